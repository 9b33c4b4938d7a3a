// How the key range of a decode step is cut into pieces: host and device arithmetic without CUDA, so that it can be checked on
// the CPU.
//
// The keys of a sequence are counted in units of 2^unit_log2 keys (one stage of the split kernel's ring, 64 keys, unless the
// step is so large that the units of all sequences would not fit an int).  A "group" is a sequence with the key/value heads that
// one team of CTAs takes at a time; the groups lie one behind the other in an order of all units, which is cut into runs of
// equal length, one per team.  A team works on the piece of each group that its run covers.
//
// A piece costs about a stage and a half besides its keys (its start, the merge of the warps, a partial to write and read; with 8
// query heads in a group about six).  Where the runs can be cut so that every team has one piece (`aligned`: a group then takes a
// multiple of the run in the order), that is preferred to somewhat shorter runs that cross from one group to the next.  us, runs that
// cross -> aligned: B = 8, T = 4096, 6 heads, G = 2, d = 64: 15.5 -> 13.1; lengths uniform in [1, 4096], B = 8, 2 heads, G = 4,
// d = 128: 13.8 -> 9.5; B = 128, lengths to 1000, 1 head, G = 8, d = 128: 21.9 -> 16.7.  Longer aligned runs than these lose
// again (B = 16, T = 2048, 6 heads, G = 2, d = 64: runs of 22 that cross 14.0, aligned ones of 32 16.6).
#pragma once

#if defined(__CUDACC__)
#define MODA_HD __host__ __device__ __forceinline__
#else
#define MODA_HD inline
#endif

namespace moda {

constexpr int kDecodeStageKeys = 64;
constexpr int kDecodeStageLog2 = 6;
constexpr int kDecodeMaxSplits = 128;                      // partials of a group that the workspace holds

MODA_HD int decode_units(int len, int unit_log2) { return ((len - 1) >> unit_log2) + 1; }      // len >= 1
MODA_HD int decode_ceil_div(int a, int b) { return (a + b - 1) / b; }
MODA_HD int decode_run(int total, int teams, int min_run) {
    const int run = decode_ceil_div(total, teams);
    return run > min_run ? run : min_run;
}
// The longest aligned run that is better than runs of `run` units that cross groups; G: query heads of a group.
MODA_HD int decode_aligned_run(int run, int G) { return run + 1 + run / 8 + (G == 8 ? 6 : 0); }

// Unit of a step of at most T_kv keys per sequence: the units of all groups, rounded up to aligned runs, stay below 2^30.
inline int decode_unit_log2(long long groups, int T_kv) {
    int u = kDecodeStageLog2;
    while (groups * decode_units(T_kv, u) > (1ll << 28) && u < 30) ++u;
    return u;
}
// Shortest run: four units, one for each pair of consumer warps (a shorter run takes as long), and enough that no group is cut
// into more than kDecodeMaxSplits - 1 pieces.
inline int decode_min_run(int T_kv, int unit_log2) {
    const int cap = decode_ceil_div(decode_units(T_kv, unit_log2), kDecodeMaxSplits - 2);
    return cap > 4 ? cap : 4;
}

// The cut: length of a run, and whether groups take whole runs.
struct DecodeCut {
    int run;
    int aligned;
};
// All sequences have T_kv keys.
inline DecodeCut decode_cut_equal(int groups, int T_kv, int unit_log2, int teams, int G) {
    const int ns = decode_units(T_kv, unit_log2), least = decode_min_run(T_kv, unit_log2);
    DecodeCut cut{decode_run(groups * ns, teams, least), 0};
    if (groups <= teams) {
        int pieces = teams / groups;                       // that many per group have a team each
        const int even = decode_ceil_div(ns, pieces);
        const int run = even > least ? even : least;
        if (run <= decode_aligned_run(cut.run, G)) cut = DecodeCut{run, 1};
    }
    return cut;
}

struct DecodePiece {
    int b, head_team;            // sequence; team of heads within it
    int k_begin, k_end;          // keys
    int index, pieces;           // which piece of its group, and of how many
};

// The pieces of one team's run.  `Len` gives the keys of a sequence.
struct DecodeWalk {
    int b, head_team, ns, stride;   // group: its sequence and team of heads, its units, and the units that it takes in the order
    int start, at, end;             // its first unit and the next one of ours in the order of all; end of our run

    MODA_HD static int stride_of(int ns, const DecodeCut& cut) {
        return cut.aligned ? decode_ceil_div(ns, cut.run) * cut.run : ns;
    }
    // `b0`: sequence that the run starts in, `before`: units (as they stand in the order) per team of heads before it
    template <class Len>
    MODA_HD void begin(const DecodeCut& cut, int team, int total, int heads, int unit_log2, int b0, int before, const Len& len) {
        at = team * cut.run;
        end = at + cut.run < total ? at + cut.run : total;
        b = b0;
        ns = at < total ? decode_units(len(b0), unit_log2) : 1;
        stride = stride_of(ns, cut);
        head_team = (at - before * heads) / stride;
        start = before * heads + head_team * stride;
    }
    MODA_HD bool done() const { return at >= end; }
    template <class Len>
    MODA_HD DecodePiece piece(const DecodeCut& cut, int team, int unit_log2, const Len& len) const {
        DecodePiece w;
        const int s0 = at - start, s1 = end - start;
        w.b = b;
        w.head_team = head_team;
        w.k_begin = s0 << unit_log2;
        w.k_end = s1 < ns ? s1 << unit_log2 : len(b);
        const int first = start / cut.run;
        w.index = team - first;
        w.pieces = (start + ns - 1) / cut.run - first + 1;
        return w;
    }
    template <class Len>
    MODA_HD void next(const DecodeCut& cut, int heads, int unit_log2, const Len& len) {
        start += stride;
        at = start;
        if (++head_team == heads) {
            head_team = 0;
            ++b;
            if (at < end) {
                ns = decode_units(len(b), unit_log2);
                stride = stride_of(ns, cut);
            }
        }
    }
};

// Pieces of group `group` when all sequences have T_kv keys.
MODA_HD int decode_pieces_equal(const DecodeCut& cut, int group, int T_kv, int unit_log2) {
    const int ns = decode_units(T_kv, unit_log2);
    if (cut.aligned) return decode_ceil_div(ns, cut.run);
    const int start = group * ns;
    return (start + ns - 1) / cut.run - start / cut.run + 1;
}

}  // namespace moda
