// Sizes of launches that a call chooses by its shape: host arithmetic without CUDA, so that it can be checked on the CPU.
#pragma once

#include <algorithm>
#include <cmath>

namespace moda {

// Whether a d = 128 forward takes the kernel with two softmax warpgroups (moda_fwd_wide128.cuh).  It is the faster one where the key tiles
// set the pace; where the depth slots do, its ring of three units against five and the smaller register share of its depth warps
// cost it up to a fifth.  us, one warpgroup -> two (B = 2, 16 heads): l = 0: T = 128 7.2 -> 7.2, T = 1000 23.9 -> 22.2, T = 2048 57.7 -> 51.9,
// T = 8192 552 -> 481, T = 16384 2339 -> 1964.  l = 4: T = 1000 27.1 -> 25.8, T = 512 11.4 -> 11.8.  l = 8: T = 4096 238 -> 223, T = 2048 84.0 -> 84.3,
// T = 1000 33.1 -> 37.9.  l = 16: T = 8192 716 -> 714 and 719 -> 650, T = 4096 268 -> 291.  l = 24: T = 16384 2545 -> 2420, T = 8192 802 -> 842.  e4m3,
// l = 8: T = 2048 73.6 -> 73.4, T = 1000 30.2 -> 33.8; l = 16: T = 8192 714 -> 631, T = 4096 235 -> 260.  2000 over 15000, l = 24, B = 4: 1192 -> 985.
// With a key tile or two there is little to alternate: T = 100, 2 heads: l = 1 7.26 -> 7.35, l = 2 7.81 -> 8.08 (e4m3 7.77 -> 8.39); T = 129: l = 1 7.68 -> 7.53, l = 2
// 8.08 -> 8.28; T = 256, B = 4, 32 heads: l = 1 16.4 -> 16.2, l = 2 17.4 -> 17.7; T = 300: l = 2 26.2 -> 26.0 (e4m3 26.1 -> 26.2).
inline bool fwd_two_softmax(int T_q, int T_kv, int l) {
    const long long keys = 2ll * T_kv - T_q;                 // twice the mean number of keys of a query: T when T_q = T_kv = T
    return keys > 128 && 128ll * l < keys && 560ll * l <= keys + 1120;
}

// How many SMs the depth part of a fused backward gets beside the sequence part.  Measured SM time: an entry of the row
// ring 1.75 us (16 SMs at it) to 2.0 us (50), e4m3 a tenth more; an iteration of the sequence part at d = 128 2.7 us
// and 5 us per key tile around them; at d = 64 11 us per key tile and 1.33 us an iteration, rising to 1.5 us for the longest (their runs
// last long enough for the clocks to come down, which the depth part, bound by HBM, does not feel).  With the share
// x = depth / (depth + sequence) of all SMs both
// parts end together; a few SMs more than that cost less than a few too few, because SMs that the depth part leaves go on
// with the sequence part.  The number is even: with an odd one a CTA shares its pair of SMs with a CTA of the sequence part,
// and the whole depth part waits for that one.
// Whole backward, us, by SMs (rounds of one count differ by 4-8 %).  d = 128, bf16:
// T = 8192, l = 16, B = 2: 34 2167, 36 2057, 38 1979, 40 2000, 44 1994 (taken: 40); T = 4096, l = 23, B = 4: 66 1664,
// 70 1602, 74 1619, 78 1634 (72).  e4m3: T = 5000, l = 23, B = 2: 64 1111, 68 1075, 72 1086, 76 1099 (70); T = 8192, l = 16: 38 1962, 42 1882,
// 46 1965 (42); T = 32768, l = 24: 18 11551, 20 11102, 24 11776 (20).  At least 16: with x from 3 to 12 every count from x + 15 % to 20 is within
// 1 % (18 shapes, counts in shuffled order; T = 65536, l = 24: 10 45.1, 16 45.4, 20 45.3 ms), and up to three too few cost 10-20 %.
// d = 64 (counts in shuffled order), bf16: T = 8192, l = 16, B = 2, 32
// heads: 32 2271, 34 2186, 36 2227, 40 2236 (36); T = 16384, l = 32, 32 heads: 34 4299, 36 4186, 38 4212, 44 4183 (38); T = 32768, l = 32, 32 heads: 18 15691,
// 20 14487, 22 13729, 24 13972, 28 13601 (22); T = 65536, l = 60, 16 heads: 18 27895, 20 27103, 22 26983 (20); e4m3: T = 5000, l = 23, B = 2, 32 heads: 58 1194, 62 1194,
// 68 1207 (62); T = 32768, l = 32: 20 14715, 22 13607, 24 13220, 28 13456 (24).
//
// With 16 units an SM or fewer the time goes in steps, by the units of the busiest SM ("rounds"): one round less is worth some SMs more, the more of
// them the fewer rounds there are; if it takes too many, the rounds stay and the count is the smallest with as many (then also below 16: 20
// units in two rounds are 10 CTAs).  us by SMs, 32 heads, B = 4, l = 6, d = 64: T = 100 (64 units, x = 47): 32 31.3, 64 21.6 (64);
// T = 300: 48 60.7, 64 57.7, 96 57.5 (48); T = 500, l = 12: 64 114.4, 80 112.5, 86 100.5, 128 112.6 (86).  d = 128, l = 6: T = 300 (384 units,
// x = 79): 78 93.3, 86 93.6, 96 96.7 (78); T = 500 (x = 74): 64 136.3, 74 131.2, 80 131.5, 86 133.8 (74); T = 1024, l = 30, e4m3, 16 heads (512 units,
// x = 115): 104 370, 124 370, 128 345 (128).
// Mean loss against the best count over 189 and, with other sizes, 150 shapes of at most 16 rounds: d = 64 1.2 and 1.8 % (with one limit of 12 % on the
// SMs that a round less may take, and 12 us a key tile: 4.0 and 2.6 %), d = 128 1.2 and 1.4 % (1.7 and 1.7 %).
inline unsigned bwd_row_ctas(int d, long long bh, int T, int l, unsigned units, unsigned sms, bool fp8) {
    const double nq = (T + 127) / 128, n = nq + 1;
    const double depth = double(units) * (l + 1) * (fp8 ? 1.9 : 1.7);
    const double seq = double(bh) * nq * (d == 128 ? 5.0 + 1.36 * n : 11.0 + (0.66 + 0.00035 * n) * n);
    const double x = sms * depth / (depth + seq);
    const auto even = [](double c) { return 2 * unsigned(std::ceil(c / 2)); };
    unsigned share = std::min(sms, std::max(16u, even(d == 128 ? 1.06 * x + 1.0 : 1.1 * x + 2.0)));
    const unsigned rounds = (units + share - 1) / share;
    if (rounds > 1 && rounds <= 16) {
        const unsigned fewer = even(std::ceil(double(units) / (rounds - 1)));
        const unsigned most = d == 128 ? 104 + 10 / (rounds - 1) : 115 + 15 / (rounds - 1);     // percent of the share
        share = (100 * fewer <= most * share && fewer <= sms) ? fewer : even(std::ceil(double(units) / rounds));
    }
    return std::min(units, std::min(share, sms));
}

// Whether the two row warpgroups of the fused backward's sequence part (d = 64) take alternate iterations, or share each (moda_bwd_fused.cuh).
// A CTA has G (tiles + 1) / 2 iterations in the mean; with few of them the one or two that do not come in pairs weigh more than what the
// pairs win.  Whole backward, l = 0, us, shared / alternate, by batch x heads: T = 100: 1 x 2 10.5 / 11.3, 8 x 32 19.8 / 21.4; T = 256: 12.2 / 12.8, 41.9 / 45.0; T = 512:
// 15.1 / 15.4, 93.0 / 96.7; T = 640: 16.5 / 16.5, 124 / 128; T = 768 (twice the mean = 7): 18.0 / 17.7, 2 x 16 27.7 / 28.2, 156 / 160; T = 900 (9): 20.7 / 20.0,
// 36.3 / 35.7, 218 / 220; T = 1200: 23.6 / 22.4, 45.9 / 45.0, 303 / 303; T = 2000: 31.8 / 29.6, 88.3 / 85.3, 4 x 32 331 / 322.  G = 4: T = 100 (8) 15.8 / 16.0,
// T = 300 (16) 27.2 / 26.4; G = 8: T = 100 (16) 21.3 / 20.9, T = 256 (24) 38.1 / 36.1.
inline bool bwd_alternates(int d, int T, int G) { return d == 64 && G * ((T + 127) / 128 + 1) > 7; }

}  // namespace moda
