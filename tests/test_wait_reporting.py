"""How kernels report a wait that ran out, as far as their sources show it (the GPU test follows one report to the host)."""
import os
import re

from paper_2603_15619_b200 import build


def source(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_the_first_site_of_a_cta_is_kept():
    # the code goes into the CTA's abort word by compare-and-swap from 0, never by a plain store
    ptx = source("sm100_ptx.cuh")
    wait = ptx[ptx.index("void mbar_wait("):ptx.index("void mbar_wait2(")]
    assert "atom.shared.cas.b32" in wait and "st.volatile.shared" not in wait


def kernels(text):
    for m in re.finditer(r"__global__", text):
        name = re.search(r"(\w+)\(", re.sub(r"__launch_bounds__\([^)]*\)", "", text[m.end():m.end() + 400])).group(1)
        start = end = text.index("{", m.end())
        depth = 0
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        yield name, text[start:end]


def test_every_kernel_that_waits_tears_down_with_the_report():
    # mbar_wait only marks the CTA: a kernel without the tear-down would return garbage with status 0
    seen = set()
    for f in sorted(os.listdir(build.CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        for name, body in kernels(source(f)):
            waits = [m.end() for m in re.finditer(r"\bmbar_wait2?\(", body)]
            if not waits:
                continue
            seen.add(name)
            calls = [m.start() for m in re.finditer(r"\babort_teardown\(", body)]
            assert len(calls) == 1 and calls[0] > max(waits), name
            # one elected thread reports; all threads pass a barrier before and after
            assert re.search(r"__syncthreads\(\);\s*abort_teardown\(&?\w+, \d+\);\s*(__syncthreads|cluster_sync_all)\(\);", body), name
            assert "report_abort(" not in body, name
    assert seen == {"moda_fwd_kernel", "moda_fwd2_kernel", "bwd_rows_kernel", "moda_bwd_fused_kernel", "moda_bwd_dq_kernel",
                    "moda_bwd_dkdv_kernel", "moda_kv_project_kernel", "wait_timeout_selftest_kernel"}, seen


def test_the_decode_wait_reports_its_own_site():
    # not what the abort word holds, which another wait of the CTA may have written meanwhile
    decode = source("moda_decode.cuh")
    body = dict(kernels(decode))["decode_split_tma_kernel"]
    assert "decode_wait(" in body and "mbar_wait" not in body
    wait = decode[decode.index("void decode_wait("):decode.index("decode_split_tma_kernel")]
    assert "report_abort(kStatusWaitTimeout | (site << 8));" in wait
