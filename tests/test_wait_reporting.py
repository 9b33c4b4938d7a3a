"""How kernels report a wait that ran out, as far as their sources show it (the GPU test follows one report to the host)."""
import os
import re

from paper_2603_15619_b200 import build


def source(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_the_first_site_of_a_cta_is_kept():
    # the code goes into the CTA's abort word by compare-and-swap from 0, never by a plain store
    ptx, decode = source("sm100_ptx.cuh"), source("moda_decode.cuh")
    wait = ptx[ptx.index("void mbar_wait("):ptx.index("void mbar_wait2(")]
    assert "atom.shared.cas.b32" in wait and "st.volatile.shared" not in wait
    wait = decode[decode.index("void decode_wait("):decode.index("decode_split_tma_kernel")]
    assert "atomicCAS(const_cast<int*>(abort_flag), 0," in wait and not re.search(r"\*abort_flag = ", wait)
