"""Register spills of kernels that lost time to them, from the report that ptxas wrote when the library was built."""
import os
import re
import subprocess

import pytest

from paper_2603_15619_b200 import build

REPORT = os.path.join(build.PKG, "build_ptxas.log")

# kernel: most bytes of spill stores, of spill loads
LIMITS = {
    "decode_split_tma_kernel<128, 1>": (0, 0),
    "decode_split_tma_kernel<128, 2>": (48, 60),
    "moda_fwd_kernel<128, 2, false>": (0, 0),
    "moda_fwd_kernel<128, 2, true>": (0, 0),
    "moda_fwd_kernel<128, 1, false>": (0, 0),
}


def spills():
    found, name = {}, None
    for line in open(REPORT):
        if m := re.search(r"Compiling entry function '(\S+)'", line):
            name = m.group(1)
        elif (m := re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)) and name:
            found.setdefault(name, (int(m.group(1)), int(m.group(2))))
    plain = subprocess.run(["c++filt"], input="\n".join(found), capture_output=True, text=True, check=True).stdout.splitlines()
    short = lambda n: n.split("(")[0].replace("void ", "").replace("moda::", "")
    return {short(n): v for n, v in zip(plain, found.values())}


@pytest.mark.skipif(not os.path.exists(REPORT), reason="the library was not built here")
@pytest.mark.parametrize("kernel", LIMITS)
def test_spills_stay_within_limits(kernel):
    stores, loads = spills()[kernel]
    most = LIMITS[kernel]
    assert stores <= most[0] and loads <= most[1], (kernel, stores, loads)
