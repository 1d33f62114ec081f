"""The build refuses tensor-core kernels whose register count is not the one
that their warps share out."""
import os
import re

import pytest

from paper_1704_07458_gb300 import build

SRC = os.path.join(build.CSRC, "ozaki_tc.cu")
WANT = int(re.search(r"\bkURegs = (\d+)", open(SRC).read()).group(1))


def _log(gram, update):
    entry = ("ptxas info    : Compiling entry function '_ZN3lob{}ILi6EEEv' for 'sm_103a'\n"
             "ptxas info    : Function properties for _ZN3lob{}ILi6EEEv\n"
             "    0 bytes stack frame, 0 bytes spill stores, 0 bytes spill loads\n"
             "ptxas info    : Used {} registers, used 1 barriers\n")
    return "".join(entry.format(k, k, r) for k, r in
                   (("20ozaki_gram_tc_kernel", gram), ("22ozaki_update_tc_kernel", update),
                    ("14row_exp_kernel", 32)))


def test_register_shares_are_checked():
    build.check_registers(SRC, _log(WANT, WANT))
    build.check_registers(os.path.join(build.CSRC, "spmm.cu"), "")
    for log in (_log(WANT - 8, WANT), _log(WANT, WANT + 8), ""):
        with pytest.raises(RuntimeError):
            build.check_registers(SRC, log)
