"""The build refuses a cache-fill attention whose launcher would refuse every launch for want of registers."""
import os

import pytest

from paper_2510_04147_b200 import build


def _log(*regs):
    return "".join(f"ptxas info    : Compiling entry function '_Z1k' for 'sm_100a'\nptxas info    : Used {r} registers, used 1 barriers\n" for r in regs)


def test_register_shares_of_the_cache_fill_attention():
    with open(os.path.join(build.CSRC, "attention_fill_tc.cu")) as f:
        source = f.read()
    build.check_register_shares(source, _log(168, 168))            # 256 * 208 + 128 * 80 of 384 * 168
    for log in (_log(168, 160), _log(165), ""):
        with pytest.raises(RuntimeError, match="register shares"):
            build.check_register_shares(source, log)


def test_kernels_that_shift_no_registers_are_not_looked_at():
    with open(os.path.join(build.CSRC, "gemm.cu")) as f:
        build.check_register_shares(f.read(), _log(96))
