"""npp_gemm_bf16 refuses an output that is not 16-byte aligned before anything
reaches the device (its stores would fault there)."""
import ctypes

import pytest

from paper_1904_06680_gb300 import npp


@pytest.mark.parametrize("shift", [4, 8, 12])
def test_unaligned_output_is_refused(shift):
    with pytest.raises(npp.NppError, match="C must be 16-byte aligned"):
        npp._check(npp.lib().npp_gemm_bf16(ctypes.c_void_p(1 << 20), ctypes.c_void_p(1 << 20),
                                           ctypes.c_void_p((1 << 20) + shift), 128, 128, 64, None))
