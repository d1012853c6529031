"""The tensor-memory instructions are the whole warp's (.sync.aligned): where
lane-dependent code precedes one, the source has a __syncwarp or a warp-wide
vote between them (a compiler that happens to bring the lanes together again
hides its absence, so this is checked in the text)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1904_06680_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _body(code, start):
    """The braces' content of the definition that begins with `start`."""
    i = code.index("{", code.index(start))
    depth = 0
    for j in range(i, len(code)):
        depth += {"{": 1, "}": -1}.get(code[j], 0)
        if depth == 0:
            return code[i:j]
    raise AssertionError(start)


def _tmem_net():
    return _body(_code("npp_rollout.cuh"), "struct TmemNet")


def test_step_reads_ahead_after_guarded_stores():
    b = _body(_tmem_net(), "Ahead fetch_ahead() const")
    assert re.search(r"__syncwarp\(\);\s*tmem_ld16\(", b)


def test_explicit_rows_stored_after_their_guarded_loads():
    b = _body(_tmem_net(), "void load_mem(")
    for store in (r"tmem_st4\(tm \+ TAIL \+ U,", r"#pragma unroll\s*for \(int k = 0; k < B; \+\+k\) put_w2\("):
        assert re.search(r"__syncwarp\(\);\s*" + store, b), store


def test_accumulators_read_after_waits():
    """Each epilogue's wait ends in one vote, abort flag included, which brings
    the lanes together; the training epilogue's guarded reads come before its
    __syncwarp."""
    gemm, mlp = _code("npp_gemm.cu"), _code("npp_mlp.cu")
    wait = r"const bool ok = mbar_wait(?:_cluster)?\(&(?:p\.)?tfull"
    verdict = r"if \(!__all_sync\(0xffffffffu, ok && [^{|]*\{[^}]*break;\s*\}\s*tc_fence_after"
    assert len(re.findall(wait, gemm)) == len(re.findall(verdict, gemm)) == 2
    assert len(re.findall(wait, mlp)) == len(re.findall(r"if \(!epilogue_go\(p, ok\)\)", mlp)) == 4
    assert re.search(r"return __all_sync\(0xffffffffu, ok && !aborted\(p\)\);", _body(mlp, "bool epilogue_go("))
    assert re.search(r"if \(ch == 0\) fetch_rows\([^;]*;\s*__syncwarp\(\);", mlp)


@pytest.mark.parametrize("name,n", [("npp_mlp.cu", 1), ("npp_gemm.cu", 2)])
def test_allocations_after_lane_0_set_up(name, n):
    code = _code(name)
    assert len(re.findall(r"tcgen05\.alloc", code)) == n
    assert len(re.findall(r"if \(warp == 0\) \{\s*__syncwarp\(\);\s*asm volatile\(\"tcgen05\.alloc", code)) == n
