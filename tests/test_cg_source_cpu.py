"""Rules of the one-kernel CG that no result shows reliably, read from its source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1106_5908_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_vectors_never_through_the_read_only_path():
    """The kernel writes p, p2, r and x, and b may be r: none of them is loaded by __ldg,
    whose lines nothing invalidates while the kernel runs."""
    args = re.findall(r"__ldg\(((?:[^()]|\([^()]*\)|\((?:[^()]|\([^()]*\))*\))*)\)", _source("k_cg.cu"))
    assert len(args) > 5
    for arg in args:
        assert re.match(r"(q\.(order|srows|diag)|cb|m\.(rp|col)|src|static_cast<const T \*>\(m\.vs\))(\W|$)", arg.strip()), arg
    # src is a row of the matrix values
    assert re.search(r"const T \*src = vals \+", _source("k_cg.cu"))


def test_step_length_summed_in_fp64():
    """p.q is summed by FP64 FMAs of exact products whatever the vectors' type, as the
    product kernels that fuse it do."""
    src = _source("k_cg.cu")
    assert re.search(r"\bAccF64 pq;", src) and "pq.fma(pr, y)" in src
    assert "dsum = fma(widen(__ldg(x + r)), widen(q), dsum)" in _source("sell_kernel.cuh")


def test_timeouts_are_solved_on_the_other_path():
    """A grid barrier that gave up ends neither solver: both go on to the kernel-by-kernel
    path (the mixed one with its right-hand side formed anew), and the kernel leaves no
    error word behind."""
    src = _source("api.cu")
    calls = [m.end() for m in re.finditer(r"st = (?:one_kernel \? )?cg_in_one_kernel\(", src)]
    assert len(calls) == 2
    plain, mixed = (src[c:c + 900] for c in calls)
    assert "st != SPMV_ERR_UNSUPPORTED && st != SPMV_ERR_TIMEOUT) return st;" in plain
    retry = mixed[mixed.index("if (st == SPMV_ERR_TIMEOUT)"):]
    assert "cg_scale_to32(w.r64, w.r32" in retry[:retry.index("}")]
    assert "set_error" not in _source("k_cg.cu")
