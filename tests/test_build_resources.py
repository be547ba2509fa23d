"""What the compiler made of the projection kernels.  The decode-step launches rely on two resident CTAs of gemm_kernel per
SM with their rings (ptxas reports registers per thread, and a static_assert in the launcher holds the shared memory of two
CTAs within an SM's); gemm_rows_kernel takes an SM for itself.  Neither spills.  An epilogue change that blows up the
register count still passes every numerical test and silently costs 20 % of the step: this catches it without a GPU."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
REGISTERS = 65536            # of an SM, handed out in steps of 8 per thread


def _variants(source, kernel):
    """{template arguments: (registers per thread, spilled bytes)} of a kernel's instances."""
    src = os.path.join(ROOT, "paper_2511_21759_b200", "csrc", source)
    r = subprocess.run(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xptxas", "-v", "-c", src,
                        "-o", os.devnull], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-2000:]
    out = {}
    for b in re.split(r"ptxas info\s*: Compiling entry function '", r.stderr)[1:]:
        m = re.search(kernel + r"ILi(\d+)EL[ib](\d+)E", b.split("'", 1)[0])
        if m:
            spills = sum(int(x) for x in re.findall(r"(\d+) bytes spill", b))
            assert m.groups() not in out
            out[m.groups()] = (int(re.search(r"Used (\d+) registers", b).group(1)), spills)
    return out


def _fits(ctas, threads, regs):
    return ctas * threads * (-(-regs // 8) * 8) <= REGISTERS


def test_gemm_variants_fit_two_ctas_per_sm_and_spill_nothing():
    seen = _variants("gemm_tcgen05.cu", "gemm_kernel")
    # the producer's and the issuer's warp, and groups of four epilogue warps: one for partial sums (0) and 32-row tiles,
    # two for SwiGLU (1) and the LM head (3), four for the LM head at 128 rows
    groups = {("32", "0"): 1, ("64", "0"): 1, ("128", "0"): 1, ("32", "1"): 1, ("64", "1"): 2, ("128", "1"): 2,
              ("32", "3"): 1, ("64", "3"): 2, ("128", "3"): 4}
    assert set(seen) == set(groups)
    for v, (regs, spills) in seen.items():
        assert _fits(2, 64 + 128 * groups[v], regs) and spills == 0, (v, regs, spills)


def test_many_row_gemm_variants_fit_an_sm_and_spill_nothing():
    seen = _variants("gemm_rows.cu", "gemm_rows_kernel")
    # six epilogues, each with and without single weight tiles, but for the LM head's statistics (1)
    assert set(seen) == {(str(e), h) for e in range(6) for h in "01"} - {("1", "1")}
    for v, (regs, spills) in seen.items():
        assert _fits(1, 320, regs) and spills == 0, (v, regs, spills)
