"""What the kernel sources must keep that no output shows."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_13768_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_overlapped_kernels_read_by_coherent_loads():
    """A kernel launched with launch_overlapped is resident while the kernel
    before it writes the field it reads: no read-only (non-coherent) loads, nor
    plain reads through a const __restrict__ pointer, which the compiler may
    turn into them; and each waits before anything else."""
    launched = set()
    headers = {n: _read(n) for n in sorted(os.listdir(CSRC)) if n.endswith((".cuh", ".cu"))}
    for text in headers.values():
        launched |= set(re.findall(r"launch_overlapped\((\w+)<", text))
    assert launched == {"sweep_pair", "sweep_pair_k", "sweep_col", "boundary_fix"}
    for name in ("wfa_sweep.cuh", "wfa_sweep_col.cuh", "wfa_sweep_pair.cuh", "wfa_sweep_pair_k.cuh"):
        assert not re.search(r"__ldg\b|ld\.global\.nc|ldca|ld\.relaxed", headers[name]), name
    whole = "\n".join(headers.values())
    for k in launched:
        body = re.search(r"\b%s\(const __grid_constant__ SweepArgs a[^)]*\) \{(.*?)\n\}\n" % k, whole, re.S).group(1)
        assert body.index("grid_wait(tin, rk);") < min(
            body.index(s) for s in ("return", "(const S*)tin", "rk + ", "(a.c") if s in body), k
        assert "a.tin" not in body.split("grid_wait", 1)[1] and "a.rk" not in body.split("grid_wait", 1)[1], k
    cell = re.search(r"float general_cell\((.*?)\n\}\n", headers["wfa_sweep.cuh"], re.S).group(1)
    assert not re.search(r"\b(in|rk)\[", cell)
