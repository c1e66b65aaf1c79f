"""What the kernel sources must keep that no output shows."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_13768_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_overlapped_kernels_read_by_coherent_loads():
    """A kernel launched with launch_overlapped is resident while the kernel
    before it writes the field it reads: no read-only (non-coherent) loads of it,
    nor plain reads through a const __restrict__ pointer, which the compiler may
    turn into them; and each waits before anything else. 1/k alone is read by
    that path: a pass right after the kernel that wrote it does not overlap."""
    launched = set()
    headers = {n: _read(n) for n in sorted(os.listdir(CSRC)) if n.endswith((".cuh", ".cu"))}
    for text in headers.values():
        calls = re.findall(r"launch_overlapped\((\w+)<[^;]*;", text)
        launched |= set(calls)
        assert len(calls) == len(re.findall(r"launch_overlapped\(\w+<[^;]*, st, !a\.fresh_k, a[^;]*;", text))
    assert launched == {"sweep_pair", "sweep_pair_k", "sweep_col", "boundary_fix"}
    for name in ("wfa_sweep.cuh", "wfa_sweep_col.cuh", "wfa_sweep_pair.cuh", "wfa_sweep_pair_k.cuh"):
        text = re.sub(r"void (ldrk|load_rk)\((.*?)\n\s*(}|RowBuf|__device__)", "", headers[name], flags=re.S)
        text = re.sub(r"__ldg\((rk \+ \w|reinterpret_cast<const float\*>\(rp\))", "", text)
        assert not re.search(r"__ldg\b|ld\.global\.nc|ldca|ld\.relaxed", text), name
    pair_k = headers["wfa_sweep_pair_k.cuh"]
    assert not re.search(r"\b(t|T[01n]|Tc\[j\]|H\[\d\])\.load_rk", pair_k)
    whole = "\n".join(headers.values())
    for k in launched:
        body = re.search(r"\b%s\(const __grid_constant__ SweepArgs a[^)]*\) \{(.*?)\n\}\n" % k, whole, re.S).group(1)
        assert body.index("grid_wait(tin, rk);") < min(
            body.index(s) for s in ("return", "(const S*)tin", "rk + ", "(a.c") if s in body), k
        assert "a.tin" not in body.split("grid_wait", 1)[1] and "a.rk" not in body.split("grid_wait", 1)[1], k
    cell = re.search(r"float general_cell\((.*?)\n\}\n", headers["wfa_sweep.cuh"], re.S).group(1)
    assert not re.search(r"\b(in|rk)\[", cell)
    prepare = re.search(r"int prepare_k_halo\((.*?)\n\}\n", headers["wfa_grid.cu"], re.S).group(1)
    assert prepare.index("recip_kernel") < prepare.index("k_fresh = true")
    planes = re.search(r"static int planes\((.*?)\n\}\n", headers["wfa_slabs.cu"], re.S).group(1)
    assert "if (what == WFA_PLANES_RECIP_K) g->k_fresh = true;" in planes   # its caller writes the halo plane of 1/k


def _depths(body, call):
    """Brace depth, from the start of a function's text, of each place of `call`."""
    return [body[:m.start()].count("{") - body[:m.start()].count("}") for m in re.finditer(re.escape(call), body)]


def test_cg_inner_products_add_four_products_at_a_time():
    """The inner products of CG sum 4 fp32 products (a row's cells of a thread)
    between compensated additions: those additions stand in the loop over a
    thread's rows (function, if, loop), not behind it."""
    text = _read("wfa_implicit.cu")
    rows = re.search(r"void cg_rows\(.*?\) \{(.*?)\n\}\n", text, re.S).group(1)
    assert len(_depths(rows, "dot.add(")) == 2 and min(_depths(rows, "dot.add(")) >= 2
    res = re.search(r"cg_res_u\(const __grid_constant__ CgArgs a\) \{(.*?)\n\}\n", text, re.S).group(1)
    assert _depths(res, "rr.add(") == [3]   # rows present, planes, rows
