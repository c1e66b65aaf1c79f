"""The work a user of this package has it do, as measurable cases.

Every case is a whole call sequence through the public entry points
(``Grid``, ``batch_run``, ``Server``, ``stencil.compile``): inputs that a user
has in hand are made by ``prepare``, and ``run`` takes them to the result. The
library's inputs and results are host arrays by its interface, so the marching,
batched and served cases start from pinned host fields and end with the result
on the host; the expression front end works on CUDA tensors.

Kinds of case (``case["kind"]``):
  march     a solve on a grid whose coefficients are set: set the field, take
            the steps, read the field back
  solve     a solve from nothing but host arrays on an existing handle:
            conductivity, field, stability limit, steps, field and total heat
  batch     many grids of different sizes and step counts in one call
  serve     a burst of independent requests to the continuous-batching server
  implicit  backward-Euler steps by conjugate gradients
  stencil   an update written in the expression front end

Sizes are those of the package's own workloads and benchmark lines, with
ragged ones of its tests' kind in between; `draw` spreads over the range.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2209_13768_gb300 as wfa
from paper_2209_13768_gb300 import stencil as S

F32, BF16 = wfa.F32, wfa.BF16

# boundary conditions by name: six (kind, value) pairs, -x +x -y +y -z +z
D, ZF, P, DC = "dirichlet", "zeroflux", "periodic", "dirichlet_cell"
FACES = {
    "cold": [(D, 0.0)] * 6,                                     # T = 0 on every face
    "slab": [(D, 1.0), (D, 0.0)] + [(ZF, 0.0)] * 4,             # hot and cold x faces, the rest insulated
    "channel": [(P, 0.0)] * 2 + [(ZF, 0.0)] * 4,                # periodic x, walls in y and z
    "held": [(DC, 1.0)] + [(DC, 0.0)] * 5,                      # outer cell layers held, one side hot
    "torus": [(P, 0.0)] * 6,                                    # periodic on every axis
}
WIND = (0.3, 0.1, 0.05)   # cells per unit time, the advection-diffusion workload's velocity


def listed():
    return [
        # the smallest real problem: the 64^3 heat test problem, 100 steps
        # (the field fits one SM group's on-chip memory; launches dominate)
        dict(name="heat_64", kind="march", nx=64, ny=64, nz=64, storage="f32", k="uniform", faces="cold",
             advect=False, steps=100),
        # a mid-size ragged conductivity problem with bf16 storage: rows that
        # are no multiple of a vector, per-cell k, hot and cold faces
        dict(name="ragged_bf16_k", kind="march", nx=333, ny=250, nz=187, storage="bf16", k="lognormal",
             faces="slab", advect=False, steps=200),
        # the benchmark's headline workload as a user runs it: per-cell k at
        # 512^3 from host arrays to the field and its heat
        dict(name="lognormal_512", kind="solve", nx=512, ny=512, nz=512, storage="f32", k="lognormal",
             faces="slab", advect=False, steps=200),
        # the largest: advection-diffusion at 1024 x 1024 x 512, both storage types
        dict(name="advdiff_1024_f32", kind="march", nx=1024, ny=1024, nz=512, storage="f32", k="uniform",
             faces="channel", advect=True, steps=200),
        dict(name="advdiff_1024_bf16", kind="march", nx=1024, ny=1024, nz=512, storage="bf16", k="uniform",
             faces="channel", advect=True, steps=200),
        # parameter studies: 256 independent grids of 16..128 cells an edge,
        # 50..500 steps each, in one call
        dict(name="batch_256", kind="batch", count=256, lo=16, hi=128, smin=50, smax=500, shapes=4),
        # serving: a burst of 32 mixed requests (heat / advection-diffusion,
        # f32 / bf16) of 32..256 cells an edge, 50..2000 steps
        dict(name="serve_32", kind="serve", count=32, lo=32, hi=256, smin=50, smax=2000, shapes=5),
        # implicit steps: the smallest (the launch latency of a CG iteration),
        # the paper's setting at 512^3, and a stiff ragged one with per-cell k
        # (large steps are what the implicit form is for)
        dict(name="implicit_64", kind="implicit", nx=64, ny=64, nz=64, k="uniform", faces="held", dt=0.1, steps=10,
             method="classic"),
        dict(name="implicit_512", kind="implicit", nx=512, ny=512, nz=512, k="uniform", faces="held", dt=0.1,
             steps=5, method="classic"),
        dict(name="implicit_stiff_k", kind="implicit", nx=390, ny=322, nz=257, k="lognormal", faces="slab", dt=2.0,
             steps=3, method="classic"),
        # the expression front end: the paper's heat step at 512^3, and two
        # coupled fields on a ragged grid
        dict(name="stencil_heat_512", kind="stencil", update="heat", nx=512, ny=512, nz=512, steps=100),
        dict(name="stencil_coupled", kind="stencil", update="coupled", nx=203, ny=161, nz=142, steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same ranges (half the drawn cases march a grid,
    the commonest use)."""
    kind = rng.choice(["march", "march", "march", "solve", "batch", "serve", "implicit", "implicit", "stencil"])
    if kind in ("march", "solve"):
        lo = 16 if kind == "march" else 48
        n = [_log_int(rng, lo, 640) for _ in range(3)]
        cells = n[0] * n[1] * n[2]
        advect = rng.random() < 0.4
        steps = min(_log_int(rng, 20, 1000), max(20, int(6e10 / cells)))
        faces = rng.choice(["cold", "slab", "channel", "held", "torus"])
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], storage=rng.choice(["f32", "f32", "bf16"]),
                    k="uniform" if advect and rng.random() < 0.7 else rng.choice(["uniform", "lognormal", "lognormal"]),
                    faces=faces, advect=advect, steps=steps)
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 2, 256), lo=16, hi=_log_int(rng, 32, 128), smin=20,
                    smax=_log_int(rng, 50, 500), shapes=rng.randrange(1 << 20))
    if kind == "serve":
        return dict(kind=kind, count=_log_int(rng, 4, 32), lo=32, hi=_log_int(rng, 64, 224), smin=50,
                    smax=_log_int(rng, 100, 1500), shapes=rng.randrange(1 << 20))
    if kind == "implicit":
        n = [_log_int(rng, 16, 448) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], k=rng.choice(["uniform", "lognormal"]),
                    faces=rng.choice(["cold", "slab", "held", "torus"]),
                    dt=round(math.exp(rng.uniform(math.log(0.05), math.log(5.0))), 4), steps=rng.randint(1, 6),
                    method=rng.choice(["classic", "classic", "classic", "pipelined"]))
    n = [_log_int(rng, 32, 512) for _ in range(3)]
    return dict(kind=kind, update=rng.choice(["heat", "coupled"]), nx=n[0], ny=n[1], nz=n[2],
                steps=_log_int(rng, 10, 200))


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _field(shape, gen, blob):
    """Initial field (nz, ny, nx) on the GPU: uniform [0, 1), or for advection
    a Gaussian blob near the centre (its place and width from the generator)."""
    nx, ny, nz = shape
    if not blob:
        return torch.rand((nz, ny, nx), generator=gen, device="cuda")
    c = (0.45 + 0.1 * torch.rand(3, generator=gen, device="cuda")).tolist()
    sigma = max(2.0, min(shape) / 16.0) * (0.8 + 0.4 * torch.rand(1, generator=gen, device="cuda").item())
    e = [torch.exp(-((torch.arange(n, device="cuda", dtype=torch.float32) - f * n) ** 2) / (2 * sigma * sigma))
         for n, f in zip((nx, ny, nz), c)]
    return e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]


def _conductivity(shape, gen):
    nx, ny, nz = shape
    return torch.exp(0.5 * torch.randn((nz, ny, nx), generator=gen, device="cuda"))


def _pinned(t):
    h = torch.empty(t.shape, dtype=torch.float32, pin_memory=True)
    h.copy_(t)
    return h


def _single(case, seed):
    """(shape, T0, k, u, faces, dt rule) of a march / solve case, on the GPU."""
    shape = (case["nx"], case["ny"], case["nz"])
    gen = _gen(seed)
    adv = case["advect"]
    T0 = _field(shape, gen, adv)
    if case["k"] == "lognormal":
        k = _conductivity(shape, gen)
    else:
        k = 0.05 if adv else 1.0
    return shape, T0, k, (WIND if adv else (0.0, 0.0, 0.0)), FACES[case["faces"]]


def _edges(rng, lo, hi):
    return tuple(int(v) for v in np.rint(np.exp(rng.uniform(np.log(lo), np.log(hi), 3))))


def _mix(case):
    """Shapes, step counts and kinds of a batch or a burst of requests (the
    fields come from the seed; who asks for which size does not)."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["count"]):
        shape = _edges(rng, case["lo"], case["hi"])
        steps = int(rng.integers(case["smin"], case["smax"] + 1))
        heat = case["kind"] == "batch" or bool(rng.random() < 0.5)
        storage = F32 if case["kind"] == "batch" or rng.random() < 0.5 else BF16
        out.append((shape, steps, heat, storage))
    return out


def _mix_inputs(case, seed):
    """One (shape, steps, storage, T0, k, u, faces, dt or 0) per grid or request."""
    gen = _gen(seed)
    out = []
    for shape, steps, heat, storage in _mix(case):
        T0 = _field(shape, gen, not heat)
        if heat:
            out.append((shape, steps, storage, T0, _conductivity(shape, gen), (0.0, 0.0, 0.0), FACES["cold"], 0.0))
        else:
            out.append((shape, steps, storage, T0, 0.05, WIND, FACES["channel"], 1.0))
    return out


HEAT_W = 0.1
REACT = (0.08, 0.05, 0.02)   # diffusion of both coupled fields, exchange rate


def _program(update):
    if update == "heat":
        T, w = S.Field("T"), S.Param("w")
        return {T: T + w * (T[-1, 0, 0] + T[1, 0, 0] + T[0, -1, 0] + T[0, 1, 0] + T[0, 0, -1] + T[0, 0, 1] - 6 * T)}
    a, b = S.Field("a"), S.Field("b")
    da, db, q = S.Param("da"), S.Param("db"), S.Param("q")

    def lap(f):
        return f[-1, 0, 0] + f[1, 0, 0] + f[0, -1, 0] + f[0, 1, 0] + f[0, 0, -1] + f[0, 0, 1] - 6 * f

    return {a: a + da * lap(a) - q * (a - b), b: b + db * lap(b) + q * (a - b)}


def _dt_for(g, adv, uniform):
    """The workload's own dt: 1 for uniform-k advection-diffusion, else 0.9 of
    the stability limit."""
    return 1.0 if adv and uniform else 0.9 * g.stability_dt()


class _Served:
    """A server with its requests' host buffers; closed with the state."""

    def __init__(self, reqs):
        self.server = wfa.Server(64 << 30)
        self.reqs = reqs

    def __del__(self):
        try:
            self.server.close()
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("march", "solve"):
        shape, T0, k, u, faces = _single(case, seed)
        st = BF16 if case["storage"] == "bf16" else F32
        uniform = case["k"] == "uniform"
        hk = k if uniform else _pinned(k)
        g = wfa.Grid(shape, storage=st)
        g.set_bcs(faces)
        if kind == "march":
            g.set_coeffs(hk, u)
            g.set_dt(_dt_for(g, case["advect"], uniform))
        return dict(kind=kind, g=g, T0=_pinned(T0), k=hk, u=u, case=case,
                    out=torch.empty(T0.shape, dtype=torch.float32, pin_memory=True))
    if kind == "batch":
        grids, fields, outs, steps = [], [], [], []
        mix = _mix_inputs(case, seed)
        flat = torch.empty(sum(m[3].numel() for m in mix), dtype=torch.float32, pin_memory=True)   # every grid's result
        at = 0
        for shape, n, storage, T0, k, u, faces, dt in mix:
            g = wfa.Grid(shape, storage=storage)
            g.set_bcs(faces)
            g.set_coeffs(_pinned(k), u)
            g.set_dt(0.9 * g.stability_dt())
            grids.append(g)
            fields.append(_pinned(T0))
            outs.append(flat[at:at + T0.numel()])
            at += T0.numel()
            steps.append(n)
        return dict(kind=kind, grids=grids, fields=fields, outs=outs, flat=flat, steps=steps)
    if kind == "serve":
        reqs = []
        for shape, n, storage, T0, k, u, faces, dt in _mix_inputs(case, seed):
            hk = k if isinstance(k, float) else _pinned(k)
            reqs.append((shape, n, storage, _pinned(T0), hk, u, faces, dt,
                         torch.empty(T0.shape, dtype=torch.float32, pin_memory=True)))
        return dict(kind=kind, served=_Served(reqs))
    if kind == "implicit":
        shape, T0, k, u, faces = _single(dict(case, advect=False), seed)
        hk = k if case["k"] == "uniform" else _pinned(k)
        g = wfa.Grid(shape)
        g.set_bcs(faces)
        g.set_coeffs(hk, u)
        g.set_cg_method(case["method"])
        return dict(kind=kind, g=g, T0=_pinned(T0), case=case,
                    out=torch.empty(T0.shape, dtype=torch.float32, pin_memory=True))
    shape = (case["nz"], case["ny"], case["nx"])
    gen = _gen(seed)
    names = ["T"] if case["update"] == "heat" else ["a", "b"]
    start = {f: torch.rand(shape, generator=gen, device="cuda") for f in names}
    return dict(kind=kind, kernel=S.compile(_program(case["update"])), start=start, case=case)


def run(state):
    kind = state["kind"]
    if kind == "march":
        g = state["g"]
        g.set_field(state["T0"])
        g.step(state["case"]["steps"])
        return g.read_field(state["out"])
    if kind == "solve":
        g, case = state["g"], state["case"]
        g.set_coeffs(state["k"], state["u"])
        g.set_field(state["T0"])
        g.set_dt(_dt_for(g, case["advect"], case["k"] == "uniform"))
        g.step(case["steps"])
        return {"T": g.read_field(state["out"]), "heat": g.total_heat()}
    if kind == "batch":
        for g, T0 in zip(state["grids"], state["fields"]):
            g.set_field(T0)
        wfa.batch_run(state["grids"], state["steps"])
        for g, out in zip(state["grids"], state["outs"]):
            g.read_field(out)
        return state["flat"]
    if kind == "serve":
        srv = state["served"].server
        tickets = [srv.submit(shape, T0, n, out=out, storage=storage, k=k, u=u, bc=faces, dt=dt)
                   for shape, n, storage, T0, k, u, faces, dt, out in state["served"].reqs]
        return [srv.wait(t) for t in tickets]
    if kind == "implicit":
        g, case = state["g"], state["case"]
        g.set_field(state["T0"])
        iters, _ = g.implicit_step(case["dt"], case["steps"], rtol=1e-6, max_iter=1000)
        return {"T": g.read_field(state["out"]), "iterations": iters}
    fields = {f: t.clone() for f, t in state["start"].items()}
    params = {"w": HEAT_W} if state["case"]["update"] == "heat" else dict(zip(("da", "db", "q"), REACT))
    state["kernel"].run(fields, steps=state["case"]["steps"], **params)
    return fields


# -------------------------------------------------------------------- work --
ON_CHIP = 96 << 20   # a working set that the L2 holds: its field moves once a call, not once a step


def _march_work(cells, steps, es, kvar):
    """Host field in and out, conductivity in, and per step the field read and
    written and the conductivity read (the paper's A_eff, Sec. 3.1.3), unless
    the grid stays on chip. 8 flops a cell update (Sec. 3.1)."""
    per = 2 * es + (4 if kvar else 0)
    moved = per * cells * (1 if per * cells <= ON_CHIP else steps)
    return 8 * cells + moved, 8 * cells * steps


def work(case):
    kind = case["kind"]
    if kind in ("march", "solve"):
        cells = case["nx"] * case["ny"] * case["nz"]
        kvar = case["k"] == "lognormal"
        b, f = _march_work(cells, case["steps"], 2 if case["storage"] == "bf16" else 4, kvar)
        if kind == "solve":
            b += 4 * cells * (1 + kvar)   # the conductivity from the host, the field once more for its heat
        return {"bytes": b, "flops": f}
    if kind in ("batch", "serve"):
        b = f = 0
        for shape, steps, heat, storage in _mix(case):
            bi, fi = _march_work(shape[0] * shape[1] * shape[2], steps, 2 if storage == BF16 else 4, heat)
            b, f = b + bi, f + fi
        return {"bytes": b, "flops": f}
    cells = case["nx"] * case["ny"] * case["nz"]
    if kind == "implicit":
        # iterations a step: about 0.4 of the Chebyshev bound of CG (the
        # solve starts from the old field); x, r and p read and written in
        # each, 15 flops (Sec. 3.2)
        kvar = case["k"] == "lognormal"
        root = math.sqrt(1.0 + 12.0 * case["dt"] * (2.5 if kvar else 1.0))
        its = max(1, round(0.4 * math.log(2e6) / math.log((root + 1.0) / (root - 1.0)))) * case["steps"]
        b = (24 + (4 if kvar else 0)) * cells
        return {"bytes": 8 * cells + (b if b <= ON_CHIP else b * its), "flops": 15 * cells * its}
    nf = 1 if case["update"] == "heat" else 2
    moved = 8 * nf * cells
    return {"bytes": moved if moved <= ON_CHIP else moved * case["steps"], "flops": (8 if nf == 1 else 22) * cells * case["steps"]}


# ------------------------------------------------------------------- exact --
class _Plain:
    """The update in 64 bits as plain tensor arithmetic on flat arrays with a
    one-cell halo: T' = c0 T + s + sum_f w_f T_f, weights zero outside."""

    def __init__(self, shape, k, u, faces, dt):
        nx, ny, nz = shape
        self.n = (nz, ny, nx)
        kd = (k.double() if torch.is_tensor(k) else torch.full((nz, ny, nx), float(k), dtype=torch.float64, device="cuda"))
        self.faces = faces
        w = [torch.zeros_like(kd) for _ in range(6)]
        src, diag = torch.zeros_like(kd), torch.zeros_like(kd)
        self.rate = torch.zeros_like(kd)   # D_C without dt (stability limit)
        self.held = torch.zeros_like(kd, dtype=torch.bool)
        self.held_val = torch.zeros_like(kd)
        self.per = [faces[2 * a][0] == P for a in range(3)]

        def ends(a):
            ax = 2 - a
            lo = [slice(None)] * 3
            hi = [slice(None)] * 3
            lo[ax], hi[ax] = slice(0, 1), slice(-1, None)
            return ax, tuple(lo), tuple(hi)

        for a in range(3):
            ax, lo, hi = ends(a)
            ap, am = max(u[a], 0.0), max(-u[a], 0.0)
            m = kd.shape[ax]
            left, right = kd.narrow(ax, 0, m - 1), kd.narrow(ax, 1, m - 1)
            K = 2 * left * right / (left + right)
            w[2 * a].narrow(ax, 1, m - 1).copy_(K + ap)
            w[2 * a + 1].narrow(ax, 0, m - 1).copy_(K + am)
            self.rate.narrow(ax, 1, m - 1).add_(K + am)
            self.rate.narrow(ax, 0, m - 1).add_(K + ap)
            for side, sl, win, wout in ((0, lo, ap, am), (1, hi, am, ap)):
                f = 2 * a + side
                kind, val = faces[f]
                if kind == P:
                    other = hi if side == 0 else lo
                    Kp = 2 * kd[sl] * kd[other] / (kd[sl] + kd[other])
                    w[f][sl] = Kp + win
                    self.rate[sl] += Kp + wout
                elif kind == D:
                    wd = 2 * kd[sl] + win
                    src[sl] += wd * val
                    diag[sl] += wd
                    self.rate[sl] += 2 * kd[sl] + wout
                elif kind == ZF:
                    diag[sl] += win - wout   # the stopped face's self term (wout - win) T_C
                elif kind == DC:
                    self.held[sl] = True
                    self.held_val[sl] = val
        if dt is None:
            free = ~self.held
            dt = 0.9 / self.rate[free].max().item()
        self.dt = dt
        for f in range(6):
            w[f].mul_(dt)
            w[f][self.held] = 0.0
        src.mul_(dt)
        diag.mul_(dt)
        src[self.held] = 0.0
        diag[self.held] = 0.0
        self.any_held = bool(self.held.any())
        c0 = 1.0 - diag
        for f in range(6):
            c0 -= w[f]
        # flat layout with a halo of one cell
        self.py, self.px = ny + 2, nx + 2
        self.sz = self.py * self.px
        self.c0, self.src = self._pad(c0), self._pad(src)
        self.w = [self._pad(x) for x in w]
        self.shift = [-1, 1, -self.px, self.px, -self.sz, self.sz]
        del kd, K, left, right, w, src, diag, c0

    def _pad(self, t):
        nz, ny, nx = self.n
        p = torch.zeros((nz + 2, ny + 2, nx + 2), dtype=torch.float64, device="cuda")
        p[1:-1, 1:-1, 1:-1] = t
        return p.view(-1)

    def _wrap(self, flat):
        if not any(self.per):
            return
        v = flat.view(self.n[0] + 2, self.n[1] + 2, self.n[2] + 2)
        for a in range(3):
            if self.per[a]:
                ax = 2 - a
                m = v.shape[ax]
                v.narrow(ax, 0, 1).copy_(v.narrow(ax, m - 2, 1))
                v.narrow(ax, m - 1, 1).copy_(v.narrow(ax, 1, 1))

    def apply(self, flat, out, linear=False):
        """out = c0 T + s + sum_f w_f T_f on the interior planes."""
        self._wrap(flat)
        a, b = self.sz, flat.numel() - self.sz
        o = out[a:b]
        if linear:
            torch.mul(self.c0[a:b], flat[a:b], out=o)
        else:
            torch.addcmul(self.src[a:b], self.c0[a:b], flat[a:b], out=o)
        for f in range(6):
            o.addcmul_(self.w[f][a:b], flat[a + self.shift[f]:b + self.shift[f]])

    def start(self, T0):
        t = T0.double()
        if self.any_held:
            t = torch.where(self.held, self.held_val, t)
        return self._pad(t)

    def dense(self, flat):
        nz, ny, nx = self.n
        return flat.view(nz + 2, ny + 2, nx + 2)[1:-1, 1:-1, 1:-1].contiguous()

    def march(self, T0, steps, storage=F32):
        """`steps` steps; with bf16 storage the field is rounded to bf16 at the
        start and after every step (that is what such a grid holds)."""
        cur = self.start(T0.bfloat16() if storage == BF16 else T0)
        nxt = torch.zeros_like(cur)
        half = torch.empty(cur.shape, dtype=torch.bfloat16, device=cur.device) if storage == BF16 else None
        for _ in range(steps):
            self.apply(cur, nxt)
            if half is not None:
                nxt.copy_(half.copy_(nxt))
            cur, nxt = nxt, cur
        return self.dense(cur)

    def implicit(self, T0, steps, tol=1e-13):
        """T' - (explicit increment at T') = T on the free cells by CG."""
        x = self.start(T0)
        free = self._pad((~self.held).double())
        tmp, q = torch.zeros_like(x), torch.zeros_like(x)
        for _ in range(steps):
            # r = dt acc(x) with the boundary terms
            self.apply(x, tmp)
            r = (tmp - x) * free
            bb = torch.dot(x * free, x * free)
            p = r.clone()
            rr = torch.dot(r, r)
            for _ in range(2000):
                if rr.item() <= tol * tol * bb.item():
                    break
                self.apply(p, tmp, linear=True)
                torch.sub(p, tmp, out=q)   # p - (linear part of the increment)
                q.add_(p)
                q.mul_(free)
                v = p * free
                alpha = rr / torch.dot(v, q)
                x.addcmul_(v, alpha.expand_as(v))
                r.addcmul_(q, (-alpha).expand_as(q))
                new = torch.dot(r, r)
                p = r + (new / rr) * v
                rr = new
        return self.dense(x)


def exact(case, seed):
    """What `run` returns, in 64 bits with plain tensor operations (on the
    host, laid out as `run`'s outputs)."""
    kind = case["kind"]
    if kind in ("march", "solve"):
        shape, T0, k, u, faces = _single(case, seed)
        dt = 1.0 if case["advect"] and case["k"] == "uniform" else None
        T = _Plain(shape, k, u, faces, dt).march(T0, case["steps"], BF16 if case["storage"] == "bf16" else F32)
        return T.cpu() if kind == "march" else {"T": T.cpu(), "heat": T.sum().item()}
    if kind in ("batch", "serve"):
        out = []
        for shape, steps, storage, T0, k, u, faces, dt in _mix_inputs(case, seed):
            out.append(_Plain(shape, k, u, faces, dt or None).march(T0, steps, storage).cpu())
        return torch.cat([t.reshape(-1) for t in out]) if kind == "batch" else out
    if kind == "implicit":
        shape, T0, k, u, faces = _single(dict(case, advect=False), seed)
        T = _Plain(shape, k, u, faces, case["dt"]).implicit(T0, case["steps"])
        return {"T": T.cpu(), "iterations": None}
    shape = (case["nz"], case["ny"], case["nx"])
    gen = _gen(seed)
    names = ["T"] if case["update"] == "heat" else ["a", "b"]
    cur = {f: torch.rand(shape, generator=gen, device="cuda").double() for f in names}
    mid = (slice(1, -1),) * 3

    def lap(t):
        c = t[mid]
        return (t[1:-1, 1:-1, :-2] + t[1:-1, 1:-1, 2:] + t[1:-1, :-2, 1:-1] + t[1:-1, 2:, 1:-1] + t[:-2, 1:-1, 1:-1]
                + t[2:, 1:-1, 1:-1] - 6 * c)

    # parameters as the front end takes them (fp32)
    w = float(np.float32(HEAT_W))
    da, db, q = (float(np.float32(v)) for v in REACT)
    for _ in range(case["steps"]):
        if names == ["T"]:
            t = cur["T"]
            inc = w * lap(t)
            t[mid] += inc
        else:
            a, b = cur["a"], cur["b"]
            ex = q * (a[mid] - b[mid])
            ia, ib = da * lap(a) - ex, db * lap(b) + ex
            a[mid] += ia
            b[mid] += ib
    return cur
