"""The work that users of this library have it do, as measurable cases.

A case is one call sequence of the public API (paper_2401_11086_gb300) on inputs of a stated size:

* kind "box": one collide-and-stream step of a periodic 3D box (Taylor-Green fields plus seeded
  density noise);
* kind "lines": steps of a batch of 1D normal shocks with fixed end states (one shock is a batch
  of one), by lb_step or by a graph replay of the persistent launch, with the profile read out by
  lb_moments where "moments" is set;
* kind "adjoint": one step of the discrete adjoint on a batch of shocks;
* kind "fit": a forward run and its gradient with respect to the relaxation times through
  autograd.relaxation_run (checkpointed).

Cases of one step read one state buffer and write the other, so that every pass does the same
work on the same input; cases of several steps advance their state (an even number of steps, which
leaves the newest state in the first buffer) as a simulation does, on shocks that stay stable.

exact() restates the scheme in plain torch, double precision: dense moment sums, per-cell frame
changes by the Hermite recurrences, irreducible parts by harmonic decomposition of the moment
tensors as polynomials.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2401_11086_gb300 as P
from paper_2401_11086_gb300 import shocks
from paper_2401_11086_gb300.autograd import SHOCK_LOSS_MASK, relaxation_run

Q_OF = {"D3Q39": 39, "D3Q103": 103, "D3Q729": 729, "D3Q4913": 4913}
MASK = P.LB_MOM_RHO | P.LB_MOM_U | P.LB_MOM_THETA | P.LB_MOM_Q


# ------------------------------------------------------------------------------ the cases
def _lines(name, lattice, N, precision, count, lo, hi, ma_lo, ma_hi, **more):
    """count shocks of lo..hi cells, Mach numbers in [ma_lo, ma_hi]."""
    c = dict(**({"name": name} if name else {}), kind="lines", lattice=lattice, N=N, precision=precision, count=count, lo=lo, hi=hi,
             ma_lo=ma_lo, ma_hi=ma_hi, steps=1, launch="step", moments=False, model="smrt", paper_frame=False)
    c.update(more)
    return c


def listed():
    return [
        # the throughput box of the benchmark's default workload, larger than any cache
        dict(name="box_256_d3q39_f32", kind="box", lattice="D3Q39", N=3, precision="f32", nx=256, ny=256, nz=256),
        # a box for a double-precision reference run, no extent a multiple of a block
        dict(name="box_ragged_d3q39_f64", kind="box", lattice="D3Q39", N=3, precision="f64", nx=90, ny=61, nz=75),
        # the smallest configuration: one weak shock in double, advanced and read out
        _lines("shock_400_d3q39_f64", "D3Q39", 3, "f64", 1, 400, 400, 1.2, 1.3, steps=40, moments=True),
        # one Ma = 3 shock on the degree-9 set in split precision, a piece of its 20000 steps
        _lines("shock_2048_d3q103_f32c64", "D3Q103", 4, "f32c64", 1, 2048, 2048, 2.8, 3.0, steps=20),
        # the batched configuration: 64 shocks of very different lengths, one persistent launch
        # of several steps replayed from a CUDA graph
        _lines("batch64_d3q103_f32c64_graph", "D3Q103", 4, "f32c64", 64, 512, 8192, 1.2, 3.0, steps=4,
               launch="graph"),
        # the paper's velocity set over its Table 3 rows, many shocks at once, both precisions
        _lines("table3_512_d3q729_f32", "D3Q729", 5, "f32", 512, 100, 400, 1.5, 5.0, paper_frame=True),
        _lines("table3_512_d3q729_f64", "D3Q729", 5, "f64", 512, 100, 400, 1.5, 5.0, paper_frame=True),
        # the paper's own run: a single shock on 100 cells, advanced and read out
        _lines("paper_100_d3q729_f64", "D3Q729", 5, "f64", 1, 100, 100, 3.0, 3.0, steps=20, moments=True,
               paper_frame=True),
        # long shocks of the mixed-Mach batch on the paper's set, graph replay of a persistent launch
        _lines("mixed_24_d3q729_f32_graph", "D3Q729", 5, "f32", 24, 512, 8192, 1.2, 4.0, steps=4, launch="graph"),
        # Table 3's Ma = 7 row on the largest velocity set
        _lines("ma7_64_d3q4913_f64", "D3Q4913", 5, "f64", 64, 100, 400, 7.0, 7.0, paper_frame=True),
        # the reverse mode: one adjoint step on the batched shocks ...
        _lines("adjoint_batch64_d3q103", "D3Q103", 4, "f32c64", 64, 512, 8192, 1.2, 3.0) | {"kind": "adjoint"},
        # ... and a gradient of a shock-profile loss, forward and backward, checkpointed
        _lines("fit_1024_d3q103", "D3Q103", 4, "f32c64", 1, 1024, 1024, 2.8, 3.0, steps=100, every=25)
        | {"kind": "fit"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["box", "lines", "lines", "tensor", "tensor", "adjoint", "fit"])
    if kind == "box":
        precision = rng.choice(["f32", "f32", "f64", "f32c64"])
        cells = _log(rng, 4000, {"f32": 14_000_000, "f64": 1_000_000, "f32c64": 2_000_000}[precision])
        side = cells ** (1.0 / 3.0)
        nx, ny = (max(7, int(side * rng.uniform(0.6, 1.6))) for _ in range(2))
        return dict(kind="box", lattice="D3Q39", N=3, precision=precision, nx=nx, ny=ny,
                    nz=max(7, min(int(cells / (nx * ny)), 400)))
    if kind == "lines":
        lattice = rng.choice(["D3Q39", "D3Q103", "D3Q103"])
        precision = rng.choice(["f32c64", "f32c64", "f64", "f32"])
        count, hi = _log(rng, 1, 64), _log(rng, 200, 8192)
        lo = max(100, hi // rng.choice([1, 3, 16]))
        ma = (1.2, 1.4) if lattice == "D3Q39" else (1.2, 3.0)
        steps = 1 if count * hi > 40_000 else rng.choice([4, 10, 20])
        return _lines("", lattice, 3 if lattice == "D3Q39" else 4, precision, count, lo, hi, *ma, steps=steps,
                      launch=rng.choice(["step", "graph"]) if steps > 1 else "step",
                      model=rng.choice(["smrt", "smrt", "es_bgk"]))
    if kind == "tensor":
        lattice = rng.choice(["D3Q729", "D3Q729", "D3Q4913"])
        big = lattice == "D3Q4913"
        precision = rng.choice(["f32", "f64"])
        count, hi = _log(rng, 1, 64 if big else 512), rng.randint(60, 400)
        return _lines("", lattice, rng.choice([4, 5, 5]), precision, count, rng.randint(40, hi), hi,
                      *((7.0, 7.0) if big else (1.5, 3.0)), paper_frame=True,
                      model=rng.choice(["smrt", "smrt", "es_bgk"]))
    if kind == "adjoint":
        lattice = rng.choice(["D3Q39", "D3Q103", "D3Q103", "D3Q729"])
        count, hi = _log(rng, 1, 64), (rng.randint(60, 400) if lattice == "D3Q729" else _log(rng, 200, 6000))
        return _lines("", lattice, {"D3Q39": 3, "D3Q103": 4, "D3Q729": 5}[lattice],
                      "f64" if lattice == "D3Q729" else rng.choice(["f64", "f32c64"]), count, max(40, hi // 4), hi,
                      *((1.2, 1.4) if lattice == "D3Q39" else (1.5, 3.0))) | {"kind": "adjoint"}
    lattice = rng.choice(["D3Q39", "D3Q103"])
    n = _log(rng, 100, 2000)
    return _lines("", lattice, 3 if lattice == "D3Q39" else 4, rng.choice(["f64", "f32c64"]), 1, n, n,
                  *((1.2, 1.4) if lattice == "D3Q39" else (2.0, 3.0)), steps=rng.choice([20, 40, 60]),
                  every=rng.choice([10, 20])) | {"kind": "fit"}


def _lengths(case):
    """The lengths belong to the case (its size), not to the seed of its inputs."""
    rng = np.random.default_rng(case["count"] * 1009 + case["lo"] * 31 + case["hi"])
    if case["hi"] >= 4 * case["lo"] and case["hi"] > 1000:  # spread over powers of two
        return rng.choice([n for k in range(16) if (n := case["lo"] << k) <= case["hi"]], size=case["count"])
    return rng.integers(case["lo"], case["hi"] + 1, size=case["count"])


def _cells(case):
    return case["nx"] * case["ny"] * case["nz"] if case["kind"] == "box" else int(_lengths(case).sum())


def work(case):
    q, N, cells = Q_OF[case["lattice"]], case["N"], _cells(case)
    elem = 8 if case["precision"] == "f64" else 4
    steps = case.get("steps", 1)
    # per cell and step: each population enters N + 1 sums of powers and leaves by a polynomial
    # of degree N (the first and last factored pass), and the collision acts on the moments
    flops = 4.0 * q * (N + 1) + 30.0 * math.comb(N + 3, 3)
    bytes_ = 2.0 * q * elem * cells  # the state in, the state out
    if case["kind"] == "adjoint":
        return {"bytes": q * (elem + 16.0) * cells, "flops": 2.0 * flops * cells}
    if case["kind"] == "fit":  # the initial state in, profiles and gradients out
        return {"bytes": (q * elem + 5 * 8.0) * cells, "flops": 3.0 * flops * cells * steps}
    return {"bytes": bytes_ + (8 * 8.0 * cells if case.get("moments") else 0.0), "flops": flops * cells * steps}


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def prepare(case, seed):
    d = P.lb_lattice_named(case["lattice"])
    rng = np.random.default_rng(seed)
    if case["kind"] == "box":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        ctx = P.lb_init_lattice(P.LatticeDesc(d.e, d.w, d.c, d.degree), nx, ny, nz, N=case["N"],
                                precision=case["precision"])
        taus = [r * 2.0 * d.c for r in shocks.TAU_RATIOS_SMRT[: shocks.ntau(case["N"])]]
        P.lb_set_relaxation(ctx, taus, True, 1.0)
        ax = [torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n) for n in (nz, ny, nx)]
        Z, Y, X = torch.meshgrid(*ax, indexing="ij")
        rho = 1.0 + 1e-3 * torch.randn(nz * ny * nx, dtype=torch.float64, device="cuda", generator=_gen(seed))
        u = torch.stack([0.05 * X.sin() * Y.cos() * Z.cos(), -0.05 * X.cos() * Y.sin() * Z.cos(),
                         torch.zeros_like(X)]).reshape(3, -1).contiguous()
        del X, Y, Z
        fa = ctx.new_state()
        P.lb_fill_equilibrium(ctx, fa, rho, u, torch.ones_like(rho))
        return {"case": case, "d": d, "ctx": ctx, "fa": fa, "fb": ctx.new_state(),
                "params": [{"taus": taus}]}
    lengths = _lengths(case)
    theta1 = None
    if case["paper_frame"] and case["lattice"] == "D3Q4913":
        machs, theta1 = [7.0] * len(lengths), [shocks.TABLE3_THETA1_D1Q17[7.0]] * len(lengths)
    elif case["paper_frame"]:
        rows = [m for m in (3.0, 1.5, 5.0) if case["ma_lo"] <= m <= case["ma_hi"]]
        machs = [rows[j % len(rows)] for j in range(len(lengths))]
        theta1 = [shocks.TABLE3_THETA1[m] for m in machs]
    else:
        machs = rng.uniform(case["ma_lo"], case["ma_hi"], size=len(lengths))
    ctx, fa, params = shocks.setup_batch(d, case["N"], machs, lengths, precision=case["precision"],
                                         width=float(rng.uniform(4.0, 10.0)), theta1=theta1)
    if case["model"] == "es_bgk" and case["kind"] == "lines":
        P.lb_set_collision_model(ctx, -1, P.LB_MODEL_ES_BGK, -0.5)
    # a state out of equilibrium, as the collision meets it
    fa *= 1.0 + 1e-3 * torch.randn(fa.shape, dtype=fa.dtype, device="cuda", generator=_gen(seed))
    s = {"case": case, "d": d, "ctx": ctx, "fa": fa, "params": params, "lengths": lengths}
    if case["kind"] == "lines":
        s["fb"] = ctx.new_state()
        if case["launch"] == "graph":
            P.lb_set_schedule(ctx, 128, 0, 1)
    elif case["kind"] == "adjoint":
        s["lam"] = 1e-3 * torch.randn(ctx.state_elems, dtype=torch.float64, device="cuda", generator=_gen(seed + 1))
        s["lam_out"] = torch.zeros_like(s["lam"])
    else:
        p = params[0]
        P.lb_set_relaxation(ctx, p["taus"], True, 1.0, p["left"], p["right"])
        s["tau"] = torch.tensor(np.asarray(p["taus"]) * (1.0 + rng.uniform(-0.2, 0.2, len(p["taus"]))),
                                requires_grad=True)
        fields = shocks.tanh_fields(p, int(lengths[0]), 6.0)  # the profile to be matched
        s["target"] = torch.zeros(5, ctx.cells, dtype=torch.float64, device="cuda")
        s["target"][0] = torch.from_numpy(fields[0])
        s["target"][1] = torch.from_numpy(fields[2])
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["kind"] == "adjoint":
        dtau = torch.zeros(len(s["params"][0]["taus"]), dtype=torch.float64, device="cuda")
        P.lb_step_adjoint(ctx, s["fa"], s["lam"], s["lam_out"], dtau)
        return {"lam": s["lam_out"].view(ctx.lattice.q, ctx.plane_stride)[:, : ctx.cells], "dtau": dtau}
    if case["kind"] == "fit":
        s["tau"].grad = None
        m = relaxation_run(ctx, s["tau"], s["fa"], case["steps"], checkpoint_every=case["every"], mask=SHOCK_LOSS_MASK)
        ((m - s["target"]) ** 2).sum().backward()
        return {"moments": m.detach(), "grad": s["tau"].grad}
    step = P.lb_step_graph if case.get("launch") == "graph" else P.lb_step
    out = step(ctx, s["fa"], s["fb"], case.get("steps", 1))
    got = {"f": ctx.planes(out)}
    if case.get("moments"):
        got["moments"] = P.lb_moments(ctx, out, MASK)
    return got


# ------------------------------------------------------------------------------ 64-bit values
def _multi(N):
    """Multi-indices of order <= N: by order, then descending lexicographically."""
    return [(a, b, n - a - b) for n in range(N + 1) for a in range(n, -1, -1) for b in range(n - a, -1, -1)]


def _fact(a):
    return math.factorial(a[0]) * math.factorial(a[1]) * math.factorial(a[2])


def _irreducible(n):
    """Projectors of the order-n symmetric tensors (components d_beta) onto their parts (n, m):
    the tensor as the polynomial sum_beta d_beta x^beta / beta! splits into |x|^(2m) times a
    harmonic polynomial of degree n - 2m."""
    mono = lambda k: [a for a in _multi(k) if sum(a) == k]  # noqa: E731
    cols, owner = [], []
    for m in range(n // 2 + 1):
        k = n - 2 * m
        src, low = mono(k), mono(k - 2) if k >= 2 else []
        lap = np.zeros((max(len(low), 1), len(src)))
        for j, a in enumerate(src):
            for ax in range(3):
                if a[ax] >= 2:
                    b = list(a)
                    b[ax] -= 2
                    lap[low.index(tuple(b)), j] += a[ax] * (a[ax] - 1)
        _, sv, vt = np.linalg.svd(lap)
        for h in vt[int((sv > 1e-9).sum()):]:
            poly = dict(zip(src, h))
            for _ in range(m):  # times |x|^2
                nxt = {}
                for a, v in poly.items():
                    for ax in range(3):
                        b = list(a)
                        b[ax] += 2
                        nxt[tuple(b)] = nxt.get(tuple(b), 0.0) + v
                poly = nxt
            cols.append([poly.get(a, 0.0) * _fact(a) for a in mono(n)])
            owner.append(m)
    B = np.array(cols).T
    inv = np.linalg.inv(B)
    return [B[:, np.array(owner) == m] @ inv[np.array(owner) == m] for m in range(n // 2 + 1)]


class _Scheme:
    """One velocity set and order in double precision on the GPU."""

    def __init__(self, d, N):
        dev = dict(dtype=torch.float64, device="cuda")
        self.N, self.idx = N, _multi(N)
        self.xi = torch.tensor(d.e.astype(np.float64) * d.c, **dev)
        self.w = torch.tensor(d.w, **dev)
        self.e, self.c, self.q = d.e.astype(np.int64), d.c, int(d.q)
        pw = torch.stack([self.xi ** j for j in range(N + 1)])  # [j][i][axis]
        he = [torch.ones_like(self.xi), self.xi]
        for j in range(1, N):
            he.append(self.xi * he[j] - j * he[j - 1])
        self.mono = torch.stack([pw[a, :, 0] * pw[b, :, 1] * pw[c, :, 2] for a, b, c in self.idx])
        self.herm = torch.stack([he[a][:, 0] * he[b][:, 1] * he[c][:, 2] / _fact((a, b, c)) for a, b, c in self.idx])
        self.proj = {n: [torch.tensor(p, **dev) for p in _irreducible(n)] for n in range(2, N + 1)}
        self.pos = torch.tensor([(a * (N + 1) + b) * (N + 1) + c for a, b, c in self.idx], device="cuda")
        self.slot = {a: k for k, a in enumerate(self.idx)}
        self.of = {n: [k for k, a in enumerate(self.idx) if sum(a) == n] for n in range(N + 1)}
        self.unit = self.mono @ self.w  # raw moments of the weights

    def _axes(self, C, v):
        """sum over (a', b', c') of prod_k C[k][a_k][a'_k] v_(a', b', c'): [M][cells] -> [M][cells]."""
        n = self.N + 1
        g = torch.zeros(n ** 3, v.shape[1], dtype=v.dtype, device=v.device).index_copy(0, self.pos, v).view(n, n, n, -1)
        g = torch.einsum("axz,xbcz->abcz", C[0], g)
        g = torch.einsum("bxz,axcz->abcz", C[1], g)
        g = torch.einsum("cxz,abxz->abcz", C[2], g)
        return g.reshape(n ** 3, -1)[self.pos]

    def _rows(self, rows):
        n = self.N + 1
        z = torch.zeros_like(rows[0][0])
        return torch.stack([torch.stack([r[j] if j < len(r) else z for j in range(n)]) for r in rows])

    def macro(self, df):
        """rho, u (relative to the frame), theta, full raw moments of populations w + df."""
        R = self.mono @ df
        s = self.slot
        rho = 1.0 + R[0]
        u = [R[s[a]] / rho for a in ((1, 0, 0), (0, 1, 0), (0, 0, 1))]
        e3 = R[s[2, 0, 0]] + R[s[0, 2, 0]] + R[s[0, 0, 2]]
        theta = 1.0 + (e3 - 3.0 * R[0] - rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)) / (3.0 * rho)
        return rho, u, theta, R + self.unit[:, None]

    def local(self, u, theta, R):
        """d_beta = sum f He_beta((xi - u) / sqrt(theta)) from the raw moments R."""
        s = theta.sqrt()
        C = []
        for k in range(3):  # rows: He_j((x - u) / s) as polynomials in x
            one = torch.ones_like(s)
            rows = [[one], [-u[k] / s, one / s]]
            for j in range(1, self.N):
                a, b = rows[j], rows[j - 1]
                z = torch.zeros_like(s)
                up, lo, lowest = [z] + [v / s for v in a], [v * (-u[k] / s) for v in a] + [z], b + [z, z]
                rows.append([x + y - j * w for x, y, w in zip(up, lo, lowest)])
            C.append(self._rows(rows))
        return self._axes(C, R)

    def absolute(self, u, theta, d):
        """a_alpha = sum f He_alpha(xi) from the local coefficients d."""
        s = theta.sqrt()
        D = []
        for k in range(3):  # rows: He_j(u + s y) in He_i(y)
            one, z = torch.ones_like(s), torch.zeros_like(s)
            rows = [[one], [u[k], s]]
            for j in range(1, self.N):
                a, b = rows[j], rows[j - 1]
                nxt = [z] * (j + 2)
                for i, v in enumerate(a):
                    nxt[i] = nxt[i] + u[k] * v
                    nxt[i + 1] = nxt[i + 1] + s * v
                    if i:
                        nxt[i - 1] = nxt[i - 1] + i * s * v
                for i, v in enumerate(b):
                    nxt[i] = nxt[i] - j * v
                rows.append(nxt)
            D.append(self._rows(rows))
        return self._axes(D, d)

    def equilibrium(self, rho, u, theta):
        """Deviations of the order-N equilibrium: [q][cells]."""
        d = torch.zeros(len(self.idx), rho.numel(), dtype=rho.dtype, device=rho.device)
        d[0] = rho
        a = self.absolute(u, theta, d)
        a = torch.cat([a[:1] - 1.0, a[1:]])
        return self.w[:, None] * (self.herm.T @ a)

    def collide(self, df, tau, maxwell, es_b):
        """tau: [parts][cells or 1] continuous times at rho = 1."""
        rho, u, theta, R = self.macro(df)
        d = self.local(u, theta, R)
        new, k = [None] * len(self.idx), 0
        zero = torch.zeros_like(rho)
        for n in range(self.N + 1):
            sl = self.of[n]
            if n < 2:
                for j in sl:
                    new[j] = rho if n == 0 else zero
                continue
            blk = d[sl]
            if es_b is None:
                out = 0.0
                for p in self.proj[n]:
                    t = (tau[k] / rho if maxwell else tau[k]) + 0.5
                    out = out + (1.0 - 1.0 / t) * (p @ blk)
                    k += 1
            else:
                t = (tau[0] / rho if maxwell else tau[0]) + 0.5
                bp = 1.0 - (1.0 - es_b) * t / (t - 0.5 * es_b)
                target = bp * blk if n == 2 else torch.zeros_like(blk)
                if n == 4:
                    dd = lambda i, j: d[self.slot[tuple(int(i == q) + int(j == q) for q in range(3))]]  # noqa: E731
                    rows = []
                    for j in sl:
                        i0, i1, i2, i3 = [ax for ax in range(3) for _ in range(self.idx[j][ax])]
                        rows.append(dd(i0, i1) * dd(i2, i3) + dd(i0, i2) * dd(i1, i3) + dd(i0, i3) * dd(i1, i2))
                    target = bp ** 2 / rho * torch.stack(rows)
                out = blk + (target - blk) / t
            for r, j in enumerate(sl):
                new[j] = out[r]
        a = self.absolute(u, theta, torch.stack(new))
        a = torch.cat([a[:1] - 1.0, a[1:]])
        return self.w[:, None] * (self.herm.T @ a)


def _chunks(fn, df, size, *cellwise):
    """fn over column blocks of df (and of the per-cell tensors)."""
    out = [fn(df[:, i : i + size], *[t[:, i : i + size] for t in cellwise]) for i in range(0, df.shape[1], size)]
    return torch.cat(out, 1)


class _Lines:
    """Pull streaming of a batch of lines with fixed end states."""

    def __init__(self, sch, s):
        self.sch = sch
        L = torch.tensor(np.asarray(s["lengths"], dtype=np.int64), device="cuda")
        self.inst = torch.repeat_interleave(torch.arange(len(L), device="cuda"), L)
        off = torch.cumsum(L, 0) - L
        x = torch.arange(int(L.sum()), device="cuda") - off[self.inst]
        kx = torch.tensor([p["kx"] for p in s["params"]], device="cuda")[self.inst]
        ends = []
        for side in ("left", "right"):
            vals = torch.tensor([[p[side]["rho"], p[side]["u"][0] - sch.c * p["kx"], p[side]["u"][1], p[side]["u"][2],
                                  p[side]["theta"]] for p in s["params"]], dtype=torch.float64, device="cuda").T
            ends.append(sch.equilibrium(vals[0], [vals[1], vals[2], vals[3]], vals[4]))
        self.groups = []
        for ex in sorted(set(sch.e[:, 0].tolist())):
            rows = torch.tensor(np.flatnonzero(sch.e[:, 0] == ex), device="cuda")
            src = x - ex - kx
            bad = torch.nonzero((src < 0) | (src >= L[self.inst])).ravel()
            left = (src[bad] < 0)[None]
            fix = torch.where(left, ends[0][rows][:, self.inst[bad]], ends[1][rows][:, self.inst[bad]])
            ok = torch.minimum(src.clamp(min=0), L[self.inst] - 1) + off[self.inst]
            self.groups.append((rows, ok, bad, fix))
        self.order = torch.argsort(torch.cat([g[0] for g in self.groups]))

    def pull(self, f):
        out = []
        for rows, ok, bad, fix in self.groups:
            out.append(f[rows][:, ok].index_copy(1, bad, fix))
        return torch.cat(out)[self.order]


def _moment_rows(sch, df, ubar, full):
    rho, u, theta, R = sch.macro(df)
    d = sch.local(u, theta, R)
    s = sch.slot
    h = 0.5 * theta * theta.sqrt()
    q = [h * (d[s[3, 0, 0]] + d[s[1, 2, 0]] + d[s[1, 0, 2]]), h * (d[s[2, 1, 0]] + d[s[0, 3, 0]] + d[s[0, 1, 2]]),
         h * (d[s[2, 0, 1]] + d[s[0, 2, 1]] + d[s[0, 0, 3]])]
    vel = [u[0] + ubar, u[1], u[2]] if full else []
    return torch.stack([rho, *vel, theta, *q])


def exact(case, seed):
    cells = _cells(case)
    if case["kind"] != "box" and cells * Q_OF[case["lattice"]] * case["steps"] > 400_000_000:
        return None
    s = prepare(case, seed)
    ctx, d, N = s["ctx"], s["d"], case["N"]
    sch = _Scheme(d, N)
    size = max(2048, (1 << 25) // (N + 1) ** 3)
    f = ctx.planes(s["fa"]).double()
    if case["kind"] == "box":
        nz, ny, nx = case["nz"], case["ny"], case["nx"]
        g = torch.stack([torch.roll(f[i].view(nz, ny, nx), (int(ez), int(ey), int(ex)), (0, 1, 2)).reshape(-1)
                         for i, (ex, ey, ez) in enumerate(sch.e)])
        tau = torch.tensor(s["params"][0]["taus"], dtype=torch.float64, device="cuda")[:, None]
        return {"f": _chunks(lambda v: sch.collide(v, tau, True, None), g, size)}
    ln = _Lines(sch, s)
    tau = torch.tensor([p["taus"] for p in s["params"]], dtype=torch.float64, device="cuda").T[:, ln.inst]
    ubar = torch.tensor([p["kx"] for p in s["params"]], dtype=torch.float64, device="cuda")[ln.inst] * d.c
    es_b = -0.5 if case["model"] == "es_bgk" and case["kind"] == "lines" else None
    if case["kind"] == "adjoint":
        lam = s["lam"].view(sch.q, ctx.plane_stride)[:, :cells]
        g, mu, dtau = ln.pull(f), [], 0.0
        for i in range(0, cells, size):
            v = g[:, i : i + size].clone().requires_grad_(True)
            t = tau[:, i : i + size].clone().requires_grad_(True)
            a, b = torch.autograd.grad((sch.collide(v, t, True, None) * lam[:, i : i + size]).sum(), (v, t))
            mu.append(a)
            dtau = dtau + b.sum(1)
        back = torch.zeros_like(f).requires_grad_(True)  # the streaming's transpose
        (out,) = torch.autograd.grad(ln.pull(back), back, torch.cat(mu, 1))
        return {"lam": out, "dtau": dtau}
    if case["kind"] == "fit":
        t = s["tau"].detach().cuda().requires_grad_(True)
        v = f
        for _ in range(case["steps"]):
            v = torch.utils.checkpoint.checkpoint(lambda a, b: sch.collide(ln.pull(a), b[:, None], True, None), v, t,
                                                  use_reentrant=False)
        m = _moment_rows(sch, ln.pull(v), ubar, False)
        (grad,) = torch.autograd.grad(((m - s["target"]) ** 2).sum(), t)
        return {"moments": m.detach(), "grad": grad.cpu()}
    for _ in range(case["steps"]):
        f = _chunks(lambda v, t: sch.collide(v, t, True, es_b), ln.pull(f), size, tau)
    got = {"f": f}
    if case["moments"]:
        got["moments"] = _moment_rows(sch, ln.pull(f), ubar, True)
    return got
