"""The group-of-lanes step and adjoint of small double line contexts (csrc/lane_kernels.cuh) against the
kernels that run one thread per cell, at the sizes where their blocks can go wrong: lines shorter
than a block's cells, one cell more or less than a block or a tile, several instances, both group
sizes (608 cells is the boundary on 152 SMs), fixed and periodic ends, both collision models.

Both sides are double with the same formulas and other summation orders: 1e-13 of the largest value
(a few hundred roundings of 2^-53). A larger grid of the same cells takes the one-thread adjoint."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2401_11086_gb300 as P  # noqa: E402
from paper_2401_11086_gb300 import shocks  # noqa: E402

SETS = [("D3Q39", 3, 1.25), ("D3Q103", 3, 2.0), ("D3Q103", 4, 2.0)]
LENGTHS = [[1], [3, 8, 9], [127, 128, 129, 40], [600, 17], [700, 33, 5]]


def _noise(t, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(t.shape, dtype=torch.float64, device="cuda", generator=g)


@pytest.mark.parametrize("name,N,Ma", SETS)
@pytest.mark.parametrize("lengths", LENGTHS)
@pytest.mark.parametrize("es", [False, True])
def test_step_matches_one_thread_per_cell(name, N, Ma, lengths, es):
    d = P.lb_lattice_named(name)
    ctx, f, _ = shocks.setup_batch(d, N, [Ma] * len(lengths), lengths, precision="f64", width=4.0)
    if es:
        P.lb_set_collision_model(ctx, -1, P.LB_MODEL_ES_BGK, -0.5)
    f *= 1.0 + 0.02 * _noise(f, 1)
    got = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)).clone()
    P.lb_set_schedule(ctx, 128, 0, 0)                     # a set schedule: one thread per cell
    want = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1))
    assert P.lb_poll_status(ctx)[0] == 0
    assert ((got - want).abs().max() / want.abs().max()).item() < 1e-13


@pytest.mark.parametrize("name,N,Ma", SETS[1:])
def test_periodic_step_matches_one_thread_per_cell(name, N, Ma):
    d = P.lb_lattice_named(name)
    nx = 133
    ctx = P.lb_init_lattice(P.LatticeDesc(d.e, d.w, d.c, d.degree, (1, 0, 0)), nx, N=N, precision="f64")
    P.lb_set_relaxation(ctx, [0.9] * shocks.ntau(N), False, 1.0)
    one = torch.ones(nx, dtype=torch.float64, device="cuda")
    f = ctx.new_state()
    P.lb_fill_equilibrium(ctx, f, one, torch.stack([0.3 * one + d.c, 0.1 * one, 0 * one]).contiguous(), one)
    f *= 1.0 + 0.02 * _noise(f, 2)
    got = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)).clone()
    P.lb_set_schedule(ctx, 64, 0, 0)
    want = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1))
    assert ((got - want).abs().max() / want.abs().max()).item() < 1e-13


@pytest.mark.parametrize("name,N,Ma", SETS)
@pytest.mark.parametrize("lengths", LENGTHS)
@pytest.mark.parametrize("precision", ["f64", "f32c64"])
def test_adjoint_matches_one_thread_per_cell(name, N, Ma, lengths, precision):
    """The same instances alone, and followed by a long one that makes the grid large."""
    d = P.lb_lattice_named(name)
    res = []
    for extra in ([], [8192]):
        ls = list(lengths) + extra
        ctx, f, p = shocks.setup_batch(d, N, [Ma] * len(ls), ls, precision=precision, width=4.0)
        n = sum(lengths)
        lam, out = (torch.zeros(ctx.state_elems, dtype=torch.float64, device="cuda") for _ in range(2))
        ctx.planes(lam)[:, :n] = _noise(torch.empty(d.q, n), 3)
        ctx.planes(f)[:, :n] *= (1.0 + 0.02 * _noise(torch.empty(d.q, n), 4)).to(f.dtype)
        dtau = torch.zeros(len(p[0]["taus"]), dtype=torch.float64, device="cuda")
        P.lb_step_adjoint(ctx, f, lam, out, dtau)          # lam is zero on the long instance
        res.append((ctx.planes(out)[:, :n].clone(), dtau))
    for g, w in zip(*res):
        assert torch.isfinite(g).all() and ((g - w).abs().max() / w.abs().max()).item() < 1e-13
