"""The group-of-lanes adjoint step of small periodic D3Q39 / D3Q103 lines (csrc/lane_kernels.cuh) against the
kernel that runs one thread per cell, which a larger grid of the same lines takes: a line of the least
length (reach of the set + frame shift, every pull wrapped somewhere) and ragged ones, both group sizes
(608 cells is the boundary on 152 SMs), double and float states.

Both sides are double with the same formulas and other summation orders: 1e-13 of the largest value, as for
fixed ends. The output starts as NaN, so that a slot left unwritten shows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2401_11086_gb300 as P  # noqa: E402
from paper_2401_11086_gb300 import shocks  # noqa: E402


def _noise(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


@pytest.mark.parametrize("name,N", [("D3Q39", 3), ("D3Q103", 3), ("D3Q103", 4)])
@pytest.mark.parametrize("more", [[], [133], [133, 9, 700]])
@pytest.mark.parametrize("shift", [1, -2])
@pytest.mark.parametrize("precision", ["f64", "f32", "f32c64"])
def test_periodic_adjoint_matches_one_thread_per_cell(name, N, more, shift, precision):
    d = P.lb_lattice_named(name)
    lengths = [int(np.abs(d.e[:, 0]).max()) + abs(shift)] + more
    n = sum(lengths)
    res = []
    for extra in ([], [8192]):
        ctx = P.lb_init_lattice(P.LatticeDesc(d.e, d.w, d.c, d.degree, (shift, 0, 0)), 0, N=N, precision=precision,
                                nx_per_instance=lengths + extra)
        taus = [0.9 + 0.1 * k for k in range(shocks.ntau(N))]
        P.lb_set_relaxation(ctx, taus, True, 1.0)
        one = torch.ones(ctx.cells, dtype=torch.float64, device="cuda")
        f = ctx.new_state()
        P.lb_fill_equilibrium(ctx, f, one, torch.stack([(0.3 + shift * d.c) * one, 0.1 * one, 0 * one]).contiguous(), one)
        ctx.planes(f)[:, :n] *= (1.0 + 0.02 * _noise((d.q, n), 4)).to(f.dtype)
        lam = torch.zeros(ctx.state_elems, dtype=torch.float64, device="cuda")
        ctx.planes(lam)[:, :n] = _noise((d.q, n), 3)  # zero on the long line
        out = torch.full_like(lam, float("nan"))
        dtau = torch.zeros(len(taus), dtype=torch.float64, device="cuda")
        P.lb_step_adjoint(ctx, f, lam, out, dtau)
        res.append((ctx.planes(out)[:, :n].clone(), dtau))
    for got, want in zip(*res):
        assert torch.isfinite(got).all() and ((got - want).abs().max() / want.abs().max()).item() < 1e-13
