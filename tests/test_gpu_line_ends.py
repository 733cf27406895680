"""1D lines at their ends and in numbers: many short lines on groups of lanes."""
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


@pytest.mark.parametrize("name,N,Ma", [("D3Q39", 3, 1.25), ("D3Q103", 4, 2.0)])
@pytest.mark.parametrize("lengths", [[1] * 40 + [8] * 9 + [9, 7, 129], [8] * 300, [1] * 700, [3000] + [1, 2] * 200])
def test_many_short_lines_on_groups_of_lanes(name, N, Ma, lengths):
    """Both group sizes, lines shorter and one cell longer than a block's cells: one thread per cell to
    1e-13 of the largest value (the same formulas in double, other summation orders)."""
    ctx, f, _ = shocks.setup_batch(P.lb_lattice_named(name), N, [Ma] * len(lengths), lengths, precision="f64", width=4.0)
    f *= 1.0 + 0.02 * _noise(f.shape, 1)
    assert P.lb_get_schedule(ctx)["tile_width"] == 1
    out = ctx.new_state()
    out.fill_(float("nan"))
    got = ctx.planes(P.lb_step(ctx, f, out, 1)).clone()
    P.lb_set_schedule(ctx, 32, 0, 0)
    want = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1))
    assert torch.isfinite(got).all() and P.lb_poll_status(ctx)[0] == 0
    assert ((got - want).abs().max() / want.abs().max()).item() < 1e-13
