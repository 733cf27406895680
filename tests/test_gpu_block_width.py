"""Float tensor-product contexts without a set schedule step in 128- or 64-cell tiles, whichever takes
fewer rounds of resident blocks (float_block_width in csrc/api.cu): the step gives the same bits as
under either width set by hand. Batches on both sides of the rule, with lines of one cell, of one cell
more or less than a tile, and shorter than the reach of the velocity set."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2401_11086_gb300 as P  # noqa: E402
from paper_2401_11086_gb300 import shocks  # noqa: E402


@pytest.mark.parametrize("name,Ma,theta1", [("D3Q729", 3.0, 0.333), ("D3Q4913", 7.0, 0.071)])
@pytest.mark.parametrize("lengths", [[1, 7, 63, 64, 65, 127, 128, 129], [128] * 40, [65] * 60, [400] * 50])
def test_default_width_gives_the_same_bits(name, Ma, theta1, lengths):
    d = P.lb_lattice_named(name)
    n = len(lengths)
    ctx, f, _ = shocks.setup_batch(d, 5, [Ma] * n, lengths, precision="f32", width=0.0, theta1=[theta1] * n)
    g = torch.Generator(device="cuda").manual_seed(7)
    f *= 1.0 + 1e-3 * torch.randn(f.shape, dtype=f.dtype, device="cuda", generator=g)
    P.lb_step(ctx, f, ctx.new_state(), 1)
    first = P.lb_get_schedule(ctx)["tile_width"]
    got = None if first == 1 else ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)).clone()
    runs = []
    for width in (128, 64, 32):
        P.lb_set_schedule(ctx, width, 0, 0)
        runs.append(ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)).clone())
    assert P.lb_poll_status(ctx)[0] == 0
    for r in runs[1:] + ([got] if got is not None else []):
        assert torch.equal(r, runs[0])
