"""1D lines at their ends and in numbers: many short lines on groups of lanes, wrapped pulls of periodic
split-precision lines, and frame shifts that a periodic axis cannot hold."""
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


@pytest.mark.parametrize("name,N", [("D3Q39", 3), ("D3Q103", 3), ("D3Q103", 4)])
@pytest.mark.parametrize("shift", [1, -2])
@pytest.mark.parametrize("persistent", [0, 1])
def test_periodic_split_lines_staged_and_direct(name, N, shift, persistent):
    """Split-precision periodic lines in the library's velocity order (pulls staged per warp, the wrapped ones
    loaded) against a permuted order (every pull loaded), from the least length on. Both form the same
    values; a last-bit difference before the stochastic rounding may turn it by one spacing of a float, at
    most 2^-23 of the largest value in each of three steps, while a wrong wrap errs by the 2 % noise."""
    d = P.lb_lattice_named(name)
    order = np.random.default_rng(0).permutation(d.q)
    least = int(np.abs(d.e[:, 0]).max()) + abs(shift)
    lengths = [least, 31, 33, 133, 512]
    noise = _noise((d.q, sum(lengths)), 5)
    res = []
    for o in (np.arange(d.q), order):
        ctx = P.lb_init_lattice(P.LatticeDesc(d.e[o], d.w[o], d.c, d.degree, (shift, 0, 0)), 0, N=N, precision="f32c64",
                                nx_per_instance=lengths)
        P.lb_set_relaxation(ctx, [1.1 + 0.1 * k for k in range(shocks.ntau(N))], True, 1.0)
        P.lb_set_schedule(ctx, 64, 0, persistent)
        one = torch.ones(ctx.cells, dtype=torch.float64, device="cuda")
        f = ctx.new_state()
        P.lb_fill_equilibrium(ctx, f, one, torch.stack([(0.2 + shift * d.c) * one, 0.1 * one, 0 * one]).contiguous(), one)
        ctx.planes(f)[:] *= (1.0 + 0.02 * noise[torch.from_numpy(o).cuda()]).to(f.dtype)
        out = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 3))
        assert P.lb_poll_status(ctx)[0] == 0
        got = torch.empty_like(out)
        got[torch.from_numpy(o).cuda()] = out
        res.append(got.double())
    assert ((res[0] - res[1]).abs().max() / res[1].abs().max()).item() < 3 * 2.0 ** -23


@pytest.mark.parametrize("name,N,precision", [("D3Q39", 3, "f64"), ("D3Q103", 4, "f32c64"), ("D3Q729", 4, "f32")])
def test_frame_shift_beyond_a_periodic_line_is_refused(name, N, precision):
    """Pulls wrap once: reach + |k_x| above the length of a periodic instance is refused by lb_set_frame_shift
    as it is by lb_init_lattice, and nothing changes; the largest shift that fits, and any shift of a line
    with fixed ends, are taken."""
    d = P.lb_lattice_named(name)
    reach = int(np.abs(d.e[:, 0]).max())
    desc = P.LatticeDesc(d.e, d.w, d.c, d.degree, (0, 0, 0))
    ctx = P.lb_init_lattice(desc, 0, N=N, precision=precision, nx_per_instance=[40, 20])
    for instance, kx in ((1, 21 - reach), (1, reach - 21), (-1, 21 - reach), (0, 41 - reach), (0, -2 ** 31), (0, 2 ** 31 - 1)):
        with pytest.raises(P.SmrtError) as e:
            P.lb_set_frame_shift(ctx, instance, kx)
        assert e.value.status == 1
    P.lb_set_frame_shift(ctx, 1, 20 - reach)
    P.lb_set_frame_shift(ctx, 0, reach - 40)
    P.lb_set_frame_shift(P.lb_init_lattice(desc, 0, N=N, precision=precision, bc_x=1, nx_per_instance=[4]), 0, 50)
    if name == "D3Q39":
        box = P.lb_init_lattice(desc, 12, 9, 9, N=N, precision=precision)
        P.lb_set_frame_shift(box, -1, 12 - reach)
        with pytest.raises(P.SmrtError):
            P.lb_set_frame_shift(box, -1, 13 - reach)
