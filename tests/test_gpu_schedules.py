"""Launch schedules of 1D-line contexts: what a context runs by default, what lb_get_schedule says of
it, and that changing the schedule between graph replays changes nothing but the launch."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2401_11086_gb300 as P  # noqa: E402
from paper_2401_11086_gb300 import shocks  # noqa: E402
from paper_2401_11086_gb300.autotune import tuned_schedule  # noqa: E402


def _float_shocks(name, lengths):
    d = P.lb_lattice_named(name)
    Ma, theta1 = (3.0, 0.333) if name == "D3Q729" else (7.0, 0.071)
    n = len(lengths)
    ctx, f, _ = shocks.setup_batch(d, 5, [Ma] * n, lengths, precision="f32", width=0.0, theta1=[theta1] * n)
    g = torch.Generator(device="cuda").manual_seed(7)
    f *= 1.0 + 1e-3 * torch.randn(f.shape, dtype=f.dtype, device="cuda", generator=g)
    return ctx, f


# more than 32 cells per SM on 152 SMs, below which D3Q729 takes one block per cell
BATCHES = [[128] * 40, [1, 63, 64, 65, 127, 129, 200] * 8, [400] * 20]


@pytest.mark.parametrize("name", ["D3Q729", "D3Q4913"])
@pytest.mark.parametrize("lengths", BATCHES)
@pytest.mark.parametrize("first,then", [(None, 128), (None, 64), (128, 64), (64, 32)])
def test_graph_follows_a_change_of_tile_width(name, lengths, first, then):
    """lb_step_graph under one width (None: the default), then under another, on the same buffers and
    step count: bit for bit the persistent steps that the graphs hold."""
    ctx, f = _float_shocks(name, lengths)
    default = P.lb_get_schedule(ctx)["tile_width"]
    if first is not None or default == 1:  # one block per cell has no graph form
        P.lb_set_schedule(ctx, first or 64, 0, 0)
    fa, fb = f.clone(), ctx.new_state()
    P.lb_step_graph(ctx, fa, fb, 2)
    P.lb_set_schedule(ctx, then, 0, 0)
    P.lb_step_graph(ctx, fa, fb, 2)
    ga, gb = f.clone(), ctx.new_state()
    for width in (first or (64 if default == 1 else default), then):
        P.lb_set_schedule(ctx, width, 0, 1)
        P.lb_step(ctx, ga, gb, 2)
    assert P.lb_poll_status(ctx)[0] == 0
    assert torch.equal(ctx.planes(fa), ctx.planes(ga)) and torch.equal(ctx.planes(fb), ctx.planes(gb))


def test_reported_width_is_the_one_that_runs():
    """Float D3Q729 batches on both sides of the width rule, ragged ones among them, all above the size of
    one block per cell: lb_get_schedule names the default width, 64 and 128 both occur, and setting the
    reported schedule, or the other width, gives the default's bits."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cells = 32 * sms + 1
    ragged = [1, 7, 63, 64, 65, 127, 128, 129]
    batches = [[128] * (cells // 128 + 2), ragged * (cells // sum(ragged) + 1), [128] * sms, [1000] * sms]
    seen = set()
    for lengths in batches:
        ctx, f = _float_shocks("D3Q729", lengths)
        s = P.lb_get_schedule(ctx)
        assert s["tile_width"] in (64, 128) and s["persistent"] == 0
        seen.add(s["tile_width"])
        want = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)).clone()
        for width in (s["tile_width"], 192 - s["tile_width"]):
            P.lb_set_schedule(ctx, width, s["blocks_per_sm"], s["persistent"], s["tensor_cores"])
            assert torch.equal(ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)), want)
    assert seen == {64, 128}


# ------------------------------------------------------------------ groups of lanes (tile width 1)
LANES = [("D3Q39", 3, 1.25), ("D3Q103", 4, 2.0)]


def _shocks(name, N, Ma, lengths, precision="f64"):
    ctx, f, _ = shocks.setup_batch(P.lb_lattice_named(name), N, [Ma] * len(lengths), lengths, precision=precision,
                                   width=4.0)
    g = torch.Generator(device="cuda").manual_seed(7)
    f *= 1.0 + 1e-3 * torch.randn(f.shape, dtype=f.dtype, device="cuda", generator=g)
    return ctx, f


@pytest.mark.parametrize("name,N,Ma", LANES)
@pytest.mark.parametrize("lengths", [[400], [130, 7, 300]])
def test_small_double_lines_keep_their_default_schedule(name, N, Ma, lengths, tmp_path):
    """The schedule that a small double line context starts on is reported, set again after others, chosen
    by the autotuner (by more than a factor of two at these sizes) and stored, with the same bits."""
    ctx, f = _shocks(name, N, Ma, lengths)
    step = lambda c, nsteps=3: c.planes(P.lb_step(c, f.clone(), c.new_state(), nsteps)).clone()  # noqa: E731
    want = step(ctx)
    s = P.lb_get_schedule(ctx)
    assert (s["tile_width"], s["persistent"]) == (1, 0)
    put = lambda q: P.lb_set_schedule(ctx, q["tile_width"], q["blocks_per_sm"], q["persistent"],  # noqa: E731
                                      q["tensor_cores"])
    put(s)
    assert torch.equal(step(ctx), want)
    P.lb_set_schedule(ctx, 32, 0, 1)
    other = step(ctx)
    assert not torch.equal(other, want) and ((other - want).abs().max() / want.abs().max()).item() < 1e-13
    put(s)
    assert torch.equal(step(ctx), want)
    best = P.lb_autotune(ctx, f.clone(), ctx.new_state(), 20)
    assert best["tile_width"] == 1 and P.lb_get_schedule(ctx)["tile_width"] == 1
    assert torch.equal(step(ctx), want)
    path = str(tmp_path / "sched.json")
    P.lb_set_schedule(ctx, 64, 0, 0)
    assert tuned_schedule(ctx, f, lengths, trial_steps=20, path=path)["tile_width"] == 1
    again, _ = _shocks(name, N, Ma, lengths)
    P.lb_set_schedule(again, 64, 0, 0)
    tuned_schedule(again, f, lengths, trial_steps=20, path=path)  # from the file
    assert torch.equal(step(again), want)
    assert P.lb_poll_status(ctx)[0] == 0


def test_width_one_is_refused_elsewhere():
    """Tile width 1 stays unsupported for persistent launches, float states and grids above 32 cells per SM,
    and a refused schedule leaves the context as it was."""
    big = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    for lengths, precision, persistent in (([400], "f64", 1), ([400], "f32", 0), ([400], "f32c64", 0),
                                           ([big], "f64", 0)):
        ctx, f = _shocks("D3Q39", 3, 1.25, lengths, precision)
        before = P.lb_get_schedule(ctx)
        with pytest.raises(P.SmrtError) as e:
            P.lb_set_schedule(ctx, 1, 0, persistent)
        assert e.value.status == 5 and P.lb_get_schedule(ctx) == before


# ------------------------------------------------------------------ blocks of the persistent launch
@pytest.mark.parametrize("name,N,Ma,precision,cells", [("D3Q729", 4, 3.0, "f64", 20), ("D3Q4913", 5, 7.0, "f64", 40),
                                                       ("D3Q103", 4, 2.0, "f32c64", 40), ("D3Q39", 3, 1.25, "f32c64", 40)])
@pytest.mark.parametrize("per_sm", [1, 3.2, 6.5])
def test_open_number_of_blocks_gives_the_same_bits(name, N, Ma, precision, cells, per_sm):
    """The persistent launch that leaves its blocks open (blocks_per_sm 0), below, in and above the range where
    it takes fewer than fit, against one block per SM: the same kernel on another grid."""
    count = int(per_sm * torch.cuda.get_device_properties(0).multi_processor_count)
    theta1 = {"D3Q729": [0.333] * count, "D3Q4913": [0.071] * count}.get(name)
    ctx, f, _ = shocks.setup_batch(P.lb_lattice_named(name), N, [Ma] * count, [cells] * count, precision=precision,
                                   width=0.0, theta1=theta1)
    for width in (128, 64):
        runs = []
        for blocks in (0, 1):
            P.lb_set_schedule(ctx, width, blocks, 1)
            runs.append(ctx.planes(P.lb_step(ctx, f.clone(), ctx.new_state(), 3)).clone())
            assert P.lb_poll_status(ctx)[0] == 0
            if precision != "f64":  # the step counter seeds the stochastic rounding: start both alike
                ctx, _, _ = shocks.setup_batch(P.lb_lattice_named(name), N, [Ma] * count, [cells] * count,
                                               precision=precision, width=0.0, theta1=theta1)
        assert torch.equal(runs[0], runs[1])


def test_periodic_float_lines_start_on_128_cell_tiles(name="D3Q729"):
    """At sizes where lines with fixed ends start on 64-cell tiles; the bits of either width."""
    d = P.lb_lattice_named(name)
    lengths = [128] * (32 * torch.cuda.get_device_properties(0).multi_processor_count // 128 + 2)
    assert P.lb_get_schedule(_float_shocks(name, lengths)[0])["tile_width"] == 64
    ctx = P.lb_init_lattice(P.LatticeDesc(d.e, d.w, d.c, d.degree, (1, 0, 0)), 0, N=5, precision="f32",
                            nx_per_instance=lengths)
    assert P.lb_get_schedule(ctx)["tile_width"] == 128
    P.lb_set_relaxation(ctx, [2.0] * shocks.ntau(5), True, 1.0)
    one = torch.ones(ctx.cells, dtype=torch.float64, device="cuda")
    f = ctx.new_state()
    P.lb_fill_equilibrium(ctx, f, one, torch.stack([d.c * one, 0 * one, 0 * one]).contiguous(), one)
    g = torch.Generator(device="cuda").manual_seed(7)
    f *= 1.0 + 1e-3 * torch.randn(f.shape, dtype=f.dtype, device="cuda", generator=g)
    want = ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)).clone()
    for width in (128, 64):
        P.lb_set_schedule(ctx, width, 0, 0)
        assert torch.equal(ctx.planes(P.lb_step(ctx, f, ctx.new_state(), 1)), want)
    assert P.lb_poll_status(ctx)[0] == 0
