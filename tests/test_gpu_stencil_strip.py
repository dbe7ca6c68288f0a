"""GPU parity of the column-strip kernel of 2-D stencils (several time steps
per sweep in registers) against the oracle: strips that end inside a vector,
runs of one row, fewer steps than a sweep, domains narrower than one strip.
fp64 within 1e-12 of the local value (floored at 1e-3 of the field maximum);
fp32 / bf16 storage bit for bit against the low-precision oracle."""
import numpy as np
import pytest

from paper_2204_02064_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def rel_err(g, o):
    floor = 1e-3 * max(np.max(np.abs(o)), 1e-300)
    return float(np.max(np.abs(g - o) / np.maximum(np.abs(o), floor)))


@pytest.fixture(scope="module")
def ctx():
    from paper_2204_02064_gb300 import api
    return api.Context(0)


CASES = [
    # grid shape (y, x), time steps, steps per sweep (0: the planner's), runs of rows (0: the planner's)
    ((9, 16), 5, 0, 0),
    ((37, 131), 9, 0, 0),
    ((64, 121), 4, 0, 64),
    ((50, 241), 7, 0, 3),
    ((23, 368), 1, 0, 5),
    ((301, 120), 6, 2, 7),
    ((200, 257), 11, 1, 0),
    ((130, 488), 10, 4, 0),
]


@pytest.mark.parametrize("name", ["2d5pt", "2ds9pt", "2d9pt", "2d25pt"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("shape,steps,ts,runs", CASES)
def test_strips_match_oracle(ctx, oracle, name, dtype, shape, steps, ts, runs):
    from paper_2204_02064_gb300 import api
    if dtype == "bf16":
        shape = (shape[0], shape[1] // 8 * 8)
    offs, w = inputs.shape_offsets(name), inputs.workload_weights(name, seed=5)
    st = api.Stencil(ctx, shape, offs, w, dtype=dtype, boundary=0.375)
    st.set_plan(kernel=api.KERNEL_STRIP, planes_per_barrier=ts, tiles=(0, 0, runs))
    src = torch.from_numpy(inputs.stencil_field(shape, 47)).to(TT[dtype]).cuda()
    st.set_field(src)
    try:
        stats = st.run(steps, stats=True)
    except api.PerksError as e:  # this number of steps per sweep is not compiled for the shape
        assert ts > 0 and e.name == "UNSUPPORTED"
        st.set_plan(kernel=api.KERNEL_STRIP, tiles=(0, 0, runs))
        stats = st.run(steps, stats=True)
    assert stats["kernel"] == api.KERNEL_STRIP
    out = torch.empty_like(src)
    st.get_field(out)
    torch.cuda.synchronize()
    st.close()
    if dtype == "f64":
        ref = oracle.stencil_run(src.cpu().numpy(), offs, w, steps, boundary=0.375)
        assert rel_err(out.cpu().numpy(), ref) <= 1e-12
    else:
        ref = oracle.stencil_run_lowp(src.float().cpu().numpy(), offs, w, steps, dtype, boundary=0.375)
        got = out.float().cpu().numpy()
        assert np.array_equal(got, ref), float(np.max(np.abs(got - ref)))


def test_strip_barrier_timeout_and_trace(ctx, oracle):
    """A barrier wait between two sweeps that gives up is reported and the
    context keeps working; a traced run marks every step (another kernel)."""
    from paper_2204_02064_gb300 import api
    f = inputs.stencil_field((1200, 1024), 48)
    offs, w = inputs.shape_offsets("2d9pt"), inputs.workload_weights("2d9pt")
    st = api.Stencil(ctx, f.shape, offs, w)
    src = torch.from_numpy(f).cuda()
    st.set_field(src)
    assert st.describe(20)["kernel"] == api.KERNEL_STRIP
    ctx.set_barrier_timeout(0)
    try:
        with pytest.raises(api.PerksError) as ei:
            st.run(20, stats=True)
        assert ei.value.name == "BARRIER_TIMEOUT"
    finally:
        ctx.set_barrier_timeout(2_000_000_000)
    st.set_field(src)
    st.set_trace(3)
    stats = st.run(6, stats=True)
    assert stats["kernel"] != api.KERNEL_STRIP and st.trace().shape == (4, stats["grid_blocks"], 2)
    out = torch.empty_like(src)
    st.get_field(out)
    assert rel_err(out.cpu().numpy(), oracle.stencil_run(f, offs, w, 6)) <= 1e-12


#: Steps per sweep the strips are compiled for.
COMPILED = {"f64": {"2d5pt": (1, 2), "2d9pt": (1, 2), "2ds9pt": (1, 2), "2d25pt": (1,)},
            "f32": {"2d5pt": (4,), "2d9pt": (4,), "2ds9pt": (2, 4), "2d25pt": (2,)}}
COMPILED["bf16"] = COMPILED["f32"]


@pytest.mark.parametrize("name", ["2d5pt", "2ds9pt", "2d9pt", "2d25pt"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("nx", [120, 257])
@pytest.mark.parametrize("ts", [1, 2, 4])
def test_every_number_of_steps_per_sweep(ctx, oracle, name, dtype, nx, ts):
    """Each compiled number of steps per sweep, for runs of one to nine steps (whole sweeps, and every remainder), is
    what runs; the others are refused."""
    from paper_2204_02064_gb300 import api
    shape = (301, nx // 8 * 8 if dtype == "bf16" else nx)
    offs, w = inputs.shape_offsets(name), inputs.workload_weights(name, seed=5)
    st = api.Stencil(ctx, shape, offs, w, dtype=dtype, boundary=0.375)
    src = torch.from_numpy(inputs.stencil_field(shape, 49)).to(TT[dtype]).cuda()
    st.set_plan(kernel=api.KERNEL_STRIP, planes_per_barrier=ts, tiles=(0, 0, 7))
    if ts not in COMPILED[dtype][name]:
        with pytest.raises(api.PerksError) as ei:
            st.run(1)
        assert ei.value.name == "UNSUPPORTED"
        return
    for steps in range(1, 10):
        st.set_field(src)
        stats = st.run(steps, stats=True)
        assert (stats["kernel"], stats["planes_per_sync"], stats["tiles_z"]) == (api.KERNEL_STRIP, ts, 7)
        out = torch.empty_like(src)
        st.get_field(out)
        torch.cuda.synchronize()
        if dtype == "f64":
            ref = oracle.stencil_run(src.cpu().numpy(), offs, w, steps, boundary=0.375)
            assert rel_err(out.cpu().numpy(), ref) <= 1e-12
        else:
            ref = oracle.stencil_run_lowp(src.float().cpu().numpy(), offs, w, steps, dtype, boundary=0.375)
            assert np.array_equal(out.float().cpu().numpy(), ref)
    st.close()
