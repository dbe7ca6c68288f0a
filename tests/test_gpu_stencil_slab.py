"""GPU parity of the slab-streaming kernel (3-D) and the patch kernel (small
2-D domains) against the oracle, at the edges of their tiles: rows that no
vector width divides, fewer rows than a thread owns, columns cut in the middle
of a block's share, halos as deep as a tile, fewer steps than an exchange.
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


def _check(ctx, oracle, name, dtype, shape, steps, kernel, **plan):
    from paper_2204_02064_gb300 import api
    offs, w = inputs.shape_offsets(name), inputs.workload_weights(name, seed=5)
    st = api.Stencil(ctx, shape, offs, w, dtype=dtype, boundary=0.375)
    st.set_plan(kernel=kernel, **plan)
    src = torch.from_numpy(inputs.stencil_field(shape, 51)).to(TT[dtype]).cuda()
    st.set_field(src)
    stats = st.run(steps, stats=True)
    assert stats["kernel"] == kernel
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
    return stats


@pytest.mark.parametrize("name", ["3d7pt", "3d13pt", "3d27pt", "poisson"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("shape,steps", [((7, 6, 16), 4), ((61, 9, 33), 3), ((23, 67, 129), 2), ((40, 37, 255), 3),
                                         ((30, 129, 72), 2), ((331, 5, 40), 3)])
def test_slab_matches_oracle(ctx, oracle, name, dtype, shape, steps):
    from paper_2204_02064_gb300 import api
    if dtype == "bf16":
        shape = shape[:2] + (shape[2] // 8 * 8,)
    _check(ctx, oracle, name, dtype, shape, steps, api.KERNEL_SLAB)


@pytest.mark.parametrize("name", ["2d5pt", "2ds9pt", "2d9pt", "2d25pt"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("shape,steps,tiles", [((8, 16), 5, 0), ((16, 24), 7, 3), ((64, 104), 1, 13), ((131, 93), 10, 0),
                                               ((257, 64), 3, 1), ((90, 328), 6, 0)])
def test_patch_matches_oracle(ctx, oracle, name, dtype, shape, steps, tiles):
    from paper_2204_02064_gb300 import api
    if dtype == "bf16":
        shape = (shape[0], shape[1] // 8 * 8)
    stats = _check(ctx, oracle, name, dtype, shape, steps, api.KERNEL_PATCH, tiles=(tiles, 0, 0))
    assert stats["cached_cells"] == shape[0] * shape[1]


def test_patch_wait_timeout_reported(ctx, oracle):
    """A block that waits for its neighbours past the limit ends the run with
    BARRIER_TIMEOUT; the context keeps working."""
    from paper_2204_02064_gb300 import api
    f = inputs.stencil_field((256, 256), 52)
    offs, w = inputs.shape_offsets("2d5pt"), inputs.workload_weights("2d5pt")
    st = api.Stencil(ctx, f.shape, offs, w)
    src = torch.from_numpy(f).cuda()
    st.set_field(src)
    assert st.describe(40)["kernel"] == api.KERNEL_PATCH
    ctx.set_barrier_timeout(0)
    try:
        with pytest.raises(api.PerksError) as ei:
            st.run(40, stats=True)
        assert ei.value.name == "BARRIER_TIMEOUT"
    finally:
        ctx.set_barrier_timeout(2_000_000_000)
    st.set_field(src)
    st.run(13, stats=True)
    out = torch.empty_like(src)
    st.get_field(out)
    torch.cuda.synchronize()
    assert rel_err(out.cpu().numpy(), oracle.stencil_run(f, offs, w, 13)) <= 1e-12


def test_plan_is_kept_until_the_request_changes(ctx):
    """Runs of one stencil reuse its plan; set_plan, a trace and the autotuner still take effect."""
    from paper_2204_02064_gb300 import api
    st = api.Stencil(ctx, (96, 128), inputs.shape_offsets("2d9pt"), inputs.workload_weights("2d9pt"), dtype="f32")
    first = st.describe(10)
    assert st.describe(10) == first
    st.set_plan(kernel=api.KERNEL_STRIP, tiles=(0, 0, 7))
    assert st.describe(10)["kernel"] == api.KERNEL_STRIP and st.describe(10)["tiles_z"] == 7
    st.set_plan(kernel=api.KERNEL_STRIP, tiles=(0, 0, 5))
    assert st.describe(10)["tiles_z"] == 5
    st.reset_plan()
    assert st.describe(10) == first
    st.set_trace(2)
    assert st.describe(10)["kernel"] == api.KERNEL_STREAMING
    st.set_trace(0)
    assert st.describe(10) == first
    st.close()


@pytest.mark.parametrize("name", ["3d7pt", "3d13pt", "3d27pt", "poisson"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("nx", [33, 40])
@pytest.mark.parametrize("parts", [47, 9, 8, 7, 6, 5, 2, 1])
def test_slab_parts_of_every_depth(ctx, oracle, name, dtype, nx, parts):
    """A column of 47 planes cut into parts of 1, 5, 6, 7, 8, 9, 23 and 47: ring slots filled again, the planes in the
    middle of a part without checks, for every remainder of the unrolled loops."""
    from paper_2204_02064_gb300 import api
    if dtype == "bf16":
        nx = nx // 8 * 8
    stats = _check(ctx, oracle, name, dtype, (47, 9, nx), 3, api.KERNEL_SLAB, tiles=(1, 1, parts))
    assert stats["tiles_z"] == parts
    # (fp64 without parts: the planner's own equal shares)
    assert stats["grid_blocks"] == (47 if dtype == "f64" and parts == 1 else parts)


@pytest.mark.parametrize("name", ["3d7pt", "3d13pt", "3d27pt", "poisson"])
@pytest.mark.parametrize("dtype,nx", [("f64", 9), ("f64", 16), ("f32", 9), ("f32", 16), ("bf16", 16)])
def test_slab_equal_shares_across_columns(ctx, oracle, name, dtype, nx):
    """Equal shares of seven planes that run from one column into the next (two parts per column would leave a fifth of
    the blocks idle): 61 columns of 35 planes, in fp64 one long column too."""
    from paper_2204_02064_gb300 import api
    rows = 32 * (4 if dtype == "f32" and name in ("3d27pt", "poisson") else 2)   # of a column of 8 lanes a row
    shapes = [(35, 60 * rows + 5, nx)] + ([(2200, 9, nx)] if dtype == "f64" else [])
    for shape in shapes:
        stats = _check(ctx, oracle, name, dtype, shape, 2, api.KERNEL_SLAB)
        columns = stats["tiles_x"] * stats["tiles_y"]
        assert columns == (61 if shape[0] == 35 else 1) and stats["tiles_z"] == 1
        assert stats["grid_blocks"] * 6 < columns * shape[0]
