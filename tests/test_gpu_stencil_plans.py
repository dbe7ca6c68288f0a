"""What a stencil does under a plan that names the column-strip, slab or patch
kernel and in the calls that plan is not made for: traced runs, per-step runs,
captured runs, tilings the kernel cannot take.  fp64 within 1e-12 of the local
value (floored at 1e-3 of the field maximum); fp32 bit for bit."""
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


# kernel, stencil, grid shape
NAMED = [("STRIP", "2d9pt", (200, 256)), ("STRIP", "2d5pt", (1200, 1024)), ("PATCH", "2d5pt", (96, 128)),
         ("SLAB", "3d7pt", (20, 24, 32)), ("SLAB", "3d27pt", (33, 29, 40))]


class Case:
    def __init__(self, ctx, name, shape, dtype="f64"):
        from paper_2204_02064_gb300 import api
        self.dtype = dtype
        self.offs, self.w = inputs.shape_offsets(name), inputs.workload_weights(name, seed=5)
        self.st = api.Stencil(ctx, shape, self.offs, self.w, dtype=dtype, boundary=0.25)
        self.src = torch.from_numpy(inputs.stencil_field(shape, 81)).to(TT[dtype]).cuda()
        self.st.set_field(self.src)

    def check(self, oracle, steps):
        out = torch.empty_like(self.src)
        self.st.get_field(out)
        torch.cuda.synchronize()
        f = self.src.cpu().numpy()
        if self.dtype == "f64":
            assert rel_err(out.cpu().numpy(), oracle.stencil_run(f, self.offs, self.w, steps, boundary=0.25)) <= 1e-12
        else:
            ref = oracle.stencil_run_lowp(f, self.offs, self.w, steps, self.dtype, boundary=0.25)
            assert np.array_equal(out.float().cpu().numpy(), ref)


@pytest.mark.parametrize("kernel,name,shape", NAMED)
def test_trace_under_a_plan_that_names_a_kernel_without_marks(ctx, oracle, kernel, name, shape):
    """A traced run marks every step whatever the plan names; without the trace the plan holds again."""
    from paper_2204_02064_gb300 import api
    c = Case(ctx, name, shape)
    want = getattr(api, "KERNEL_" + kernel)
    c.st.set_plan(kernel=want)
    assert c.st.run(2, stats=True)["kernel"] == want
    c.st.set_trace(3)
    assert c.st.describe(5)["kernel"] in (api.KERNEL_RESIDENT, api.KERNEL_STREAMING)
    stats = c.st.run(5, stats=True)
    tr = c.st.trace().astype(np.int64)
    assert tr.shape == (4, stats["grid_blocks"], 2)
    assert (tr[1:] > 0).all() and (tr[1:, :, 1] >= tr[1:, :, 0]).all()
    c.st.set_trace(0)
    assert c.st.run(1, stats=True)["kernel"] == want
    c.check(oracle, 8)
    c.st.close()


@pytest.mark.parametrize("name,shape", [("2d9pt", (200, 256)), ("3d27pt", (33, 29, 40))])
def test_autotune_then_trace(ctx, oracle, name, shape):
    """The plan the autotuner leaves, whichever kernel it names, can be traced; tuned under a
    trace it names one that marks its steps."""
    from paper_2204_02064_gb300 import api
    c = Case(ctx, name, shape)
    c.st.autotune(probe_steps=4)
    c.st.set_trace(2)
    stats = c.st.run(3, stats=True)
    assert c.st.trace().shape == (3, stats["grid_blocks"], 2)
    assert c.st.autotune(probe_steps=4)["kernel"] in ("resident", "streaming")
    c.check(oracle, 3)
    c.st.close()


@pytest.mark.parametrize("kernel,name,shape", NAMED)
def test_per_step_run_under_a_plan_that_names_a_persistent_kernel(ctx, oracle, kernel, name, shape):
    """Such a plan's tiles (as the autotuner leaves them) are the persistent kernel's; a per-step run takes its own."""
    from paper_2204_02064_gb300 import api
    c = Case(ctx, name, shape)
    want = getattr(api, "KERNEL_" + kernel)
    c.st.set_plan(kernel=want)
    d = c.st.describe(4)
    c.st.set_plan(kernel=want, tiles=(d["tiles_x"], d["tiles_y"], d["tiles_z"]))
    assert c.st.run(2, stats=True)["kernel"] == want
    c.st.run(3, api.PER_STEP)
    assert c.st.run(1, stats=True)["kernel"] == want
    c.check(oracle, 6)
    c.st.close()


@pytest.mark.parametrize("first", ["trace", "plan"])
@pytest.mark.parametrize("name,shape,dtype", [("2d5pt", (96, 128), "f64"), ("2d5pt", (1200, 1024), "f64"),
                                              ("3d27pt", (33, 29, 40), "f32")])
def test_captured_run_after_a_run_of_another_kernel(ctx, oracle, name, shape, dtype, first):
    """Whichever persistent kernel ran first (a traced run's, a plan's), a later run by default needs no allocation and
    can be captured in a graph."""
    from paper_2204_02064_gb300 import api
    c = Case(ctx, name, shape, dtype)
    if first == "trace":
        c.st.set_trace(2)
        c.st.run(4)
        c.st.set_trace(0)
    else:
        c.st.set_plan(kernel=api.KERNEL_STREAMING, tiles=(0, 0, 0))
        c.st.run(4)
        c.st.reset_plan()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.st.run(8)            # an even number of exchanges or sweeps: every replay starts where the last ended
    graph.replay()
    torch.cuda.synchronize()
    c.check(oracle, 12)
    c.st.close()


def test_tilings_a_kernel_cannot_take_are_refused(ctx, oracle):
    """Strips, slabs and patches take the tiles they are asked for or refuse them; the planner's own are taken."""
    from paper_2204_02064_gb300 import api
    flat, box = Case(ctx, "2d9pt", (200, 256)), Case(ctx, "3d7pt", (30, 70, 96), "f32")
    for c, kernel, bad in ((flat, api.KERNEL_STRIP, [(17, 0, 0), (0, 2, 0)]),
                           (flat, api.KERNEL_PATCH, [(0, 2, 0), (200, 0, 0)]),
                           (box, api.KERNEL_SLAB, [(17, 0, 0), (0, 17, 0), (2, 2, 0), (0, 0, 31)])):
        c.st.set_plan(kernel=kernel)
        d = c.st.describe(4)
        own = (d["tiles_x"], d["tiles_y"], d["tiles_z"])
        c.st.set_plan(kernel=kernel, tiles=own)
        assert c.st.describe(4) == d
        for tiles in bad:
            c.st.set_plan(kernel=kernel, tiles=tiles)
            with pytest.raises(api.PerksError) as ei:
                c.st.run(1)
            assert ei.value.name == "UNSUPPORTED"
    # rows of 32, 16 or 8 lanes, four cells each, two rows per thread: columns of 128 x 16, 64 x 32 or 32 x 64 cells
    steps = 0
    for tiles in ((1, 5, 0), (2, 3, 0), (3, 2, 5), (2, 0, 7), (0, 0, 7), (0, 5, 30)):
        box.st.set_plan(kernel=api.KERNEL_SLAB, tiles=tiles)
        d = box.st.run(3, stats=True)
        steps += 3
        assert d["kernel"] == api.KERNEL_SLAB
        assert all(want in (0, got) for want, got in zip(tiles, (d["tiles_x"], d["tiles_y"], d["tiles_z"])))
        assert d["grid_blocks"] <= 2 * ctx.info()["sm_count"]
    box.check(oracle, steps)
    flat.st.close()
    box.st.close()
