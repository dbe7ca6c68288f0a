"""GPU parity of the warm-start network's kernels against the oracle, and
the gain of the trained network as a CG warm start.

Forward: F32 storage within 1e-4 of the fp64 oracle (relative to the output's
max); BF16 storage against the oracle with every activation rounded to bf16
as the kernels store it (1e-2: an fp32 sum that lands on a bf16 rounding
boundary may round the other way).  Gradients: F32 storage within 1e-4 of
the oracle's reverse-mode gradient (relative to the largest component); the
oracle's gradient is itself pinned by central differences.
"""
import numpy as np
import pytest

from paper_2204_02064_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

C1 = 32
DIL = (1, 2, 4, 8)


@pytest.fixture(scope="module")
def ctx():
    from paper_2204_02064_gb300 import api
    return api.Context(0)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _params(seed, scale=1.0):
    rng = np.random.default_rng(seed)
    parts = []
    for co, ci in [(C1, 2), (C1, C1), (C1, C1), (1, C1)]:
        parts += [rng.standard_normal(co * ci * 9) * scale * np.sqrt(2.0 / (9 * ci)),
                  rng.standard_normal(co) * 0.05]
    return np.concatenate(parts).astype(np.float32)


def _case(nimg, ny, nx, seed):
    k, f = inputs.poisson_problems(max(ny, nx), nimg, seed=seed, ell=4.0)
    return k[:, :ny, :nx].copy(), f[:, :ny, :nx].copy()


def _features(k, f, rnd=lambda a: a):
    return np.stack([rnd(np.log(k)), rnd(f)], axis=1)


@pytest.mark.parametrize("shape", [(2, 20, 23), (1, 16, 16), (3, 37, 5)])
def test_forward_f32_matches_oracle(ctx, oracle, shape):
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = shape
    k, f = _case(nimg, ny, nx, 41)
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1)
    p = _params(3)
    net.params = p
    net.scale = 2.5
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), u)
    torch.cuda.synchronize()
    x = _features(k, f, lambda a: a.astype(np.float32).astype(np.float64))
    ref = np.stack([oracle.warmnet_forward(p.astype(np.float64), x[i], C1, DIL) for i in range(nimg)]) * 2.5
    got = u.cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref))


def test_forward_bf16_matches_rounded_oracle(ctx, oracle):
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 2, 33, 40
    k, f = _case(nimg, ny, nx, 42)
    net = api.WarmNet(ctx, storage=api.BF16, dilations=DIL, seed=1)
    p = _params(4)
    net.params = p
    net.scale = 1.0
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), u)
    torch.cuda.synchronize()
    rb = oracle.bf16_round
    x = _features(k, f, lambda a: rb(a.astype(np.float32)).astype(np.float64))
    pd = p.astype(np.float64)
    offs, o = [], 0
    for co, ci in [(C1, 2), (C1, C1), (C1, C1), (1, C1)]:
        W = pd[o:o + co * ci * 9].reshape(co, ci, 3, 3)
        o += co * ci * 9
        B = pd[o:o + co]
        o += co
        offs.append((W, B))
    ref = []
    for i in range(nimg):
        y = x[i]
        for l, (W, B) in enumerate(offs):
            y = oracle.conv2d(y, W, B, DIL[l])
            if l < 3:
                y = rb(np.maximum(y, 0).astype(np.float32)).astype(np.float64)
        ref.append(y[0])
    ref = np.stack(ref)
    got = u.cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-2 * np.max(np.abs(ref))


@pytest.mark.parametrize("shape", [(2, 20, 23), (3, 16, 33)])
def test_gradient_f32_matches_oracle(ctx, oracle, shape):
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = shape
    k, f = _case(nimg, ny, nx, 43)
    u = inputs.uniform(44, nimg * ny * nx).reshape(nimg, ny, nx) * 3.0 - 1.0
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1)
    p = _params(5)
    net.params = p
    net.scale = 1.5
    loss, g = net.gradient(_dev(k), _dev(f), _dev(u))
    x = _features(k, f, lambda a: a.astype(np.float32).astype(np.float64))
    ref_loss, ref_g = oracle.warmnet_grad(p.astype(np.float64), x, u / 1.5, C1, DIL)
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    assert np.max(np.abs(g - ref_g)) <= 1e-4 * np.max(np.abs(ref_g))


def test_gradient_bf16_close_to_oracle(ctx, oracle):
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 2, 24, 24
    k, f = _case(nimg, ny, nx, 45)
    u = inputs.uniform(46, nimg * ny * nx).reshape(nimg, ny, nx) * 2.0 - 1.0
    net = api.WarmNet(ctx, storage=api.BF16, dilations=DIL, seed=1)
    p = _params(6)
    net.params = p
    loss, g = net.gradient(_dev(k), _dev(f), _dev(u))
    x = _features(k, f)
    ref_loss, ref_g = oracle.warmnet_grad(p.astype(np.float64), x, u, C1, DIL)
    assert loss == pytest.approx(ref_loss, rel=5e-2)
    assert np.linalg.norm(g - ref_g) <= 5e-2 * np.linalg.norm(ref_g)


def test_adam_step_matches_formula(ctx):
    """One Adam step from zero moments moves every parameter by
    lr * g / (|g| + eps) (bias-corrected first step)."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 1, 16, 16
    k, f = _case(nimg, ny, nx, 47)
    u = inputs.uniform(48, nimg * ny * nx).reshape(nimg, ny, nx)
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=2)
    p0 = net.params
    _, g = net.gradient(_dev(k), _dev(f), _dev(u))
    net.train_step(_dev(k), _dev(f), _dev(u), lr=1e-3)
    p1 = net.params
    expect = p0 - 1e-3 * g / (np.abs(g) + 1e-8)
    assert np.max(np.abs(p1 - expect)) <= 1e-6


def _solve(ctx, k, f, x0=None, rtol=1e-8):
    from paper_2204_02064_gb300 import api
    P = api.Poisson(ctx, k)
    x = torch.zeros_like(f) if x0 is None else x0.clone()
    res = P.solve(f, x, rtol=rtol)
    return x, res


def _timed_solve(ctx, k, f, net=None, rtol=1e-8):
    """Wall time (CUDA events) of one batched solve to rtol, the network's
    inference included when `net` gives the start; returns (ms, stats)."""
    from paper_2204_02064_gb300 import api
    P = api.Poisson(ctx, k)
    x = torch.zeros_like(f)
    torch.cuda.synchronize()
    s = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(s)
    if net is not None:
        net.predict(k, f, x)
    P.solve(f, x, rtol=rtol, stats=False)
    e1.record(s)
    e1.synchronize()
    ms = e0.elapsed_time(e1)
    x2 = torch.zeros_like(f)
    if net is not None:
        net.predict(k, f, x2)
    res = P.solve(f, x2, rtol=rtol)
    P.close()
    return ms, res


def test_trained_net_gains_over_zero_start(ctx):
    """Train on solver-generated pairs, then solve held-out problems to 1e-8
    from zero and from the network's prediction: both reach the tolerance
    (CG decides), and the warm start needs fewer iterations and less wall
    time, its inference included (medians of five alternated timed solves
    of each start)."""
    from paper_2204_02064_gb300 import api
    n, ntrain, ntest = 64, 512, 64
    k, f = inputs.poisson_problems_device(n, ntrain + ntest, seed=inputs.SEED_POISSON, ell=4.0)
    u, res = _solve(ctx, k[:ntrain].contiguous(), f[:ntrain].contiguous(), rtol=1e-10)
    assert res["max_true_rel_residual"] <= 1e-10
    net = api.WarmNet(ctx, storage=api.BF16, dilations=DIL, seed=3)
    losses = net.fit(k[:ntrain].contiguous(), f[:ntrain].contiguous(), u, batch=16, epochs=30, lr=2e-3)
    assert losses[-1] < 0.5 * losses[0]
    kt, ft = k[ntrain:].contiguous(), f[ntrain:].contiguous()
    _, zero = _solve(ctx, kt, ft)
    u0 = torch.zeros_like(ft)
    net.predict(kt, ft, u0)
    _, warm = _solve(ctx, kt, ft, x0=u0)
    assert zero["max_true_rel_residual"] <= 1e-8 and warm["max_true_rel_residual"] <= 1e-8
    print("zero-start mean iterations %.1f, warm-start %.1f, losses %s"
          % (zero["mean_iterations"], warm["mean_iterations"], losses[[0, -1]]))
    assert warm["mean_iterations"] < zero["mean_iterations"]
    t_zero, t_warm = [], []
    for rep in range(5):
        for which in ((0, 1) if rep % 2 == 0 else (1, 0)):
            ms, r = _timed_solve(ctx, kt, ft, net if which else None)
            assert r["max_true_rel_residual"] <= 1e-8
            (t_warm if which else t_zero).append(ms)
    print("zero-start ms %s, warm-start ms %s" % (sorted(t_zero), sorted(t_warm)))
    assert np.median(t_warm) < np.median(t_zero)


def _pool(a, F):
    n, ny, nx = a.shape
    return a.reshape(n, ny // F, F, nx // F, F).mean(axis=(2, 4))


def _bilinear(c, F):
    """Cell-centred bilinear interpolation of (n, H, W) to (n, H F, W F), clamped."""
    n, H, W = c.shape
    yc = np.clip((np.arange(H * F) + 0.5) / F - 0.5, 0, H - 1)
    xc = np.clip((np.arange(W * F) + 0.5) / F - 0.5, 0, W - 1)
    y0 = np.floor(yc).astype(int)
    x0 = np.floor(xc).astype(int)
    y1 = np.minimum(y0 + 1, H - 1)
    x1 = np.minimum(x0 + 1, W - 1)
    wy = (yc - y0)[:, None]
    wx = (xc - x0)[None, :]
    out = np.empty((n, H * F, W * F))
    for i in range(n):
        o = c[i]
        out[i] = (1 - wy) * ((1 - wx) * o[y0][:, x0] + wx * o[y0][:, x1]) + wy * ((1 - wx) * o[y1][:, x0] + wx * o[y1][:, x1])
    return out


@pytest.mark.parametrize("F", [2, 4])
def test_pooled_forward_matches_oracle(ctx, oracle, F):
    """Coarse-grid mode: inputs averaged over F x F blocks, the network on the
    coarse grid, the output interpolated bilinearly back to the fine cells."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 2, 32, 40
    k, f = _case(nimg, ny, nx, 51)
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1, pool=F)
    p = _params(7)
    net.params = p
    net.scale = 3.0
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), u)
    torch.cuda.synchronize()
    x = np.stack([_pool(np.log(k), F), _pool(f, F)], axis=1).astype(np.float32).astype(np.float64)
    coarse = np.stack([oracle.warmnet_forward(p.astype(np.float64), x[i], C1, DIL) for i in range(nimg)])
    ref = _bilinear(coarse, F) * 3.0
    got = u.cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref))
    with pytest.raises(api.PerksError):
        net.predict(_dev(k[:, :31, :]), _dev(f[:, :31, :]), torch.zeros((nimg, 31, nx), dtype=torch.float64,
                                                                       device="cuda"))


def test_pooled_gradient_matches_oracle(ctx, oracle):
    from paper_2204_02064_gb300 import api
    F, nimg, ny, nx = 2, 2, 24, 30
    k, f = _case(nimg, ny, nx, 52)
    u = inputs.uniform(53, nimg * ny * nx).reshape(nimg, ny, nx) * 2.0 - 1.0
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1, pool=F)
    p = _params(8)
    net.params = p
    net.scale = 0.5
    loss, g = net.gradient(_dev(k), _dev(f), _dev(u))
    x = np.stack([_pool(np.log(k), F), _pool(f, F)], axis=1).astype(np.float32).astype(np.float64)
    ref_loss, ref_g = oracle.warmnet_grad(p.astype(np.float64), x, _pool(u, F) / 0.5, C1, DIL)
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    assert np.max(np.abs(g - ref_g)) <= 1e-4 * np.max(np.abs(ref_g))


def _dyadic_params(seed):
    """Network parameters on coarse binary grids: layer-1 weights in
    {-3..3}/16, inner weights sparse in {-1, 0, 1}/64, output weights in
    {-1, 0, 1}/64, biases in {-8..8}/256 -- every value exact in bf16."""
    def u(n, k):
        return inputs.uniform(inputs.substream(seed, k), n)
    parts = [(np.floor(u(C1 * 2 * 9, 1) * 7) - 3) / 16, (np.floor(u(C1, 2) * 17) - 8) / 256]
    for l, (co, ci) in enumerate([(C1, C1), (C1, C1), (1, C1)]):
        a, s = u(co * ci * 9, 3 + 2 * l), u(co * ci * 9, 4 + 2 * l)
        w = np.where(a < 0.25, np.where(s < 0.5, -1.0, 1.0), 0.0) if co > 1 else np.floor(s * 3) - 1
        parts += [w / 64, (np.floor(u(co, 10 + l) * 17) - 8) / 256]
    return np.concatenate(parts).astype(np.float32)


def _rounded_oracle(oracle, p, x):
    """The fp64 oracle network with every hidden activation rounded to bf16
    (as the kernels store it); also returns, per layer, log2 of the largest
    sum of |terms| in units of the layer's value grid (the bits an exact sum
    needs)."""
    pd = p.astype(np.float64)
    layers, o = [], 0
    for co, ci in [(C1, 2), (C1, C1), (C1, C1), (1, C1)]:
        W = pd[o:o + co * ci * 9].reshape(co, ci, 3, 3)
        o += co * ci * 9
        layers.append((W, pd[o:o + co]))
        o += co
    rb = oracle.bf16_round
    out, bits = [], 0.0
    for i in range(x.shape[0]):
        y = x[i]
        for l, (W, B) in enumerate(layers):
            g = 0
            while not np.all(np.round(y * 2.0 ** g) == y * 2.0 ** g):
                g += 1
            gw = 0
            while not np.all(np.round(np.concatenate([W.ravel(), B]) * 2.0 ** gw)
                             == np.concatenate([W.ravel(), B]) * 2.0 ** gw):
                gw += 1
            sabs = oracle.conv2d(np.abs(y), np.abs(W), np.abs(B), DIL[l])
            bits = max(bits, float(np.log2(sabs.max() * 2.0 ** (g + gw) + 1)))
            y = oracle.conv2d(y, W, B, DIL[l])
            if l < 3:
                y = rb(np.maximum(y, 0).astype(np.float32)).astype(np.float64)
        out.append(y[0])
    return np.stack(out), bits


@pytest.mark.parametrize("shape", [(2, 7, 300), (1, 33, 128), (3, 16, 40)])
@pytest.mark.parametrize("tc", [True, False])
def test_bf16_layers_match_rounded_oracle_exactly(ctx, oracle, shape, tc):
    """BF16 storage, inner layers as tcgen05 implicit GEMMs (tc) or on the
    CUDA cores: with inputs and parameters on coarse binary grids every
    product and partial sum is exact in fp32 (the test checks that the
    largest sum needs < 24 bits), so in any summation order each layer's
    fp32 result is the exact one, and rounding it to bf16 gives the same
    bits as the oracle rounded the same way.  The output must equal the
    rounded oracle element for element, ragged 128-pixel tiles included."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = shape
    k = np.ones((nimg, ny, nx))                                   # log k = 0 exactly
    f = (np.floor(inputs.uniform(inputs.substream(78, nx), nimg * ny * nx) * 9) - 4).reshape(nimg, ny, nx) / 4
    p = _dyadic_params(77)
    ref, bits = _rounded_oracle(oracle, p, _features(k, f))
    assert bits < 24, bits
    net = api.WarmNet(ctx, storage=api.BF16, dilations=DIL, seed=1)
    net.set_tensor_cores(tc)
    net.params = p
    net.scale = 1.0
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), u)
    torch.cuda.synchronize()
    got = u.cpu().numpy()
    net.close()
    assert np.max(np.abs(ref)) > 1e-3
    assert np.array_equal(got, ref), np.max(np.abs(got - ref))


@pytest.mark.parametrize("shape", [(2, 7, 300), (3, 16, 40)])
def test_tensor_core_layers_close_to_rounded_oracle(ctx, oracle, shape):
    """Random parameters (not bf16-exact; the tensor-core operands round them
    to bf16): the tcgen05 forward against the bf16-rounded oracle, per
    element, within 2e-2 of the output's largest magnitude."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = shape
    k, f = _case(nimg, ny, nx, 61)
    p = _params(9)
    x = _features(k, f, lambda a: oracle.bf16_round(a.astype(np.float32)).astype(np.float64))
    ref, _ = _rounded_oracle(oracle, p, x)
    net = api.WarmNet(ctx, storage=api.BF16, dilations=DIL, seed=1)
    net.set_tensor_cores(True)
    net.params = p
    net.scale = 1.0
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), u)
    torch.cuda.synchronize()
    got = u.cpu().numpy()
    net.close()
    assert np.max(np.abs(got - ref)) <= 2e-2 * np.max(np.abs(ref))
    assert np.corrcoef(got.ravel(), ref.ravel())[0, 1] > 0.999


def _pass_through_params(channel):
    """Parameters that hand input channel `channel` (positive) through the centre taps unchanged."""
    p = np.zeros(32 * 2 * 9 + 32 + 2 * (32 * 32 * 9 + 32) + 32 * 9 + 1, dtype=np.float32)
    at = 0
    for layer, (ci, co) in enumerate(((2, 32), (32, 32), (32, 32), (32, 1))):
        p[at + (channel if layer == 0 else 0) * 9 + 4] = 1.0
        at += co * ci * 9 + co
    return p


@pytest.mark.parametrize("F,shape", [(1, (2, 5, 7)), (2, (1, 6, 258)), (3, (2, 9, 771)), (5, (1, 35, 45)),
                                     (8, (2, 136, 72)), (16, (1, 48, 272)), (31, (1, 62, 93)), (32, (1, 64, 96))])
@pytest.mark.parametrize("channel", [0, 1])
def test_pooling_and_interpolation(ctx, F, shape, channel):
    """Block means of log k and f, and the interpolation back, through a network
    that passes one channel on.  Both sides round a mean to fp32 once (half an
    ulp, 2^-24 each); everything else is fp64."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = shape
    n = nimg * ny * nx
    k = np.exp(40.0 * inputs.uniform(61, n)).reshape(shape)   # logs 0..40: the exponents' sum carries the mean
    f = 1.0 + inputs.uniform(62, n).reshape(shape)
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1, pool=F)
    net.params = _pass_through_params(channel)
    net.scale = 2.0
    ref = _bilinear(_pool(np.log(k) if channel == 0 else f, F), F) * 2.0
    # u at an odd offset too: rows that 16-byte stores cannot write
    for off in (0, 1):
        flat = torch.full((n + 1 + off,), -7.0, dtype=torch.float64, device="cuda")
        u = flat[off:off + n].reshape(shape)
        net.predict(_dev(k), _dev(f), u)
        torch.cuda.synchronize()
        assert np.max(np.abs(u.cpu().numpy() - ref)) <= 2.0 ** -22 * np.max(np.abs(ref))
        assert bool((flat[off + n:] == -7.0).all()) and bool((flat[:off] == -7.0).all())


@pytest.mark.parametrize("F", [1, 4])
@pytest.mark.parametrize("value", [5e-324, 1e-310, 2.2250738585072014e-308, 1.7e308])
def test_log_of_extreme_coefficients(ctx, F, value):
    """A subnormal, the smallest normal and a huge coefficient: the mean log of their coarse cell, from a
    network that subtracts ReLU(-x) from ReLU(x) (fp32 rounding of a mean, as above)."""
    from paper_2204_02064_gb300 import api
    ny, nx = 4 * F, 8 * F
    k = np.full((1, ny, nx), np.e)
    k[0, F, 3 * F - 1] = value
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1, pool=F)
    p = _pass_through_params(0)
    p[2 * 9 + 4] = -1.0
    a1 = 32 * 2 * 9 + 32
    p[a1 + (32 + 1) * 9 + 4] = 1.0
    a2 = a1 + 32 * 32 * 9 + 32
    p[a2 + (32 + 1) * 9 + 4] = 1.0
    p[a2 + 32 * 32 * 9 + 32 + 9 + 4] = -1.0
    net.params = p
    net.scale = 1.0
    u = torch.zeros((1, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(np.zeros_like(k)), u)
    torch.cuda.synchronize()
    ref = _bilinear(_pool(np.log(k), F), F)
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 2.0 ** -22 * np.max(np.abs(ref))


@pytest.mark.parametrize("F,ny,nx,nimg", [(1, 13, 300, 75), (2, 40, 258, 61), (3, 60, 255, 97), (8, 64, 264, 150),
                                          (32, 64, 320, 500)])
def test_pooling_rounds_of_jobs(ctx, F, ny, nx, nimg):
    """Large batches pool several rows of coarse cells per round, single images
    one: the same bits for every image, a partly filled last round included."""
    from paper_2204_02064_gb300 import api
    k = np.exp(6.0 * inputs.uniform(71, nimg * ny * nx) - 3.0).reshape(nimg, ny, nx)
    f = (2.0 * inputs.uniform(72, nimg * ny * nx) - 1.0).reshape(nimg, ny, nx)
    k[nimg - 1, 0, 0] = 5e-324                                    # a logarithm of its own
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=3, pool=F)
    net.scale = 1.5
    dk, df = _dev(k), _dev(f)
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(dk, df, u)
    one = torch.zeros((1, ny, nx), dtype=torch.float64, device="cuda")
    for i in (0, 1, nimg // 2, nimg - 2, nimg - 1):
        net.predict(dk[i:i + 1].contiguous(), df[i:i + 1].contiguous(), one)
        torch.cuda.synchronize()
        assert torch.equal(one[0], u[i]), i
    net.close()


@pytest.mark.parametrize("F", [1, 2, 3, 8, 32])
@pytest.mark.parametrize("amp", [1e-5, 1e-7, 1e-9, 1e-12, 2e-16, 0.0])
def test_log_of_coefficients_near_one(ctx, F, amp):
    """Coefficients 1 + amp x [-1/4, 1]: the mean log keeps its digits however small it is, from the network of the
    test above (fp32 rounding of a mean); a field of ones gives 0."""
    from paper_2204_02064_gb300 import api
    ny, nx = 4 * F, 8 * F
    k = 1.0 + amp * (1.25 * inputs.uniform(91, ny * nx).reshape(1, ny, nx) - 0.25)
    net = api.WarmNet(ctx, storage=api.F32, dilations=DIL, seed=1, pool=F)
    p = _pass_through_params(0)
    p[2 * 9 + 4] = -1.0
    a1 = 32 * 2 * 9 + 32
    p[a1 + (32 + 1) * 9 + 4] = 1.0
    a2 = a1 + 32 * 32 * 9 + 32
    p[a2 + (32 + 1) * 9 + 4] = 1.0
    p[a2 + 32 * 32 * 9 + 32 + 9 + 4] = -1.0
    net.params = p
    net.scale = 1.0
    u = torch.zeros((1, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(np.zeros_like(k)), u)
    torch.cuda.synchronize()
    ref = _bilinear(_pool(np.log(k), F), F)
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 2.0 ** -22 * np.max(np.abs(ref))


@pytest.mark.parametrize("dil", [(16, 16, 16, 16), (3, 12, 5, 16), (1, 7, 13, 2)])
def test_forward_bf16_other_dilations(ctx, oracle, dil):
    """The tensor-core layers' staged halo, operand strides and shared memory follow the dilation, up to the largest
    the ABI takes; tolerance as for the default dilations (a sum on a bf16 rounding boundary)."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 2, 53, 70
    k, f = _case(nimg, ny, nx, 51)
    net = api.WarmNet(ctx, storage=api.BF16, dilations=dil, seed=1)
    p = _params(8)
    net.params = p
    net.scale = 1.0
    u = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), u)
    torch.cuda.synchronize()
    rb = oracle.bf16_round
    x = _features(k, f, lambda a: rb(a.astype(np.float32)).astype(np.float64))
    pd, ref = p.astype(np.float64), []
    for i in range(nimg):
        y, o = x[i], 0
        for l, (co, ci) in enumerate([(C1, 2), (C1, C1), (C1, C1), (1, C1)]):
            W, B = pd[o:o + co * ci * 9].reshape(co, ci, 3, 3), pd[o + co * ci * 9:o + co * ci * 9 + co]
            o += co * ci * 9 + co
            y = oracle.conv2d(y, W, B, dil[l])
            if l < 3:
                y = rb(np.maximum(y, 0).astype(np.float32)).astype(np.float64)
        ref.append(y[0])
    ref = np.stack(ref)
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 1e-2 * np.max(np.abs(ref))


@pytest.mark.parametrize("dil", [(16, 11, 3, 16), (5, 8, 11, 13)])
def test_f32_other_dilations(ctx, oracle, dil):
    """Forward and gradient in fp32 at dilations whose tiles are mostly halo (11: the widest the inner layers' forward
    takes); tolerances of the default dilations."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 2, 37, 51
    k, f = _case(nimg, ny, nx, 52)
    u = inputs.uniform(53, nimg * ny * nx).reshape(nimg, ny, nx) * 3.0 - 1.0
    net = api.WarmNet(ctx, storage=api.F32, dilations=dil, seed=1)
    p = _params(9)
    net.params = p
    net.scale = 1.5
    out = torch.zeros((nimg, ny, nx), dtype=torch.float64, device="cuda")
    net.predict(_dev(k), _dev(f), out)
    torch.cuda.synchronize()
    x = _features(k, f, lambda a: a.astype(np.float32).astype(np.float64))
    ref = np.stack([oracle.warmnet_forward(p.astype(np.float64), x[i], C1, dil) for i in range(nimg)]) * 1.5
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-4 * np.max(np.abs(ref))
    loss, g = net.gradient(_dev(k), _dev(f), _dev(u))
    ref_loss, ref_g = oracle.warmnet_grad(p.astype(np.float64), x, u / 1.5, C1, dil)
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    assert np.max(np.abs(g - ref_g)) <= 1e-4 * np.max(np.abs(ref_g))


def test_gradient_bf16_other_dilations(ctx, oracle):
    """bf16 gradient at the widest dilation the inner layers' weight gradient takes (14); the next one is an error, and
    leaves the context usable."""
    from paper_2204_02064_gb300 import api
    nimg, ny, nx = 2, 40, 44
    k, f = _case(nimg, ny, nx, 54)
    u = inputs.uniform(55, nimg * ny * nx).reshape(nimg, ny, nx) * 2.0 - 1.0
    wide = api.WarmNet(ctx, storage=api.BF16, dilations=(1, 2, 15, 8), seed=1)
    with pytest.raises(api.PerksError):
        wide.gradient(_dev(k), _dev(f), _dev(u))
    wide.close()
    dil = (2, 14, 12, 16)
    net = api.WarmNet(ctx, storage=api.BF16, dilations=dil, seed=1)
    p = _params(10)
    net.params = p
    loss, g = net.gradient(_dev(k), _dev(f), _dev(u))
    x = _features(k, f)
    ref_loss, ref_g = oracle.warmnet_grad(p.astype(np.float64), x, u, C1, dil)
    assert loss == pytest.approx(ref_loss, rel=5e-2)
    assert np.linalg.norm(g - ref_g) <= 5e-2 * np.linalg.norm(ref_g)
