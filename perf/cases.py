"""The work that users of this library have it do, as measurable cases.

listed() holds fixed cases, draw() more of the same ranges; prepare() makes
what a program has in hand before the call, run() is one pass through the
public entry points, work() what a pass cannot do without, and exact() the
result in 64-bit floating point by plain torch.

Families (the "kind" of a case):
  stencil  set_field, a run of time steps, get_field on one domain;
  batch    the same for many uneven 2-D domains in one launch;
  cg       a sparse SPD system solved to a relative residual of 1e-10;
  poisson  batched variable-coefficient Poisson problems solved by CG;
  predict  the warm-start network's first guess for a batch of problems;
  grad     loss and parameter gradient of one training minibatch.
Every object is used with its default plan, as a program does that does not
tune by hand.
"""
import functools
import math

import numpy as np
import torch

from paper_2204_02064_gb300 import api, inputs

TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # The smallest domain of the benchmark: latency of a time step and of the call.
        dict(name="2d5pt-f64-256", kind="stencil", shape="2d5pt", dtype="f64", nx=256, ny=256, nz=1, steps=100),
        # A 2-D domain of the stencil suite's size, larger than the on-chip memory in use.
        dict(name="2d5pt-f32-3072", kind="stencil", shape="2d5pt", dtype="f32", nx=3072, ny=3072, nz=1, steps=100),
        # A 3-D domain that fits on chip for all steps.
        dict(name="3d7pt-f32-192", kind="stencil", shape="3d7pt", dtype="f32", nx=192, ny=192, nz=192, steps=100),
        # The headline domain, in double precision.
        dict(name="3d7pt-f64-384", kind="stencil", shape="3d7pt", dtype="f64", nx=384, ny=384, nz=384, steps=40),
        # The same domain with 16-bit storage.
        dict(name="3d7pt-bf16-384", kind="stencil", shape="3d7pt", dtype="bf16", nx=384, ny=384, nz=384, steps=40),
        # A ragged box: extents that no vector width divides, 27 points.
        dict(name="3d27pt-f32-ragged", kind="stencil", shape="3d27pt", dtype="f32", nx=251, ny=246, nz=233, steps=20),
        # Many uneven 2-D domains advanced together (half 9-point, half 25-point boxes).
        dict(name="batch-f32-64", kind="batch", dtype="f32", count=64, lo=128, hi=2048, seed=2, steps=40),
        # A million unknowns with scattered columns, double precision.
        dict(name="cg-f64-1M", kind="cg", matrix="random", mode="f64", nx=1 << 20, ny=1),
        # One implicit step of a diffusion problem on a 2-D grid: mixed precision with refinement.
        dict(name="cg-ir-grid-701x613", kind="cg", matrix="grid", mode="ir", nx=701, ny=613),
        # Large Poisson problems given a bounded number of iterations each.
        dict(name="poisson-512-x64", kind="poisson", nx=512, ny=512, count=64, iters=24),
        # First guesses for a whole batch of Poisson problems (network on the 8x coarsened grid).
        dict(name="predict-bf16-256", kind="predict", storage="bf16", side=512, count=256, pool=8),
        # One training minibatch of that network.
        dict(name="grad-bf16-16", kind="grad", storage="bf16", side=512, count=16, pool=8),
    ]


# ------------------------------------------------------------------ drawing

#: Cell-point updates of the largest listed stencil (384^3 cells, 40 steps, 7 points).
MOST_UPDATES = 384 ** 3 * 40 * 7


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_stencil(rng):
    shape = rng.choice(["2d5pt", "2d5pt", "2ds9pt", "2d9pt", "2d25pt", "3d7pt", "3d7pt", "3d13pt", "3d27pt", "poisson"])
    dtype = rng.choice(["f64", "f32", "bf16"])
    npts = len(inputs.shape_offsets(shape))
    if inputs.SHAPES[shape][1] == 2:
        nx, ny, nz = _log_int(rng, 64, 4096), _log_int(rng, 64, 4096), 1
    else:
        nx, ny, nz = (_log_int(rng, 32, 384) for _ in range(3))
    # half of the domains have a row length that 16-byte vectors divide; bf16 needs it
    if dtype == "bf16" or rng.random() < 0.5:
        nx = max(8, nx // 8 * 8)
    steps = _log_int(rng, 10, 200)
    steps = max(4, min(steps, MOST_UPDATES // (nx * ny * nz * npts)))
    return dict(kind="stencil", shape=shape, dtype=dtype, nx=nx, ny=ny, nz=nz, steps=steps)


def _draw_batch(rng):
    return dict(kind="batch", dtype=rng.choice(["f32", "f32", "f64"]), count=rng.randint(8, 48), lo=128,
                hi=_log_int(rng, 256, 1600) // 8 * 8, seed=rng.randint(0, 10 ** 6), steps=_log_int(rng, 5, 40))


def _draw_cg(rng):
    n = _log_int(rng, 2000, 1 << 20)
    if rng.random() < 0.5:
        return dict(kind="cg", matrix="random", mode=rng.choice(["f64", "ir"]), nx=n, ny=1)
    nx = max(20, int(math.sqrt(n) * rng.uniform(0.7, 1.4)))
    return dict(kind="cg", matrix="grid", mode=rng.choice(["f64", "ir"]), nx=nx, ny=max(20, n // nx))


def _draw_poisson(rng):
    nx, ny = _log_int(rng, 48, 512), _log_int(rng, 48, 512)
    cells = _log_int(rng, 1 << 18, 1 << 24)
    # small grids are solved to the tolerance (iters = 0), large ones given a budget
    iters = 0 if max(nx, ny) <= 128 else rng.randint(12, 24)
    if iters == 0:
        cells = min(cells, 1 << 20)
    return dict(kind="poisson", nx=nx, ny=ny, count=max(1, min(256, cells // (nx * ny))), iters=iters)


def _draw_net(rng, kind):
    pool = rng.choice([1, 4, 8, 8, 16])
    side = pool * max(16 // pool, _log_int(rng, 96, 512) // pool)
    cells = _log_int(rng, 1 << 18, 1 << 26) if kind == "predict" else _log_int(rng, 1 << 17, 1 << 22)
    cells = min(cells, (1 << 21 if kind == "predict" else 1 << 17) * pool * pool)  # bounded work at pool 1
    return dict(kind=kind, storage=rng.choice(["bf16", "bf16", "f32"]), side=side,
                count=max(1, min(256, cells // (side * side))), pool=pool)


def draw(rng):
    u = rng.random()
    if u < 0.5:
        return _draw_stencil(rng)
    if u < 0.6:
        return _draw_batch(rng)
    if u < 0.75:
        return _draw_cg(rng)
    if u < 0.85:
        return _draw_poisson(rng)
    return _draw_net(rng, "predict" if u < 0.93 else "grad")


# ------------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=None)
def _context():
    return api.Context(0)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rand(shape, seed, dtype=torch.float64):
    return torch.rand(shape, generator=_gen(seed), dtype=torch.float64, device="cuda").to(dtype)


def _field_shape(case):
    return (case["ny"], case["nx"]) if case["nz"] == 1 else (case["nz"], case["ny"], case["nx"])


def _batch_domains(case):
    return inputs.batch_domains(case["count"], seed=case["seed"], lo=case["lo"], hi=case["hi"])


def _csr(case, seed):
    """(rowptr int32, col int32, val float64, b) on the GPU."""
    g = _gen(seed)
    if case["matrix"] == "random":
        # every row draws 3..31 partners; A_ij = A_ji in [-1, 0); diagonal 1.05 x the row's absolute sum
        n = case["nx"]
        k = torch.randint(3, 32, (n,), generator=g, device="cuda")
        rows = torch.repeat_interleave(torch.arange(n, device="cuda"), k)
        cols = torch.randint(0, n - 1, (rows.numel(),), generator=g, device="cuda")
        cols += (cols >= rows)
        key = torch.unique(torch.minimum(rows, cols) * n + torch.maximum(rows, cols))
        i, j = key // n, key % n
        v = torch.rand(key.numel(), generator=g, dtype=torch.float64, device="cuda") - 1.0
        factor = 1.05
    else:
        # (I + dt L) of one implicit diffusion step with varying conductivity on an ny x nx grid
        nx, ny = case["nx"], case["ny"]
        n = nx * ny
        at = torch.arange(n, device="cuda").reshape(ny, nx)
        i = torch.cat([at[:, :-1].reshape(-1), at[:-1].reshape(-1)])
        j = torch.cat([at[:, 1:].reshape(-1), at[1:].reshape(-1)])
        v = -25.0 * (0.5 + torch.rand(i.numel(), generator=g, dtype=torch.float64, device="cuda"))
        factor = 1.0
    absrow = torch.zeros(n, dtype=torch.float64, device="cuda")
    r, c, a = torch.cat([i, j]), torch.cat([j, i]), torch.cat([v, v])
    order = torch.argsort(r * n + c)
    r, c, a = r[order], c[order], a[order]
    first = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    first[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    # row sums as differences of one running sum would lose digits: a segmented sum instead
    absrow = torch.segment_reduce(a.abs(), "sum", offsets=first)
    diag = factor * absrow + (1.0 if case["matrix"] == "grid" else 0.0)
    at = torch.arange(n, device="cuda")
    r, c, a = torch.cat([r, at]), torch.cat([c, at]), torch.cat([a, diag])
    order = torch.argsort(r * n + c)
    first = first + torch.arange(n + 1, device="cuda")
    b = 2.0 * torch.rand(n, generator=g, dtype=torch.float64, device="cuda") - 1.0
    return first.int(), c[order].int(), a[order].contiguous(), b


def _poisson_inputs(ny, nx, count, seed):
    k, f = inputs.poisson_problems_device(max(nx, ny), count, seed=seed)
    return k[:, :ny, :nx].contiguous(), f[:, :ny, :nx].contiguous()


def _net_weights(seed):
    """Weights of a network as a program loads them: He-scaled normals, small biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for cin, cout in ((2, 32), (32, 32), (32, 32), (32, 1)):
        parts.append(rng.standard_normal(cout * cin * 9) * math.sqrt(2.0 / (9 * cin)))
        parts.append(0.1 * rng.standard_normal(cout))
    return np.concatenate(parts).astype(np.float32)


def _net_inputs(case, seed):
    k, f = _poisson_inputs(case["side"], case["side"], case["count"], seed)
    u = None
    if case["kind"] == "grad":  # smooth targets
        c = torch.randn((case["count"], 1, 8, 8), generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
        u = 100.0 * torch.nn.functional.interpolate(c, size=(case["side"],) * 2, mode="bilinear", align_corners=False)
        u = u[:, 0].contiguous()
    return k, f, u


NET_SCALE = 100.0


def prepare(case, seed):
    ctx = _context()
    kind = case["kind"]
    if kind == "stencil":
        shape = _field_shape(case)
        st = api.Stencil(ctx, shape, inputs.shape_offsets(case["shape"]), inputs.workload_weights(case["shape"]),
                         dtype=case["dtype"])
        src = _rand(shape, seed, TORCH[case["dtype"]])
        return dict(case=case, st=st, src=src, out=torch.empty_like(src))
    if kind == "batch":
        doms = _batch_domains(case)
        src = [_rand(d["shape"], seed + i, TORCH[case["dtype"]]) for i, d in enumerate(doms)]
        return dict(case=case, batch=api.Batch(ctx, doms, dtype=case["dtype"]), src=src,
                    out=[torch.empty_like(s) for s in src])
    if kind == "cg":
        rowptr, col, val, b = _csr(case, seed)
        return dict(case=case, op=api.CsrOperator(ctx, rowptr, col, val), b=b, x=torch.zeros_like(b))
    if kind == "poisson":
        k, f = _poisson_inputs(case["ny"], case["nx"], case["count"], seed)
        return dict(case=case, op=api.Poisson(ctx, k), b=f, x=torch.zeros_like(f))
    k, f, u = _net_inputs(case, seed)
    net = api.WarmNet(ctx, storage=api.DTYPES[case["storage"]], pool=case["pool"])
    net.params = _net_weights(seed)
    net.scale = NET_SCALE
    return dict(case=case, net=net, k=k, f=f, u=torch.empty_like(f) if u is None else u)


# --------------------------------------------------------------------- pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "stencil":
        st = state["st"]
        st.set_field(state["src"])
        st.run(case["steps"])
        return st.get_field(state["out"])
    if kind == "batch":
        batch = state["batch"]
        for i, s in enumerate(state["src"]):
            batch.set_field(i, s)
        batch.run(case["steps"])
        for i, o in enumerate(state["out"]):
            batch.get_field(i, o)
        return state["out"]
    if kind == "cg":
        x = state["x"].zero_()
        state["op"].solve(state["b"], x, rtol=1e-10, mode=api.CG_FP64 if case["mode"] == "f64" else api.CG_FP32_IR)
        return x
    if kind == "poisson":
        x = state["x"].zero_()
        if case["iters"]:
            state["op"].solve(state["b"], x, rtol=1e-8, max_iter=case["iters"], stats=False)
        else:
            state["op"].solve(state["b"], x, rtol=1e-10, stats=False)
        return x
    if kind == "predict":
        state["net"].predict(state["k"], state["f"], state["u"])
        return state["u"]
    loss, grad = state["net"].gradient(state["k"], state["f"], state["u"])
    return dict(loss=np.float32(loss), grad=grad)


def work(case):
    kind = case["kind"]
    if kind == "stencil":
        cells = case["nx"] * case["ny"] * case["nz"]
        npts = len(inputs.shape_offsets(case["shape"]))
        return dict(bytes=2.0 * cells * BYTES[case["dtype"]], flops=2.0 * npts * cells * case["steps"])
    if kind == "batch":
        doms = _batch_domains(case)
        cells = [d["shape"][0] * d["shape"][1] for d in doms]
        return dict(bytes=2.0 * sum(cells) * BYTES[case["dtype"]],
                    flops=2.0 * case["steps"] * sum(c * len(d["weights"]) for c, d in zip(cells, doms)))
    if kind == "cg":
        n = case["nx"] * case["ny"]
        nnz, iters = (35 * n, 50) if case["matrix"] == "random" else (5 * n, 150)
        return dict(bytes=12.0 * nnz + 20.0 * n, flops=iters * (2.0 * nnz + 10.0 * n))
    if kind == "poisson":
        n = case["nx"] * case["ny"] * case["count"]
        iters = case["iters"] or 10 * max(case["nx"], case["ny"])
        return dict(bytes=24.0 * n, flops=20.0 * n * iters)
    fine = case["side"] ** 2 * case["count"]
    macs = 9 * (2 * 32 + 2 * 32 * 32 + 32) * (fine // case["pool"] ** 2)
    return dict(bytes=24.0 * fine, flops=2.0 * macs * (1 if kind == "predict" else 3))


# ------------------------------------------------------------- 64-bit result

def _exact_stencil(src, offsets, weights, steps):
    v = src.double()
    if v.dim() == 2:
        v = v[None]
    r = max(abs(c) for o in offsets for c in o)
    nz, ny, nx = v.shape
    rz = r if any(o[2] for o in offsets) else 0
    pad = torch.zeros((nz + 2 * rz, ny + 2 * r, nx + 2 * r), dtype=torch.float64, device=v.device)
    for _ in range(steps):
        pad[rz:rz + nz, r:r + ny, r:r + nx] = v
        v = torch.zeros_like(v)
        for (dx, dy, dz), w in zip(offsets, weights):
            v.add_(pad[rz + dz:rz + dz + nz, r + dy:r + dy + ny, r + dx:r + dx + nx], alpha=float(w))
    return v.reshape(src.shape)


def _exact_cg(apply, b, dot, iters=None, rtol=1e-14, most=20000):
    """Conjugate gradient from zero: `iters` iterations, or to rtol."""
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), dot(r, r)
    stop = rtol * rtol * rr
    for it in range(iters if iters is not None else most):
        if iters is None and it % 10 == 0 and bool((rr <= stop).all()):
            break
        q = apply(p)
        pq = dot(p, q)
        alpha = torch.where(pq > 0, rr / pq, torch.zeros_like(rr))
        x += alpha * p
        r -= alpha * q
        rn = dot(r, r)
        p = r + torch.where(rr > 0, rn / rr, torch.zeros_like(rr)) * p
        rr = rn
    return x


def _poisson_apply(k):
    fx = torch.cat([k[:, :, :1], 2 * k[:, :, :-1] * k[:, :, 1:] / (k[:, :, :-1] + k[:, :, 1:]), k[:, :, -1:]], 2)
    fy = torch.cat([k[:, :1], 2 * k[:, :-1] * k[:, 1:] / (k[:, :-1] + k[:, 1:]), k[:, -1:]], 1)
    dg = fx[:, :, :-1] + fx[:, :, 1:] + fy[:, :-1] + fy[:, 1:]

    def apply(v):
        q = dg * v
        q[:, :, 1:] -= fx[:, :, 1:-1] * v[:, :, :-1]
        q[:, :, :-1] -= fx[:, :, 1:-1] * v[:, :, 1:]
        q[:, 1:] -= fy[:, 1:-1] * v[:, :-1]
        q[:, :-1] -= fy[:, 1:-1] * v[:, 1:]
        return q
    return apply


def _exact_net(x, w, dil=(1, 2, 4, 8)):
    """The network's output for the inputs x (count, 2, H, W) with flat weights w, as sums over the nine taps."""
    at = 0
    for layer, (cin, cout) in enumerate(((2, 32), (32, 32), (32, 32), (32, 1))):
        wl = w[at:at + cout * cin * 9].reshape(cout, cin, 9)
        at += cout * cin * 9
        d, (h, wd) = dil[layer], x.shape[-2:]
        pad = torch.nn.functional.pad(x, (d, d, d, d))
        y = w[at:at + cout].reshape(1, cout, 1, 1).expand(x.shape[0], cout, h, wd)
        at += cout
        for tap in range(9):
            ky, kx = tap // 3 * d, tap % 3 * d
            y = y + torch.einsum("oc,bchw->bohw", wl[:, :, tap], pad[:, :, ky:ky + h, kx:kx + wd])
        x = torch.relu(y) if layer < 3 else y
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "stencil":
        src = _rand(_field_shape(case), seed, TORCH[case["dtype"]])
        return _exact_stencil(src, inputs.shape_offsets(case["shape"]), inputs.workload_weights(case["shape"]),
                              case["steps"])
    if kind == "batch":
        return [_exact_stencil(_rand(d["shape"], seed + i, TORCH[case["dtype"]]), d["offsets"], d["weights"],
                               case["steps"]) for i, d in enumerate(_batch_domains(case))]
    if kind == "cg":
        rowptr, col, val, b = _csr(case, seed)
        a = torch.sparse_csr_tensor(rowptr.long(), col.long(), val, size=(b.numel(), b.numel()))
        return _exact_cg(lambda v: torch.mv(a, v), b, torch.dot)
    if kind == "poisson":
        k, f = _poisson_inputs(case["ny"], case["nx"], case["count"], seed)
        return _exact_cg(_poisson_apply(k), f, lambda u, v: (u * v).sum((1, 2), keepdim=True),
                         iters=case["iters"] or None)
    k, f, u = _net_inputs(case, seed)
    w = torch.from_numpy(_net_weights(seed)).cuda().double()
    pooled = lambda v: torch.nn.functional.avg_pool2d(v[:, None], case["pool"])  # noqa: E731
    if kind == "predict":
        out = []
        per = max(1, (1 << 20) * case["pool"] ** 2 // case["side"] ** 2)  # images at a time: bounded memory
        for i in range(0, case["count"], per):
            y = _exact_net(torch.cat([pooled(k[i:i + per].log()), pooled(f[i:i + per])], 1), w)
            out.append(torch.nn.functional.interpolate(y, scale_factor=case["pool"], mode="bilinear",
                                                       align_corners=False)[:, 0])
        return NET_SCALE * torch.cat(out)
    w.requires_grad_(True)
    y = _exact_net(torch.cat([pooled(k.log()), pooled(f)], 1), w)
    loss = (y - pooled(u) / NET_SCALE).square().mean()
    loss.backward()
    return dict(loss=loss.detach().reshape(()), grad=w.grad)
