"""The per-brick MLP initializer on the device against the float64 oracle: the fused brick
render + L1 kernel (value and gradient), the network's forward and its weight gradients, and a
training run whose loss falls."""
import numpy as np
import pytest
import torch

from oracle import mlp as OM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gsct():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_01844_gb300 as g
    from paper_2604_01844_gb300 import build

    build.build()
    return g


def test_brick_loss_matches_oracle(gsct):
    B = gsct.binding
    rng = np.random.default_rng(0)
    nb = 6
    raw = rng.standard_normal((nb, 352)) * 0.6
    raw.reshape(nb, 32, 11)[:, :, 3:6] += 0.8
    target = rng.random((nb, 4096)) * 0.5
    raw32, tgt32 = raw.astype(np.float32), target.astype(np.float32)
    y = torch.zeros((nb, 384), device="cuda")
    y[:, :352] = torch.from_numpy(raw32).cuda()
    t = torch.from_numpy(tgt32).cuda()
    loss = torch.zeros(1, device="cuda")
    dy = torch.zeros((nb, 384), device="cuda")
    B.check(B.lib().gs_brick_loss(B.ptr(y), 384, B.ptr(t), nb, B.ptr(loss), B.ptr(dy), 384, None,
                                  torch.cuda.current_stream().cuda_stream), "brick_loss")
    torch.cuda.synchronize()
    rr = torch.from_numpy(raw32.astype(np.float64)).requires_grad_(True)
    want = OM.brick_l1(rr, torch.from_numpy(tgt32.astype(np.float64)))
    (g,) = torch.autograd.grad(want, rr)
    assert abs(float(loss) - float(want)) <= 1e-5 * abs(float(want))
    got = dy[:, :352].cpu().double()
    scale = float(g.abs().max())
    assert float((got - g).abs().max()) <= 2e-3 * scale, float((got - g).abs().max() / scale)


# boxes inside the region, clipped by it and covering it; thin and rotated Gaussians
@pytest.mark.parametrize("log_scale,spread,rot", [(-3.0, 0.0, 0.5), (0.0, 0.7, 1.0), (2.0, 0.2, 0.5),
                                                  (3.0, 0.0, 0.0)])
def test_brick_loss_boxes(gsct, log_scale, spread, rot):
    """The rendering within 1e-3 of its peak (the quadratic form's FP32 terms reach about 2e3,
    6 x 2^-24 of them is 7e-4 of the exponent) but for pairs at the cut (q within 0.01 of 9),
    and the gradient as in the test above."""
    B = gsct.binding
    rng = np.random.default_rng(5)
    nb = 3
    raw = rng.standard_normal((nb, 32, 11)).astype(np.float32)
    raw[..., 0:3] *= 2.0  # tanh towards the cell's corners
    raw[..., 3:6] = log_scale + spread * raw[..., 3:6]
    raw[..., 6:10] *= rot
    tgt = rng.random((nb, 4096)).astype(np.float32)
    y = torch.zeros((nb, 384), device="cuda")
    y[:, :352] = torch.from_numpy(raw.reshape(nb, 352)).cuda()
    loss, dy = torch.zeros(1, device="cuda"), torch.zeros((nb, 384), device="cuda")
    out = torch.full((nb, 4096), float("nan"), device="cuda")
    B.check(B.lib().gs_brick_loss(B.ptr(y), 384, B.ptr(torch.from_numpy(tgt).cuda()), nb,
                                  B.ptr(loss), B.ptr(dy), 384, B.ptr(out),
                                  torch.cuda.current_stream().cuda_stream), "brick_loss")
    torch.cuda.synchronize()
    rr = torch.from_numpy(raw.reshape(nb, 352).astype(np.float64)).requires_grad_(True)
    c, s, q, rho = (x.detach() for x in OM.decode(rr.reshape(nb, 32, 11)))
    ax = torch.arange(16, dtype=torch.float64) + 0.5
    zz, yy, xx = torch.meshgrid(ax, ax, ax, indexing="ij")
    d = torch.stack([xx, yy, zz], -1).reshape(1, 1, -1, 3) - c[:, :, None, :]
    u = torch.einsum("ngva,ngab->ngvb", d, OM.quat_rot(q)) / s[:, :, None, :]
    qf = (u * u).sum(-1)
    edge = torch.where((qf - 9).abs() < 0.01, rho[:, :, None] * np.exp(-4.49), 0 * qf).sum(1)
    want = torch.where(qf < 9, rho[:, :, None] * torch.exp(-0.5 * qf), 0 * qf).sum(1)
    err = (out.cpu().double() - want).abs()
    assert bool((err <= 1e-3 * want.max() + edge).all()), float(err.max())
    (g,) = torch.autograd.grad(OM.brick_l1(rr, torch.from_numpy(tgt.astype(np.float64))), rr)
    got = dy[:, :352].cpu().double()
    assert float((got - g).abs().max()) <= 2e-3 * float(g.abs().max())


# one row and column, parts of a 32-column group, rows that eight CTAs share unevenly
@pytest.mark.parametrize("rows,cols", [(1, 1), (7, 33), (1000, 96), (4099, 384)])
def test_colsum(gsct, rows, cols):
    """At most rows / 256 additions per thread, then 5 + 3 levels: each rounds to 2^-24 of the sum
    of magnitudes."""
    B = gsct.binding
    x = torch.from_numpy(np.random.default_rng(rows).standard_normal((rows, cols)).astype(np.float32))
    out = torch.full((cols,), float("nan"), device="cuda")
    B.check(B.lib().gs_colsum(B.ptr(x.cuda()), rows, cols, B.ptr(out),
                              torch.cuda.current_stream().cuda_stream), "colsum")
    tol = (rows / 256 + 9 + 8) * 2.0 ** -24 * x.double().abs().sum(0) + 1e-30
    assert bool(((out.cpu().double() - x.double().sum(0)).abs() <= tol).all())


def _mlp_ref(m):
    Ws = [w.detach().cpu().double() for w in m.W]
    bs = [b.detach().cpu().double() for b in m.b]
    return Ws, bs


def test_mlp_forward_and_weight_gradients(gsct):
    from paper_2604_01844_gb300.mlp import BrickMLP

    m = BrickMLP(seed=3)
    rng = np.random.default_rng(1)
    M = 256
    x = torch.from_numpy(rng.random((M, 4096)).astype(np.float32))
    x16 = x.to(torch.bfloat16).cuda()
    y = m.forward(x16)
    Ws, bs = _mlp_ref(m)
    Ws = [w.requires_grad_(True) for w in Ws]
    bs = [b.requires_grad_(True) for b in bs]
    yref = OM.mlp_forward(x.double(), Ws, bs)
    got = y.cpu().double()
    assert float((got - yref).abs().max()) <= 2e-2 * float(yref.abs().max()) + 1e-3
    gy = torch.from_numpy(rng.standard_normal((M, 384)).astype(np.float32))
    gy[:, 352:] = 0
    m.backward(gy.cuda())
    (yref * gy.double()).sum().backward()
    torch.cuda.synchronize()
    for gw, ref in zip(m.grads, [w.grad for w in Ws] + [b.grad for b in bs]):
        g = gw.cpu().double()
        scale = float(ref.abs().max()) + 1e-12
        assert float((g - ref).abs().max()) <= 5e-2 * scale, float((g - ref).abs().max() / scale)


def test_mlp_training_reduces_brick_loss(gsct):
    """Bricks of smooth random blobs; 60 Adam steps roughly halve the render L1."""
    from paper_2604_01844_gb300.mlp import BrickMLP

    rng = np.random.default_rng(2)
    M = 256
    ax = np.arange(16) + 0.5
    zz, yy, xx = np.meshgrid(ax, ax, ax, indexing="ij")
    tgt = np.zeros((M, 4096), dtype=np.float32)
    for b in range(M):
        for _ in range(3):
            c = rng.uniform(3, 13, 3)
            s = rng.uniform(1.5, 4)
            tgt[b] += (rng.uniform(0.3, 1.0) * np.exp(-((xx - c[0]) ** 2 + (yy - c[1]) ** 2 +
                                                       (zz - c[2]) ** 2) / (2 * s * s))).ravel()
    noisy = tgt + 0.05 * rng.standard_normal(tgt.shape).astype(np.float32)
    x16 = torch.from_numpy(noisy).to(torch.bfloat16).cuda()
    t = torch.from_numpy(tgt).cuda()
    m = BrickMLP(seed=4)
    losses = []
    for it in range(60):
        loss = torch.zeros(1, device="cuda")
        m.train_step(x16, t, loss, lr=1e-3)
        losses.append(float(loss))
    assert int(m.err.item()) == 0
    assert losses[-1] < 0.6 * losses[0], losses[::10]


# ------------------------------------------------------------------------------------------
# The network entry points of the C ABI (gs_mlp_train_step, gs_mlp_infer) against the
# sequence of primitive library calls they stand for
# ------------------------------------------------------------------------------------------
def _primitive_train_step(B, m, x16, target, loss, lr, M):
    """Forward GEMMs -> gs_brick_loss -> transposes and backward GEMMs -> per-tensor Adam ->
    step increment, each a separate library call on the network's tensors."""
    L = B.lib()
    s = torch.cuda.current_stream().cuda_stream
    err = m.err

    def gemm(a, b, Mr, N, K, bias=None, relu=False, c32=None, c16=None):
        B.check(L.gs_gemm_bf16(B.ptr(a), B.ptr(b), Mr, N, K, B.ptr(bias), 1 if relu else 0,
                               B.ptr(c32), B.ptr(c16), N, B.ptr(err), s), "gemm")

    h = []
    a, K = x16, 4096
    for li in range(3):
        hb = torch.empty((M, 256), dtype=torch.bfloat16, device="cuda")
        gemm(a, m.W16[li], M, 256, K, bias=m.b[li], relu=True, c16=hb)
        h.append(hb)
        a, K = hb, 256
    y = torch.empty((M, 384), device="cuda")
    gemm(a, m.W16[3], M, 384, 256, bias=m.b[3], c32=y)
    dy = torch.zeros((M, 384), device="cuda")
    B.check(L.gs_brick_loss(B.ptr(y), 384, B.ptr(target), M, B.ptr(loss), B.ptr(dy), 384, None,
                            s), "brick_loss")
    acts = [x16] + h
    g32, width = dy, 384
    g16 = torch.empty((M, 384), dtype=torch.bfloat16, device="cuda")
    B.check(L.gs_f32_to_bf16(B.ptr(g32), B.ptr(g16), g32.numel(), s), "f32_to_bf16")
    for li in (3, 2, 1, 0):
        k_in = acts[li].shape[1]
        B.check(L.gs_colsum(B.ptr(g32), M, width, B.ptr(m.grads[4 + li]), s), "colsum")
        gT = torch.empty((width, M), dtype=torch.bfloat16, device="cuda")
        aT = torch.empty((k_in, M), dtype=torch.bfloat16, device="cuda")
        B.check(L.gs_transpose_bf16(B.ptr(g16), M, width, B.ptr(gT), s), "transpose")
        B.check(L.gs_transpose_bf16(B.ptr(acts[li]), M, k_in, B.ptr(aT), s), "transpose")
        gemm(gT, aT, width, k_in, M, c32=m.grads[li])
        if li == 0:
            break
        WT = torch.empty((k_in, width), dtype=torch.bfloat16, device="cuda")
        B.check(L.gs_transpose_bf16(B.ptr(m.W16[li]), width, k_in, B.ptr(WT), s), "transpose")
        gp = torch.empty((M, k_in), device="cuda")
        gemm(g16, WT, M, k_in, width, c32=gp)
        g16p = torch.empty((M, k_in), dtype=torch.bfloat16, device="cuda")
        B.check(L.gs_relu_mask_bf16(B.ptr(gp), B.ptr(h[li - 1]), gp.numel(), B.ptr(g16p), s),
                "relu_mask")
        g32, g16, width = gp, g16p, k_in
    # per-tensor Adam on views of the flat moments
    off = 0
    views = []
    for p in m.params:
        views.append((m.flat_m[off:off + p.numel()], m.flat_v[off:off + p.numel()]))
        off += p.numel()
    for i, (p, g, (mm, vv)) in enumerate(zip(m.params, m.grads, views)):
        B.check(L.gs_adam_flat(B.ptr(p), B.ptr(mm), B.ptr(vv), B.ptr(g), p.numel(),
                               B.ptr(m.step_count), lr, 0.9, 0.999, 1e-8,
                               B.ptr(m.W16[i]) if i < 4 else None, s), "adam_flat")
    B.check(L.gs_step_incr(B.ptr(m.step_count), s), "step_incr")


def test_exported_train_step_equals_primitive_sequence(gsct):
    """Three steps of gs_mlp_train_step and of the primitive call sequence from the same
    start: parameters, bf16 weights, Adam moments and gradients equal bit for bit."""
    from paper_2604_01844_gb300.mlp import BrickMLP

    B = gsct.binding
    rng = np.random.default_rng(9)
    M = 256
    x = torch.from_numpy(rng.random((3, M, 4096)).astype(np.float32))
    t = torch.from_numpy((rng.random((3, M, 4096)) * 0.4).astype(np.float32)).cuda()
    a, b = BrickMLP(seed=5), BrickMLP(seed=5)
    la, lb = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    for k in range(3):
        x16 = x[k].to(torch.bfloat16).cuda()
        a.train_step(x16, t[k], la, lr=1e-3)
        _primitive_train_step(B, b, x16, t[k], lb, 1e-3, M)
    torch.cuda.synchronize()
    assert int(a.err.item()) == 0 and int(b.err.item()) == 0
    assert int(a.step_count.item()) == 3 == int(b.step_count.item())
    for name, u, v in (("params", a.flat, b.flat), ("bf16 weights", a.flat16, b.flat16),
                       ("m", a.flat_m, b.flat_m), ("v", a.flat_v, b.flat_v),
                       ("grad", a.flat_grad, b.flat_grad)):
        assert torch.equal(u, v), (name, float((u.float() - v.float()).abs().max()))
    # the loss is summed over the bricks with float atomics: equal up to their order
    assert abs(float(la) - float(lb)) <= 1e-6 * abs(float(lb))


def test_train_step_large_batch_equals_primitive_sequence(gsct):
    """A batch whose GEMMs fill the SMs (128 x 256 tiles in every operand form) against the
    primitive calls, which transpose their operands in memory: the same products in the same
    order, so the gradients are equal bit for bit."""
    from paper_2604_01844_gb300.mlp import BrickMLP

    B = gsct.binding
    M = 19456
    g = torch.Generator(device="cuda").manual_seed(3)
    x16 = torch.rand(M, 4096, device="cuda", generator=g).to(torch.bfloat16)
    t = 0.4 * torch.rand(M, 4096, device="cuda", generator=g)
    a, b = BrickMLP(seed=5), BrickMLP(seed=5)
    la, lb = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    a.train_step(x16, t, la, lr=1e-3)
    _primitive_train_step(B, b, x16, t, lb, 1e-3, M)
    torch.cuda.synchronize()
    assert int(a.err.item()) == 0 and int(b.err.item()) == 0
    assert torch.equal(a.flat_grad, b.flat_grad)


def test_infer_equals_forward_and_decode(gsct):
    from paper_2604_01844_gb300.mlp import BrickMLP

    B = gsct.binding
    rng = np.random.default_rng(10)
    M = 128
    m = BrickMLP(seed=6)
    x16 = torch.from_numpy(rng.random((M, 4096)).astype(np.float32)).to(torch.bfloat16).cuda()
    geo = torch.from_numpy(np.stack([rng.uniform(-1, 1, M), rng.uniform(-1, 1, M),
                                     rng.uniform(-1, 1, M), np.full(M, 2 / 256)],
                                    1).astype(np.float32)).cuda()
    got = m.infer_gaussians(x16, geo, 1.7)
    y = m.forward(x16)
    want = [torch.empty((M * 32, 4), device="cuda") for _ in range(3)]
    B.check(B.lib().gs_brick_decode(B.ptr(y), 384, B.ptr(geo), M, 1.7, *[B.ptr(w) for w in want],
                                    torch.cuda.current_stream().cuda_stream), "decode")
    torch.cuda.synchronize()
    for u, v in zip(got, want):
        assert torch.equal(u, v)


def test_colsum_of_the_longest_column(gsct):
    """2^31 - 1 rows, the most an int holds: every row is read, and none beyond the last."""
    B = gsct.binding
    x = torch.zeros((2 ** 31 - 1, 1), device="cuda")
    x[0], x[2 ** 30], x[2 ** 31 - 9:] = 1.0, 2.0, 4.0
    out = torch.full((1,), -1.0, device="cuda")
    B.check(B.lib().gs_colsum(B.ptr(x), x.shape[0], 1, B.ptr(out),
                              torch.cuda.current_stream().cuda_stream), "colsum")
    assert float(out) == 1.0 + 2.0 + 4.0 * 8


# the input gradient's tiles of 64 columns (2432 and 4736 bricks), 128 (4864) and 256 (19456); the
# weight gradients, of at most 32 x 2 or 3 tiles of 128, take 64 whatever the batch
@pytest.mark.parametrize("M", [2432, 4736, 4864, 19456])
def test_train_step_tiles_equal_primitive_sequence(gsct, M):
    """Every tile of the stored-operand GEMMs against the primitive calls on transposed copies: the
    same products in the same order, so the gradients are equal bit for bit."""
    from paper_2604_01844_gb300.mlp import BrickMLP

    B = gsct.binding
    g = torch.Generator(device="cuda").manual_seed(M)
    x16 = torch.rand(M, 4096, device="cuda", generator=g).to(torch.bfloat16)
    t = 0.4 * torch.rand(M, 4096, device="cuda", generator=g)
    a, b = BrickMLP(seed=5), BrickMLP(seed=5)
    la, lb = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    a.train_step(x16, t, la, lr=1e-3)
    _primitive_train_step(B, b, x16, t, lb, 1e-3, M)
    assert int(a.err.item()) == 0 and int(b.err.item()) == 0
    assert torch.equal(a.flat_grad, b.flat_grad) and bool((a.flat_grad != 0).any())


# the narrowest matrix that takes a thread per column (128 columns an SM) and one column less
@pytest.mark.parametrize("less", [0, 1])
@pytest.mark.parametrize("rows", [1, 9, 500])
def test_colsum_of_wide_matrices(gsct, rows, less):
    """Kahan's sum is within 2 x 2^-24 of the sum of magnitudes (and 500 additions' second order), the
    tree of the other route within (rows / 256 + 17) x 2^-24."""
    B = gsct.binding
    cols = 128 * torch.cuda.get_device_properties(0).multi_processor_count - less
    x = torch.randn(rows, cols, device="cuda", generator=torch.Generator("cuda").manual_seed(rows))
    x[0, 7] = float("inf")
    out = torch.full((cols,), float("nan"), device="cuda")
    B.check(B.lib().gs_colsum(B.ptr(x), rows, cols, B.ptr(out),
                              torch.cuda.current_stream().cuda_stream), "colsum")
    tol = (3 if less == 0 else rows / 256 + 17) * 2.0 ** -24 * x.double().abs().sum(0) + 1e-30
    assert float(out[7]) == float("inf")
    out[7], x[0, 7], tol[7] = 0.0, 0.0, float("inf")
    assert bool(((out.double() - x.double().sum(0)).abs() <= tol).all())
