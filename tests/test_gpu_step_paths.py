"""Branches of the whole step against fp64 references of the same step (noise by the sequential paths, which have their own
tests), at the sizes where a tile, a remainder or a range ends."""
import math

import numpy as np
import pytest
import torch

from util import TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dp():
    import paper_2009_03106_b200 as pkg
    pkg.load_library()
    return pkg


def _spread(B, scale=4.0):
    """Factors of the examples' gradients, from 1 / scale to scale, in mixed order: norms on both sides of the threshold."""
    f = torch.exp(torch.linspace(-1.0, 1.0, B, device="cuda") * math.log(scale))
    gen = torch.Generator(device="cuda"); gen.manual_seed(B)
    return f[torch.randperm(B, generator=gen, device="cuda")]


def _rel(got, ref):
    got, ref = got.double(), ref.double()
    return ((got - ref).norm() / ref.norm()).item()


# ---------------------------------------------------------------------------
# element-wise layers: clipped sums from the stored per-example gradients, against fp64 and against the second pass over the
# inputs (taken when the workspace lacks the room, and by layers of fewer than 8 positions)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,T,widths", [(1, 8, (1,)), (7, 9, (33, 4, 130)), (65, 40, (512, 31)), (129, 8, (64,) * 17)])
def test_elementwise_grads_from_stored_rows(dp, dtype, B, T, widths):
    gen = torch.Generator(device="cuda"); gen.manual_seed(B + T)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    C, sigma, seed = 1.0, 0.5, 11
    layers = []
    for k, d in enumerate(widths):
        t = 3 if k == 2 else T
        H = torch.randn(B, t, d, generator=gen, device="cuda").to(td)
        Z = (torch.randn(B, t, d, generator=gen, device="cuda") * (2.0 / (t * sum(widths))) ** 0.5).to(td)
        layers.append(dp.ModelLayer(dp.DPCLIP_KIND_ELEMENTWISE, H, Z, k % 3 != 1))
    full, small = dp.ModelPlan(layers), dp.ModelPlan(layers)
    small.workspace = small.workspace[:256]
    grads = [((y.A.double() * y.Zbar.double()).sum(1), y.Zbar.double().sum(1) if y.has_bias else None) for y in layers]
    norms = sum(g.pow(2).sum(1) + (0 if s is None else s.pow(2).sum(1)) for g, s in grads).sqrt()
    clip = (C / norms).clamp(max=1.0)
    for sg in (0.0, sigma):
        for plan in (full, small):
            plan.run(C, sg, seed)
        torch.cuda.synchronize()
        assert dp.dpclip_read_status(full.workspace) == 0
        for l, (g, s) in enumerate(grads):
            for out, other, ref in ((full.gW[l], small.gW[l], g), (full.gb[l], small.gb[l], s)):
                if ref is None:
                    continue
                if sg == 0.0:
                    assert _rel(out, (clip[:, None] * ref).sum(0)) <= TOL["f32"]["grad"]      # sums in fp32 of exact inputs
                else:
                    # the same draws on either path: what differs is the sum below them
                    assert (out - other).abs().max().item() <= 1e-5 * max(1.0, out.abs().max().item())
    assert ((full.norms.double() - norms).abs() / norms).max().item() <= TOL["f32"]["norm"]


def test_elementwise_grads_of_an_example_that_overflows(dp):
    # finite inputs, a per-example sum beyond fp32: infinite norm, factor 0, nothing of it in the sum
    B, T, d = 5, 16, 40
    H = torch.randn(B, T, d, device="cuda"); Z = torch.randn(B, T, d, device="cuda") * 1e-3
    H[2, :, 7] = 3e30; Z[2, :, 7] = 1e20
    plan = dp.ModelPlan([dp.ModelLayer(dp.DPCLIP_KIND_ELEMENTWISE, H, Z, True)])
    plan.run(1.0, 0.0, 0)
    torch.cuda.synchronize()
    keep = [0, 1, 3, 4]
    ref = (H[keep].double() * Z[keep].double()).sum((0, 1))
    assert torch.isinf(plan.norms[2]) and plan.clip[2].item() == 0.0
    assert _rel(plan.gW[0], ref) <= 1e-5 and np.isfinite(plan.gb[0].cpu().numpy()).all()


def test_elementwise_overflow_beside_an_infinite_input(dp):
    # columns 4 to 7 belong to one thread: an infinite input in column 5 makes that column's sum NaN (0 times infinity) and no other
    B, T, d = 5, 16, 40
    H = torch.randn(B, T, d, device="cuda"); Z = torch.randn(B, T, d, device="cuda") * 1e-3
    H[2, :, 7] = 3e30; Z[2, :, 7] = 1e20
    H[2, 0, 5] = math.inf
    plan = dp.ModelPlan([dp.ModelLayer(dp.DPCLIP_KIND_ELEMENTWISE, H, Z, True)])
    plan.run(1.0, 0.0, 0)
    torch.cuda.synchronize()
    assert plan.clip[2].item() == 0.0
    ref = (H[[0, 1, 3, 4]].double() * Z[[0, 1, 3, 4]].double()).sum((0, 1))
    others = [c for c in range(d) if c != 5]
    assert torch.isnan(plan.gW[0][5]) and _rel(plan.gW[0][others], ref[others]) <= 1e-5
    assert torch.isfinite(plan.gb[0]).all()


# sums from stored rows by eight warps (up to 256 examples), 32 and clusters of CTAs, around the ends of each
@pytest.mark.parametrize("B", [256, 257, 1024, 1025, 2049, 5000, 9000])
@pytest.mark.parametrize("d", [31, 64])
def test_elementwise_grads_of_many_examples(dp, B, d):
    gen = torch.Generator(device="cuda"); gen.manual_seed(B)
    H = torch.randn(B, 8, d, generator=gen, device="cuda")
    Z = torch.randn(B, 8, d, generator=gen, device="cuda") * _spread(B)[:, None, None] / (16 * d) ** 0.5
    plan = dp.ModelPlan([dp.ModelLayer(dp.DPCLIP_KIND_ELEMENTWISE, H, Z, True), dp.ModelLayer(dp.DPCLIP_KIND_ELEMENTWISE, H, Z, False)])
    plan.run(1.0, 0.0, 0)
    torch.cuda.synchronize()
    g, s = (H.double() * Z.double()).sum(1), Z.double().sum(1)
    clip = (1.0 / (2 * g.pow(2).sum(1) + s.pow(2).sum(1)).sqrt()).clamp(max=1.0)
    assert clip.max().item() == 1.0 and clip.min().item() < 0.5
    for got, ref in ((plan.gW[0], g), (plan.gb[0], s), (plan.gW[1], g)):
        assert _rel(got, (clip[:, None] * ref).sum(0)) <= TOL["f32"]["grad"]


# ---------------------------------------------------------------------------
# convolutions from feature maps, copied as patch matrices: widths that are no multiple of 16 bytes, several examples per CTA,
# channel blocks with a remainder, strides, paddings beyond the map, odd rows of narrow layers
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,B,C,size,d_out,k,stride,pad,cm", [
    ("f32", 9, 40, (8, 8), 160, 3, 1, 1, True), ("f32", 33, 33, (13, 10), 48, 3, 1, 1, True), ("f32", 16, 3, (32, 32), 32, 3, 1, 1, True),
    ("f32", 24, 3, (33, 31), 30, 3, 1, 1, True), ("f32", 8, 72, (12, 20), 64, 5, 2, 2, False), ("f32", 40, 64, (4, 4), 130, 3, 1, 1, True),
    ("f32", 4, 48, (56, 56), 16, 1, 2, 0, True), ("bf16", 9, 40, (8, 8), 160, 3, 1, 1, True), ("bf16", 33, 33, (13, 10), 48, 3, 1, 1, True),
    ("bf16", 16, 64, (16, 16), 128, 3, 2, 1, True), ("bf16", 50, 100, (4, 6), 40, 3, 1, 1, False), ("bf16", 5, 24, (28, 28), 72, 5, 1, 4, True),
    ("bf16", 3, 20, (56, 40), 200, 3, 3, 0, True), ("bf16", 64, 80, (7, 7), 33, 2, 1, 3, True),
    ("bf16", 40, 32, (14, 14), 64, 3, 2, 0, True), ("bf16", 40, 32, (14, 14), 64, 3, 1, 1, True), ("f32", 80, 24, (6, 7), 64, 3, 2, 0, True),
    ("f32", 70, 36, (10, 5), 48, 2, 2, 0, True)])
def test_convolutions_from_feature_maps(dp, dtype, B, C, size, d_out, k, stride, pad, cm):
    _check_convolution(dp, dtype, B, C, size, d_out, (k, k), stride, pad, cm)


def _check_convolution(dp, dtype, B, C, size, d_out, k, stride, pad, cm, offset=0):
    gen = torch.Generator(device="cuda"); gen.manual_seed(7)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    n = B * C * size[0] * size[1]
    X = torch.randn(n + offset, generator=gen, device="cuda").to(td)[offset:].view(B, C, *size)
    T = ((size[0] + 2 * pad - k[0]) // stride + 1) * ((size[1] + 2 * pad - k[1]) // stride + 1)
    Z = (torch.randn(B, T, d_out, generator=gen, device="cuda") * _spread(B)[:, None, None] / (T * d_out * C * k[0] * k[1]) ** 0.5).to(td)
    plan = dp.ModelPlan([dp.ModelLayer(dp.DPCLIP_KIND_CONV, X, Z.transpose(1, 2).contiguous() if cm else Z, True,
                                       conv=(*k, stride, pad), z_channel_major=cm)])
    plan.run(1.0, 0.0, 0)
    torch.cuda.synchronize()
    assert dp.dpclip_read_status(plan.workspace) == 0
    A = torch.nn.functional.unfold(X.double(), k, padding=pad, stride=stride).transpose(1, 2)
    G = torch.einsum("bto,bti->boi", Z.double(), A)
    gb = Z.double().sum(1)
    norms = (G.pow(2).sum((1, 2)) + gb.pow(2).sum(1)).sqrt()
    clip = (1.0 / norms).clamp(max=1.0)
    assert B < 3 or (clip.max().item() == 1.0 and clip.min().item() < 0.5)
    tol = TOL[dtype]
    assert ((plan.norms.double() - norms).abs() / norms).max().item() <= tol["norm"]
    assert _rel(plan.gW[0], (clip[:, None, None] * G).sum(0)) <= tol["grad"]
    assert _rel(plan.gb[0], (clip[:, None] * gb).sum(0)) <= tol["grad"]
    return plan


# rows of positions that a CTA takes in parts: windows that begin inside the padding, rows that are no multiple of a load or of a part,
# strides, one window per position, inputs that begin off a 16-byte boundary
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,C,size,d_out,k,stride,pad,offset", [
    (16, 24, (1, 300), 64, (1, 3), 1, 1, 0), (4, 24, (1, 301), 96, (1, 9), 1, 0, 0), (4, 64, (1, 4096), 64, (1, 3), 2, 0, 0), (4, 24, (1, 16000), 32, (1, 9), 1, 0, 0),
    (3, 20, (9, 72), 64, (3, 3), 1, 1, 0), (3, 16, (12, 130), 64, (5, 5), 1, 2, 0), (3, 16, (20, 200), 64, (3, 3), 2, 1, 1), (4, 10, (7, 257), 64, (2, 7), 1, 9, 0),
    (3, 16, (3, 2001), 64, (3, 2), 3, 3, 2), (3, 8, (40, 600), 64, (16, 16), 4, 0, 4), (16, 8, (64, 6000), 64, (16, 16), 64, 0, 0), (8, 3, (20, 1000), 32, (7, 7), 2, 3, 0)])
def test_convolutions_of_long_rows(dp, dtype, B, C, size, d_out, k, stride, pad, offset):
    plan = _check_convolution(dp, dtype, B, C, size, d_out, k, stride, pad, True, offset)
    T = ((size[0] + 2 * pad - k[0]) // stride + 1) * ((size[1] + 2 * pad - k[1]) // stride + 1)
    macs = B * T * C * k[0] * k[1] * d_out
    if macs >= (4 if dtype == "bf16" else 32) << 20:              # from here on the patch matrix is copied
        assert plan.workspace.numel() >= B * T * C * k[0] * k[1] * (2 if dtype == "bf16" else 4)


# ---------------------------------------------------------------------------
# classifier heads of one position on their own: rows and columns around the kernel's 64, odd rows, noise, 1025 examples (the
# tile kernel again)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,d_in,d_out,lda", [(1, 1, 1, 1), (64, 256, 10, 256), (65, 63, 16, 63), (130, 130, 7, 131), (1024, 65, 2, 66), (1025, 64, 3, 64)])
def test_heads_of_few_outputs(dp, dtype, B, d_in, d_out, lda):
    gen = torch.Generator(device="cuda"); gen.manual_seed(B)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    A = torch.randn(B, 1, lda, generator=gen, device="cuda").to(td)[:, :, :d_in]
    Z = torch.randn(B, 1, d_out, generator=gen, device="cuda").to(td)
    clip = torch.rand(B, generator=gen, device="cuda")
    ws = torch.zeros(max(dp.dpclip_workspace_bytes(B, 1, d_in, d_out, 0 if dtype == "f32" else 1), 256), dtype=torch.uint8, device="cuda")
    gW, gb = torch.full((d_out, d_in), 9.0, device="cuda"), torch.full((d_out,), 9.0, device="cuda")
    for c in (clip, None):
        dp.dpclip_clipped_grad(A, Z, c, gW, gb, ws)
        w = torch.ones(B, device="cuda") if c is None else c
        zc = w.double()[:, None] * Z[:, 0].double()
        # bf16 operands that TMA can address take the tensor cores, which round c zb to bf16
        tol = 1e-2 if dtype == "bf16" and d_in % 8 == 0 and d_out % 8 == 0 else 1e-5
        assert _rel(gW, zc.T @ A[:, 0].double()) <= tol and _rel(gb, zc.sum(0)) <= tol
    # with noise: the same sum followed by the same draws
    dp.dpclip_add_noise(gW, 0.5, 1.0, 3, 4); dp.dpclip_add_noise(gb, 0.5, 1.0, 3, 5)
    nW, nb = torch.empty_like(gW), torch.empty_like(gb)
    dp.dpclip_clipped_grad_noise(A, Z, None, nW, nb, 0.5, 1.0, 3, 4, 5, ws)
    torch.cuda.synchronize()
    assert (nW - gW).abs().max().item() <= 1e-5 * gW.abs().max().item() and (nb - gb).abs().max().item() <= 1e-5 * gb.abs().max().item()


# ---------------------------------------------------------------------------
# clipped sums on CTA pairs: tiles narrower than 256 columns and of at most 256 rows (one sub-tile), widths around their ends, in
# shared launches and alone, with two-term sums (copied operands) and without
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("d_in,d_out", [(300, 300), (264, 520), (32, 640), (288, 136), (1100, 256), (520, 257), (768, 769), (296, 1024), (24, 512)])
@pytest.mark.parametrize("odd", [0, 2])
def test_clipped_sums_on_pairs_of_cut_tiles(dp, d_in, d_out, odd):
    gen = torch.Generator(device="cuda"); gen.manual_seed(d_in)
    B, T = 24, 50
    shapes = [(d_in + odd, d_out), (d_out, d_in + odd), (d_in + odd, d_out + odd)]
    layers = []
    for i, o in shapes:
        A = torch.randn(B, T, i, generator=gen, device="cuda").bfloat16()
        Z = (torch.randn(B, T, o, generator=gen, device="cuda") * _spread(B)[:, None, None] / (3 * T * i * o) ** 0.5).bfloat16()
        layers.append(dp.Layer(A, Z, True))
    plan = dp.StepPlan(layers)
    plan.run(1.0, 0.0, 0)
    torch.cuda.synchronize()
    assert dp.dpclip_read_status(plan.workspace) == 0
    sums = [(torch.einsum("bto,bti->boi", y.Zbar.double(), y.A.double()), y.Zbar.double().sum(1)) for y in layers]
    norms = sum(G.pow(2).sum((1, 2)) + g.pow(2).sum(1) for G, g in sums).sqrt()
    clip = (1.0 / norms).clamp(max=1.0)
    assert clip.max().item() == 1.0 and clip.min().item() < 0.5
    assert ((plan.norms.double() - norms).abs() / norms).max().item() <= 5e-6           # exact products, sums in fp32
    for l, (G, g) in enumerate(sums):
        i, o = shapes[l]
        # one bf16 rounding of a scaled operand; copied layers hold it in two terms (relative error 2^-18).  Layers TMA cannot address are
        # copied from 32 M multiply-adds on.
        copied = (i % 8 or o % 8) and i * o * B * T >= 32 << 20
        assert _rel(plan.gW[l], (clip[:, None, None] * G).sum(0)) <= (1e-5 if copied else 4e-3), l
        assert _rel(plan.gb[l], (clip[:, None] * g).sum(0)) <= 1e-5


# ---------------------------------------------------------------------------
# launches that start behind their predecessor's tail.  Steps whose first launch does (T = 1 models in two launches) and updates, right
# behind a memset, a copy, a kernel or a join, recorded and not: equal to the same with every launch in order.  And per-layer factors from the
# tail of the norm launch.
# ---------------------------------------------------------------------------
def _other_work(kind):
    """Something that still runs when the next launch is made, its last node of the given kind."""
    x, y = torch.zeros(1 << 24, device="cuda"), torch.ones(1 << 24, device="cuda")
    side = torch.cuda.Stream()

    def run():
        if kind == "memset":
            y.mul_(1.0)
            x.zero_()
        elif kind == "copy":
            x.copy_(y)
        elif kind == "kernel":
            x.add_(y)
        elif kind == "join":
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                x.add_(y)
            torch.cuda.current_stream().wait_stream(side)
    return run


def _recorded(fn):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream(priority=-1)):
        fn()
    return graph


@pytest.mark.parametrize("before", ["nothing", "memset", "copy", "kernel", "join"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("model", ["t1", "streams"])
def test_launches_behind_other_work(dp, path_switch, model, dtype, before):
    gen = torch.Generator(device="cuda"); gen.manual_seed(3)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    B = 96
    shapes = [(1, 1000, 520), (1, 520, 640), (1, 640, 10)] if model == "t1" else [(40, 264, 520), (40, 520, 264), (1, 640, 136)]
    layers = [dp.Layer(torch.randn(B, T, i, generator=gen, device="cuda").to(td),
                       (torch.randn(B, T, o, generator=gen, device="cuda") * _spread(B)[:, None, None] / (T * i * o) ** 0.5).to(td), True)
              for T, i, o in shapes]
    plan, work = dp.StepPlan(layers), _other_work(before)
    theta0 = torch.randn(plan.flat.numel(), generator=gen, device="cuda")
    theta = theta0.clone()

    def step():
        work()                                            # right in front of the step's first launch
        if model == "t1":
            plan.run(1.0, 0.1, 5)
        else:
            plan.run_streams(1.0, 0.1, 5, branches=4)
        dp.dpclip_dp_sgd_step(theta, plan.flat, 0.5, 1.0, 0.1, 7, 9, 1e-2)           # right behind the join of a step on several streams
        work()
        dp.dpclip_dp_sgd_step(theta, plan.flat, 0.5, 1.0, 0.1, 7, 11, 1e-2)

    def result(run):
        plan.flat.zero_(); plan.clip.zero_(); theta.copy_(theta0)
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        assert all(dp.dpclip_read_status(w) == 0 for w in plan.workspaces())
        return plan.clip.clone(), plan.flat.clone(), theta.clone()

    step()
    torch.cuda.synchronize()
    got = [result(step), result(_recorded(step).replay)]
    path_switch("DPCLIP_NO_OVERLAP", "1")
    want = result(step)
    # sums of norms and of windows may add up in another order from run to run
    for clip, flat, th in got:
        assert _rel(clip, want[0]) <= 1e-5 and _rel(flat, want[1]) <= 1e-4 and _rel(th, want[2]) <= 1e-4


@pytest.mark.parametrize("dtype,T,d", [("bf16", 50, 300), ("bf16", 256, 128), ("f32", 64, 192), ("f32", 48, 146)])
def test_per_layer_factors_of_recorded_steps(dp, dtype, T, d):
    gen = torch.Generator(device="cuda"); gen.manual_seed(T)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    B, n = 40, 3
    layers = [dp.Layer(torch.randn(B, T, d, generator=gen, device="cuda").to(td),
                       (torch.randn(B, T, 2 * d, generator=gen, device="cuda") * 1e-2).to(td), True) for _ in range(n)]
    plan, C = dp.StepPlan(layers), [0.5, 1.0, 2.0]
    theta = torch.randn(plan.flat.numel(), generator=gen, device="cuda")

    def step():
        clip = dp.dpclip_step_per_layer(plan, C, 0.1, 5)
        dp.dpclip_dp_sgd_step(theta, plan.flat, 0.5, 1.0, 0.1, 7, 9, 1e-2)
        return clip

    theta0 = theta.clone()
    want = [step().clone(), plan.flat.clone(), theta.clone()]
    theta.copy_(theta0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        clip = step()
    graph.replay()
    torch.cuda.synchronize()
    assert dp.dpclip_read_status(plan.workspace) == 0
    for l, (y, c) in enumerate(zip(layers, C)):
        G = torch.einsum("bto,bti->boi", y.Zbar.double(), y.A.double())
        norm = (G.pow(2).sum((1, 2)) + y.Zbar.double().sum(1).pow(2).sum(1)).sqrt()
        assert ((clip[l].double() - (c / norm).clamp(max=1.0)).abs()).max().item() <= TOL[dtype]["norm"]
    assert _rel(clip, want[0]) <= 1e-5 and _rel(plan.flat, want[1]) <= 1e-4 and _rel(theta, want[2]) <= 1e-4


# ---------------------------------------------------------------------------
# models of T = 1 layers in two launches: batches and widths around the stages and tiles, heads of few outputs, noise, the
# accumulation windows (B > 128 in fp32, > 768 in bf16), and the one launch that a header-sized workspace leaves
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,widths", [(1, (640, 520, 8)), (31, (1000, 512, 10)), (33, (784, 1000, 1000, 10)), (65, (512, 136, 520, 1)), (129, (264, 1096, 17 * 8)),
                                      (257, (2048, 264, 16)), (800, (384, 768, 24)), (2048, (128, 2200, 10))])
def test_t1_models_in_two_launches(dp, dtype, B, widths):
    gen = torch.Generator(device="cuda"); gen.manual_seed(B)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    layers = []
    for k, (i, o) in enumerate(zip(widths, widths[1:])):
        A = torch.randn(B, 1, i, generator=gen, device="cuda").to(td)
        Z = (torch.randn(B, 1, o, generator=gen, device="cuda") * torch.rand(B, 1, 1, generator=gen, device="cuda") * 2 / (i * o) ** 0.5).to(td)
        layers.append(dp.Layer(A, Z, k % 3 != 1))
    full, small = dp.StepPlan(layers), dp.StepPlan(layers)
    small.workspace = small.workspace[:256]
    n2 = sum(y.Zbar.double().pow(2).sum((1, 2)) * (y.A.double().pow(2).sum((1, 2)) + (1 if y.has_bias else 0)) for y in layers)
    clip = (0.7 / n2.sqrt()).clamp(max=1.0)
    counts = []
    for plan in (full, small):
        n0 = dp.dpclip_launch_count()
        plan.run(0.7, 0.0, 1)
        torch.cuda.synchronize()
        counts.append(dp.dpclip_launch_count() - n0)
        assert dp.dpclip_read_status(plan.workspace) == 0
        assert ((plan.norms.double() - n2.sqrt()) / n2.sqrt()).abs().max().item() <= TOL["f32"]["norm"]
        for l, y in enumerate(layers):
            zc = clip[:, None] * y.Zbar[:, 0].double()
            assert _rel(plan.gW[l], zc.T @ y.A[:, 0].double()) <= (TOL["f32"]["grad"] if dtype == "f32" else 4e-3)
            if y.has_bias:
                assert _rel(plan.gb[l], zc.sum(0)) <= 1e-5
    assert counts == [2, 1]
    # the same draws on top of either
    base = [p.flat.clone() for p in (full, small)]
    for plan in (full, small):
        plan.run(0.7, 0.3, 5)
    torch.cuda.synchronize()
    noise = [p.flat - b for p, b in zip((full, small), base)]
    assert (noise[0] - noise[1]).abs().max().item() <= 1e-4 * max(1.0, base[0].abs().max().item())


# bias sums of heads whose rows take no vector loads: every number of columns up to 16, batches around the rows in flight
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,d_out", [(1, 1), (297, 2), (300, 3), (64, 5), (2048, 7), (129, 9), (1025, 10), (333, 13), (700, 15), (96, 16)])
def test_t1_bias_sums_of_heads(dp, dtype, B, d_out):
    gen = torch.Generator(device="cuda"); gen.manual_seed(B)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    layers = []
    for i, o in ((640, 520), (520, 136), (136, d_out)):
        A = torch.randn(B, 1, i, generator=gen, device="cuda").to(td)
        Z = (torch.randn(B, 1, o, generator=gen, device="cuda") * _spread(B)[:, None, None] / (3 * i * o) ** 0.5).to(td)
        layers.append(dp.Layer(A, Z, True))
    plan = dp.StepPlan(layers)
    n2 = sum(y.Zbar.double().pow(2).sum((1, 2)) * (y.A.double().pow(2).sum((1, 2)) + 1) for y in layers)
    clip = (1.0 / n2.sqrt()).clamp(max=1.0)
    n0 = dp.dpclip_launch_count()
    plan.run(1.0, 0.0, 1)
    torch.cuda.synchronize()
    assert dp.dpclip_launch_count() - n0 == 2 and dp.dpclip_read_status(plan.workspace) == 0
    for l, y in enumerate(layers):
        zc = clip[:, None] * y.Zbar[:, 0].double()
        assert _rel(plan.gb[l], zc.sum(0)) <= 1e-5 * max(1.0, (zc.abs().sum(0).norm() / zc.sum(0).norm()).item() ** 0.5)
        assert _rel(plan.gW[l], zc.T @ y.A[:, 0].double()) <= (TOL["f32"]["grad"] if dtype == "f32" else 4e-3)


# ---------------------------------------------------------------------------
# fp32 norms on CTA pairs of examples of one window (up to 128 positions) and of more, every width of the N side
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("T", [2, 31, 33, 128, 129])
@pytest.mark.parametrize("d_in,d_out", [(520, 136), (264, 196), (500, 260), (256, 256)])
def test_fp32_norms_of_short_examples(dp, T, d_in, d_out):
    gen = torch.Generator(device="cuda"); gen.manual_seed(T)
    B = -(-(1 << 25) // (T * d_in * d_out)) + 1                   # just above the size that takes the tensor cores
    A = torch.randn(B, T, d_in, generator=gen, device="cuda")
    Z = torch.randn(B, T, d_out, generator=gen, device="cuda") * 1e-2
    ws = torch.zeros(dp.dpclip_workspace_bytes(B, T, d_in, d_out), dtype=torch.uint8, device="cuda")
    sq = torch.empty(B, device="cuda")
    dp.dpclip_layer_sqnorms(A, Z, True, sq, ws)
    torch.cuda.synchronize()
    assert dp.dpclip_read_status(ws) == 0
    ref = torch.stack([(Z[b].double().T @ A[b].double()).pow(2).sum() + Z[b].double().sum(0).pow(2).sum() for b in range(B)])
    assert ((sq.double().sqrt() - ref.sqrt()) / ref.sqrt()).abs().max().item() <= TOL["f32"]["norm"]
