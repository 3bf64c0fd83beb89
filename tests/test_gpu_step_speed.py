"""Steps that once lost time: each against another form of the same work on the same GPU, with a margin well above what two runs
differ by."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dp():
    import paper_2009_03106_b200 as pkg
    pkg.load_library()
    return pkg


def _times(*steps, reps=10, rounds=9):
    """Least time of each step in microseconds: ten to a graph, the graphs in turn (the rate of a training loop)."""
    graphs = []
    for step in steps:
        step()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=torch.cuda.Stream(priority=-1)):
            for _ in range(reps):
                step()
        graphs.append(g)
    best = [float("inf")] * len(steps)
    for _ in range(rounds):
        for k, g in enumerate(graphs):
            g.replay()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                g.replay()
            b.record()
            torch.cuda.synchronize()
            best[k] = min(best[k], a.elapsed_time(b) * 1e3 / (10 * reps))
    return best


def _dense(B, T, d_in, d_out, dtype):
    A = torch.randn(B, T, d_in, device="cuda").to(dtype)
    Z = torch.randn(B, T, d_out, device="cuda") * (torch.exp((torch.rand(B, 1, 1, device="cuda") * 2 - 1) * math.log(4.0)) / math.sqrt(T * d_in * d_out))
    return A, Z.to(dtype)


def _conv(dp, B, C, size, d_out, k, stride, pad, dtype):
    X = torch.relu(torch.randn(B, C, *size, device="cuda")).to(dtype)
    T = ((size[0] + 2 * pad - k[0]) // stride + 1) * ((size[1] + 2 * pad - k[1]) // stride + 1)
    Z = (torch.randn(B, d_out, T, device="cuda") / math.sqrt(T * d_out * C * k[0] * k[1])).to(dtype)
    return dp.ModelLayer(dp.DPCLIP_KIND_CONV, X, Z, True, conv=(*k, stride, pad), z_channel_major=True)


# patch matrices of maps with an odd number of elements, loaded element by element, beside maps of one element more a channel
def test_patch_matrices_of_odd_maps(dp):
    odd = dp.ModelPlan([_conv(dp, 16, 96, (33, 31), 24, (3, 3), 1, 1, torch.bfloat16)])
    even = dp.ModelPlan([_conv(dp, 16, 96, (32, 32), 24, (3, 3), 1, 1, torch.bfloat16)])
    t_odd, t_even = _times(lambda: odd.run(1.0, 0.0, 1), lambda: even.run(1.0, 0.0, 1))
    assert t_odd <= 1.15 * t_even, (t_odd, t_even)


# element-wise layers of many examples: the sums from stored per-example gradients beside the second pass over the inputs, which a
# workspace without room for them leaves
@pytest.mark.parametrize("B,T,d", [(4096, 8, 64), (16384, 8, 64), (2048, 32, 256)])
def test_elementwise_sums_of_many_examples(dp, B, T, d):
    H, Z = _dense(B, T, d, d, torch.bfloat16)
    stored, second = (dp.ModelPlan([dp.ModelLayer(dp.DPCLIP_KIND_ELEMENTWISE, H, Z, True)]) for _ in range(2))
    second.workspace = second.workspace[:256]
    a, b = _times(lambda: stored.run(1.0, 0.05, 1), lambda: second.run(1.0, 0.05, 1))
    assert a <= 1.05 * b, (a, b)


# heads of few outputs and many examples beside the tile kernel, which a head of 17 outputs takes: as many tiles
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("B,d_in", [(512, 300), (1024, 1000)])
def test_heads_of_few_outputs_and_many_examples(dp, dtype, B, d_in):
    steps = []
    for o in (10, 17):
        A, Z = _dense(B, 1, d_in, o, dtype)
        gW, gb, clip = torch.empty(o, d_in, device="cuda"), torch.empty(o, device="cuda"), torch.rand(B, device="cuda")
        ws = torch.zeros(max(256, dp.dpclip_workspace_bytes(B, 1, d_in, o, dp.DPCLIP_F32 if dtype == torch.float32 else dp.DPCLIP_BF16)), dtype=torch.uint8, device="cuda")
        steps.append(lambda A=A, Z=Z, gW=gW, gb=gb, ws=ws: dp.dpclip_clipped_grad_noise(A, Z, clip, gW, gb, 0.05, 1.0, 3, 4, 5, ws))
    few, wide = _times(*steps)
    assert few <= 1.25 * wide, (few, wide)


# models of T = 1 layers: the bias sums of a head whose rows take no vector loads beside the same model without them, and the two launches
# beside the one cooperative launch, many examples and few tiles
@pytest.mark.parametrize("dtype,widths", [(torch.bfloat16, (784, 1000, 1000, 10)), (torch.float32, (256, 640, 640, 10))])
def test_bias_sums_of_a_head_of_few_outputs(dp, dtype, widths):
    data = [_dense(2048, 1, i, o, dtype) for i, o in zip(widths, widths[1:])]
    plans = [dp.StepPlan([dp.Layer(A, Z, k < len(data) - 1 or bias) for k, (A, Z) in enumerate(data)]) for bias in (True, False)]
    a, b = _times(*[lambda p=p: p.run(1.0, 0.05, 1) for p in plans])
    assert a <= 1.1 * b, (a, b)


@pytest.mark.parametrize("widths", [(2000, 300, 300, 300, 300, 300, 300, 2), (784, 1000, 1000, 10)])
def test_two_launches_of_many_examples(dp, path_switch, widths):
    plan = dp.StepPlan([dp.Layer(*_dense(2048, 1, i, o, torch.float32), True) for i, o in zip(widths, widths[1:])])
    two, = _times(lambda: plan.run(1.0, 0.05, 1))
    path_switch("DPCLIP_NO_T1_PLANES", "1")
    one, = _times(lambda: plan.run(1.0, 0.05, 1))
    assert two <= 1.02 * one, (two, one)


# reduces of few CTAs, and of full tiles on all SMs, beside the same step with every launch in order
@pytest.mark.parametrize("dtype,B,T,d_in,d_out", [(torch.float32, 64, 200, 192, 256), (torch.float32, 32, 300, 256, 512),
                                                  (torch.bfloat16, 512, 64, 256, 512), (torch.bfloat16, 16, 512, 1024, 1024)])
def test_reduces_beside_the_sums(dp, path_switch, dtype, B, T, d_in, d_out):
    plan = dp.StepPlan([dp.Layer(*_dense(B, T, d_in, d_out, dtype), True)])
    behind, = _times(lambda: plan.run(1.0, 0.05, 1))
    path_switch("DPCLIP_NO_OVERLAP", "1")
    ordered, = _times(lambda: plan.run(1.0, 0.05, 1))
    assert behind <= 1.05 * ordered, (behind, ordered)


# a long chain of few CTAs beside the shared fp32 norms, which fill every SM: on four streams the two run side by side
def test_small_layers_beside_the_shared_fp32_norms(dp):
    f = torch.float32
    layers = [_conv(dp, 18, 3, (28, 28), 64, (3, 3), 1, 1, f), _conv(dp, 18, 64, (28, 28), 256, (3, 3), 1, 1, f),
              _conv(dp, 18, 256, (28, 28), 256, (3, 3), 2, 1, f), _conv(dp, 18, 256, (14, 14), 256, (3, 3), 1, 1, f)]
    plan = dp.ModelPlan(layers)
    four, one = _times(lambda: plan.run_streams(1.0, 0.05, 1, branches=4), lambda: plan.run(1.0, 0.05, 1), reps=1)
    assert four <= 0.95 * one, (four, one)
