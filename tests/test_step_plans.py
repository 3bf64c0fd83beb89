"""Plans of whole steps, worked out on the host (no GPU): which convolutions are copied as patch matrices, and what planning costs."""
import time

import pytest

FAKE = 1 << 20                    # an aligned address that nothing reads


@pytest.fixture(scope="module")
def binding():
    from paper_2009_03106_b200 import binding as b
    b.load_library()
    return b


def _conv(b, C, H, W, d_out, k, stride, pad):
    kh, kw = k
    m = b._CModelLayer()
    m.kind, m.z_channel_major = b.DPCLIP_KIND_CONV, 1
    m.conv = b._CConv(C, H, W, kh, kw, stride, pad)
    m.layer = b._CLayer(FAKE, 0, FAKE, 0, 0, C * kh * kw, d_out, 1, 0, FAKE, C * kh * kw, FAKE)
    return m


def _plan(b, layers, B, dtype):
    arr = (b._CModelLayer * len(layers))(*layers)
    return lambda: b.load_library().dpclip_model_workspace_bytes(arr, len(layers), B, dtype)


# long rows: the window of a CTA does not grow with the row, so the layers are copied whatever their width
@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("B,C,H,W,d_out,k,stride,pad", [
    (16, 64, 1, 16000, 64, (1, 9), 1, 0), (16, 64, 1, 4096, 64, (1, 3), 2, 0), (8, 32, 64, 4096, 32, (3, 3), 1, 1),
    (8, 8, 300, 600, 32, (16, 16), 4, 0), (4, 8, 64, 60000, 64, (16, 16), 64, 0), (4, 64, 1, 500000, 64, (1, 1), 1, 0), (16, 64, 1, 300, 64, (1, 3), 1, 1)])
def test_convolutions_of_long_rows_are_copied(binding, dtype, B, C, H, W, d_out, k, stride, pad):
    T = ((H + 2 * pad - k[0]) // stride + 1) * ((W + 2 * pad - k[1]) // stride + 1)
    copies = B * T * (C * k[0] * k[1] + d_out) * (2 if dtype else 4)
    assert _plan(binding, [_conv(binding, C, H, W, d_out, k, stride, pad)], B, dtype)() >= copies


# the plan of a step that is not recorded is made in every call: about as long as the launches of one kernel (3 us here; a search for bank
# paddings at every size tried took 30 us)
def test_planning_a_convolution_step_takes_microseconds(binding):
    k3 = (3, 3)
    plan = _plan(binding, [_conv(binding, 3, 32, 32, 64, k3, 1, 1), _conv(binding, 64, 32, 32, 128, k3, 2, 1),
                           _conv(binding, 128, 16, 16, 256, k3, 2, 1), _conv(binding, 256, 8, 8, 256, k3, 1, 1)], 64, 1)
    best = float("inf")
    for _ in range(2000):
        t = time.perf_counter()
        plan()
        best = min(best, time.perf_counter() - t)
    assert best < 12e-6, best
