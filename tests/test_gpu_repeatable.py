"""Which block calls give the same bits every time. A tile of the MLP's second
GEMM (and of an in-place out-projection) whose K range is cut is summed by
several CTAs in whatever order they come; that is done only at widths that are
a multiple of 256 from 1024 on, with more 256 x 256 tiles than CTA pairs. Every
other call repeats itself exactly; where K is cut, two runs differ by no more
than the order of a few fp32 sums."""
import numpy as np
import pytest
import torch

from paper_2606_13898_gb300 import inputs as I

from .gpu_helpers import lib_ready, to_dev_i32

pytestmark = pytest.mark.gpu


def runs(H, d, heads, T, lens, fp8, in_place, n):
    """n outputs of one block on the same inputs, and the residual stream's largest value."""
    rng = np.random.default_rng(d + T + sum(lens))
    B, rows = len(lens), sum(lens)
    cu = to_dev_i32(np.concatenate([[0], np.cumsum(lens)]))
    w = I.make_weights(d, True, seed=d + T)
    sh = H.Shape(B=B, H=64, W=64, d=d, T=T, heads=heads, mlp=1)
    u = torch.from_numpy(rng.standard_normal((B * T + rows, d)).astype(np.float32)).cuda()
    out = torch.empty_like(u)
    need = (H.hilo_block_fp8_workspace_bytes if fp8 else H.hilo_block_workspace_bytes)(sh, rows)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    fn = H.hilo_block_forward_fp8 if fp8 else H.hilo_block_forward
    dw = (H.DeviceWeightsFP8 if fp8 else H.DeviceWeights).from_host(w)
    got = []
    for _ in range(n):
        if in_place:
            out.copy_(u)
        src = out if in_place else u
        fn(sh, dw, cu, rows, src, src[B * T:], H.HILO_F32, out, ws, need)
        H.hilo_sync_status()
        got.append(out.clone())
    return got


@pytest.mark.parametrize("d,heads,T,lens,fp8,in_place", [
    (512, 8, 64, [601], 0, 0),
    (640, 5, 77, [333], 0, 1),
    (1024, 16, 64, [300], 0, 0),   # a multiple of 256, fewer tiles than pairs
    (1024, 8, 0, [900], 1, 1),
    (1152, 9, 77, [65, 700], 0, 0),
    (1152, 18, 154, [1508], 0, 0),
    (1280, 10, 0, [1500], 1, 0),
    (3072, 24, 64, [500], 0, 0),
])
def test_block_repeats_itself_exactly(d, heads, T, lens, fp8, in_place):
    got = runs(lib_ready(), d, heads, T, lens, fp8, in_place, 12)
    assert all(torch.equal(g, got[0]) for g in got[1:])


def test_block_with_k_cut_repeats_up_to_the_order_of_sums():
    """3072 channels, 2389 rows: 120 tiles on at most 76 pairs. Up to 8 partial sums
    and the residual, each no larger than 2^6 here, are added in fp32 in some order:
    two orders differ by at most 2 * 8 * 2^-24 * 2^6 = 6.2e-5."""
    got = runs(lib_ready(), 3072, 24, 154, [2235], 0, 0, 4)
    assert float(got[0].abs().max()) < 2.0 ** 6
    for g in got[1:]:
        assert float((g - got[0]).abs().max()) <= 6.2e-5
