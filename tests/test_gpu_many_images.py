"""Attention over many images: the schedule goes through up to 8 images one after
another and through more 32 at a time, keeps the row offsets in shared memory up
to 4096 images, and walks on from a job's image to the next one's. Results at
those edges (images of different and of equal length, empty ones, more and fewer
query tiles than SMs), and the cost of one image more."""
import numpy as np
import pytest
import torch

from oracle import hilo_oracle as O

from .gpu_helpers import assert_block_close, lib_ready, to_dev_i32
from .test_gpu_kernels import bits, scaled_weights

pytestmark = pytest.mark.gpu


def lengths(B, kind, T):
    rng = np.random.default_rng(B)
    if kind == "equal":
        return [40] * B
    lens = rng.integers(1, 300 if B < 200 else 4, B)
    if T:  # (the oracle has no softmax over nothing)
        lens[rng.random(B) < 0.2] = 0
        lens[-1] = 0
    return lens.tolist()


@pytest.mark.parametrize("T", [0, 3])
@pytest.mark.parametrize("B,kind", [(2, "mixed"), (8, "mixed"), (9, "mixed"), (31, "mixed"), (32, "equal"), (33, "mixed"), (65, "equal"),
                                    (97, "mixed"), (130, "equal"), (4096, "mixed"), (4097, "mixed")])
def test_attention_of_many_images(B, kind, T):
    H = lib_ready()
    rng = np.random.default_rng(B + T)
    d, heads, lens = 128, 2, lengths(B, kind, T)
    rows = sum(lens)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    ut, ui = bits(rng.standard_normal((B * T, d))), bits(rng.standard_normal((rows, d)))
    w = scaled_weights(rng, d, False, std=1.0 / np.sqrt(d))
    sh = H.Shape(B=B, H=64, W=64, d=d, T=T, heads=heads, mlp=0)
    out = torch.empty(B * T + rows, d, dtype=torch.float32, device="cuda")
    wsb = H.hilo_block_workspace_bytes(sh, rows)
    ws = torch.full((wsb,), 0xFF, dtype=torch.uint8, device="cuda")
    H.hilo_block_forward(sh, H.DeviceWeights.from_host(w), to_dev_i32(cu), rows, H.bf16_from_bits(ut) if T else None,
                         H.bf16_from_bits(ui), H.HILO_BF16, out, ws, wsb)
    H.hilo_sync_status()
    ot, oi = O.block(ut, ui, cu, T, w, heads, False)
    got = out.cpu().numpy()
    if T:
        assert_block_close(got[:B * T], ot, "text rows")
    assert_block_close(got[B * T:], oi, "image rows")


def block_time(H, B):
    """Milliseconds of a block without MLP over B images of 64 rows, best of 20."""
    d, rows = 128, 64 * B
    rng = np.random.default_rng(0)
    sh = H.Shape(B=B, H=64, W=64, d=d, T=8, heads=2, mlp=0)
    w = H.DeviceWeights.from_host(scaled_weights(rng, d, False, std=1.0 / np.sqrt(d)))
    cu = to_dev_i32(np.arange(B + 1) * 64)
    ut = torch.randn(8 * B, d, device="cuda").bfloat16()
    ui = torch.randn(rows, d, device="cuda").bfloat16()
    out = torch.empty(8 * B + rows, d, dtype=torch.float32, device="cuda")
    wsb = H.hilo_block_workspace_bytes(sh, rows)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    times = []
    for _ in range(25):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            H.hilo_block_forward(sh, w, cu, rows, ut, ui, H.HILO_BF16, out, ws, wsb)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / 4)
    return min(times[5:])


def test_one_image_more_costs_one_image_more():
    """Offsets read again from global memory for every job, from image 0 on, once
    made 129 images take 283 us where 128 took 76."""
    H = lib_ready()
    t128, t129, t256 = (block_time(H, B) for B in (128, 129, 256))
    assert t129 < 1.5 * t128, (t128, t129)
    assert t256 < 4.0 * t128, (t128, t256)
