"""The block's GEMMs at the edges of their tiles: 32-row units (one row, a unit
less or more by one), text and image groups cut to different heights, feature
counts that end half-way into a 256-feature tile (d an odd multiple of 128),
tail tiles cut by rows, and along K (MLP2 of 1280 channels, 80 tiles). bf16
rows and fp32 rows in; against the fp64 oracle within the block tolerance (max-abs 2e-2,
rel-L2 1e-2, as for every block test: bf16 operands, fp32 sums)."""
import numpy as np
import pytest
import torch

from oracle import hilo_oracle as O
from paper_2606_13898_gb300 import inputs as I

from .gpu_helpers import assert_block_close, lib_ready, to_dev_i32

pytestmark = pytest.mark.gpu


def check_block(d, heads, T, lens, f32):
    """One block against the oracle; rows past the used ones hold NaN before and are
    not written."""
    H = lib_ready()
    rng = np.random.default_rng(d + T + sum(lens) + f32)
    B, rows = len(lens), sum(lens)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    cap = rows + 40  # rows past the used ones hold NaN and must not matter
    w = I.make_weights(d, True, seed=d + T)
    ut = rng.standard_normal((B * T, d)).astype(np.float32)
    ui = rng.standard_normal((rows, d)).astype(np.float32)
    if not f32:
        ut, ui = I.f32_to_bf16_bits(ut), I.f32_to_bf16_bits(ui)
    dev = (lambda a: torch.from_numpy(a).cuda()) if f32 else H.bf16_from_bits
    img = torch.full((cap, d), float("nan"), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    img[:rows] = dev(ui)
    sh = H.Shape(B=B, H=64, W=64, d=d, T=T, heads=heads, mlp=1)
    out = torch.full((B * T + cap, d), 7.0, dtype=torch.float32, device="cuda")
    wsb = H.hilo_block_workspace_bytes(sh, cap)
    ws = torch.full((wsb,), 0xFF, dtype=torch.uint8, device="cuda")  # NaN
    H.hilo_block_forward(sh, H.DeviceWeights.from_host(w), to_dev_i32(cu), cap, dev(ut) if T else None, img,
                         H.HILO_F32 if f32 else H.HILO_BF16, out, ws, wsb)
    H.hilo_sync_status()
    ot, oi = O.block(ut, ui, cu, T, w, heads, True)
    got = out.cpu().numpy()
    if T:
        assert_block_close(got[:B * T], ot, "text rows")
    assert_block_close(got[B * T:B * T + rows], oi, "image rows")
    assert np.all(got[B * T + rows:] == 7.0), "rows past the used ones were written"


@pytest.mark.parametrize("f32", [0, 1])
@pytest.mark.parametrize("d,heads,T,lens", [
    (128, 1, 0, [1]),            # one row, no text: a single one-unit tile
    (128, 2, 33, [31]),          # units of 33 and 31 rows
    (384, 3, 1, [257, 95]),      # N = 1152, 384, 1536: half-empty last feature tiles
    (640, 5, 77, [333]),
    (512, 8, 64, [601]),         # MLP2 with K = 2048
    (1152, 9, 77, [65, 700]),
])
def test_block_at_tile_edges(d, heads, T, lens, f32):
    check_block(d, heads, T, lens, f32)


# Up to K = 512 the plan prices tiles by their epilogues: several rounds of whole tiles
# and tiles cut by rows, on both sides of that K
@pytest.mark.parametrize("d,heads,T,lens", [(128, 2, 154, [2235]), (256, 4, 0, [4096]), (384, 6, 64, [1700, 700]),
                                            (512, 8, 0, [2389]), (640, 5, 33, [2389])])
def test_block_of_short_k(d, heads, T, lens):
    check_block(d, heads, T, lens, 0)


def test_block_with_tiles_cut_along_k():
    """16 x 5 tiles of 256 x 256 on at most 76 pairs: MLP2's last round is cut along K = 5120."""
    check_block(1280, 10, 0, [4096], 1)
