"""The selector's mask dilation: a 16 x 16-token tile reads its halo of up to 64
tokens as rows of bits. Radii around the word edges, masks at the grid's corners
and edges, grids smaller and larger than the halo; and its cost, which must not
depend on how many tokens the threshold selects."""
import numpy as np
import pytest
import torch
from scipy import ndimage

from oracle import hilo_oracle as O
from paper_2606_13898_gb300 import inputs as I

from .gpu_helpers import lib_ready
from .test_gpu_select import run_select

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0, 1, 7, 8, 9, 15, 16, 17, 24, 31, 32, 40, 63, 64])
@pytest.mark.parametrize("Hh,W", [(4, 6), (36, 18), (20, 150)])
def test_dilation_at_word_edges(Hh, W, radius):
    H = lib_ready()
    rng = np.random.default_rng(radius + W)
    B, N = 3, Hh * W
    img = I.make_image(B, Hh, W, 8, 1, seed=W)
    mask = np.zeros((B, N), np.uint8)
    mask[0, [0, N - 1]] = 1                       # opposite corners
    mask[1, rng.integers(0, N, 3)] = [1, 128, 255]  # anywhere, any nonzero byte
    grown = ndimage.maximum_filter(mask.reshape(B, Hh, W), size=(1, 2 * radius + 1, 2 * radius + 1), mode="constant")
    for thr in (0.4, 2.0):                        # 2.0: no token by its magnitude
        got = run_select(H, img, mask, Hh, W, 8, radius, thr)
        assert np.array_equal(got, O.sobel_select(img, (grown != 0).reshape(B, N).astype(np.uint8), Hh, W, 8, 0, thr))


def select_time(H, radius, thr):
    """Milliseconds of one selection over 64 x 64 tokens with an empty mask, best of 20."""
    sh = H.Shape(B=1, H=64, W=64, d=128)
    n = H.hilo_sobel_workspace_bytes(sh)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    img = torch.rand(1, 1024, 1024, 3, device="cuda")
    mask = torch.zeros(64 * 64, dtype=torch.uint8, device="cuda")
    keep = torch.empty(64 * 64, dtype=torch.uint8, device="cuda")
    times = []
    for _ in range(25):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(8):
            H.hilo_sobel_select(sh, img, 3, 16, mask, radius, thr, keep, ws, n)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / 8)
    return min(times[5:])


def test_dilation_costs_little_at_any_radius():
    """A window of bytes per token once made radius 64 take 991 us where radius 1
    takes 10."""
    H = lib_ready()
    near = select_time(H, 1, 0.1)
    for thr in (0.1, 2.0):
        assert select_time(H, 64, thr) < 4 * near + 0.01, thr
