"""The bandwidth kernels and the attention's schedule where their code changes
path: the score where a thread takes one more group of channels; the split at
the sizes where a thread's number of tokens doubles, for one image, clusters of
images (2, 5, 8) and more than a cluster (9), in each mode and on arrays that
allow no wide load; low-frequency rows in one and several slices; the three unpools on fp32 arrays that allow 32-byte accesses
and that do not; e4m3 rows at the ends of the widths that stay in registers;
LayerNorm rows below, at and above one pass of the resident groups; attention
over images of different length, with more query tiles than SMs, and more images
than the offsets kept in shared memory; the selector's tiles for every number of
channels."""
import numpy as np
import pytest
import torch

from oracle import hilo_oracle as O
from paper_2606_13898_gb300 import inputs as I

from .gpu_helpers import assert_block_close, lib_ready, to_dev_i32
from .test_gpu_kernels import bits, check_split, scaled_weights
from .test_gpu_select import run_select

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    return lib_ready()


def offset_by_one(a):
    """A device copy of the array one element past an aligned address."""
    t = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    buf[1:] = t
    return buf[1:]


@pytest.mark.parametrize("d", [1024, 1152, 2048, 2176, 3200, 4096])
def test_score_at_groups_per_thread(H, d):
    rng = np.random.default_rng(d)
    x = bits(rng.standard_normal((2, 6, 4, d)) * rng.uniform(0.1, 10, size=(2, 6, 4, 1)))
    s = torch.empty(48, dtype=torch.float32, device="cuda")
    H.hilo_score(H.Shape(B=2, H=6, W=4, d=d), H.bf16_from_bits(x), s)
    H.hilo_sync_status()
    ref = O.score(x)
    assert np.array_equal(s.cpu().numpy().view(np.uint32), ref.reshape(-1).view(np.uint32))


@pytest.mark.parametrize("mode", ["plain1", "plain2", "regions2", "lf4"])
@pytest.mark.parametrize("B", [1, 2, 5, 8, 9])
@pytest.mark.parametrize("Hh,W", [(4, 4), (64, 64), (64, 68), (64, 128), (64, 132), (128, 128), (128, 132)])
def test_split_at_tokens_per_thread(H, Hh, W, B, mode):
    rng = np.random.default_rng(Hh * W + B)
    N = Hh * W
    s = (rng.integers(0, 300, size=(B, N)) * 0.25).astype(np.float32)
    mask = (rng.random((B, N)) < 0.05).astype(np.uint8)
    kk = rng.integers(1, N // 2, size=B).astype(np.int32)
    km = rng.integers(1, N // 2, size=B).astype(np.int32)
    levels, lf = (2 if mode[-1] == "2" else 1), (4 if mode == "lf4" else 0)
    sh = H.Shape(B=B, H=Hh, W=W, d=128, levels=levels, lf=lf)
    sp = H.SplitBuffers.alloc(sh)
    sp.labels = offset_by_one(sp.labels.cpu().numpy())
    (H.hilo_split_regions if mode == "regions2" else H.hilo_split)(
        sh, offset_by_one(s), offset_by_one(mask), to_dev_i32(kk), to_dev_i32(km), sp)
    H.hilo_sync_status()
    ref = (O.split(s, mask, kk, km, Hh, W, levels, lf=lf) if lf else
           O.split(s, mask, kk, km, Hh, W, levels, granular=mode == "regions2"))
    check_split(sp, ref, B, N)


@pytest.mark.parametrize("levels,lf", [(1, 0), (2, 0), (1, 2), (1, 4), (1, 8)])
@pytest.mark.parametrize("d", [128, 256, 384, 512, 640, 1024, 1152, 3072, 3200])
def test_pack_at_warps_per_row(H, d, levels, lf):
    """Every number of warps per row, of rows per CTA and of chunks in flight, for rows
    that are no multiple of a CTA's, and a capacity that ends within an image."""
    rng = np.random.default_rng(d + levels + lf)
    B, Hh, W = 3, 16, 24
    N = Hh * W
    x = bits(rng.standard_normal((B, Hh, W, d)))
    kk = np.array([0, N // 3, N], np.int32)
    mask = (rng.random((B, N)) < 0.02).astype(np.uint8)
    ref = O.split(O.score(x), mask, kk, kk // 2, Hh, W, levels, **({"lf": lf} if lf else {}))
    sh = H.Shape(B=B, H=Hh, W=W, d=d, levels=levels, lf=lf)
    rows = int(ref.cu_img[-1])
    sp = H.SplitBuffers.alloc(sh)
    for name in ("labels", "counts", "cu_img", "tok_row"):
        getattr(sp, name).copy_(torch.from_numpy(getattr(ref, name).reshape(-1)))
    sp.row_src[:rows].copy_(torch.from_numpy(ref.row_src))
    want = O.pack(x, ref, lf) if lf else O.pack(x, ref)
    for cap in (rows + 3, rows - 7):
        packed = torch.full((rows + 3, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        H.hilo_pack(sh, H.bf16_from_bits(x), sp, packed, cap)
        H.hilo_sync_status()
        n = min(cap, rows)
        assert np.array_equal(H.bits_from_bf16(packed[:n]), want[:n])
        assert torch.isnan(packed[n:].float()).all()


@pytest.mark.parametrize("B", [1, 2])
@pytest.mark.parametrize("lf,d", [(2, 1152), (4, 1024), (4, 1152), (8, 128), (8, 2176), (8, 4096)])
def test_pack_low_frequency_slices(H, lf, d, B):
    rng = np.random.default_rng(lf + d + B)
    Hh, W = 16, 24
    N = Hh * W
    x = bits(rng.standard_normal((B, Hh, W, d)))
    kk = rng.integers(0, N + 1, size=B).astype(np.int32)
    ref = O.split(O.score(x), (rng.random((B, N)) < 0.1).astype(np.uint8), kk, kk, Hh, W, 1, lf=lf)
    sh = H.Shape(B=B, H=Hh, W=W, d=d, lf=lf)
    cap, rows = H.hilo_row_capacity(sh), int(ref.cu_img[-1])
    sp = H.SplitBuffers.alloc(sh)
    for name in ("labels", "counts", "cu_img", "tok_row"):
        getattr(sp, name).copy_(torch.from_numpy(getattr(ref, name).reshape(-1)))
    sp.row_src[:rows].copy_(torch.from_numpy(ref.row_src))
    packed = torch.full((cap, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    H.hilo_pack(sh, H.bf16_from_bits(x), sp, packed, cap)
    H.hilo_sync_status()
    assert np.array_equal(H.bits_from_bf16(packed[:rows]), O.pack(x, ref, lf))
    assert torch.isnan(packed[rows:].float()).all()


def check_unpacks(H, B, Hh, W, d, off):
    """The three unpools on fp32 arrays `off` floats past a 32-byte boundary."""
    rng = np.random.default_rng(d + off)
    N = Hh * W
    x = bits(rng.standard_normal((B, Hh, W, d)))
    ref = O.split(O.score(x), (rng.random((B, N)) < 0.1).astype(np.uint8), np.array([N // 4, 5], np.int32),
                  np.array([N // 4, 9], np.int32), Hh, W, 2)
    rows = int(ref.cu_img[-1])
    pk, out = O.pack(x, ref), rng.standard_normal((rows, d)).astype(np.float32)
    sh = H.Shape(B=B, H=Hh, W=W, d=d, levels=2)
    sp = H.SplitBuffers.alloc(sh)
    sp.labels.copy_(torch.from_numpy(ref.labels.reshape(-1)))
    sp.tok_row.copy_(torch.from_numpy(ref.tok_row.reshape(-1)))
    buf = torch.full((rows * d + 8,), float("nan"), dtype=torch.float32, device="cuda")
    od = buf[off:off + rows * d]
    od.copy_(torch.from_numpy(out.reshape(-1)))
    xd, pd = H.bf16_from_bits(x), H.bf16_from_bits(pk)
    ybuf = torch.full((B * N * d + 8,), 7.0, dtype=torch.float32, device="cuda")
    y = ybuf[off:off + B * N * d]
    for want, call in ((O.unpack(out, ref), lambda: H.hilo_unpack(sh, od, sp, y)),
                       (O.unpack_delta(out, pk, x, ref), lambda: H.hilo_unpack_delta(sh, od, pd, xd, sp, y))):
        ybuf.fill_(7.0)
        call()
        H.hilo_sync_status()
        assert np.array_equal(y.cpu().numpy().reshape(want.shape), want)
        assert torch.all(ybuf[:off] == 7.0) and torch.all(ybuf[off + B * N * d:] == 7.0)
    H.hilo_unpack_update(sh, od, sp, xd, 0.035)
    H.hilo_sync_status()
    assert np.array_equal(H.bits_from_bf16(xd).reshape(x.shape), O.update(x, O.unpack(out, ref).reshape(x.shape), 0.035))


@pytest.mark.parametrize("off", [0, 4])  # floats past a 32-byte boundary: 32- and 16-byte accesses
@pytest.mark.parametrize("d", [128, 384, 3072, 4096])
def test_unpack_at_both_alignments(H, d, off):
    check_unpacks(H, 2, 8, 12, d, off)


@pytest.mark.parametrize("off", [0, 4])
@pytest.mark.parametrize("d", [128, 256])  # one piece per lane; more tokens than resident warps
def test_unpack_of_short_rows(H, d, off):
    check_unpacks(H, 2, 64, 132, d, off)


@pytest.mark.parametrize("dtype,cols", [("bf16", 8), ("bf16", 4096), ("bf16", 4104), ("bf16", 12288),
                                        ("bf16", 12296), ("f16", 4096), ("f16", 4104), ("f16", 12296),
                                        ("f32", 4104)])
@pytest.mark.parametrize("rows", [1, 1000])
def test_quantize_rows_at_register_widths(H, dtype, cols, rows):
    rng = np.random.default_rng(cols + rows)
    x = (rng.standard_normal((rows, cols)) * np.exp(rng.uniform(-8, 8, (rows, 1)))).astype(np.float32)
    x[rows // 2, -1] = 20000.0  # the row's largest value in its last column
    if dtype == "bf16":
        xb = bits(x)
        src, code, xf = H.bf16_from_bits(xb), H.HILO_BF16, O.bf16_to_f32(xb)
    elif dtype == "f16":
        xh = np.clip(x, -60000, 60000).astype(np.float16)
        src, code, xf = torch.from_numpy(xh).cuda(), H.HILO_F16, xh.astype(np.float32)
    else:
        src, code, xf = torch.from_numpy(x).cuda(), H.HILO_F32, x
    q = torch.full((rows + 1, cols), 0x55, dtype=torch.uint8, device="cuda")
    sc = torch.empty(rows, dtype=torch.float32, device="cuda")
    H.hilo_quantize_rows_e4m3(src, code, rows, cols, q, sc)
    H.hilo_sync_status()
    cref, sref = O.quantize_rows(xf)
    got = q.cpu().numpy()
    assert np.array_equal(got[:rows], cref) and np.all(got[rows] == 0x55)
    assert np.array_equal(sc.cpu().numpy(), sref)


@pytest.mark.parametrize("dtype,cols", [("bf16", 2048), ("bf16", 2056), ("f16", 6144), ("f16", 6152), ("f32", 2048)])
def test_quantize_rows_at_piece_counts(H, dtype, cols):
    """One to two and three to six pieces of a row per thread, more rows than CTAs."""
    test_quantize_rows_at_register_widths(H, dtype, cols, 1300)


@pytest.mark.parametrize("f32", [0, 1])
@pytest.mark.parametrize("rows", [1, 911, 1830])
@pytest.mark.parametrize("d", [128, 640, 4096])
def test_layernorm_rows(H, d, rows, f32):
    """The LayerNorm rows of a block (first region of its workspace). Each is
    the fp64 value rounded to bf16 (2^-9 relative), after fp32 sums over d
    elements (mean and variance within d 2^-24 of their terms, 3e-4 at most)."""
    rng = np.random.default_rng(d + rows)
    u = (rng.standard_normal((rows, d)) * 3 + 1).astype(np.float32)
    if not f32:
        u = bits(u)
    zeros = I.BlockWeights(**{s: I.StreamWeights(
        w_qkv=np.zeros((3 * d, d), np.uint16), b_qkv=np.zeros(3 * d, np.uint16),
        w_o=np.zeros((d, d), np.uint16), b_o=np.zeros(d, np.uint16)) for s in ("txt", "img")})
    sh = H.Shape(B=1, H=64, W=64, d=d, T=0, heads=d // 128, mlp=0)
    out = torch.empty(rows, d, dtype=torch.float32, device="cuda")
    wsb = H.hilo_block_workspace_bytes(sh, rows)
    ws = torch.full((wsb,), 0xFF, dtype=torch.uint8, device="cuda")  # NaN
    H.hilo_block_forward(sh, H.DeviceWeights.from_host(zeros), to_dev_i32([0, rows]), rows, None,
                         torch.from_numpy(u).cuda() if f32 else H.bf16_from_bits(u),
                         H.HILO_F32 if f32 else H.HILO_BF16, out, ws, wsb)
    H.hilo_sync_status()
    got = ws[:rows * d * 2].view(torch.bfloat16).view(rows, d).float().cpu().numpy().astype(np.float64)
    ref = O.layer_norm(u.astype(np.float64) if f32 else O.bf16_to_f32(u).astype(np.float64))
    assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 3e-4)


@pytest.mark.parametrize("d,rows", [(128, 1), (128, 3647), (128, 3649), (256, 1825), (256, 5000), (384, 2000)])
def test_layernorm_rows_of_narrow_groups(H, d, rows):
    """A warp or 64 threads per row: 12 or 6 rows per CTA, below and above one pass."""
    test_layernorm_rows(H, d, rows, rows % 2)


@pytest.mark.parametrize("d,heads,T,lens", [
    (1024, 16, 64, [130, 900, 5, 0]),      # 240 query tiles of images 1 to 9 tiles long
    (1024, 8, 0, [257, 2050]),             # 160 tiles, hd 128, no text
    (128, 2, 0, [5, 150] * 65),            # 130 images: offsets read from memory
    (128, 1, 3, [0] * 3 + [129] * 125),    # 128 images: the last that fit in shared memory
])
def test_attention_images_of_different_length(H, d, heads, T, lens):
    rng = np.random.default_rng(d + heads + len(lens))
    B, rows = len(lens), sum(lens)
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


@pytest.mark.parametrize("patch", [8, 16])
@pytest.mark.parametrize("C", [1, 2, 3, 4])
def test_sobel_tiles_of_every_pixel_width(H, C, patch):
    """Full-width tiles (vector loads), a partial one at the right edge, and flat
    image parts (magnitude 0) beside infinite and huge pixels (magnitude inf, NaN)."""
    rng = np.random.default_rng(C + patch)
    B, Hh, W = 2, 6, 18
    img = rng.random((B, Hh * patch, W * patch, C)).astype(np.float32)
    img[0, : 2 * patch] = 0.5
    mask = np.zeros((B, Hh * W), np.uint8)
    mask[:, 5] = 1
    for thr in (0.1, 0.7):
        assert np.array_equal(run_select(H, img, mask, Hh, W, patch, 1, thr),
                              O.sobel_select(img, mask, Hh, W, patch, 1, thr))
    img[1, patch, patch] = np.inf
    img[1, 3 * patch + 2, 9 * patch] = 3e38
    with np.errstate(all="ignore"):
        assert np.array_equal(run_select(H, img, mask, Hh, W, patch, 0, 0.1),
                              O.sobel_select(img, mask, Hh, W, patch, 0, 0.1))
