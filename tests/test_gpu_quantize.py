"""GPU parity: NVFP4 quantizer (metis_quantize_nvfp4) against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import gauss, nvfp4 as onv
from paper_2509_00404_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2509_00404_b200 import binding as B
    h = B.Handle(0)
    yield B, h
    h.close()


def _adversarial(rng, rows, cols):
    """Heavy-tailed rows, exact ties, zero blocks, signed zeros, block maxima on E4M3 boundaries."""
    x = rng.standard_normal((rows, cols)) * np.exp(rng.uniform(-4, 4, (rows, 1)))
    x[1, :16] = 0.0
    x[2, 16:32] = -0.0
    x[3, :16] = np.array([6, 5, 3.5, 2.5, 1.75, 1.25, 0.75, 0.25, -6, -5, -3.5, -2.5, -1.75, -1.25, -0.75, -0.25])
    x[4, :16] = 448.0 * 6 / 7
    x[5, 32:48] = 1e-30
    x = synth.to_bf16_values(x.astype(np.float32))
    return x


def _compare(B, h, x, xd, axes, rounding, layout, seed=1234, tensor_scale=None):
    from gpu_util import nv_to_numpy
    bc, br = h.quantize_nvfp4(xd, axes, rounding, seed=seed, layout=layout, tensor_scale=tensor_scale)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    for t, axis in ((bc, onv.AXIS_COLS), (br, onv.AXIS_ROWS)):
        if t is None:
            continue
        c, s, ts = nv_to_numpy(t)
        oc, os_, ots = onv.quantize(x, axis, rounding, seed=seed, tensor_scale=tensor_scale)
        assert ts == ots
        assert np.array_equal(s, os_)
        assert np.array_equal(c, oc)


@pytest.mark.parametrize("rounding", [0, 1])
@pytest.mark.parametrize("layout", [0, 1])
def test_quantizer_bit_exact_both_axes(ctx, rounding, layout):
    from gpu_util import to_dev_bf16
    B, h = ctx
    rng = np.random.default_rng(10 + rounding)
    x = _adversarial(rng, 320, 448)                  # spans several 128-tiles with a ragged tail in both directions
    _compare(B, h, x, to_dev_bf16(x), B.BLOCKS_BOTH, rounding, layout)


@pytest.mark.parametrize("rounding", [0, 1])
def test_quantizer_strided_views_and_unaligned_scale_rows(ctx, rounding):
    """The paths beside the fast one: a BF16 operand that is a column slice of a wider tensor (leading dimension larger
    than the width, rows starting 16 bytes off a 32-byte boundary: no 32-byte loads), and a linear scale layout whose
    rows are not a multiple of four blocks (scale bytes written one by one)."""
    from gpu_util import to_dev_bf16
    B, h = ctx
    rng = np.random.default_rng(40 + rounding)
    x = _adversarial(rng, 336, 400)                              # 25 and 21 blocks per stored row
    wide = torch.zeros((336, 400 + 24), dtype=torch.bfloat16, device="cuda")
    wide[:, 8:408] = to_dev_bf16(x)
    view = wide[:, 8:408]
    assert view.data_ptr() % 32 == 16 and view.stride(0) == 424
    _compare(B, h, x, view, B.BLOCKS_BOTH, rounding, B.SF_LINEAR)
    _compare(B, h, np.ascontiguousarray(x[:320, :384]), wide[:320, 8:392], B.BLOCKS_BOTH, rounding, B.SF_TILED)   # tiled scales want multiples of 64
    _compare(B, h, x, to_dev_bf16(x), B.BLOCKS_BOTH, rounding, B.SF_LINEAR)


def test_quantizer_fp32_input_given_scale_and_single_axis(ctx):
    B, h = ctx
    rng = np.random.default_rng(3)
    x = (rng.standard_normal((64, 128)) * 3).astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    _compare(B, h, x, xd, B.BLOCKS_ALONG_COLS, B.ROUND_RNE, B.SF_LINEAR, tensor_scale=np.float32(0.01))
    _compare(B, h, x, xd, B.BLOCKS_ALONG_ROWS, B.ROUND_SR, B.SF_TILED, tensor_scale=np.float32(0.004))  # saturates some blocks
    _compare(B, h, x, xd, B.BLOCKS_ALONG_COLS, B.ROUND_SR, B.SF_LINEAR)


def test_quantizer_all_zero_and_tiny_shapes(ctx):
    B, h = ctx
    x = np.zeros((16, 64), dtype=np.float32)
    _compare(B, h, x, torch.from_numpy(x).cuda(), B.BLOCKS_BOTH, B.ROUND_RNE, B.SF_LINEAR)
    x = np.full((16, 16), -2.5, dtype=np.float32)
    _compare(B, h, x, torch.from_numpy(x).cuda(), B.BLOCKS_BOTH, B.ROUND_SR, B.SF_LINEAR)


def test_every_fp32_tie_and_neighbour_rounds_like_the_oracle(ctx):
    """All seven E2M1 midpoints, +-1 ulp, both signs, placed in blocks whose scale is exactly 1."""
    B, h = ctx
    mids = np.array([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0], dtype=np.float32)
    vals = np.concatenate([mids, np.nextafter(mids, np.float32(0)), np.nextafter(mids, np.float32(9))])
    vals = np.concatenate([vals, -vals]).astype(np.float32)           # 42 values
    x = np.zeros((16, 64), dtype=np.float32)
    x[:, 0] = 6.0
    x[:, 16] = 6.0
    x[:, 32] = 6.0
    x[:, 48] = 6.0
    flat = x.reshape(-1)
    slots = [i for i in range(flat.size) if i % 16 != 0][: vals.size]
    flat[slots] = vals
    _compare(B, h, x, torch.from_numpy(x).cuda(), B.BLOCKS_ALONG_COLS, B.ROUND_RNE, B.SF_LINEAR, tensor_scale=np.float32(1.0))


def test_rejects_bad_arguments(ctx):
    B, h = ctx
    x = torch.zeros((16, 24), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.MetisError):
        h.quantize_nvfp4(x, B.BLOCKS_ALONG_COLS, layout=B.SF_LINEAR)            # cols not a multiple of 16
    x = torch.zeros((16, 48), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.MetisError):
        h.quantize_nvfp4(x, B.BLOCKS_ALONG_COLS, layout=B.SF_TILED)             # tiled scales need a multiple of 64


def test_quantile_table_matches_oracle(ctx):
    B, h = ctx
    ref = gauss.quantile_level(np.arange(65536))
    assert np.array_equal(h.quantile_table(), (ref.view(np.uint32) >> 16).astype(np.uint16))


@pytest.mark.parametrize("case", [(128, 256, 1, "bf16"), (200, 192, 0, "fp32"), (1024, 4096, 1, "bf16")], ids=lambda c: "%dx%d_%s_%s" % (c[0], c[1], "sr" if c[2] else "rne", c[3]))
def test_random_hadamard_recipe_matches_the_oracle_byte_for_byte(case):
    """The comparison recipe of Section 4 (random Hadamard transform of every 16-block, then NVFP4 with stochastic
    rounding): codes, scale bytes and tensor scale against the oracle, and the product-preserving property on the
    GPU's own bytes."""
    from oracle import hadamard as ohad
    from gpu_util import nv_to_numpy
    from paper_2509_00404_b200 import binding as B, synth
    rows, cols, rounding, dt = case
    x, _ = synth.llama_like(rows, cols, 1.0, 900 + rows, rank=8)
    if dt == "fp32":
        x = (x * np.float32(1.2345)).astype(np.float32)
    xd = torch.from_numpy(x).cuda() if dt == "fp32" else torch.from_numpy(x).to(torch.bfloat16).cuda()
    h = B.Handle(0)
    try:
        layout = B.SF_TILED if cols % 64 == 0 else B.SF_LINEAR
        t = h.quantize_rht_nvfp4(xd, rounding=rounding, seed=17, layout=layout)
        torch.cuda.synchronize()
        assert h.device_status() == 0
        c, s, ts = nv_to_numpy(t)
        oc, os_, ots = ohad.quantize_rht(x, rounding, seed=17)
        assert ts == ots and np.array_equal(s, os_) and np.array_equal(c, oc)
        back = ohad.rht_inverse(onv.dequantize(c, s, ts), 17)
        assert np.linalg.norm(back - x) / np.linalg.norm(x) < 0.2
    finally:
        h.close()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rows,cols,pad", [(16, 64, 0), (16, 64, 8), (33, 64, 4), (130, 1088, 64), (70, 2112, 16), (64, 16448, 4), (3, 16448, 64), (4096, 2112, 0)])
def test_tensor_amax_sees_every_element(ctx, dtype, rows, cols, pad):
    """The tensor scale is amax / 2688 whichever element is the largest: corners, the ends of a row, a middle row, and every
    column of one row (operands of one short row group, rows of several segments, contiguous ones and strided ones, whose rows
    always start on 16-byte boundaries).  The columns beyond the operand hold larger values and must not count."""
    B, h = ctx
    if dtype == torch.bfloat16 and pad % 8:
        pad += 4                                     # the library wants rows on 16-byte boundaries
    full = torch.rand((rows, cols + pad), device="cuda").to(dtype)
    full[:, cols:] = 1000.0
    x = full[:, :cols]
    spots = {(0, 0), (0, cols - 1), (rows - 1, 0), (rows - 1, cols - 1), (rows // 2, cols // 2)} | {(rows // 3, c) for c in range(0, cols, max(1, cols // 37))}
    for r, c in sorted(spots):
        old = x[r, c].clone()
        x[r, c] = -7.0
        t, _ = h.quantize_nvfp4(x)
        assert t.tensor_scale.item() == float(np.float32(7.0) / np.float32(2688.0)), (r, c)
        x[r, c] = old
    x[rows - 1, cols // 2] = float("nan")
    h.quantize_nvfp4(x)
    torch.cuda.synchronize()
    assert h.device_status() != 0


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_stochastic_rounding_of_saturated_and_exact_blocks(ctx, dtype):
    """Blocks whose scale is clamped at 448 (a tensor scale far too small: most elements saturate at 6), blocks whose maximum
    falls exactly on an E4M3 scale, values on the E2M1 grid (never rounded up, whatever the draw) and just above it, and
    tiny ones: byte for byte the oracle's codes."""
    B, h = ctx
    rng = np.random.default_rng(77)
    x = rng.standard_normal((192, 320)).astype(np.float32)
    x[:32] *= 1e4
    x[32:48] = np.tile(np.array([0, 0.5, 1, 1.5, 2, 3, 4, 6], dtype=np.float32), 40)
    x[48:64] = np.tile(np.array([0.5, 1, 1.5, 2, 3, 4, 5.96875, 6], dtype=np.float32) * np.float32(1.0078125), 40)
    x[64:80] *= 1e-6
    x[::3] *= -1
    x = synth.to_bf16_values(x)
    xd = torch.from_numpy(x).to(dtype).cuda()
    for ts in (None, 1.0 / 448, 1.0):
        _compare(B, h, x, xd, B.BLOCKS_BOTH, onv.ROUND_SR, B.SF_TILED, tensor_scale=ts)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rounding", [onv.ROUND_RNE, onv.ROUND_SR])
def test_a_nan_is_stored_as_six_and_its_block_is_scaled_by_the_others(ctx, dtype, rounding):
    """With a caller's tensor scale no amax check sees a NaN: it becomes +6 times the block scale, in ordinary, saturated and zero
    blocks and beside an infinity, and every other element keeps the code that it has with a zero in the NaN's place.  A block
    of nothing else gets the largest scale."""
    from gpu_util import nv_to_numpy
    B, h = ctx
    rng = np.random.default_rng(78)
    x = synth.to_bf16_values(rng.standard_normal((192, 192)).astype(np.float32))
    x[16:32] *= 4096.0
    x[32:48] = 0.0
    nan = np.zeros(x.shape, dtype=bool)
    nan[::5, ::7] = True                             # several in a block and one, in either orientation
    nan[48:96] = False
    nan[50, 3] = nan[70, 100] = True
    nan[112:128] = False
    nan[112:128, 64:80] = True
    x[nan] = 0.0
    x[80, 40] = np.inf
    xn = np.where(nan, np.float32("nan"), x).astype(np.float32)
    ts = np.float32(1.0 / 448)
    bc, br = h.quantize_nvfp4(torch.from_numpy(xn).to(dtype).cuda(), B.BLOCKS_BOTH, rounding, seed=5, layout=B.SF_TILED, tensor_scale=ts)
    torch.cuda.synchronize()
    for t, axis, at in ((bc, onv.AXIS_COLS, nan), (br, onv.AXIS_ROWS, nan.T)):
        c, s, _ = nv_to_numpy(t)
        with np.errstate(invalid="ignore", over="ignore"):
            oc, os_, _ = onv.quantize(np.where(np.isinf(x), np.float32(3e38), x), axis, rounding, seed=5, tensor_scale=ts)
        os_ = np.where(at.reshape(at.shape[0], -1, 16).all(axis=2), np.uint8(126), os_)
        assert np.array_equal(s, os_)
        assert np.array_equal(c[~at], oc[~at]) and bool((c[at] == 7).all())


@pytest.mark.parametrize("tensor_scale", [1.0 / 448, 0.013, 2.0 ** -80, 2.0 ** 98])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rounding", [onv.ROUND_RNE, onv.ROUND_SR])
def test_whole_tiles_and_block_scales_at_their_edges(ctx, dtype, rounding, tensor_scale):
    """Matrices of whole tiles have a kernel of their own, and the block scale's quotient is formed from a reciprocal where the tensor scale
    allows it and divided where not (2^-80): blocks whose maximum is every E4M3 value times 6 tensor scales, the numbers beside it, and
    ones far below the smallest scale, byte for byte the oracle's codes, from a contiguous operand and from a view with rows off the
    32-byte boundary (the general kernel)."""
    B, h = ctx
    rng = np.random.default_rng(79)
    ts = np.float32(tensor_scale)
    x = rng.uniform(-1, 1, (256, 384)).astype(np.float32)
    grid = np.array([onv.E4M3_POS[b] for b in range(1, 127)], dtype=np.float32) * (np.float32(6) * ts)
    edge = np.stack([grid, np.nextafter(grid, np.float32(0)), np.nextafter(grid, np.float32(np.inf)), grid * np.float32(2.0 ** -25)]).reshape(-1)
    blocks = x.reshape(-1, 16)
    blocks[: edge.size] *= edge[:, None]
    blocks[: edge.size, 5] = edge
    blocks[edge.size:] *= ts * np.float32(40)
    blocks[-3:] *= np.float32(2.0 ** -36)
    if dtype == torch.bfloat16:
        x = synth.to_bf16_values(x)
    xd = torch.from_numpy(x).to(dtype).cuda()
    _compare(B, h, x, xd, B.BLOCKS_BOTH, rounding, B.SF_TILED, tensor_scale=ts)
    wide = torch.zeros((256, 384 + 8), dtype=dtype, device="cuda")
    wide[:, 8:] = xd
    _compare(B, h, x, wide[:, 8:], B.BLOCKS_BOTH, rounding, B.SF_TILED, tensor_scale=ts)
    _compare(B, h, x[:128, :128].copy(), xd[:128, :128].contiguous(), B.BLOCKS_ALONG_ROWS, rounding, B.SF_TILED, tensor_scale=ts)


@pytest.mark.parametrize("dtype,rows,cols,pad", [(torch.float32, 37, 1088, 64), (torch.float32, 41, 2752, 64), (torch.bfloat16, 5, 2112, 64), (torch.bfloat16, 9, 6208, 8),
                                                 (torch.bfloat16, 10083, 8192, 16), (torch.float32, 10081, 4096, 0)])
def test_tensor_amax_of_few_threads_a_row_and_beyond_the_l2(ctx, dtype, rows, cols, pad):
    """Strided rows that are cut into units of 32, 64 or 128 threads (with rows left over in the last unit), and tensors just above 5/4 of the
    L2, a CTA per unit: the largest element counts wherever it stands, and those beyond the operand's columns do not."""
    B, h = ctx
    full = torch.rand((rows, cols + pad), device="cuda").to(dtype)
    full[:, cols:] = 1000.0
    x = full[:, :cols]
    step = 16 // x.element_size()
    spots = {(0, 0), (0, cols - 1), (rows - 1, 0), (rows - 1, cols - 1)} | {(rows - 1 - i, (i * 37 * step + i) % cols) for i in range(min(rows, 24))} | {(rows // 2, c) for c in range(0, cols, max(step, cols // 24))}
    out = h.quantize_nvfp4(x, layout=B.SF_LINEAR)
    for r, c in sorted(spots):
        old = x[r, c].clone()
        x[r, c] = -7.0
        t, _ = h.quantize_nvfp4(x, layout=B.SF_LINEAR, out=out)
        assert t.tensor_scale.item() == float(np.float32(7.0) / np.float32(2688.0)), (r, c)
        x[r, c] = old
