"""GPU parity: the split-FP4 linear layer end to end (Eq. 2, Eq. 3, weight gradient) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import layer as olay, nvfp4 as onv, split as osp
from paper_2509_00404_b200 import synth

pytestmark = pytest.mark.gpu

TOL = 2e-3        # relative Frobenius error of layer outputs / gradients against the oracle's own split-FP4 result


@pytest.fixture(scope="module")
def ctx():
    from paper_2509_00404_b200 import binding as B
    h = B.Handle(0)
    yield B, h
    h.close()


def _check_e2e(case, errors, *pairs, base_tol=TOL):
    from gpu_util import check_e2e
    return check_e2e(case, errors, pairs, base_tol)


def _oracle_from_gpu_operand(op, k):
    """Dequantize the library's own quantized pieces in float64 (isolates the GEMM composition from the split)."""
    from gpu_util import nv_dequant
    res_c = nv_dequant(op.res_by_cols) if op.res_by_cols else None
    res_r = nv_dequant(op.res_by_rows).T if op.res_by_rows else None
    if k == 0:
        z = np.zeros((op.rows, op.cols))
        return z, res_c, res_r
    lq, rq = nv_dequant(op.left_q)[:k].T, nv_dequant(op.right_q)[:k].T
    low = (lq * op.sigma.cpu().numpy().astype(np.float64)) @ rq.T
    return low, res_c, res_r


def test_small_config_forward(ctx):
    from gpu_util import to_dev_bf16, rel_fro
    B, h = ctx
    c = synth.config_small()
    xo = h.split(to_dev_bf16(c["x"]), 4, 4, sketch=B.SKETCH_FULL, seed=1)
    wo = h.split(to_dev_bf16(c["w"]), 4, 4, sketch=B.SKETCH_FULL, seed=2)
    y = h.linear_fwd(xo, wo)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    xq = olay.quantize_operand(c["x"], 4, 4, osp.MODE_FULL, 1)
    wq = olay.quantize_operand(c["w"], 4, 4, osp.MODE_FULL, 2)
    _check_e2e("small_config_forward_128tok_256to256_k4", {"y": rel_fro(y.cpu().numpy(), olay.linear_fwd(xq, wq))}, (xo, xq), (wo, wq))
    # composition alone, on the library's own codes: tight
    lx, rxc, _ = _oracle_from_gpu_operand(xo, 4)
    lw, rwc, _ = _oracle_from_gpu_operand(wo, 4)
    assert rel_fro(y.cpu().numpy(), (lx + rxc) @ (lw + rwc).T) < 2e-5


@pytest.mark.parametrize("k", [0, 8])
def test_forward_and_backward_medium(ctx, k):
    from gpu_util import to_dev_bf16, rel_fro
    B, h = ctx
    l, m, n, p = 512, 384, 256, 8 if k else 0
    x, _ = synth.llama_like(l, m, 1.0, 51, rank=8)
    w, _ = synth.llama_like(n, m, 0.02, 52, rank=8)
    d, _ = synth.llama_like(l, n, 1e-4, 53, rank=8)
    xo = h.split(to_dev_bf16(x), k, p, sketch=B.SKETCH_SAMPLED, seed=1)
    wo = h.split(to_dev_bf16(w), k, p, sketch=B.SKETCH_FULL, seed=2)
    do = h.split(to_dev_bf16(d), k, p, sketch=B.SKETCH_SAMPLED, seed=3, rounding=B.ROUND_SR)
    y = h.linear_fwd(xo, wo)
    dx, dw = h.linear_bwd(do, xo, wo)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    xq = olay.quantize_operand(x, k, p, osp.MODE_SAMPLED, 1)
    wq = olay.quantize_operand(w, k, p, osp.MODE_FULL, 2)
    dq = olay.quantize_operand(d, k, p, osp.MODE_SAMPLED, 3, onv.ROUND_SR)
    _check_e2e("medium_512tok_384to256_k%d" % k,
               {"y": rel_fro(y.cpu().numpy(), olay.linear_fwd(xq, wq)), "dx": rel_fro(dx.cpu().numpy(), olay.linear_dgrad(dq, wq)),
                "dw": rel_fro(dw.cpu().numpy(), olay.linear_wgrad(dq, xq))}, (xo, xq), (wo, wq), (do, dq))
    lx, rxc, rxr = _oracle_from_gpu_operand(xo, k)
    lw, rwc, rwr = _oracle_from_gpu_operand(wo, k)
    ld, rdc, rdr = _oracle_from_gpu_operand(do, k)
    assert rel_fro(y.cpu().numpy(), (lx + rxc) @ (lw + rwc).T) < 2e-5
    assert rel_fro(dx.cpu().numpy(), (ld + rdc) @ (lw + rwr)) < 2e-5
    assert rel_fro(dw.cpu().numpy(), (ld + rdr).T @ (lx + rxr)) < 2e-5


@pytest.mark.parametrize("k", [0, 8, 128])
def test_layer_on_the_oracles_own_bytes(ctx, k):
    """No discontinuity in the way: the ORACLE's codes, scale bytes, tensor scales and singular values are uploaded
    into the library's operands, so both sides multiply exactly the same quantized tensors.  Eq. 2, Eq. 3 and the
    weight gradient must then agree with the oracle's float64 evaluation to FP32-accumulation accuracy, with no
    allowance of any kind."""
    from gpu_util import rel_fro, operand_from_oracle
    B, h = ctx
    l, m, n, p = (512, 384, 256, 8 if k else 0) if k <= 64 else (1024, 768, 640, 8)      # k = 128: the wide-rank composition
    x, _ = synth.llama_like(l, m, 1.0, 51, rank=max(k, 8))
    w, _ = synth.llama_like(n, m, 0.02, 52, rank=max(k, 8))
    d, _ = synth.llama_like(l, n, 1e-4, 53, rank=max(k, 8))
    xq = olay.quantize_operand(x, k, p, osp.MODE_SAMPLED, 1)
    wq = olay.quantize_operand(w, k, p, osp.MODE_FULL, 2)
    dq = olay.quantize_operand(d, k, p, osp.MODE_SAMPLED, 3, onv.ROUND_SR)
    xo, wo, do = (operand_from_oracle(B, q) for q in (xq, wq, dq))
    y = h.linear_fwd(xo, wo)
    fg = tuple(torch.full(sh, float("nan"), device="cuda") for sh in ((k, n), (k,), (k, m))) if k else None
    dx, dw = h.linear_bwd(do, xo, wo, factor_grads=fg)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    errs = (rel_fro(y.cpu().numpy(), olay.linear_fwd(xq, wq)), rel_fro(dx.cpu().numpy(), olay.linear_dgrad(dq, wq)),
            rel_fro(dw.cpu().numpy(), olay.linear_wgrad(dq, xq)))
    print("layer on the oracle's bytes, k = %d: y %.2e dx %.2e dw %.2e" % (k, *errs))
    assert max(errs) < 2e-5
    if k:
        du, ds, dv = olay.factor_grads(olay.linear_wgrad(dq, xq), wq)
        d_left, d_sigma, d_right = fg
        assert rel_fro(d_right.cpu().numpy().T, du) < 2e-5 and rel_fro(d_left.cpu().numpy().T, dv) < 2e-5
        assert rel_fro(d_sigma.cpu().numpy(), ds) < 2e-5


@pytest.mark.parametrize("dw_dtype", [torch.float32, torch.bfloat16])
def test_factor_gradients(ctx, dw_dtype):
    """dL/dU, dL/dS, dL/dV of the weight factors (Section 3.2) against the oracle."""
    from gpu_util import to_dev_bf16, rel_fro, nv_dequant
    B, h = ctx
    l, m, n, k, p = 256, 448, 192, 12, 4
    x, _ = synth.llama_like(l, m, 1.0, 61, rank=8)
    w, _ = synth.llama_like(n, m, 0.02, 62, rank=8)
    d, _ = synth.llama_like(l, n, 1e-4, 63, rank=8)
    xo = h.split(to_dev_bf16(x), k, p, sketch=B.SKETCH_SAMPLED, seed=1)
    wo = h.split(to_dev_bf16(w), k, p, sketch=B.SKETCH_FULL, seed=2)
    do = h.split(to_dev_bf16(d), k, p, sketch=B.SKETCH_SAMPLED, seed=3, rounding=B.ROUND_SR)
    d_left = torch.full((k, n), float("nan"), device="cuda")
    d_sigma = torch.full((k,), float("nan"), device="cuda")
    d_right = torch.full((k, m), float("nan"), device="cuda")
    dx, dw = h.linear_bwd(do, xo, wo, out_dtype=dw_dtype, factor_grads=(d_left, d_sigma, d_right))
    torch.cuda.synchronize()
    assert h.device_status() == 0
    # (a) the three contractions themselves, from the library's own dw and dequantized factors, in float64
    dwn = dw.float().cpu().numpy().astype(np.float64)
    lq, rq = nv_dequant(wo.left_q)[:k].T, nv_dequant(wo.right_q)[:k].T            # n x k (V), m x k (U)
    sig = wo.sigma.cpu().numpy().astype(np.float64)
    assert rel_fro(d_left.cpu().numpy().T, (dwn @ rq) * sig) < 1e-5
    assert rel_fro(d_right.cpu().numpy().T, (dwn.T @ lq) * sig) < 1e-5
    assert rel_fro(d_sigma.cpu().numpy(), np.einsum("jt,ji,it->t", lq, dwn, rq)) < 1e-5
    # (b) end to end against the oracle's own split, quantization and weight gradient
    xq = olay.quantize_operand(x, k, p, osp.MODE_SAMPLED, 1)
    wq = olay.quantize_operand(w, k, p, osp.MODE_FULL, 2)
    dq = olay.quantize_operand(d, k, p, osp.MODE_SAMPLED, 3, onv.ROUND_SR)
    du, ds, dv = olay.factor_grads(olay.linear_wgrad(dq, xq), wq)
    base = TOL if dw_dtype == torch.float32 else 3 * TOL                          # a BF16 dw carries 2^-9 per entry
    _check_e2e("factor_gradients_256tok_448to192_k12_dw_%s" % ("fp32" if dw_dtype == torch.float32 else "bf16"),
               {"dU": rel_fro(d_right.cpu().numpy().T, du), "dV": rel_fro(d_left.cpu().numpy().T, dv),
                "dS": rel_fro(d_sigma.cpu().numpy(), ds)}, (xo, xq), (wo, wq), (do, dq), base_tol=base)


@pytest.mark.parametrize("l,n,m,k,dtype,pad", [
    (128, 64, 64, 4, torch.float32, 0),            # one strip, one ragged chunk, the smallest rank
    (128, 320, 2112, 20, torch.float32, 2),        # rows that start off the 16-byte boundary: element loads
    (128, 2112, 320, 36, torch.bfloat16, 2),
    (256, 1088, 960, 64, torch.bfloat16, 0),
    (256, 576, 1024, 68, torch.float32, 0),        # more than 64 vectors: a second pass with four of them
    (256, 9536, 192, 8, torch.float32, 0),         # a long contraction for few columns: clusters of eight
])
def test_factor_gradient_strips_and_chunks(ctx, l, n, m, k, dtype, pad):
    """The contractions against float64 from the library's own dw and factors.  Every product is exact and a partial sum runs
    over at most a few hundred FP32 additions of at most twelve tensor-core adds each: 2e-6 of the result in norm."""
    from gpu_util import rel_fro, nv_dequant
    B, h = ctx
    torch.manual_seed(n + k)
    xo = h.split(torch.randn(l, m, device="cuda").to(torch.bfloat16), 0, 0)
    do = h.split(torch.randn(l, n, device="cuda").to(torch.bfloat16), 0, 0)
    wo = B.Operand(n, m, k)
    wo.left_q, wo.right_q = h.quantize_nvfp4(torch.randn(k, n, device="cuda"))[0], h.quantize_nvfp4(torch.randn(k, m, device="cuda"))[0]
    wo.sigma.copy_(torch.rand(k, device="cuda") + 0.5)
    fg = (torch.full((k, n), float("nan"), device="cuda"), torch.full((k,), float("nan"), device="cuda"), torch.full((k, m), float("nan"), device="cuda"))
    dw = torch.empty((n, m + pad), dtype=dtype, device="cuda")[:, :m]
    h.linear_bwd(do, xo, wo, need_dx=False, out=(None, dw), factor_grads=fg)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    dwn = dw.float().cpu().numpy().astype(np.float64)
    lq, rq, sig = nv_dequant(wo.left_q)[:k].T, nv_dequant(wo.right_q)[:k].T, wo.sigma.cpu().numpy().astype(np.float64)
    assert rel_fro(fg[0].cpu().numpy().T, (dwn @ rq) * sig) < 2e-6
    assert rel_fro(fg[2].cpu().numpy().T, (dwn.T @ lq) * sig) < 2e-6
    assert rel_fro(fg[1].cpu().numpy(), np.einsum("jt,ji,it->t", lq, dwn, rq)) < 1e-5


@pytest.mark.parametrize("l,n,m,k,dtype,pad", [
    (64, 64, 9280, 8, torch.float32, 0),           # ten chunks per CTA, the last one half: the ring goes round twice
    (64, 9280, 128, 24, torch.bfloat16, 0),
    (64, 192, 9280, 48, torch.float32, 2),
])
def test_factor_gradients_of_a_long_contraction(ctx, l, n, m, k, dtype, pad):
    """More chunks per CTA than the ring holds, in both directions; the bounds of the test above."""
    test_factor_gradient_strips_and_chunks(ctx, l, n, m, k, dtype, pad)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("peak", [3.4e38, 1e39])
def test_factor_gradients_of_an_overflowing_weight_gradient(ctx, dtype, peak):
    """Entries of dW that are infinite, or finite in FP32 and infinite in BF16: alone in a row or column, two of the same and two of
    opposite sign in one, in the first and the last chunk.  The gradients are what FP32 products and sums give: infinite, a NaN
    only for 0 * inf and inf - inf, finite where the factor's entry keeps them so, and untouched elsewhere."""
    from gpu_util import rel_fro, nv_to_numpy, nv_dequant
    B, h = ctx
    l, n, m, k = 128, 320, 448, 20
    rng = np.random.default_rng(5)
    spots = [(3, 5, 1), (64, 200, -1), (64, 447, -1), (130, 17, 1), (130, 260, -1), (319, 128, 1), (200, 300, 1), (210, 300, 1), (220, 310, -1), (221, 310, 1)]
    dy, x = np.zeros((l, n), dtype=np.float32), np.zeros((l, m), dtype=np.float32)
    dy[len(spots):] = 1e-4 * rng.standard_normal((l - len(spots), n)); x[len(spots):] = 1e-4 * rng.standard_normal((l - len(spots), m))
    for t, (r, c, sgn) in enumerate(spots):
        dy[t, r], x[t, c] = sgn, 1.0
    do, xo = (h.split(torch.from_numpy(a).cuda().to(torch.bfloat16), 0, 0) for a in (dy, x))
    xo.res_by_rows.tensor_scale.fill_(1.0)
    do.res_by_rows.tensor_scale.fill_(peak / 2688.0 ** 2)          # both maxima are stored as 448 * 6
    torch.manual_seed(3)
    wo = B.Operand(n, m, k)
    wo.left_q, wo.right_q = h.quantize_nvfp4(torch.randn(k, n, device="cuda"))[0], h.quantize_nvfp4(torch.randn(k, m, device="cuda"))[0]
    wo.sigma.copy_(torch.rand(k, device="cuda") + 0.5)
    fg = (torch.empty((k, n), device="cuda"), torch.empty(k, device="cuda"), torch.empty((k, m), device="cuda"))
    dw = torch.empty((n, m), dtype=dtype, device="cuda")
    h.linear_bwd(do, xo, wo, need_dx=False, out=(None, dw), factor_grads=fg)
    torch.cuda.synchronize()
    dwn = dw.float().cpu().numpy().astype(np.float64)
    big = np.abs(dwn) > 3.39e38
    assert int(big.sum()) == len(spots) and bool(np.isinf(dwn[big]).all()) == (peak > 3.4e38 or dtype == torch.bfloat16)
    sig = wo.sigma.cpu().numpy().astype(np.float64)
    for got, fac, mat in ((fg[0], wo.right_q, dwn), (fg[2], wo.left_q, dwn.T)):
        codes, _, ts = nv_to_numpy(fac)
        unscaled = (nv_dequant(fac)[:k] / float(ts)).T              # the sums are over E2M1 * E4M3 values, the FP32 scales come last
        with np.errstate(invalid="ignore", over="ignore"):
            sums = np.zeros((mat.shape[0], k))
            for c in range(mat.shape[1]):                           # an FP32 sum that has overflowed stays infinite
                sums += mat[:, c:c + 1] * unscaled[c]
                sums = np.where(np.abs(sums) > 3.4028236e38, np.copysign(np.inf, sums), sums)
            want = sums * float(ts) * sig
            want = np.where(np.abs(want) > 3.4028236e38, np.copysign(np.inf, want), want)
        got = got.cpu().numpy().T.astype(np.float64)
        assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
        rows = np.abs(mat).max(axis=1) > 3.39e38
        fin = np.isfinite(want)
        assert np.isinf(want[rows]).any() and fin[~rows].all()
        assert rel_fro(got[~rows], want[~rows]) < 2e-6
        assert np.allclose(got[rows][fin[rows]], want[rows][fin[rows]], rtol=1e-5, atol=2e-6 * np.abs(want[~rows]).max())


def test_factor_gradients_need_the_weight_gradient(ctx):
    from gpu_util import to_dev_bf16
    B, h = ctx
    c = synth.config_small()
    xo = h.split(to_dev_bf16(c["x"]), 4, 4, sketch=B.SKETCH_FULL, seed=1)
    wo = h.split(to_dev_bf16(c["w"]), 4, 4, sketch=B.SKETCH_FULL, seed=2)
    do = h.split(torch.randn(128, 256, device="cuda").to(torch.bfloat16), 4, 4, sketch=B.SKETCH_FULL, seed=3)
    g = torch.zeros((4, 256), device="cuda")
    with pytest.raises(RuntimeError):
        h.linear_bwd(do, xo, wo, need_dw=False, factor_grads=(g, None, None))


@pytest.mark.parametrize("kp", [(12, 4), (24, 8), (40, 0), (48, 8), (64, 8)])
def test_rank_and_oversampling_range(ctx, kp):
    """Ranks that are not multiples of 16 (padded coefficient blocks), no oversampling, and the largest rank."""
    from gpu_util import to_dev_bf16, rel_fro
    B, h = ctx
    k, p = kp
    l, m, n = 512, 768, 640
    x, _ = synth.llama_like(l, m, 1.0, 91, rank=max(k, 8))
    w, _ = synth.llama_like(n, m, 0.02, 92, rank=max(k, 8))
    d, _ = synth.llama_like(l, n, 1e-4, 93, rank=max(k, 8))
    xo = h.split(to_dev_bf16(x), k, p, sketch=B.SKETCH_SAMPLED, seed=1)
    wo = h.split(to_dev_bf16(w), k, p, sketch=B.SKETCH_FULL, seed=2)
    do = h.split(to_dev_bf16(d), k, p, sketch=B.SKETCH_SAMPLED, seed=3, rounding=B.ROUND_SR)
    y = h.linear_fwd(xo, wo)
    dx, dw = h.linear_bwd(do, xo, wo)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    xq = olay.quantize_operand(x, k, p, osp.MODE_SAMPLED, 1)
    wq = olay.quantize_operand(w, k, p, osp.MODE_FULL, 2)
    dq = olay.quantize_operand(d, k, p, osp.MODE_SAMPLED, 3, onv.ROUND_SR)
    for op, q in ((xo, xq), (wo, wq), (do, dq)):
        assert np.max(np.abs(op.sigma.cpu().numpy()[:k] - q.sigma) / q.sigma) < 1e-3
    _check_e2e("rank_range_512tok_768to640_k%d_p%d" % (k, p),
               {"y": rel_fro(y.cpu().numpy(), olay.linear_fwd(xq, wq)), "dx": rel_fro(dx.cpu().numpy(), olay.linear_dgrad(dq, wq)),
                "dw": rel_fro(dw.cpu().numpy(), olay.linear_wgrad(dq, xq))}, (xo, xq), (wo, wq), (do, dq))


def test_ragged_layer_through_the_two_cta_gemm(ctx):
    """l, m, n above 256 but not multiples of the 256-wide GEMM tiles: ragged tiles in every product, the fused
    low-rank correction boxes, tensor stores clipped at the matrix edge."""
    from gpu_util import to_dev_bf16, rel_fro
    B, h = ctx
    l, m, n, k, p = 320, 448, 320, 8, 4
    x, _ = synth.llama_like(l, m, 1.0, 81, rank=8)
    w, _ = synth.llama_like(n, m, 0.02, 82, rank=8)
    d, _ = synth.llama_like(l, n, 1e-4, 83, rank=8)
    xo = h.split(to_dev_bf16(x), k, p, sketch=B.SKETCH_SAMPLED, seed=1)
    wo = h.split(to_dev_bf16(w), k, p, sketch=B.SKETCH_FULL, seed=2)
    do = h.split(to_dev_bf16(d), k, p, sketch=B.SKETCH_SAMPLED, seed=3, rounding=B.ROUND_SR)
    y = h.linear_fwd(xo, wo)
    dx, dw = h.linear_bwd(do, xo, wo)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    lx, rxc, rxr = _oracle_from_gpu_operand(xo, k)
    lw, rwc, rwr = _oracle_from_gpu_operand(wo, k)
    ld, rdc, rdr = _oracle_from_gpu_operand(do, k)
    assert rel_fro(y.cpu().numpy(), (lx + rxc) @ (lw + rwc).T) < 2e-5
    assert rel_fro(dx.cpu().numpy(), (ld + rdc) @ (lw + rwr)) < 2e-5
    assert rel_fro(dw.cpu().numpy(), (ld + rdr).T @ (lx + rxr)) < 2e-5
    xq = olay.quantize_operand(x, k, p, osp.MODE_SAMPLED, 1)
    wq = olay.quantize_operand(w, k, p, osp.MODE_FULL, 2)
    dq = olay.quantize_operand(d, k, p, osp.MODE_SAMPLED, 3, onv.ROUND_SR)
    _check_e2e("ragged_320tok_448to320_k8",
               {"y": rel_fro(y.cpu().numpy(), olay.linear_fwd(xq, wq)), "dx": rel_fro(dx.cpu().numpy(), olay.linear_dgrad(dq, wq)),
                "dw": rel_fro(dw.cpu().numpy(), olay.linear_wgrad(dq, xq))}, (xo, xq), (wo, wq), (do, dq))


@pytest.mark.parametrize("l,n,m,kd,kx,kw", [
    (64, 192, 64, 4, 4, 4),               # one K block of each product, a residual product with an odd number of 64-column tiles
    (128, 448, 192, 8, 12, 4),            # residual product in the group, unequal ranks
    (320, 2112, 576, 36, 32, 40),         # 33-vector remainders of the finishing kernel, ragged K
    (512, 256, 4160, 16, 16, 16),         # contractions of 17 K blocks divided by eight, of one and of two beside them
    (4096, 256, 320, 64, 48, 64),         # 64 vectors beside 48: two 32-vector groups, one row per warp
    (9216, 256, 256, 16, 20, 12), (9216, 256, 256, 40, 36, 64),           # two rows per warp (from 7105 rows on), one and two 32-vector groups
    (19200, 256, 256, 16, 20, 12), (19200, 256, 256, 40, 36, 64),         # four rows per warp (from 14209 on); more CTAs than SMs: four stages, two CTAs an SM
    (256, 512, 768, 72, 64, 64),          # a rank above 64 beside ranks below it
    (1024, 4096, 4096, 128, 100, 128),    # ranks above 64 whose contractions would fill a second round of CTAs
])
def test_skinny_products_in_one_launch(ctx, l, n, m, kd, kx, kw):
    """Forward and both gradients against float64 products of the library's own codes (exact codes, FP32 sums: 2e-5)."""
    from gpu_util import to_dev_bf16, rel_fro
    B, h = ctx
    t = [synth.planted(r, c, 8, 100 * s * (np.sqrt(r) + np.sqrt(c)), 10 * s * (np.sqrt(r) + np.sqrt(c)), s, sd)[0]
         for r, c, s, sd in ((l, m, 1.0, 71), (n, m, 0.02, 72), (l, n, 1e-4, 73))]
    xo, wo, do = (h.split(to_dev_bf16(a), k, 4, sketch=B.SKETCH_FULL, seed=i) for i, (a, k) in enumerate(zip(t, (kx, kw, kd))))
    y = h.linear_fwd(xo, wo)
    dx, dw = h.linear_bwd(do, xo, wo)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    lx, rxc, rxr = _oracle_from_gpu_operand(xo, kx)
    lw, rwc, rwr = _oracle_from_gpu_operand(wo, kw)
    ld, rdc, rdr = _oracle_from_gpu_operand(do, kd)
    assert rel_fro(y.cpu().numpy(), (lx + rxc) @ (lw + rwc).T) < 2e-5
    assert rel_fro(dx.cpu().numpy(), (ld + rdc) @ (lw + rwr)) < 2e-5
    assert rel_fro(dw.cpu().numpy(), (ld + rdr).T @ (lx + rxr)) < 2e-5


@pytest.mark.parametrize("side", ["x", "w", "dy"])
@pytest.mark.parametrize("rows,k", [(7107, 32), (7107, 48), (14211, 12), (14211, 64), (16386, 32)])
def test_plain_operand_of_any_number_of_rows_beside_a_factored_one(ctx, side, rows, k):
    """metis_quantize_nvfp4 takes any number of rows, so a plain activation, weight or gradient may leave the finishing kernel (two rows a warp
    from 7105 on, four from 14209 on) a warp that the extent cuts.  Products against float64 ones of the library's own codes, in a workspace of exactly the
    plan's bytes between guard bytes."""
    from gpu_util import to_dev_bf16, rel_fro, nv_dequant, Guarded
    B, h = ctx
    few, inner = 320, 256
    t = synth.planted(rows, inner, 8, 100 * (np.sqrt(rows) + 16), 10 * (np.sqrt(rows) + 16), 1.0, 75)[0]
    plain = B.Operand(rows, inner, 0, B.BLOCKS_ALONG_COLS)
    plain.res_by_cols, _ = h.quantize_nvfp4(to_dev_bf16(t), axes=B.BLOCKS_ALONG_COLS)
    shape = (inner, few) if side == "dy" else (few, inner)
    wide = h.split(to_dev_bf16(synth.planted(*shape, 8, 60.0, 6.0, 0.02, 76)[0]), k, 4, sketch=B.SKETCH_FULL, seed=3)
    low, by_cols, by_rows = _oracle_from_gpu_operand(wide, k)
    q = nv_dequant(plain.res_by_cols)
    kx, up = (2 * k + 63) // 64 * 64, lambda n: (n + 255) // 256 * 256
    ws = Guarded((4 * 64 * 64 + sum(up(4 * r * k) + up(2 * r * kx) for r in (rows, few)),), torch.uint8)
    own, h.workspace = h.workspace, lambda n: ws.view
    try:
        if side == "dy":
            got, _ = h.linear_bwd(plain, None, wide, need_dw=False)
            want = q @ (low + by_rows)
        elif side == "x":
            got, want = h.linear_fwd(plain, wide), q @ (low + by_cols).T
        else:
            got, want = h.linear_fwd(wide, plain), (low + by_cols) @ q.T
        torch.cuda.synchronize()
    finally:
        h.workspace = own
    assert h.device_status() == 0
    assert rel_fro(got.cpu().numpy(), want) < 2e-5
    ws.check("workspace")


def test_wide_rank_beside_more_columns_than_a_grid_has_rows_of_blocks(ctx):
    """A product of few rows (256) and 2^22 columns at a rank above 64: the tiled step on the rows' operand counts its blocks by the rows.  The
    first and the last 256 columns are, bit for bit, those of the same call on a weight of these rows alone."""
    B, h = ctx
    l, n, m, k = 256, 1 << 22, 64, 72
    g = torch.Generator(device="cuda").manual_seed(77)
    xo, wo = B.Operand(l, m, 0, B.BLOCKS_ALONG_COLS), B.Operand(n, m, k, B.BLOCKS_ALONG_COLS)
    for t in (xo.res_by_cols, wo.res_by_cols, wo.left_q, wo.right_q):
        t.codes.random_(0, 256, generator=g)
        t.scales.random_(0x28, 0x40, generator=g)
        t.tensor_scale.fill_(0.01)
    wo.sigma.uniform_(0.5, 2.0, generator=g)

    def part(rows):
        p = B.Operand(256, m, k, B.BLOCKS_ALONG_COLS)
        p.right_q, p.sigma = wo.right_q, wo.sigma
        p.res_by_cols.codes, p.left_q.codes = wo.res_by_cols.codes[rows], wo.left_q.codes[:, rows.start // 2: rows.stop // 2].contiguous()
        p.res_by_cols.scales, p.left_q.scales = (t.scales[rows.start * 4 * u: rows.stop * 4 * u] for t, u in ((wo.res_by_cols, 1), (wo.left_q, 2)))
        p.res_by_cols.tensor_scale, p.left_q.tensor_scale = wo.res_by_cols.tensor_scale, wo.left_q.tensor_scale
        return h.linear_fwd(xo, p, out_dtype=torch.bfloat16)

    first, last = part(slice(0, 256)), part(slice(n - 256, n))
    ws = torch.empty(4 * 8192 + (n + l) * (4 * k + 2 * 192) + 2048, dtype=torch.uint8, device="cuda")
    own, h.workspace = h.workspace, lambda nbytes: ws
    try:
        y = h.linear_fwd(xo, wo, out_dtype=torch.bfloat16)
        torch.cuda.synchronize()
    finally:
        h.workspace = own
    assert h.device_status() == 0 and bool(torch.isfinite(first).all()) and float(first.float().std()) > 0
    assert torch.equal(y[:, :256], first) and torch.equal(y[:, n - 256:], last)


@pytest.mark.parametrize("kd,kx", [(256, 256), (0, 256), (256, 8)])
def test_rank_256_products_of_long_and_deep_operands(ctx, kd, kx):
    """From 8192 rows and 2^26 residual elements on, the products with 256 factor vectors run beside the grouped ones, on two streams: weight
    gradient of operands with random codes against their float64 product (exact codes, FP32 sums)."""
    B, h = ctx
    n = 8192
    g = torch.Generator(device="cuda").manual_seed(79)
    e2m1 = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64, device="cuda")

    def value(t):
        c = torch.stack((t.codes & 15, t.codes >> 4), dim=2).reshape(t.rows, -1).int()
        s = t.linear_scales().cuda().view(torch.float8_e4m3fn).double()
        return (e2m1[c].reshape(t.rows, -1, 16) * s[:, :, None]).reshape(t.rows, -1) * t.tensor_scale.double()

    def operand(k):
        op = B.Operand(n, n, k, B.BLOCKS_ALONG_ROWS)
        for t, scale in ((op.res_by_rows, 0.01), (op.left_q, 0.003), (op.right_q, 0.003)):
            t.codes.random_(0, 256, generator=g)
            t.scales.random_(0x28, 0x40, generator=g)
            t.tensor_scale.fill_(scale)
        op.sigma.uniform_(0.5, 2.0, generator=g)
        v = value(op.res_by_rows).T
        return op, v + (value(op.left_q).T * op.sigma.double()) @ value(op.right_q) if k else v

    do, d = operand(kd)
    xo, x = operand(kx)
    _, dw = h.linear_bwd(do, xo, None, need_dx=False)
    torch.cuda.synchronize()
    assert h.device_status() == 0
    want = d.T @ x
    assert float((dw.double() - want).norm() / want.norm()) < 2e-5


def test_bf16_output(ctx):
    from gpu_util import to_dev_bf16, rel_fro
    B, h = ctx
    c = synth.config_small()
    xo = h.split(to_dev_bf16(c["x"]), 4, 4, sketch=B.SKETCH_FULL, seed=1)
    wo = h.split(to_dev_bf16(c["w"]), 4, 4, sketch=B.SKETCH_FULL, seed=2)
    y32 = h.linear_fwd(xo, wo)
    y16 = h.linear_fwd(xo, wo, out_dtype=torch.bfloat16)
    torch.cuda.synchronize()
    assert rel_fro(y16.float().cpu().numpy(), y32.cpu().numpy()) < 4e-3


def test_repeated_calls_are_bit_identical(ctx):
    """Same inputs, same seeds: every byte of every output is the same from call to call.  The decomposition, the
    forward and the backward fork into the handle's side streams (the backward into all of them), so a missing join
    or a shared intermediate would show up here as a changed bit."""
    from gpu_util import to_dev_bf16
    B, h = ctx
    l, m, n, k, p = 1024, 768, 512, 16, 8
    x, _ = synth.llama_like(l, m, 1.0, 61, rank=16)
    w, _ = synth.llama_like(n, m, 0.02, 62, rank=16)
    d, _ = synth.llama_like(l, n, 1e-4, 63, rank=16)
    xd, wd, dd = to_dev_bf16(x), to_dev_bf16(w), to_dev_bf16(d)

    def run():
        xo = h.split(xd, k, p, sketch=B.SKETCH_SAMPLED, seed=1)
        wo = h.split(wd, k, p, sketch=B.SKETCH_FULL, seed=2)
        do = h.split(dd, k, p, sketch=B.SKETCH_SAMPLED, seed=3, rounding=B.ROUND_SR)
        y = h.linear_fwd(xo, wo, out_dtype=torch.bfloat16)
        dx, dw = h.linear_bwd(do, xo, wo)
        torch.cuda.synchronize()
        return [y, dx, dw, xo.left, xo.right, xo.sigma, do.res_by_cols.codes, do.res_by_rows.codes, wo.left_q.codes]

    first = [t.clone() for t in run()]
    for _ in range(5):
        again = run()
        assert all(torch.equal(a, b) for a, b in zip(first, again))
    assert h.device_status() == 0


def test_concurrent_step_replayed_many_times_is_bit_identical():
    """The whole step of a 4096-token layer - three decompositions on three streams, forward and backward - captured
    once and replayed 1500 times: every replay must reproduce the first one bit for bit.  Kernels of different
    operands overlap differently from replay to replay, which is what exposes a missing ordering between a buffer's
    readers and the copy that refills it (such a gap once let one step in a few hundred through with a 32 x 8 patch of
    wrong residual values)."""
    from paper_2509_00404_b200 import binding as B
    l = m = n = 4096
    k, p = 32, 8
    x, w, d = synth.planted_device(l, m, 32, 1.0, 11), synth.planted_device(n, m, 32, 0.02, 12), synth.planted_device(l, n, 32, 1e-4, 13)
    hx, hw, hd = B.Handle(0), B.Handle(0), B.Handle(0)
    try:
        xo, wo, do = B.Operand(l, m, k), B.Operand(n, m, k), B.Operand(l, n, k)
        y = torch.empty((l, n), dtype=torch.bfloat16, device="cuda")
        dx, dw = torch.empty((l, m), dtype=torch.bfloat16, device="cuda"), torch.empty((n, m), dtype=torch.bfloat16, device="cuda")
        sw, sd = torch.cuda.Stream(), torch.cuda.Stream()
        e0, ew, ex, eb = (torch.cuda.Event() for _ in range(4))

        def step():
            main = torch.cuda.current_stream()
            e0.record(main); sw.wait_event(e0); sd.wait_event(e0)
            with torch.cuda.stream(sw):
                hw.split(w, k, p, sketch=B.SKETCH_FULL, seed=2, out=wo, stream=sw)
                ew.record(sw)
            hx.split(x, k, p, sketch=B.SKETCH_SAMPLED, seed=1, out=xo)
            ex.record(main)
            main.wait_event(ew)
            hx.linear_fwd(xo, wo, out=y)
            with torch.cuda.stream(sd):
                hd.split(d, k, p, sketch=B.SKETCH_SAMPLED, seed=3, rounding=B.ROUND_SR, out=do, stream=sd)
                sd.wait_event(ex); sd.wait_event(ew)
                hd.linear_bwd(do, xo, wo, out=(dx, dw), stream=sd)
                eb.record(sd)
            main.wait_event(eb)

        for _ in range(2):
            step()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            step()
        g.replay()
        torch.cuda.synchronize()
        watched = [y, dx, dw, xo.res_by_cols.codes, xo.res_by_rows.codes, wo.res_by_cols.codes, wo.res_by_rows.codes,
                   do.res_by_cols.codes, do.res_by_rows.codes, xo.res_by_cols.scales, do.res_by_rows.scales]
        first = [t.clone() for t in watched]
        bad = 0
        for _ in range(1500):
            g.replay()
            bad += int(not all(torch.equal(a, b) for a, b in zip(first, watched)))
        torch.cuda.synchronize()
        assert bad == 0, "%d of 1500 replays differ from the first" % bad
        assert (hx.device_status() | hw.device_status() | hd.device_status()) == 0
    finally:
        for h in (hx, hw, hd):
            h.close()
