"""Kernel-level parity of the CUDA library against the fp64 oracle (GPU only).

Each test calls one kernel through the C ABI of include/flglm_kernels.h on seeded
inputs that are exactly representable in bf16, and compares with the oracle's
function of the same step (or, for the plain contractions, with the fp64 product
that defines them).  Shapes span several tiles and a ragged tail.
"""

import numpy as np
import pytest
import torch

from oracle import flglm_oracle as O
from tests._gpu import (bits, dev_bf16, dev_f32, dev_i32, f64, flglm, need_gpu, rel_inf, rnd_bf16_f64,
                        rope_table)

pytestmark = pytest.mark.gpu

# bf16 output rounding is 2^-9 relative; fp32 accumulation over K adds far less.
GEMM_TOL = 1e-2


@pytest.fixture(scope="module")
def F():
    need_gpu()
    return flglm()


def _store(mat: np.ndarray, mn_major: bool):
    """Device copy of a logical [rows, K] operand: row-major as is (K-major), or its
    transpose [K, rows] (MN-major).  Returns (tensor, leading dim)."""
    if mn_major:
        t = dev_bf16(np.ascontiguousarray(mat.T))
        return t, mat.shape[0]
    return dev_bf16(mat), mat.shape[1]


TILES = ["auto", "128x128", "128x256", "pair"]


def tile_id(F, name):
    return {"auto": F.FL_TILE_AUTO, "128x128": F.FL_TILE_128x128, "128x256": F.FL_TILE_128x256,
            "pair": F.FL_TILE_256x256_PAIR}[name]


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("layout", [(0, 0), (0, 1), (1, 1)], ids=["fwd", "dgrad", "wgrad"])
@pytest.mark.parametrize("shape", [(200, 256, 320), (136, 384, 200), (1000, 1024, 512), (64, 128, 64),
                                   (8, 256, 4096), (520, 768, 72), (104, 512, 256), (4000, 4096, 520)])
def test_gemm_layouts(F, layout, shape, tile):
    """Every operand layout and tile shape.  (104, 512, 256): the odd CTA of a pair loads
    rows wholly past M; (4000, 4096, 520): several 256 x 256 tiles per CTA pair, so both
    accumulator buffers and the 6-stage ring wrap, with a ragged last k-block."""
    M, N, K = shape
    a_mn, b_mn = layout
    if tile in ("128x256", "pair") and N % 256:
        pytest.skip("256-column tiles need N % 256 == 0")
    rng = np.random.default_rng(M * 7 + N + K + 31 * a_mn + 17 * b_mn)
    A = rnd_bf16_f64(rng, (M, K))
    B = rnd_bf16_f64(rng, (N, K))
    dA, lda = _store(A, bool(a_mn))
    dB, ldb = _store(B, bool(b_mn))
    D = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    F.gemm(M, N, K, dA, lda, a_mn, dB, ldb, b_mn, D, N, tile=tile_id(F, tile))
    torch.cuda.synchronize()
    ref = A @ B.T
    assert rel_inf(f64(D), ref) < GEMM_TOL


def test_gemm_accumulate_f32_repeated(F):
    """fp32 read-modify-write epilogue (weight gradients accumulate across calls)."""
    M, N, K = 384, 512, 300
    rng = np.random.default_rng(5)
    A = rnd_bf16_f64(rng, (M, K))
    B = rnd_bf16_f64(rng, (N, K))
    C0 = rng.standard_normal((M, N)).astype(np.float32)
    dA, lda = _store(A, True)
    dB, ldb = _store(B, True)
    D = dev_f32(C0)
    for _ in range(2):
        F.gemm(M, N, K, dA, lda, 1, dB, ldb, 1, D, N, epilogue=F.FL_EPI_ACCUM_F32)
    torch.cuda.synchronize()
    ref = C0.astype(np.float64) + 2 * (A @ B.T)
    assert rel_inf(f64(D), ref) < 1e-5


@pytest.mark.parametrize("tile", ["auto", "pair"])
def test_gemm_epilogues(F, tile):
    M, N, K = 192, 512, 256
    t = tile_id(F, tile)
    rng = np.random.default_rng(11)
    A = rnd_bf16_f64(rng, (M, K))
    B = rnd_bf16_f64(rng, (N, K), 0.1)
    bias = rng.standard_normal(N).astype(np.float32)
    R = rnd_bf16_f64(rng, (M, N))
    dA, lda = _store(A, False)
    dB, ldb = _store(B, False)
    db = dev_f32(bias)
    dR = dev_bf16(R)
    acc = A @ B.T
    alpha = 1.7
    # bias + gelu, pre-activation kept
    D = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    U = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_BIAS_GELU, bias=db, aux_out=U, ld_aux_out=N)
    torch.cuda.synchronize()
    u = acc + bias[None, :]
    assert rel_inf(f64(U), u) < GEMM_TOL
    assert rel_inf(f64(D), O.gelu(u)) < GEMM_TOL
    # bias + alpha * residual
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_BIAS_RESID, bias=db, aux=dR, ld_aux=N,
           alpha=alpha)
    torch.cuda.synchronize()
    assert rel_inf(f64(D), u + alpha * R) < GEMM_TOL
    # alpha * residual, no bias
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_RESID, aux=dR, ld_aux=N, alpha=alpha)
    torch.cuda.synchronize()
    assert rel_inf(f64(D), acc + alpha * R) < GEMM_TOL
    # gelu' of a stored pre-activation; its column sums added to a vector (the up-projection
    # bias gradient of the backward)
    c0 = rng.standard_normal(N).astype(np.float32)
    cs = dev_f32(c0)
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_GELU_BWD, aux=dR, ld_aux=N, colsum=cs)
    torch.cuda.synchronize()
    du = acc * O.gelu_grad(R)
    assert rel_inf(f64(D), du) < GEMM_TOL
    assert rel_inf(f64(cs) - c0, du.sum(axis=0)) < 1e-4
    # plain store with bias
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_STORE, bias=db)
    torch.cuda.synchronize()
    assert rel_inf(f64(D), u) < GEMM_TOL


@pytest.mark.parametrize("tile", ["auto", "pair"])
@pytest.mark.parametrize("hd", [64, 128])
def test_gemm_rope_epilogue(F, hd, tile):
    nh = 2
    H = nh * hd
    M, N, K = 130, 3 * H, 256
    if tile == "pair" and N % 256:
        pytest.skip("256-column tiles need N % 256 == 0")
    rng = np.random.default_rng(hd)
    A = rnd_bf16_f64(rng, (M, K))
    B = rnd_bf16_f64(rng, (N, K), 0.1)
    bias = rng.standard_normal(N).astype(np.float32)
    pos = rng.integers(0, 300, size=M).astype(np.int32)
    rd = hd // 2
    tab = rope_table(300, rd, 10000.0)
    dA, lda = _store(A, False)
    dB, ldb = _store(B, False)
    D = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, epilogue=F.FL_EPI_BIAS_ROPE, bias=dev_f32(bias),
           pos=dev_i32(pos), rope_tab=dev_f32(tab), n_heads=nh, head_dim=hd, rotary_dim=rd, tile=tile_id(F, tile))
    torch.cuda.synchronize()
    qkv = A @ B.T + bias[None, :]
    cos, sin = O.rope_cos_sin(pos, rd, 10000.0)
    q = O.rope_rotate(qkv[:, :H].reshape(M, nh, hd), cos, sin, rd).reshape(M, H)
    k = O.rope_rotate(qkv[:, H:2 * H].reshape(M, nh, hd), cos, sin, rd).reshape(M, H)
    ref = np.concatenate([q, k, qkv[:, 2 * H:]], axis=1)
    assert rel_inf(f64(D), ref) < GEMM_TOL


@pytest.mark.parametrize("H", [256, 768, 3072, 4096])  # 768: one chunk per thread; 3072: six warps
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_layernorm_fwd_bwd(F, H, dtype):
    T = 77
    rng = np.random.default_rng(H + (dtype == "f32"))
    if dtype == "f32":
        x = (2.0 * rng.standard_normal((T, H))).astype(np.float32).astype(np.float64)
        dev_io = dev_f32
        dt = F.FL_DT_F32
    else:
        x = rnd_bf16_f64(rng, (T, H), 2.0)
        dev_io = dev_bf16
        dt = F.FL_DT_BF16
    g = (1 + 0.2 * rng.standard_normal(H)).astype(np.float32)
    be = (0.2 * rng.standard_normal(H)).astype(np.float32)
    dx_, dg_, db_ = dev_io(x), dev_f32(g), dev_f32(be)
    y = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    mean = torch.empty(T, dtype=torch.float32, device="cuda")
    rstd = torch.empty(T, dtype=torch.float32, device="cuda")
    F.fl_k_layernorm_fwd(T, H, dx_, dg_, db_, 1e-5, y, mean, rstd, x_dtype=dt)
    torch.cuda.synchronize()
    yr, mur, rsr = O.layer_norm_fwd(x, g.astype(np.float64), be.astype(np.float64), 1e-5)
    assert rel_inf(f64(y), yr) < 1e-2
    np.testing.assert_allclose(f64(mean), mur, rtol=0, atol=1e-5)
    np.testing.assert_allclose(f64(rstd), rsr, rtol=1e-4)
    # backward, with and without the alpha-scaled residual gradient; bf16 and fp32 dx
    if dtype == "f32":
        dy = rng.standard_normal((T, H)).astype(np.float32).astype(np.float64)
        res = rng.standard_normal((T, H)).astype(np.float32).astype(np.float64)
    else:
        dy = rnd_bf16_f64(rng, (T, H))
        res = rnd_bf16_f64(rng, (T, H))
    ws = torch.empty(F.fl_k_layernorm_bwd_workspace(T, H) // 4 + 64, dtype=torch.float32, device="cuda")
    for use_res in (False, True):
        dxo = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
        dxf = torch.empty((T, H), dtype=torch.float32, device="cuda")
        dgam = dev_f32(np.full(H, 0.5, np.float32))
        dbet = dev_f32(np.full(H, -0.25, np.float32))
        F.fl_k_layernorm_bwd(T, H, dev_io(dy), dx_, mean, rstd, dg_, dev_io(res) if use_res else None, 3.0,
                             dxo, dgam, dbet, ws, io_dtype=dt, dx_f32=dxf)
        torch.cuda.synchronize()
        dxr, dgr, dbr = O.layer_norm_bwd(dy, x, mur, rsr, g.astype(np.float64))
        if use_res:
            dxr = dxr + 3.0 * res
        assert rel_inf(f64(dxo), dxr) < 1e-2
        assert rel_inf(f64(dxf), dxr) < 1e-4
        assert rel_inf(f64(dgam) - 0.5, dgr) < 1e-4
        assert rel_inf(f64(dbet) + 0.25, dbr) < 1e-4


def test_layernorm_unsupported_widths(F):
    """Hidden sizes the forward has no launch shape for (an odd multiple of 256 above 2048, a
    width not a multiple of 256) and a negative row count are refused before any launch."""
    H = 2304
    x = torch.zeros((4, 4096), dtype=torch.bfloat16, device="cuda")
    v = torch.zeros(4096, device="cuda")
    y = torch.full((4, 4096), 1.0, dtype=torch.bfloat16, device="cuda")
    st = torch.zeros(4, device="cuda")
    for h, code in ((H, -7), (200, -7)):
        with pytest.raises(F.FlError) as ei:
            F.fl_k_layernorm_fwd(4, h, x, v, v, 1e-5, y, st, st)
        assert ei.value.code == code
    with pytest.raises(F.FlError) as ei:
        F.fl_k_layernorm_fwd(-1, 256, x, v, v, 1e-5, y, st, st)
    assert ei.value.code == -1
    torch.cuda.synchronize()
    assert (y == 1.0).all() and not st.any()


@pytest.mark.parametrize("tile", ["auto", "pair"])
def test_gemm_fp32_residual_epilogues(F, tile):
    """fp32 residual stream: D fp32 = acc + bias + alpha * R, with R an fp32 tensor or its
    LayerNorm recomputed in fp32 from the row statistics."""
    M, N, K = 200, 512, 256
    t = tile_id(F, tile)
    rng = np.random.default_rng(12)
    A = rnd_bf16_f64(rng, (M, K))
    B = rnd_bf16_f64(rng, (N, K), 0.1)
    bias = rng.standard_normal(N).astype(np.float32)
    X = (3.0 * rng.standard_normal((M, N)) + 0.5).astype(np.float32)
    g = (1 + 0.2 * rng.standard_normal(N)).astype(np.float32)
    be = (0.2 * rng.standard_normal(N)).astype(np.float32)
    _, mu, rs = O.layer_norm_fwd(X.astype(np.float64), g.astype(np.float64), be.astype(np.float64), 1e-5)
    dA, lda = _store(A, False)
    dB, ldb = _store(B, False)
    acc = A @ B.T
    D = torch.empty((M, N), dtype=torch.float32, device="cuda")
    dX = dev_f32(X)
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_BIAS_RESID, bias=dev_f32(bias), aux=dX, ld_aux=N,
           alpha=7.5, aux_dtype=F.FL_DT_F32, d_dtype=F.FL_DT_F32)
    torch.cuda.synchronize()
    assert rel_inf(f64(D), acc + bias[None, :] + 7.5 * X) < 1e-5
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_BIAS_RESID, bias=dev_f32(bias), aux=dX, ld_aux=N,
           alpha=7.5, aux_dtype=F.FL_DT_F32, d_dtype=F.FL_DT_F32, ln_mean=dev_f32(mu), ln_rstd=dev_f32(rs),
           ln_gamma=dev_f32(g), ln_beta=dev_f32(be))
    torch.cuda.synchronize()
    lnx = (X - mu[:, None]) * rs[:, None] * g[None, :] + be[None, :]
    assert rel_inf(f64(D), acc + bias[None, :] + 7.5 * lnx) < 1e-5
    F.gemm(M, N, K, dA, lda, 0, dB, ldb, 0, D, N, tile=t, epilogue=F.FL_EPI_RESID, aux=dX, ld_aux=N, alpha=-2.0,
           aux_dtype=F.FL_DT_F32, d_dtype=F.FL_DT_F32)
    torch.cuda.synchronize()
    assert rel_inf(f64(D), acc - 2.0 * X) < 1e-5


@pytest.mark.parametrize("hd", [64, 128])
def test_attention_fwd_bwd(F, hd):
    seqs = [1, 64, 100, 130, 7, 64, 200] + ([520, 1030] if hd == 128 else [])
    nh = 2
    H = nh * hd
    cu = np.cumsum([0] + seqs).astype(np.int32)
    T = int(cu[-1])
    rng = np.random.default_rng(hd + 3)
    qkv = rnd_bf16_f64(rng, (T, 3 * H))
    do = rnd_bf16_f64(rng, (T, H))
    dqkv_ = dev_bf16(qkv)
    dcu = dev_i32(cu)
    ntiles = F.fl_k_attention_tiles(cu)
    assert ntiles == sum((L + 63) // 64 for L in seqs)
    tiles = torch.empty(ntiles * 2, dtype=torch.int32, device="cuda")
    o = torch.full((T, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((nh, T), dtype=torch.float32, device="cuda")
    F.fl_k_attention_fwd(T, nh, hd, dqkv_, cu, dcu, tiles, o, lse)
    torch.cuda.synchronize()
    q = qkv[:, :H].reshape(T, nh, hd)
    k = qkv[:, H:2 * H].reshape(T, nh, hd)
    v = qkv[:, 2 * H:].reshape(T, nh, hd)
    o_ref, lse_ref = O.attention_fwd(q, k, v, cu)
    assert rel_inf(f64(o), o_ref.reshape(T, H)) < 2e-2
    np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=2e-2)
    # backward (inverse rotary rotation folded in, as the server uses it)
    rd = hd // 2
    pos = np.concatenate([np.arange(L) for L in seqs]).astype(np.int32)
    tab = rope_table(max(seqs), rd, 10000.0)
    delta = torch.empty((nh, T), dtype=torch.float32, device="cuda")
    dq = torch.full((T, 3 * H), float("nan"), dtype=torch.bfloat16, device="cuda")
    # the kernel differentiates through its own saved O (bf16), as the server does
    F.fl_k_attention_bwd(T, nh, hd, dqkv_, o, lse, dev_bf16(do), cu, dcu, tiles, delta, dev_f32(tab), rd, dq)
    torch.cuda.synchronize()
    dqr, dkr, dvr = O.attention_bwd(do.reshape(T, nh, hd), q, k, v, cu)
    cos, sin = O.rope_cos_sin(pos, rd, 10000.0)
    dq_ref = O.rope_rotate(dqr, cos, sin, rd, inverse=True).reshape(T, H)
    dk_ref = O.rope_rotate(dkr, cos, sin, rd, inverse=True).reshape(T, H)
    got = f64(dq)
    assert rel_inf(got[:, :H], dq_ref) < 5e-2
    assert rel_inf(got[:, H:2 * H], dk_ref) < 5e-2
    assert rel_inf(got[:, 2 * H:], dvr.reshape(T, H)) < 5e-2


def test_adamw(F):
    n = 4096 + 64
    rng = np.random.default_rng(9)
    w = rng.standard_normal(n).astype(np.float32) * 0.02
    m = np.zeros(n, np.float32)
    v = np.zeros(n, np.float32)
    dw, dm, dv = dev_f32(w), dev_f32(m), dev_f32(v)
    wb = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    ref_w, ref_m, ref_v = w.astype(np.float64), m.astype(np.float64), v.astype(np.float64)
    for t in range(1, 4):
        g = (rng.standard_normal(n) * 1e-3).astype(np.float32)
        dg = dev_f32(g)
        F.fl_k_adamw(n, dw, dg, dm, dv, wb, 1e-3, 0.9, 0.999, 1e-8, 0.01, 1 - 0.9 ** t, 1 - 0.999 ** t)
        torch.cuda.synchronize()
        # the C ABI carries the hyperparameters as fp32: the oracle gets the same values
        f = lambda x: float(np.float32(x))
        ref_w, ref_m, ref_v = O.adamw_update(ref_w, g.astype(np.float64), ref_m, ref_v, t, f(1e-3), f(0.9),
                                             f(0.999), f(1e-8), f(0.01))
        assert not f64(dg).any()
    assert rel_inf(f64(dw), ref_w) < 1e-5
    assert rel_inf(f64(dm), ref_m) < 1e-5
    assert rel_inf(f64(dv), ref_v) < 1e-5
    np.testing.assert_array_equal(bits(wb), bits(dw.to(torch.bfloat16)))


def test_colsum(F):
    T, N = 1000, 768
    rng = np.random.default_rng(2)
    x = rnd_bf16_f64(rng, (T, N))
    out = dev_f32(np.ones(N, np.float32))
    F.fl_k_colsum(T, N, dev_bf16(x), out)
    torch.cuda.synchronize()
    np.testing.assert_allclose(f64(out), 1.0 + x.sum(0), rtol=1e-5, atol=1e-4)


def test_pack_clients_bitexact(F):
    rng = np.random.default_rng(4)
    H = 256
    lens = [3, 1, 64, 17, 200]
    clients = [dev_bf16(rnd_bf16_f64(rng, (2, L, H))) for L in lens]
    nbytes = [c.numel() * 2 for c in clients]
    packed = torch.empty(sum(c.numel() for c in clients), dtype=torch.bfloat16, device="cuda")
    F.fl_k_pack_clients(clients, nbytes, packed, scatter=False)
    back = [torch.empty_like(c) for c in clients]
    F.fl_k_pack_clients(back, nbytes, packed, scatter=True)
    torch.cuda.synchronize()
    want = np.concatenate([bits(c).reshape(-1) for c in clients])
    np.testing.assert_array_equal(bits(packed), want)
    for a, b in zip(back, clients):
        np.testing.assert_array_equal(bits(a), bits(b))


@pytest.mark.parametrize("hd", [64, 128])
def test_attention_bwd_many_units(F, hd):
    """Many more (tile, head) units than SMs, so that every persistent backward CTA walks
    several units (the next unit's tiles loading while a unit's output leaves): every
    element of dqkv written (NaN-filled before), sampled heads against the oracle, and the
    rope table's alignment checked before any launch."""
    nh = 32 if hd == 128 else 40
    H = nh * hd
    seqs = [256] * 24 + [1, 130, 300, 77, 512, 64]
    cu = np.cumsum([0] + seqs).astype(np.int32)
    T = int(cu[-1])
    rng = np.random.default_rng(hd + 11)
    qkv = rnd_bf16_f64(rng, (T, 3 * H))
    do = rnd_bf16_f64(rng, (T, H))
    dqkv_, dcu = dev_bf16(qkv), dev_i32(cu)
    tiles = torch.empty(F.fl_k_attention_tiles(cu) * 2, dtype=torch.int32, device="cuda")
    o = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((nh, T), dtype=torch.float32, device="cuda")
    F.fl_k_attention_fwd(T, nh, hd, dqkv_, cu, dcu, tiles, o, lse)
    rd = hd // 2
    pos = np.concatenate([np.arange(L) for L in seqs]).astype(np.int32)
    tab = dev_f32(rope_table(max(seqs), rd, 10000.0))
    delta = torch.empty((nh, T), dtype=torch.float32, device="cuda")
    dq = torch.full((T, 3 * H), float("nan"), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(F.FlError, match="aligned"):
        F.fl_k_attention_bwd(T, nh, hd, dqkv_, o, lse, dev_bf16(do), cu, dcu, tiles, delta, tab.view(-1)[2:], rd, dq)
    F.fl_k_attention_bwd(T, nh, hd, dqkv_, o, lse, dev_bf16(do), cu, dcu, tiles, delta, tab, rd, dq)
    torch.cuda.synchronize()
    got = f64(dq)
    assert np.isfinite(got).all()
    cos, sin = O.rope_cos_sin(pos, rd, 10000.0)
    heads = [0, nh // 2 + 1, nh - 1]
    sel = lambda base: np.concatenate([np.arange(base + h * hd, base + (h + 1) * hd) for h in heads])
    q = qkv[:, sel(0)].reshape(T, len(heads), hd)
    k = qkv[:, sel(H)].reshape(T, len(heads), hd)
    v = qkv[:, sel(2 * H)].reshape(T, len(heads), hd)
    dos = do[:, sel(0)].reshape(T, len(heads), hd)
    dqr, dkr, dvr = O.attention_bwd(dos, q, k, v, cu)
    n = len(heads) * hd
    assert rel_inf(got[:, sel(0)], O.rope_rotate(dqr, cos, sin, rd, inverse=True).reshape(T, n)) < 5e-2
    assert rel_inf(got[:, sel(H)], O.rope_rotate(dkr, cos, sin, rd, inverse=True).reshape(T, n)) < 5e-2
    assert rel_inf(got[:, sel(2 * H)], dvr.reshape(T, n)) < 5e-2


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("seqs", [[256] * 10 + [1, 130], [256] * 6 + [1, 300, 130, 700], [128] * 11 + [1, 77, 64]])
def test_attention_bwd_unit_order(F, hd, seqs):
    """Units taken in a fixed stride (two tiles per segment at most) or handed out while the
    kernel runs (three and more), several per SM, probabilities and score gradients made in two
    passes or (one tile per segment, as short ones alone) in one: the bits of every segment alone."""
    nh = 16
    H, rd = nh * hd, hd // 2
    g = torch.Generator(device="cuda").manual_seed(hd + len(seqs))
    T = sum(seqs)
    qkv = torch.randn((T, 3 * H), generator=g, device="cuda").bfloat16()
    do = torch.randn((T, H), generator=g, device="cuda").bfloat16()
    tab = dev_f32(rope_table(max(seqs), rd, 10000.0))

    def backward(lens, qkv, do):
        cu = np.cumsum([0] + lens).astype(np.int32)
        T, dcu = int(cu[-1]), dev_i32(cu)
        tiles = torch.empty(F.fl_k_attention_tiles(cu) * 2, dtype=torch.int32, device="cuda")
        o = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
        lse, delta = torch.empty((2, nh, T), dtype=torch.float32, device="cuda")
        dq = torch.full((T, 3 * H), float("nan"), dtype=torch.bfloat16, device="cuda")
        F.fl_k_attention_fwd(T, nh, hd, qkv, cu, dcu, tiles, o, lse)
        F.fl_k_attention_bwd(T, nh, hd, qkv, o, lse, do, cu, dcu, tiles, delta, tab, rd, dq)
        torch.cuda.synchronize()
        return dq

    got, at = backward(seqs, qkv, do), 0
    for L in seqs:
        want = backward([L], qkv[at:at + L].clone(), do[at:at + L].clone())
        assert torch.isfinite(want).all()
        assert torch.equal(got[at:at + L].view(torch.int16), want.view(torch.int16)), L
        at += L


@pytest.mark.parametrize("hd", [64, 128])
def test_attention_forward_output_alignment(F, hd):
    """An output that is only 16-byte aligned takes the narrower stores: the same bits."""
    nh, lens = 4, [130, 1, 128, 40]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    T, H = int(cu[-1]), nh * hd
    g = torch.Generator(device="cuda").manual_seed(hd)
    qkv = torch.randn((T, 3 * H), generator=g, device="cuda").bfloat16()
    tiles = torch.empty(2 * F.fl_k_attention_tiles(cu), dtype=torch.int32, device="cuda")
    out = []
    for off in (0, 8):
        o = torch.zeros(T * H + 16, dtype=torch.bfloat16, device="cuda")[off:off + T * H]
        lse = torch.empty((nh, T), device="cuda")
        F.fl_k_attention_fwd(T, nh, hd, qkv, cu, dev_i32(cu), tiles, o, lse)
        out.append((bits(o), lse))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("hd,Lp", [(64, 16), (128, 100)])
def test_attention_with_prefix(F, hd, Lp):
    """P-tuning v2 prefix (App. A): every query also sees Lp prefix keys/values (one or two
    64-key tiles, the second partial); prefix gradients are summed over all segments."""
    seqs = [1, 64, 100, 7, 130]
    nh = 2
    H = nh * hd
    cu = np.cumsum([0] + seqs).astype(np.int32)
    T = int(cu[-1])
    rng = np.random.default_rng(hd + Lp)
    qkv = rnd_bf16_f64(rng, (T, 3 * H))
    pk = rnd_bf16_f64(rng, (Lp, H))
    pv = rnd_bf16_f64(rng, (Lp, H))
    do = rnd_bf16_f64(rng, (T, H))
    dqkv_, dcu = dev_bf16(qkv), dev_i32(cu)
    dpk_, dpv_ = dev_bf16(pk), dev_bf16(pv)
    tiles = torch.empty(F.fl_k_attention_tiles(cu) * 2, dtype=torch.int32, device="cuda")
    o = torch.full((T, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((nh, T), dtype=torch.float32, device="cuda")
    F.fl_k_attention_fwd(T, nh, hd, dqkv_, cu, dcu, tiles, o, lse, dpk_, dpv_, Lp)
    torch.cuda.synchronize()
    q = qkv[:, :H].reshape(T, nh, hd)
    k = qkv[:, H:2 * H].reshape(T, nh, hd)
    v = qkv[:, 2 * H:].reshape(T, nh, hd)
    ppk, ppv = pk.reshape(Lp, nh, hd), pv.reshape(Lp, nh, hd)
    o_ref, lse_ref = O.attention_fwd(q, k, v, cu, ppk, ppv)
    assert rel_inf(f64(o), o_ref.reshape(T, H)) < 2e-2
    np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=2e-2)
    delta = torch.empty((nh, T), dtype=torch.float32, device="cuda")
    dq = torch.full((T, 3 * H), float("nan"), dtype=torch.bfloat16, device="cuda")
    gpk = dev_f32(np.full((Lp, H), 0.25, np.float32))
    gpv = torch.zeros((Lp, H), dtype=torch.float32, device="cuda")
    F.fl_k_attention_bwd(T, nh, hd, dqkv_, o, lse, dev_bf16(do), cu, dcu, tiles, delta, None, 0, dq,
                         dpk_, dpv_, Lp, gpk, gpv)
    torch.cuda.synchronize()
    dqr, dkr, dvr, dpkr, dpvr = O.attention_bwd(do.reshape(T, nh, hd), q, k, v, cu, ppk, ppv)
    got = f64(dq)
    assert rel_inf(got[:, :H], dqr.reshape(T, H)) < 5e-2
    assert rel_inf(got[:, H:2 * H], dkr.reshape(T, H)) < 5e-2
    assert rel_inf(got[:, 2 * H:], dvr.reshape(T, H)) < 5e-2
    assert rel_inf(f64(gpk) - 0.25, dpkr.reshape(Lp, H)) < 5e-2   # accumulated onto the 0.25
    assert rel_inf(f64(gpv), dpvr.reshape(Lp, H)) < 5e-2


@pytest.mark.parametrize("nh,hd,seqs", [(16, 64, [70] * 11), (32, 128, [40] * 6), (4, 64, [9] * 39),
                                        (16, 128, [300, 1, 128, 5, 260, 129, 2])])
def test_attention_prefix_slices(F, nh, hd, seqs):
    """Prefix gradients where the query tiles do not divide into a slice per SM (11 tiles for 10
    slices, 6 for 5, 39 for 38 on 152 SMs), and with more slices times heads than SMs, whose units
    are handed out while the kernel runs: every tile's share, added once."""
    Lp, H = 24, nh * hd
    cu = np.cumsum([0] + seqs).astype(np.int32)
    T = int(cu[-1])
    rng = np.random.default_rng(nh + hd)
    qkv, do = rnd_bf16_f64(rng, (T, 3 * H)), rnd_bf16_f64(rng, (T, H))
    pk, pv = rnd_bf16_f64(rng, (Lp, H)), rnd_bf16_f64(rng, (Lp, H))
    dqkv_, dcu, dpk_, dpv_ = dev_bf16(qkv), dev_i32(cu), dev_bf16(pk), dev_bf16(pv)
    tiles = torch.empty(F.fl_k_attention_tiles(cu) * 2, dtype=torch.int32, device="cuda")
    o = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    lse, delta = torch.empty((2, nh, T), dtype=torch.float32, device="cuda")
    F.fl_k_attention_fwd(T, nh, hd, dqkv_, cu, dcu, tiles, o, lse, dpk_, dpv_, Lp)
    dq = torch.empty((T, 3 * H), dtype=torch.bfloat16, device="cuda")
    gpk, gpv = torch.zeros((2, Lp, H), dtype=torch.float32, device="cuda")
    F.fl_k_attention_bwd(T, nh, hd, dqkv_, o, lse, dev_bf16(do), cu, dcu, tiles, delta, None, 0, dq,
                         dpk_, dpv_, Lp, gpk, gpv)
    torch.cuda.synchronize()
    r = lambda x: x.reshape(-1, nh, hd)
    _, _, _, dpkr, dpvr = O.attention_bwd(r(do), r(qkv[:, :H]), r(qkv[:, H:2 * H]), r(qkv[:, 2 * H:]), cu, r(pk), r(pv))
    assert rel_inf(f64(gpk), dpkr.reshape(Lp, H)) < 5e-2
    assert rel_inf(f64(gpv), dpvr.reshape(Lp, H)) < 5e-2


@pytest.mark.parametrize("tile", ["auto", "pair"])
@pytest.mark.parametrize("M,N,K,mn", [(200, 384, 136, 1), (256, 512, 64, 1), (130, 256, 96, 0), (600, 1024, 520, 1)])
def test_gemm_adamw_epilogue(F, M, N, K, mn, tile):
    """The weight-gradient GEMM with the AdamW update in its epilogue equals the plain fp32
    gradient GEMM followed by the separate AdamW kernel: weights, moments and the bf16
    copy; ragged rows, every tile shape (N = 384 takes 128-column tiles)."""
    if tile == "pair" and N % 256:
        pytest.skip("256-column tiles need N % 256 == 0")
    rng = np.random.default_rng(M + N)
    A = rnd_bf16_f64(rng, (M, K))
    B = rnd_bf16_f64(rng, (N, K))
    dA, lda = _store(A, bool(mn))
    dB, ldb = _store(B, bool(mn))
    w0 = (0.05 * rng.standard_normal((M, N))).astype(np.float32)
    m0 = (0.01 * rng.standard_normal((M, N))).astype(np.float32)
    v0 = (1e-3 * rng.random((M, N))).astype(np.float32)
    lr, b1, b2, eps, wd, t = 1e-3, 0.9, 0.999, 1e-8, 0.01, 3
    bc1, bc2 = 1.0 - b1 ** t, 1.0 - b2 ** t
    # reference: g = A B^T stored in fp32, then fl_k_adamw
    g = torch.empty((M, N), dtype=torch.float32, device="cuda")
    F.gemm(M, N, K, dA, lda, mn, dB, ldb, mn, g, N, epilogue=F.FL_EPI_STORE_F32)
    wr, mr, vr = dev_f32(w0), dev_f32(m0), dev_f32(v0)
    wbr = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    F.fl_k_adamw(M * N, wr, g, mr, vr, wbr, lr, b1, b2, eps, wd, bc1, bc2)
    # fused
    wf, mf, vf = dev_f32(w0), dev_f32(m0), dev_f32(v0)
    wbf = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    ga = F.fl_gemm_args(M, N, K, F.ptr(dA), lda, mn, F.ptr(dB), ldb, mn, F.ptr(wf), N, F.FL_EPI_ADAMW)
    ga.aux_out, ga.ld_aux_out = F.ptr(wbf), N
    ga.adam_m, ga.adam_v = F.ptr(mf), F.ptr(vf)
    ga.lr, ga.beta1, ga.beta2, ga.eps, ga.weight_decay = lr, b1, b2, eps, wd
    ga.inv_bc1, ga.inv_bc2 = 1.0 / np.float32(bc1), 1.0 / np.float32(bc2)
    ga.tile = tile_id(F, tile)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    F.fl_k_gemm(ga, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for got, want in ((wf, wr), (mf, mr), (vf, vr)):
        assert rel_inf(f64(got), f64(want)) < 1e-5
    np.testing.assert_array_equal(bits(wbf), bits(wf.to(torch.bfloat16)))


@pytest.mark.parametrize("layout", [(0, 0), (0, 1), (1, 1)], ids=["fwd", "dgrad", "wgrad"])
@pytest.mark.parametrize("M,N,K", [(8, 128, 8), (72, 4096, 4040), (128, 4096, 4096), (136, 1280, 4168), (264, 4096, 136),
                                   (304, 4096, 200), (512, 4096, 1024), (520, 2176, 72)])
def test_gemm_picked_tile_bit_identical(F, M, N, K, layout):
    """The tile the library picks (narrow ones here: few tiles, ragged rows, odd and ragged
    counts of k-blocks) gives the bits of the 128 x 128 tile for every epilogue: each output
    sums over K in the same order whatever the tile, which client-batching relies on."""
    a_mn, b_mn = layout
    g = torch.Generator(device="cuda").manual_seed(M + N + K)

    def rnd(*shape, dt=torch.bfloat16, s=1.0):
        return (s * torch.randn(shape, generator=g, device="cuda")).to(dt)
    A = rnd(*((K, M) if a_mn else (M, K)))
    B = rnd(*((K, N) if b_mn else (N, K)), s=0.05)
    lda, ldb = (M if a_mn else K), (N if b_mn else K)
    bias, aux16, aux32 = rnd(N, dt=torch.float32), rnd(M, N), rnd(M, N, dt=torch.float32)
    mu, rs, ga = rnd(M, dt=torch.float32), rnd(M, dt=torch.float32), rnd(N, dt=torch.float32)
    pos = torch.arange(M, device="cuda", dtype=torch.int32)
    tab = rnd(M, 32, 2, dt=torch.float32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    f32 = dict(aux_dtype=F.FL_DT_F32, d_dtype=F.FL_DT_F32)
    cases = [(torch.bfloat16, dict(epilogue=F.FL_EPI_STORE, bias=bias)), (torch.float32, dict(epilogue=F.FL_EPI_STORE_F32)),
             (torch.float32, dict(epilogue=F.FL_EPI_ACCUM_F32)),
             (torch.bfloat16, dict(epilogue=F.FL_EPI_BIAS_GELU, bias=bias, ld_aux_out=N, aux_out="u")),
             (torch.bfloat16, dict(epilogue=F.FL_EPI_GELU_BWD, aux=aux16, ld_aux=N, colsum="c")),
             (torch.float32, dict(epilogue=F.FL_EPI_BIAS_RESID, bias=bias, aux=aux32, ld_aux=N, alpha=7.5, ln_mean=mu,
                                  ln_rstd=rs, ln_gamma=ga, ln_beta=bias, **f32))]
    if N % 384 == 0 or N == 4096:
        cases.append((torch.bfloat16, dict(epilogue=F.FL_EPI_BIAS_ROPE, bias=bias, pos=pos, rope_tab=tab, n_heads=N // 384,
                                           head_dim=128, rotary_dim=64)))
    for dt, kw in cases:
        got = []
        for tile in (F.FL_TILE_AUTO, F.FL_TILE_128x128):
            D = torch.ones((M, N), dtype=dt, device="cuda")
            u, c = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda"), torch.zeros(N, device="cuda")
            k = {n: {"u": u, "c": c}[v] if isinstance(v, str) else v for n, v in kw.items()}
            F.gemm(M, N, K, A, lda, a_mn, B, ldb, b_mn, D, N, status=status, tile=tile, **k)
            got.append((D, u, c))
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        (D0, u0, c0), (D1, u1, c1) = got
        assert torch.equal(D0.view(torch.int32 if dt == torch.float32 else torch.int16),
                           D1.view(torch.int32 if dt == torch.float32 else torch.int16)), kw["epilogue"]
        assert torch.equal(u0.view(torch.int16), u1.view(torch.int16))
        # column sums: atomic sums of at most M fp32 values in any order
        assert (c0 - c1).abs().max() <= 2.0 ** -22 * M * max(1.0, float(D1.float().abs().max())) if kw["epilogue"] == F.FL_EPI_GELU_BWD else True


@pytest.mark.parametrize("M,N,K", [(8, 256, 8), (264, 512, 1016), (264, 512, 1024), (2056, 4096, 200), (4104, 8192, 72)])
def test_gemm_fp32_gradient_bit_identical(F, M, N, K):
    """The pair tile's fp32 gradient epilogue (rows past M, rows longer than the output, one
    tile to several per pair, one and two problems) gives the bits of the 128 x 128 tile,
    stored and added, and touches nothing past column N; so does the tile the library picks
    (outputs past the L2's size among them)."""
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn((K, M), generator=g, device="cuda").bfloat16()
    B = torch.randn((K, N), generator=g, device="cuda").bfloat16()
    D0 = torch.randn((2, M, N + 8), generator=g, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for epi in (F.FL_EPI_STORE_F32, F.FL_EPI_ACCUM_F32):
        for n in (1, 2):
            got = []
            for tile in (F.FL_TILE_256x256_PAIR, F.FL_TILE_AUTO, F.FL_TILE_128x128):
                D = D0.clone()
                F.fl_k_gemm_multi([F.gemm_args(M, N, K, A, M, 1, B, N, 1, D[r], N + 8, epilogue=epi, tile=tile)
                                   for r in range(n)], status)
                got.append(D)
            torch.cuda.synchronize()
            assert int(status.item()) == 0
            for D in got[:2]:
                assert torch.equal(D.view(torch.int32), got[2].view(torch.int32)), (epi, n)
                assert torch.equal(D[:, :, N:], D0[:, :, N:])


@pytest.mark.parametrize("K", [64, 3072])
@pytest.mark.parametrize("eps", [0.0, 1e-44, 1e-40, 1e-30])
def test_gemm_adamw_epilogue_tiny_eps(F, K, eps):
    """Denominators down to nothing: rows with a zero gradient and zero moments keep their weights
    with any eps above 0 (0 / 0 without one), rows with an infinite one move by what the separate
    kernel says, as do the others (two ulps of the update)."""
    M, N = 256, 512
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.randn((K, M), generator=g, device="cuda").bfloat16()
    A[:, 16:48] = 0
    A[:, 48:50] *= 1e-25                     # the squares underflow
    B = torch.randn((K, N), generator=g, device="cuda").bfloat16()
    w0 = 0.05 * torch.randn((M, N), generator=g, device="cuda")
    m0 = torch.zeros((M, N), device="cuda")
    m0[60, :8] = float("inf")
    lr, b1, b2, wd = 1e-3, 0.9, 0.999, 0.01
    grad = torch.zeros((M, N), device="cuda")
    F.gemm(M, N, K, A, M, 1, B, N, 1, grad, N, epilogue=F.FL_EPI_STORE_F32)
    wr, mr, vr, wbr = w0.clone(), m0.clone(), torch.zeros_like(w0), torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    F.fl_k_adamw(M * N, wr, grad.clone(), mr, vr, wbr, lr, b1, b2, eps, wd, 0.1, 0.001)
    w, m, v, wb = w0.clone(), m0.clone(), torch.zeros_like(w0), torch.empty_like(wbr)
    F.gemm(M, N, K, A, M, 1, B, N, 1, w, N, epilogue=F.FL_EPI_ADAMW, adam_m=m, adam_v=v, aux_out=wb, ld_aux_out=N,
           lr=lr, beta1=b1, beta2=b2, eps=eps, weight_decay=wd, inv_bc1=1 / 0.1, inv_bc2=1 / 0.001)
    torch.cuda.synchronize()
    assert torch.equal(w.isnan(), wr.isnan()) and torch.equal(w.isinf(), wr.isinf())
    assert bool(w[16:48].isnan().any()) == (eps == 0.0)
    ok = wr.isfinite()
    assert ((w - wr).abs()[ok] <= 2.0 ** -22 * ((w0 - wr).abs() + w0.abs())[ok]).all()


@pytest.mark.parametrize("K", [8, 2048, 3064, 3072, 3080])
def test_gemm_adamw_epilogue_against_exact(F, K):
    """The fused update on both sides of the contraction length where its epilogue changes,
    ragged rows, two problems in one launch: against the update in 64 bits of the very
    gradient the GEMM makes.  Bound per weight: half an ulp of the result and of the update's
    last product, and 8 ulps of lr * ratio for the moments, the quotient and the root (each
    correctly rounded or within one ulp); gradients span the range down to zero."""
    M, N = 264, 512
    rng = np.random.default_rng(K)
    lr, b1, b2, eps, wd, t = 1e-3, 0.9, 0.999, 1e-8, 0.01, 3
    f = [np.float32(x) for x in (lr, b1, b2, eps, wd)]
    inv1, inv2 = np.float32(1.0 / np.float32(1.0 - b1 ** t)), np.float32(1.0 / np.float32(1.0 - b2 ** t))
    A = rnd_bf16_f64(rng, (M, K))
    A[:8] = 0.0  # rows with a zero gradient
    A[8:64] *= 2.0 ** -rng.integers(0, 60, (56, 1))
    dA, lda = _store(A, True)
    dB, ldb = _store(rnd_bf16_f64(rng, (N, K)), True)
    w0 = (0.05 * rng.standard_normal((2, M, N))).astype(np.float32)
    w0[:, :, :64] = 0.0
    m0 = (0.01 * rng.standard_normal((2, M, N))).astype(np.float32)
    v0 = (1e-3 * rng.random((2, M, N))).astype(np.float32)
    m0[:, :8], v0[:, :8] = 0.0, 0.0
    m0[:, 8:64] = 0.0
    v0[:, 8:64] = 0.0
    g = torch.empty((M, N), dtype=torch.float32, device="cuda")
    F.gemm(M, N, K, dA, lda, 1, dB, ldb, 1, g, N, epilogue=F.FL_EPI_STORE_F32, tile=F.FL_TILE_256x256_PAIR)
    w, m, v = dev_f32(w0), dev_f32(m0), dev_f32(v0)
    wb = torch.empty((2, M, N), dtype=torch.bfloat16, device="cuda")
    F.fl_k_gemm_multi([F.gemm_args(M, N, K, dA, lda, 1, dB, ldb, 1, w[r], N, epilogue=F.FL_EPI_ADAMW, adam_m=m[r], adam_v=v[r],
                                   aux_out=wb[r], ld_aux_out=N, lr=lr, beta1=b1, beta2=b2, eps=eps, weight_decay=wd,
                                   inv_bc1=float(inv1), inv_bc2=float(inv2), tile=F.FL_TILE_256x256_PAIR) for r in range(2)])
    torch.cuda.synchronize()
    lr, b1, b2, eps, wd = (float(x) for x in f)
    g = f64(g)
    me = b1 * m0.astype(np.float64) + (1.0 - b1) * g
    ve = b2 * v0.astype(np.float64) + (1.0 - b2) * g * g
    ratio = me * float(inv1) / (np.sqrt(ve * float(inv2)) + eps)
    we = w0 - lr * (ratio + wd * w0.astype(np.float64))
    u = 2.0 ** -24
    # the new first moment is a sum of two terms of either sign: its rounding is relative to them
    terms = (b1 * np.abs(m0) + (1.0 - b1) * np.abs(g)) * float(inv1) / (np.sqrt(ve * float(inv2)) + eps)
    bound = u * (1.01 * np.abs(we) + 16.0 * lr * (terms + wd * np.abs(w0))) + 1e-30
    assert (np.abs(f64(w) - we) <= bound).all()
    np.testing.assert_array_equal(bits(wb), bits(w.to(torch.bfloat16)))


def test_zero_size_calls(F):
    """Degenerate sizes: a GEMM of M = 0 rows, LayerNorm forward and backward over T = 0
    rows, AdamW over 0 parameters, column sums over 0 rows, and attention over one empty
    segment are no-ops that succeed and leave every output untouched."""
    H, N, K = 256, 256, 64
    A = torch.zeros((8, K), dtype=torch.bfloat16, device="cuda")
    B = torch.zeros((N, K), dtype=torch.bfloat16, device="cuda")
    D = torch.full((8, N), 7.0, dtype=torch.bfloat16, device="cuda")
    F.gemm(0, N, K, A, K, 0, B, K, 0, D, N)
    x = torch.zeros((8, H), dtype=torch.bfloat16, device="cuda")
    gam = torch.ones(H, device="cuda")
    bet = torch.zeros(H, device="cuda")
    y = torch.full((8, H), 3.0, dtype=torch.bfloat16, device="cuda")
    mean = torch.full((8,), 5.0, device="cuda")
    rstd = torch.full((8,), 5.0, device="cuda")
    F.fl_k_layernorm_fwd(0, H, x, gam, bet, 1e-5, y, mean, rstd)
    dgam = torch.full((H,), 2.0, device="cuda")
    dbet = torch.full((H,), 2.0, device="cuda")
    ws = torch.empty(max(F.fl_k_layernorm_bwd_workspace(1, H), 16), dtype=torch.uint8, device="cuda")
    F.fl_k_layernorm_bwd(0, H, x, x, mean, rstd, gam, None, 0.0, y, dgam, dbet, ws)
    w = torch.full((8,), 4.0, device="cuda")
    F.fl_k_adamw(0, w, w, w, w, None, 1e-3, 0.9, 0.999, 1e-8, 0.0, 0.1, 0.001)
    cs = torch.full((N,), 6.0, device="cuda")
    F.fl_k_colsum(0, N, D, cs)
    nh, hd = 2, 128
    qkv = torch.zeros((8, 3 * nh * hd), dtype=torch.bfloat16, device="cuda")
    cu = np.array([0, 0], np.int32)
    tiles = torch.zeros(16, dtype=torch.int32, device="cuda")
    o = torch.full((8, nh * hd), 9.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((nh, 8), 9.0, device="cuda")
    assert F.fl_k_attention_tiles(cu) == 0
    F.fl_k_attention_fwd(0, nh, hd, qkv, cu, dev_i32(cu), tiles, o, lse)
    torch.cuda.synchronize()
    assert (D == 7.0).all() and (y == 3.0).all() and (mean == 5.0).all() and (rstd == 5.0).all()
    assert (dgam == 2.0).all() and (dbet == 2.0).all() and (w == 4.0).all() and (cs == 6.0).all()
    assert (o == 9.0).all() and (lse == 9.0).all() and not tiles.any()
