"""Client parts of the split (§3.1) on the GPU: embedding + block 0 at the bottom, block
N-1 + final LayerNorm + LM head + cross-entropy at the top, the full split round with the
server, and client averaging (§3.3).  Parity against the fp64 oracle (GPU only)."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import flglm_oracle as O
from tests._gpu import bits, dev_bf16_from_bits, dev_i32, f64, flglm, need_gpu, rel_inf
from tests.test_gpu_server import GRAD_TOL, OUT_TOL, check_updated_weights

pytestmark = pytest.mark.gpu

LOSS_TOL = 1e-2


@pytest.fixture(scope="module")
def F():
    need_gpu()
    return flglm()


def tiny_client(**kw):
    return syn.CONFIGS["tiny"].with_(client_batch=2, seq_lens=(64,), vocab=1000, lr=1e-3, **kw)


def bf16_dev(x64):
    return dev_bf16_from_bits(syn.f32_to_bf16_bits(np.asarray(x64, np.float32)))


def part_tensors(cfg):
    n_blk = 14 if cfg.prefix_len else 12
    out = [(F_part, t) for F_part in ("bottom", "top") for t in range(n_blk)]
    return out + [("embed", 0), ("head", 0), ("final_ln", 0), ("final_ln", 1)]


PART_IDS = {"bottom": 0, "top": 1, "embed": 2, "head": 3, "final_ln": 4}


def test_client_init_matches_generator(F):
    cfg = tiny_client(prefix_len=8)
    cl = F.Client(F.make_client_cfg(cfg, cfg.tokens), cfg.seed)
    want = syn.init_client(cfg)
    for part, t in part_tensors(cfg):
        got = cl.get_param(PART_IDS[part], t)
        w = want[part][t].reshape(-1)
        ulps = np.abs(got.view(np.int32).astype(np.int64) - w.astype(np.float32).view(np.int32).astype(np.int64))
        assert ulps.max() <= 1, (part, t, ulps.max())
    cl.close()


def client_round(F, cfg, ctx=None, mp=None, check_step=True, params=None):
    """One client alone (its bottom output handed straight to its top), GPU against the
    oracle on the same bf16 hand-offs."""
    cl = F.Client(F.make_client_cfg(cfg, cfg.tokens), cfg.seed)
    if params is None:
        params = syn.init_client(cfg)
    else:   # explicit values: loaded into the client, the oracle takes the same ones
        for part, t in part_tensors(cfg):
            cl.set_param(PART_IDS[part], t, params[part][t])
    tokens = syn.client_tokens(cfg, 0)
    labels = syn.client_labels(tokens, ctx)
    b, L = tokens.shape
    h0 = torch.empty((b, L, cfg.hidden), dtype=torch.bfloat16, device="cuda")
    cl.bottom_forward(dev_i32(tokens), L, h0, context_lens=ctx, mask_pos=mp)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    gh = torch.empty_like(h0)
    cl.top_forward_backward(h0, dev_i32(labels), loss, gh)
    gh_bits = bits(gh)
    cl.bottom_backward(gh)
    cl.sync()
    ref = O.OracleClient(cfg, params)
    h0_ref = ref.bottom_forward(tokens, ctx, mp)
    assert rel_inf(f64(h0), h0_ref) < OUT_TOL
    # the top and the bottom backward see the GPU's bf16 hand-offs, as the protocol sends them
    loss_ref, gh_ref = ref.top_forward_backward(syn.bf16_bits_to_f64(bits(h0)).reshape(b, L, -1), labels)
    assert abs(float(loss.item()) - loss_ref) / abs(loss_ref) < LOSS_TOL, (loss.item(), loss_ref)
    assert rel_inf(f64(gh), gh_ref) < GRAD_TOL
    ref.bottom_backward(syn.bf16_bits_to_f64(gh_bits).reshape(b, L, -1))
    trained = set(ref.trained())
    gref = {}
    for part, t in part_tensors(cfg):
        g = cl.get_grad(PART_IDS[part], t)
        gr = ref.grads[part][t].reshape(-1)
        gref[(part, t)] = gr.copy()
        if (part, t) in trained:
            e = rel_inf(g, gr)
            assert e < GRAD_TOL, ("grad", part, t, e)
        elif part not in ("bottom", "top"):
            assert not g.any()   # frozen: no gradient kept
    if check_step:
        cl.step(cfg.lr)
        ref.step(cfg.lr)
        cl.sync()
        for part, t in part_tensors(cfg):
            w0 = np.asarray(params[part][t], np.float32).reshape(-1)
            w = cl.get_param(PART_IDS[part], t)
            if (part, t) in trained:
                check_updated_weights(w, ref.params[part][t].reshape(-1), w0, gref[(part, t)], cfg.lr, (part, t))
            else:
                np.testing.assert_array_equal(w, w0)
    cl.close()


def test_client_parity(F):
    client_round(F, tiny_client())


def test_client_parity_glm_ptuning(F):
    """The paper's client: GLM blank-infilling rows, P-tuning v2 prefixes in both client
    blocks, everything else frozen."""
    cfg = tiny_client(prefix_len=16, freeze_base=1)
    ctx = [40, 63]
    client_round(F, cfg, ctx=ctx, mp=[39, 10])


def test_split_round_matches_oracle(F):
    """The whole protocol of §3.1 on one GPU: two clients' bottoms, one client-batched
    server call (§3.3), the clients' tops, the server backward, the clients' bottom
    backwards and every step, against the oracle client/server composition."""
    cfg = syn.CONFIGS["tiny"].with_(n_blocks=2, client_batch=2, seq_lens=(64, 48), vocab=1000, lr=1e-3)
    K, b = cfg.K, cfg.client_batch
    ctx_all, mp_all = syn.glm_structure(cfg)
    ccfgs = [cfg.with_(seq_lens=(L,)) for L in cfg.seq_lens]
    srv = F.Server(F.make_cfg(cfg, cfg.tokens), cfg.seed)
    clients = [F.Client(F.make_client_cfg(c, c.tokens), cfg.seed) for c in ccfgs]
    toks = [syn.client_tokens(cfg, k) for k in range(K)]
    ctxs = [ctx_all[k * b:(k + 1) * b] for k in range(K)]
    mps = [mp_all[k * b:(k + 1) * b] for k in range(K)]
    labs = [syn.client_labels(toks[k], ctxs[k]) for k in range(K)]
    h0 = [torch.empty((b, L, cfg.hidden), dtype=torch.bfloat16, device="cuda") for L in cfg.seq_lens]
    for k in range(K):
        clients[k].bottom_forward(dev_i32(toks[k]), cfg.seq_lens[k], h0[k], ctxs[k], mps[k])
    hs = [torch.empty_like(x) for x in h0]
    srv.forward(h0, cfg.seq_lens, hs, context_lens=ctx_all, mask_pos=mp_all)
    losses = [torch.zeros(1, dtype=torch.float32, device="cuda") for _ in range(K)]
    gh = [torch.empty_like(x) for x in h0]
    for k in range(K):
        clients[k].top_forward_backward(hs[k], dev_i32(labs[k]), losses[k], gh[k])
    g0 = [torch.empty_like(x) for x in h0]
    srv.backward(gh, g0)
    for k in range(K):
        clients[k].bottom_backward(g0[k])
        clients[k].sync()
    srv.sync()
    # oracle: the same composition in fp64
    cp = syn.init_client(cfg)
    rcl = [O.OracleClient(c, cp) for c in ccfgs]
    rsrv = O.OracleServer(cfg)
    rh0 = [rcl[k].bottom_forward(toks[k], ctxs[k], mps[k]) for k in range(K)]
    rhs = rsrv.forward(rh0, ctx_all, mp_all)
    rtop = [rcl[k].top_forward_backward(rhs[k], labs[k]) for k in range(K)]
    rg0 = rsrv.backward([g for _, g in rtop])
    for k in range(K):
        rcl[k].bottom_backward(rg0[k])
        assert rel_inf(f64(h0[k]), rh0[k]) < OUT_TOL
        assert rel_inf(f64(hs[k]), rhs[k]) < OUT_TOL
        assert abs(losses[k].item() - rtop[k][0]) / rtop[k][0] < LOSS_TOL
        assert rel_inf(f64(gh[k]), rtop[k][1]) < GRAD_TOL
        assert rel_inf(f64(g0[k]), rg0[k]) < GRAD_TOL
        for part, t in part_tensors(cfg):
            e = rel_inf(clients[k].get_grad(PART_IDS[part], t), rcl[k].grads[part][t].reshape(-1))
            assert e < GRAD_TOL, ("client", k, part, t, e)
    for bb in range(cfg.n_blocks):
        for t in range(12):
            assert rel_inf(srv.get_grad(bb, t), rsrv.grads[bb][t].reshape(-1)) < GRAD_TOL, ("server", bb, t)
    # steps (each client against its oracle), then the end-of-period client averaging (§3.3)
    gref = [{(p, t): rcl[k].grads[p][t].reshape(-1).copy() for p, t in part_tensors(cfg)} for k in range(K)]
    for c in clients:
        c.step(cfg.lr)
    srv.step(cfg.lr)
    for k in range(K):
        rcl[k].step(cfg.lr)
        for part, t in part_tensors(cfg):
            w0 = np.asarray(cp[part][t], np.float32).reshape(-1)
            check_updated_weights(clients[k].get_param(PART_IDS[part], t), rcl[k].params[part][t].reshape(-1), w0,
                                  gref[k][(part, t)], cfg.lr, (k, part, t))
    before = {(p, t): [c.get_param(PART_IDS[p], t) for c in clients] for p, t in part_tensors(cfg)}
    F.fl_client_average(clients)
    inv = np.float32(1.0) / np.float32(K)
    for (p, t), ws in before.items():
        want = (ws[0] + ws[1]) * inv
        for c in clients:
            np.testing.assert_array_equal(c.get_param(PART_IDS[p], t), want)
    for c in clients:
        c.close()
    srv.close()


def test_client_average_is_the_mean(F):
    """fl_client_average writes the fp32 mean (summed in client order) into every client."""
    cfg = tiny_client()
    cls = [F.Client(F.make_client_cfg(cfg, cfg.tokens), s) for s in (1, 2, 3)]
    before = {(p, t): [c.get_param(PART_IDS[p], t) for c in cls] for p, t in part_tensors(cfg)}
    F.fl_client_average(cls)
    inv = np.float32(1.0) / np.float32(3.0)
    for (p, t), ws in before.items():
        want = ((ws[0] + ws[1]) + ws[2]) * inv
        for c in cls:
            np.testing.assert_array_equal(c.get_param(PART_IDS[p], t), want)
    with pytest.raises(F.FlError):
        F.fl_client_average([cls[0], cls[0]])
    for c in cls:
        c.close()


def test_client_errors(F):
    cfg = tiny_client()
    cl = F.Client(F.make_client_cfg(cfg, cfg.tokens), 0)
    b, L, H = 2, 64, cfg.hidden
    h = torch.zeros((b, L, H), dtype=torch.bfloat16, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    labels = dev_i32(np.full((b, L), -1, np.int32))
    with pytest.raises(F.FlError) as ei:        # top before bottom
        cl.top_forward_backward(h, labels, loss, h)
    assert ei.value.code == -3
    with pytest.raises(F.FlError) as ei:        # too many tokens
        cl.bottom_forward(dev_i32(np.zeros((b, 65), np.int32)), 65, h)
    assert ei.value.code == -1
    bad = np.zeros((b, L), np.int32)
    bad[1, 5] = cfg.vocab                       # out-of-range token: embeds as zeros, reported at sync
    cl.bottom_forward(dev_i32(bad), L, h)
    with pytest.raises(F.FlError) as ei:
        cl.bottom_forward(dev_i32(bad), L, h)   # round already open
    assert ei.value.code == -3
    with pytest.raises(F.FlError) as ei:
        cl.sync()
    assert ei.value.code == -1
    lab = np.full((b, L), -1, np.int32)
    lab[0, 3] = cfg.vocab + 7                   # label >= vocab: ignored, reported
    cl.top_forward_backward(h, dev_i32(lab), loss, h)
    with pytest.raises(F.FlError) as ei:
        cl.sync()
    assert ei.value.code == -1
    assert float(loss.item()) == 0.0            # no valid target: zero loss
    cl.bottom_backward(h)
    cl.step(1e-3)
    cl.sync()
    cl.close()


@pytest.mark.slow
def test_client_chatglm6b_shapes(F):
    """The ChatGLM-6B client: H 4096, 32 x 128 heads, FFN 16384, vocabulary 130528 (head
    padded to 130560), one GLM row of 96 tokens, all client parameters trained."""
    cfg = syn._glm("client6b", 1, 1, 1, (96,)).with_(vocab=syn.CHATGLM6B_VOCAB, lr=1e-4)
    rng = np.random.default_rng(6)

    def draw(shape):
        return (0.02 * rng.standard_normal(shape, dtype=np.float32))

    params = {}
    for part in ("bottom", "top"):
        ts = [draw(s) for s in syn.param_shapes(cfg)]
        for t in (syn.T_G1, syn.T_G2):
            ts[t] = 1.0 + ts[t]
        params[part] = ts
    params["embed"] = [draw((cfg.vocab, cfg.hidden))]
    params["head"] = [draw((cfg.vocab, cfg.hidden))]
    params["final_ln"] = [1.0 + draw(cfg.hidden), draw(cfg.hidden)]
    client_round(F, cfg, ctx=[70], mp=[69], check_step=False, params=params)


@pytest.mark.parametrize("V,ld", [(1000, 1024), (130528, 130560), (5, 8)])
def test_cross_entropy_kernel(F, V, ld):
    """The row kernel against the oracle: loss, per-row losses and the logit gradient,
    ragged vocabulary tails, padded columns zero, rows without a target."""
    rng = np.random.default_rng(V)
    T = 37
    logits = np.zeros((T, ld), np.float32)
    logits[:, :V] = (2.0 * rng.standard_normal((T, V))).astype(np.float32)
    labels = rng.integers(0, V, size=T).astype(np.int32)
    labels[[0, 9, 30]] = -1
    dl = torch.from_numpy(logits).cuda()
    row = torch.empty(T, dtype=torch.float32, device="cuda")
    dlog = torch.full((T, ld), 7.0, dtype=torch.bfloat16, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    cnt = torch.empty(1, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    F.fl_k_cross_entropy(T, V, ld, dl, dev_i32(labels), row, dlog, loss, cnt, st)
    torch.cuda.synchronize()
    ref_loss, ref_d = O.cross_entropy(logits[:, :V].astype(np.float64), labels)
    assert int(cnt.item()) == T - 3 and int(st.item()) == 0
    assert abs(loss.item() - ref_loss) / ref_loss < 1e-5
    got = f64(dlog)
    assert not got[:, V:].any()
    assert rel_inf(got[:, :V], ref_d) < 1e-2        # bf16 gradient
    assert not got[[0, 9, 30]].any()


@pytest.mark.parametrize("rows", ["cta", "cluster", "one"])
@pytest.mark.parametrize("V,ld", [(16381, 16384), (16385, 16388), (32766, 32768), (32769, 32776), (65536, 65540),
                                  (131071, 131072), (131073, 131076)])
def test_cross_entropy_row_lengths(F, V, ld, rows):
    """Row lengths on both sides of every change of kernel, by more rows than half of the SMs (a
    CTA each), by as many (where long rows take a cluster each, two rows per cluster) and by one;
    columns that are masked (-inf, the lowest float) or far apart, a label on the last column, rows
    without a target before and after others of their cluster; each probability within 8 fp32
    ulps plus one bf16 rounding of the result."""
    g = torch.Generator(device="cuda").manual_seed(V)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = {"cta": max(90, sms // 2 + 1), "cluster": sms // 2, "one": 1}[rows]
    assert rows != "cluster" or T > 2 * sms // 8 + 5
    x = 2.0 * torch.randn((T, ld), generator=g, device="cuda")
    x[:, V:] = float("inf")  # padding is not read into the softmax
    lab = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    lab[0] = V - 1
    if T > 1:
        x[1, : V // 2] = -float("inf")
        x[2, 3:V:7] = torch.finfo(torch.float32).min
        x[3, 5] += 80.0
        x[4, :V] -= 1000.0
        lab[1], lab[5], lab[T - 1] = V - 1, -1, -3
    row = torch.empty(T, device="cuda")
    dlog = torch.full((T, ld), 7.0, dtype=torch.bfloat16, device="cuda")
    loss = torch.empty(1, device="cuda")
    cnt = torch.empty(1, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    F.fl_k_cross_entropy(T, V, ld, x, lab, row, dlog, loss, cnt, st)
    torch.cuda.synchronize()
    n = T - 2 if T > 1 else 1
    assert int(cnt.item()) == n and int(st.item()) == 0
    xd, ld_ = x[:, :V].double(), lab.long()
    lse = torch.logsumexp(xd, 1)
    keep = ld_ >= 0
    want_row = torch.where(keep, lse - xd.gather(1, ld_.clamp(min=0)[:, None])[:, 0], torch.zeros_like(lse))
    # fp32: the exponent's argument is rounded (|x - max| <= 2^11 here), and so is the loss itself
    assert ((row.double() - want_row).abs() <= 2.0 ** -21 * (1.0 + want_row.abs() + lse.abs())).all()
    assert abs(loss.item() - want_row.sum().item() / n) <= 2e-6 * max(1.0, want_row.sum().item() / n)
    p = torch.exp(xd - lse[:, None])
    p[torch.arange(T, device="cuda"), ld_.clamp(min=0)] -= 1.0
    want = p * keep[:, None] / n
    err = (dlog[:, :V].double() - want).abs()
    assert (err <= 2.0 ** -8 * want.abs() + 2.0 ** -18 / n + 1e-38).all()
    assert not dlog[:, V:].any() and not dlog[~keep].any()


@pytest.mark.parametrize("V,ld", [(9000, 16400), (32768, 32768), (60000, 65536), (131072, 131072)])
@pytest.mark.parametrize("few", [True, False])
def test_cross_entropy_masked_low_rows(F, V, ld, few):
    """Rows whose live columns lie in some of a cluster's column ranges only (masked with -inf, or
    a vocabulary that ends before the last ranges), their maximum far below zero or above: no
    range without a live column turns into NaN; the lowest logits give probability 0."""
    g = torch.Generator(device="cuda").manual_seed(V)
    T = 6 if few else torch.cuda.get_device_properties(0).multi_processor_count
    x = 2.0 * torch.randn((T, ld), generator=g, device="cuda")
    x[:, V:] = float("nan")
    col = torch.arange(V, device="cuda")
    live = [(col // 2048) % 8 == 1, (col // 1024) % 2 == 0, col < 2048, col == 1, col >= V - 5, col >= 0]
    shift = [-100.0, -1000.0, -95.0, -300.0, 200.0, -150.0]
    lab = torch.zeros(T, device="cuda", dtype=torch.int32)
    for i in range(T):
        k = i % 6
        x[i, :V] += shift[k]
        x[i, :V][~live[k]] = -float("inf")
        lab[i] = int(col[live[k]][-1])
    row = torch.empty(T, device="cuda")
    dlog = torch.full((T, ld), 7.0, dtype=torch.bfloat16, device="cuda")
    loss = torch.empty(1, device="cuda")
    cnt = torch.empty(1, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    F.fl_k_cross_entropy(T, V, ld, x, lab, row, dlog, loss, cnt, st)
    torch.cuda.synchronize()
    xd = x[:, :V].double()
    lse = torch.logsumexp(xd, 1)
    want = torch.exp(xd - lse[:, None])
    want[torch.arange(T, device="cuda"), lab.long()] -= 1.0
    want /= T
    # as above: the exponent's argument, of at most 2^11, is rounded to fp32
    assert not dlog[:, V:].any()
    assert ((dlog[:, :V].double() - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -12 * want.abs() + 2.0 ** -18 / T).all()
    want_row = lse - xd.gather(1, lab.long()[:, None])[:, 0]
    assert ((row.double() - want_row).abs() <= 2.0 ** -21 * (1.0 + want_row.abs() + lse.abs())).all()
    x[2, 0] = float("nan")  # a row that holds a NaN is NaN, its padding stays zero
    F.fl_k_cross_entropy(T, V, ld, x, lab, row, dlog, loss, cnt, st)
    torch.cuda.synchronize()
    assert dlog[2, :V].isnan().all() and not dlog[:, V:].any() and dlog[[0, 1, 3], :V].isfinite().all()


@pytest.mark.parametrize("H,off", [(256, 0), (256, 2), (258, 0), (4096, 4)])
def test_embedding_scatter_alignment(F, H, off):
    """Vector and element-wise reductions by the alignment of the gradient and the width."""
    g = torch.Generator(device="cuda").manual_seed(H + off)
    V, T = 50, 200
    tok = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    tok[7] = V
    buf = torch.randn(T * H + off, generator=g, device="cuda").bfloat16()
    dx = buf[off:]
    dE = torch.zeros(V * H + 4, device="cuda")[: V * H]
    F.fl_k_embedding_scatter_add(T, H, tok, V, dx, dE)
    torch.cuda.synchronize()
    ok = tok < V
    want = torch.zeros((V, H), device="cuda", dtype=torch.float64).index_add_(0, tok[ok].long(), dx.view(T, H)[ok].double())
    # at most T fp32 additions per element, in any order
    assert ((dE.view(V, H).double() - want).abs() <= T * 2.0 ** -23 * 6.0).all()


def test_embedding_kernels(F):
    rng = np.random.default_rng(5)
    V, H, T = 300, 256, 77
    table = rng.standard_normal((V, H)).astype(np.float32)
    tb = syn.bf16_bits_to_f32(syn.f32_to_bf16_bits(table))
    tokens = rng.integers(0, V, size=T).astype(np.int32)
    tokens[[3, 4]] = tokens[2]                      # repeated ids: their gradients add up
    tokens[10] = V                                  # out of range: zero row, flagged
    out = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    F.fl_k_embedding_gather(T, H, dev_i32(tokens), bf16_dev(tb), V, out, st)
    dx = rng.standard_normal((T, H))
    dxb = syn.bf16_bits_to_f64(syn.f32_to_bf16_bits(dx.astype(np.float32)))
    dE = torch.zeros((V, H), dtype=torch.float32, device="cuda")
    F.fl_k_embedding_scatter_add(T, H, dev_i32(tokens), V, bf16_dev(dxb), dE)
    torch.cuda.synchronize()
    ok = tokens < V
    want = np.zeros((T, H))
    want[ok] = tb[tokens[ok]]
    np.testing.assert_array_equal(f64(out), want)
    assert int(st.item()) == 1
    np.testing.assert_allclose(f64(dE), O.embedding_bwd(dxb[ok], tokens[ok], V), rtol=1e-6, atol=1e-5)
