"""Server-level parity: fl_server_create/forward/backward/step on the GPU against the
fp64 oracle server (GPU only).

Tolerances (per tensor, ||gpu - oracle||_inf / ||oracle||_inf): output states 2e-2,
input-state and weight gradients 5e-2, weights after one AdamW step 1e-3.  Packing,
unpacking and segment indexing are bit-exact (client-batching invariant on the GPU).
"""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import flglm_oracle as O
from tests._gpu import bits, dev_bf16_from_bits, f64, flglm, need_gpu, rel_inf

pytestmark = pytest.mark.gpu

OUT_TOL, GRAD_TOL, W_TOL = 2e-2, 5e-2, 1e-3


@pytest.fixture(scope="module")
def F():
    need_gpu()
    return flglm()


def make_server(F, cfg, max_tokens=None, seed=None, fused_step_min_tokens=1):
    """fused_step_min_tokens=1: fl_server_backward_step always takes the fused path (the
    test blocks hold far fewer weights than the library fuses by itself)."""
    mt = max_tokens or cfg.tokens
    return F.Server(F.make_cfg(cfg, mt, fused_step_min_tokens=fused_step_min_tokens),
                    cfg.seed if seed is None else seed)


def run_gpu(F, srv, cfg, states_bits, grads_bits):
    states = [dev_bf16_from_bits(s) for s in states_bits]
    outs = [torch.empty_like(s) for s in states]
    srv.forward(states, cfg.seq_lens, outs)
    gouts = [dev_bf16_from_bits(g) for g in grads_bits]
    gins = [torch.empty_like(s) for s in states]
    srv.backward(gouts, gins)
    srv.sync()
    return outs, gins


def test_create_init_matches_generator(F):
    cfg = syn.CONFIGS["tiny"]
    srv = make_server(F, cfg)
    for t in range(12):
        got = srv.get_param(0, t)
        want = syn.init_tensor(cfg, 0, t).reshape(-1)
        # device and host libm may differ by an ulp in double before the fp32 rounding
        ulps = np.abs(got.view(np.int32).astype(np.int64) - want.view(np.int32).astype(np.int64))
        assert ulps.max() <= 1, (t, ulps.max())
        assert (ulps == 0).mean() > 0.999
    srv.close()


def check_updated_weights(w, w_ref, w0, g_ref, lr, where):
    """Weights after one AdamW step.  The first Adam step moves each weight by about
    lr * sign(g), a jump at g = 0, so an element whose reference gradient is below the
    gradient precision may legitimately move the other way.  Some gradients are zero in
    exact arithmetic (the key bias on the un-rotated dims only shifts every score of a
    row by the same amount, which softmax ignores), so their sign is rounding noise.
    The 1e-3 bound applies to elements whose gradient is resolved (>= the gradient
    tolerance x max); elements with a significant gradient (>= 1e-2 x max) must move the
    same way (under 2% flipped, mean update error under 5% of lr)."""
    w = w.astype(np.float64)
    den = np.abs(w_ref).max()
    gmax = max(np.abs(g_ref).max(), 1e-30)
    resolved = np.abs(g_ref) >= GRAD_TOL * gmax
    if resolved.any():
        assert np.abs(w - w_ref)[resolved].max() / den < W_TOL, where
    significant = np.abs(g_ref) >= 1e-2 * gmax
    if significant.any():
        err = np.abs((w - w0) - (w_ref - w0.astype(np.float64)))[significant]
        assert np.mean(err) < 0.05 * lr, (where, np.mean(err) / lr)
        assert np.mean(err > lr) < 0.02, (where, np.mean(err > lr))


def parity_case(F, cfg, check_step=True, fused=False):
    params = syn.init_params(cfg)
    srv = make_server(F, cfg)
    for b in range(cfg.n_blocks):
        for t in range(12):
            srv.set_param(b, t, params[b][t])
    states = syn.client_states(cfg)
    grads = syn.client_grads(cfg)
    if fused:   # backward + AdamW in one call: compare outputs, input grads and updated weights
        st = [dev_bf16_from_bits(s) for s in states]
        outs = [torch.empty_like(s) for s in st]
        srv.forward(st, cfg.seq_lens, outs)
        gins = [torch.empty_like(s) for s in st]
        srv.backward_step([dev_bf16_from_bits(g) for g in grads], gins, cfg.lr)
        srv.sync()
        ref = O.OracleServer(cfg, params)
        ro = ref.forward([syn.bf16_bits_to_f64(s) for s in states])
        rg = ref.backward([syn.bf16_bits_to_f64(g) for g in grads])
        gref = [[ref.grads[b][t].reshape(-1).copy() for t in range(12)] for b in range(cfg.n_blocks)]
        ref.step(cfg.lr)
        for k in range(cfg.K):
            assert rel_inf(f64(outs[k]), ro[k]) < OUT_TOL
            assert rel_inf(f64(gins[k]), rg[k]) < GRAD_TOL
        for b in range(cfg.n_blocks):
            for t in range(12):
                check_updated_weights(srv.get_param(b, t), ref.params[b][t].reshape(-1),
                                      params[b][t].reshape(-1), gref[b][t], cfg.lr, (b, t))
                m, v = srv.get_adam_moments(b, t)
                assert rel_inf(m, ref.m[b][t].reshape(-1)) < GRAD_TOL
                assert not srv.get_grad(b, t).any()
        srv.close()
        return
    outs, gins = run_gpu(F, srv, cfg, states, grads)
    ref = O.OracleServer(cfg, params)
    ro = ref.forward([syn.bf16_bits_to_f64(s) for s in states])
    rg = ref.backward([syn.bf16_bits_to_f64(g) for g in grads])
    for k in range(cfg.K):
        assert rel_inf(f64(outs[k]), ro[k]) < OUT_TOL, ("out", k, rel_inf(f64(outs[k]), ro[k]))
        assert rel_inf(f64(gins[k]), rg[k]) < GRAD_TOL, ("grad_in", k, rel_inf(f64(gins[k]), rg[k]))
    for b in range(cfg.n_blocks):
        for t in range(12):
            g = srv.get_grad(b, t)
            e = rel_inf(g, ref.grads[b][t].reshape(-1))
            assert e < GRAD_TOL, ("wgrad", b, syn.TENSOR_NAMES[t], e)
    if check_step:
        gref = [[ref.grads[b][t].reshape(-1).copy() for t in range(12)] for b in range(cfg.n_blocks)]
        srv.step(cfg.lr)
        ref.step(cfg.lr)
        srv.sync()
        for b in range(cfg.n_blocks):
            for t in range(12):
                check_updated_weights(srv.get_param(b, t), ref.params[b][t].reshape(-1),
                                      params[b][t].reshape(-1), gref[b][t], cfg.lr, (b, t))
                m, v = srv.get_adam_moments(b, t)
                assert rel_inf(m, ref.m[b][t].reshape(-1)) < GRAD_TOL
                assert not srv.get_grad(b, t).any()
    srv.close()


@pytest.mark.parametrize("rfl", [1, 0], ids=["glm_block", "pre_ln"])
def test_tiny_config_parity(F, rfl):
    parity_case(F, syn.CONFIGS["tiny"].with_(residual_from_ln=rfl))


@pytest.mark.parametrize("rfl", [1, 0], ids=["glm_block", "pre_ln"])
def test_tiny_config_parity_fused_step(F, rfl):
    parity_case(F, syn.CONFIGS["tiny"].with_(residual_from_ln=rfl), fused=True)


def test_fused_step_equals_backward_then_step(F):
    """Two steps of fl_server_backward_step against fl_server_backward + fl_server_step
    on identically seeded servers (the fused AdamW epilogue uses the same fp32 formula;
    the LayerNorm parameter gradients are summed with atomics, so their summation order,
    and the last bits of those updates, may differ between runs)."""
    cfg = syn.CONFIGS["tiny"].with_(n_blocks=2, seq_lens=(64, 40))
    states = [dev_bf16_from_bits(s) for s in syn.client_states(cfg)]
    grads = [dev_bf16_from_bits(g) for g in syn.client_grads(cfg)]
    a, b = make_server(F, cfg), make_server(F, cfg)
    outs = [torch.empty_like(s) for s in states]
    gi = [torch.empty_like(s) for s in states]
    for _ in range(2):
        a.forward(states, cfg.seq_lens, outs)
        a.backward(grads, gi)
        a.step(1e-3)
        b.forward(states, cfg.seq_lens, outs)
        b.backward_step(grads, gi, 1e-3)
    a.sync()
    b.sync()
    for blk in range(cfg.n_blocks):
        for t in range(12):
            wa, wb = a.get_param(blk, t), b.get_param(blk, t)
            assert rel_inf(wb, wa) < 1e-5, (blk, t)
            ma, va = a.get_adam_moments(blk, t)
            mb, vb = b.get_adam_moments(blk, t)
            assert rel_inf(mb, ma) < 1e-5 and rel_inf(vb, va) < 1e-5
    # with gradients pending from an earlier backward, the call falls back to backward + step
    b.forward(states, cfg.seq_lens, outs)
    b.backward(grads, gi)
    b.forward(states, cfg.seq_lens, outs)
    b.backward_step(grads, gi, 1e-3)
    b.sync()
    a.close()
    b.close()


def test_backward_step_below_the_fusion_crossover(F):
    """By default a block of few weights takes backward + step inside
    fl_server_backward_step; two steps of it give the weights of the forced fused path
    (up to the rounding of the atomic bias sums)."""
    cfg = syn.CONFIGS["tiny"].with_(n_blocks=2, seq_lens=(64, 40))
    states = [dev_bf16_from_bits(s) for s in syn.client_states(cfg)]
    grads = [dev_bf16_from_bits(g) for g in syn.client_grads(cfg)]
    a, b = make_server(F, cfg, fused_step_min_tokens=0), make_server(F, cfg)
    outs = [torch.empty_like(s) for s in states]
    gi = [torch.empty_like(s) for s in states]
    for _ in range(2):
        for srv in (a, b):
            srv.forward(states, cfg.seq_lens, outs)
            srv.backward_step(grads, gi, 1e-3)
    a.sync()
    b.sync()
    for blk in range(cfg.n_blocks):
        for t in range(12):
            assert rel_inf(a.get_param(blk, t), b.get_param(blk, t)) < 1e-5, (blk, t)
    a.close()
    b.close()


def test_backward_step_default_at_hidden_1024(F):
    """Hidden 1024 (12.6M matrix weights per block): what the library picks by itself against the
    separate update, over two steps (up to the rounding of the atomic bias sums)."""
    cfg = syn.CONFIGS["tiny"].with_(hidden=1024, n_heads=16, ffn_hidden=4096, client_batch=1, seq_lens=(300, 77))
    g = torch.Generator(device="cuda").manual_seed(5)
    states = [torch.randn((1, n, 1024), generator=g, device="cuda").bfloat16() for n in cfg.seq_lens]
    grads = [(1e-3 * torch.randn((1, n, 1024), generator=g, device="cuda")).bfloat16() for n in cfg.seq_lens]
    a, b = (make_server(F, cfg, fused_step_min_tokens=n) for n in (0, 1 << 30))
    for _ in range(2):
        for srv in (a, b):
            outs, gi = [torch.empty_like(x) for x in states], [torch.empty_like(x) for x in states]
            srv.forward(states, cfg.seq_lens, outs)
            srv.backward_step(grads, gi, 1e-3)
            srv.sync()
    for t in range(12):
        assert rel_inf(a.get_param(0, t), b.get_param(0, t)) < 1e-5, t
    a.close()
    b.close()


def test_ragged_small_parity(F):
    cfg = syn.CONFIGS["tiny"].with_(n_blocks=2, client_batch=1, seq_lens=(1, 17, 64, 65, 130, 3))
    parity_case(F, cfg)


def test_block6b_parity(F):
    """One ChatGLM-6B-shaped block (H 4096, 32 x 128, F 16384), K=4 x 512, full size."""
    parity_case(F, syn.CONFIGS["block6b"], check_step=True)


def test_client_batching_invariant_bitexact(F):
    """§3.3 stacks clients without mixing them: each client's outputs and input gradients
    from the packed call equal (bit for bit) those of calling the server with that client
    alone; the packed weight gradients equal the sum of the per-client ones."""
    cfg = syn.CONFIGS["tiny"].with_(n_blocks=2, client_batch=2, seq_lens=(64, 20, 130))
    states = syn.client_states(cfg)
    grads = syn.client_grads(cfg)
    srv = make_server(F, cfg)
    outs, gins = run_gpu(F, srv, cfg, states, grads)
    gsum = [[np.zeros(srv.numel(t)) for t in range(12)] for _ in range(cfg.n_blocks)]
    packed_g = [[srv.get_grad(b, t).astype(np.float64) for t in range(12)] for b in range(cfg.n_blocks)]
    srv.close()
    for k in range(cfg.K):
        c1 = cfg.with_(seq_lens=(cfg.seq_lens[k],))
        s1 = make_server(F, c1, max_tokens=cfg.tokens, seed=cfg.seed)
        o1, g1 = run_gpu(F, s1, c1, [states[k]], [grads[k]])
        np.testing.assert_array_equal(bits(o1[0]), bits(outs[k]))
        np.testing.assert_array_equal(bits(g1[0]), bits(gins[k]))
        for b in range(cfg.n_blocks):
            for t in range(12):
                gsum[b][t] += s1.get_grad(b, t)
        s1.close()
    for b in range(cfg.n_blocks):
        for t in range(12):
            assert rel_inf(packed_g[b][t], gsum[b][t]) < 1e-3


def test_serial_accumulation_and_state_errors(F):
    """Serial strategy (§3.3): forward/backward per client without a step accumulates the
    weight gradients; protocol-order violations are reported as FL_ERR_STATE."""
    cfg = syn.CONFIGS["tiny"]
    srv = make_server(F, cfg)
    dummy = [torch.empty((cfg.client_batch, cfg.seq_lens[0], cfg.hidden), dtype=torch.bfloat16, device="cuda")]
    with pytest.raises(F.FlError) as ei:
        srv.backward(dummy, dummy)
    assert ei.value.code == -3
    states = syn.client_states(cfg)
    grads = syn.client_grads(cfg)
    for k in range(cfg.K):
        ck = cfg.with_(seq_lens=(cfg.seq_lens[k],))
        run_gpu(F, srv, ck, [states[k]], [grads[k]])
    ser = [srv.get_grad(0, t) for t in range(12)]
    srv.close()
    srv2 = make_server(F, cfg)
    run_gpu(F, srv2, cfg, states, grads)
    for t in range(12):
        assert rel_inf(ser[t], srv2.get_grad(0, t)) < 1e-3
    # step while a forward is pending
    st = [dev_bf16_from_bits(s) for s in states]
    outs = [torch.empty_like(s) for s in st]
    srv2.forward(st, cfg.seq_lens, outs)
    with pytest.raises(F.FlError) as ei:
        srv2.step(1e-4)
    assert ei.value.code == -3
    with pytest.raises(F.FlError) as ei:
        srv2.forward(st, cfg.seq_lens, outs)
    assert ei.value.code == -3
    srv2.close()


def test_argument_errors(F):
    cfg = syn.CONFIGS["tiny"]
    srv = make_server(F, cfg, max_tokens=256)
    st = [torch.empty((2, 64, 256), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    with pytest.raises(F.FlError) as ei:      # 3 x 2 x 64 = 384 tokens > 256
        srv.forward(st, [64, 64, 64], st)
    assert ei.value.code == -2
    with pytest.raises(F.FlError) as ei:
        srv.forward(st[:1], [0], st[:1])
    assert ei.value.code == -1
    base = torch.empty(2 * 64 * 256 + 8, dtype=torch.bfloat16, device="cuda")
    mis = base[1:1 + 2 * 64 * 256]            # 2-byte offset: not 16-byte aligned
    with pytest.raises(F.FlError) as ei:
        srv.forward([mis], [64], [st[0]])
    assert ei.value.code == -1
    with pytest.raises(F.FlError) as ei:
        srv.forward([], [], [])
    assert ei.value.code == -1
    srv.sync()
    srv.close()


@pytest.mark.parametrize("fused", [False, True], ids=["step", "backward_step"])
def test_tiny_parity_weight_decay(F, fused):
    """Decoupled weight decay lambda = 0.01 (the paper trains with none; the AdamW of the
    library takes it as a parameter): the step, and the step fused into the backward."""
    parity_case(F, syn.CONFIGS["tiny"].with_(weight_decay=0.01), fused=fused)


def fp32_oracle_case(F, cfg):
    """GPU forward + backward against the fp32 C++ oracle (single precision throughout, the
    precision the tolerances were written for), the same seeded weights and inputs."""
    from oracle import oracle32 as O32
    params = syn.init_params(cfg)
    srv = make_server(F, cfg)
    for b in range(cfg.n_blocks):
        for t in range(12):
            srv.set_param(b, t, params[b][t])
    states = syn.client_states(cfg)
    grads = syn.client_grads(cfg)
    outs, gins = run_gpu(F, srv, cfg, states, grads)
    H = cfg.hidden
    x = np.concatenate([syn.bf16_bits_to_f64(s).reshape(-1, H) for s in states])
    dy = np.concatenate([syn.bf16_bits_to_f64(g).reshape(-1, H) for g in grads])
    cu = np.concatenate([[0], np.cumsum([L for L in cfg.seq_lens for _ in range(cfg.client_batch)])])
    g32 = [[np.zeros(p.shape, np.float32) for p in blk] for blk in params]
    y, dx = O32.server_fwd_bwd(cfg, params, g32, cu, x, dy)
    y_gpu = np.concatenate([f64(o).reshape(-1, H) for o in outs])
    dx_gpu = np.concatenate([f64(g).reshape(-1, H) for g in gins])
    assert rel_inf(y_gpu, y) < OUT_TOL, rel_inf(y_gpu, y)
    assert rel_inf(dx_gpu, dx) < GRAD_TOL, rel_inf(dx_gpu, dx)
    for b in range(cfg.n_blocks):
        for t in range(12):
            e = rel_inf(srv.get_grad(b, t), g32[b][t].reshape(-1))
            assert e < GRAD_TOL, ("wgrad", b, syn.TENSOR_NAMES[t], e)
    srv.close()


def test_tiny_parity_vs_fp32_oracle(F):
    """The one-block H=256 workload (K=2 x 2 rows x 64 tokens) against the fp32 oracle."""
    fp32_oracle_case(F, syn.CONFIGS["tiny"])


def test_block6b_segment_parity_vs_fp32_oracle(F):
    """One ChatGLM-6B-shaped block (H=4096, 32 x 128, F=16384) on one 512-token client of
    the one-block workload, against the fp32 oracle."""
    fp32_oracle_case(F, syn.CONFIGS["block6b"].with_(seq_lens=(512,)))
