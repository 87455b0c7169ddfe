"""GPU vs oracle parity of the DiT-MoE block's attention path (Sec. 4.1),
through the C ABI (marked gpu).

Every layer of every step is teacher-forced (see gpu_harness): the oracle's
attention of the GPU's block input must match the recomputed a rows, the
kept rows must be untouched, u must equal bf16(x + a), and the MoE
sub-layer is then checked with the router input the sync rule prescribes.
Cases cover every built head size (64, 72, 80, 96, 128), samples that are
ragged against the 64-row query blocks and the 128-row GEMM tiles, one
sample per step (seq_len 0), the three attention policies, a shared expert,
the full-size 12-head block of the D 768 stack, and degenerate steps.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_harness import np_of, run_trajectory  # noqa: E402
from paper_2606_15615_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for gpu-marked tests")
    from paper_2606_15615_gb300 import build
    build.build()
    from paper_2606_15615_gb300 import moeca
    return moeca


def drift(x0, rng, n, sigma):
    xs = [x0]
    for _ in range(1, n):
        xs.append((xs[-1] + sigma * rng.standard_normal(x0.shape)).astype(np.float32))
    return [W.round_to_bf16(x) for x in xs]


def make_block_stack(M, T, D, H, E, k, F, L=1, S=0, n_shared=0, seed=0, wscale=0.05, **cfg_kw):
    ws = []
    for l in range(L):
        w, _, _ = W.tiny_layer(300 + 10 * seed + l, T, D, E, k, F, n_shared=n_shared, dtype="bf16",
                               bias=n_shared > 0, wscale=wscale)
        w.update(W.tiny_attn(300 + 10 * seed + l, D, dtype="bf16", wscale=wscale))
        ws.append(w)
    cfg = M.moeca_config_default(n_layers=L, hidden=D, ffn=F, n_experts=E, top_k=k, n_shared=n_shared,
                                 max_tokens=cfg_kw.pop("max_tokens", T), dtype=M.MOECA_BF16,
                                 n_heads=H, seq_len=S, **cfg_kw)
    return M.Stack(cfg, ws), cfg, ws


@pytest.mark.parametrize("impl", [2, 1])
@pytest.mark.parametrize("D,H,S,T", [(256, 4, 200, 400), (576, 8, 104, 312), (320, 4, 72, 216),
                                     (384, 4, 136, 272), (384, 3, 264, 528)])
def test_sync_blocks_every_head_size(M, D, H, S, T, impl):
    """Heads of 64, 72, 80, 96 and 128 channels; samples ragged against the
    64 / 128-row query blocks, the 128-key blocks and the 128-row tiles; two
    layers; a full step every 3; the tcgen05 core (2) and the mma.sync core (1)."""
    st, cfg, ws = make_block_stack(M, T, D, H, 8, 2, 256, L=2, S=S, seed=D + H, tau0=0.72, refresh_period=3,
                                   attn_impl=impl)
    rng = np.random.default_rng(D + H)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 5, 0.08)
    rep, _ = run_trajectory(st, cfg, ws, xs)
    cache_rows = rep.attn_rows - 2 * 2 * T          # full steps 0 and 3, two layers
    assert rep.reused > 0 and rep.recomputed > 0
    assert 0 < cache_rows < 2 * 3 * T, rep          # some, not all, tokens recompute attention
    stats = st.stats()
    assert stats["attn_recomputed"] == rep.attn_rows
    st.close()


@pytest.mark.parametrize("policy", [1, 2])
def test_stale_and_full_policies(M, policy):
    """Table 4's "without sync update" (attention reused on every cache step)
    and the always-recompute policy that routes on the fresh input."""
    T, D, H, S = 256, 256, 4, 128
    st, cfg, ws = make_block_stack(M, T, D, H, 8, 2, 256, L=2, S=S, seed=7, tau0=0.72, attn_policy=policy)
    rng = np.random.default_rng(70 + policy)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 4, 0.08)
    rep, _ = run_trajectory(st, cfg, ws, xs)
    assert rep.attn_rows == (2 * T if policy == 1 else 2 * 4 * T)
    assert rep.reused > 0
    st.close()


def test_one_sample_shared_expert(M):
    """seq_len 0 (every token attends to all T rows) with a shared expert
    under the synchronized rule."""
    T, D, H = 296, 256, 2
    st, cfg, ws = make_block_stack(M, T, D, H, 4, 2, 192, L=1, S=0, n_shared=1, seed=8, tau0=0.7)
    rng = np.random.default_rng(80)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 4, 0.05)
    rep, _ = run_trajectory(st, cfg, ws, xs)
    assert rep.reused > 0 and rep.attn_rows > T
    st.close()


def test_sync_block_shared_expert_always(M):
    """A shared expert recomputed for every token (shared_policy 1) under the
    sync rule: a token that keeps its attention (empty recompute set) still
    has a shared-expert row, whose input the preparation kernel gathers."""
    T, D, H, S = 256, 256, 4, 128
    st, cfg, ws = make_block_stack(M, T, D, H, 4, 2, 192, L=2, S=S, n_shared=1, seed=9, tau0=0.8, shared_policy=1)
    rng = np.random.default_rng(90)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 4, 0.03)
    rep, _ = run_trajectory(st, cfg, ws, xs)
    stats = st.stats()
    assert stats["tokens_fully_reused"] > 0 and stats["shared_recomputed"] == 2 * 4 * T
    st.close()


def test_block_full_size_d768_12_heads(M):
    """The 12-head block of the D 768 stack at full size (T 2048 = 8 samples
    of 256, E 16, top-2, F 3072), two of its layers, three steps."""
    wl = W.workload("dit_d768_h12_e16_k2_f3072_t2048_l12_bf16")
    ws = []
    for l in range(2):
        w = W.make_layer_weights(wl, l)
        w.update(W.make_attn_weights(wl, l))
        ws.append(w)
    cfg = M.moeca_config_default(n_layers=2, hidden=wl.hidden, ffn=wl.ffn, n_experts=wl.n_experts,
                                 top_k=wl.top_k, max_tokens=wl.n_tokens, dtype=M.MOECA_BF16,
                                 n_heads=wl.n_heads, seq_len=wl.seq, tau0=0.665)
    st = M.Stack(cfg, ws)
    xs = list(W.trajectory(wl, n_steps=3))
    rep, _ = run_trajectory(st, cfg, ws, xs)
    assert rep.reused > 0 and 2 * 2 * wl.n_tokens > rep.attn_rows - 2 * wl.n_tokens > 0
    st.close()


def test_repeated_input_all_reused_is_bitwise_previous_output(M):
    """tau0 = +inf with the same input: no branch and no attention row is
    recomputed and the output repeats the previous step exactly."""
    T, D, H, S = 208, 256, 4, 104
    st, cfg, ws = make_block_stack(M, T, D, H, 8, 2, 256, L=2, S=S, seed=9, tau0=math.inf)
    rng = np.random.default_rng(90)
    x = torch.from_numpy(W.round_to_bf16(rng.standard_normal((T, D)).astype(np.float32))).cuda().to(torch.bfloat16)
    o0 = st.step(x, 0).clone()
    o1 = st.step(x, 1).clone()
    torch.cuda.synchronize()
    assert torch.equal(o0, o1)
    s = st.stats()
    assert s["attn_recomputed"] == 2 * T and s["reused"] == 2 * T * 2
    st.close()


def test_token_count_change_and_empty_step(M):
    """A new T forces a full step (every token's attention); T = 0 is a no-op."""
    D, H, S = 256, 4, 64
    st, cfg, ws = make_block_stack(M, 256, D, H, 8, 2, 256, L=1, S=S, seed=10, tau0=0.72)
    rng = np.random.default_rng(100)
    a = drift(rng.standard_normal((256, D)).astype(np.float32), rng, 2, 0.05)
    b = drift(rng.standard_normal((128, D)).astype(np.float32), rng, 2, 0.05)
    flags = []
    rep, _ = run_trajectory(st, cfg, ws, a + b, refresh_flags=flags)
    assert flags == [True, False, True, False]
    st.step(torch.empty((0, D), dtype=torch.bfloat16, device="cuda"), 9)
    with pytest.raises(M.MoecaError):
        st.step(torch.zeros((100, D), dtype=torch.bfloat16, device="cuda"), 10)   # not a multiple of 64
    st.close()
    st2, _, _ = make_block_stack(M, 60, D, H, 8, 2, 256, L=1, S=20, seed=10)
    with pytest.raises(M.MoecaError):
        st2.step(torch.zeros((60, D), dtype=torch.bfloat16, device="cuda"), 0)    # samples of 20 rows: not a multiple of 8
    st2.close()


@pytest.mark.parametrize("policy", [0, 1])
def test_separate_kernel_path(M, policy):
    """The SIMT FFN takes the separate router / select / compact kernels, so
    u = x + a^{t0} and the FFN row gather run as their own launches."""
    T, D, H, S = 256, 256, 4, 128
    st, cfg, ws = make_block_stack(M, T, D, H, 8, 2, 256, L=2, S=S, seed=11, tau0=0.72, attn_policy=policy,
                                   ffn_impl=M.MOECA_FFN_SIMT)
    rng = np.random.default_rng(110 + policy)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 4, 0.08)
    rep, _ = run_trajectory(st, cfg, ws, xs)
    assert rep.reused > 0 and rep.attn_rows >= 2 * T + (1 if policy == 0 else 0)
    st.close()


def test_tcgen05_and_mma_sync_cores_agree(M):
    """The two attention cores on the same block inputs: a rows within bf16
    rounding of each other (different summation order, same math)."""
    T, D, H, S = 512, 512, 4, 256
    outs = []
    for impl in (2, 1):
        st, cfg, ws = make_block_stack(M, T, D, H, 8, 2, 256, L=1, S=S, seed=12, tau0=0.72, attn_impl=impl)
        rng = np.random.default_rng(120)
        xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 3, 0.08)
        for t, x in enumerate(xs):
            st.step(torch.from_numpy(x).cuda().to(torch.bfloat16), t)
        torch.cuda.synchronize()
        outs.append(np_of(st.get_state(0)["attn_a"]).astype(np.float64))
        st.close()
    err = np.linalg.norm(outs[0] - outs[1]) / np.linalg.norm(outs[1])
    assert err < 1e-2, err


def test_sixteen_token_prep_blocks(M):
    """D 1536 with attention leaves room for 16-token preparation blocks only:
    each block must write the FFN-row map of its own tokens alone (the lanes
    past its 16 tokens belong to the next block)."""
    T, D, H, S = 256, 1536, 12, 128
    st, cfg, ws = make_block_stack(M, T, D, H, 4, 2, 256, L=1, S=S, n_shared=1, seed=13, tau0=0.7)
    rng = np.random.default_rng(130)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 3, 0.08)
    # Outputs of magnitude ~40 here: the max-abs bound follows the bf16
    # step of the value (see output_abs_bound).
    rep, _ = run_trajectory(st, cfg, ws, xs)
    assert rep.reused > 0 and rep.attn_rows > T
    st.close()


@pytest.mark.parametrize("impl", [2, 1])
def test_huge_activations_stay_finite(M, impl):
    """Block inputs of magnitude 2e4 put the scaled scores near 1e9-1e10: the
    softmax must use one rounded product for the maximum and the exponent,
    or the largest term overflows 2^x (untrained deep stacks grow this big).
    At this scale bf16 rounding of q and k moves the scores by about 1e7, so
    the softmax is an argmax that rounding decides: the check is that every
    step completes and stays finite, not parity."""
    T, D, H, S = 1024, 256, 2, 512
    st, cfg, ws = make_block_stack(M, T, D, H, 8, 2, 256, L=1, S=S, seed=14, wscale=0.2, tau0=0.72, attn_impl=impl)
    rng = np.random.default_rng(140)
    x0 = (2.0e4 * rng.standard_normal((T, D))).astype(np.float32)
    for t, x in enumerate(drift(x0, rng, 3, 200.0)):
        out = st.step(torch.from_numpy(x).cuda().to(torch.bfloat16), t)
        torch.cuda.synchronize()
        st.stats()  # raises on a device status (e.g. NaN routing)
        assert torch.isfinite(out.float()).all()
        assert torch.isfinite(st.get_state(0)["attn_a"].float()).all()
    assert st.stats()["attn_recomputed"] > T
    st.close()


def test_wide_block_separate_path(M):
    """D 2560 with 20 heads of 128: the preparation kernel does not fit next to
    the cached attention rows, so the separate router / select / compact
    kernels run with the tensor-core FFN; the output projection takes 256-wide
    tiles (residual epilogue over eight chunks)."""
    T, D, H, S = 256, 2560, 20, 256
    st, cfg, ws = make_block_stack(M, T, D, H, 4, 2, 512, L=1, S=S, n_shared=1, seed=15, wscale=0.02, tau0=0.7)
    rng = np.random.default_rng(150)
    xs = drift(rng.standard_normal((T, D)).astype(np.float32), rng, 3, 0.08)
    rep, _ = run_trajectory(st, cfg, ws, xs)
    assert rep.reused > 0 and rep.attn_rows > T
    st.close()


def test_full_step_sees_projection_weights_a_kernel_just_before_wrote(M):
    """w_qkv and w_o changed in place by kernels of the caller's, the last one
    right before a full step (whose first launch reads w_qkv), with and without
    a synchronisation in between: the same bits."""
    T, D, H, S = 512, 768, 12, 256
    rng = np.random.default_rng(160)
    x = torch.from_numpy(W.round_to_bf16(rng.standard_normal((T, D)).astype(np.float32))).cuda().to(torch.bfloat16)
    outs = []
    for wait in (True, False):
        w, _, _ = W.tiny_layer(16, T, D, 8, 2, 256, dtype="bf16", wscale=0.05)
        w.update(W.tiny_attn(16, D, dtype="bf16", wscale=0.05))
        w = {q: torch.from_numpy(v).cuda().to(torch.bfloat16) if q in ("w_qkv", "w_o") else v for q, v in w.items()}
        cfg = M.moeca_config_default(n_layers=1, hidden=D, ffn=256, n_experts=8, top_k=2, max_tokens=T, n_heads=H,
                                     seq_len=S, dtype=M.MOECA_BF16, tau0=0.72, refresh_period=1)
        st = M.Stack(cfg, [w])
        assert w["w_qkv"].data_ptr() in {k.data_ptr() for k in st._keep}  # the caller's tensor itself
        for t in range(6):
            w["w_o"].neg_()
            w["w_qkv"].mul_(-0.5 if t % 2 else -2.0)
            if wait:
                torch.cuda.synchronize()
            outs.append(st.step(x, t))
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        st.close()
    for a, b in zip(outs[:6], outs[6:]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("L", [1, 3])
def test_projection_maps_are_built_once(M, L):
    """Steps of a block stack encode one tensor map each, of the step's input
    (the warp-level attention core has none), not several per layer: the other
    projections read the handle's buffers.  Inputs in changing buffers and
    token counts below max_tokens, with the results of a handle of that size."""
    D, H, S = 256, 4, 40
    rng = np.random.default_rng(170)
    big, _, _ = make_block_stack(M, 240, D, H, 8, 2, 256, L=L, S=S, seed=17, tau0=0.72, attn_impl=1)
    for T in (120, 200, 40):
        ref, _, _ = make_block_stack(M, T, D, H, 8, 2, 256, L=L, S=S, seed=17, tau0=0.72, attn_impl=1)
        xs = [torch.from_numpy(x).cuda().to(torch.bfloat16)
              for x in drift(rng.standard_normal((T, D)).astype(np.float32), rng, 3, 0.1)]
        want = [ref.step(x, t) for t, x in enumerate(xs)]
        before = M.LIB.moeca_probe_maps_encoded()
        got = [big.step(x, t) for t, x in enumerate(xs)]
        assert M.LIB.moeca_probe_maps_encoded() - before == len(xs)
        torch.cuda.synchronize()
        assert ref.stats()["attn_recomputed"] > 0
        for a, b in zip(want, got):
            assert torch.equal(a, b)
        ref.close()
    big.close()
