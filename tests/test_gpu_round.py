"""GPU round parity against the oracle, batch invariance, forcing and edge cases."""
import numpy as np
import pytest
import torch

import synth
from oracle import decode as od
from oracle.model import Decoder
from tests.gpu_util import NEAR_TIE, decode_all, gpu_accept, lockstep, new_engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny():
    w = synth.make_weights(synth.TINY, seed=synth.WEIGHT_SEED)
    return synth.TINY, w, Decoder(synth.TINY, w)


@pytest.fixture(scope="module")
def tiny_gain():
    cfg = synth.TINY.with_(n_heads=8, n_kv_heads=4)   # GQA group 2 on the tiny decoder
    w = synth.make_weights(cfg, seed=7, gain_std=0.1)
    return cfg, w, Decoder(cfg, w)


def test_tiny_workload_lockstep(tiny):
    """Tiny decoder workload: prefix 448 visual + 64 text, K = 8, about 64 rounds."""
    cfg, w, dec = tiny
    wl = synth.WORKLOADS["tiny"]
    prompt = wl.prompts()[0]
    eng = new_engine(cfg, w, max_ctx=1024, max_K=8, max_prefill=512)
    st, stats = lockstep(eng, dec, prompt, wl.K, wl.max_new, check_logits=True)
    print(f"\ntiny lockstep: {stats}")
    assert st.done and len(st.out) == wl.max_new
    assert stats.rounds >= 30
    assert stats.max_logit_err <= 3e-2
    eng.close()


@pytest.mark.parametrize("K,n_vis,n_text", [(0, 40, 23), (1, 64, 0), (4, 0, 65), (15, 100, 27),
                                            (16, 127, 1)])
def test_tiny_gqa_gains_lockstep(tiny_gain, K, n_vis, n_text):
    """GQA group 2, non-unit norm gains, ragged prefixes around page edges, K in 0..16."""
    cfg, w, dec = tiny_gain
    prompt = synth.make_prompt(cfg, n_vis, n_text, index=K)
    eng = new_engine(cfg, w, max_ctx=512, max_K=16, max_prefill=96)   # prefill in chunks
    st, stats = lockstep(eng, dec, prompt, K, 48, check_logits=True)
    print(f"\nK={K}: {stats}")
    assert st.done and len(st.out) == 48
    eng.close()


def test_gpu_self_spec_equals_gpu_ar(tiny_gain):
    """Batch-invariant kernels: the GPU's self-speculative output equals its own
    greedy AR (K = 0) output token for token (the paper's AR-equivalence, here
    exact because a row's arithmetic does not depend on the window it sits in)."""
    cfg, w, _ = tiny_gain
    eng = new_engine(cfg, w, max_ctx=1024, max_K=16, max_prefill=256)
    prompt = synth.make_prompt(cfg, 200, 50, index=11)
    slots = torch.tensor([0], dtype=torch.int32, device=eng.device)
    outs = {}
    for K in (0, 3, 8, 16):
        x0 = eng.prefill(0, prompt.vis, prompt.text, 200)
        outs[K] = [x0] + decode_all(eng, slots, K, 400)[0]
        assert len(outs[K]) == 200
    assert outs[3] == outs[0] and outs[8] == outs[0] and outs[16] == outs[0]
    eng.close()


def test_forced_acceptance_hits_schedule(tiny_gain):
    """Forcing d_1..d_L to the greedy continuation makes the verifier accept exactly L."""
    cfg, w, _ = tiny_gain
    K, max_new = 16, 300
    eng = new_engine(cfg, w, max_ctx=2048, max_K=K, max_prefill=256)
    prompt = synth.make_prompt(cfg, 300, 20, index=12)
    slots = torch.tensor([0], dtype=torch.int32, device=eng.device)
    x0 = eng.prefill(0, prompt.vis, prompt.text, max_new + K + 4)
    ref = [x0] + decode_all(eng, slots, K, 1000)[0]
    P = prompt.length
    teacher = np.full(P + len(ref) + 4, -1, np.int32)
    teacher[P:P + len(ref)] = ref
    sched = synth.accept_schedule("geometric", K, 1, 200)
    from paper_2609_26638_gb300 import gs
    t_dev = torch.from_numpy(teacher).to(eng.device)
    s_dev = torch.from_numpy(sched).to(eng.device)
    force = gs.gs_force(teacher=t_dev.data_ptr(), teacher_stride=teacher.shape[0],
                        L_sched=s_dev.data_ptr(), L_stride=sched.shape[1])
    x0b = eng.prefill(0, prompt.vis, prompt.text, max_new)
    assert x0b == x0
    dev = eng.device
    out_tok = torch.zeros((1, K + 2), dtype=torch.int32, device=dev)
    cnt = torch.zeros(1, dtype=torch.int32, device=dev)
    done = torch.zeros(1, dtype=torch.int32, device=dev)
    torch.cuda.synchronize(dev)
    got = [x0]
    r = 0
    while True:
        eng.round(slots, K, out_tok, cnt, done, force=force)
        eng.stream.synchronize()
        c = int(cnt.cpu()[0])
        got.extend(out_tok.cpu().numpy()[0, :c].tolist())
        if int(done.cpu()[0]):
            break
        assert c == int(sched[0, r]) + 2, (r, c, sched[0, r])
        r += 1
    assert got == ref[:max_new]
    eng.check()
    eng.close()


def test_batch_equals_single_and_ragged_finish(tiny_gain):
    """Three sequences with different prefixes and caps decoded as one batch give
    the same tokens as each decoded alone; finished ones commit nothing more."""
    cfg, w, _ = tiny_gain
    K = 6
    eng = new_engine(cfg, w, max_batch=4, max_ctx=1024, max_K=K, max_prefill=256)
    prompts = [synth.make_prompt(cfg, nv, nt, index=20 + i)
               for i, (nv, nt) in enumerate([(63, 2), (130, 5), (10, 1)])]
    caps = [40, 17, 29]
    single = []
    for i, p in enumerate(prompts):
        x0 = eng.prefill(i, p.vis, p.text, caps[i])
        single.append([x0] + decode_all(eng, torch.tensor([i], dtype=torch.int32, device=eng.device),
                                         K, 100)[0])
    x0s = [eng.prefill(i, p.vis, p.text, caps[i]) for i, p in enumerate(prompts)]
    slots = torch.tensor([2, 0, 1], dtype=torch.int32, device=eng.device)   # any slot order
    outs = decode_all(eng, slots, K, 100)
    batch = {2: outs[0], 0: outs[1], 1: outs[2]}
    for i in range(3):
        assert [x0s[i]] + batch[i] == single[i]
        assert len(single[i]) == caps[i]
    eng.close()


def test_stop_token_truncates(tiny_gain):
    cfg, w, dec = tiny_gain
    prompt = synth.make_prompt(cfg, 50, 10, index=31)
    ar = od.ar_decode(dec, od.prefill(dec, prompt.vis, prompt.text, 512, 40))
    eos = ar[9]
    eng = new_engine(cfg, w, max_ctx=512, max_K=8, max_prefill=128, eos=eos)
    st, stats = lockstep(eng, dec, prompt, 8, 40, eos=eos)
    assert st.done and st.out[-1] == eos and eos not in st.out[:-1]
    eng.close()


def test_bad_requests_raise(tiny):
    from paper_2609_26638_gb300 import gs
    cfg, w, _ = tiny
    eng = new_engine(cfg, w, max_ctx=256, max_K=4, max_prefill=128)
    dev = eng.device
    slots = torch.tensor([0], dtype=torch.int32, device=dev)
    o = torch.zeros((1, 8), dtype=torch.int32, device=dev)
    c = torch.zeros(1, dtype=torch.int32, device=dev)
    d = torch.zeros(1, dtype=torch.int32, device=dev)
    with pytest.raises(gs.GsError) as e:
        eng.round(slots, 5, o, c, d)                         # K > max_K
    assert e.value.code == gs.GS_ERR_INVALID_ARG
    force = gs.gs_force(teacher=o.data_ptr(), teacher_stride=8, L_sched=c.data_ptr(), L_stride=1)
    with pytest.raises(gs.GsError) as e:                     # forcing is a greedy-only hook
        gs.gs_round(eng.handle, slots.data_ptr(), 1, 2, gs.GS_ACCEPT_STOCHASTIC, force,
                    o.data_ptr(), c.data_ptr(), d.data_ptr())
    assert e.value.code == gs.GS_ERR_INVALID_ARG
    with pytest.raises(gs.GsError) as e:
        gs.gs_round(eng.handle, slots.data_ptr(), 1, 2, 7, None, o.data_ptr(), c.data_ptr(),
                    d.data_ptr())
    assert e.value.code == gs.GS_ERR_INVALID_ARG
    with pytest.raises(gs.GsError) as e:
        eng.set_sampling(0.0, 1)
    assert e.value.code == gs.GS_ERR_INVALID_ARG
    p = synth.make_prompt(cfg, 200, 10)
    with pytest.raises(gs.GsError) as e:
        eng.prefill(0, p.vis, p.text, 100)                   # 210 + 100 + 6 > 256
    assert e.value.code == gs.GS_ERR_OOM
    with pytest.raises(gs.GsError):
        eng.prefill(3, p.vis[:8], p.text[:2], 4)             # slot out of range
    # an unprefilled slot is "done": a round commits nothing
    eng.round(slots, 2, o, c, d)
    eng.stream.synchronize()
    assert int(c.cpu()[0]) == 0 and int(d.cpu()[0]) == 1
    # out-of-range token id: the kernel clamps it and raises the device check
    bad = p.text[:4].copy()
    bad[1] = cfg.vocab + 5
    eng.prefill(0, None, bad, 4)
    with pytest.raises(gs.GsError) as e:
        eng.check()
    assert e.value.code == gs.GS_ERR_DEVICE_CHECK
    eng.check()                                            # cleared
    eng.close()


def test_bounded_wait_times_out_and_context_survives(tiny_gain):
    """Failure detection without a GPU fault: a probe kernel waits, through the
    bounded mbarrier wait every pipeline uses, on a barrier nothing arrives on,
    with a 20 ms limit.  The wait runs out, gs_sync_check reports
    GS_ERR_TIMEOUT (then the word is clear), and the context stays usable: the
    rounds that follow commit the same tokens as before the probe."""
    from paper_2609_26638_gb300 import gs
    cfg, w, _ = tiny_gain
    eng = new_engine(cfg, w, max_ctx=512, max_K=8, max_prefill=128)
    prompt = synth.make_prompt(cfg, 40, 12, index=17)
    slots = torch.tensor([0], dtype=torch.int32, device=eng.device)
    eng.prefill(0, prompt.vis, prompt.text, 24)
    before = decode_all(eng, slots, 8, 12)[0]
    gs.gs_wait_probe(eng.handle, 20000)
    with pytest.raises(gs.GsError) as e:
        eng.check()
    assert e.value.code == gs.GS_ERR_TIMEOUT
    eng.check()                                            # cleared
    with pytest.raises(gs.GsError) as e:
        gs.gs_wait_probe(eng.handle, 0)
    assert e.value.code == gs.GS_ERR_INVALID_ARG
    eng.prefill(0, prompt.vis, prompt.text, 24)
    after = decode_all(eng, slots, 8, 12)[0]
    assert after == before
    eng.close()


def test_round_profile_matches_round(tiny_gain):
    """gs_round_profile runs the same round as gs_round (same committed tokens
    and state) and reports one timed entry per kernel launch, in launch order:
    window, embed, per layer QKV / attention / O / gate-up / down, LM head, for
    the draft and the verify forward, then accept."""
    cfg, w, _ = tiny_gain
    eng = new_engine(cfg, w, max_ctx=1024, max_K=16, max_prefill=256)
    prompt = synth.make_prompt(cfg, 120, 30, index=3)
    dev = eng.device
    slots = torch.tensor([0], dtype=torch.int32, device=dev)
    K = 6
    bufs = [torch.zeros((1, K + 2), dtype=torch.int32, device=dev),
            torch.zeros(1, dtype=torch.int32, device=dev),
            torch.zeros(1, dtype=torch.int32, device=dev)]
    eng.prefill(0, prompt.vis, prompt.text, 100)
    ref = []
    for _ in range(3):
        eng.round(slots, K, *bufs)
        eng.stream.synchronize()
        ref.append(bufs[0].cpu().numpy()[0, :int(bufs[1].cpu()[0])].tolist())
    ref_state = eng.state(0)
    eng.prefill(0, prompt.vis, prompt.text, 100)
    got = []
    for _ in range(3):
        prof = eng.round_profile(slots, K, *bufs)
        got.append(bufs[0].cpu().numpy()[0, :int(bufs[1].cpu()[0])].tolist())
    assert got == ref
    assert eng.state(0) == ref_state
    fwd = ["embed"] + ["qkv", "attention", "o_proj", "gate_up", "down"] * cfg.n_layers + ["lm_head"]
    assert [k for k, _ in prof] == ["window"] + fwd + ["window"] + fwd + ["accept"]
    assert len(prof) == gs_launches(eng)
    assert all(ms > 0 for _, ms in prof)
    eng.check()
    eng.close()


def gs_launches(eng):
    from paper_2609_26638_gb300 import gs
    return gs.gs_round_launches(eng.handle)


@pytest.mark.parametrize("K,split_pages,max_ctx", [(16, 0, 512), (31, 0, 512), (31, 1, 2048)])
def test_windows_of_more_than_128_rows_at_a_page_edge(K, split_pages, max_ctx):
    """GQA group 8: a window's (K + 1) * 8 rows exceed one query block of 128, and
    the second block's key limits lie inside the window.  The first window starts
    a few slots below a page edge, so its own slots complete a page that an item
    loads first: that page counts as committed for no block of the window.
    Clusters of items and (32 items of one page) persistent CTAs; in lock-step
    with the oracle, and as graph launches equal to greedy AR token for token."""
    cfg = synth.TINY.with_(n_heads=16, n_kv_heads=2)
    w = synth.make_weights(cfg, seed=9, gain_std=0.1)
    prompt = synth.make_prompt(cfg, 100, 22, index=K)          # n = 122, edges at 128 and 192
    eng = new_engine(cfg, w, max_ctx=max_ctx, max_K=K, max_prefill=128, split_pages=split_pages)
    st, stats = lockstep(eng, Decoder(cfg, w), prompt, K, 48, check_logits=True)
    print(f"\nK={K}: {stats}")
    assert st.done and len(st.out) == 48
    slots = torch.tensor([0], dtype=torch.int32, device=eng.device)
    outs = []
    for k in (0, K):
        x0 = eng.prefill(0, prompt.vis, prompt.text, 80)
        outs.append([x0] + decode_all(eng, slots, k, 80)[0])
    assert len(outs[0]) == 80 and outs[1] == outs[0]
    eng.close()


def _merge_tickets(eng):
    """The attention's merge tickets, one int32 per (query block, KV head): a view
    into the engine's workspace, found from its end (the pieces behind the tickets,
    each starting on 256 bytes).  The denoising step counts lie on the way."""
    c, up = eng.cfg, lambda n: (n + 255) // 256 * 256
    W, G = c.max_K + 1, c.n_heads // c.n_kv_heads
    rows = c.max_batch * W
    weights = sum(t.numel() for lw in eng.layers for n, t in lw.items() if n.startswith("w_"))
    weights += eng.w["lm_head"].numel()
    off = eng.ws_bytes
    for nbytes in (2 * weights, 16 * rows, 4 * rows * c.vocab, 4 * rows * c.vocab,
                   8 * rows * (c.vocab // 128), 8 * rows * (c.vocab // 128), 256):
        off -= up(nbytes)
    words = eng.workspace.view(torch.int32)
    off -= up(4 * c.max_batch)
    steps = words[off // 4:off // 4 + c.max_batch]
    off -= 2 * up(4 * c.max_batch) + up(4 * rows)
    qb = 128 // G
    n_sub = -(-W // min(W, qb))
    T_max = up(max(rows, c.max_prefill, 256))
    blocks = max(c.max_batch * n_sub, -(-min(c.max_prefill, T_max) // qb))
    off -= up(4 * blocks * c.n_kv_heads)
    return words[off // 4:off // 4 + blocks * c.n_kv_heads], steps


def test_timeout_report_resets_the_merge_tickets(tiny_gain):
    """A launch whose wait runs out drops work items, which can leave merge tickets
    behind; with one left, a later launch would merge before its last item has
    arrived.  The report of the failure clears them: tickets are planted and the
    failure raised from the host, and after gs_sync_check the words are zero and a
    decode through the persistent attention (32 items of one page) commits what it
    did before."""
    from paper_2609_26638_gb300 import gs
    cfg, w, _ = tiny_gain
    eng = new_engine(cfg, w, max_batch=2, max_ctx=2048, max_K=8, max_prefill=256, split_pages=1)
    prompt = synth.make_prompt(cfg, 300, 12, index=41)
    slots = torch.tensor([0], dtype=torch.int32, device=eng.device)
    tickets, steps = _merge_tickets(eng)
    out = torch.zeros((3, 8), dtype=torch.int32, device=eng.device)
    eng.prefill(0, prompt.vis, prompt.text, 40)
    eng.diffusion_block(slots, 4, 2.0, out[0], out[1], out[2])
    eng.stream.synchronize()
    assert steps.tolist() == [4, 0]                      # the view is where it is said to be
    eng.prefill(0, prompt.vis, prompt.text, 40)
    before = decode_all(eng, slots, 8, 40)[0]
    assert not tickets.any()
    tickets.fill_(1)
    torch.cuda.synchronize()
    gs.gs_wait_probe(eng.handle, 1000)
    with pytest.raises(gs.GsError) as e:
        eng.check()
    assert e.value.code == gs.GS_ERR_TIMEOUT
    torch.cuda.synchronize()
    assert not tickets.any()
    eng.prefill(0, prompt.vis, prompt.text, 40)
    assert decode_all(eng, slots, 8, 40)[0] == before
    eng.close()


def test_calls_after_an_earlier_failure(tiny_gain):
    """A call that failed on the host (a round while its stream is being captured)
    leaves nothing behind for the calls after it: the attention and the projection
    judge their own launches only."""
    from paper_2609_26638_gb300 import gs
    cfg, w, _ = tiny_gain
    eng = new_engine(cfg, w, max_ctx=256, max_K=4, max_prefill=128)
    dev = eng.device
    o = torch.zeros((1, 8), dtype=torch.int32, device=dev)
    slots = torch.zeros(1, dtype=torch.int32, device=dev)
    M, N, K = 100, 256, 256
    x = torch.randn(M, K, device=dev).half()
    wl = torch.randn(N, K, device=dev).half()
    y = torch.zeros(M, N, dtype=torch.float16, device=dev)
    sl = torch.zeros(gs.gs_linear_scratch_bytes(M, N, 1), dtype=torch.uint8, device=dev)
    q = torch.randn(1, 5, 8, 64, device=dev).half()
    kv = torch.randn(2, 2, 4, 64, 64, device=dev).half()
    pt = torch.tensor([[1, 0]], dtype=torch.int32, device=dev)
    n = torch.tensor([70], dtype=torch.int32, device=dev)
    out = torch.zeros_like(q)
    sa = torch.zeros(gs.gs_attention_scratch_bytes(1, 5, 8, 4, 2, 1), dtype=torch.uint8, device=dev)
    s = torch.cuda.current_stream(dev).cuda_stream

    def calls():
        gs.gs_attention(1, q.data_ptr(), kv.data_ptr(), 2, pt.data_ptr(), 2, n.data_ptr(), 1, 5, 8, 4,
                        out.data_ptr(), sa.data_ptr(), sa.numel(), 1, s)
        gs.gs_linear(x.data_ptr(), wl.data_ptr(), y.data_ptr(), M, N, K, gs.EPI_STORE_F16, 1,
                     sl.data_ptr(), sl.numel(), s)
        torch.cuda.synchronize()
        return out.clone(), y.clone()

    want = calls()

    def fail():
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(eng.stream):
            graph.capture_begin(capture_error_mode="thread_local")
            with pytest.raises(gs.GsError) as e:
                gs.gs_round(eng.handle, slots.data_ptr(), 1, 2, gs.GS_ACCEPT_GREEDY, None,
                            o.data_ptr(), o.data_ptr(), o.data_ptr())
            assert e.value.code == gs.GS_ERR_CUDA
            graph.capture_end()

    fail()
    for got, ref in zip(calls(), want):
        assert torch.equal(got, ref)
    fail()
    gs.gs_linear(x.data_ptr(), wl.data_ptr(), y.data_ptr(), M, N, K, gs.EPI_STORE_F16, 1,
                 sl.data_ptr(), sl.numel(), s)
    torch.cuda.synchronize()
    eng.close()


def test_engine_after_an_earlier_failure(tiny_gain):
    """The same for the calls of a decoder: one is built and prefilled after a round
    that could not be captured."""
    from paper_2609_26638_gb300 import gs
    cfg, w, _ = tiny_gain
    eng = new_engine(cfg, w, max_ctx=256, max_K=4, max_prefill=128)
    o = torch.zeros((1, 8), dtype=torch.int32, device=eng.device)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(eng.stream):
        graph.capture_begin(capture_error_mode="thread_local")
        with pytest.raises(gs.GsError) as e:
            gs.gs_round(eng.handle, o.data_ptr(), 1, 2, gs.GS_ACCEPT_GREEDY, None, o.data_ptr(),
                        o.data_ptr(), o.data_ptr())
        assert e.value.code == gs.GS_ERR_CUDA and "Capture" in str(e.value)
        graph.capture_end()
    p = synth.make_prompt(cfg, 20, 5, index=1)
    x0 = eng.prefill(0, p.vis, p.text, 8)
    other = new_engine(cfg, w, max_ctx=256, max_K=4, max_prefill=128)
    assert other.prefill(0, p.vis, p.text, 8) == x0
    eng.close()
    other.close()


def test_wide_model_batch_equals_single():
    """d_model 4096: the QKV projection's split forms clusters of eight also above 64
    rows.  Eight sequences in one batch (136 rows) commit what each commits alone
    (17 rows, and 17-row windows are in lock-step with the oracle)."""
    cfg = synth.TINY.with_(n_layers=1, d_model=4096, n_heads=8, n_kv_heads=4)
    w = synth.make_weights(cfg, seed=13)
    K, B, cap = 16, 8, 24
    eng = new_engine(cfg, w, max_batch=B, max_ctx=256, max_K=K, max_prefill=128)
    prompts = [synth.make_prompt(cfg, 20 + 9 * i, 5, index=60 + i) for i in range(B)]
    st, stats = lockstep(eng, Decoder(cfg, w), prompts[0], K, cap, check_logits=True)
    assert st.done
    single = []
    for i, p in enumerate(prompts):
        eng.prefill(i, p.vis, p.text, cap)
        single.append(decode_all(eng, torch.tensor([i], dtype=torch.int32, device=eng.device), K, 40)[0])
    for i, p in enumerate(prompts):
        eng.prefill(i, p.vis, p.text, cap)
    slots = torch.arange(B, dtype=torch.int32, device=eng.device)
    assert decode_all(eng, slots, K, 40) == single
    eng.close()


def test_weights_of_a_little_more_than_one_wave():
    """Gate/up (160 tiles) and LM head (153 tiles) of one to one and a half tiles per
    SM: one sequence in lock-step with the oracle (17-row windows), and a batch of
    five (85 rows) commits what each commits alone."""
    cfg = synth.TINY.with_(n_layers=1, n_heads=8, n_kv_heads=4, d_ffn=10240, vocab=153 * 128)
    w = synth.make_weights(cfg, seed=17)
    K, B, cap = 16, 5, 24
    eng = new_engine(cfg, w, max_batch=B, max_ctx=256, max_K=K, max_prefill=128)
    prompts = [synth.make_prompt(cfg, 20 + 9 * i, 5, index=80 + i) for i in range(B)]
    st, stats = lockstep(eng, Decoder(cfg, w), prompts[0], K, cap, check_logits=True)
    assert st.done
    single = []
    for i, p in enumerate(prompts):
        eng.prefill(i, p.vis, p.text, cap)
        single.append(decode_all(eng, torch.tensor([i], dtype=torch.int32, device=eng.device), K, 40)[0])
    for i, p in enumerate(prompts):
        eng.prefill(i, p.vis, p.text, cap)
    slots = torch.arange(B, dtype=torch.int32, device=eng.device)
    assert decode_all(eng, slots, K, 40) == single
    eng.close()
