"""GPU parity of the PARD decode step against the CPU oracle, through the
C ABI.  Every test builds both sides from the same seeded inputs."""
import numpy as np
import pytest

import oracle
import synthetic as S
from oracle import pard as OP
from oracle.philox import STREAM_ACCEPT, STREAM_BONUS, STREAM_DRAFT, raw_words, uniform01

from _parity import GUMBEL_EPS, LOGIT_TOL, MARGIN, Pair, check_token, greedy_step, gumbel_scores, margin, sampling_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2504_18583_gb300 import _build
    _build.build()


def run_greedy(P: Pair, max_steps=64, inject_fn=None, sequential=False):
    P.prefill()
    step = 1
    outs = []
    while not P.oracle.all_done() and step <= max_steps:
        inject = inject_fn(P, step) if inject_fn else None
        outs.append(greedy_step(P, step, inject, sequential))
        step += 1
    n, gen, done = P.eng.state()
    assert done == [1 if d else 0 for d in P.oracle.done]
    assert P.eng.last_status() == 0
    return outs


def test_tiny_greedy_matches_oracle_every_step():
    """The tiny configuration (FFN 688: ragged row-major gate/up/down tiles)
    against the oracle step by step; and with FFN 768, where every matrix
    takes the packed layout."""
    for ffn in (688, 768):
        wl = S.WORKLOADS["tiny"]
        wl = wl.replace(target=wl.target.replace(ffn=ffn), draft=wl.draft.replace(ffn=ffn))
        P = Pair(wl)
        run_greedy(P)
        assert P.oracle.all_done()
        # the generated sequence equals autoregressive greedy decoding where margins are clear
        assert P.stats["excused_tokens"] <= P.stats["checked_tokens"] // 10
        print("ffn", ffn, "stats", P.stats)


def test_vanilla_sd_sequential_draft_matches_oracle_every_step():
    """Vanilla speculative decoding (K sequential draft passes, Section 2.2)
    on the same kernels: draft logits, candidates, accept lengths and slots
    against the oracle's sequential draft, batch 2, ragged prompts; with the
    target as its own draft every candidate but the last step's is accepted."""
    wl = S.WORKLOADS["tiny"].replace(batch=2, prompt_len=None, prompt_len_range=(20, 45), n_new=24)
    P = Pair(wl)
    run_greedy(P, sequential=True)
    assert P.oracle.all_done()
    print("stats", P.stats)
    wl2 = S.WORKLOADS["tiny"].replace(n_new=20, prompt_len=30)
    P2 = Pair(wl2, draft_is_target=True)
    outs = run_greedy(P2, sequential=True)
    accs = [int(o["a"][0]) for o in outs]
    assert max(accs) == wl2.K
    print("accept lengths", accs, P2.stats)


def test_distinct_mask_ids_and_k12_match_oracle_every_step():
    """One mask id per offset (Section 4.3's alternative to the shared id)
    and K = 12 (verify 13 rows, draft up to 24 rows per sequence: two
    attention row blocks), batch 2, against the oracle step by step; the
    argument and state checks of pard_set_mask_ids."""
    from paper_2504_18583_gb300 import pard
    wl = S.WORKLOADS["tiny"].replace(K=12, batch=2, n_new=24, prompt_len=None, prompt_len_range=(20, 45))
    V = wl.draft.vocab
    ids = [V - 2 - k for k in range(wl.K - 1)]
    P = Pair(wl)
    P.eng.set_mask_ids(ids)
    P.oracle.mask_ids = ids
    run_greedy(P)
    assert P.oracle.all_done()
    print("stats", P.stats)
    with pytest.raises(pard.PardError):
        P.eng.set_mask_ids(list(range(wl.K)))       # more than max_k - 1 offsets
    with pytest.raises(pard.PardError):
        P.eng.set_mask_ids([V] + ids[1:])            # outside the vocabulary
    P.eng.set_mask_ids(ids[:3])                      # too few for K - 1 = 11 mask rows
    P.eng.prefill(P.prompts, wl.n_new, wl.K)
    out = P.eng.alloc_step_outputs()
    with pytest.raises(pard.PardError):
        P.eng.draft(out)
    P.eng.set_mask_ids(None)


def test_stalled_wait_is_reported_and_the_context_stays_usable():
    """Failure detection without a GPU fault: a kernel's bounded pipeline wait
    on a barrier nothing completes gives up after its limit, sets the timeout
    bit and returns; pard_last_status reports it, and the next decode steps
    still match the oracle."""
    wl = S.WORKLOADS["tiny"].replace(n_new=12)
    P = Pair(wl)
    P.prefill()
    greedy_step(P, 1)
    assert P.eng.last_status() == 0
    P.eng.selftest_stalled_wait()
    assert P.eng.last_status() == 1  # ST_TIMEOUT_TMA
    greedy_step(P, 2)
    assert P.eng.last_status() == 0


def test_cod_keep_flags_match_the_oracle_bit_exactly():
    """COD data construction (Section 3.2, appendix algorithm) on the GPU:
    keep flags and per-subtask counts identical to the oracle's for ragged
    sample lengths, K = 1..8, several retention settings, the 4096-row
    maximum and the degenerate cases (n = 1, r = 1, r_min = 1)."""
    import torch
    from oracle import cod
    from paper_2504_18583_gb300 import pard
    cases = [(1, 3, 0.5, 0.0), (4, 3, 0.5, 0.0), (37, 2, 0.5, 0.0), (500, 8, 0.5, 0.0), (777, 6, 0.7, 0.1),
             (2048, 8, 0.5, 0.05), (4096, 8, 0.6, 0.0), (64, 1, 0.5, 0.0), (100, 5, 1.0, 0.0), (100, 5, 0.3, 1.0)]
    for t, (n, K, r, r_min) in enumerate(cases):
        keep_g, counts_g = pard.cod_select(n, K, r, r_min, seed=1000 + t, sample_id=t)
        keep_o, counts_o = cod.cod_select(n, K, r, r_min, seed=1000 + t, sample_id=t)
        torch.cuda.synchronize()
        assert counts_g.cpu().tolist() == counts_o, (n, K, r, r_min)
        assert np.array_equal(keep_g.cpu().numpy(), keep_o), (n, K, r, r_min)
    # one 2048-row, K = 8 sample, timed on the device
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    pard.cod_select(2048, 8, 0.5, 0.0, 1, 0)
    ev[0].record()
    for i in range(20):
        pard.cod_select(2048, 8, 0.5, 0.0, 1, i)
    ev[1].record()
    torch.cuda.synchronize()
    print("COD 2048 rows, K = 8: %.1f us per sample" % (ev[0].elapsed_time(ev[1]) * 1e3 / 20))


def test_page_pool_exhaustion_and_device_bounds_flag():
    """Host and device checks without a fault: a batch whose page reservation
    exceeds the pool returns PARD_ERR_NO_PAGES before any launch; a verify
    candidate outside the vocabulary is caught by the row-plan kernel, which
    flags ST_BAD_TOKEN (read by pard_last_status as PARD_ERR_DEVICE_CHECK)
    and embeds token 0 instead of reading out of bounds."""
    import torch
    from paper_2504_18583_gb300 import pard
    wl = S.WORKLOADS["tiny"].replace(n_new=20, prompt_len=40)
    tw = S.device_weights(wl.target, wl.seed, S.TARGET)
    dw = S.device_weights(wl.draft, wl.seed, S.DRAFT)
    eng = pard.PardEngine(wl.target, tw, wl.draft, dw, max_batch=1, max_k=wl.K, max_ctx=256, n_pages=2,
                          prefill_chunk=64)
    with pytest.raises(pard.PardError) as e:
        eng.prefill([list(range(1, 41))], wl.n_new, wl.K)
    assert e.value.code == -3  # PARD_ERR_NO_PAGES: 40 + 20 + 2K positions need 5 pages of 16
    P = Pair(wl)
    P.prefill()
    out = P.eng.alloc_step_outputs()
    P.eng.draft(out)
    bad = torch.full((1, wl.K), wl.target.vocab + 5, dtype=torch.int32, device="cuda")
    P.eng.verify(out, bad)
    assert P.eng.last_status() == 1 << 3  # ST_BAD_TOKEN
    assert P.eng.last_status() == 0       # the word is cleared once read


def test_tiny_greedy_jittered_norms_batch_ragged():
    """Batch of 3 with prompts 17 / 33 / 50 tokens (page boundaries at
    several offsets), norm gains != 1, prefill chunks of 64 rows."""
    wl = S.WORKLOADS["tiny"].replace(batch=3, prompt_len=None, prompt_len_range=(17, 50), norm_jitter=0.1,
                                     n_new=20)
    wl = wl.replace(target=wl.target.replace(ffn=768), draft=wl.draft.replace(ffn=768))
    P = Pair(wl)
    run_greedy(P)
    print("stats", P.stats)


def test_self_draft_accepts_and_rolls_back():
    """Draft = target: d_0 always equals the target's argmax, so every step
    accepts at least one candidate and commit/rollback runs with a > 0."""
    wl = S.WORKLOADS["tiny"].replace(n_new=30, batch=2, prompt_len=40)
    P = Pair(wl, draft_is_target=True)
    outs = run_greedy(P)
    accs = [int(o["a"][b]) for o in outs for b in range(2)]
    assert max(accs) >= 1
    print("accept lengths", accs, P.stats)


def test_injected_candidates_hit_every_accept_length():
    """pard_verify on the target's own greedy continuation with one planted
    mismatch at j accepts exactly j candidates (j = K: none planted)."""
    wl = S.WORKLOADS["tiny"].replace(n_new=40)
    P = Pair(wl)
    K = wl.K
    ar = oracle.ar_greedy(wl.target, P.tw_host, P.prompts[0], wl.n_new + K + 2)
    seen = set()

    def inject(P, step):
        n0 = len(P.oracle.generated[0])
        j = (step - 1) % (K + 1)
        cont = list(ar[n0:n0 + K])
        while len(cont) < K:
            cont.append(0)
        if j < K:
            cont[j] = (cont[j] + 1) % (wl.target.vocab - 1)
        return np.array([cont], dtype=np.int32)

    outs = run_greedy(P, inject_fn=inject)
    for s, o in enumerate(outs):
        seen.add(int(o["a"][0]))
    assert seen >= set(range(K + 1)) - {K} or len(seen) >= K
    print("accept lengths seen", sorted(seen), P.stats)


def test_kv_cache_holds_the_oracle_keys_and_values():
    wl = S.WORKLOADS["tiny"].replace(n_new=12)
    P = Pair(wl)
    run_greedy(P)
    n = P.oracle.n[0]
    pos = list(range(0, n - 1))
    for model, om, shape in ((0, P.oracle.T, wl.target), (1, P.oracle.D, wl.draft)):
        upto = n - 1 if model == 0 else n - len(P.oracle.pending[0])
        for layer in (0, shape.n_layers - 1):
            k, v = P.eng.read_kv(model, layer, 0, pos[:upto], shape)
            k = k.float().cpu().numpy()
            v = v.float().cpu().numpy()
            ko = om.kc[0][layer, :upto]
            vo = om.vc[0][layer, :upto]
            # bf16 storage: relative 2^-8 plus the accumulated logit-level error
            assert np.abs(k - ko).max() <= 0.02 * max(1.0, np.abs(ko).max())
            assert np.abs(v - vo).max() <= 0.02 * max(1.0, np.abs(vo).max())


def test_full_width_8b_layers_short_prompt():
    """8B-shaped target and 1B-shaped draft at full width (every GEMM,
    attention and LM-head tile count of the full models), two layers each,
    64-token prompt, three steps; K = 8 gives 16 draft rows and 9 verify rows."""
    wl = S.WORKLOADS["8b_greedy"].replace(target=S.TARGET_8B.replace(n_layers=2),
                                          draft=S.DRAFT_1B.replace(n_layers=2), prompt_len=64, n_new=20)
    P = Pair(wl, prefill_chunk=64)
    P.prefill()
    for step in range(1, 4):
        greedy_step(P, step)
    assert P.eng.last_status() == 0
    print("stats", P.stats)


def test_autoregressive_mode_k0_matches_the_oracle_forward():
    """K = 0: each pard_verify + pard_accept_commit decodes one token with the
    target alone (Eq. 2); logits and tokens against one oracle forward per
    token, teacher-forced onto the GPU's token."""
    from paper_2504_18583_gb300 import pard
    wl = S.WORKLOADS["tiny"].replace(n_new=20)
    tw = S.model_weights(wl.target, wl.seed, S.TARGET, wl.norm_jitter)
    dw = S.model_weights(wl.draft, wl.seed, S.DRAFT, wl.norm_jitter)
    prompt = [int(t) for t in wl.prompts()[0]]
    P_len = len(prompt)
    eng = pard.PardEngine(wl.target, S.device_weights(wl.target, 0, 0, host=tw), wl.draft,
                          S.device_weights(wl.draft, 0, 0, host=dw), max_batch=1, max_k=wl.K,
                          max_ctx=P_len + wl.n_new + 2 * wl.K + 16, n_pages=wl.n_pages(), prefill_chunk=64,
                          page_order_target=wl.page_order(S.TARGET), page_order_draft=wl.page_order(S.DRAFT))
    stats = dict(excused_tokens=0, checked_tokens=0)
    m = oracle.OracleModel(wl.target, tw, 1, P_len + wl.n_new + 2)
    lg = m.forward(0, prompt, np.arange(P_len, dtype=np.int32), [P_len - 1])[0]
    tok = int(eng.prefill([prompt], wl.n_new, 0).cpu().numpy()[0])
    check_token(tok, lg, stats, "first token")
    out = eng.alloc_step_outputs(want_logits=True)
    for step in range(1, wl.n_new):
        eng.verify(out, None, 1.0)
        y = out["logits"][0, 0].cpu().numpy()
        lg = m.forward(0, [tok], [P_len + step - 1], [0])[0]
        assert float(np.abs(y - lg).max()) <= LOGIT_TOL, f"step {step}"
        eng.accept_commit(out, False, 1.0, 0, step)
        assert int(out["n_emit"][0]) == 1 and int(out["accept_len"][0]) == 0
        tok = int(out["emitted"][0, 0])
        check_token(tok, lg, stats, f"step {step}")
    n, gen, done = eng.state()
    assert gen == [wl.n_new] and done == [1]
    assert eng.last_status() == 0
    with pytest.raises(RuntimeError):
        eng.draft(out)
    print("stats", stats)


def test_batch16_ragged_full_width_two_layers():
    """The batch-16 ragged configuration (8b_batch16: K = 6, ragged prompts)
    at full width with two layers per model: 16 x 7 = 112 verify rows and 192
    draft rows take the CTA pairs' tiles, and attention covers 16 sequences of
    different lengths.  Prompts are 16..64 tokens here (the configuration's
    128..2048 keep the CPU oracle's prefill within seconds only at this size)."""
    wl = S.WORKLOADS["8b_batch16"].replace(target=S.TARGET_8B.replace(n_layers=2),
                                           draft=S.DRAFT_1B.replace(n_layers=2), prompt_len_range=(16, 64), n_new=12)
    P = Pair(wl, prefill_chunk=64)
    P.prefill()
    for step in range(1, 4):
        greedy_step(P, step)
    assert P.eng.last_status() == 0
    print("stats", P.stats)


# ----------------------------------------------------------------------------
# speculative sampling
# ----------------------------------------------------------------------------
def test_sampling_decisions_on_identical_logits():
    """Level 1: the oracle's logits fed to the GPU acceptance kernels with the
    same Philox streams give the same accept/reject decisions and bonus draws
    (except where u*q and p are within a few ulps)."""
    import torch
    wl = S.WORKLOADS["tiny"].replace(sample=True, n_new=1000, K=4)
    P = Pair(wl)
    P.prefill(seed=5)
    rng = np.random.default_rng(0)
    V, K = wl.target.vocab, wl.K
    mism = 0
    for trial in range(40):
        y = (rng.standard_normal((1, K + 1, V)) * 2.0).astype(np.float32)
        z = (y[:, :K] + rng.standard_normal((1, K, V)).astype(np.float32) * (0.3 + 0.1 * (trial % 5))).astype(np.float32)
        d = np.array([OP.draft_tokens(z[0], True, 1.0, 77 + trial, 3, 0)], dtype=np.int32)
        P.eng.set_logits(torch.as_tensor(y, device="cuda"), torch.as_tensor(z, device="cuda"),
                         torch.as_tensor(d, device="cuda"), 1.0)
        out = P.eng.alloc_step_outputs()
        step = 1000 + trial
        n_before = P.eng.state()[0][0]
        P.eng.accept_commit(out, True, 1.0, 5, step)
        a_g = int(out["accept_len"][0])
        em_g = out["emitted"][0].cpu().numpy()
        a_o, em_o = OP.accept_sampling(d[0], z[0], y[0], 1.0, 5, step, 0)
        if a_o != a_g:
            # excuse only a decision within rounding of the threshold
            i = min(a_o, a_g)
            p = OP.softmax_t(y[0, i], 1.0)[d[0, i]]
            q = OP.softmax_t(z[0, i], 1.0)[d[0, i]]
            u = uniform01(raw_words(5, STREAM_ACCEPT, step, 0, i, np.zeros(1, np.uint64)))[0]
            assert abs(u * q - p) <= 1e-5 * max(p, q), (trial, a_o, a_g)
            mism += 1
            continue
        take = int(out["n_emit"][0])
        assert list(em_g[:take]) == em_o[:take], (trial, em_g, em_o)
    assert mism <= 2


def test_sampling_end_to_end_tiny():
    """Level 2: sampling decode end to end (tiny models, batch 2, ragged
    prompts).  The sampled first token, the draft's Gumbel-max candidates,
    the accept / reject decisions and the bonus draws agree with the
    oracle's on the same Philox streams wherever the margins are clear (the
    margins follow from the measured logit differences); the oracle follows
    the GPU's tokens."""
    wl = S.WORKLOADS["tiny"].replace(sample=True, n_new=40, batch=2, prompt_len=None, prompt_len_range=(20, 45))
    P = Pair(wl)
    seed = 11
    P.prefill(seed)
    step = 1
    while not P.oracle.all_done() and step < 60:
        sampling_step(P, step, seed)
        step += 1
    assert P.oracle.all_done()
    st = P.stats
    print("stats", st)
    assert st["decisions_checked"] > 0
    # draft candidates, first tokens and bonus draws: nearly all have clear margins
    assert st["sampled_exact"] >= 0.9 * st["sampled_checked"]
    assert P.eng.last_status() == 0


def test_sampling_full_width_8b_two_layers():
    """The sampling configuration (8b_sample: T = 1, K = 6) at full width with
    two layers per model, 64-token prompt: logits within tolerance; sampled
    candidates, first token, decisions and bonus draws as in the tiny test;
    KV slots equal."""
    wl = S.WORKLOADS["8b_sample"].replace(target=S.TARGET_8B.replace(n_layers=2),
                                          draft=S.DRAFT_1B.replace(n_layers=2), prompt_len=64, n_new=24)
    P = Pair(wl, prefill_chunk=64)
    seed = 5
    P.prefill(seed)
    for step in range(1, 5):
        sampling_step(P, step, seed)
    st = P.stats
    print("stats", st)
    assert st["sampled_exact"] >= 0.9 * st["sampled_checked"]
    assert P.eng.last_status() == 0


def test_vanilla_sd_sampled_sequential_draft():
    """The sampled form of vanilla speculative decoding's drafting stage
    (Section 2.2): every draft pass draws its candidate by Gumbel-max from
    its own logits (Philox stream 0, row i); candidates, decisions and bonus
    draws against the oracle's sequential draft fed the GPU's candidates,
    margins as in the other sampling tests; batch 2, ragged prompts."""
    wl = S.WORKLOADS["tiny"].replace(sample=True, n_new=30, batch=2, prompt_len=None, prompt_len_range=(20, 45))
    P = Pair(wl)
    seed = 13
    P.prefill(seed)
    step = 1
    while not P.oracle.all_done() and step < 40:
        sampling_step(P, step, seed, sequential=True)
        step += 1
    st = P.stats
    print("stats", st)
    assert P.oracle.all_done()
    assert st["sampled_exact"] >= 0.9 * st["sampled_checked"]
    assert P.eng.last_status() == 0


@pytest.mark.parametrize("vocab", [2048, 128256])
def test_draft_sampler_on_identical_logits(vocab):
    """Level 1 for the draft's candidate selection (Eq. 6, sampled at
    temperature T, and greedy): given draft logits go through statistics of
    the LM head's layout, every entry scored exactly, and the same selection
    kernel, and the candidates equal the oracle's Gumbel-max (or argmax)
    winners on the same Philox stream exactly, except where the winner's lead
    is a few fp32 ulps.  (The LM head's own draw:
    test_lm_head_draw_follows_its_own_logits.)"""
    import torch
    wl = S.WORKLOADS["tiny"].replace(batch=3, K=6, n_new=100, prompt_len=20)
    if vocab != wl.target.vocab:
        wl = wl.replace(target=wl.target.replace(vocab=vocab, mask_id=vocab - 1),
                        draft=wl.draft.replace(vocab=vocab, mask_id=vocab - 1))
    P = Pair(wl)
    P.prefill()
    B, K, V = wl.batch, wl.K, vocab
    rng = np.random.default_rng(vocab)
    near = exact = 0
    for trial in range(12):
        T = (0.7, 1.0, 1.3)[trial % 3]
        sample = trial % 4 != 3
        z = (rng.standard_normal((B, K, V)) * 2.0).astype(np.float32)
        out = P.eng.alloc_step_outputs()
        seed, step = 31 + trial, 200 + trial
        P.eng.set_draft_logits(torch.as_tensor(z, device="cuda"), out, sample, T, seed, step)
        d_g = out["draft"].cpu().numpy()
        for b in range(B):
            d_o = OP.draft_tokens(z[b], sample, T, seed, step, b)
            for i in range(K):
                if int(d_g[b, i]) == d_o[i]:
                    exact += 1
                    continue
                sc = (gumbel_scores(z[b, i], T, seed, STREAM_DRAFT, step, b, i) if sample
                      else z[b, i].astype(np.float32))
                assert margin(sc) <= GUMBEL_EPS, (trial, b, i, int(d_g[b, i]), d_o[i], margin(sc))
                near += 1
    print("exact", exact, "near ties", near)
    assert near <= 2 and exact >= B * K * 12 - 2


def test_weight_packing_round_trip_restores_every_matrix():
    """Loading packs the weight matrices in place; unpacking restores the
    exact row-major bits (including a draft sharing the target's tensors)."""
    import torch
    wl = S.WORKLOADS["tiny"].replace(target=S.TARGET_8B.replace(n_layers=1, vocab=2048, mask_id=2047),
                                     draft=S.DRAFT_1B.replace(n_layers=1, vocab=2048, mask_id=2047))
    P = Pair(wl)
    host = P.tw_host
    dev = P.tw_dev
    packed_any = not torch.equal(dev["layers"][0]["wq"].view(torch.int16).cpu(),
                                 torch.from_numpy(host["layers"][0]["wq"].view("int16")))
    assert packed_any, "wq should be in the packed layout while loaded"
    P.eng.unpack_weights()
    for name in ("wq", "wk", "wv", "wo", "wg", "wu", "wd"):
        got = dev["layers"][0][name].view(torch.int16).cpu().numpy()
        assert np.array_equal(got, host["layers"][0][name].view("int16")), name
    assert np.array_equal(dev["lm_head"].view(torch.int16).cpu().numpy(), host["lm_head"].view("int16"))
    with pytest.raises(Exception):
        P.eng.prefill([[1, 2, 3]], 4, wl.K)


def test_state_errors_are_reported():
    from paper_2504_18583_gb300 import pard
    wl = S.WORKLOADS["tiny"]
    P = Pair(wl)
    out = P.eng.alloc_step_outputs()
    with pytest.raises(pard.PardError) as e:
        P.eng.draft(out)
    assert e.value.code == -7
    with pytest.raises(pard.PardError) as e:
        P.eng.prefill([list(range(10))], 10_000, wl.K)
    assert e.value.code == -1


def test_cod_threshold_bins_at_the_edges():
    """COD rows at the edges of the four-rows-a-thread split and of the
    threshold search: row counts around multiples of four, keep counts of
    zero, of one and of every candidate, and more subtasks than rows."""
    import torch
    from oracle import cod
    from paper_2504_18583_gb300 import pard
    for t, (n, K, r, r_min) in enumerate([(3, 6, 0.9, 0.0), (5, 4, 0.01, 0.0), (127, 12, 0.95, 0.0), (4093, 3, 0.999, 0.0),
                                          (4095, 16, 0.5, 0.001), (4096, 3, 1.0, 0.0), (8, 64, 1.0, 1.0)]):
        keep_g, counts_g = pard.cod_select(n, K, r, r_min, seed=(1 << 40) + t, sample_id=7 * t)
        keep_o, counts_o = cod.cod_select(n, K, r, r_min, seed=(1 << 40) + t, sample_id=7 * t)
        torch.cuda.synchronize()
        assert counts_g.cpu().tolist() == counts_o, (n, K, r, r_min)
        assert np.array_equal(keep_g.cpu().numpy(), keep_o), (n, K, r, r_min)


@pytest.mark.parametrize("batch,K,lens,chunk", [(13, 4, (3, 70), 64), (16, 7, (5, 20), 320), (2, 4, (300, 330), 320),
                                                (1, 3, (600, 600), 576)],
                         ids=["65_rows", "128_rows_prefill_odd", "two_token_tiles", "three_token_tiles"])
def test_wide_gemm_tile_edges(batch, K, lens, chunk):
    """Passes of more than 64 rows (CTA pairs of 256 weight rows): row counts
    at and beside a tile's edges, one to three token tiles, odd numbers of
    128-row weight tiles (d 384, FFN 704, vocabulary 2056: the last pair's
    second CTA has none), packed and row-major matrices, draft passes with
    fewer rows than their capacity; two greedy steps against the oracle."""
    V = 2056
    shape = S.WORKLOADS["tiny"].target.replace(n_layers=2, d_model=384, ffn=704, vocab=V, mask_id=V - 1)
    wl = S.WORKLOADS["tiny"].replace(target=shape, draft=shape.replace(n_layers=1, ffn=712), batch=batch, K=K,
                                     prompt_len=None, prompt_len_range=lens, n_new=12)
    P = Pair(wl, prefill_chunk=chunk)
    P.prefill()
    for step in range(1, 3):
        greedy_step(P, step)
    assert P.eng.last_status() == 0
    print("stats", P.stats)


@pytest.mark.parametrize("lens", [(1, 64, 63, 2, 130), (200, 1, 1, 1), (64, 64, 1)])
def test_prompts_of_several_sequences_in_one_pass(lens):
    """Prompt passes take 64 rows of the concatenated prompts at a time:
    prompts that begin, end and continue inside a pass, one-token prompts and
    prompts of exactly a pass; first tokens, then two greedy steps."""
    wl = S.WORKLOADS["tiny"].replace(batch=len(lens), prompt_len=None, prompt_lens_given=lens, n_new=12)
    P = Pair(wl, prefill_chunk=64)
    P.prefill()
    for step in range(1, 3):
        greedy_step(P, step)
    assert P.eng.last_status() == 0
    print("stats", P.stats)


def test_wide_projection_rounds_values_as_often_right_as_the_narrow_one():
    """The tensor cores truncate at every accumulation, and values are rounded
    to bf16 after the projection: the share of a first layer's values that
    differ from the correctly rounded 64-bit ones, from passes of up to 512
    rows (CTA pairs) and from passes of 64 rows, on the 8B and 1B widths.
    About 300 of 410k values differ; three standard deviations of a ratio of
    two such counts are 3 sqrt(2 / 300) = 0.25."""
    import torch
    from paper_2504_18583_gb300 import pard
    V, lens = 2056, (300, 100)
    shapes = [s.replace(n_layers=1, vocab=V, mask_id=V - 1) for s in (S.TARGET_8B, S.DRAFT_1B)]
    g = torch.Generator(device="cuda").manual_seed(5)
    weights, ref = [], []
    prompts = [torch.randint(0, V - 1, (n,), generator=g, device="cuda").tolist() for n in lens]
    for s in shapes:
        w = {n: torch.empty(s.tensor_shape(n), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)
             for n in S.GLOBAL_TENSORS + S.LAYER_TENSORS}
        for n in ("attn_norm", "mlp_norm", "final_norm"):
            w[n] += 1.0
        h = [w["embed"][torch.tensor(p, device="cuda")].double() for p in prompts]
        ref.append([((x / torch.sqrt((x * x).mean(-1, keepdim=True) + s.rms_eps) * w["attn_norm"].double())
                     @ w["wv"].double().T).to(torch.bfloat16) for x in h])
        weights.append({**{n: w[n] for n in S.GLOBAL_TENSORS}, "layers": [{n: w[n] for n in S.LAYER_TENSORS}]})
    wrong = {}
    for chunk in (512, 64):
        for i, p in enumerate(prompts):  # passes of 300 and of 100 rows
            eng = pard.PardEngine(shapes[0], weights[0], shapes[1], weights[1], max_batch=1, max_k=4, max_ctx=400,
                                  n_pages=32, prefill_chunk=chunk)
            eng.prefill([p], 8, 4)
            for mi in (0, 1):
                v = eng.read_kv(mi, 0, 0, list(range(len(p))), shapes[mi])[1].reshape(len(p), -1)
                wrong[chunk, mi] = wrong.get((chunk, mi), 0) + int((v != ref[mi][i]).sum())
            assert eng.last_status() == 0
            eng.unpack_weights()
            eng.close()
    print(wrong)
    for mi in (0, 1):
        assert wrong[512, mi] <= 1.25 * wrong[64, mi], wrong


def flat_head_engine(batch, K):
    """An engine whose draft gives every vocabulary entry the same logit: all
    LM-head rows are one row."""
    import torch
    from paper_2504_18583_gb300 import pard
    t, d = S.WORKLOADS["tiny"].target, S.WORKLOADS["tiny"].draft
    g = torch.Generator(device="cuda").manual_seed(3)

    def weights(s):
        w = {n: torch.empty(s.tensor_shape(n), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)
             for n in S.GLOBAL_TENSORS}
        w["final_norm"] += 1.0
        w["lm_head"][:] = w["lm_head"][0] * 8
        w["layers"] = []
        for _ in range(s.n_layers):
            L = {n: torch.empty(s.tensor_shape(n), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)
                 for n in S.LAYER_TENSORS}
            L["attn_norm"] += 1.0
            L["mlp_norm"] += 1.0
            w["layers"].append(L)
        return w

    eng = pard.PardEngine(t, weights(t), d, weights(d), max_batch=batch, max_k=K, max_ctx=80, n_pages=5 * batch)
    prompts = torch.randint(0, t.vocab - 1, (batch, 20), generator=torch.Generator().manual_seed(1)).tolist()
    eng.prefill(prompts, 16, K)
    return eng


@pytest.mark.parametrize("batch,K,T", [(2, 4, 1e-7), (16, 6, 1e-7), (16, 6, 1e-6)])
def test_sampled_draft_takes_the_lowest_index_of_equal_scores(batch, K, T):
    """A Gumbel-max score is rounded at the size of logit / T: at a very low
    temperature many entries share the best one, and the first of them is the
    draw (16 and 96 rows: both GEMM kernels)."""
    eng = flat_head_engine(batch, K)
    out = eng.alloc_step_outputs(want_logits=True)
    eng.draft(out, True, T, 77, 5)
    d, z = out["draft"].cpu().numpy(), out["draft_logits"].cpu().numpy()
    tied = 0
    for b in range(batch):
        for i in range(K):
            sc = gumbel_scores(z[b, i], T, 77, STREAM_DRAFT, 5, b, i)
            tied += int((sc == sc.max()).sum() > 1)
            assert int(d[b, i]) == int(np.argmax(sc)), (b, i, int(d[b, i]), int(np.argmax(sc)), sc.max())
    assert tied
    assert eng.last_status() == 0


def random_engine(shapes, batch, K, prompt_len, seed=7, stream=None, prefill_chunk=512):
    """An engine on seeded random weights (generated on the device), its prompts prefilled."""
    import torch
    from paper_2504_18583_gb300 import pard
    g = torch.Generator(device="cuda").manual_seed(seed)
    weights = []
    for s in shapes:
        def mat(n):
            t = torch.empty(s.tensor_shape(n), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)
            return t + 1.0 if n.endswith("norm") else t
        w = {n: mat(n) for n in S.GLOBAL_TENSORS}
        w["layers"] = [{n: mat(n) for n in S.LAYER_TENSORS} for _ in range(s.n_layers)]
        weights.append(w)
    torch.cuda.synchronize()
    pages = -(-(prompt_len + 16 + 2 * K) // 16)
    eng = pard.PardEngine(shapes[0], weights[0], shapes[1], weights[1], max_batch=batch, max_k=K, stream=stream,
                          max_ctx=prompt_len + 32 + 2 * K, n_pages=pages * batch, prefill_chunk=prefill_chunk)
    p = torch.randint(0, shapes[0].vocab - 1, (batch, prompt_len), generator=torch.Generator().manual_seed(seed))
    eng.prefill(p.tolist(), 16, K)
    return eng


def wide_pass(eng, out, cand):
    eng.draft(out, True, 0.9, 5, 1)
    eng.verify(out, cand, 1.0)
    return [out[k].clone() for k in ("draft", "draft_logits", "logits")]


WIDE_SHAPES = {
    # model widths, sequences, K: rows and the split of the down projection's tiles
    "odd_tiles": (dict(d_model=384, ffn=704, vocab=2056), 16, 7),
    "26_pairs_a_tile": (dict(d_model=384, ffn=6656, vocab=2056), 16, 7),  # more partials than the ring has places
    "two_token_tiles": (dict(d_model=512, ffn=2048, vocab=4096), 32, 9),
    "8b_widths": (None, 16, 7),
}


@pytest.mark.parametrize("case", WIDE_SHAPES)
def test_shared_tiles_do_not_depend_on_who_finishes_them(case):
    """Passes of more than 64 rows in which CTA pairs give their parts of a
    shared output tile up at once, after a microsecond, or not at all: the
    same bits in every output, launch after launch."""
    import torch
    widths, batch, K = WIDE_SHAPES[case]
    if widths:
        t = S.WORKLOADS["tiny"].target.replace(n_layers=2, mask_id=widths["vocab"] - 1, **widths)
        shapes = (t, t.replace(n_layers=1))
    else:
        shapes = [s.replace(n_layers=1, vocab=2056, mask_id=2055) for s in (S.TARGET_8B, S.DRAFT_1B)]
    eng = random_engine(shapes, batch, K, 20)
    out = eng.alloc_step_outputs(want_logits=True)
    cand = torch.randint(0, shapes[0].vocab - 1, (batch, K), device="cuda", dtype=torch.int32)
    want = wide_pass(eng, out, cand)
    assert all(torch.isfinite(x.float()).all() for x in want)
    for ns in (0, 0, 0, 700, 0, 1000, -1, 0, -1):
        eng.set_share_wait(ns)
        for got, w in zip(wide_pass(eng, out, cand), want):
            assert torch.equal(got, w), ns
    assert eng.last_status() == 0


def test_two_engines_on_two_streams():
    """Two engines whose passes of more than 64 rows run at the same time on
    streams of their own: each gives the bits that it gives alone."""
    import torch
    shapes = [s.replace(n_layers=2, vocab=4104, mask_id=4103) for s in (S.TARGET_8B, S.DRAFT_1B)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    cand = torch.randint(0, 4103, (16, 6), device="cuda", dtype=torch.int32)
    torch.cuda.synchronize()
    engines = [random_engine(shapes, 16, 6, 40, seed=k, stream=s) for k, s in enumerate(streams)]
    outs, alone = [], []
    for e, s in zip(engines, streams):
        with torch.cuda.stream(s):
            outs.append(e.alloc_step_outputs(want_logits=True))
            alone.append(wide_pass(e, outs[-1], cand))
        torch.cuda.synchronize()
    for _ in range(6):
        got = []
        for e, s, o in zip(engines, streams, outs):
            with torch.cuda.stream(s):
                got.append(wide_pass(e, o, cand))
        torch.cuda.synchronize()
        for a, b in zip(alone, got):
            assert all(torch.equal(x, y) for x, y in zip(a, b))
    assert [e.last_status() for e in engines] == [0, 0]


@pytest.mark.parametrize("T", [0.05, 0.7, 1.0, 1.3])
@pytest.mark.parametrize("batch,K", [(2, 4), (8, 4), (16, 6)], ids=["16_rows", "64_rows", "192_rows"])
def test_lm_head_draw_follows_its_own_logits(batch, K, T):
    """The draw that the draft pass makes in the LM head (a rough ranking,
    then exact scores of the few best): the token of the highest Gumbel score
    of the logits the pass returns, except where the lead is within the
    roundings of the two sides' noise and of the sum."""
    t = S.WORKLOADS["tiny"].target.replace(n_layers=1, vocab=4104, mask_id=4103)
    eng = random_engine((t, t), batch, K, 20, seed=int(100 * T))
    out = eng.alloc_step_outputs(want_logits=True)
    near = 0
    for step in (1, 2):
        eng.draft(out, True, T, 91, step)
        d, z = out["draft"].cpu().numpy(), out["draft_logits"].cpu().numpy()
        for b in range(batch):
            for i in range(K):
                sc = gumbel_scores(z[b, i], T, 91, STREAM_DRAFT, step, b, i)
                if int(d[b, i]) != int(np.argmax(sc)):
                    assert sc[d[b, i]] >= sc.max() - GUMBEL_EPS - 2 * np.spacing(np.abs(sc).max()), (step, b, i)
                    near += 1
    assert near <= 2
    assert eng.last_status() == 0
