"""The allocation-free acceptance entry point gives the same results as the
context-based path (pard_set_logits + pard_accept_commit) on the same
inputs, for two calls in a row (greedy and sampling), through the C ABI.

This file is collected last on purpose: pard_accept_noalloc is an interface
for callers that cannot provide device memory (no device allocator, or an
engine that forbids allocation on its serving path), and its scratch lives in
a fixed device array shared by all calls."""
import numpy as np
import pytest

import synthetic as S
from oracle import pard as OP

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,K,vocab", [(1, 4, 2048), (3, 4, 2048), (16, 8, 128256)],
                         ids=["b1k4", "b3k4", "b16k8_full_vocab"])
def test_noalloc_acceptance_matches_context_path_twice(batch, K, vocab):
    """Four calls in a row (two sampled, two greedy) at batch 1, at batch 3,
    and at the scratch's limits (batch 16, K = 8, the 128256-entry
    vocabulary: every row pitch and tile count of its fixed layout)."""
    import torch
    from _parity import Pair
    from paper_2504_18583_gb300 import _build, pard
    _build.build()
    wl = S.WORKLOADS["tiny"].replace(sample=True, n_new=100000, K=K, batch=batch, prompt_len=20)
    if vocab != wl.target.vocab:
        wl = wl.replace(target=wl.target.replace(vocab=vocab, mask_id=vocab - 1),
                        draft=wl.draft.replace(vocab=vocab, mask_id=vocab - 1))
    P = Pair(wl)
    P.prefill(seed=3)
    B, V = wl.batch, vocab
    rng = np.random.default_rng(11 + batch)
    lib = pard.lib()
    stream = P.eng.stream.cuda_stream
    for call, sample in enumerate((True, True, False, False)):
        y = (rng.standard_normal((B, K + 1, V)) * 2.0).astype(np.float32)
        z = (y[:, :K] + rng.standard_normal((B, K, V)).astype(np.float32) * 0.5).astype(np.float32)
        d = np.array([OP.draft_tokens(z[b], True, 1.0, 900 + call, 2, b) for b in range(B)], dtype=np.int32)
        if call == 1:
            d[:, 1:] = np.argmax(y[:, 1:K], axis=-1)  # some acceptance deep into the draft
        yt, zt, dt = (torch.as_tensor(a, device="cuda") for a in (y, z, d))
        step = 50 + call
        # existing path
        P.eng.set_logits(yt, zt, dt, 1.0)
        out = P.eng.alloc_step_outputs()
        P.eng.accept_commit(out, sample, 1.0, 7, step)
        # allocation-free path, same inputs
        acc2 = torch.full((B,), -9, dtype=torch.int32, device="cuda")
        em2 = torch.full((B, K + 1), -9, dtype=torch.int32, device="cuda")
        code = lib.pard_accept_noalloc(yt.data_ptr(), zt.data_ptr(), dt.data_ptr(), B, K, V, int(sample), 1.0, 7,
                                       step, acc2.data_ptr(), em2.data_ptr(), stream)
        assert code == 0, pard.pard_last_error()
        torch.cuda.synchronize()
        assert torch.equal(acc2, out["accept_len"]), (call, acc2, out["accept_len"])
        assert torch.equal(em2, out["emitted"]), (call, em2, out["emitted"])
    # sizes beyond the static scratch are refused with a message
    code = lib.pard_accept_noalloc(yt.data_ptr(), zt.data_ptr(), dt.data_ptr(), 17, K, V, 0, 1.0, 0, 0,
                                   acc2.data_ptr(), em2.data_ptr(), stream)
    assert code == -1 and "static scratch" in pard.pard_last_error()
    assert P.eng.last_status() == 0


@pytest.mark.parametrize("vocab", [8, 2040, 2056, 4104])
def test_noalloc_tile_edges_masked_rows_and_unaligned_logits(vocab):
    """The statistics' 2048-entry tiles at vocabularies just below and above
    their multiples, with whole stretches of the logits masked to -inf, from
    arrays that start 4 bytes off a 16-byte boundary: the same as the oracle's
    acceptance rule."""
    import torch
    from paper_2504_18583_gb300 import _build, pard
    _build.build()
    B, K = 2, 5
    rng = np.random.default_rng(vocab)
    for sample in (True, False):
        y = (rng.standard_normal((B, K + 1, vocab)) * 2.0).astype(np.float32)
        y[:, :, : vocab // 2] = -np.inf
        z = y[:, :K] + np.where(np.isinf(y[:, :K]), 0, 0.4 * rng.standard_normal((B, K, vocab))).astype(np.float32)
        d = np.argmax(z, axis=-1).astype(np.int32)
        hold = [torch.empty(a.size + 1, dtype=torch.float32, device="cuda") for a in (y, z)]
        for h, a in zip(hold, (y, z)):
            h[1:].copy_(torch.from_numpy(a.reshape(-1)))
        dt = torch.as_tensor(d, device="cuda")
        acc = torch.empty(B, dtype=torch.int32, device="cuda")
        em = torch.empty((B, K + 1), dtype=torch.int32, device="cuda")
        code = pard.lib().pard_accept_noalloc(hold[0][1:].data_ptr(), hold[1][1:].data_ptr(), dt.data_ptr(), B, K, vocab,
                                              int(sample), 1.0, 21, 4, acc.data_ptr(), em.data_ptr(),
                                              torch.cuda.current_stream().cuda_stream)
        assert code == 0, pard.pard_last_error()
        for b in range(B):
            with np.errstate(divide="ignore", invalid="ignore"):
                a_o, em_o = (OP.accept_sampling(d[b], z[b], y[b], 1.0, 21, 4, b) if sample
                             else OP.accept_greedy(d[b], y[b]))
            assert int(acc[b]) == a_o, (sample, b)
            assert em[b].tolist()[:a_o + 1] == [int(t) for t in em_o], (sample, b)


@pytest.mark.parametrize("T", [1e-3, 0.05, 0.7, 1.3])
def test_noalloc_sampling_at_other_temperatures(T):
    """Temperatures other than 1, down to scores of several thousand (where
    the draw's sum is rounded to 1e-3 and several entries can share the best
    score): accept lengths and tokens of the oracle's rule, the bonus token
    except where its lead is within the two sides' roundings."""
    import torch
    from _parity import GUMBEL_EPS, gumbel_scores
    from oracle.philox import STREAM_BONUS
    from paper_2504_18583_gb300 import _build, pard
    _build.build()
    B, K, vocab = 16, 3, 4104
    rng = np.random.default_rng(int(T * 1000))
    y = (rng.standard_normal((B, K + 1, vocab)) * 2.0).astype(np.float32)
    y[: B // 2] = np.round(y[: B // 2])  # many equal logits
    z = y[:, :K] + (T * rng.standard_normal((B, K, vocab))).astype(np.float32)
    z[: B // 4] = y[: B // 4, :K]  # p = q: every candidate is accepted, the bonus comes from the last row
    d = np.array([OP.draft_tokens(z[b], True, T, 8, 4, b) for b in range(B)], dtype=np.int32)
    yt, zt, dt = (torch.as_tensor(a, device="cuda") for a in (y, z, d))
    acc = torch.empty(B, dtype=torch.int32, device="cuda")
    em = torch.empty((B, K + 1), dtype=torch.int32, device="cuda")
    code = pard.lib().pard_accept_noalloc(yt.data_ptr(), zt.data_ptr(), dt.data_ptr(), B, K, vocab, 1, T, 21, 4,
                                          acc.data_ptr(), em.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert code == 0, pard.pard_last_error()
    exact = 0
    for b in range(B):
        with np.errstate(divide="ignore", invalid="ignore"):
            a_o, em_o = OP.accept_sampling(d[b], z[b], y[b], T, 21, 4, b)
        assert int(acc[b]) == a_o, b
        got = em[b].tolist()[:a_o + 1]
        assert got[:a_o] == [int(x) for x in em_o[:a_o]], b
        if got[a_o] == int(em_o[a_o]):
            exact += 1
        elif a_o == K:
            sc = gumbel_scores(y[b, K], T, 21, STREAM_BONUS, 4, b, 0)
            assert sc[got[a_o]] >= sc.max() - GUMBEL_EPS - 2 * np.spacing(np.abs(sc).max()), b
    assert exact >= B - 1
    assert (acc.cpu().numpy()[: B // 4] == K).all()
