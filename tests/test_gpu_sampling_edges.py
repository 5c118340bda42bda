"""Sampling at the ends of what the entry points take: proposals that are no
vocabulary ids, and temperatures so low that the scores z / T + G are rounded
far above the noise."""
import numpy as np
import pytest

from paper_2609_32869_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("with_q", [False, True])
def test_a_proposal_outside_the_vocabulary_is_rejected(with_q):
    """A forced proposal that is no id is recorded in the error word and
    rejected, wherever it stands (also behind a rejection): tokens, counts and
    state equal those of a run that proposes a suppressed id in its place,
    which has probability 0."""
    import torch
    from paper_2609_32869_gb300 import binding as B
    from paper_2609_32869_gb300.session import Session, upload_weights
    cfg, n, steps = syn.TINY, 9, 3
    K, V = cfg.block_k, cfg.vocab
    dev = upload_weights(syn.make_weights(cfg, seed=2))
    never = 777
    sup = np.zeros(V, np.uint8)
    sup[never] = 1
    d_sup = torch.from_numpy(sup).cuda()
    fq = torch.randn(n, K, V, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    bad = np.array([-1, V, 2**31 - 1, -2**31], np.int64).astype(np.int32)
    forced = [syn.random_tokens(cfg, (n, K), seed=40 + i) for i in range(steps)]
    holes = np.zeros((n, K), bool)
    for i in range(n):
        holes[i, i % K:] = True     # from its i-th proposal on ...
        holes[i, (i + 2) % K] = False  # ... but one

    def run(fill):
        s = Session(cfg, dev, max_batch=n)
        s.prefill(np.arange(n, dtype=np.int32), syn.encoder_output(cfg, 1, seed=2)[np.zeros(n, int)],
                  syn.prompts(cfg, n, length=5, seed=3), np.full(n, 60, np.int32))
        out, err = [], 0
        for i, f in enumerate(forced):
            f = f.copy()
            f[holes] = fill[:holes.sum()]
            toks, cnt = s.step(forced=f, sp=B.sample_params(0.9, 50 + i, d_sup), forced_q=fq if with_q else None)
            out += [toks.cpu().numpy().copy(), cnt.cpu().numpy().copy()]
            out += [s.state()[k].copy() for k in ("len", "anchor", "remaining", "done")]
            err |= s.error(clear=True)
        s.close()
        return out, err

    want, err = run(np.full(n * K, never, np.int32))
    assert err == 0
    got, err = run(np.resize(bad, n * K))
    assert err == B.WF_DEV_ERR_TOKEN
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
    assert max(c.max() for c in want[1::6]) > 1  # some proposals were accepted


@pytest.mark.parametrize("T", [1e-3, 1e-5, 1e-6, 1e-9, 1e-40])
def test_low_temperature_draws_follow_the_rounded_scores(T):
    """A draw is the argmax of fl(fl(z / T) + G), -inf for a suppressed id, the
    lowest id on ties.  One vocabulary tile of equal rows is left unsuppressed,
    so its ids have the same logit and the draw hangs on G as far as the sum's
    rounding keeps it: down to ties of all ids.  Draws that turn on less than
    2e-6 of G (its logarithms' rounding on either side) are left out."""
    import torch
    from oracle import philox
    from paper_2609_32869_gb300 import binding as B
    from paper_2609_32869_gb300.session import Session, upload_weights
    cfg, n, seed = syn.TINY, 7, 91
    K, V = cfg.block_k, cfg.vocab
    ws = syn.make_weights(cfg, seed=4)
    ws.target["tok_emb"][128:256] = ws.target["tok_emb"][128]
    sup = np.ones(V, np.uint8)
    sup[128:256] = 0
    d_sup = torch.from_numpy(sup).cuda()
    sp = B.sample_params(T, seed, d_sup)
    s = Session(cfg, upload_weights(ws), max_batch=n, keep_logits=True)
    s.prefill(np.arange(n, dtype=np.int32), syn.encoder_output(cfg, 1, seed=2)[np.zeros(n, int)],
              syn.prompts(cfg, n, length=5, seed=3), np.full(n, 60, np.int32))
    s.draft(sp=sp)
    z = s.view(B.WF_VIEW_DRAFT_LOGITS, torch.float32, (n, K + 1, V)).cpu().numpy()
    cand = s.view(B.WF_VIEW_CANDIDATES, torch.int32, (n, K)).cpu().numpy()
    compared = 0
    for i in range(n):
        for j in range(1, K + 1):
            x = np.full(V, -np.inf, np.float32)
            with np.errstate(over="ignore"):
                x[128:256] = z[i, j, 128:256] / np.float32(T)
            g = philox.gumbel_noise(seed, i, 1, j, philox.TAG_DRAFT, V)
            lo, hi = x + (g - np.float32(2e-6)), x + (g + np.float32(2e-6))
            near = hi >= lo.max()  # the ids that can be largest: one, or sums that are known
            if near.sum() == 1 or (lo == hi)[near].all():
                assert cand[i, j - 1] == int(np.argmax(x + g)), (i, j)
                compared += 1
    assert compared > n * K // 2 and s.error() == 0
    s.close()
