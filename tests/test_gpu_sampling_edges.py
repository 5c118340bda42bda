"""Sampling at the ends of what the entry points take: temperatures so low that
the scores z / T + G are rounded far above the noise."""
import numpy as np
import pytest

from paper_2609_32869_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1e-3, 1e-5, 1e-6, 1e-9, 1e-40])
def test_low_temperature_draws_follow_the_rounded_scores(T):
    """A draw is the argmax of fl(fl(z / T) + G), the lowest id on ties.  One
    vocabulary tile of equal rows is left unsuppressed, so its ids have the
    same logit and the draw hangs on G as far as the sum's rounding keeps it:
    down to ties of all ids.  Draws that turn on less than 2e-6 of G (its
    logarithms' rounding on either side) are left out."""
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
            with np.errstate(over="ignore"):
                x = z[i, j, 128:256] / np.float32(T)
            g = philox.gumbel_noise(seed, i, 1, j, philox.TAG_DRAFT, V)[128:256]
            lo, hi = x + (g - np.float32(2e-6)), x + (g + np.float32(2e-6))
            # the ids that can be largest; the draw is known if their sums are
            if (hi >= lo.max()).any() and (lo == hi)[hi >= lo.max()].all():
                assert cand[i, j - 1] == 128 + int(np.argmax(x + g)), (i, j)
                compared += 1
    assert compared > n * K // 2 and s.error() == 0
    s.close()
