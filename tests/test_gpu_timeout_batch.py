"""Failure detection in the kernels of a step (GPU): the bounded waits of the
warp-level projections (one sequence, or several by option), of the cluster
split-K projections, of the pair kernel, split and unsplit (the output head),
and of the walking cross-attention run out during one step, as in
test_gpu_timeout.py, and the handle recovers.  Every copy and matrix
instruction still completes; the waits only give up before it does, and the
kernels then wait (bounded) for what they have in flight."""
import numpy as np
import pytest

from paper_2609_32869_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _steps(s, forced, sp):
    out = []
    for f in forced:
        toks, cnt = s.step(forced=f, sp=sp)
        st = s.state()
        out += [toks.cpu().numpy().copy(), cnt.cpu().numpy().copy(), st["len"].copy(), st["anchor"].copy()]
    return out


def _timeout_and_recover(cfg, n, T, limits, skinny=False):
    import torch
    from paper_2609_32869_gb300 import binding as B
    from paper_2609_32869_gb300.session import Session, upload_weights
    dev = upload_weights(syn.make_weights(cfg, seed=0, ln_noise=True))
    enc = syn.encoder_output(cfg, 1, seed=1)[np.zeros(n, int)]
    prompt = syn.prompts(cfg, n, length=4, seed=1)
    slots = np.arange(n, dtype=np.int32)
    forced = [syn.random_tokens(cfg, (n, cfg.block_k), seed=70 + i) for i in range(2)]
    sp = B.sample_params(T, 5) if T else None

    def session():
        s = Session(cfg, dev, max_batch=n)
        if skinny:
            B.wf_set_option(s.h, B.WF_OPT_SKINNY, 1)
        s.prefill(slots, enc, prompt, np.full(n, 60, np.int32), sp=sp)
        return s

    s = session()
    want = _steps(s, forced, sp)
    assert s.error() == 0
    s.close()
    s = session()
    for limit in limits:
        B.wf_set_option(s.h, B.WF_OPT_SPIN_LIMIT, limit)
        s.step(forced=forced[0], sp=sp)  # returns: every wait is bounded
        torch.cuda.synchronize()
        assert s.error(clear=True) & B.WF_DEV_ERR_TIMEOUT
        B.wf_set_option(s.h, B.WF_OPT_SPIN_LIMIT, 0)
        s.reset_slots(slots)
        assert s.compact() == n
        for a, b in zip(want, _steps(s, forced, sp)):
            assert np.array_equal(a, b)
        assert s.error() == 0
        s.reset_slots(slots)
        assert s.compact() == n
    s.close()


@pytest.mark.parametrize("n", [1, 5])
def test_warp_level_projections_give_up_and_the_handle_recovers(n):
    _timeout_and_recover(syn.TINY, n, 0.0, (32,), skinny=True)


# 18 rows: cluster split-K; 108 rows: pairs of SMs (tiny widths, one chunk of
# several k-steps or three)
@pytest.mark.parametrize("n,T", [(2, 0.0), (12, 0.0), (12, 0.8)])
def test_projections_give_up_and_the_handle_recovers(n, T):
    _timeout_and_recover(syn.TINY, n, T, (32, 400))


def test_the_walk_gives_up_and_its_counters_return_to_zero():
    """52 sequences of 6 heads are two (sequence, head) groups per SM: walking
    CTAs, most of whose shares cut a group that another CTA finishes.  A count
    left behind by a CTA that gave up would merge that group too early, or
    never, in the steps that follow."""
    _timeout_and_recover(syn.TINY, 52, 0.0, (32, 400, 3000))
