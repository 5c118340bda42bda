"""Projections of many token rows (pairs of SMs on 256-row weight tiles): their
rows equal, bit for bit, those of the small launches that the cluster split-K
kernel runs, at tile edges and ragged sizes, and through every epilogue of a
decode step."""
import numpy as np
import pytest

from paper_2609_32869_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


# (N, K): splits of 10, 5, 4, 16 (5 k-steps each), 3, one k-step per chunk at
# the least, ragged N (one odd CTA without weight rows, odd output stride)
SHAPES = [(1280, 1280), (3840, 1280), (5120, 1280), (1280, 5120), (1152, 384), (1000, 128), (130, 192), (1281, 64)]


@pytest.mark.parametrize("N,K", SHAPES)
def test_wide_rows_equal_small_launches(N, K):
    import torch
    from paper_2609_32869_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(N + K)
    M = 1031
    x = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    w = (0.02 * torch.randn(N, K, generator=g, device="cuda")).bfloat16()
    b = (0.02 * torch.randn(N, generator=g, device="cuda")).bfloat16()

    def run(lo, hi, offset=0):
        buf = torch.full(((hi - lo) * N + offset,), float("nan"), device="cuda")
        y = buf[offset:].view(hi - lo, N)
        B.wf_gemm_bf16(x[lo:hi], w, b, y, hi - lo, N, K, None, 0)
        return y

    want = torch.cat([run(lo, min(M, lo + 40)) for lo in range(0, M, 40)])  # cluster split-K
    for m in (41, 65, 96, 97, 129, 257, 288, 833, M):
        assert torch.equal(run(0, m), want[:m]), m
    assert torch.equal(run(0, 300, offset=1), want[:300])  # an output that is only 4-byte aligned
    bound = K * 2.0 ** -23 * (x.double().abs() @ w.double().abs().T) + 1e-6
    assert ((want.double() - (x.double() @ w.double().T + b.double())).abs() <= bound).all()


@pytest.mark.parametrize("n", [11, 30, 57])
def test_step_rows_do_not_depend_on_batch(n):
    """n * 9 > 96 rows against a two-sequence handle of the same requests:
    logits, taps and tokens of a step are the same bits (query, key/value,
    residual, GELU and history epilogues, and the acoustic projection)."""
    import torch
    from paper_2609_32869_gb300 import binding as B
    from paper_2609_32869_gb300.session import Session, upload_weights
    cfg = syn.TINY
    dev = upload_weights(syn.make_weights(cfg, seed=3, ln_noise=True))
    enc = syn.encoder_output(cfg, 3, seed=1)
    prompt = syn.prompts(cfg, 3, length=7, seed=1)
    pick = np.arange(n) % 3
    rows, V = cfg.block_k + 1, cfg.vocab

    def step(which):
        k = len(which)
        s = Session(cfg, dev, max_batch=k, keep_logits=True)
        s.prefill(np.arange(k, dtype=np.int32), enc[which], prompt[which], np.full(k, 60, np.int32))
        for _ in range(2):
            toks, cnt = s.step()
        out = [s.view(B.WF_VIEW_TARGET_LOGITS, torch.float32, (k, rows, V)).clone(),
               s.view(B.WF_VIEW_DRAFT_LOGITS, torch.float32, (k, rows, V)).clone(),
               s.view(B.WF_VIEW_TAPS, torch.bfloat16, (k, rows, cfg.n_taps * cfg.d_model)).clone(),
               toks.clone(), cnt.clone()]
        assert s.error() == 0
        s.close()
        return out

    big = step(pick)
    for pair in ((0, 1), (1, 2)):
        small = step(np.array(pair))
        for a, b in zip(big, small):
            for i in (pair[0], pair[0] + 3 * ((n - 3) // 3)):
                assert torch.equal(a[i], b[0])
                assert torch.equal(a[i + pair[1] - pair[0]], b[1])


@pytest.mark.parametrize("T,mask", [(0.25, False), (0.7, True), (1.0, False), (30.0, True)])
def test_sampling_head_draws_the_exact_argmax(T, mask):
    """The head's Gumbel-max draw (ids screened by an estimate, the survivors
    scored exactly) is the argmax of x + G over every id that is not
    suppressed, on the GPU's own logits with the oracle's noise, wherever the
    two best scores differ by more than the logarithms' rounding (1e-4 at
    scores below 20).  Odd vocabulary, whole vocabulary tiles suppressed."""
    import torch
    from oracle import philox
    from paper_2609_32869_gb300 import binding as B
    from paper_2609_32869_gb300.session import Session, upload_weights
    cfg, n, seed = syn.TINY, 13, 77
    K, V = cfg.block_k, cfg.vocab
    dev = upload_weights(syn.make_weights(cfg, seed=4))
    enc = syn.encoder_output(cfg, 1, seed=2)[np.zeros(n, int)]
    prompt = syn.prompts(cfg, n, length=5, seed=3)
    sup = np.zeros(V, np.uint8)
    if mask:
        sup[syn.uniform_int(5, "sup", (V // 3,), 0, V - 1)] = 1
        sup[128:384] = 1
    d_sup = torch.from_numpy(sup).cuda()
    sp = B.sample_params(T, seed, d_sup if mask else None)
    s = Session(cfg, dev, max_batch=n, keep_logits=True)
    s.prefill(np.arange(n, dtype=np.int32), enc, prompt, np.full(n, 60, np.int32))
    s.draft(sp=sp)
    z = s.view(B.WF_VIEW_DRAFT_LOGITS, torch.float32, (n, K + 1, V)).cpu().numpy()
    cand = s.view(B.WF_VIEW_CANDIDATES, torch.int32, (n, K)).cpu().numpy()
    clear = 0
    for i in range(n):
        for j in range(1, K + 1):
            x = z[i, j] / np.float32(T) + philox.gumbel_noise(seed, i, 1, j, philox.TAG_DRAFT, V)
            x[sup != 0] = -np.inf
            top = np.argsort(x)[-2:]
            if x[top[1]] - x[top[0]] > 1e-4:
                assert cand[i, j - 1] == top[1], (i, j)
                clear += 1
    assert clear > n * K // 2 and s.error() == 0
    s.close()
