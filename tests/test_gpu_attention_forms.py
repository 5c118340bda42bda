"""The forms of an attention launch (cluster, split blocks, one CTA per group,
walking CTAs) give the same bits and read nothing past the visible keys: a
large launch equals launches of its sequences alone, with NaN in every cache
row that no query sees."""
import numpy as np
import pytest

from oracle import decoder as od
from paper_2609_32869_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

# (mode, ctx, rps, n_seq, heads, cache lengths): cross-attention shares that cut
# groups, a block of 44 and of one frame, two query groups, one row; text caches
# at the edges of the 64-row copies, of a block and of the cache
CASES = [
    (2, 1500, 9, 17, 20, None), (2, 300, 1, 40, 12, None), (2, 257, 17, 20, 20, None), (2, 512, 16, 31, 20, None),
    (2, 200, 9, 3, 20, None), (2, 40, 3, 2, 4, None), (2, 1500, 9, 9, 20, None),
    (0, 448, 9, 16, 20, (0, 54, 55, 56, 63, 118, 119, 246, 247, 248, 255, 256, 310, 311, 430, 439)),
    (1, 448, 9, 16, 20, (0, 54, 55, 56, 63, 118, 119, 246, 247, 248, 255, 256, 310, 311, 430, 439)),
    (0, 448, 223, 4, 20, (0, 0, 33, 225)), (0, 448, 1, 5, 20, (0, 63, 64, 255, 447)),
]


@pytest.mark.parametrize("mode,ctx,rps,n_seq,H,lengths", CASES)
def test_forms_agree_and_read_only_visible_keys(mode, ctx, rps, n_seq, H, lengths):
    import torch
    from paper_2609_32869_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(ctx + rps)
    d = H * 64
    slots = np.random.RandomState(n_seq).permutation(n_seq).astype(np.int32)
    base = np.zeros(n_seq, np.int32)
    if lengths:
        base[slots] = lengths
    q = torch.randn(n_seq * rps, d, generator=g, device="cuda").bfloat16()
    k = torch.randn(n_seq, H, ctx, 64, generator=g, device="cuda").bfloat16()
    v = torch.randn(n_seq, H, ctx, 64, generator=g, device="cuda").bfloat16()
    if mode != 2:
        for s in range(n_seq):
            k[s, :, base[s] + rps:] = float("nan")
            v[s, :, base[s] + rps:] = float("nan")
    db = torch.from_numpy(base).cuda()

    def run(rows, sl):
        n = len(sl)
        out = torch.full((n * rps, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        nb = B.wf_attention_scratch_bytes(n, rps, H, ctx)
        sc = torch.full((nb,), 255, dtype=torch.uint8, device="cuda")  # scratch comes uninitialised
        B.wf_attention(rows, k, v, torch.from_numpy(np.ascontiguousarray(sl)).cuda(), db, n, rps, H, ctx, mode,
                       mode == 1, 10000.0, out, sc, nb)
        return out

    big = run(q, slots)
    for i in range(n_seq):
        assert torch.equal(big[i * rps:(i + 1) * rps], run(q[i * rps:(i + 1) * rps], slots[i:i + 1])), i
    for i in (0, n_seq - 1):
        s = int(slots[i])
        n_keys = ctx if mode == 2 else int(base[s]) + rps
        f = lambda t: t.float().cpu().numpy().astype(np.float64)  # noqa: E731
        qi, at = f(q[i * rps:(i + 1) * rps]), base[s] + np.arange(rps)
        ki, vi = (f(t[s, :, :n_keys]).transpose(1, 0, 2).reshape(n_keys, d) for t in (k, v))
        if mode == 1:
            qi, ki = od.rope(qi, at, H, 10000.0), od.rope(ki, np.arange(n_keys), H, 10000.0)
        vis = np.arange(n_keys)[None, :] <= at[:, None] if mode == 0 else None
        want = od.multi_head_attention(qi, ki, vi, H, vis)
        np.testing.assert_allclose(f(big[i * rps:(i + 1) * rps]), want, atol=2e-2, rtol=1e-2)
