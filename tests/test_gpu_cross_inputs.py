"""Cross-attention of many sequences on the inputs that its entry point takes
besides plain queries and keys: rotated by position (`rope`), and with frames
whose scores are -inf.  A large launch equals launches of its sequences alone,
bit for bit, and the oracle."""
import numpy as np
import pytest

from oracle import decoder as od

pytestmark = pytest.mark.gpu


def _calls(n_seq, rps, H, ctx, rope, edit=None):
    """(rows per sequence of one launch, of one launch each, of the oracle)."""
    import torch
    from paper_2609_32869_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(ctx + rps)
    d = H * 64
    slots = np.random.RandomState(n_seq).permutation(n_seq).astype(np.int32)
    q = torch.randn(n_seq * rps, d, generator=g, device="cuda").bfloat16()
    k = torch.randn(n_seq, H, ctx, 64, generator=g, device="cuda").bfloat16()
    v = torch.randn(n_seq, H, ctx, 64, generator=g, device="cuda").bfloat16()
    if edit:
        edit(q.view(n_seq * rps, H, 64), k)

    def run(rows, sl, noalloc=False):
        n = len(sl)
        out = torch.full((n * rps, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        ds = torch.from_numpy(np.ascontiguousarray(sl)).cuda()
        if noalloc:
            B.wf_attention_noalloc(rows, k, v, ds, None, n, rps, H, ctx, 2, rope, 10000.0, out)
            return out
        nb = B.wf_attention_scratch_bytes(n, rps, H, ctx)
        sc = torch.full((nb,), 255, dtype=torch.uint8, device="cuda")
        B.wf_attention(rows, k, v, ds, None, n, rps, H, ctx, 2, rope, 10000.0, out, sc, nb)
        return out

    big = run(q, slots)
    if B.wf_attention_scratch_bytes(n_seq, rps, H, ctx) <= 8 << 20:
        assert torch.equal(big, run(q, slots, noalloc=True))
    alone = torch.cat([run(q[i * rps:(i + 1) * rps], slots[i:i + 1]) for i in range(n_seq)])
    f = lambda t: t.float().cpu().numpy().astype(np.float64)  # noqa: E731
    want = []
    for i in (0, n_seq - 1):
        s = int(slots[i])
        qi = f(q[i * rps:(i + 1) * rps])
        ki, vi = (f(t[s]).transpose(1, 0, 2).reshape(ctx, d) for t in (k, v))
        if rope:
            qi, ki = od.rope(qi, np.arange(rps), H, 10000.0), od.rope(ki, np.arange(ctx), H, 10000.0)
        want.append(od.multi_head_attention(qi, ki, vi, H))
    ends = np.concatenate([f(big[:rps]), f(big[-rps:])])
    return big, alone, ends, np.concatenate(want)


# (sequences, rows, heads, frames): two (sequence, head, query group)s per SM
# and one fewer, one and two query groups, blocks of 256 frames cut short
@pytest.mark.parametrize("n_seq,rps,H,ctx", [(17, 9, 20, 300), (15, 9, 20, 300), (16, 1, 20, 1500), (9, 17, 20, 513),
                                             (53, 9, 6, 257)])
def test_positions_rotate_whatever_the_number_of_sequences(n_seq, rps, H, ctx):
    import torch
    big, alone, ends, want = _calls(n_seq, rps, H, ctx, 1)
    assert torch.equal(big, alone)
    # bf16 output rounding (2^-8 relative) dominates the fp32 arithmetic
    np.testing.assert_allclose(ends, want, atol=2e-2, rtol=1e-2)


# frames whose keys are -inf against positive queries: slices of 32 keys, a
# whole block of 256, the cut last block, and all but one frame
@pytest.mark.parametrize("n_seq,rps,H,ctx,masked", [
    (17, 9, 20, 600, ((64, 128),)), (17, 9, 20, 600, ((0, 33), (256, 512))), (17, 9, 20, 600, ((512, 600),)),
    (9, 17, 20, 513, ((0, 256), (288, 513))), (53, 9, 6, 300, ((0, 299),)), (15, 9, 20, 600, ((64, 128), (256, 512)))])
def test_masked_frames_have_weight_zero(n_seq, rps, H, ctx, masked):
    import torch

    def edit(q, k):
        q[..., 0] = 1.0
        for a, b in masked:
            k[:, :, a:b, 0] = float("-inf")

    big, alone, ends, want = _calls(n_seq, rps, H, ctx, 0, edit)
    assert torch.isfinite(big.float()).all()
    assert torch.equal(big, alone)
    np.testing.assert_allclose(ends, want, atol=2e-2, rtol=1e-2)


# (sequences, rows, heads, frames): one CTA per group from 81% of a wave of
# three CTAs on each of 152 SMs (370 of 456 groups) to a whole one, walking CTAs
# on either side; two query groups over more and over less than 88 MiB of keys
# and values
@pytest.mark.parametrize("n_seq,rps,H,ctx", [(369, 3, 1, 300), (370, 3, 1, 300), (456, 3, 1, 300), (457, 3, 1, 300),
                                             (13, 17, 20, 1500), (11, 17, 24, 1300), (16, 17, 15, 1500)])
def test_forms_agree_where_they_change(n_seq, rps, H, ctx):
    import torch
    big, alone, ends, want = _calls(n_seq, rps, H, ctx, 0)
    assert torch.equal(big, alone)
    np.testing.assert_allclose(ends, want, atol=2e-2, rtol=1e-2)


# more queries than frames: their positions run past the frames'
@pytest.mark.parametrize("n_seq,rps,H,ctx", [(3, 209, 12, 42), (2, 300, 4, 257), (1, 17, 1, 1), (40, 65, 6, 64)])
def test_queries_past_the_frames_rotate_by_their_positions(n_seq, rps, H, ctx):
    import torch
    big, alone, ends, want = _calls(n_seq, rps, H, ctx, 1)
    assert torch.equal(big, alone)
    np.testing.assert_allclose(ends, want, atol=2e-2, rtol=1e-2)
