"""Many short work items per thread block: each is found and decoded one ahead, its results are stored while the next
one runs, and its buffers come back in between.  A head's results must not depend on what the block did before, and
sampled heads are what the float64 oracle gives."""
import math

import pytest

import oracle
from parity_util import BF16_REL_FRO, rel_fro, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,H_kv,N,D,causal,padded", [
    (40, 16, 16, 100, 128, False, False),    # one key tile, one query tile: every item is one step
    (24, 16, 16, 130, 128, True, False),     # one and two steps
    (24, 16, 4, 130, 64, True, False),       # grouped heads
    (24, 16, 16, 300, 64, False, False),     # three key tiles of three steps
    (24, 16, 16, 300, 128, True, False),
    (24, 16, 16, 300, 64, False, True),      # lengths 0 to N: items that only write zeros
    (24, 16, 16, 300, 128, True, True),
    (24, 16, 16, 600, 64, False, False),     # the narrow shape of heads of 64; so many heads that items are drawn
    (24, 16, 16, 800, 64, True, False),
    (12, 16, 4, 700, 64, True, False),
    (12, 16, 16, 1000, 64, False, True),
    (40, 16, 16, 260, 128, True, False),     # drawn items of one to three steps
])
def test_results_do_not_depend_on_the_items_before(B, H, H_kv, N, D, causal, padded):
    import torch
    import paper_2409_04431_b200 as sa
    g = torch.Generator(device="cuda").manual_seed(7 * N + D)
    q, k, v, d_o = (torch.randn((B, h, N, D), generator=g, device="cuda").to(torch.bfloat16) for h in (H, H_kv, H_kv, H))
    scale, bias = 1.0 / math.sqrt(D), -math.log(N)
    lens = torch.randint(0, N + 1, (B,), generator=g, device="cuda", dtype=torch.int32) if padded else None

    def run(lo, hi):
        x = [t[lo:hi].contiguous() for t in (q, k, v, d_o)]
        if padded:
            o = sa.sigattn_fwd_varlen(*x[:3], scale, bias, lens[lo:hi].contiguous(), causal)
            return (o, *sa.sigattn_bwd_varlen(*x, scale, bias, lens[lo:hi].contiguous(), causal)[:3])
        o = sa.sigattn_fwd_gqa(*x[:3], scale, bias, causal)
        return (o, *sa.sigattn_bwd_gqa(*x, scale, bias, causal)[:3])

    whole = run(0, B)
    names = "o dq dk dv".split()
    again = [run(0, B) for _ in range(3)]   # back to back: the next launch's blocks set up while the last ones end
    sa.sigattn_check()
    for repetition in again:
        for name, a, b in zip(names, whole, repetition):
            assert b.isfinite().all(), name
            if name != "dq":   # (dQ is summed over the key tiles in the order in which they arrive)
                assert torch.equal(a, b), name
            else:
                assert ((a.float() - b.float()).norm() <= 1e-3 * a.float().norm()).item()
    # the heads in halves of the batch: other items before each of them.  dK and dV of a key/value head with one query
    # head are one item's sums, the same to the last bit.  Otherwise what a row sums up is the same, up to the bf16
    # rounding of parts where a launch divides items: 2^-8 of the value and of the largest addend
    for lo, hi in ((0, B // 2), (B // 2, B)):
        part = run(lo, hi)
        for name, a, b in zip(names, whole, part):
            if H == H_kv and name in ("dk", "dv"):
                assert torch.equal(a[lo:hi], b), name
            a, b = a[lo:hi].float(), b.float()
            assert ((a - b).norm() <= 6e-3 * b.norm()).item(), name
    sa.sigattn_check()
    group = H // H_kv
    for b, h in ((0, 0), (B // 2, H_kv // 2), (B - 1, H_kv - 1)):
        kv, qs = (slice(b, b + 1), slice(h, h + 1)), (slice(b, b + 1), slice(h * group, (h + 1) * group))
        x = [to_host(t[i]) for t, i in zip((q, k, v, d_o), (qs, kv, kv, qs))]
        more = {"seqlens": [int(lens[b])]} if padded else {}
        refs = (oracle.sigattn_fwd(*x[:3], scale, bias, causal, **more), *oracle.sigattn_bwd(*x, scale, bias, causal, **more))
        for name, t, i, r in zip(names, whole, (qs, qs, kv, kv), refs):
            assert rel_fro(to_host(t[i]), r) < BF16_REL_FRO, (name, b, h)
