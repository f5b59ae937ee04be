"""GPU parity of the decoding kernel that divides a head's keys over a thread-block cluster: every cluster
size, the edges of its row count and of a key tile, against the float64 oracle, through the C ABI."""
import math

import numpy as np
import pytest

import oracle
from paper_2409_04431_b200 import inputs
from parity_util import BF16_REL_FRO, max_abs, rel_fro, to_device, to_host

pytestmark = pytest.mark.gpu


def _run(B, H, H_kv, N_q, N_k, D, causal, with_slopes):
    import torch
    import paper_2409_04431_b200 as sa
    q, _, _, _ = inputs.random_case(B, H, N_q, D, 301)
    _, k, v, _ = inputs.random_case(B, H_kv, N_k, D, 302)
    slopes = np.exp2(-8.0 * np.arange(1, H + 1) / H).astype(np.float32) if with_slopes else None
    bias = (-math.log(N_k) + 0.3 * np.random.default_rng(303).standard_normal((B, H))).astype(np.float32)
    tq, tk, tv = (to_device(t, "bf16") for t in (q, k, v))
    sl = None if slopes is None else torch.from_numpy(slopes).cuda()
    tb = torch.from_numpy(bias).cuda()
    before = sa.sigattn_launch_count()
    o = sa.sigattn_fwd_decode(tq, tk, tv, 1.0 / math.sqrt(D), tb, causal, sl)
    launches = sa.sigattn_launch_count() - before
    again = sa.sigattn_fwd_decode(tq, tk, tv, 1.0 / math.sqrt(D), tb, causal, sl)
    sa.sigattn_check()
    g = to_host(o)
    ref = oracle.sigattn_fwd(q, k, v, 1.0 / math.sqrt(D), bias.astype(np.float64), causal, slopes)
    assert np.isfinite(g).all()
    assert rel_fro(g, ref) < BF16_REL_FRO, rel_fro(g, ref)
    assert max_abs(g, ref) < 2e-2 * max(1.0, float(np.abs(ref).max()))
    return launches, torch.equal(o, again)


@pytest.mark.parametrize("B,H,H_kv,N_q,N_k,D,causal,with_slopes", [
    (1, 8, 2, 1, 2048, 128, True, False),      # 16 key tiles over 16 thread blocks, one each
    (1, 8, 2, 1, 4000, 64, True, True),        # 32 tiles over 16, ragged last tile
    (1, 32, 8, 1, 2000, 128, True, False),     # eight heads over clusters of eight
    (2, 64, 32, 1, 300, 128, True, True),      # 64 heads, 3 tiles: clusters of two, shares of one and two tiles
    (3, 100, 50, 1, 260, 64, True, False),     # 150 heads: one thread block per head, two per SM
    (2, 16, 16, 64, 1000, 128, True, False),   # 64 rows, the most the kernel takes
    (1, 16, 16, 17, 130, 64, True, True),      # 17 rows (padded to 32), second tile of two keys
    (80, 2, 2, 1, 700, 128, False, False),     # 160 heads without a mask, six tiles each, two per SM
    (40, 4, 4, 64, 900, 128, True, True),      # 64 rows and more heads than SMs: the large ring
    (1, 1, 1, 2, 129, 64, False, False),       # two keys' worth of a second tile, one head
])
def test_decode_one_cluster_per_head(B, H, H_kv, N_q, N_k, D, causal, with_slopes):
    launches, same = _run(B, H, H_kv, N_q, N_k, D, causal, with_slopes)
    assert launches == 1      # the cluster adds its parts itself: nothing to convert
    assert same               # ... in rank order


@pytest.mark.parametrize("B,H,H_kv,N_q,N_k,D,causal,with_slopes", [
    (1, 2, 1, 1, 16500, 64, True, True),       # 129 tiles: the fewest that one head divides over several clusters
    (1, 8, 8, 2, 17000, 128, True, False),     # eight heads, four clusters of four each
])
def test_decode_several_clusters_per_head(B, H, H_kv, N_q, N_k, D, causal, with_slopes):
    launches, _ = _run(B, H, H_kv, N_q, N_k, D, causal, with_slopes)
    assert launches == 2      # sums in scratch, then converted


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("N_k", [300, 2000, 2048])
def test_decode_values_that_are_not_finite(N_k, causal):
    """NaN in one cached key reaches every head that reads it; Inf in a query, whose logits are +-Inf, weighs the keys
    with 1 and 0 (also where the last tile holds rows that do not exist)."""
    import torch
    import paper_2409_04431_b200 as sa
    H, H_kv, D = 8, 2, 128
    g = torch.Generator(device="cuda").manual_seed(N_k)
    q = torch.randn((1, H, 1, D), generator=g, device="cuda").to(torch.bfloat16)
    k, v = (torch.randn((1, H_kv, N_k, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    a = (1.0 / math.sqrt(D), -math.log(N_k), causal)
    clean = sa.sigattn_fwd_decode(q, k, v, *a)
    bad = k.clone()
    bad[0, 0, 17, 5] = float("nan")
    o = sa.sigattn_fwd_decode(q, bad, v, *a)
    assert bool(torch.isnan(o[0, :4]).all()) and torch.equal(o[0, 4:], clean[0, 4:])
    inf = q.clone()
    inf[0, 3, 0, 7] = float("inf")
    o = sa.sigattn_fwd_decode(inf, k, v, *a)
    sa.sigattn_check()
    want = (k[0, 0, :, 7] > 0).double().cpu() @ v[0, 0].double().cpu()
    assert rel_fro(to_host(o)[0, 3, 0], want.numpy()) < BF16_REL_FRO
    keep = [h for h in range(H) if h != 3]
    assert torch.equal(o[0, keep], clean[0, keep])
