"""The backward of heads of 64 in its narrow shape (long sequences), causal: grouped heads, the query heads or the query
tiles of an item divided, padded batches, packed documents and key/value shards, with several items per thread block;
sampled heads against the float64 oracle."""
import math

import numpy as np
import pytest

import oracle
from parity_util import BF16_REL_FRO, max_abs, rel_fro, to_host

pytestmark = pytest.mark.gpu

D, SCALE = 64, 0.125
NAMES = ("dQ", "dK", "dV")


def _inputs(B, H, H_kv, N, N_k=None, seed=23):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    shapes = (H, N), (H_kv, N_k or N), (H_kv, N_k or N), (H, N)
    return [torch.randn((B, h, n, D), generator=g, device="cuda").to(torch.bfloat16) for h, n in shapes]


def _spoil(q, k, v):
    """Leaves blocks full of NaN behind, which the allocator hands out again for results of these sizes."""
    import torch
    [torch.full_like(t, float("nan")) for t in (q, k, v)]


def _slopes(H, with_slopes):
    import torch
    if not with_slopes:
        return None, None
    s = np.exp2(-8.0 * np.arange(1, H + 1) / H).astype(np.float32)
    return s, torch.from_numpy(s).cuda()


def _close(got, ref, name):
    assert np.isfinite(got).all(), name
    assert rel_fro(got, ref) < BF16_REL_FRO, (name, rel_fro(got, ref))
    assert max_abs(got, ref) < 2e-2 * max(1.0, float(np.abs(ref).max())), name


def _check(x, grads, db, heads, slopes, rows=slice(None), bias=None, **more):
    """heads: (batch, key/value head), each with all query heads that read it; db: [batch or sequence, query head]."""
    group = x[0].shape[1] // x[1].shape[1]
    got_db, ref_db = [], []
    for b, h in heads:
        kv, qs = (slice(b, b + 1), slice(h, h + 1), rows), (slice(b, b + 1), slice(h * group, (h + 1) * group), rows)
        t = [to_host(a[s]) for a, s in zip(x, (qs, kv, kv, qs))]
        lens = {"seqlens": [more["seqlens"][b]]} if "seqlens" in more else {}
        a = (*t, SCALE, bias, True, None if slopes is None else slopes[qs[1]], 1024)
        for name, g, s, r in zip(NAMES, grads, (qs, kv, kv), oracle.sigattn_bwd(*a, **lens)):
            _close(to_host(g[s]), r, f"{name}[{b},{h}]")
        if db is not None:
            got_db.append(db[more.get("db_row", b), qs[1]].cpu().numpy().astype(np.float64))
            ref_db.append(oracle.sigattn_bwd_dbias(*a, **lens)[0])
    if db is not None:   # a sum of signed terms per head: compared over the sampled heads together
        assert rel_fro(np.stack(got_db), np.stack(ref_db)) < BF16_REL_FRO


@pytest.mark.parametrize("B,N,with_slopes,want_dbias", [
    (8, 3000, False, True),     # 768 items
    (8, 3000, True, False),
    (2, 3050, True, True),      # few items: the query heads of a key/value head divided over several, whose parts add up
    (2, 3050, False, False),
])
def test_grouped_heads(B, N, with_slopes, want_dbias):
    import paper_2409_04431_b200 as sa
    H, H_kv = 16, 4
    x = _inputs(B, H, H_kv, N)
    slopes, sl = _slopes(H, with_slopes)
    bias = -math.log(N)
    _spoil(*x[:3])
    *out, db = sa.sigattn_bwd_gqa(*x, SCALE, bias, True, sl, want_dbias=want_dbias)
    sa.sigattn_check()
    _check(x, out, db, [(0, 0), (B - 1, 3)], slopes, bias=bias)


def test_divided_query_tiles():
    """One sequence, two heads: the query tiles of a key tile divided over two items."""
    import paper_2409_04431_b200 as sa
    N = 2900
    x = _inputs(1, 2, 2, N)
    _spoil(*x[:3])
    out = sa.sigattn_bwd(*x, SCALE, -math.log(N), True)
    sa.sigattn_check()
    _check(x, out, None, [(0, 0), (0, 1)], None, bias=-math.log(N))


@pytest.mark.parametrize("with_slopes,want_dbias", [(False, True), (True, False)])
def test_padded_batch(with_slopes, want_dbias):
    import torch
    import paper_2409_04431_b200 as sa
    B, H, N = 8, 4, 4200
    lens = [1500, 0, 1, N, 130, 128, 2000, 3001]
    x = _inputs(B, H, H, N)
    slopes, sl = _slopes(H, with_slopes)
    _spoil(*x[:3])
    tl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    *out, db = sa.sigattn_bwd_varlen(*x, SCALE, -7.0, tl, True, sl, want_dbias=want_dbias)
    sa.sigattn_check()
    _check(x, out, db, [(0, 1), (2, 0), (4, 3)], slopes, bias=-7.0, seqlens=lens)
    for t in out:
        assert bool(torch.isfinite(t).all())
        assert all(not bool(t[b, :, n:].any()) for b, n in enumerate(lens))


@pytest.mark.parametrize("H,H_kv,with_slopes,want_dbias", [(16, 16, False, True), (16, 4, True, True), (16, 4, False, False)])
def test_packed_documents(H, H_kv, with_slopes, want_dbias):
    import torch
    import paper_2409_04431_b200 as sa
    lens = [1700, 3301, 1000, 2399]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    x = _inputs(1, H, H_kv, int(cu[-1]))
    slopes, sl = _slopes(H, with_slopes)
    bias = -np.log(np.array(lens, dtype=np.float64))
    tb = torch.from_numpy(np.repeat(bias[:, None], H, axis=1).astype(np.float32)).cuda().contiguous()
    _spoil(*x[:3])
    *out, db = sa.sigattn_bwd_ragged(*x, torch.from_numpy(cu).cuda(), SCALE, tb, True, sl, want_dbias=want_dbias)
    sa.sigattn_check()
    for s, heads in ((0, [(0, 0)]), (2, [(0, 1), (0, H_kv - 1)]), (3, [(0, 2)])):
        _check(x, out, db, heads, slopes, rows=slice(int(cu[s]), int(cu[s + 1])), bias=float(bias[s]), db_row=s)
    assert all(bool(torch.isfinite(t).all()) for t in out)


def test_key_value_shard():
    """The shard's gradients are added to what is there: two calls give twice the oracle's."""
    import torch
    import paper_2409_04431_b200 as sa
    H, H_kv, N, N_k, pos0 = 8, 2, 2900, 900, -300
    x = _inputs(1, H, H_kv, N, N_k)
    acc = torch.zeros(x[0].shape, dtype=torch.float32, device="cuda")
    dk, dv = torch.zeros_like(x[1]), torch.zeros_like(x[2])
    for _ in range(2):
        sa.sigattn_bwd_shard_acc_kv(*x, acc, dk, dv, SCALE, -7.0, pos0, True)
    sa.sigattn_check()
    t = [to_host(a[:, s]) for a, s in zip(x, (slice(0, 4), slice(0, 1), slice(0, 1), slice(0, 4)))]
    refs = oracle.sigattn_bwd(*t, SCALE, -7.0, True, row_block=1024, pos0=pos0)
    _close(SCALE * to_host(acc[:, :4]), 2 * refs[0], "dQ")
    # dK, dV: every addition (two calls, four parts of the query heads each) rounds the sum to bf16, uniformly within
    # 2^-9 of it: 2^-9 sqrt(8 / 3), and the parts are smaller than the sum
    for name, g, r in zip(NAMES[1:], (dk, dv), refs[1:]):
        assert rel_fro(to_host(g[:, :1]), 2 * r) < BF16_REL_FRO * math.sqrt(2.0), name
