"""Calls whose heads are handed out in groups, the last one smaller than the others, and forwards whose items are cut
unevenly over two thread blocks: sampled heads on both sides of every border against the float64 oracle."""
import math

import numpy as np
import pytest

import oracle
from parity_util import BF16_REL_FRO, max_abs, rel_fro, to_host

pytestmark = pytest.mark.gpu


def _normal(*shape):
    import torch
    return torch.randn(shape, generator=_normal.g, device="cuda").to(torch.bfloat16)


@pytest.fixture(autouse=True)
def _seed():
    import torch
    _normal.g = torch.Generator(device="cuda").manual_seed(17)


def _close(got, ref, name):
    assert np.isfinite(got).all(), name
    assert rel_fro(got, ref) < BF16_REL_FRO, (name, rel_fro(got, ref))
    assert max_abs(got, ref) < 2e-2 * max(1.0, float(np.abs(ref).max())), name


def _check_heads(q, k, v, d_o, out, heads, scale, bias, causal, slopes=None, lens=None, row_block=None):
    """out: (O, dQ, dK, dV); heads: key/value heads (batch, head), each with all query heads that read it."""
    group = q.shape[1] // k.shape[1]
    for b, h in heads:
        kv, qs = (slice(b, b + 1), slice(h, h + 1)), (slice(b, b + 1), slice(h * group, (h + 1) * group))
        t = [to_host(x[s]) for x, s in ((q, qs), (k, kv), (v, kv), (d_o, qs))]
        more = {"seqlens": [lens[b]]} if lens is not None else {}
        sl = None if slopes is None else slopes[qs[1]]
        refs = (oracle.sigattn_fwd(*t[:3], scale, bias, causal, sl, row_block, **more),
                *oracle.sigattn_bwd(*t, scale, bias, causal, sl, row_block, **more))
        for name, x, s, r in zip(("O", "dQ", "dK", "dV"), out, (qs, qs, kv, kv), refs):
            _close(to_host(x[s]), r, f"{name}[{b},{h}]")


@pytest.mark.parametrize("B,H,N,D,causal,with_slopes", [
    (8, 30, 700, 128, True, False),    # 240 heads in groups of 93, 93 and 54
    (8, 30, 700, 128, False, True),
    (20, 30, 600, 64, False, False),   # 600 heads in groups of 218, 218 and 164
    (20, 30, 600, 64, True, True),
])
def test_plain(B, H, N, D, causal, with_slopes):
    import torch
    import paper_2409_04431_b200 as sa
    q, k, v, d_o = (_normal(B, H, N, D) for _ in range(4))
    slopes = np.exp2(-8.0 * np.arange(1, H + 1) / H).astype(np.float32) if with_slopes else None
    sl = None if slopes is None else torch.from_numpy(slopes).cuda()
    a = (1.0 / math.sqrt(D), -math.log(N), causal)
    out = (sa.sigattn_fwd(q, k, v, *a, sl), *sa.sigattn_bwd(q, k, v, d_o, *a, sl))
    sa.sigattn_check()
    n = 32 * 2 ** 20 // (N * D * 4)   # heads of a group
    edges = [0, n - 1, n, 2 * n - 1, 2 * n, B * H - 1]
    _check_heads(q, k, v, d_o, out, [divmod(e, H) for e in edges], *a, slopes)
    assert all(bool(torch.isfinite(t).all()) for t in out)


@pytest.mark.parametrize("B,H,H_kv,N,heads,row_block", [
    (8, 120, 30, 700, [0, 22, 23, 92, 93, 229, 230, 239], None),   # forward: groups of 93 key/value heads, backward: of 23
    (1, 12, 3, 8192, [1, 2], 1024),      # the query heads of a key/value head divided over two items; groups of 2 and 1
])
def test_grouped_heads(B, H, H_kv, N, heads, row_block):
    import paper_2409_04431_b200 as sa
    D = 128
    q, d_o, k, v = _normal(B, H, N, D), _normal(B, H, N, D), _normal(B, H_kv, N, D), _normal(B, H_kv, N, D)
    a = (1.0 / math.sqrt(D), -math.log(N), True)
    out = (sa.sigattn_fwd_gqa(q, k, v, *a), *sa.sigattn_bwd_gqa(q, k, v, d_o, *a)[:3])
    sa.sigattn_check()
    _check_heads(q, k, v, d_o, out, [divmod(e, H_kv) for e in heads], *a, row_block=row_block)


def test_padded_batch():
    import torch
    import paper_2409_04431_b200 as sa
    B, H, N, D = 30, 30, 700, 128      # 900 heads: groups of 93, the last one of 63
    q, k, v, d_o = (_normal(B, H, N, D) for _ in range(4))
    lens = np.random.default_rng(3).integers(1, N + 1, B)
    lens[[0, 5, 27]] = [N, 0, 1]
    tl = torch.from_numpy(lens.astype(np.int32)).cuda()
    scale, bias = 1.0 / math.sqrt(D), -5.0
    out = (sa.sigattn_fwd_varlen(q, k, v, scale, bias, tl, False), *sa.sigattn_bwd_varlen(q, k, v, d_o, scale, bias, tl, False)[:3])
    sa.sigattn_check()
    edges = [0, 92, 93, 5 * H + 7, 5 * 93, 27 * H + 26, 9 * 93 - 1, 9 * 93, B * H - 1]
    _check_heads(q, k, v, d_o, out, [divmod(e, H) for e in edges], scale, bias, False, lens=[int(n) for n in lens])
    for t in out:
        assert bool(torch.isfinite(t).all()) and not bool(t[5].any()) and not bool(t[27, :, 1:].any())


@pytest.mark.parametrize("N_q,N_k,with_slopes", [(700, 8192, False), (1024, 8192, True), (600, 8100, False)])
def test_items_cut_unevenly(N_q, N_k, with_slopes):
    """96 or 128 items of about equal cost on 148 SMs."""
    import torch
    import paper_2409_04431_b200 as sa
    H, H_kv, D = 32, 8, 128
    q, k, v = _normal(1, H, N_q, D), _normal(1, H_kv, N_k, D), _normal(1, H_kv, N_k, D)
    slopes = np.exp2(-8.0 * np.arange(1, H + 1) / H).astype(np.float32) if with_slopes else None
    sl = None if slopes is None else torch.from_numpy(slopes).cuda()
    scale, bias = 1.0 / math.sqrt(D), -math.log(N_k)
    o = sa.sigattn_fwd_nk(q, k, v, scale, bias, True, sl)
    assert torch.equal(o, sa.sigattn_fwd_nk(q, k, v, scale, bias, True, sl))   # the sum of two shares has no order
    sa.sigattn_check()
    for h in (0, 13, 31):
        kv = slice(h // 4, h // 4 + 1)
        ref = oracle.sigattn_fwd(to_host(q[:, h:h + 1]), to_host(k[:, kv]), to_host(v[:, kv]), scale, bias, True,
                                 None if slopes is None else slopes[h:h + 1])
        _close(to_host(o[:, h:h + 1]), ref, f"O[{h}]")
