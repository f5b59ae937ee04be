"""GPU parity of the kernels for short sequences (heads of 64, N <= 256) at the edges of their column counts,
against the float64 oracle, and on more heads than fit the GPU at once, against the general kernels."""
import math

import numpy as np
import pytest

import oracle
from paper_2409_04431_b200 import inputs
from parity_util import assert_bf16_close, to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 33, 96, 160, 161, 192, 193, 224, 225, 240])
@pytest.mark.parametrize("causal,with_slopes", [(False, False), (True, True), (False, True)])
def test_short_edges(N, causal, with_slopes):
    import torch
    import paper_2409_04431_b200 as sa
    B, H, D = 1, 3, 64
    q, k, v, d_o = inputs.random_case(B, H, N, D, 400 + N)
    slopes = (0.5 ** np.arange(1, H + 1)).astype(np.float32) if with_slopes else None
    sl = None if slopes is None else torch.from_numpy(slopes).cuda()
    tq, tk, tv, tdo = (to_device(t, "bf16") for t in (q, k, v, d_o))
    scale, bias = 1.0 / math.sqrt(D), -math.log(N)
    o = sa.sigattn_fwd(tq, tk, tv, scale, bias, causal, sl)
    grads = sa.sigattn_bwd(tq, tk, tv, tdo, scale, bias, causal, sl)
    sa.sigattn_check()
    assert_bf16_close(to_host(o), oracle.sigattn_fwd(q, k, v, scale, bias, causal, slopes), "O")
    for name, g, r in zip(("dQ", "dK", "dV"), grads, oracle.sigattn_bwd(q, k, v, d_o, scale, bias, causal, slopes)):
        assert_bf16_close(to_host(g), r, name)


@pytest.mark.parametrize("B,N,causal", [(40, 197, False), (30, 256, True), (61, 100, False)])
def test_short_many_heads_equal_the_general_kernels(B, N, causal):
    """The same weights, rounded at the same places and summed in the same order: O, dK and dV of the padded-batch
    entry points with full lengths (the general kernels) are bit-identical."""
    import torch
    import paper_2409_04431_b200 as sa
    H, D = 12, 64
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v, d_o = (torch.randn((B, H, N, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(4))
    full = torch.full((B,), N, dtype=torch.int32, device="cuda")
    scale, bias = 1.0 / math.sqrt(D), -math.log(N)
    assert torch.equal(sa.sigattn_fwd(q, k, v, scale, bias, causal), sa.sigattn_fwd_varlen(q, k, v, scale, bias, full, causal))
    a = sa.sigattn_bwd(q, k, v, d_o, scale, bias, causal)
    b = sa.sigattn_bwd_varlen(q, k, v, d_o, scale, bias, full, causal)
    sa.sigattn_check()
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    assert float((a[0].float() - b[0].float()).norm() / b[0].float().norm()) < 1e-3   # dQ: fp32 sums in another order


@pytest.mark.parametrize("kind,H,H_kv,N", [
    ("plain", 3, 3, 300), ("causal", 3, 3, 700), ("grouped", 4, 2, 385), ("padded", 2, 2, 520), ("packed", 2, 1, 900),
])
def test_wide_backward_at_64(kind, H, H_kv, N):
    """The four-group shape of the backward (typical sequences up to 1280 rows, heads of 64): every kind of call that
    reaches it, with a ragged last tile, several query tiles per item and several items per thread block."""
    import torch
    import paper_2409_04431_b200 as sa
    B, D, causal = (1 if kind == "packed" else 2), 64, kind in ("causal", "packed")
    q, _, _, d_o = inputs.random_case(B, H, N, D, 500 + N)
    _, k, v, _ = inputs.random_case(B, H_kv, N, D, 501 + N)
    tq, tk, tv, tdo = (to_device(t, "bf16") for t in (q, k, v, d_o))
    scale, bias, more = 1.0 / math.sqrt(D), -math.log(N), {}
    if kind == "padded":
        lens = [N, N // 3]
        out = sa.sigattn_bwd_varlen(tq, tk, tv, tdo, scale, bias, torch.tensor(lens, dtype=torch.int32, device="cuda"), causal)
        more = {"seqlens": lens}
    elif kind == "packed":
        cu = np.array([0, 10, 300, 301, N], dtype=np.int32)
        out = sa.sigattn_bwd_ragged(tq, tk, tv, tdo, torch.from_numpy(cu).cuda(), scale, bias, causal)
        more = {"cu_seqlens": cu}
    else:
        out = sa.sigattn_bwd_gqa(tq, tk, tv, tdo, scale, bias, causal, want_dbias=True)
    sa.sigattn_check()
    for name, g, r in zip(("dQ", "dK", "dV"), out, oracle.sigattn_bwd(q, k, v, d_o, scale, bias, causal, None, **more)):
        assert_bf16_close(to_host(g), r, name)


@pytest.mark.parametrize("H,H_kv,N,causal", [(3, 3, 500, False), (3, 3, 530, False), (4, 2, 500, False), (4, 2, 530, False),
                                             (4, 2, 890, True), (4, 2, 910, True)])
def test_backward_shapes_meet_at_64(H, H_kv, N, causal):
    """ALiBi on both sides of the lines between the wide and the narrow backward: 512 rows without a mask, 900 rows of
    a causal call with grouped heads (two thirds of them count as typical)."""
    import torch
    import paper_2409_04431_b200 as sa
    B, D = 1, 64
    q, _, _, d_o = inputs.random_case(B, H, N, D, 600 + N)
    _, k, v, _ = inputs.random_case(B, H_kv, N, D, 601 + N)
    slopes = (0.5 ** np.arange(1, H + 1)).astype(np.float32)
    tq, tk, tv, tdo = (to_device(t, "bf16") for t in (q, k, v, d_o))
    scale, bias = 1.0 / math.sqrt(D), -math.log(N)
    out = sa.sigattn_bwd_gqa(tq, tk, tv, tdo, scale, bias, causal, torch.from_numpy(slopes).cuda())
    sa.sigattn_check()
    for name, g, r in zip(("dQ", "dK", "dV"), out, oracle.sigattn_bwd(q, k, v, d_o, scale, bias, causal, slopes)):
        assert_bf16_close(to_host(g), r, name)
