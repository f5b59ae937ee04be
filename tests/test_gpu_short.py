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
    """The four-group shape of the backward (short sequences, heads of 64): every kind of call that reaches it, with a
    ragged last tile and several query tiles per item."""
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
    """ALiBi at lengths of 500 and 900 rows, where both shapes of the backward have served."""
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


@pytest.mark.parametrize("kind,N,causal,with_slopes", [
    ("plain", 320, False, False), ("plain", 321, False, False),       # wide up to 320 rows
    ("plain", 752, True, False), ("plain", 753, True, True),          # 500, two thirds of the rows count as typical
    ("grouped", 480, False, True), ("grouped", 481, False, False),
    ("grouped", 542, True, True), ("grouped", 543, True, False),      # 360
    ("padded", 901, False, False), ("padded", 902, True, False),      # 450, half of the rows
    ("padded", 501, False, True), ("padded", 502, False, True),       # 250
    ("packed", 1280, True, False), ("packed", 1281, True, False),     # rows per document
    ("packed", 900, False, True), ("packed", 901, False, True),
])
def test_backward_on_both_sides_of_the_wide_shapes_lines(kind, N, causal, with_slopes):
    """The last length that the wide shape of the backward serves and the first of the narrow one, for each kind of call."""
    import torch
    import paper_2409_04431_b200 as sa
    B, D = (1 if kind == "packed" else 2), 64
    H, H_kv = (4, 2) if kind == "grouped" else (2, 2)
    q, _, _, d_o = inputs.random_case(B, H, N, D, 700 + N)
    _, k, v, _ = inputs.random_case(B, H_kv, N, D, 701 + N)
    slopes = (0.5 ** np.arange(1, H + 1)).astype(np.float32) if with_slopes else None
    sl = None if slopes is None else torch.from_numpy(slopes).cuda()
    t = [to_device(x, "bf16") for x in (q, k, v, d_o)]
    scale, bias, more = 1.0 / math.sqrt(D), -math.log(N), {}
    if kind == "padded":
        lens = [N, N // 3]
        out = sa.sigattn_bwd_varlen(*t, scale, bias, torch.tensor(lens, dtype=torch.int32, device="cuda"), causal, sl)
        more = {"seqlens": lens}
    elif kind == "packed":
        cu = np.array([0, N], dtype=np.int32)
        out = sa.sigattn_bwd_ragged(*t, torch.from_numpy(cu).cuda(), scale, bias, causal, sl)
        more = {"cu_seqlens": cu}
    elif kind == "grouped":
        out = sa.sigattn_bwd_gqa(*t, scale, bias, causal, sl)
    else:
        out = sa.sigattn_bwd(*t, scale, bias, causal, sl)
    sa.sigattn_check()
    for name, g, r in zip(("dQ", "dK", "dV"), out, oracle.sigattn_bwd(q, k, v, d_o, scale, bias, causal, slopes, **more)):
        assert_bf16_close(to_host(g), r, name)
