"""Kernels that may begin while the one before them still runs: chains of calls in which each reads what the one
before wrote give the same bits as the same chains with a synchronisation after every call."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,B,H,N,D,dtype", [
    ("forward", 1, 12, 197, 64, "bf16"), ("forward", 2, 4, 600, 128, "bf16"), ("forward", 1, 2, 100, 64, "fp32"),
    ("backward", 2, 12, 197, 64, "bf16"), ("backward", 1, 6, 700, 64, "bf16"), ("backward", 1, 4, 520, 128, "bf16"),
    ("backward", 1, 2, 100, 128, "fp32"), ("decode", 2, 8, 2000, 128, "bf16"), ("decode", 40, 8, 300, 64, "bf16"),
])
def test_chained_calls(kind, B, H, N, D, dtype):
    import torch
    import paper_2409_04431_b200 as sa
    g = torch.Generator(device="cuda").manual_seed(7)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    q, k, v, d_o = (torch.randn((B, H, n, D), generator=g, device="cuda").to(t) for n in (1 if kind == "decode" else N, N, N, N))
    scale, bias = 1.0 / math.sqrt(D), -math.log(N)
    ws = torch.empty(max(1, sa.sigattn_bwd_workspace_bytes(B, H, N, D, 0)), dtype=torch.uint8, device="cuda")

    def chain(sync):
        x, buf = q.clone(), [torch.empty_like(q) for _ in range(2)]
        for step in range(24):
            if kind == "forward":
                x = sa.sigattn_fwd(x, k, v, scale, bias, True, out=buf[step & 1])
            elif kind == "decode":
                x = sa.sigattn_fwd_decode(x, k, v, scale, bias, True, out=buf[step & 1])
            else:   # dV (its bits do not depend on timing) becomes the next call's dO, by way of the forward
                dv = sa.sigattn_bwd(q, k, v, x, scale, bias, True, workspace=ws)[2]
                x = sa.sigattn_fwd(dv, k, v, scale, bias, True, out=buf[step & 1])
            if sync:
                torch.cuda.synchronize()
        sa.sigattn_check()
        return x.clone()

    assert torch.equal(chain(False), chain(True))
