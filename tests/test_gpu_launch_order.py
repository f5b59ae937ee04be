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


@pytest.mark.parametrize("kind", ["forward", "backward"])
def test_replayed_calls_share_nothing_with_calls_in_flight(kind):
    """A captured call whose work items are drawn (so many heads of long sequences that they are handed out in groups)
    replays while a call on another stream, which has fewer items than the GPU has SMs, draws its own, after about as many
    launches as a rotation of 1024 shared slots takes to come round to the captured one: both write what they write alone."""
    import torch
    import paper_2409_04431_b200 as sa
    H, N, D = 21, 16384, 64
    g = torch.Generator(device="cuda").manual_seed(9)
    q, k, v, d_o = (torch.randn((1, H, N, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(4))
    a = (1.0 / math.sqrt(D), -math.log(N), True)
    T = 16384
    sq, sk, sv, sdo = (torch.randn((1, 1, T, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(4))
    cu = torch.tensor([0, T], dtype=torch.int32, device="cuda")
    sa_ = (1.0 / math.sqrt(D), -5.0, True)
    ws = torch.empty(sa.sigattn_bwd_workspace_bytes(1, H, N, D, 0), dtype=torch.uint8, device="cuda")
    small_ws = torch.empty(sa.sigattn_bwd_workspace_bytes(1, 1, T, D, 0), dtype=torch.uint8, device="cuda")
    outs, small_out = [torch.empty_like(q) for _ in range(3)], torch.empty_like(sq)

    def large():
        if kind == "forward":
            return [sa.sigattn_fwd(q, k, v, *a, out=outs[0])]
        return list(sa.sigattn_bwd(q, k, v, d_o, *a, workspace=ws, out=tuple(outs)))

    def small():
        if kind == "forward":
            return [sa.sigattn_fwd_ragged(sq, sk, sv, cu, *sa_, out=small_out)]
        return list(sa.sigattn_bwd_ragged(sq, sk, sv, sdo, cu, *sa_, workspace=small_ws)[:3])

    def differ(x, y):   # dQ (the first of a backward's results) is a sum in order of arrival, the others are exact
        d = [float((s.float() - t.float()).norm() / t.float().norm()) for s, t in zip(x, y)]
        return not all(e <= (1e-3 if kind == "backward" and i == 0 else 0.0) for i, e in enumerate(d)), d

    ref, small_ref = [t.clone() for t in large()], [t.clone() for t in small()]
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        large()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(1021):
            small()
    for _ in range(6):
        for t in outs + [small_out]:
            t.fill_(float("nan"))
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            got = small()
        graph.replay()
        torch.cuda.synchronize()
        for what, x, y in (("replayed", outs, ref), ("in flight", got, small_ref)):
            wrong, d = differ(x, y)
            assert not wrong, (what, d)
    sa.sigattn_check()
