"""The compiled host side of the calls: what it refuses, which stream it launches on, what it returns."""
import math

import pytest

pytestmark = pytest.mark.gpu


def _qkv(B=1, H=2, N=40, D=64, dtype=None):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    return [torch.randn((B, H, N, D), generator=g, device="cuda").to(dtype or torch.bfloat16) for _ in range(4)]


def test_refuses_what_the_kernels_could_not_read():
    import torch
    import paper_2409_04431_b200 as sa
    q, k, v, d_o = _qkv()
    a = (0.125, -3.0)
    for bad in (k.cpu(), k.float(), k[:, :, :20].contiguous(), k.transpose(1, 2), None, 3):
        with pytest.raises(ValueError):
            sa.sigattn_fwd(q, bad, v, *a)
        with pytest.raises(ValueError):
            sa.sigattn_bwd(q, k, v, bad, *a)
    with pytest.raises(TypeError):
        sa.sigattn_fwd(*(t.half() for t in (q, k, v)), *a)
    with pytest.raises(ValueError):
        sa.sigattn_fwd(q, k, v, *a, out=torch.empty_like(q, dtype=torch.float32))
    with pytest.raises(ValueError):
        sa.sigattn_bwd(q, k, v, d_o, *a, out=(q, k))
    with pytest.raises(ValueError):
        sa.sigattn_bwd(q, k, v, d_o, *a, workspace=torch.empty(1 << 20, device="cuda"))
    with pytest.raises(sa.SigattnError) as e:
        sa.sigattn_bwd(q, k, v, d_o, *a, workspace=torch.empty(64, dtype=torch.uint8, device="cuda"))
    assert e.value.code == -5
    for bias in (torch.zeros(2, device="cuda"), torch.zeros((1, 2)), torch.zeros((1, 2), dtype=torch.float64, device="cuda")):
        with pytest.raises(ValueError):
            sa.sigattn_fwd_gqa(q, k, v, 0.125, bias)
    with pytest.raises(ValueError):
        sa.sigattn_fwd_varlen(q, k, v, *a, torch.tensor([40, 40], dtype=torch.int32, device="cuda"))


def test_outputs_and_streams():
    """Given outputs come back as the same objects; the current stream and an explicit one (object or handle) see
    the launches: work queued behind a long spin on that stream reads what was written before it."""
    import torch
    import paper_2409_04431_b200 as sa
    q, k, v, d_o = _qkv()
    a = (1.0 / math.sqrt(64), -math.log(40))
    ref = sa.sigattn_fwd(q, k, v, *a)
    out = torch.empty_like(q)
    assert sa.sigattn_fwd(q, k, v, *a, out=out) is out and torch.equal(out, ref)
    grads = tuple(torch.empty_like(q) for _ in range(3))
    got = sa.sigattn_bwd(q, k, v, d_o, *a, out=grads)
    assert all(x is y for x, y in zip(got, grads))
    assert sa.sigattn_bwd_nk(q, k, v, d_o, *a)[3] is None
    assert sa.sigattn_bwd_nk(q, k, v, d_o, *a, want_dbias=True)[3].shape == (1, 2)
    side = torch.cuda.Stream()
    for how in ("current", "object", "handle"):
        late = torch.zeros_like(q)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            late.add_(torch.randn(2048, 2048, device="cuda").mm(torch.randn(2048, 2048, device="cuda"))[0, 0] * 0)
            late.copy_(q)
            if how == "current":
                o = sa.sigattn_fwd(late, k, v, *a)
        if how != "current":
            o = sa.sigattn_fwd(late, k, v, *a, stream=side if how == "object" else side.cuda_stream)
        side.synchronize()
        assert torch.equal(o, ref), how


@pytest.mark.parametrize("how", ["list", "generator", "map", "stacked tensor"])
def test_gradients_into_any_iterable_of_three(how):
    """`out` may be whatever unpacks into three tensors; what the call hands back is alive and is what it wrote, also
    where the iterable kept no reference to the tensors (freed ones would be handed out again by the allocations here)."""
    import torch
    import paper_2409_04431_b200 as sa
    q, k, v, d_o = _qkv(N=300)
    a = (1.0 / math.sqrt(64), -math.log(300))
    ref = sa.sigattn_bwd(q, k, v, d_o, *a)
    out = {"list": lambda: [torch.empty_like(q) for _ in range(3)], "generator": lambda: (torch.empty_like(q) for _ in range(3)),
           "map": lambda: map(torch.empty_like, (q, k, v)), "stacked tensor": lambda: torch.empty((3, *q.shape), dtype=q.dtype, device="cuda")}[how]()
    got = sa.sigattn_bwd(q, k, v, d_o, *a, out=out)
    later = [torch.full_like(q, 7.0) for _ in range(6)]
    assert len(got) == 3 and len(later) == 6 and all(isinstance(x, torch.Tensor) for x in got)
    assert torch.equal(got[1], ref[1]) and torch.equal(got[2], ref[2])
    assert float((got[0].float() - ref[0].float()).norm() / ref[0].float().norm()) < 1e-3   # dQ: fp32 sums in another order
    if how == "stacked tensor":
        assert all(x.data_ptr() == out[i].data_ptr() for i, x in enumerate(got))
    for wrong in ((q, k), (q, k, v, d_o), iter([q, k])):
        with pytest.raises(ValueError):
            sa.sigattn_bwd(q, k, v, d_o, *a, out=wrong)
    with pytest.raises(TypeError):
        sa.sigattn_bwd(q, k, v, d_o, *a, out=3)


@pytest.mark.parametrize("what", ["forward", "backward"])
def test_other_threads_run_while_a_launch_waits(what):
    """A launch blocks when the stream's queue is full; the calls do not hold the interpreter lock meanwhile.  The stream
    is kept busy for about half a second and more launches are queued than it takes; the longest pause of a thread that
    only counts has to be far shorter than the wait (the interpreter's own switch interval is 5 ms)."""
    import threading
    import time
    import torch
    import paper_2409_04431_b200 as sa
    q, k, v, d_o = _qkv()
    o, grads = torch.empty_like(q), tuple(torch.empty_like(q) for _ in range(3))
    a = (0.125, -3.0)
    call = {"forward": lambda: sa.sigattn_fwd(q, k, v, *a, out=o), "backward": lambda: sa.sigattn_bwd(q, k, v, d_o, *a, out=grads)}[what]
    call()
    torch.cuda.synchronize()
    stop, pauses = threading.Event(), []

    def count():
        last = time.perf_counter()
        while not stop.is_set():
            time.sleep(0.0005)
            now = time.perf_counter()
            pauses.append(now - last)
            last = now

    counter = threading.Thread(target=count)
    counter.start()
    try:
        torch.cuda._sleep(1_000_000_000)
        t0 = time.perf_counter()
        longest = 0.0
        for _ in range(4000):
            t1 = time.perf_counter()
            call()
            longest = max(longest, time.perf_counter() - t1)
            if time.perf_counter() - t0 > 5.0:
                break
    finally:
        stop.set()
        counter.join()
        torch.cuda.synchronize()
    assert longest > 0.2, longest          # some launch did wait for the queue
    assert max(pauses) < 0.5 * longest, (max(pauses), longest)


@pytest.mark.parametrize("how", ["object", "handle"])
@pytest.mark.parametrize("what", ["backward", "decode", "forward", "static scratch"])
def test_memory_of_calls_on_another_stream(what, how):
    """An explicit stream that is not the current one, with everything allocated by the call: its scratch and results
    share no memory with what the current stream has in use, before the call or after it."""
    import torch
    import paper_2409_04431_b200 as sa
    spin = 100_000_000   # about 50 ms
    B, H, N, D = (2, 8, 400, 64) if what != "decode" else (1, 2, 1, 128)   # the latter: sums of several clusters in scratch
    g = torch.Generator(device="cuda").manual_seed(3)
    q, d_o = (torch.randn((B, H, N, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    k, v = (torch.randn((B, H, 70000 if what == "decode" else N, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    a = (1.0 / math.sqrt(D), -math.log(k.shape[2]))
    call = {"backward": lambda **x: sa.sigattn_bwd(q, k, v, d_o, *a, **x)[0], "forward": lambda **x: sa.sigattn_fwd(q, k, v, *a, **x),
            "decode": lambda **x: sa.sigattn_fwd_decode(q, k, v, *a, **x),
            "static scratch": lambda **x: sa.sigattn_bwd_static_scratch(q, k, v, d_o, *a, **x)[0]}[what]
    ref = call()
    side = torch.cuda.Stream()
    stream = side if how == "object" else side.cuda_stream
    scratch = {"backward": sa.sigattn_bwd_workspace_bytes(B, H, N, D, 0), "decode": sa.sigattn_fwd_decode_workspace_bytes(B, H, N, D, 0)}.get(what, 0)
    sizes = [n for n in (scratch, q.numel() * 2) if n]

    def close(x):
        return float((x.float() - ref.float()).norm() / ref.float().norm()) < 1e-3   # (fp32 sums in another order)

    torch.cuda.synchronize()
    # memory that the current stream still writes when the call on the other one has long ended
    before = [torch.empty(n, dtype=torch.uint8, device="cuda") for n in sizes for _ in range(3)]
    torch.cuda._sleep(spin)
    for x in before:
        x.fill_(255)
    del before, x
    got = call(stream=stream)
    torch.cuda.synchronize()
    assert close(got)
    # memory that the current stream takes and fills while the call's kernels have not begun
    with torch.cuda.stream(side):
        torch.cuda._sleep(spin)
    got = call(stream=stream)
    after = [torch.full((n,), 7, dtype=torch.uint8, device="cuda") for n in sizes for _ in range(3)]
    torch.cuda.synchronize()
    assert close(got) and all(bool((x == 7).all()) for x in after)
    # a result that the current stream still reads when it is dropped
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda._sleep(spin)
    kept = got.clone()
    del got
    with torch.cuda.stream(side):
        later = [torch.zeros_like(q) for _ in range(6)]
    torch.cuda.synchronize()
    assert close(kept) and len(later) == 6
    sa.sigattn_check()


def test_refuses_scratch_the_kernels_could_not_use():
    import torch
    import paper_2409_04431_b200 as sa
    q, k, v, d_o = _qkv(N=300)
    a = (0.125, -5.0)
    size = sa.sigattn_bwd_workspace_bytes(1, 2, 300, 64, 0)
    ok = torch.empty(size, dtype=torch.uint8, device="cuda")
    bad = (torch.empty(size, dtype=torch.uint8), torch.empty(size // 4, device="cuda"), torch.empty(2 * size, dtype=torch.uint8, device="cuda")[::2], size)
    for w in bad:
        with pytest.raises(ValueError):
            sa.sigattn_bwd(q, k, v, d_o, *a, workspace=w)
        with pytest.raises(ValueError):
            sa.sigattn_fwd_decode(q[:, :, :1].contiguous(), k, v, *a, workspace=w)
    for w, code in ((ok[:size - 1], -5), (torch.empty(size + 16, dtype=torch.uint8, device="cuda")[16:], -3)):
        with pytest.raises(sa.SigattnError) as e:
            sa.sigattn_bwd(q, k, v, d_o, *a, workspace=w)
        assert e.value.code == code
    sa.sigattn_bwd(q, k, v, d_o, *a, workspace=ok)
    sa.sigattn_check()
