"""Entry points called from other host threads than the one that made their
plans: every call succeeds and gives the values of a call made alone."""
import threading

import pytest
import torch

from paper_2609_24294_gb300 import zfpx as z

pytestmark = pytest.mark.gpu


def f64(rate):
    x = torch.randn((4, 8, 32), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(rate))
    s = torch.zeros(z.zfpx_stream_bytes_f64(rate, (32, 8, 4)), dtype=torch.uint8, device="cuda")
    return lambda stream: z.zfpx_encode_f64(rate, x, s, stream=stream), [s]


def rfft(n):
    x = torch.randn((1, 4, n), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    re, im = (torch.zeros((1, 4, n // 2), device="cuda") for _ in range(2))
    return lambda stream: z.zfpx_rfft_lon(x, re, im, stream=stream), [re, im]


def fused(n):
    x = torch.randn((4, 4, n), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    plan = z.Plan.for_fields(x, 1, 1, 0, 3)
    recv = torch.zeros(plan.buffer_bytes(8), dtype=torch.uint8, device="cuda")
    z.zfpx_pack_compress(plan, 8, x, recv, layout=z.LAYOUT_RECV)
    re, im = (torch.zeros((4, 4, n // 2), device="cuda") for _ in range(2))
    work = z.zfpx_decompress_rfft(plan, 8, recv, re, im)
    return lambda stream: z.zfpx_decompress_rfft(plan, 8, recv, re, im, work=work, stream=stream), [re, im]


def legendre(nlev):
    plan = z.Legendre(8, 7)
    g = torch.Generator("cuda").manual_seed(nlev)
    re, im = (torch.randn((nlev, 8, 8), device="cuda", generator=g) for _ in range(2))
    a = [torch.zeros((nlev, plan.ncoeffs), device="cuda") for _ in range(2)]
    return lambda stream: plan.forward(re, im, *a, stream=stream), a


def new_thread_runs(fn, times=1):
    """A thread, started, that calls fn; failures end up in its list."""
    failed = []

    def loop():
        try:
            for _ in range(times):
                fn()
        except Exception as e:
            failed.append(e)

    t = threading.Thread(target=loop)
    t.start()
    return t, failed


# a thread whose first CUDA call is the library's (the stream is made elsewhere)
@pytest.mark.parametrize("make,size", [(f64, 8), (rfft, 64), (fused, 64), (legendre, 8)])
def test_first_call_of_a_thread(make, size):
    fn, outs = make(size)
    st = torch.cuda.Stream()
    fn(st)
    torch.cuda.synchronize()
    want = [o.clone() for o in outs]
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    t, failed = new_thread_runs(lambda: fn(st))
    t.join()
    torch.cuda.synchronize()
    assert not failed
    assert all(torch.equal(o, w) for o, w in zip(outs, want))


# The limit on dynamic shared memory belongs to the kernel: no call may lower what
# another has asked for.  float64 rates of 49664 and 51712 bytes; the others'
# smallest and a large launch.
@pytest.mark.parametrize("make,sizes", [(f64, (28, 32)), (rfft, (20, 8100)), (fused, (20, 3750)), (legendre, (8, 96))])
def test_calls_of_two_sizes_from_four_threads(make, sizes):
    calls = []
    for size in sizes:
        fn, outs = make(size)
        fn(torch.cuda.current_stream())
        calls.append((fn, outs, [o.clone() for o in outs], torch.cuda.Stream()))
    for _, outs, _, _ in calls:
        for o in outs:
            o.zero_()
    torch.cuda.synchronize()
    threads = [new_thread_runs(lambda fn=fn, st=st: fn(st), 6000) for fn, _, _, st in calls for _ in range(2)]
    for t, _ in threads:
        t.join()
    torch.cuda.synchronize()
    assert not any(failed for _, failed in threads)
    for _, outs, want, _ in calls:
        assert all(torch.equal(o, w) for o, w in zip(outs, want))
