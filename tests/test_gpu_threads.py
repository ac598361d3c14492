"""Calls from several threads, each on a stream of its own: the same bits as one call after the other, and no call fails because another
thread's asks the same kernel for less shared memory."""
import threading

import pytest
import torch

from paper_2511_05534_b200 import binding as F

pytestmark = pytest.mark.gpu


def _call(U, H, G, L, W, B):
    """A compression with its own buffers: (call, outputs)."""
    gen = torch.Generator(device="cuda").manual_seed(L + B)
    q, k, v = (torch.randn((U, h, t, 128), generator=gen, device="cuda").bfloat16() for h, t in ((H * G, W), (H, L), (H, L)))
    m = (torch.arange(L, device="cuda") % 70 < 50).to(torch.uint8)[None].repeat(U, 1)
    p = F.Params(U, H * G, H, 128, L, W, B, theta=0.3, tau=2.0, tau_mode=F.TAU_REL)
    k_out, v_out = (torch.zeros((U, H, B, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ws = F.alloc_workspace(p)
    return lambda: F.flowmm_compress_layer(p, q, k, v, m, k_out, v_out, ws), (k_out, v_out), ws


def test_first_call_of_a_thread():
    """A thread that has not used CUDA before: the first thing it does is a call that describes tensors to the driver."""
    call, outs, ws = _call(1, 4, 4, 400, 32, 16)
    call()
    want = [o.clone() for o in outs]
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    errors = []

    def work():
        try:
            call()
        except Exception as e:                                      # (an assertion of a thread would go unseen)
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not errors and F.flowmm_last_device_status(ws) == 0
    assert all(torch.equal(o, w) for o, w in zip(outs, want))


# pairs of calls that meet in a kernel with different needs of shared memory
@pytest.mark.parametrize("shapes", [
    ((1, 4, 4, 400, 32, 16), (1, 4, 8, 1000, 64, 200)),             # scoring by clusters, selection, merge on the tensor cores
    ((20, 4, 1, 200, 32, 1), (20, 4, 1, 640, 32, 64)),              # matching and merge in one launch
    ((1, 4, 1, 3000, 32, 300), (1, 4, 1, 9000, 32, 900)),           # lists by clusters, selection by clusters
    ((40, 4, 1, 1500, 32, 300), (50, 4, 1, 4000, 32, 800)),         # lists of a block per head
])
def test_threads_with_calls_of_other_sizes(shapes):
    calls = [_call(*s) for s in shapes for _ in range(2)]
    expected = []
    for call, outs, _ in calls:
        call()
        expected.append([o.clone() for o in outs])
        for o in outs:
            o.zero_()
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(300):
                    calls[i][0]()
                torch.cuda.current_stream().synchronize()
        except Exception as e:                                      # (an assertion of a thread would go unseen)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    for (_, outs, ws), want in zip(calls, expected):
        assert F.flowmm_last_device_status(ws) == 0
        assert all(torch.equal(o, w) for o, w in zip(outs, want))
