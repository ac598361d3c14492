"""Calls from several threads."""
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
