"""wd_finalize beside another host thread's network calls: a call keeps the
scratch that it has."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_finalize_leaves_a_running_calls_scratch():
    import torch
    import paper_0810_5365_gb300 as W
    dims = (8, 8, 8, 8)
    g = torch.Generator(device="cuda").manual_seed(7)
    rnd = lambda n: torch.randn(n, device="cuda", generator=g)  # noqa: E731
    gauge = (0.3 * rnd(W.wd_gauge_bytes(dims, W.WD_F32, 12) // 4)).view(torch.uint8)
    w, x = 0.2 * rnd(W.WD_NN_PARAMS), rnd(W.nn_field_bytes(dims, 4) // 4)

    def apply(flags):
        o = torch.zeros_like(x)
        W.wd_nn_apply_ex(o, x, w, gauge, dims, flags)
        return o

    ref = [apply(f) for f in (0, W.WD_NN_BF16)]
    torch.cuda.synchronize()
    outs = []
    t = threading.Thread(target=lambda: outs.extend(apply((0, W.WD_NN_BF16)[k % 2]) for k in range(400)))
    t.start()
    while t.is_alive():
        W.wd_finalize()
    t.join()
    assert len(outs) == 400 and all(torch.equal(o, ref[k % 2]) for k, o in enumerate(outs))
