"""Each synchronous network call has its own error flag: a wait that gives up in
another host thread is not reported by it, and it does not clear that thread's."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_error_flags_of_two_host_threads():
    import torch
    import paper_0810_5365_gb300 as W
    dims = (4, 4, 4, 4)
    g = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda n: torch.randn(n, device="cuda", generator=g)  # noqa: E731
    gauge = (0.3 * rnd(W.wd_gauge_bytes(dims, W.WD_F32, 12) // 4)).view(torch.uint8)
    w, x = 0.2 * rnd(9 * 8 * 4 * 2), rnd(W.nn_field_bytes(dims, 4) // 4)
    out = torch.zeros(W.nn_field_bytes(dims, 8) // 4, device="cuda")
    delta, grad = torch.zeros_like(out), torch.zeros(9 * 8 * 4 * 2, device="cuda")
    wn, outn = 0.2 * rnd(W.WD_NN_PARAMS), torch.zeros_like(x)
    calls = [lambda: W.wd_nn_layer(out, x, w, 4, 8, gauge, dims),
             lambda: W.wd_nn_wgrad(grad, x, delta, 4, 8, gauge, dims),
             lambda: W.wd_nn_apply(outn, x, wn, gauge, dims),
             lambda: W.wd_nn_apply_ex(outn, x, wn, gauge, dims, W.WD_NN_BF16)]
    for c in calls:
        c()
    W.wd_wait_selftest(10)
    torch.cuda.synchronize()
    stop, status, failed = threading.Event(), [], []

    def waits():  # bounded waits that run out (about 20 us each), one call after another
        while not stop.is_set():
            status.append(W.wd_wait_selftest(200))

    t = threading.Thread(target=waits)
    t.start()
    try:
        for k in range(2000):
            try:
                calls[k % 4]()
            except W.WdError as e:
                failed.append(e)
    finally:
        stop.set()
        t.join()
    assert not failed and len(status) > 100
    assert all(s == W.WD_ERR_TIMEOUT for s in status)
