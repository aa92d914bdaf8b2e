"""The kept scratch of the synchronous network calls: growing, shrinking,
another stream, after wd_finalize, and above the size that is kept."""
import pytest

pytestmark = pytest.mark.gpu


def test_network_calls_share_one_scratch():
    import torch
    import paper_0810_5365_gb300 as W

    def case(dims, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        rnd = lambda n: torch.randn(n, device="cuda", generator=g)  # noqa: E731
        gauge = (0.3 * rnd(W.wd_gauge_bytes(dims, W.WD_F32, 12) // 4)).view(torch.uint8)
        return dims, gauge, 0.2 * rnd(W.WD_NN_PARAMS), rnd(W.nn_field_bytes(dims, 4) // 4), rnd(W.nn_field_bytes(dims, 8) // 4)

    def run(c):
        dims, gauge, w, x, y = c
        outs = []
        for flags in (0, W.WD_NN_BF16, W.WD_NN_EVEN, W.WD_NN_BF16 | W.WD_NN_EVEN):
            o = torch.zeros_like(x)
            W.wd_nn_apply_ex(o, x, w, gauge, dims, flags)
            outs.append(o)
        o = torch.zeros_like(x)
        W.wd_nn_apply(o, x, w, gauge, dims)
        grad = torch.zeros(9 * 8 * 8 * 2, device="cuda")
        W.wd_nn_wgrad(grad, y, y, 8, 8, gauge, dims)
        return outs + [o, grad]

    # 44^3 x 32: 2 x 654 MB of FP32 activations, more than is kept
    cases = [case((4, 6, 4, 8), 1), case((8, 8, 8, 10), 2), case((44, 44, 44, 32), 3)]
    W.wd_finalize()
    ref = []
    for c in cases:            # each alone, on fresh scratch
        ref.append(run(c))
        W.wd_finalize()
    side = torch.cuda.Stream()
    try:
        for k in (0, 1, 2, 0, 2, 1):
            W.wd_set_stream(side if k == 1 else None)
            side.wait_stream(torch.cuda.current_stream())
            got = run(cases[k])
            side.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, ref[k])), k
    finally:
        W.wd_set_stream(None)
        W.wd_finalize()


def test_two_host_threads_do_not_share_it():
    import threading
    import torch
    import paper_0810_5365_gb300 as W
    dims = (8, 8, 8, 8)
    g = torch.Generator(device="cuda").manual_seed(7)
    rnd = lambda n: torch.randn(n, device="cuda", generator=g)  # noqa: E731
    gauge = (0.3 * rnd(W.wd_gauge_bytes(dims, W.WD_F32, 12) // 4)).view(torch.uint8)
    work = [(0.2 * rnd(W.WD_NN_PARAMS), rnd(W.nn_field_bytes(dims, 4) // 4)) for _ in range(2)]

    def apply(w, x):
        o = torch.zeros_like(x)
        W.wd_nn_apply_ex(o, x, w, gauge, dims, W.WD_NN_BF16)
        return o

    ref = [apply(*c) for c in work]
    outs = [[], []]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=lambda k=k: outs[k].extend(apply(*work[k]) for _ in range(100))) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in (0, 1):
        assert len(outs[k]) == 100 and all(torch.equal(o, ref[k]) for o in outs[k])
