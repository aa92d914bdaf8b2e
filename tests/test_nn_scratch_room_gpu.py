"""The network calls' kept scratch gives way to an allocation that finds no room."""
import pytest

pytestmark = pytest.mark.gpu


def test_kept_scratch_gives_way():
    import torch
    import paper_0810_5365_gb300 as W
    dims = (24, 24, 24, 32)
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda n: torch.randn(n, device="cuda", generator=g)  # noqa: E731
    gauge = (0.3 * rnd(W.wd_gauge_bytes(dims, W.WD_F32, 12) // 4)).view(torch.uint8)
    w, x = 0.2 * rnd(W.WD_NN_PARAMS), rnd(W.nn_field_bytes(dims, 4) // 4)
    out, ref = torch.zeros_like(x), torch.zeros_like(x)
    kept = 2 * W.nn_field_bytes(dims, 8)  # two fields of eight channels
    W.wd_finalize()
    W.wd_nn_apply(ref, x, w, gauge, dims)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    # 412 GB of scratch for 2^30 sites: refused before anything is read
    with pytest.raises(W.WdError):
        W.wd_nn_apply(out, x, w, gauge, (128, 128, 128, 512))
    assert torch.cuda.mem_get_info()[0] - before >= kept - (4 << 20)
    W.wd_nn_apply(out, x, w, gauge, dims)
    assert torch.equal(out, ref)
    W.wd_finalize()
