"""FP16 hopping on lattices whose links exceed L2, where CTAs bring links into
L2 ahead of their use: the bits of the kernel that does not (staged
neighbours), of every CTA size, and of a lattice cut below the line."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _fields(dims, seed):
    import torch
    import paper_0810_5365_gb300 as W
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = W.wd_spinor_bytes(dims, 0, W.WD_F16)
    V = int(np.prod(dims))
    npad = (V // 2 + 31) // 32 * 32
    inp = torch.zeros(n, dtype=torch.uint8, device="cuda")
    h = torch.rand(npad * 24, device="cuda", generator=g) * 2 - 1
    inp[:npad * 48] = h.half().view(torch.uint8)
    inp[npad * 48:npad * 52] = torch.rand(npad, device="cuda", generator=g).add(0.5).view(torch.uint8)
    gauge = (torch.rand(W.wd_gauge_bytes(dims, W.WD_F16, 12) // 2, device="cuda", generator=g) - 0.5).half()
    return inp, gauge.view(torch.uint8), n


@pytest.mark.parametrize("dims", [(32, 32, 32, 46), (30, 26, 34, 70)])
def test_prefetching_launches_give_the_same_bits(dims):
    import torch
    import paper_0810_5365_gb300 as W
    assert W.wd_gauge_bytes(dims, W.WD_F16, 12) > torch.cuda.get_device_properties(0).L2_cache_size
    inp, gauge, n = _fields(dims, 3)

    def run(recon, parity, norm=None, block=0):
        out = torch.zeros(n, dtype=torch.uint8, device="cuda")
        W.wd_dslash_set_block(block)
        try:
            W.wd_dslash_ex(out, inp, gauge, parity, 1, -0.2, None, 0.0, None, 0.0, norm, dims, W.WD_F16, recon)
        finally:
            W.wd_dslash_set_block(0)
        return out

    for parity in (0, 1):
        ref = run(12, parity, block=64)
        assert torch.equal(ref, run(12, parity, block=128)) and torch.equal(ref, run(12, parity, block=256))
        norm = torch.zeros(1, dtype=torch.float64, device="cuda")
        assert torch.equal(ref, run(12, parity, norm))
        if (dims[0] * dims[1] // 2) % 32 == 0:
            assert torch.equal(ref, run(12 | W.WD_STAGE_NEIGHBOURS, parity))
        # temporal gauge: time links are not loaded, ahead of use neither
        tg = run(12 | W.WD_TEMPORAL_GAUGE, parity, block=64)
        assert torch.equal(tg, run(12 | W.WD_TEMPORAL_GAUGE, parity, block=256)) and not torch.equal(tg, ref)
