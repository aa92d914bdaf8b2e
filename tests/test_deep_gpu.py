"""FP32 and FP16 hopping on lattices whose CTAs all fit on the SMs at 128
registers, against the kernel of the larger ones: the same field repeated along
t, on both sides of the line between them, gives the same bits away from the
time boundary (where the antiperiodic sign differs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,copies", [((6, 10, 14, 26), 8), ((16, 16, 16, 38), 2), ((16, 16, 16, 20), 2)])
@pytest.mark.parametrize("prec,recon", [("f32", 12), ("f32", 18), ("f16", 12)])
@pytest.mark.parametrize("tg", [0, 1])
def test_both_sides_of_the_line_agree(dims, copies, prec, recon, tg):
    import torch
    import paper_0810_5365_gb300 as W
    prec = {"f32": W.WD_F32, "f16": W.WD_F16}[prec]
    gen = torch.Generator(device="cuda").manual_seed(11)
    V, T = int(np.prod(dims)), dims[3]
    U = torch.rand(4, V, 18, dtype=torch.float64, device="cuda", generator=gen) - 0.5
    psi, x = (torch.randn(V // 2, 24, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2))
    line = 4 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    assert V // 2 <= line < copies * V // 2

    def run(n, parity, dagger, epilogue, norm, block):
        d = dims[:3] + (n * T,)
        g = W.alloc_gauge(d, prec, recon)
        W.wd_pack_gauge(g, U.repeat(1, n, 1).reshape(-1), d, prec, recon)
        f = []
        for v, q in ((psi, 1 - parity), (x, parity)):
            f.append(W.alloc_spinor(d, q, prec))
            W.wd_pack_spinor(f[-1], v.repeat(n, 1).reshape(-1), d, q, prec)
        out = W.alloc_spinor(d, parity, prec)
        nrm = torch.zeros(1, dtype=torch.float64, device="cuda") if norm else None
        W.wd_dslash_set_block(block)
        try:
            W.wd_dslash_ex(out, f[0], g, parity, dagger, -0.3, f[1] if epilogue else None, 0.7, None, 0.0, nrm, d,
                           prec, recon | (W.WD_TEMPORAL_GAUGE if tg else 0))
        finally:
            W.wd_dslash_set_block(0)
        r = torch.empty(n * V // 2 * 24, dtype=torch.float64, device="cuda")
        W.wd_unpack_spinor(r, out, d, parity, prec)
        if norm:  # FP32 sums of a site and a CTA's 128 sites
            assert abs(nrm.item() - (r * r).sum().item()) <= 2e-6 * nrm.item()
        return r.view(n, T, -1)

    for parity, dagger, epilogue, norm, block in ((0, 0, 0, 0, 64), (1, 1, 0, 0, 128), (0, 1, 1, 0, 256),
                                                  (1, 0, 0, 1, 0), (0, 1, 1, 1, 0)):
        small, large = run(1, parity, dagger, epilogue, norm, block), run(copies, parity, dagger, epilogue, norm, block)
        for c in range(copies):
            assert torch.equal(small[0, 1:-1], large[c, 1:-1])
        assert torch.equal(small[0, 0], large[0, 0]) and torch.equal(small[0, -1], large[-1, -1])
