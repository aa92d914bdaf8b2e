"""Fused norms of lattices with more than 12 x 256 block partials (the second
trip of the partial sums), against the sum over the output in FP64."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(32, 32, 32, 24), (32, 32, 32, 26), (40, 32, 32, 38)])  # 3072, 3328, 6080 CTAs
@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_fused_norms_of_many_blocks(dims, prec):
    import torch
    import paper_0810_5365_gb300 as W
    p = {"f64": W.WD_F64, "f32": W.WD_F32, "f16": W.WD_F16}[prec]
    V = dims[0] * dims[1] * dims[2] * dims[3]
    g = torch.Generator(device="cuda").manual_seed(9)
    # any links serve (18 reals; FP16 holds 12); sizes vary over the lattice, so that a lost partial shows
    links = 0.3 * torch.randn(4 * V * 18, dtype=torch.float64, device="cuda", generator=g)
    recon = 12 if prec == "f16" else 18
    gauge = W.alloc_gauge(dims, p, recon)
    W.wd_pack_gauge(gauge, links, dims, p, recon)
    del links
    fields, outs = [], []
    for _ in range(2):
        c = torch.randn(V // 2 * 24, dtype=torch.float64, device="cuda", generator=g)
        c *= (1 + torch.arange(V // 2, device="cuda") / V).repeat_interleave(24)
        f = W.alloc_spinor(dims, W.WD_ODD, p)
        W.wd_pack_spinor(f, c, dims, W.WD_ODD, p)
        fields.append(f)
    # a block sums 128 sites of 24 terms in the working precision: 24 in a row, then pairs
    tol = (24 + 8) * 2.0 ** (-53 if prec == "f64" else -24) + 1e-14

    def norm_of(o):
        back = torch.empty(V // 2 * 24, dtype=torch.float64, device="cuda")
        W.wd_unpack_spinor(back, o, dims, W.WD_EVEN, p)
        return float((back * back).sum())

    for f in fields:
        o, n = W.alloc_spinor(dims, W.WD_EVEN, p), torch.zeros(1, dtype=torch.float64, device="cuda")
        W.wd_dslash_ex(o, f, gauge, W.WD_EVEN, 0, 0.7, None, 0.0, None, 0.0, n, dims, p, recon)
        outs.append(norm_of(o))
        assert abs(float(n) - outs[-1]) <= tol * outs[-1]
    both, o2 = torch.cat(fields), torch.cat([W.alloc_spinor(dims, W.WD_EVEN, p)] * 2)
    n2 = torch.zeros(2, dtype=torch.float64, device="cuda")
    W.wd_dslash_mrhs(o2, both, gauge, W.WD_EVEN, 0, 0.7, None, 0.0, 2, n2, dims, p, recon)
    assert all(abs(float(a) - b) <= tol * b for a, b in zip(n2, outs))
