"""Small components beside large ones in the FP64 hopping: the fixed-point sum
(csrc/wd_fix64.cuh) gives each component the bits of the FP64 chain, on the host
against long double, and on the GPU against the oracle."""
import numpy as np
import pytest

import oracle
from synth import fields
from tests.test_fix64 import _inputs
from tests.test_fix64_links import run_host


def test_every_component_is_as_exact_as_the_chain(tmp_path):
    run_host(tmp_path, "fix64_small_check")


def _diagonal_links(dims, seed=11):
    """Diagonal SU(3) links: colours do not mix."""
    rng = np.random.default_rng(seed)
    V = int(np.prod(dims))
    p = rng.uniform(0, 2 * np.pi, (4, V, 3))
    p[..., 2] = -p[..., 0] - p[..., 1]
    U = np.zeros((4, V, 3, 3), dtype=complex)
    for c in range(3):
        U[..., c, c] = np.exp(1j * p[..., c])
    return U


def _hop(half, U, dims, recon, dagger):
    import paper_0810_5365_gb300 as W
    from tests._wdutil import pack_gauge, pack_spinor, unpack_spinor
    g, i, o = pack_gauge(U, dims, W.WD_F64, recon), pack_spinor(half, dims, 1, W.WD_F64), W.alloc_spinor(dims, 0, W.WD_F64)
    W.wd_dslash_ex(o, i, g, 0, dagger, 1.0, None, 0.0, None, 0.0, None, dims, W.WD_F64, recon)
    return unpack_spinor(o, dims, 0, W.WD_F64)


def _terms(half, U, dims):
    """Per even site: a bound for the sum of the moduli that make up a component, [Vh, 3] by colour."""
    full = oracle.embed(half, dims, 1)
    x = fields.coords(dims).T
    V, stride = int(np.prod(dims)), np.cumprod([1, *dims[:3]])
    size = 2 * np.abs(full).max(axis=1)  # two spins of the projection
    S = np.zeros((V, 3))
    for mu in range(4):
        n = np.arange(V) + stride[mu] * (((x[mu] + 1) % dims[mu]) - x[mu])
        S += np.einsum("vab,vb->va", np.abs(U[mu]), size[n])
        S[n] += np.einsum("vba,vb->va", np.abs(U[mu]), size)
    return oracle.restrict(S[:, None, :].repeat(4, 1) + 0j, dims, 0)[:, 0].real


# roundings of a component: projection 1, product 6, sum 8, each 2^-53 of its
# terms; times sqrt(2) for the modulus, times two for the oracle's own, and as
# many again for the rebuilt row of 12-real links
TOL = {18: 2 * 1.42 * 15 * 2.0 ** -53, 12: 4 * 1.42 * 15 * 2.0 ** -53}


@pytest.mark.gpu
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dims", [(6, 4, 4, 6), (8, 2, 6, 4), (10, 6, 2, 14)])
def test_small_colours_keep_their_bits(dims, recon):
    for U in (_diagonal_links(dims), fields.unit_links(dims)):
        for k in (0, 1, 3, 4, 5, 6, 8, 20, 45, 60, 200):
            psi = fields.gaussian_spinor(dims, seed=k + 1)
            psi[..., 1] *= 2.0 ** -k
            half = oracle.restrict(psi, dims, 1)
            for dagger in (0, 1):
                got, want = _hop(half, U, dims, recon, dagger), oracle.hop_block(0, half, U, dims, dagger=bool(dagger))
                err, S = np.abs(got - want), _terms(half, U, dims)
                assert np.all(err <= TOL[recon] * S[:, None, :]), (k, (err / S[:, None, :]).max(axis=(0, 1)))


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["gaussian", "unit", "point", "sizes", "large", "small", "tiny", "links 1.5",
                                  "links 0.01"])
@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("dims", [(6, 4, 4, 6), (4, 6, 10, 2)])
def test_each_component_to_its_own_terms(form, recon, dims):
    if recon == 12 and form.startswith("links"):
        pytest.skip("12-real storage is for SU(3) links")
    U, psi = _inputs(form, dims)
    half = oracle.restrict(psi, dims, 1)
    scale = np.abs(half).max()  # (the oracle's sums of 1e250 and 1e-280 stay in range)
    for dagger in (0, 1):
        got, want = _hop(half, U, dims, recon, dagger), oracle.hop_block(0, half, U, dims, dagger=bool(dagger))
        S = _terms(half / scale, U, dims) * scale
        assert np.all(np.abs(got - want) <= TOL[recon] * S[:, None, :])
