"""FP64 hopping with 18-real links that are not of order one: in fixed point too
(csrc/wd_fix64.cuh), on the host against long double and on the GPU against the
oracle."""
import numpy as np
import pytest

import oracle
from synth import fields
from tests.test_fix64_links import run_host
from tests.test_fix64_small import TOL, _hop, _terms


def test_sized_links_are_taken_and_no_less_exact(tmp_path):
    run_host(tmp_path, "fix64_sized_check")


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["tadpole", "some", "spread", "anisotropic", "large", "tiny", "vanishing"])
@pytest.mark.parametrize("dims", [(6, 4, 4, 6), (4, 2, 10, 4)])
def test_links_of_any_size(form, dims):
    rng = np.random.default_rng(5)
    U = fields.su3_links(dims, workers=1).copy()
    V = U.shape[1]
    if form == "tadpole":
        U *= 1.15
    elif form == "some":
        U[:, rng.random(V) < 0.05] *= 1.3
    elif form == "spread":
        U *= 2.0 ** rng.uniform(-6, 6, (4, V, 1, 1))
    elif form == "anisotropic":
        U[:3] *= 0.05
        U[3] *= 5
    elif form == "large":
        U *= 1e25     # beyond the fixed-point range
    elif form == "tiny":
        U *= 1e-25
    else:
        U[:, rng.random(V) < 0.5] = 0
    half = oracle.restrict(fields.gaussian_spinor(dims), dims, 1)
    for dagger in (0, 1):
        got, want = _hop(half, U, dims, 18, dagger), oracle.hop_block(0, half, U, dims, dagger=bool(dagger))
        assert np.all(np.abs(got - want) <= TOL[18] * _terms(half, U, dims)[:, None, :])
