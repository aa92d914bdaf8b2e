"""The fixed-point FP64 hopping sum (csrc/wd_fix64.cuh): its arithmetic on the
host against long double, and on the GPU the forms of input that decide
between it and the FP64 chain."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from synth import fields

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_site_is_no_less_exact_than_the_fp64_chain(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "fix64_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", str(exe), os.path.join(HERE, "host", "fix64_check.cu")],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    last = r.stdout.strip().splitlines()[-1].split()
    assert last[0] == "OK" and float(last[2]) <= 1.0, r.stdout


def _inputs(form, dims):
    U, psi = fields.su3_links(dims, workers=1), fields.gaussian_spinor(dims)
    if form == "unit":
        U = fields.unit_links(dims)
    elif form == "point":         # one spin-colour of one odd site
        psi = np.zeros_like(psi)
        psi[1, 2, 1] = 1
    elif form == "sizes":         # neighbours of very different sizes
        psi = psi * 10.0 ** np.linspace(-12, 12, len(psi))[:, None, None]
    elif form == "large":
        psi = psi * 1e250
    elif form == "small":
        psi = psi * 1e-250
    elif form == "tiny":          # below the fixed-point range
        psi = psi * 1e-280
    elif form == "links 1.5":     # not SU(3): some sites' links are refused, others are not
        U = U.copy()
        U[:, ::3] *= 1.5
    elif form == "links 0.01":
        U = U.copy()
        U[1, ::2] *= 0.01
    return U, psi


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["gaussian", "unit", "point", "sizes", "large", "small", "tiny", "links 1.5",
                                  "links 0.01"])
@pytest.mark.parametrize("recon", [18, 12])
def test_fp64_hopping_over_the_forms_of_input(form, recon):
    import torch
    import paper_0810_5365_gb300 as W
    from tests._wdutil import pack_gauge, pack_spinor, unpack_spinor
    if recon == 12 and form.startswith("links"):
        pytest.skip("12-real storage is for SU(3) links")
    dims = (6, 4, 4, 6)
    U, psi = _inputs(form, dims)
    src = oracle.restrict(psi, dims, 1)
    g, i = pack_gauge(U, dims, W.WD_F64, recon), pack_spinor(src, dims, 1, W.WD_F64)
    x = oracle.restrict(fields.gaussian_spinor(dims, seed=5), dims, 0) * np.abs(src).max()
    xp = pack_spinor(x, dims, 0, W.WD_F64)
    for dagger in (0, 1):
        o = W.alloc_spinor(dims, 0, W.WD_F64)
        W.wd_dslash_ex(o, i, g, 0, dagger, 1.0, None, 0.0, None, 0.0, None, dims, W.WD_F64, recon)
        got, want = unpack_spinor(o, dims, 0, W.WD_F64), oracle.hop_block(0, src, U, dims, dagger=bool(dagger))
        # per site, relative to what its neighbours bring: eight hops, each term to 2^-53
        mag = oracle.hop_block(0, np.abs(src) + 0j, np.abs(U) + 0j, dims)
        scale = np.abs(mag).max(axis=(1, 2))
        full = np.maximum(scale, np.abs(want).max(axis=(1, 2)))
        ok = full > 0
        assert np.all(got[~ok] == 0)
        if form == "sizes":
            assert np.linalg.norm(got - want) <= 1e-13 * np.linalg.norm(want)
        else:
            err = np.abs(got - want).max(axis=(1, 2))
            assert np.all(err[ok] <= 1e-13 * np.maximum(full[ok], np.abs(src).max() * (form != "point")))
        # four right-hand sides give the single field's bits
        o4, i4 = torch.cat([o] * 4), torch.cat([i] * 4)
        W.wd_dslash_mrhs(o4, i4, g, 0, dagger, 1.0, None, 0.0, 4, None, dims, W.WD_F64, recon)
        assert all(torch.equal(o4[k * o.numel():(k + 1) * o.numel()], o) for k in range(4))
        W.wd_dslash_ex(o, i, g, 0, dagger, -0.5, xp, 0.25, None, 0.0, None, dims, W.WD_F64, recon)
        got = unpack_spinor(o, dims, 0, W.WD_F64)
        assert np.linalg.norm(got - (-0.5 * want + 0.25 * x)) <= 1e-13 * (np.linalg.norm(want) + np.linalg.norm(x))


@pytest.mark.gpu
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_fp64_hopping_keeps_non_finite_values(value):
    import paper_0810_5365_gb300 as W
    from tests._wdutil import pack_gauge, pack_spinor, unpack_spinor
    dims = (6, 4, 4, 6)
    U, psi = _inputs("gaussian", dims)
    src = oracle.restrict(psi, dims, 1)
    hit = np.zeros_like(src)
    hit[7] = src[7]
    touched = np.abs(oracle.hop_block(0, hit, U, dims)).max(axis=(1, 2)) > 0
    want = oracle.hop_block(0, src, U, dims)
    src[7, 1, 2] = value
    o = W.alloc_spinor(dims, 0, W.WD_F64)
    W.wd_dslash_ex(o, pack_spinor(src, dims, 1, W.WD_F64), pack_gauge(U, dims, W.WD_F64, 18), 0, 0, 1.0, None, 0.0,
                   None, 0.0, None, dims, W.WD_F64, 18)
    got = unpack_spinor(o, dims, 0, W.WD_F64)
    assert touched.sum() == 8 and not np.isfinite(got[touched]).all(axis=(1, 2)).any()
    assert np.abs(got[~touched] - want[~touched]).max() <= 1e-13 * np.abs(want).max()
