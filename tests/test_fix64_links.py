"""Links and neighbours at the edge of what the fixed-point FP64 hopping sum
(csrc/wd_fix64.cuh) takes: on the host, and on the GPU against the other
precisions and the oracle."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from synth import fields

HERE = os.path.dirname(os.path.abspath(__file__))


def run_host(tmp_path, name):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / name
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", str(exe), os.path.join(HERE, "host", name + ".cu")], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().splitlines()[-1].startswith("OK"), r.stdout + r.stderr
    return r.stdout


def test_links_that_do_not_fit_are_seen_beside_zero_neighbours(tmp_path):
    run_host(tmp_path, "fix64_links_check")


@pytest.mark.gpu
@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("recon", [18, 12])
def test_non_finite_links_beside_zero_neighbours(value, recon):
    """Where the FP32 kernel gives NaN (0 times the link's value) the FP64 one does too."""
    import paper_0810_5365_gb300 as W
    from tests._wdutil import pack_gauge, pack_spinor, unpack_spinor
    dims = (6, 4, 4, 6)
    U = fields.su3_links(dims, workers=1).copy()
    for k, (mu, site) in enumerate([(0, 10), (1, 100), (2, 201), (3, 333), (3, 570)]):
        U[mu, site, k % 2, k % 3] = value
    for src in ("zero", "point"):
        psi = np.zeros((np.prod(dims), 4, 3), dtype=complex)
        if src == "point":
            psi[1, 2, 1] = psi[101, 0, 0] = 1
        half = oracle.restrict(psi, dims, 1)
        bad = {}
        for prec in (W.WD_F64, W.WD_F32):
            o = W.alloc_spinor(dims, 0, prec)
            W.wd_dslash_ex(o, pack_spinor(half, dims, 1, prec), pack_gauge(U, dims, prec, recon), 0, 0, 1.0, None, 0.0,
                           None, 0.0, None, dims, prec, recon)
            bad[prec] = ~np.isfinite(unpack_spinor(o, dims, 0, prec)).all(axis=(1, 2))
        assert bad[W.WD_F32].any() and np.array_equal(bad[W.WD_F64], bad[W.WD_F32])
