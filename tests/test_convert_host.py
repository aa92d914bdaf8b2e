"""The integer float <-> double conversions of csrc/wd_common.cuh, compiled as
host code and compared bit for bit with the language's own."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_conversions_match_the_language(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "convert_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", str(exe), os.path.join(HERE, "host", "convert_check.cu")],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout + r.stderr


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 6, 2, 10), (6, 4, 6, 10), (14, 10, 6, 8)])
def test_pack_and_unpack_layouts(dims):
    """Packed words against the documented layout, half and full, every format;
    32-site groups that are part full, and rows that switch parity inside one."""
    import numpy as np
    import torch
    import paper_0810_5365_gb300 as W
    from synth import fields
    V = int(np.prod(dims))
    npad = (V // 2 + 31) // 32 * 32
    U, psi = fields.su3_links(dims, workers=1), fields.gaussian_spinor(dims)
    psi[0] = 0
    psi[V - 1, 1, 1] = 1e-42            # a denormal float
    src = torch.from_numpy(psi.view(np.float64).copy()).cuda()
    half = [fields.to_half(psi, dims, p) for p in (0, 1)]

    def words(z, per, prec):            # [sites][12] complex -> blocks of 32 sites, groups of `per` reals
        r = np.zeros((npad, z.shape[1] * 2))
        r[:len(z)] = z.reshape(len(z), -1).view(np.float64)
        return r.reshape(npad // 32, 32, -1, per).transpose(0, 2, 1, 3).reshape(-1).astype(prec)

    for prec, dt, per, nb in ((W.WD_F64, np.float64, 2, 192), (W.WD_F32, np.float32, 4, 96)):
        full = torch.zeros(W.wd_spinor_bytes(dims, W.WD_FULL, prec), dtype=torch.uint8, device="cuda")
        W.wd_pack_spinor(full, src, dims, W.WD_FULL, prec)
        rows = full.cpu().numpy().reshape(2, -1)[:, :npad * nb].copy().view(dt)
        for p in (0, 1):
            want = words(half[p].reshape(-1, 12), per, dt)
            assert np.array_equal(rows[p], want)
            one = torch.zeros(W.wd_spinor_bytes(dims, p, prec), dtype=torch.uint8, device="cuda")
            W.wd_pack_spinor(one, torch.from_numpy(half[p].reshape(-1).view(np.float64).copy()).cuda(), dims, p, prec)
            assert np.array_equal(one.cpu().numpy()[:npad * nb].view(dt), want)
            back = torch.zeros(V // 2 * 24, dtype=torch.float64, device="cuda")
            W.wd_unpack_spinor(back, one, dims, p, prec)
            assert np.array_equal(back.cpu().numpy(), half[p].reshape(-1).view(np.float64).astype(dt).astype(np.float64))
        back = torch.zeros(V * 24, dtype=torch.float64, device="cuda")
        W.wd_unpack_spinor(back, full, dims, W.WD_FULL, prec)
        assert np.array_equal(back.cpu().numpy(), psi.reshape(-1).view(np.float64).astype(dt).astype(np.float64))
        for recon in (12, 18):
            g = torch.zeros(W.wd_gauge_bytes(dims, prec, recon), dtype=torch.uint8, device="cuda")
            W.wd_pack_gauge(g, torch.from_numpy(U.reshape(-1).view(np.float64).copy()).cuda(), dims, prec, recon)
            got = g.cpu().numpy()[:8 * npad * recon * np.dtype(dt).itemsize].view(dt)
            gper = 2 if prec == W.WD_F64 or recon == 18 else 4
            want = np.concatenate([words(fields.to_half(U[mu], dims, p).reshape(-1, 9)[:, :recon // 2], gper, dt)
                                   for mu in range(4) for p in (0, 1)])
            assert np.array_equal(got, want)
    # FP16: the largest component of each site is its scale
    f16 = torch.zeros(W.wd_spinor_bytes(dims, 0, W.WD_F16), dtype=torch.uint8, device="cuda")
    W.wd_pack_spinor(f16, torch.from_numpy(half[0].reshape(-1).view(np.float64).copy()).cuda(), dims, 0, W.WD_F16)
    raw = f16.cpu().numpy()
    r = np.zeros((npad, 24), np.float32)
    r[:V // 2] = half[0].reshape(-1, 12).view(np.float64).astype(np.float32)
    sc = np.abs(r).max(axis=1)
    assert np.array_equal(raw[npad * 48:npad * 52].view(np.float32), sc)
    h = raw[:npad * 48].copy().view(np.float16).reshape(npad // 32, 3, 32, 8).transpose(0, 2, 1, 3).reshape(npad, 24)
    assert np.abs(h.astype(np.float64) * sc[:, None] - r).max() <= 2.0 ** -11 * sc.max() * 1.001
