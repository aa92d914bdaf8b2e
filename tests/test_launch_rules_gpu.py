"""Launch rules of the solvers: overlapped and plain graph edges on both sides
of the line between them, and batches of one problem (a parameter that holds
one) against the same problem twice (the full table)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(dims, nrhs, seed):
    import torch
    V = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(seed)
    U = torch.zeros(4, V, 3, 3, dtype=torch.complex128, device="cuda")
    # diagonal SU(3) links with random phases
    ph = 0.4 * torch.randn(4, V, 2, dtype=torch.float64, device="cuda", generator=g)
    ph = torch.cat([ph, -ph.sum(-1, keepdim=True)], -1)
    U[..., range(3), range(3)] = torch.exp(1j * ph)
    b = torch.randn(nrhs, V, 12, dtype=torch.complex128, device="cuda", generator=g)
    return torch.view_as_real(U).reshape(-1), torch.view_as_real(b).reshape(-1)


@pytest.mark.parametrize("dims,prec", [((4, 4, 4, 6), "f16"), ((24, 24, 24, 16), "f16"), ((16, 16, 16, 48), "f32"),
                                       ((24, 24, 24, 18), "f32")])
@pytest.mark.parametrize("solver", [0, 1])
def test_overlapped_and_plain_iterations_agree(dims, prec, solver):
    import torch
    import paper_0810_5365_gb300 as W
    U, b = _problem(dims, 1, 3)
    p = W.wd_solve_params_default()
    p.inner_prec, p.solver = (W.WD_F16 if prec == "f16" else W.WD_F32), solver
    out = []
    for overlap in (1, 0):
        W.wd_set_launch_overlap(overlap)
        W.wd_finalize()
        try:
            x = torch.zeros_like(b)
            info = W.wd_solve_ex(x, b, U, 0.1, dims, p)
        finally:
            W.wd_set_launch_overlap(1)
        assert info["true_residual"] <= 1e-10
        out.append(x)
    assert torch.equal(*out)


@pytest.mark.parametrize("prec", ["f16", "f32", "f64"])
def test_one_problem_and_the_same_twice(prec):
    import torch
    import paper_0810_5365_gb300 as W
    dims, nrhs = (4, 6, 4, 10), 3
    U, b = _problem(dims, nrhs, 5)
    p = W.wd_solve_params_default()
    p.inner_prec = {"f16": W.WD_F16, "f32": W.WD_F32, "f64": W.WD_F64}[prec]
    p.inner_recon = 12 if prec != "f64" else 18
    xs = [torch.zeros_like(b) for _ in range(3)]
    one = dict(dims=dims, kappa=0.11, nrhs=nrhs, gauge=U, b=b)
    W.wd_solve_batch([dict(one, x=xs[0])], p)
    W.wd_solve_batch([dict(one, x=xs[1]), dict(one, x=xs[2])], p)
    assert torch.equal(xs[0], xs[1]) and torch.equal(xs[1], xs[2])
