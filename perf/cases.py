"""The work that users of libwd have it do, through the Python binding of its C ABI.

A case is one kind of call on one lattice:

  dslash  wd_dslash / wd_dslash_dag: the hopping term on one parity, or D on the full lattice
  mhat    wd_mhat: the even-odd operator 1 - kappa^2 H_eo H_oe or its adjoint
  mrhs    wd_dslash_mrhs with its fused norms: one gauge field, many right-hand sides
  blas    wd_norm2, wd_cdot, wd_axpby: what a user's own Krylov loop does between operators
  load    wd_pack_gauge, wd_pack_spinor, wd_unpack_spinor: a configuration and a source in, a field out
  layer   wd_nn_layer and wd_nn_wgrad: a layer of the network forward, and its weight gradient
  net     wd_nn_apply_ex: the learned preconditioner as the flexible CG applies it
  solve   wd_solve_ex: one mixed-precision solve
  batch   wd_solve_batch: several right-hand sides of one gauge field

Links are reunitarised SU(3) matrices near the identity (mean link about 0.94), spinors complex
Gaussian or point sources, as in the tests and the benchmark of this repository.
"""
import math

import torch

import paper_0810_5365_gb300 as W

PREC = {"f64": W.WD_F64, "f32": W.WD_F32, "f16": W.WD_F16}
PARITY = {"even": W.WD_EVEN, "odd": W.WD_ODD, "full": W.WD_FULL}
CD = torch.complex128


def listed():
    return [
        # the smallest lattice of the batched configuration: launches and latency are all there is
        dict(name="dslash f32 8^4", kind="dslash", dims="8x8x8x8", prec="f32", parity="even", dagger=0),
        # a ragged mid-size lattice (no extent a power of two, a last tile that is part full), FP16,
        # the adjoint: half of a normal-equations step
        dict(name="mhat f16 dag ragged", kind="mhat", dims="14x10x18x22", prec="f16", recon=12, dagger=1),
        # the headline throughput lattice in the two bulk precisions
        dict(name="dslash f32 32^3x64", kind="dslash", dims="32x32x32x64", prec="f32", parity="even", dagger=0),
        dict(name="dslash f16 32^3x64", kind="dslash", dims="32x32x32x64", prec="f16", parity="odd", dagger=0),
        # the FP64 operator on the full lattice: residuals, and plain FP64 work
        dict(name="D f64 24^3x48", kind="dslash", dims="24x24x24x48", prec="f64", parity="full", dagger=0),
        # twelve spin-colour sources of one configuration, as a batched solver applies the operator
        dict(name="mrhs f32 12 24^3x48", kind="mrhs", dims="24x24x24x48", prec="f32", recon=12, nrhs=12, dagger=0),
        # vector work of a user's own Krylov loop
        dict(name="blas f32 24^3x48", kind="blas", dims="24x24x24x48", prec="f32"),
        # a configuration and a source brought in, a solution read out
        dict(name="load f32 24^3x48", kind="load", dims="24x24x24x48", prec="f32", recon=12),
        # training: the middle layer of the network forward, and its weight gradient
        dict(name="layer 8-8 16^3x32", kind="layer", dims="16x16x16x32", cin=8, cout=8),
        # inference: the preconditioner N_e of the flexible CG
        dict(name="net bf16 even 32^3x64", kind="net", dims="32x32x32x64", bf16=1, even=1),
        # one mixed-precision solve, FP16 inner iterations
        dict(name="solve f16 24^3x48", kind="solve", dims="24x24x24x48", prec="f16", kappa=0.137, solver="cg"),
        # the twelve point sources of a propagator, solved together
        dict(name="batch f32 12 24^3x48", kind="batch", dims="24x24x24x48", prec="f32", kappa=0.136, nrhs=12,
             source="point"),
    ]


# The relative residual that a solve asks for: tight enough that two roundings of one solve agree to
# about 1e-11 (at the default 1e-10 they agree to about 1e-9 where D is near critical).
TOL = 1e-12


def _draw_dims(rng, lo, hi):
    """Even extents, volumes spread over the logarithm between lo and hi, t the longest more often than not."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = (v / rng.choice([1, 2, 2])) ** 0.25
        d = [max(4, 2 * round(side * math.exp(rng.uniform(-0.3, 0.3)) / 2)) for _ in range(3)]
        d.append(max(4, 2 * round(v / (d[0] * d[1] * d[2]) / 2)))
        n = d[0] * d[1] * d[2] * d[3]
        if lo <= n <= hi and d[3] <= 128:
            return "x".join(map(str, d))


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "mhat", "mrhs", "blas", "load", "layer", "net", "solve", "batch"])
    small, large = 8 ** 4, 32 ** 3 * 64
    if kind == "dslash":
        prec = rng.choice(["f64", "f32", "f16"])
        return dict(kind=kind, dims=_draw_dims(rng, small, large // 2 if prec == "f64" else large), prec=prec,
                    parity=rng.choice(["even", "odd", "full"]), dagger=rng.randrange(2))
    if kind == "mhat":
        prec = rng.choice(["f64", "f32", "f16"])
        return dict(kind=kind, dims=_draw_dims(rng, small, large // 2), prec=prec,
                    recon=12 if prec == "f16" else rng.choice([12, 18]), dagger=rng.randrange(2))
    if kind == "mrhs":
        prec = rng.choice(["f32", "f16"])
        return dict(kind=kind, dims=_draw_dims(rng, small, 24 ** 3 * 48), prec=prec,
                    recon=12 if prec == "f16" else rng.choice([12, 18]), nrhs=rng.randint(2, 12),
                    dagger=rng.randrange(2))
    if kind in ("blas", "load"):
        c = dict(kind=kind, dims=_draw_dims(rng, small, 24 ** 3 * 48), prec=rng.choice(["f64", "f32", "f16"]))
        if kind == "load":
            c["recon"] = 12 if c["prec"] == "f16" else rng.choice([12, 18])
        return c
    if kind == "layer":
        cin, cout = rng.choice([(4, 8), (8, 8), (8, 4)])
        return dict(kind=kind, dims=_draw_dims(rng, small, 16 ** 3 * 32), cin=cin, cout=cout)
    if kind == "net":
        return dict(kind=kind, dims=_draw_dims(rng, small, large), bf16=rng.randrange(2), even=rng.randrange(2))
    if kind == "solve":
        solver = rng.choice(["cg", "cg", "bicgstab"])
        return dict(kind=kind, dims=_draw_dims(rng, small, 16 ** 3 * 32), prec=rng.choice(["f32", "f16"]),
                    kappa=round(rng.uniform(0.11, 0.12 if solver == "bicgstab" else 0.137), 4), solver=solver)
    return dict(kind=kind, dims=_draw_dims(rng, small, 16 ** 3 * 32), prec=rng.choice(["f32", "f16"]),
                kappa=round(rng.uniform(0.11, 0.136), 4), nrhs=rng.randint(2, 12),
                source=rng.choice(["point", "gaussian"]))


# ---------------------------------------------------------------------------
# inputs: canonical FP64 fields, made on the GPU from the seed
# ---------------------------------------------------------------------------

def _dims(case):
    return tuple(int(v) for v in case["dims"].split("x"))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 64 + stream)


def _mul(a, b):
    """a b for [n, 3, 3] matrices."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _links(dims, seed, eps=0.3):
    """complex128 [4, V, 3, 3]: exp(i eps H), H Gaussian traceless Hermitian, reunitarised into SU(3)."""
    V, g = _volume(dims), _gen(seed, 1)
    U = torch.empty(4, V, 3, 3, dtype=CD, device="cuda")
    for mu in range(4):
        a = torch.randn(V, 3, 3, dtype=CD, device="cuda", generator=g)
        a = 0.5j * eps * (a + a.mH)
        a = a - a.diagonal(dim1=1, dim2=2).mean(-1)[:, None, None] * torch.eye(3, dtype=CD, device="cuda")
        a2 = _mul(a, a)
        u = torch.eye(3, dtype=CD, device="cuda") + a + a2 / 2 + _mul(a, a2) / 6
        r0 = u[:, 0] / u[:, 0].norm(dim=1, keepdim=True)
        r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(1, keepdim=True) * r0
        r1 = r1 / r1.norm(dim=1, keepdim=True)
        U[mu] = torch.stack([r0, r1, torch.linalg.cross(r0, r1, dim=1).conj()], 1)
    return U


def _gaussian(shape, seed, stream):
    """Complex normals, real and imaginary parts N(0, 1/2)."""
    return torch.randn(*shape, dtype=CD, device="cuda", generator=_gen(seed, stream))


def _parity_sites(dims, parity):
    x = [torch.arange(n, device="cuda") for n in dims]
    par = (x[3][:, None, None, None] + x[2][None, :, None, None] + x[1][None, None, :, None] + x[0]) & 1
    return torch.nonzero(par.reshape(-1) == parity).reshape(-1)


def _sources(case, seed):
    """Right-hand sides [nrhs, V, 4, 3] of a solve."""
    V, n = _volume(_dims(case)), case.get("nrhs", 1)
    if case.get("source") == "point":
        b = torch.zeros(n, V, 12, dtype=CD, device="cuda")
        for r in range(n):
            b[r, 0, r % 12] = 1
        return b.reshape(n, V, 4, 3)
    return _gaussian((n, V, 4, 3), seed, 3)


def _gamma():
    """Chiral basis: gamma_k = [[0, -i s_k], [i s_k, 0]], gamma_t = [[0, 1], [1, 0]]."""
    s = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=CD)
    g = torch.zeros(4, 4, 4, dtype=CD)
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * s[k], 1j * s[k]
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2)
    return g


NET = [(4, 8, 1), (8, 8, 1j), (8, 4, -1j)]


def _layer_weights(cin, cout, c, kappa=0.137):
    """[9, cout, cin]: 1 + c kappa H on the first four channels."""
    w, g = torch.zeros(9, cout, cin, dtype=CD), _gamma()
    n = min(cin, cout)
    w[0, :n, :n] = torch.eye(n)
    for mu in range(4):
        w[1 + 2 * mu, :4, :4] = c * kappa * (torch.eye(4) - g[mu])
        w[2 + 2 * mu, :4, :4] = c * kappa * (torch.eye(4) + g[mu])
    return w


def _weights(layers, seed):
    """The weights of the layers as training leaves them: the hopping series, perturbed."""
    return [_layer_weights(i, o, c).cuda() + 0.01 * _gaussian((9, o, i), seed, 10 + k)
            for k, (i, o, c) in enumerate(layers)]


def _flat(ws):
    return torch.cat([torch.view_as_real(w).reshape(-1) for w in ws]).float().contiguous()


def _real(z):
    return torch.view_as_real(z.contiguous()).reshape(-1)


# ---------------------------------------------------------------------------
# packed buffers
# ---------------------------------------------------------------------------

def _buffer(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")  # (padding sites stay zero)


def _packed(z, dims, parity, prec):
    buf = _buffer(W.wd_spinor_bytes(dims, parity, prec))
    W.wd_pack_spinor(buf, _real(z), dims, parity, prec)
    return buf


def _packed_gauge(U, dims, prec, recon):
    buf = _buffer(W.wd_gauge_bytes(dims, prec, recon))
    W.wd_pack_gauge(buf, _real(U), dims, prec, recon)
    return buf


def _padded(dims):
    return (_volume(dims) // 2 + 31) // 32 * 32


def _values(buf, dims, prec, halves=1):
    """The numbers that packed half fields hold, as views of their buffer."""
    n, per = _padded(dims), {W.WD_F64: 192, W.WD_F32: 96, W.WD_F16: 52}[prec]
    rows = buf.view(halves, -1)[:, :n * per]
    if prec == W.WD_F64:
        return {"v": rows.view(torch.float64)}
    if prec == W.WD_F32:
        return {"v": rows.view(torch.float32)}
    return {"h": rows[:, :n * 48].view(torch.float16), "s": rows[:, n * 48:].view(torch.float32)}


def _layout(z, dims, prec):
    """_values() of half fields z [halves, Vh, 12], from 64 bits."""
    m, n = z.shape[0], _padded(dims)
    z = torch.cat([z, torch.zeros(m, n - z.shape[1], 12, dtype=CD, device=z.device)], 1)
    r = torch.view_as_real(z)
    if prec == W.WD_F16:
        s = r.abs().amax(dim=(2, 3))
        r = r / torch.where(s > 0, s, torch.ones_like(s))[:, :, None, None]
    k = {W.WD_F64: 12, W.WD_F32: 6, W.WD_F16: 3}[prec]
    v = r.reshape(m, n // 32, 32, k, 24 // k).permute(0, 1, 3, 2, 4).reshape(m, -1)
    return {"h": v, "s": s} if prec == W.WD_F16 else {"v": v}


def _nn_pack(z, dims):
    """A field [V, C, 3] in the packed FP32 full layout of C channels (here in 64 bits)."""
    C, n = z.shape[1], _padded(dims)
    half = W.nn_field_bytes(dims, C) // 8
    out = torch.zeros(2, half, dtype=torch.float64, device="cuda")
    for p in (0, 1):
        h = z[_parity_sites(dims, p)].reshape(-1, 3 * C)
        h = torch.cat([h, torch.zeros(n - h.shape[0], 3 * C, dtype=CD, device="cuda")])
        v = torch.view_as_real(h).reshape(n // 32, 32, 3 * C // 2, 4).permute(0, 2, 1, 3).reshape(-1)
        out[p, :v.numel()] = v
    return out.reshape(-1)


# ---------------------------------------------------------------------------
# prepare, run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    V, prec = _volume(dims), PREC.get(case.get("prec", "f32"))
    s = dict(case=case, dims=dims, prec=prec, kind=kind)
    if kind == "dslash":
        par = PARITY[case["parity"]]
        src = W.WD_FULL if par == W.WD_FULL else 1 - par
        s.update(parity=par, gauge=_packed_gauge(_links(dims, seed), dims, prec, 12),
                 inp=_packed(_gaussian((V if src == W.WD_FULL else V // 2, 12), seed, 2), dims, src, prec),
                 out=_buffer(W.wd_spinor_bytes(dims, par, prec)))
    elif kind == "mhat":
        n = W.wd_spinor_bytes(dims, W.WD_EVEN, prec)
        s.update(gauge=_packed_gauge(_links(dims, seed), dims, prec, case["recon"]),
                 inp=_packed(_gaussian((V // 2, 12), seed, 2), dims, W.WD_EVEN, prec), out=_buffer(n), tmp=_buffer(n))
    elif kind == "mrhs":
        n, nr = W.wd_spinor_bytes(dims, W.WD_EVEN, prec), case["nrhs"]
        src, x = _gaussian((nr, V // 2, 12), seed, 2), _gaussian((nr, V // 2, 12), seed, 4)
        s.update(gauge=_packed_gauge(_links(dims, seed), dims, prec, case["recon"]),
                 inp=torch.cat([_packed(z, dims, W.WD_ODD, prec) for z in src]),
                 x=torch.cat([_packed(z, dims, W.WD_EVEN, prec) for z in x]), out=_buffer(n * nr),
                 norm=torch.zeros(nr, dtype=torch.float64, device="cuda"))
    elif kind == "blas":
        x, y = _gaussian((2, V // 2, 12), seed, 2)
        s.update(x=_packed(x, dims, W.WD_EVEN, prec), y=_packed(y, dims, W.WD_EVEN, prec),
                 dots=torch.zeros(4, dtype=torch.float64, device="cuda"))
    elif kind == "load":
        s.update(U=_real(_links(dims, seed)), psi=_real(_gaussian((V, 12), seed, 2)),
                 gauge=_buffer(W.wd_gauge_bytes(dims, prec, case["recon"])),
                 spinor=_buffer(W.wd_spinor_bytes(dims, W.WD_FULL, prec)),
                 back=torch.zeros(V * 24, dtype=torch.float64, device="cuda"))
    elif kind == "layer":
        ci, co = case["cin"], case["cout"]
        c = next(c for i, o, c in NET if (i, o) == (ci, co))
        s.update(gauge=_packed_gauge(_links(dims, seed), dims, W.WD_F32, 12), w=_flat(_weights([(ci, co, c)], seed)),
                 inp=_nn_pack(_gaussian((V, ci, 3), seed, 2), dims).float(),
                 delta=_nn_pack(_gaussian((V, co, 3), seed, 4), dims).float(),
                 out=torch.zeros(W.nn_field_bytes(dims, co) // 4, dtype=torch.float32, device="cuda"),
                 grad=torch.zeros(9 * co * ci * 2, dtype=torch.float32, device="cuda"))
    elif kind == "net":
        s.update(gauge=_packed_gauge(_links(dims, seed), dims, W.WD_F32, 12), w=_flat(_weights(NET, seed)),
                 inp=_nn_pack(_gaussian((V, 4, 3), seed, 2), dims).float(),
                 out=torch.zeros(W.nn_field_bytes(dims, 4) // 4, dtype=torch.float32, device="cuda"))
    else:
        p = W.wd_solve_params_default()
        p.inner_prec, p.tol = prec, TOL
        if case.get("solver") == "bicgstab":
            p.solver = W.WD_SOLVER_BICGSTAB
        b = _real(_sources(case, seed))
        s.update(U=_real(_links(dims, seed)), b=b, x=torch.zeros_like(b), params=p)
    s["result"] = _result(s)
    return s


def _result(s):
    """The outputs of a pass, as views of the state's buffers."""
    c, dims, prec, kind = s["case"], s["dims"], s["prec"], s["kind"]
    if kind == "dslash":
        return _values(s["out"], dims, prec, 2 if s["parity"] == W.WD_FULL else 1)
    if kind == "mhat":
        return _values(s["out"], dims, prec)
    if kind == "mrhs":
        return {"norm": s["norm"], **_values(s["out"], dims, prec, c["nrhs"])}
    if kind == "blas":
        return {"dots": s["dots"], **_values(s["y"], dims, prec)}
    if kind == "load":
        n = _padded(dims)
        if prec == W.WD_F16:
            links = s["gauge"][:8 * n * 24].view(torch.float16)
        else:
            links = s["gauge"][:8 * n * c["recon"] * (8 if prec == W.WD_F64 else 4)].view(
                torch.float64 if prec == W.WD_F64 else torch.float32)
        return {"links": links, "back": s["back"], **_values(s["spinor"], dims, prec, 2)}
    return {k: s[k] for k in ("out", "grad", "x") if k in s}


def run(s):
    c, dims, prec, kind = s["case"], s["dims"], s["prec"], s["kind"]
    if kind == "dslash":
        (W.wd_dslash_dag if c["dagger"] else W.wd_dslash)(s["out"], s["inp"], s["gauge"], 0.1365, s["parity"], dims,
                                                          prec)
    elif kind == "mhat":
        W.wd_mhat(s["out"], s["inp"], s["gauge"], s["tmp"], 0.137, c["dagger"], dims, prec, c["recon"])
    elif kind == "mrhs":
        W.wd_dslash_mrhs(s["out"], s["inp"], s["gauge"], W.WD_EVEN, c["dagger"], -0.0185, s["x"], 1.0, c["nrhs"],
                         s["norm"], dims, prec, c["recon"])
    elif kind == "blas":
        W.wd_norm2(s["dots"], s["x"], dims, W.WD_EVEN, prec)
        W.wd_cdot(s["dots"].data_ptr() + 16, s["x"], s["y"], dims, W.WD_EVEN, prec)
        W.wd_axpby(1.0, s["x"], 0.375, s["y"], dims, W.WD_EVEN, prec)
    elif kind == "load":
        W.wd_pack_gauge(s["gauge"], s["U"], dims, prec, c["recon"])
        W.wd_pack_spinor(s["spinor"], s["psi"], dims, W.WD_FULL, prec)
        W.wd_unpack_spinor(s["back"], s["spinor"], dims, W.WD_FULL, prec)
    elif kind == "layer":
        W.wd_nn_layer(s["out"], s["inp"], s["w"], c["cin"], c["cout"], s["gauge"], dims)
        W.wd_nn_wgrad(s["grad"], s["inp"], s["delta"], c["cin"], c["cout"], s["gauge"], dims)
    elif kind == "net":
        W.wd_nn_apply_ex(s["out"], s["inp"], s["w"], s["gauge"], dims,
                         (W.WD_NN_BF16 if c["bf16"] else 0) | (W.WD_NN_EVEN if c["even"] else 0))
    elif kind == "solve":
        W.wd_solve_ex(s["x"], s["b"], s["U"], c["kappa"], dims, s["params"])
    else:
        W.wd_solve_batch([dict(dims=dims, kappa=c["kappa"], nrhs=c["nrhs"], gauge=s["U"], b=s["b"], x=s["x"])],
                         s["params"])
    return s["result"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    dims, kind = _dims(case), case["kind"]
    V = _volume(dims)
    spinor = {"f64": 192, "f32": 96, "f16": 52}.get(case.get("prec"), 96)
    link = {"f64": 8, "f32": 4, "f16": 2}.get(case.get("prec"), 4) * case.get("recon", 12)
    if kind == "dslash":  # per output site: eight links, its share of the input, itself
        n = V if case["parity"] == "full" else V // 2
        return {"bytes": n * (8 * link + 2 * spinor) if case["parity"] != "full" else n * (4 * link + 2 * spinor),
                "flops": 1320 * n}
    if kind == "mhat":  # the links once, the input once, the output once
        return {"bytes": 4 * V * link + V * spinor, "flops": V // 2 * (2 * 1320 + 48)}
    if kind == "mrhs":
        return {"bytes": 4 * V * link + 3 * case["nrhs"] * V // 2 * spinor, "flops": case["nrhs"] * V // 2 * 1416}
    if kind == "blas":  # two fields in, one out
        return {"bytes": 3 * V // 2 * spinor, "flops": V // 2 * 240}
    if kind == "load":
        return {"bytes": 4 * V * (144 + link) + V * (192 + spinor) + V * 192, "flops": 0}
    if kind in ("layer", "net"):
        layers = [(case["cin"], case["cout"])] if kind == "layer" else [(i, o) for i, o, _ in NET]
        mix = sum(9 * 3 * 8 * i * o for i, o in layers) * V
        hop = sum(8 * 66 * i for i, _ in layers) * V
        if kind == "layer":  # forward and weight gradient
            return {"bytes": 4 * V * 48 + V * 24 * (case["cin"] + 2 * case["cout"]), "flops": 2 * mix + hop}
        share = 0.5 if case["even"] else 1.0
        return {"bytes": 4 * V * 48 + 2 * 96 * V * share, "flops": (mix + hop) * share}
    # the links and the sources in, the solutions out; the operator 60 times a source on both parities
    n = case.get("nrhs", 1)
    return {"bytes": 4 * V * 144 + 2 * n * V * 192, "flops": 60 * n * 1320 * V}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _hops(phi, U, dims):
    """T_d phi for d = 1..8 on the full lattice: forward and backward in x, y, z, t (phi [V, C, 3])."""
    shape = (dims[3], dims[2], dims[1], dims[0])
    f = phi.reshape(*shape, *phi.shape[1:])
    for mu in range(4):
        u, ax = U[mu].reshape(*shape, 3, 3), 3 - mu
        fwd = torch.roll(f, -1, ax)
        if mu == 3:
            fwd[-1] = -fwd[-1]
        yield (u.unsqueeze(-3) * fwd.unsqueeze(-2)).sum(-1).reshape(phi.shape)
        bwd = torch.roll((u.mH.unsqueeze(-3) * f.unsqueeze(-2)).sum(-1), 1, ax)
        if mu == 3:
            bwd[0] = -bwd[0]
        yield bwd.reshape(phi.shape)


def _hopping(psi, U, dims, dagger=False):
    """H psi or H^+ psi (psi [V, 4, 3])."""
    g = _gamma().to(psi.device) * (-1 if dagger else 1)
    out = torch.zeros_like(psi)
    for d, t in enumerate(_hops(psi, U, dims)):
        gt = torch.einsum("st,vtc->vsc", g[d // 2], t)
        out += t + gt if d & 1 else t - gt
    return out


def _hop_half(half, U, dims, parity, dagger=False):
    """H restricted: a half field [Vh, 12] of the other parity -> one of `parity`."""
    full = torch.zeros(_volume(dims), 12, dtype=CD, device="cuda")
    full[_parity_sites(dims, 1 - parity)] = half
    h = _hopping(full.reshape(-1, 4, 3), U, dims, dagger).reshape(-1, 12)
    return h[_parity_sites(dims, parity)]


def _layer(phi, w, U, dims):
    y = torch.einsum("oi,via->voa", w[0], phi)
    for d, t in enumerate(_hops(phi, U, dims)):
        y += torch.einsum("oi,via->voa", w[d + 1], t)
    return y


def _solve(b, U, kappa, dims):
    """D x = b by CG on the normal equations, to the accuracy of 64 bits."""
    def op(v, dag=False):
        return v - kappa * _hopping(v, U, dims, dag)

    x, r = torch.zeros_like(b), b.clone()
    for _ in range(2):  # the second time from the residual itself
        s = op(r, True)
        p, y, res = s.clone(), torch.zeros_like(b), r.clone()
        gam, stop = s.abs().square().sum(), 1e-28 * s.abs().square().sum()
        for _ in range(2000):
            if gam <= stop:
                break
            q = op(p)
            a = gam / q.abs().square().sum()
            y += a * p
            res -= a * q
            s = op(res, True)
            new = s.abs().square().sum()
            p = s + (new / gam) * p
            gam = new
        x += y
        r = b - op(x)
    return x


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    V, prec = _volume(dims), PREC.get(case.get("prec", "f32"))
    if kind == "blas":
        x, y = _gaussian((2, V // 2, 12), seed, 2)
        d = (x.conj() * y).sum()
        return {"dots": torch.stack([x.abs().square().sum(), 0 * d.real, d.real, d.imag]),
                **_layout((x + 0.375 * y)[None], dims, prec)}
    if kind in ("solve", "batch") and case.get("nrhs", 1) * V > 24 ** 3 * 48:
        return None
    U = _links(dims, seed)
    if kind == "load":
        psi = _gaussian((V, 12), seed, 2)
        halves = torch.stack([psi[_parity_sites(dims, p)] for p in (0, 1)])
        n, nc = _padded(dims), case["recon"] // 2
        u = torch.zeros(4, 2, n, nc, dtype=CD, device="cuda")
        for p in (0, 1):
            u[:, p, :V // 2] = U[:, _parity_sites(dims, p)].reshape(4, V // 2, 9)[:, :, :nc]
        r = torch.view_as_real(u).reshape(8, n // 32, 32, 2 * nc)
        if prec == W.WD_F16:  # U00 U01 U02 U10 of all regions, then U11 U12
            links = torch.cat([r[..., :8].reshape(-1), r[..., 8:].reshape(-1)])
        else:
            k = {W.WD_F64: nc, W.WD_F32: nc if nc == 9 else nc // 2}[prec]
            links = r.reshape(8, n // 32, 32, k, 2 * nc // k).permute(0, 1, 3, 2, 4).reshape(-1)
        return {"links": links, "back": _real(psi), **_layout(halves, dims, prec)}
    if kind == "dslash":
        if case["parity"] == "full":
            psi = _gaussian((V, 12), seed, 2).reshape(V, 4, 3)
            d = (psi - 0.1365 * _hopping(psi, U, dims, case["dagger"])).reshape(V, 12)
            return _layout(torch.stack([d[_parity_sites(dims, p)] for p in (0, 1)]), dims, prec)
        h = _hop_half(_gaussian((V // 2, 12), seed, 2), U, dims, PARITY[case["parity"]], case["dagger"])
        return _layout(-0.1365 * h[None], dims, prec)
    if kind == "mhat":
        v = _gaussian((V // 2, 12), seed, 2)
        t = _hop_half(v, U, dims, 1, case["dagger"])
        return _layout((v - 0.137 ** 2 * _hop_half(t, U, dims, 0, case["dagger"]))[None], dims, prec)
    if kind == "mrhs":
        nr = case["nrhs"]
        src, x = _gaussian((nr, V // 2, 12), seed, 2), _gaussian((nr, V // 2, 12), seed, 4)
        o = torch.stack([-0.0185 * _hop_half(src[r], U, dims, 0, case["dagger"]) + x[r] for r in range(nr)])
        return {"norm": o.abs().square().sum((1, 2)), **_layout(o, dims, prec)}
    if kind == "layer":
        ci, co = case["cin"], case["cout"]
        w, = _weights([next(n for n in NET if n[:2] == (ci, co))], seed)
        phi, delta = _gaussian((V, ci, 3), seed, 2), _gaussian((V, co, 3), seed, 4)
        t = [phi] + list(_hops(phi, U, dims))
        grad = torch.stack([torch.einsum("voa,via->oi", delta, z.conj()) for z in t])
        return {"out": _nn_pack(_layer(phi, w, U, dims), dims), "grad": _real(grad)}
    if kind == "net":
        phi, par = _gaussian((V, 4, 3), seed, 2), _parity_sites(dims, 1)
        if case["even"]:
            phi[par] = 0
        for w in _weights(NET, seed):
            phi = _layer(phi, w, U, dims)
        if case["even"]:
            phi[par] = 0
        return {"out": _nn_pack(phi, dims)}
    return {"x": torch.cat([_real(_solve(b, U, case["kappa"], dims)) for b in _sources(case, seed)])}
