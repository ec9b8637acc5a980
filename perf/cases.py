"""The work that users of this library have it do, as cases that can be timed and checked.

``listed()`` names twelve of them, ``draw(rng)`` gives another of the same ranges, ``prepare(case, seed)``
builds what a program holds before the call (hierarchy handle, fields on the GPU), ``run(state)`` makes one
pass through the public binding, ``work(case)`` counts the bytes and flops that no implementation can avoid
and ``exact(case, seed)`` computes the same result in 64 bits with plain torch.

Operator cases use SU(3) links 1 + eps (A - A^+) / 2, reunitarised (the generator of the repository's
bandwidth lattice); whole solves use beta = 6.0 heatbath fields of at most 8^4, tiled to the lattice as the
32^3 x 64 solve of the benchmark does.
"""
import math

import numpy as np
import torch

from paper_0811_4331_gb300 import inputs
from paper_0811_4331_gb300 import wilson_mg as wm

PRECS = {"f64": 0, "f32": 1, "f16": 2, "bf16": 3}
CX_BYTES = {"f64": 16, "f32": 8, "f16": 4, "bf16": 4}
EPS = 0.3        # disorder of the operator cases' links
SWEEPS = 6       # relaxation sweeps of the operator cases' null vectors
TOL = 1e-12      # relative residual of the solves
HEATBATH = 30    # heatbath sweeps of the solves' fields
MASS = 0.05      # of the operator cases


def listed():
    return [
        # the smoother's stencil of an 8^3 x 16 solve: the smallest call, called thousands of times a solve
        {"name": "dslash_f16_8x8x8x16", "kind": "dslash", "prec": "f16", "x": 8, "y": 8, "z": 8, "t": 16, "nrhs": 1},
        # the stencil of a large lattice, fields far above the L2
        {"name": "dslash_f16_32x32x32x64", "kind": "dslash", "prec": "f16", "x": 32, "y": 32, "z": 32, "t": 64,
         "nrhs": 1},
        # the Krylov operator of a propagator: twelve spin-colour sources at once
        {"name": "dslash_f32_16x16x16x32_12", "kind": "dslash", "prec": "f32", "x": 16, "y": 16, "z": 16, "t": 32,
         "nrhs": 12},
        # the true residual of every solve, and the operator of the FP64 solvers
        {"name": "dslash_f64_16x16x16x32", "kind": "dslash", "prec": "f64", "x": 16, "y": 16, "z": 16, "t": 32,
         "nrhs": 1},
        # two smoothing steps on a lattice with odd and unequal extents
        {"name": "mr_bf16_18x14x10x21", "kind": "mr", "prec": "bf16", "x": 18, "y": 14, "z": 10, "t": 21, "nrhs": 1,
         "steps": 2},
        # the even-odd smoother's operator, twelve sources
        {"name": "schur_f16_16x16x16x32_12", "kind": "schur", "prec": "f16", "x": 16, "y": 16, "z": 16, "t": 32,
         "nrhs": 12},
        # the two transfers of a 24-source cycle (12 point and 12 Gaussian sources in the benchmark)
        {"name": "restrict_f16_16x16x16x32_24", "kind": "restrict", "prec": "f16", "x": 16, "y": 16, "z": 16, "t": 32,
         "block": 4, "nv": 24, "nrhs": 24},
        {"name": "prolong_f16_16x16x16x32_24", "kind": "prolong", "prec": "f16", "x": 16, "y": 16, "z": 16, "t": 32,
         "block": 4, "nv": 24, "nrhs": 24},
        # the coarse stencil of that cycle, and the same operator with one source in FP32
        {"name": "coarse_mma_16x16x16x32_24", "kind": "coarse", "prec": "f32", "mma": 1, "x": 16, "y": 16, "z": 16,
         "t": 32, "block": 4, "nv": 24, "nrhs": 24},
        {"name": "coarse_f32_16x16x16x32", "kind": "coarse", "prec": "f32", "mma": 0, "x": 16, "y": 16, "z": 16,
         "t": 32, "block": 4, "nv": 24, "nrhs": 1},
        # the benchmark's step: null vectors, retarget to four masses, four solves side by side
        {"name": "sweep_8x8x8x16", "kind": "sweep", "x": 8, "y": 8, "z": 8, "t": 16, "nv": 20, "sweeps": 300,
         "masses": 4},
        # a propagator: twelve sources on a three-level hierarchy that the program keeps
        {"name": "propagator_16x16x16x32", "kind": "propagator", "x": 16, "y": 16, "z": 16, "t": 32, "nv": 24,
         "nrhs": 12},
    ]


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "dslash", "mr", "schur", "restrict", "prolong", "coarse", "coarse",
                       "sweep", "propagator"])
    case = {"kind": kind}
    if kind in ("dslash", "mr", "schur"):
        unit = 2 if kind == "schur" else 1
        sites = math.exp(rng.uniform(math.log(256), math.log(1 << 20)))
        ext = [max(unit, unit * round(sites ** 0.25 * math.exp(rng.uniform(-0.35, 0.35)) / unit)) for _ in range(4)]
        V = ext[0] * ext[1] * ext[2] * ext[3]
        case["prec"] = rng.choice(["f16", "f16", "bf16", "f32", "f32", "f64"])
        # the FP64 stencil is far slower per site, so its fields stay smaller
        room = max(1, (150000 if case["prec"] == "f64" else 2000000) // V)
        case["nrhs"] = 1 if kind == "mr" else min(room, rng.choice([1, 1, 2, 3, 4, 6, 8, 12, 24]))
        if kind == "mr":
            case["steps"] = rng.choice([1, 2, 4])
    elif kind in ("restrict", "prolong", "coarse"):
        block = rng.choice([2, 4, 4])
        sites = math.exp(rng.uniform(math.log(4 if kind == "coarse" else 2), math.log(512)))  # coarse sites
        ext = [block * max(1, round(sites ** 0.25 * math.exp(rng.uniform(-0.5, 0.5)))) for _ in range(4)]
        while ext[0] * ext[1] * ext[2] * ext[3] > 131072:
            ext[ext.index(max(ext))] -= block
        case["block"] = block
        case["nv"] = rng.choice([8, 12, 16, 20, 24, 24, 28, 32])
        case["nrhs"] = rng.choice([1, 2, 4, 6, 9, 12, 16, 24])
        if kind == "coarse":
            case["mma"] = rng.choice([0, 1, 1])
            case["prec"] = "f32" if case["mma"] else rng.choice(["f32", "f64"])
        else:
            case["prec"] = rng.choice(["f16", "f16", "bf16", "f32", "f64"])
    elif kind == "sweep":
        ext = [4 * rng.choice([1, 2]), 4 * rng.choice([1, 2]), 8, 8 * rng.choice([1, 2])]
        case.update(nv=rng.choice([16, 20]), sweeps=rng.choice([100, 200, 300]), masses=rng.choice([1, 2, 3, 4]))
    else:
        ext = [8 * rng.choice([1, 2]), 8 * rng.choice([1, 2]), 16, 8 * rng.choice([1, 2, 3, 4])]
        case.update(nv=rng.choice([16, 20, 24]), nrhs=rng.choice([1, 2, 4, 6, 8, 12]))
    case.update(x=ext[0], y=ext[1], z=ext[2], t=ext[3])
    return case


# ---------------------------------------------------------------- inputs


def _dims(case):
    return (case["x"], case["y"], case["z"], case["t"])


def _volume(case):
    return case["x"] * case["y"] * case["z"] * case["t"]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _randn(shape, gen, dtype=torch.complex128):
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype)


def _links(dims, gen):
    """(4, Lt, Lz, Ly, Lx, 3, 3) SU(3) links near the identity."""
    shape = (4,) + tuple(reversed(dims)) + (3, 3)
    a = _randn(shape, gen) * math.sqrt(2.0)  # re and im ~ N(0, 1)
    m = torch.eye(3, device="cuda", dtype=torch.complex128) + 0.5 * EPS * (a - a.mH)
    r0 = m[..., 0, :]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    r1 = m[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], dim=-2).contiguous()


def _heatbath_links(dims, seed):
    """beta = 6.0 links of a lattice of extents at most 8, tiled to dims."""
    base = list(dims)
    for i in range(4):
        while base[i] > 8:
            base[i] //= 2
    U = torch.from_numpy(inputs.heatbath_gauge(tuple(base), 6.0, HEATBATH, int(seed))).cuda()
    reps = [d // b for d, b in zip(dims, base)]
    return U.repeat(1, reps[3], reps[2], reps[1], reps[0], 1, 1).contiguous()


def _field(shape, prec, gen):
    """A Gaussian field in internal storage."""
    if prec == "f64":
        return _randn(shape, gen)
    x = _randn(shape, gen, torch.complex64)
    if prec == "f32":
        return x
    return torch.view_as_real(x).to(torch.float16 if prec == "f16" else torch.bfloat16).contiguous()


def _level1(case):
    """Extents of the first coarse level and the block that takes it to the second."""
    ext = [d // case["block"] for d in _dims(case)]
    return ext, [2 if e % 2 == 0 else 1 for e in ext]


def _starts(case, gen):
    """Start vectors of the null-vector setup, external layout, on the host as the binding takes them."""
    V = _volume(case)
    out = [_randn((case["nv"], V, 12), gen)]
    if case["kind"] == "coarse":
        ext, _ = _level1(case)
        out.append(_randn((2, ext[0] * ext[1] * ext[2] * ext[3], 2 * case["nv"]), gen))
    return out


def _operator_handle(case, U, starts):
    prec = PRECS[case["prec"]]
    kw = dict(mixed=0) if prec == 0 else dict(mixed=1, fine_prec=prec)
    if case["kind"] in ("dslash", "mr", "schur"):
        p = wm.mg_default_params(n_levels=1, **kw)
        return wm.mg_setup(U, _dims(case), MASS, p)
    block = [(case["block"],) * 4]
    nv, sweeps = [case["nv"]], [SWEEPS]
    if case["kind"] == "coarse":  # a third level, so that level 1 keeps its operator in the cycle's precisions
        block.append(tuple(_level1(case)[1]))
        nv.append(2)
        sweeps.append(1)
        kw["coarse_mma"] = case["mma"]
    p = wm.mg_default_params(n_levels=len(nv) + 1, block=block, nv=nv, setup_sweeps=sweeps, defer_coarsest=1, **kw)
    return wm.mg_setup(U, _dims(case), MASS, p, starts=[s.cpu().numpy() for s in starts])


def _shapes(case):
    """Internal shapes of the input and the output of an operator case."""
    V, R = _volume(case), case["nrhs"]
    fine = (R, 3, V, 4)
    if case["kind"] in ("dslash", "mr"):
        return fine, fine
    if case["kind"] == "schur":
        return (R, 3, V // 2, 4), (R, 3, V // 2, 4)
    ext, _ = _level1(case)
    coarse = (R, 2 * case["nv"], ext[0] * ext[1] * ext[2] * ext[3])
    return {"restrict": (fine, coarse), "prolong": (coarse, fine), "coarse": (coarse, coarse)}[case["kind"]]


def _in_out_prec(case):
    """Storage of input and output: 16-bit transfers have FP32 on the coarse side."""
    p = case["prec"]
    c = "f64" if p == "f64" else "f32"
    return {"restrict": (p, c), "prolong": (c, p)}.get(case["kind"], (p, p))


def _operator_inputs(case, seed):
    gen = _generator(seed)
    U = _links(_dims(case), gen)
    starts = _starts(case, gen) if "nv" in case else []
    return U, starts, _field(_shapes(case)[0], _in_out_prec(case)[0], gen)


# the solves' quark masses: beta = 6.0 fields of this kind have their critical mass near -0.75
SWEEP_MASSES = [-0.62, -0.65, -0.67, -0.68]
PROPAGATOR_MASS = -0.66


def _sources(case, count, seed):
    return _randn((count,) + tuple(reversed(_dims(case))) + (4, 3), _generator(seed)) * math.sqrt(2.0)


# ---------------------------------------------------------------- prepare and run


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        p = wm.mg_default_params(n_levels=2, block=[(4, 4, 4, 4)], nv=[case["nv"]], setup_sweeps=[case["sweeps"]],
                                 mixed=1, fine_prec=wm.MG_F16, seed=7, defer_coarsest=1)
        return {"kind": kind, "dims": _dims(case), "U": _heatbath_links(_dims(case), seed), "params": p,
                "masses": SWEEP_MASSES[-case["masses"]:], "b": _sources(case, 1, seed)[0],
                "streams": [torch.cuda.Stream() for _ in range(case["masses"])]}
    if kind == "propagator":
        p = wm.mg_default_params(n_levels=3, block=[(4, 4, 4, 4), (2, 2, 2, 2)], nv=[case["nv"], case["nv"]],
                                 setup_sweeps=[300, 100], mixed=1, fine_prec=wm.MG_F16, seed=7, coarse_mma=1)
        h = wm.mg_setup(_heatbath_links(_dims(case), seed), _dims(case), PROPAGATOR_MASS, p)
        return {"kind": kind, "h": h, "b": _sources(case, case["nrhs"], seed)}
    U, starts, inp = _operator_inputs(case, seed)
    h = _operator_handle(case, U, starts)
    out = torch.empty_like(_field(_shapes(case)[1], _in_out_prec(case)[1], _generator(0)))
    state = {"kind": kind, "h": h, "prec": PRECS[case["prec"]], "nrhs": case["nrhs"], "in": inp, "out": out}
    if kind == "mr":
        state.update(x=torch.empty_like(inp), steps=case["steps"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "sweep":
        masses, b = state["masses"], state["b"]
        base = wm.mg_setup(state["U"], state["dims"], masses[-1], state["params"])
        hs = wm.mg_retarget_batch(base, masses)
        xs = [torch.zeros_like(b) for _ in masses]
        for q in state["streams"]:
            q.wait_stream(torch.cuda.current_stream())
        wm.mg_solve_many(hs, [b] * len(masses), xs, TOL, streams=state["streams"])
        for h in hs:
            wm.mg_destroy(h)
        wm.mg_destroy(base)
        return xs
    if kind == "propagator":
        x = torch.zeros_like(state["b"])
        wm.mg_solve(state["h"], state["b"], x, TOL)
        return x
    h, prec, inp, out, nrhs = state["h"], state["prec"], state["in"], state["out"], state["nrhs"]
    if kind == "dslash":
        wm.dslash_apply(h, prec, inp, out, nrhs)
    elif kind == "schur":
        wm.schur_apply(h, prec, inp, out, nrhs)
    elif kind == "restrict":
        wm.restrict_apply(h, 0, prec, inp, out, nrhs)
    elif kind == "prolong":
        wm.prolong_apply(h, 0, prec, inp, out, nrhs)
    elif kind == "coarse":
        wm.coarse_apply(h, 1, prec, inp, out, nrhs)
    else:
        state["x"].zero_()
        wm.mr_apply(h, 0, prec, inp, state["x"], out, state["steps"])
        return [state["x"], out]
    return out


# ---------------------------------------------------------------- work

HOP_FLOPS = 1368  # of D at one site


def work(case):
    V, kind = _volume(case), case["kind"]
    if kind == "sweep":
        # links and source in, solutions out; relaxation of the null vectors and about 40 cycles of five
        # stencils and one outer stencil per mass
        m = case["masses"]
        return {"bytes": 16.0 * V * (36 + 12 + 12 * m),
                "flops": float(HOP_FLOPS) * V * (case["nv"] * case["sweeps"] + 240 * m)}
    if kind == "propagator":
        return {"bytes": 16.0 * V * 24 * case["nrhs"] + 24.0 * 4 * V,
                "flops": float(HOP_FLOPS) * V * 300 * case["nrhs"]}
    R = case["nrhs"]
    pi, po = _in_out_prec(case)
    n_in, n_out = (math.prod(s) for s in _shapes(case))
    vectors = n_in * CX_BYTES[pi] + n_out * CX_BYTES[po]
    links = 24.0 * V * CX_BYTES[case["prec"]]  # two rows of four links
    if kind == "dslash" or kind == "schur":
        return {"bytes": vectors + links, "flops": float(HOP_FLOPS) * V * R}
    if kind == "mr":
        return {"bytes": vectors + n_out * CX_BYTES[po] + links, "flops": (HOP_FLOPS + 100.0) * V * (case["steps"] + 1)}
    if kind == "coarse":
        nc = 2 * case["nv"]
        sites = n_in // (R * nc)
        cell = 4 if case["mma"] else CX_BYTES[case["prec"]]
        return {"bytes": vectors + 9.0 * nc * nc * sites * cell, "flops": 8.0 * 9 * nc * nc * sites * R}
    return {"bytes": vectors + 12.0 * case["nv"] * V * CX_BYTES[case["prec"]], "flops": 8.0 * 12 * case["nv"] * V * R}


# ---------------------------------------------------------------- 64-bit values with plain torch

# gamma_mu [[0, X], [X^+, 0]] in the chiral basis: X = -i sigma_k for x, y, z and 1 for t
_SIGMA = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
_GAMMA_X = [-1j * _SIGMA[0], -1j * _SIGMA[1], -1j * _SIGMA[2], np.eye(2)]


def _su3(U, h, dagger):
    """U h or U^+ h on the last axis of h (..., spin, colour)."""
    out = None
    for b in range(3):
        col = U[..., b, :].conj() if dagger else U[..., :, b]
        term = col.unsqueeze(-2) * h[..., b:b + 1]
        out = term if out is None else out + term
    return out


def _spin2(m, h):
    """The 2 x 2 matrix m on the spin axis of h (..., 2, 3); every row of m has one entry."""
    rows = []
    for i in range(2):
        j = int(np.argmax(np.abs(m[i])))
        rows.append(complex(m[i, j]) * h[..., j, :])
    return torch.stack(rows, dim=-2)


def _dirac(U, psi, mass):
    """D psi for psi (R, Lt, Lz, Ly, Lx, 4, 3)."""
    out = (4.0 + mass) * psi
    for mu in range(4):
        axis, X = 4 - mu, _GAMMA_X[mu]
        Xi = X.conj().T
        for fwd in (True, False):
            s = 1.0 if fwd else -1.0
            h = psi[..., :2, :] - s * _spin2(X, psi[..., 2:, :])  # upper half of (1 -+ gamma) psi
            if fwd:
                g = _su3(U[mu], torch.roll(h, -1, axis), False)
            else:
                g = torch.roll(_su3(U[mu], h, True), 1, axis)
            out[..., :2, :] -= 0.5 * g
            out[..., 2:, :] += 0.5 * s * _spin2(Xi, g)
    return out


def _to_lattice(f, case):
    """Internal level-0 field (R, 3, V, 4[, 2]) -> (R, Lt, Lz, Ly, Lx, 4, 3) complex128."""
    f = torch.view_as_complex(f.double().contiguous()) if f.dim() == 5 else f.to(torch.complex128)
    return f.permute(0, 2, 1, 3).reshape((f.shape[0],) + tuple(reversed(_dims(case))) + (4, 3))


def _from_lattice(psi):
    V = psi[0].numel() // 12
    return psi.reshape(psi.shape[0], V, 3, 4).permute(0, 2, 1, 3).contiguous()


def _parity(case):
    axes = [torch.arange(n, device="cuda") for n in reversed(_dims(case))]
    return sum(torch.meshgrid(*axes, indexing="ij")).flatten() % 2


def _schur(U, case, half):
    """S = M - H_eo H_oe / (4 M) on an internal even half field."""
    M = 4.0 + MASS
    even = (_parity(case) == 0).nonzero().flatten()
    f = torch.view_as_complex(half.double().contiguous()) if half.dim() == 5 else half.to(torch.complex128)
    full = torch.zeros(f.shape[:2] + (_volume(case), 4), dtype=torch.complex128, device="cuda")
    full[:, :, even] = f
    psi = _to_lattice(full, case)
    hop = lambda v: 2.0 * (M * v - _dirac(U, v, MASS))  # noqa: E731  (D = M - H / 2)
    out = M * psi - hop(hop(psi)) / (4.0 * M)
    return _from_lattice(out)[:, :, even]


def _mr_step(U, x, r, omega=0.8):
    """One under-relaxed minimal-residual step of every right-hand side."""
    p = _dirac(U, r, MASS)
    dims = tuple(range(1, r.dim()))
    a = (p.conj() * r).sum(dims, keepdim=True) / (p.abs() ** 2).sum(dims, keepdim=True)
    return x + omega * a * r, r - omega * a * p


def _to_blocks(psi, case):
    """(R, Lt, Lz, Ly, Lx, 4, 3) -> (coarse site, chirality, R, elements of the block)."""
    b, R = case["block"], psi.shape[0]
    lt, lz, ly, lx = (d // b for d in reversed(_dims(case)))
    v = psi.reshape(R, lt, b, lz, b, ly, b, lx, b, 2, 6)
    return v.permute(1, 3, 5, 7, 9, 0, 2, 4, 6, 8, 10).reshape(lt * lz * ly * lx, 2, R, b ** 4 * 6)


def _from_blocks(v, case):
    b, R = case["block"], v.shape[2]
    lt, lz, ly, lx = (d // b for d in reversed(_dims(case)))
    v = v.reshape(lt, lz, ly, lx, 2, R, b, b, b, b, 6).permute(5, 0, 6, 1, 7, 2, 8, 3, 9, 4, 10)
    return v.reshape((R,) + tuple(reversed(_dims(case))) + (4, 3))


def _prolongator(U, case, start):
    """Orthonormal null vectors per block and chirality, (coarse site, chirality, nv, elements)."""
    x = start.reshape((case["nv"],) + tuple(reversed(_dims(case))) + (4, 3)).clone()
    r = -_dirac(U, x, MASS)
    for _ in range(SWEEPS):
        x, r = _mr_step(U, x, r)
    v = _to_blocks(x, case).contiguous()
    for k in range(case["nv"]):
        q = v[:, :, k]
        for _ in range(2 if k else 0):
            q = q - (v[:, :, :k].conj() @ q.unsqueeze(-1)).transpose(-1, -2).matmul(v[:, :, :k]).squeeze(-2)
        v[:, :, k] = q / torch.linalg.vector_norm(q, dim=-1, keepdim=True)
    return v


def _restrict(P, psi, case):
    """(R, 2 nv, coarse sites)"""
    c = torch.matmul(_to_blocks(psi, case), P.mH)  # (site, chirality, R, nv)
    return c.permute(2, 1, 3, 0).reshape(psi.shape[0], 2 * case["nv"], P.shape[0])


def _prolong(P, c, case):
    R, n, sites = c.shape
    y = c.to(torch.complex128).reshape(R, 2, n // 2, sites).permute(3, 1, 0, 2)
    return _from_blocks(torch.matmul(y, P), case)


def _solve(U, b, mass):
    """D x = b for every right-hand side by BiCGstab, restarted from the true residual."""
    dims = tuple(range(1, b.dim()))
    dot = lambda u, v: (u.conj() * v).sum(dims, keepdim=True)  # noqa: E731
    bn = dot(b, b).real.sqrt()
    x = torch.zeros_like(b)
    for _ in range(6):
        r = b - _dirac(U, x, mass)
        if float((dot(r, r).real.sqrt() / bn).max()) < 2e-14:
            break
        r = r.clone()
        hat, p, rho = r.clone(), r.clone(), dot(r, r)
        target = 1e-9 * bn if float((dot(r, r).real.sqrt() / bn).max()) > 1e-6 else 3e-15 * bn
        for it in range(1500):
            v = _dirac(U, p, mass)
            alpha = rho / dot(hat, v)
            s = r - alpha * v
            t = _dirac(U, s, mass)
            omega = dot(t, s) / dot(t, t)
            x = x + alpha * p + omega * s
            r = s - omega * t
            if it % 10 == 9 and bool((dot(r, r).real.sqrt() <= target).all()):
                break
            new = dot(hat, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        U, b = _heatbath_links(_dims(case), seed), _sources(case, 1, seed)
        return [_solve(U, b, m)[0] for m in SWEEP_MASSES[-case["masses"]:]]
    if kind == "propagator":
        return _solve(_heatbath_links(_dims(case), seed), _sources(case, case["nrhs"], seed), PROPAGATOR_MASS)
    U, starts, inp = _operator_inputs(case, seed)
    real = lambda f, prec: torch.view_as_real(f) if prec in ("f16", "bf16") else f  # noqa: E731
    if kind == "dslash":
        return real(_from_lattice(_dirac(U, _to_lattice(inp, case), MASS)), case["prec"])
    if kind == "schur":
        return real(_schur(U, case, inp), case["prec"])
    if kind == "mr":
        r = _to_lattice(inp, case)
        x = torch.zeros_like(r)
        for _ in range(case["steps"]):
            x, r = _mr_step(U, x, r)
        return [real(_from_lattice(x), case["prec"]), real(_from_lattice(r), case["prec"])]
    P = _prolongator(U, case, starts[0])
    if kind == "restrict":
        return _restrict(P, _to_lattice(inp, case), case)
    if kind == "prolong":
        return real(_from_lattice(_prolong(P, inp, case)), case["prec"])
    return _restrict(P, _dirac(U, _prolong(P, inp, case), MASS), case)
