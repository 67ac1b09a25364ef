"""Performance cases: the work that users of this framework have it do, each through the public
entry points of `paper_1311_5029_gb300`.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare(case, seed)` makes
what a program holds before the call, `run(state)` is one pass, `work(case)` the bytes and
floating-point operations that a pass cannot do without, and `exact(case, seed)` the values that
`run` stands for, in 64 bits with plain torch.

The lattices are those of the paper's and this repository's workloads (4^3 x 8, 16^3 x 32,
20^3 x 64, 28^3 x 96) and ragged ones between them; the coefficients are the workloads' placeholder
set; links are random SU(3) matrices near the identity, as in a thermalised gauge field.
"""
import math

import numpy as np
import torch

import paper_1311_5029_gb300 as ok

COEFFS = {"u0": 0.0, "am0": 0.5, "kappa": 0.0, "zeta": 1.0, "r_s": 1.0, "c_B": 1.0, "c_E": 1.0, "c_EE": 0.03,
          "c1": 0.05, "c2": 0.02, "c3": 0.04, "c4": 0.03, "c5": 0.02}
TOL = 1e-11      # true FP64 residual of every solve: the solution itself is then good to about 1e-10
DELTA = 1e-4     # reliable-update threshold of the benchmark's solves
RATE = 1e-3      # Adam rate of a training step
LAYERS = 4       # layers of the learned preconditioner

# Bytes per site of the stored W of each precision (43 colour matrices) and of one spinor field.
W_BYTES = {"f64": 6192, "df64": 6192, "f32": 3096, "w16": 1548, "tc": 1548}
SPINOR = {"f64": 192, "df64": 192, "f32": 96, "w16": 96, "tc": 96}
COPY = {"f64": ok.W_F64, "df64": ok.W_DF64, "f32": ok.W_F32, "w16": ok.W_F16, "tc": ok.W_F16_TC}
PREC = {"f64": ok.F64, "df64": ok.F64, "f32": ok.F32, "w16": ok.F32_W16, "tc": ok.F16_TC}
APPLY_FLOPS = 148 * 66   # colour matrix-vector products of one site


def listed():
    return [
        # The smallest call: one application on a test lattice, where launch and call latency count.
        {"name": "apply_f32_4x8", "kind": "apply", "x": 4, "y": 4, "z": 4, "t": 8, "bct": 1, "prec": "f32", "nrhs": 1},
        # The inner operator of every mixed-precision solve, on the benchmark's lattice.
        {"name": "apply_f32_16x32", "kind": "apply", "x": 16, "y": 16, "z": 16, "t": 32, "bct": 1, "prec": "f32", "nrhs": 1},
        # The same on the largest lattice, whose time slices of W exceed half of L2.
        {"name": "apply_f32_28x96", "kind": "apply", "x": 28, "y": 28, "z": 28, "t": 96, "bct": 1, "prec": "f32", "nrhs": 1},
        # Half-precision storage on a ragged lattice with the antiperiodic time direction of physics runs.
        {"name": "apply_w16_ragged", "kind": "apply", "x": 14, "y": 18, "z": 11, "t": 27, "bct": -1, "prec": "w16", "nrhs": 1},
        # FP64 with the copy that precompute_W stores by default.
        {"name": "apply_f64_16x32", "kind": "apply", "x": 16, "y": 16, "z": 16, "t": 32, "bct": -1, "prec": "f64", "nrhs": 1},
        # FP64 accuracy from the double-float copy: the true residuals of the solves.
        {"name": "apply_df64_16x32", "kind": "apply", "x": 16, "y": 16, "z": 16, "t": 32, "bct": 1, "prec": "df64", "nrhs": 1},
        # Several sources through the FP32 operator (an odd count on a lattice of the sweep).
        {"name": "apply_multi_f32_12x24", "kind": "apply", "x": 12, "y": 12, "z": 12, "t": 24, "bct": 1, "prec": "f32", "nrhs": 6},
        # The 12 spin-colour sources of one propagator on the tensor cores, the paper's coarse lattice.
        {"name": "apply_tc_20x64", "kind": "apply", "x": 20, "y": 20, "z": 20, "t": 64, "bct": 1, "prec": "tc", "nrhs": 12},
        # A solve with a kept W on a small lattice: bound by launches and the host's round trips.
        {"name": "solve_4x8", "kind": "solve", "x": 4, "y": 4, "z": 4, "t": 8, "bct": 1, "am0": 1.0, "fresh": False},
        # The benchmark's step: W of a new gauge field, a mixed-precision solve, release of W.
        {"name": "step_16x32", "kind": "solve", "x": 16, "y": 16, "z": 16, "t": 32, "bct": 1, "am0": 0.5, "fresh": True},
        # One propagator of a new gauge field: W, then twelve point sources in lockstep on the tensor cores.
        {"name": "propagator_20x64", "kind": "propagator", "x": 20, "y": 20, "z": 20, "t": 64, "bct": 1, "am0": 1.0, "nrhs": 12},
        # One Adam step of the learned preconditioner on a batch of (source, solution) pairs.
        {"name": "train_16x32", "kind": "train", "x": 16, "y": 16, "z": 16, "t": 32, "bct": 1, "batch": 4},
    ]


def _extents(rng, most):
    """Lattice extents whose product is spread over 256 .. `most` sites, odd ones among them."""
    target = math.exp(rng.uniform(math.log(256), math.log(most)))
    while True:
        side = target ** 0.25
        d = [max(4, min(28, round(side * math.exp(rng.uniform(-0.35, 0.25))))) for _ in range(3)]
        t = max(4, min(96, round(target / (d[0] * d[1] * d[2]))))
        if d[0] * d[1] * d[2] * t <= most:
            return {"x": d[0], "y": d[1], "z": d[2], "t": t, "bct": rng.choice([1, -1])}


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "solve", "propagator", "train"])
    if kind == "apply":
        prec = rng.choice(["f32", "f32", "w16", "f64", "df64", "tc"])
        most = {"f32": 28 ** 3 * 96, "w16": 28 ** 3 * 96, "f64": 20 ** 3 * 64, "df64": 20 ** 3 * 64, "tc": 20 ** 3 * 64}[prec]
        case = {"kind": kind, **_extents(rng, most), "prec": prec, "nrhs": 1}
        if prec == "tc":
            case["nrhs"] = rng.randint(1, 16)
        elif prec in ("f32", "w16") and rng.random() < 0.3:
            case.update(_extents(rng, 16 ** 3 * 32))
            case["nrhs"] = rng.randint(2, 12)
        return case
    if kind == "solve":
        return {"kind": kind, **_extents(rng, 16 ** 3 * 32), "am0": round(rng.uniform(0.5, 2.5), 2), "fresh": rng.random() < 0.5}
    if kind == "propagator":
        return {"kind": kind, **_extents(rng, 16 ** 3 * 32), "am0": round(rng.uniform(0.8, 2.5), 2), "nrhs": rng.randint(2, 12)}
    return {"kind": kind, **_extents(rng, 16 ** 3 * 32), "batch": rng.randint(1, 4)}


# ---------------------------------------------------------------------------- inputs
def _sites(case):
    return case["x"] * case["y"] * case["z"] * case["t"]


def _shape(case):
    return (case["t"], case["z"], case["y"], case["x"])


def _generator(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + part)
    return g


def _links(case, seed, eps=0.2):
    """[T, Z, Y, X, 4, 3, 3] SU(3) links: the Gram-Schmidt rows of 1 + i eps H, H Gaussian Hermitian."""
    n = 4 * _sites(case)
    g = _generator(seed, 1)
    a = torch.view_as_complex(torch.randn((n, 3, 3, 2), generator=g, device="cuda", dtype=torch.float64))
    m = 0.5j * eps * (a + a.conj().transpose(1, 2)) + torch.eye(3, dtype=torch.complex128, device="cuda")
    r0 = m[:, 0] / torch.linalg.vector_norm(m[:, 0], dim=1, keepdim=True)
    r1 = m[:, 1] - (r0.conj() * m[:, 1]).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    r2 = torch.stack([r0[:, 1] * r1[:, 2] - r0[:, 2] * r1[:, 1], r0[:, 2] * r1[:, 0] - r0[:, 0] * r1[:, 2],
                      r0[:, 0] * r1[:, 1] - r0[:, 1] * r1[:, 0]], dim=1).conj()
    return torch.stack([r0, r1, r2], dim=1).reshape(_shape(case) + (4, 3, 3)).contiguous()


def _gauss(case, seed, part, lead=(), dtype=torch.complex128):
    """Gaussian spinor field(s) [*lead, T, Z, Y, X, 4, 3]."""
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    shape = tuple(lead) + _shape(case) + (4, 3, 2)
    return torch.view_as_complex(torch.randn(shape, generator=_generator(seed, part), device="cuda", dtype=real))


def _point_sources(case, seed, nrhs):
    """Spin-colour point sources at one site, which the seed chooses."""
    site = int(torch.randint(_sites(case), (1,), generator=_generator(seed, 5), device="cuda"))
    b = torch.zeros((nrhs, _sites(case), 12), dtype=torch.complex128, device="cuda")
    for k in range(nrhs):
        b[k, site, k % 12] = 1.0
    return b.reshape((nrhs,) + _shape(case) + (4, 3))


def _weights(seed):
    """Weights near the identity, as a network has them early in its training."""
    w = torch.view_as_complex(0.05 * torch.randn((LAYERS, 9, 4, 4, 2), generator=_generator(seed, 6), device="cuda",
                                                 dtype=torch.float32)).to(torch.complex128)
    w[:, 0] += 0.6 * torch.eye(4, dtype=torch.complex128, device="cuda")
    return w.to(torch.complex64).to(torch.complex128)


def _bc(case):
    return (1, 1, 1, case["bct"])


def _coeffs(case):
    return dict(COEFFS, am0=case.get("am0", COEFFS["am0"]))


def _fields(case, seed):
    """The source fields of a case."""
    if case["kind"] == "apply":
        lead = () if case["nrhs"] == 1 and case["prec"] != "tc" else (case["nrhs"],)
        return _gauss(case, seed, 2, lead, torch.complex128 if case["prec"] in ("f64", "df64") else torch.complex64)
    if case["kind"] == "solve":
        return _gauss(case, seed, 2)
    if case["kind"] == "propagator":
        return _point_sources(case, seed, case["nrhs"])
    return _gauss(case, seed, 2, (case["batch"],), torch.complex64), _gauss(case, seed, 3, (case["batch"],), torch.complex64)


def prepare(case, seed):
    links = _links(case, seed)
    state = {"case": case, "fields": _fields(case, seed)}
    if case["kind"] == "apply":
        state["W"] = ok.precompute_W(links, _coeffs(case), _bc(case), COPY[case["prec"]])
        state["out"] = torch.empty_like(state["fields"])
    elif case["kind"] == "train":
        state["W"] = ok.precompute_W(links, _coeffs(case), _bc(case), ok.W_F16 | ok.W_LINKS)
        state["net"] = ok.net_create(LAYERS, _weights(seed).cpu().numpy())
    elif case["kind"] == "solve" and not case["fresh"]:
        state["W"] = ok.precompute_W(links, _coeffs(case), _bc(case), ok.W_DF64 | ok.W_F32)
    else:
        state["links"] = links
    return state


def run(state):
    case, fields = state["case"], state["fields"]
    if case["kind"] == "apply":
        if fields.dim() == 7:
            return ok.apply_M_multi(state["W"], fields, state["out"], prec=PREC[case["prec"]])
        return ok.apply_M(state["W"], fields, state["out"], prec=PREC[case["prec"]])
    if case["kind"] == "solve":
        W = state["W"] if not case["fresh"] else ok.precompute_W(state["links"], _coeffs(case), _bc(case), ok.W_DF64 | ok.W_F32)
        x, _ = ok.bicgstab(W, fields, tol=TOL, delta=DELTA)
        if case["fresh"]:
            W.free()
        return x
    if case["kind"] == "propagator":
        W = ok.precompute_W(state["links"], _coeffs(case), _bc(case), ok.W_DF64 | ok.W_F16_TC)
        x, _ = ok.bicgstab_multi(W, fields, tol=TOL, mode=ok.SOLVE_MIXED_TC | ok.SOLVE_DEFECT, delta=DELTA)
        W.free()
        return x
    loss = ok.net_train_step(state["net"], state["W"], fields[0], fields[1], lr=RATE)
    return {"loss": loss, "weights": state["net"].weights.astype(np.complex64)}


# ---------------------------------------------------------------------------- work
def work(case):
    V = _sites(case)
    if case["kind"] == "apply":
        n = case["nrhs"]
        return {"bytes": V * (W_BYTES[case["prec"]] + 2 * n * SPINOR[case["prec"]]), "flops": V * n * APPLY_FLOPS}
    if case["kind"] == "train":
        # per pair: four layers forward and three adjoint ones (links, a field in, a field out), four
        # gradients (links, two fields) and the loss with its seed
        n = case["batch"]
        return {"bytes": V * n * (7 * (288 + 192) + 4 * (288 + 192) + 3 * 96), "flops": V * n * (7 * 4224 + 4 * 4224)}
    # a solve: about this many iterations of two applications and the vector updates between them
    # (rhat; s = r - a v; x and r; p), and two FP64 residuals
    its = 20 + 20 / case["am0"]
    n = case.get("nrhs", 1)
    w = W_BYTES["f32"] if case["kind"] == "solve" else W_BYTES["tc"]
    per_it = 2 * (w + 2 * n * 96) + n * (1 + 3 + 7 + 4) * 96
    built = 576 + W_BYTES["f64"] + w if case.get("fresh", True) else 0
    return {"bytes": V * (its * per_it + 2 * n * (W_BYTES["f64"] + 3 * 192) + built),
            "flops": V * n * (2 * its + 2) * APPLY_FLOPS}


# ---------------------------------------------------------------------------- exact
_AXIS = {0: 3, 1: 2, 2: 1, 3: 0}   # direction (x, y, z, t) -> axis of [T, Z, Y, X, ...]


def _at(f, *steps):
    """The field at x + sum of (mu, n) steps, periodic."""
    for mu, n in steps:
        if n:
            f = torch.roll(f, -n, _AXIS[mu])
    return f


def _dag(m):
    return m.conj().transpose(-1, -2)


def _pauli():
    c = lambda rows: torch.tensor(rows, dtype=torch.complex128, device="cuda")  # noqa: E731
    return [c([[0, 1], [1, 0]]), c([[0, -1j], [1j, 0]]), c([[1, 0], [0, -1]])]


def _kron(s, m):
    """(2 x 2 spin) x (3 x 3 colour field): a 6 x 6 field."""
    return torch.einsum("ab,...cd->...acbd", s, m).reshape(m.shape[:-2] + (6, 6))


def _clover(U, mu, nu):
    a, b = U[mu], U[nu]
    q = a @ _at(b, (mu, 1)) @ _dag(_at(a, (nu, 1))) @ _dag(b)
    plaquette = float(torch.diagonal(q, dim1=-2, dim2=-1).sum(-1).real.mean()) / 3
    q = q + b @ _dag(_at(a, (mu, -1), (nu, 1))) @ _dag(_at(b, (mu, -1))) @ _at(a, (mu, -1))
    q = q + _dag(_at(a, (mu, -1))) @ _dag(_at(b, (mu, -1), (nu, -1))) @ _at(a, (mu, -1), (nu, -1)) @ _at(b, (nu, -1))
    q = q + _dag(_at(b, (nu, -1))) @ _at(a, (nu, -1)) @ _at(b, (mu, 1), (nu, -1)) @ _dag(a)
    return (q - _dag(q)) / 8, plaquette


def _hops(links, c):
    """(offset, 12 x 12 field) for the 27 terms of M psi, one at a time."""
    U = [links[..., mu, :, :] for mu in range(4)]
    F, plaq = {}, 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            F[mu, nu], p = _clover(U, mu, nu)
            plaq += p / 6
    u0 = c["u0"] if c["u0"] > 0 else plaq ** 0.25
    E = [-F[i, 3] for i in range(3)]
    B = [F[1, 2], -F[0, 2], F[0, 1]]
    S = _pauli()
    one = torch.eye(2, dtype=torch.complex128, device="cuda")
    eye6 = torch.eye(6, dtype=torch.complex128, device="cuda")
    ES = sum(_kron(S[i], E[i]) for i in range(3))
    BD = 1j * sum(_kron(S[i], B[i]) for i in range(3))

    def full(a, b, c_, d):
        return torch.cat([torch.cat([a, b], -1), torch.cat([c_, d], -1)], -2)

    def offset(*steps):
        v = [0, 0, 0, 0]
        for mu, n in steps:
            v[mu] += n
        return tuple(v)

    inv2k = 1 / (2 * c["kappa"]) if c["kappa"] > 0 else c["am0"] + 1 + 3 * c["r_s"] * c["zeta"] + 18 * c["c4"]
    d0 = -(c["c_B"] * c["zeta"] + 16 * c["c5"]) / (2 * u0 ** 3) * BD + u0 * inv2k * eye6
    s0 = -(c["c_E"] * c["zeta"]) / (2 * u0 ** 3) * ES
    yield (0, 0, 0, 0), full(d0, s0, -s0, d0)

    u4 = _kron(one, U[3])
    s4 = c["c_EE"] / (2 * u0 ** 4) * (u4 @ _at(ES, (3, 1)) - ES @ u4)
    zero = torch.zeros_like(u4)
    yield offset((3, 1)), full(zero, s4, s4, -u4)
    ub, sb = _dag(_at(u4, (3, -1))), _dag(_at(s4, (3, -1)))
    yield offset((3, -1)), full(-ub, -sb, -sb, zero)
    del u4, s4, ub, sb

    for i in range(3):
        ui = _kron(one, U[i])
        si = _kron(S[i], torch.eye(3, dtype=torch.complex128, device="cuda").expand(U[i].shape))
        s = 0.5 * (c["zeta"] - 2 * c["c1"] - 12 * c["c2"]) * _kron(S[i], U[i])
        s = s + c["c3"] / (2 * u0 ** 4) * (ui @ si @ _at(BD, (i, 1)) - si @ BD @ ui + 2j * _kron(one, B[i] @ U[i]))
        d = -0.5 * (c["r_s"] * c["zeta"] + 8 * c["c4"]) * ui
        for k in range(3):
            if k == i:
                continue
            j = 3 - i - k
            sign = 1.0 if (j - i) % 3 == 1 else -1.0   # epsilon_ijk
            up = U[k] @ _at(U[i], (k, 1)) @ _dag(_at(U[k], (i, 1)))
            dn = _dag(_at(U[k], (k, -1))) @ _at(U[i], (k, -1)) @ _at(U[k], (k, -1), (i, 1))
            d = d + 1j * c["c5"] / 4 * (u0 ** -2 - u0 ** -4) * sign * _kron(S[j], up - dn)
        d = d + c["c5"] / u0 ** 4 * (ui @ _at(BD, (i, 1)) + BD @ ui - 1j * _kron(S[i], U[i] @ _at(B[i], (i, 1)) + B[i] @ U[i]))
        yield offset((i, 1)), full(d, s, s, d)
        d, s = _dag(_at(d, (i, -1))), _dag(_at(s, (i, -1)))
        yield offset((i, -1)), full(d, -s, -s, d)
        uu = U[i] @ _at(U[i], (i, 1))
        d, s = c["c4"] / u0 * _kron(one, uu), (c["c1"] + 2 * c["c2"]) / (2 * u0) * _kron(S[i], uu)
        yield offset((i, 2)), full(d, s, s, d)
        d, s = _dag(_at(d, (i, -2))), _dag(_at(s, (i, -2)))
        yield offset((i, -2)), full(d, -s, -s, d)
        for j in range(i + 1, 3):
            s = c["c2"] / (2 * u0) * _kron(S[i] + S[j], U[i] @ _at(U[j], (i, 1)) + U[j] @ _at(U[i], (j, 1)))
            yield offset((i, 1), (j, 1)), full(zero, s, s, zero)
            s = -_dag(_at(s, (i, -1), (j, -1)))
            yield offset((i, -1), (j, -1)), full(zero, s, s, zero)
            s = c["c2"] / (2 * u0) * _kron(S[i] - S[j], U[i] @ _dag(_at(U[j], (j, -1), (i, 1))) + _dag(_at(U[j], (j, -1))) @ _at(U[i], (j, -1)))
            yield offset((i, 1), (j, -1)), full(zero, s, s, zero)
            s = -_dag(_at(s, (i, -1), (j, 1)))
            yield offset((i, -1), (j, 1)), full(zero, s, s, zero)


def _moved(psi, off, bct):
    """psi [T, Z, Y, X, ...] at x + off, with the boundary sign of the time direction."""
    out = _at(psi, *enumerate(off))
    if bct < 0 and off[3]:
        T = psi.shape[0]
        wraps = torch.div(torch.arange(T, device="cuda") + off[3], T, rounding_mode="floor")
        out = out * torch.where(wraps % 2 == 0, 1.0, -1.0).reshape((T,) + (1,) * (psi.dim() - 1))
    return out


def _exact_apply(links, c, bct, psi):
    """M psi for psi [T, Z, Y, X, 12, n]."""
    out = torch.zeros_like(psi)
    for off, w in _hops(links, c):
        out += w @ _moved(psi, off, bct)
        del w
    return out


def _exact_solve(links, c, bct, b):
    """x with M x = b for b [T, Z, Y, X, 12, n], by BiCGStab for each column to a residual of 1e-13."""
    offs, blocks = [], []
    for off, w in _hops(links, c):
        offs.append(off)
        blocks.append(w)
    M = torch.cat(blocks, -1).reshape(-1, 12, 27 * 12)
    del blocks

    def apply(v):
        return (M @ torch.cat([_moved(v, off, bct) for off in offs], -2).reshape(M.shape[0], 27 * 12, -1)).reshape(v.shape)

    def dot(p, q):
        return (p.conj() * q).sum((0, 1, 2, 3, 4))

    x, bb = torch.zeros_like(b), dot(b, b).real
    for _ in range(6):   # restarts from the true residual
        r = b - apply(x)
        if float((dot(r, r).real / bb).max()) < 1e-26:
            break
        rh, p, rho = r, r, dot(r, r)
        for it in range(400):
            v = apply(p)
            al = rho / dot(rh, v)
            s = r - al * v
            t = apply(s)
            om = dot(t, s) / dot(t, t)
            x = x + al * p + om * s
            r = s - om * t
            if float((dot(r, r).real / bb).max()) < 1e-27:
                break
            new = dot(rh, r)
            p = r + (new / rho) * (al / om) * (p - om * v)
            rho = new
    return x


def _exact_train(links, bct, weights, b, x):
    """The loss and the weights after one Adam step on the pairs b[k], x[k]."""
    A = weights.clone().requires_grad_(True)
    total = 0.0
    for k in range(b.shape[0]):
        v = b[k].to(torch.complex128)
        for l in range(LAYERS):
            out = torch.einsum("st,...tc->...sc", A[l, 0], v)
            for mu in range(4):
                U, unit = links[..., mu, :, :], tuple(int(m == mu) for m in range(4))
                fwd = torch.einsum("...ab,...sb->...sa", U, _moved(v, unit, bct))
                back = _moved(torch.einsum("...ba,...sb->...sa", U.conj(), v), tuple(-m for m in unit), bct)
                out = out + torch.einsum("st,...tc->...sc", A[l, 1 + 2 * mu], fwd)
                out = out + torch.einsum("st,...tc->...sc", A[l, 2 + 2 * mu], back)
            v = out
        xs = x[k].to(torch.complex128)
        loss = (v - xs).abs().square().sum() / xs.abs().square().sum() / b.shape[0]
        loss.backward()
        total += float(loss.detach())
    g = torch.view_as_real(A.grad)   # Adam's first step: both moments are the gradient's
    w = torch.view_as_real(weights) - RATE * g / (g.abs() + 1e-8)
    return {"loss": total, "weights": torch.view_as_complex(w.contiguous())}


def exact(case, seed):
    links, fields = _links(case, seed), _fields(case, seed)
    V, n = _sites(case), case.get("nrhs", 1)
    if case["kind"] == "train":
        return _exact_train(links, case["bct"], _weights(seed), *fields)
    if case["kind"] == "propagator" and V * n > 1_000_000:
        return None   # the dense solve of so many systems takes too long
    lead = fields.dim() == 7
    v = fields.reshape((n,) + _shape(case) + (12,)).permute(1, 2, 3, 4, 5, 0).to(torch.complex128)
    out = (_exact_apply if case["kind"] == "apply" else _exact_solve)(links, _coeffs(case), case["bct"], v)
    out = out.permute(5, 0, 1, 2, 3, 4).reshape((n,) + _shape(case) + (4, 3))
    return out if lead else out[0]
