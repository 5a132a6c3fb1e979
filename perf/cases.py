"""The work whose speed this library is judged by, as cases that a program can run.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of
the same ranges, ``prepare(case, seed)`` what a caller holds before the call (inputs on the GPU, a
Lattice with its links loaded), ``run(state)`` one pass through the public entry points,
``work(case)`` the bytes and operations that the pass cannot do without and ``exact(case, seed)``
the same outputs from plain torch in 64 bits.

Lattice shapes, Ls, masses and the roughness of the links (eps) are those of the tests and of the
benchmark: 4^4 x 8, 8^4 x 8, 12^4 x 12, 16^4 x 16, 16^3 x 32 x 12, 24^3 x 64 x 24, alpha 1 or 2,
M5 1.8, (m1, m2) = (0.04, 1.0) and its neighbours, tolerance 1e-10.
"""
import math

import numpy as np
import torch

from paper_1611_00298_gb300 import eofa
from paper_1611_00298_gb300.autograd import eofa_action

M5 = 1.8
BC_T = -1
PRECS = {"f64": eofa.PREC_F64, "f32": eofa.PREC_MIXED_F32, "f16": eofa.PREC_MIXED_F16}
SYSTEMS = {"dwf": eofa.SYS_DWF, "L": eofa.SYS_EOFA_L, "R": eofa.SYS_EOFA_R}
SPINOR = {"f64": 192, "f32": 96, "f16": 52}
# conjugate-gradient iterations that links of these kinds take to 1e-10 (work() only)
ITERS = 300


def _case(name, kind, dims, Ls, **kw):
    X, Y, Z, T = dims
    return dict({"name": name, "kind": kind, "X": X, "Y": Y, "Z": Z, "T": T, "Ls": Ls, "alpha": 2.0}, **kw)


def listed():
    return [
        # one small EOFA solve (action of a test lattice): launches and latency are all there is
        _case("solve_f32_4x4x4x4_8", "solve", (4, 4, 4, 4), 8, prec="f32", system="L", eps=0.3, m1=0.04, m2=1.0),
        # mixed-precision propagator solve of one source, the ordinary size
        _case("solve_f32_16x16x16x16_16", "solve", (16, 16, 16, 16), 16, prec="f32", system="dwf", eps=0.6, m1=0.04, m2=1.0),
        # an HMC force's right-handed solve on the large lattice: where trajectories spend their time
        _case("solve_f32_24x24x24x32_24", "solve", (24, 24, 24, 32), 24, prec="f32", system="R", eps=0.7, m1=0.0362, m2=1.0),
        # the same kind of solve with 16-bit storage of the inner fields
        _case("solve_f16_16x16x16x32_16", "solve", (16, 16, 16, 32), 16, prec="f16", system="L", eps=0.5, m1=0.04, m2=0.2),
        # an all-FP64 solve (reference runs, the Metropolis action when mixed precision is not wanted)
        _case("solve_f64_12x12x12x12_12", "solve", (12, 12, 12, 12), 12, prec="f64", system="dwf", eps=0.5, m1=0.04, m2=1.0),
        # several mass pairs, left and right systems on one small lattice, solved together from host arrays
        _case("batched_f32_8x8x8x8_8", "batched", (8, 8, 8, 8), 8, prec="f32", nsys=8, eps=0.5, m1=0.2, m2=0.6),
        # the Dirac operator and its adjoint on whole FP64 fields (measurements, other solvers)
        _case("apply_f64_16x16x16x32_12", "apply", (16, 16, 16, 32), 12, eps=0.5, m1=0.04),
        # the even-odd kernel behind every solve, benchmark lattice: both parities, operator and adjoint
        _case("schur_f32_24x24x24x64_24", "schur", (24, 24, 24, 64), 24, prec="f32", eps=0.7, m1=0.0362),
        # the same with 16-bit storage, an uneven lattice and an Ls that is no multiple of 8
        _case("schur_f16_6x10x14x18_10", "schur", (6, 10, 14, 18), 10, prec="f16", eps=0.5, m1=0.04),
        # differentiation of the action through the autograd wrapper: links in, gradient out
        _case("grad_f32_16x16x16x32_12", "grad", (16, 16, 16, 32), 12, prec="f32", alpha=1.0, eps=0.5, m1=0.04, m2=1.0),
        # the adjoint (force) kernel alone, from given solutions
        _case("force_24x24x24x32_24", "force", (24, 24, 24, 32), 24, eps=0.7),
        # a pure-gauge force-gradient trajectory, the inner time scale of an HMC run
        _case("gauge_md_16x16x16x32", "gauge_md", (16, 16, 16, 32), 4, eps=0.3, beta=5.7, nsteps=4),
    ]


def _dims(rng, lo, hi):
    """Even extents whose volume is spread over the logarithm of [lo, hi]."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    d = [2 * rng.randint(2, 12) for _ in range(4)]
    for _ in range(64):
        v = d[0] * d[1] * d[2] * d[3]
        if want / 1.3 <= v <= want * 1.3:
            break
        k = rng.randrange(4)
        d[k] = min(32, d[k] + 2) if v < want else max(4, d[k] - 2)
    return tuple(d)


def draw(rng):
    case = _draw(rng)
    del case["name"]
    return case


def _draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batched", "apply", "schur", "schur", "grad", "force", "gauge_md"])
    Ls = rng.choice([8, 12, 16, 24, rng.randint(4, 32)])
    alpha = rng.choice([1.0, 2.0, 2.0])
    eps = rng.choice([0.3, 0.5, 0.6, 0.7])
    m1, m2 = rng.choice([(0.04, 1.0), (0.04, 0.2), (0.2, 0.6), (0.6, 1.0)])
    if kind == "solve":
        prec = rng.choice(["f32", "f32", "f16", "f64"])
        dims = _dims(rng, 256, 20000 if prec == "f64" else 200000)
        return _case("", kind, dims, min(Ls, 12) if prec == "f64" else Ls, prec=prec, alpha=alpha, eps=eps, m1=m1,
                     m2=m2, system=rng.choice(["dwf", "L", "R"]))
    if kind == "batched":
        return _case("", kind, _dims(rng, 256, 10000), min(Ls, 16), prec=rng.choice(["f32", "f16"]),
                     nsys=rng.randint(2, 12), alpha=alpha, eps=eps, m1=m1, m2=m2)
    if kind == "grad":
        return _case("", kind, _dims(rng, 256, 65536), min(Ls, 16), prec="f32", alpha=alpha, eps=eps, m1=m1, m2=m2)
    if kind == "gauge_md":
        return _case("", kind, _dims(rng, 256, 200000), 4, eps=rng.choice([0.1, 0.3]), beta=rng.choice([5.5, 5.7, 6.0]),
                     nsteps=rng.randint(2, 4))
    dims = _dims(rng, 256, 300000)
    if kind == "force":
        return _case("", kind, dims, Ls, eps=eps)
    if kind == "apply":
        return _case("", kind, dims, Ls, alpha=alpha, eps=eps, m1=m1)
    return _case("", kind, dims, Ls, prec=rng.choice(["f32", "f16", "f64"]), alpha=alpha, eps=eps, m1=m1)


# ---------------------------------------------------------------- inputs

def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream * 7919) % (1 << 62))
    return g


def _randc(shape, gen):
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=gen) * math.sqrt(2.0)


def _hermitian(n, gen, dtype):
    """sum_a h_a lambda_a with h_a ~ N(0, 1): traceless Hermitian 3x3 matrices."""
    h = torch.randn((n, 8), dtype=torch.float64, device="cuda", generator=gen).to(dtype.to_real())
    r3 = 1.0 / math.sqrt(3.0)
    H = torch.zeros((n, 3, 3), dtype=dtype, device="cuda")
    for (a, b), (k, l) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
        H[:, a, b] = torch.complex(h[:, k], -h[:, l])
        H[:, b, a] = torch.complex(h[:, k], h[:, l])
    H[:, 0, 0] = h[:, 2] + r3 * h[:, 7]
    H[:, 1, 1] = -h[:, 2] + r3 * h[:, 7]
    H[:, 2, 2] = -2.0 * r3 * h[:, 7]
    return H


def _links(case, seed):
    """Links exp(i eps sum_a h_a lambda_a), made SU(3) to rounding; shape (T, Z, Y, X, 4, 3, 3)."""
    shape = (case["T"], case["Z"], case["Y"], case["X"], 4, 3, 3)
    H = _hermitian(math.prod(shape[:5]), _gen(seed, 1), torch.complex64)
    A = (0.125j * case["eps"]) * H
    E = torch.eye(3, dtype=A.dtype, device="cuda").expand_as(A)
    out, term = E, E
    for n in range(1, 11):
        term = term @ A / n
        out = out + term
    for _ in range(3):
        out = out @ out
    r = out.to(torch.complex128)
    r0 = r[:, 0] / torch.linalg.vector_norm(r[:, 0], dim=-1, keepdim=True)
    r1 = r[:, 1] - (r0.conj() * r[:, 1]).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    return torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], dim=1).reshape(shape)


def _dims_of(case):
    return (case["X"], case["Y"], case["Z"], case["T"])


def _shape5(case):
    return (case["Ls"], case["T"], case["Z"], case["Y"], case["X"], 4, 3)


def _systems(case):
    """The mass pairs and sides of a batched case."""
    pairs = [(case["m1"] * f, min(1.0, case["m2"] * f)) for f in (0.2, 0.5, 1.0, 1.5, 0.35, 0.75)]
    return [(("L", "R")[i % 2], *pairs[(i // 2) % len(pairs)]) for i in range(case["nsys"])]


def _fields(case, seed):
    """The case's random fields other than the links."""
    kind, n = case["kind"], 1
    if kind in ("solve", "apply", "schur"):
        return [_randc(_shape5(case), _gen(seed, 2))]
    if kind == "batched":
        return [_randc(_shape5(case), _gen(seed, 2 + i)) for i in range(case["nsys"])]
    if kind == "grad":
        return [_randc(_shape5(case)[1:], _gen(seed, 2))]
    if kind == "force":
        return [_randc(_shape5(case), _gen(seed, 2 + i)) for i in range(2)]
    n = math.prod(_dims_of(case)) * 4
    return [0.5 * _hermitian(n, _gen(seed, 2), torch.complex128).reshape(_shape5(case)[1:5] + (4, 3, 3))]


def prepare(case, seed):
    kind = case["kind"]
    U = _links(case, seed)
    f = _fields(case, seed)
    lat = eofa.Lattice(_dims_of(case), case["Ls"], bc_t=BC_T)
    s = {"case": case, "lat": lat}
    if kind == "grad":
        s["U"] = torch.view_as_real(U).requires_grad_(True)
        s["phi"] = f[0]
        return s
    lat.gauge_load_dev(U)
    if kind == "solve":
        s.update(b=f[0], x=torch.zeros_like(f[0]))
    elif kind == "batched":
        s["b"] = [t.cpu().numpy() for t in f]
        s["x"] = [np.zeros_like(b) for b in s["b"]]
        s["params"] = [lat.solve_params(system=SYSTEMS[side], alpha=case["alpha"], M5=M5, m1=a, m2=b,
                                        shift=0.0 if side == "L" else -1.0, precision=PRECS[case["prec"]], tol=1e-10)
                       for side, a, b in _systems(case)]
    elif kind == "apply":
        s.update(psi=f[0], out=torch.empty_like(f[0]), adj=torch.empty_like(f[0]))
    elif kind == "schur":
        nb = lat.field_bytes(PRECS[case["prec"]])
        s["half"] = [torch.empty(nb, dtype=torch.uint8, device="cuda") for _ in range(6)]
        lat.pack_dev(PRECS[case["prec"]], f[0], s["half"][0], s["half"][1])
    elif kind == "force":
        s.update(chi=f, F=torch.empty(lat.shapeU, dtype=torch.complex128, device="cuda"))
    else:
        s.update(U=U, P0=f[0], P=torch.empty_like(f[0]), U1=torch.empty_like(U))
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- the passes

FORCE_K = 0.9  # the coefficient k of the force cases


def _views(case, buf):
    """A half-checkerboard field as numbers: FP16 storage has its per-site scales behind the halves."""
    if case["prec"] == "f64":
        return [buf.view(torch.float64)]
    if case["prec"] == "f32":
        return [buf.view(torch.float32)]
    n = math.prod(_dims_of(case)) // 2 * case["Ls"]
    return [buf[:48 * n].view(torch.float16), buf[48 * n:52 * n].view(torch.float32)]


def run(state):
    case, lat = state["case"], state["lat"]
    kind, alpha = case["kind"], case["alpha"]
    if kind == "solve":
        lat.solve_dev(state["b"], state["x"], system=SYSTEMS[case["system"]], alpha=alpha, M5=M5, mf=case["m1"],
                      m1=case["m1"], m2=case["m2"], shift=-1.0 if case["system"] == "R" else 0.0,
                      precision=PRECS[case["prec"]], tol=1e-10)
        return state["x"]
    if kind == "batched":
        eofa.solve_batched([lat] * case["nsys"], state["params"], state["b"], state["x"])
        return state["x"]
    if kind == "apply":
        lat.dwf_apply_dev(state["psi"], state["out"], alpha, M5, case["m1"])
        lat.dwf_apply_dev(state["psi"], state["adj"], alpha, M5, case["m1"], dagger=True)
        return [state["out"], state["adj"]]
    if kind == "schur":
        prec, half = PRECS[case["prec"]], state["half"]
        for dag in (0, 1):
            lat.schur_hop_dev(prec, 0, dag, half[1], half[2 + 2 * dag], alpha, M5, case["m1"])
            lat.schur_hop_dev(prec, 1, dag, half[0], half[3 + 2 * dag], alpha, M5, case["m1"])
        return [v for h in half[2:] for v in _views(case, h)]
    if kind == "grad":
        S = eofa_action(state["U"], state["phi"], lat, alpha, M5, case["m1"], case["m2"],
                        precision=PRECS[case["prec"]], tol=1e-10)
        (G,) = torch.autograd.grad(S, state["U"])
        return [S.detach(), G]
    if kind == "force":
        lat.force_from_chi_dev(FORCE_K, state["chi"][0], state["chi"][1], state["F"])
        return state["F"]
    state["P"].copy_(state["P0"])
    lat.gauge_load_dev(state["U"])
    info = lat.hmc_trajectory_dev(state["P"], U=state["U1"], beta=case["beta"], integrator=eofa.INT_FG_QPQPQ,
                                  nsteps=case["nsteps"], tau=0.25 * case["nsteps"])
    return [state["P"], state["U1"], info["H0"]]


def work(case):
    """One pass's inputs read once and outputs written once; the arithmetic of the standard counts
    (1320 operations a site for the hop, four hops and 240 operations of vector work a
    conjugate-gradient iteration and site pair)."""
    V = math.prod(_dims_of(case))
    Ls, kind, links = case["Ls"], case["kind"], 4 * V * 144
    n5 = V * Ls
    cg = ITERS * (n5 // 2) * (4 * 1320 + 240)
    if kind == "solve":
        return {"bytes": links + 2 * 192 * n5, "flops": cg}
    if kind == "batched":
        return {"bytes": links + 2 * 192 * n5 * case["nsys"], "flops": cg * case["nsys"]}
    if kind == "apply":
        return {"bytes": links + 3 * 192 * n5, "flops": 2 * n5 * (1320 + 96)}
    if kind == "schur":
        sp = SPINOR[case["prec"]]
        return {"bytes": (links if case["prec"] == "f64" else links // 2) + 3 * sp * n5, "flops": 2 * n5 * (1320 + 168)}
    if kind == "grad":
        return {"bytes": 2 * links + 192 * V, "flops": 2 * cg}
    if kind == "force":
        return {"bytes": 2 * links + 2 * 192 * n5, "flops": 2 * 4 * n5 * (48 + 144)}
    # 4 forces a step of 4 links a site: 18 products of 3x3 matrices (198 operations each)
    return {"bytes": 4 * links, "flops": 4 * case["nsteps"] * 4 * V * 19 * 198}


# ---------------------------------------------------------------- plain torch in 64 bits

def _gammas():
    """gamma_mu in the chiral basis, [[0, A], [A^+, 0]]."""
    As = [[[0, -1j], [-1j, 0]], [[0, -1], [1, 0]], [[-1j, 0], [0, 1j]], [[1, 0], [0, 1]]]
    out = []
    for A in As:
        A = torch.tensor(A, dtype=torch.complex128, device="cuda")
        g = torch.zeros((4, 4), dtype=torch.complex128, device="cuda")
        g[:2, 2:], g[2:, :2] = A, A.conj().T
        out.append(g)
    return out


def _shift(f, mu, sign):
    """f(x + sign mu) of a (s, T, Z, Y, X, ...) field, with the time boundary's sign."""
    g = torch.roll(f, -sign, dims=4 - mu)
    if mu == 3:
        g[:, -1 if sign > 0 else 0] *= BC_T
    return g


def _colour(M, f):
    """M(x) f(x) in colour, term by term."""
    return torch.stack([sum(M[None, ..., a, b, None] * f[..., b] for b in range(3)) for a in range(3)], dim=-1)


def _hop(U, psi, dagger=False):
    sgn = -1.0 if dagger else 1.0
    out = torch.zeros_like(psi)
    for mu, g in enumerate(_gammas()):
        Um = U[..., mu, :, :]
        f = _colour(Um, _shift(psi, mu, 1))
        out -= 0.5 * (f - sgn * torch.einsum("ij,...jc->...ic", g, f))
        Ub = torch.roll(Um, 1, dims=3 - mu).conj().transpose(-1, -2)
        f = _colour(Ub, _shift(psi, mu, -1))
        out -= 0.5 * (f + sgn * torch.einsum("ij,...jc->...ic", g, f))
    return out


def _s_matrices(Ls, alpha, m):
    """(D-tilde, 1 - L) of each chirality as dense Ls x Ls matrices."""
    L = np.zeros((Ls, Ls))
    for s in range(1, Ls):
        L[s, s - 1] = 1.0
    L[0, Ls - 1] += -m
    c, d = 0.5 * alpha, 0.5
    one = np.eye(Ls)
    return [(d * (one - X) + c * (one + X), one - X) for X in (L, L.T)]


def _on_s(mats, psi):
    """The chirality-wise s-matrices applied to a field."""
    up, lo = (torch.einsum("st,t...->s...", torch.as_tensor(M, dtype=torch.complex128, device="cuda"), h)
              for M, h in zip(mats, (psi[..., :2, :], psi[..., 2:, :])))
    return torch.cat([up, lo], dim=-2)


def _g5r5(psi):
    out = psi.flip(0).clone()
    out[..., 2:, :] *= -1
    return out


def _cgnr(A, Ad, f):
    """Least-squares conjugate gradients to the rounding of 64 bits."""
    x = torch.zeros_like(f)
    for _ in range(2):
        r = f - A(x)
        s = Ad(r)
        p, gam = s.clone(), float((s.abs() ** 2).sum())
        stop = 1e-28 * gam
        for _ in range(4000):
            q = A(p)
            a = gam / float((q.abs() ** 2).sum())
            x, r = x + a * p, r - a * q
            s = Ad(r)
            new = float((s.abs() ** 2).sum())
            if new <= stop:
                break
            p, gam = s + (new / gam) * p, new
    return x


def _solution(U, b, case, side, m1, m2):
    """x of D_DWF x = b or of (H(m) + shift Delta P) x = b (left: shift 0, right: shift -1)."""
    Ls, alpha = case["Ls"], case["alpha"]
    T = _s_matrices(Ls, alpha, m2 if side == "R" else m1)
    G = [((4 - M5) * D + E) @ np.linalg.inv(D) for D, E in T]
    if side == "R":
        c, d = 0.5 * alpha, 0.5
        beta = -(c - d) / (c + d)
        k = alpha * (m2 - m1) / ((1 + m1 * beta ** Ls) * (1 + m2 * beta ** Ls))
        Om = np.array([beta ** (Ls - 1 - s) for s in range(Ls)]) / (c + d)
        G[0] = G[0] - k * np.outer(Om[::-1], Om)
    f = b if side == "dwf" else _g5r5(b)
    y = _cgnr(lambda v: _hop(U, v) + _on_s(G, v), lambda v: _hop(U, v, True) + _on_s([M.T for M in G], v), f)
    return _on_s([np.linalg.inv(D) for D, _ in T], y) if side == "dwf" else y


def _half(case, psi, parity):
    """A field's sites of one parity as (site, s, 12), the order of the packed half fields."""
    Z = [torch.arange(case[k], device="cuda") for k in ("T", "Z", "Y", "X")]
    par = (Z[0][:, None, None, None] + Z[1][:, None, None] + Z[2][:, None] + Z[3]) % 2
    return psi.reshape(case["Ls"], -1, 12)[:, (par == parity).reshape(-1)].transpose(0, 1)


def _packed(case, h):
    """A half field's numbers in the library's layout of the case's precision."""
    per = {"f64": 1, "f32": 2, "f16": 4}[case["prec"]]
    v = torch.view_as_real(h.contiguous()).reshape(h.shape[0], h.shape[1], 12 // per, 2 * per)
    if case["prec"] != "f16":
        return [v.permute(0, 2, 1, 3).reshape(-1)]
    scale = v.abs().amax(dim=(2, 3))
    return [(v / scale[..., None, None]).permute(0, 2, 1, 3).reshape(-1), scale.reshape(-1)]


def _traceless_force(U, G):
    """The force F = sum_a F^a T^a of a real function with gradient G = d/dRe U + i d/dIm U."""
    X = -U @ G.conj().transpose(-1, -2)
    A = X - X.conj().transpose(-1, -2)
    A = A - torch.diagonal(A, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3 * torch.eye(3, dtype=A.dtype, device=A.device)
    return -0.25j * A


def _gauge_action(U, beta):
    S = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            A = U[..., mu, :, :] @ torch.roll(U[..., nu, :, :], -1, dims=3 - mu)
            B = U[..., nu, :, :] @ torch.roll(U[..., mu, :, :], -1, dims=3 - nu)
            S = S + (beta / 3.0) * (3.0 - (A * B.conj()).real.sum((-1, -2))).sum()
    return S


def _gauge_md(case, U, P):
    """QPQPQ with the displaced-link force gradient."""
    h, beta = 0.25, case["beta"]
    H0 = float((P.abs() ** 2).sum() + _gauge_action(U, beta))
    lam, z = 0.5 - math.sqrt(3.0) / 6.0, (2.0 - math.sqrt(3.0)) / 12.0 * h * h

    def force(U):
        V = U.clone().requires_grad_(True)
        (G,) = torch.autograd.grad(_gauge_action(V, beta), V)
        return _traceless_force(U, G)

    def drift(U, Q, t):
        return torch.linalg.matrix_exp(1j * t * Q) @ U

    for _ in range(case["nsteps"]):
        for t in (lam * h, (1 - 2 * lam) * h):
            U = drift(U, P, t)
            P = P - (h / 2) * force(drift(U, force(U), -z))
        U = drift(U, P, lam * h)
    return [P, U, H0]


def exact(case, seed):
    kind, n5 = case["kind"], math.prod(_dims_of(case)) * case["Ls"]
    if kind == "grad" or (kind in ("solve", "batched") and n5 * case.get("nsys", 1) > 300000):
        return None  # conjugate gradients in plain torch take minutes there
    U, f = _links(case, seed), _fields(case, seed)
    if kind == "solve":
        return _solution(U, f[0], case, case["system"], case["m1"], case["m2"])
    if kind == "batched":
        return [_solution(U, b, case, *s) for b, s in zip(f, _systems(case))]
    if kind == "apply":
        D, E = zip(*_s_matrices(case["Ls"], case["alpha"], case["m1"]))
        Dw = [(4 - M5) * d + e for d, e in zip(D, E)]
        out = _hop(U, _on_s(D, f[0])) + _on_s(Dw, f[0])
        return [out, _on_s([d.T for d in D], _hop(U, f[0], True)) + _on_s([d.T for d in Dw], f[0])]
    if kind == "schur":
        Gi = [d @ np.linalg.inv((4 - M5) * d + e) for d, e in _s_matrices(case["Ls"], case["alpha"], case["m1"])]
        out = []
        for dag in (0, 1):
            v = _on_s([g.T for g in Gi] if dag else Gi, _hop(U, f[0], bool(dag)))
            for par in (0, 1):
                out += _packed(case, _half(case, v, par))
        return out
    if kind == "force":
        V = U.clone().requires_grad_(True)
        S = sum(k * (_g5r5(c).conj() * _hop(V, c)).sum().real for k, c in zip((FORCE_K, -FORCE_K), f))
        (G,) = torch.autograd.grad(S, V)
        return _traceless_force(U, G)
    return _gauge_md(case, U, f[0])
