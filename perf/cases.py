"""Performance cases of the library: what a lattice program has it do, through the public `Wilson` handle.

A case is one call (or, for `md`, the calls of one molecular-dynamics step) on one lattice:

* `apply`: one operator apply, as a program with its own Krylov solver, residual check or
  measurement code makes it: M, T^-1 and the Schur operator M-hat, in FP64 and FP32, adjoint or not;
* `solve`: M x = rhs to a 1e-10 FP64 true residual by one of the library's methods and precisions;
* `md`: a new gauge field is loaded, then the pseudofermion force and the determinant term with its
  force are taken from it, as every step of hybrid Monte Carlo does.

Every handle works on a stream of its own, as bench.py's do, and all of a pass runs on that stream.
Inputs come from the seed: links near unity with Gaussian algebra coefficients (the synthetic stand-ins
for a thermalised anisotropic ensemble), Gaussian sources, or the twelve spin-colour point sources of
a propagator. Couplings are those of the repository's workloads: kappa_s is a fraction of the free
critical value 1 / (2 (xi + 3)) and kappa_t = xi kappa_s.

FP32 applies carry FP32 rounding in their complex128 output arrays; the program that asked for them
keeps them as complex64.
"""

import math

import torch

from paper_0910_0992_gb300 import _lib as wf

METHODS = {"unprec": wf.WF_UNPREC, "eo4d": wf.WF_EO4D, "temporal": wf.WF_TEMPORAL,
           "temporal_schur": wf.WF_TEMPORAL_SCHUR, "temporal_ilu": wf.WF_TEMPORAL_ILU}
PRECISIONS = {"fp64": wf.WF_FP64, "fp32": wf.WF_FP32, "fp16mix": wf.WF_FP16MIX}
TOL = 1e-10


def _apply(name, op, L, T, nrhs, f32, dagger=False):
    return {"name": name, "kind": "apply", "op": op, "L": L, "T": T, "nrhs": nrhs, "f32": f32, "dagger": dagger,
            "xi": 3.5, "crit": 0.9, "eps": 0.25}


def _solve(name, method, precision, L, T, nrhs, xi=3.5, crit=0.9, eps=0.25, sources="gaussian"):
    return {"name": name, "kind": "solve", "method": method, "precision": precision, "L": L, "T": T, "nrhs": nrhs,
            "xi": xi, "crit": crit, "eps": eps, "sources": sources}


def listed():
    return [
        # the smallest lattice of the test workloads: a call is launches and one wait
        _apply("schur_f64_4c16", "schur", 4, 16, 1, False),
        # the paper's lattice with one source: the operator inside a program's own CG
        _apply("schur_f32_16c128", "schur", 16, 128, 1, True),
        # the adjoint on a propagator's twelve sources, the largest lattice of the benchmark
        _apply("schur_dag_f32_24c128_x12", "schur", 24, 128, 12, True, True),
        # a program's own true residual: M in FP64, on the sweep's 48-slot lines with its four sources
        _apply("M_f64_12c48_x4", "M", 12, 48, 4, False),
        # the time-line inverse alone on an odd, padded line and an odd number of sources
        _apply("Tinv_f32_10c37_x3", "Tinv", 10, 37, 3, True),
        # the headline: a propagator (twelve point sources) on 24^3 x 128
        _solve("solve_24c128_x12", "temporal_schur", "fp32", 24, 128, 12, crit=0.97, eps=0.2, sources="point"),
        # one source on the paper's lattice, where a solve is bound by latency as much as by bandwidth
        _solve("solve_16c128", "temporal_schur", "fp32", 16, 128, 1),
        # all-FP64 solve on a small lattice, as tests and reference runs make it
        _solve("solve_f64_8c32_x2", "temporal_schur", "fp64", 8, 32, 2, xi=3.0),
        # the 4-D even-odd comparator on the anisotropy sweep's 96-slot lattice with its four sources
        _solve("solve_eo4d_16c96_x4", "eo4d", "fp32", 16, 96, 4, xi=3.0),
        # the clover operator with partial temporal preconditioning and 3-D ILU
        _solve("solve_clover_ilu_16c128", "temporal_ilu", "fp32", 16, 128, 1),
        # the clover operator with its whole time-line block inverted
        _solve("solve_clover_full_16c128", "full_sw", "fp32", 16, 128, 1),
        # one molecular-dynamics step on the force workload's lattice
        {"name": "md_8c32", "kind": "md", "L": 8, "T": 32, "precision": "fp32", "xi": 3.0, "crit": 0.9, "eps": 0.25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "solve", "solve", "md"])
    if kind == "md":
        return {"kind": "md", "L": 2 * _log_int(rng, 2, 8), "T": _log_int(rng, 8, 64),
                "precision": rng.choice(["fp32", "fp64"]), "xi": 3.0, "crit": 0.9, "eps": 0.25}
    if kind == "apply":
        c = _apply("", rng.choice(["schur", "schur", "M", "Tinv"]), 2 * _log_int(rng, 2, 12), _log_int(rng, 8, 160),
                   _log_int(rng, 1, 12), rng.random() < 0.6, rng.random() < 0.5)
    else:
        method = rng.choice(["temporal_schur", "temporal_schur", "temporal_schur", "eo4d", "temporal_ilu", "full_sw"])
        T = _log_int(rng, 8, 128)
        prec = rng.choice(["fp32", "fp32", "fp64", "fp16mix"]) if method == "temporal_schur" else "fp32"
        c = _solve("", method, prec, 2 * _log_int(rng, 2, 8), T - T % 2 if method == "eo4d" else T,
                   _log_int(rng, 1, 12), xi=rng.choice([3.0, 3.5, 4.5, 6.0]))
        # FP64 and the clover methods cost several times an FP32 Wilson solve
        if prec == "fp64" or method in ("temporal_ilu", "full_sw"):
            c["nrhs"] = min(c["nrhs"], 3)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------
def _kappas(case):
    ks = case["crit"] / (2.0 * (case["xi"] + 3.0))
    return ks, case["xi"] * ks


def _gauge(L, T, eps, gen):
    """U[t][z][y][x][mu][3][3]: rows of 1 + i eps H - (eps H)^2 / 2, H a Gaussian element of su(3),
    orthonormalised (the third row the conjugate cross product of the first two)."""
    n = T * L ** 3 * 4
    h = torch.randn(n, 8, dtype=torch.float64, device="cuda", generator=gen) * (0.5 * eps)
    H = torch.zeros(n, 3, 3, dtype=torch.complex128, device="cuda")
    d = h[:, 7] / math.sqrt(3.0)
    H[:, 0, 0], H[:, 1, 1], H[:, 2, 2] = h[:, 2] + d, d - h[:, 2], -2.0 * d
    for (a, b), (re, im) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
        H[:, a, b] = torch.complex(h[:, re], -h[:, im])
        H[:, b, a] = H[:, a, b].conj()
    r0 = 1j * H[:, 0] - 0.5 * (H[:, 0, :, None] * H).sum(1)
    r1 = 1j * H[:, 1] - 0.5 * (H[:, 1, :, None] * H).sum(1)
    r0[:, 0] += 1.0
    r1[:, 1] += 1.0
    r0 /= torch.linalg.vector_norm(r0, dim=1, keepdim=True)
    for _ in range(2):
        r1 -= (r0.conj() * r1).sum(1, keepdim=True) * r0
        r1 /= torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    H[:, 0], H[:, 1], H[:, 2] = r0, r1, torch.linalg.cross(r0, r1, dim=1).conj()
    return H.reshape(T, L, L, L, 4, 3, 3)


def _gaussian(shape, gen):
    return torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=gen)


def _inputs(case, seed):
    """(U, the sources or None) of a case: everything that the seed decides."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    L, T = case["L"], case["T"]
    U = _gauge(L, T, case["eps"], gen)
    if case["kind"] == "md" or case.get("op") == "schur":
        src = _gaussian((case.get("nrhs", 1), T, L ** 3 // 2, 4, 3), gen)
    elif case.get("sources") == "point":
        src = torch.zeros(case["nrhs"], T * L ** 3, 12, dtype=torch.complex128, device="cuda")
        site = int(torch.randint(T * L ** 3, (1,), device="cuda", generator=gen))
        for k in range(case["nrhs"]):
            src[k, site, k % 12] = 1.0
        src = src.reshape(case["nrhs"], T, L, L, L, 4, 3)
    else:
        src = _gaussian((case["nrhs"], T, L, L, L, 4, 3), gen)
    return U, src


# tree-level clover coefficients of the repository's clover benchmark on 16^3 x 128, xi = 3.5
CLOVER = (0.324, 0.699)


def _is_clover(case):
    return case.get("method") in ("temporal_ilu", "full_sw")


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    ks, kt = _kappas(case)
    U, st.src = _inputs(case, seed)
    st.stream = torch.cuda.Stream()
    st.w = wf.Wilson(case["L"], case["T"], ks, kt, case["xi"], -1)
    st.w.set_stream(st.stream.cuda_stream)
    torch.cuda.synchronize()  # the handle's stream reads what the current one made
    if case["kind"] == "md":
        st.U = U  # the field of the step, loaded by every pass
    elif _is_clover(case):
        st.w.load_gauge_clover(U, *CLOVER)
    else:
        st.w.load_gauge(U)
    return st


def run(st):
    case, w = st.case, st.w
    with torch.cuda.stream(st.stream):
        if case["kind"] == "apply":
            f = {"schur": w.apply_schur, "M": w.apply_M, "Tinv": w.apply_Tinv}[case["op"]]
            out = f(st.src, dagger=case["dagger"], f32=case["f32"])
            return out.to(torch.complex64) if case["f32"] else out
        if case["kind"] == "solve":
            if case["method"] == "full_sw":
                x, _, _, status = w.solve_full_sw(st.src, TOL, PRECISIONS[case["precision"]])
            else:
                x, _, _, status = w.solve(st.src, TOL, METHODS[case["method"]], PRECISIONS[case["precision"]])
            if status != wf.WF_OK:
                raise RuntimeError("the solve did not converge")
            return x
        w.load_gauge(st.U)
        shape = (case["T"], case["L"], case["L"], case["L"], 4, 8)
        F = torch.empty(shape, dtype=torch.float64, device="cuda")
        D = torch.empty(shape, dtype=torch.float64, device="cuda")
        action, _ = wf.wf_force(w.h, st.src, F, PRECISIONS[case["precision"]], 1e-12)
        logdet = w.temporal_logdet(D)
        return {"action": action, "force": F, "logdet": logdet, "logdet_force": D}


# ---------------------------------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------------------------------
def _schur_flops(L, T):
    return (3432 * T - 576) * (L ** 3 // 2)  # the paper's count (App. B), per source


def _iterations(case):
    """CGNR iterations a solve of these couplings needs to 1e-10 (measured, rounded)."""
    if case["crit"] > 0.95:
        return 60
    return {"temporal_schur": 30, "eo4d": 54, "temporal_ilu": 34, "full_sw": 30}[case["method"]]


def work(case):
    """Inputs read once, outputs written once; a solve's inner vectors are counted once per operator
    apply, in the precision of the applies (its iterations are what the method cannot do without)."""
    L, T = case["L"], case["T"]
    V, n = L ** 3 * T, case.get("nrhs", 1)
    if case["kind"] == "apply":
        real = 4 if case["f32"] else 8
        links = 3 * (12 if case["f32"] else 18) * real
        if case["op"] == "schur":
            return {"bytes": V * links + n * V // 2 * 384, "flops": n * _schur_flops(L, T)}
        if case["op"] == "M":
            return {"bytes": V * links + n * V * 384, "flops": n * V * 1368}
        return {"bytes": n * V * 384, "flops": n * V * 4 * 18}
    applies = 2 * (_iterations(case) if case["kind"] == "solve" else 32)
    real = 8 if case["precision"] == "fp64" else 4
    links = 3 * (18 if real == 8 else 12) * real
    if case["kind"] == "md":
        return {"bytes": V * (576 + 512) + V // 2 * 192 + applies * (V * links + V * 12 * 2 * real // 2 * 2),
                "flops": applies * _schur_flops(L, T) + V * 4000}
    per_apply = V * links + n * (V // 2) * 12 * 2 * real * 2
    if _is_clover(case):
        per_apply = per_apply + V * 72 * 2 * real + n * (V // 2) * 12 * 2 * real * 2
    return {"bytes": n * V * 384 + applies * per_apply, "flops": n * (applies * _schur_flops(L, T) + 2 * V * 1368)}


# ---------------------------------------------------------------------------------------------------
# The same results in 64 bits by plain torch: fields as [spin][colour][t][z][y][x], links as
# [row][col][t][z][y][x] per direction (x, y, z, t); gamma_k = [[0, -i sigma_k], [i sigma_k, 0]]
# ---------------------------------------------------------------------------------------------------
_AXIS = (-1, -2, -3, -4)  # of x, y, z, t


def _fields(U):
    return [U[..., mu, :, :].permute(4, 5, 0, 1, 2, 3).contiguous() for mu in range(4)]


def _mul(U, h):  # U h on [spin][colour]
    return U[:, 0] * h[:, None, 0] + U[:, 1] * h[:, None, 1] + U[:, 2] * h[:, None, 2]


def _mul_dag(U, h):
    return _mul(U.conj().transpose(0, 1), h)


def _isigma(k, a):  # i sigma_k on the two spins of a
    if k == 0:
        return torch.stack([1j * a[1], 1j * a[0]])
    if k == 1:
        return torch.stack([a[1], -a[0]])
    return torch.stack([1j * a[0], -1j * a[1]])


def _hop_space(U, psi):
    up, lo = 0.0, 0.0
    u, d = psi[:2], psi[2:]
    for k in range(3):
        p = u + _isigma(k, d)  # (1 - gamma_k) psi = (p, -i sigma_k p)
        w = _mul(U[k], torch.roll(p, -1, _AXIS[k]))
        up, lo = up + w, lo - _isigma(k, w)
        m = u - _isigma(k, d)  # (1 + gamma_k) psi = (m, i sigma_k m)
        w = torch.roll(_mul_dag(U[k], m), 1, _AXIS[k])
        up, lo = up + w, lo + _isigma(k, w)
    return 0.5 * torch.cat([up, lo])


def _wrap(T, at, bc):
    s = torch.ones(T, 1, 1, 1, dtype=torch.float64, device="cuda")
    s[at] = bc
    return s


def _M(U, psi, mu, gf, A=None, bc=-1.0):
    T = psi.shape[2]
    dn = _wrap(T, T - 1, bc) * _mul(U[3], torch.roll(psi[2:], -1, -4))
    up = _wrap(T, 0, bc) * torch.roll(_mul_dag(U[3], psi[:2]), 1, -4)
    out = mu * psi - torch.cat([up, dn]) - _hop_space(U, psi) / gf
    if A is not None:
        out = out + torch.einsum("acbdtzyx,bdtzyx->actzyx", A, psi)
    return out


def _g5(psi):
    return -torch.cat([psi[2:], psi[:2]])


def _Tinv(U, eta, mu, dagger, bc=-1.0):
    """(mu psi(t) = eta(t) + U(t) psi(t+1)), or the adjoint (mu psi(t) = eta(t) + U(t-1)^dag psi(t-1)):
    the open recurrence, the product of its links, and the wrap closed by a 3x3 solve per line."""
    T, Ut = eta.shape[2], U[3]
    order = range(T) if dagger else range(T - 1, -1, -1)

    def step(t, v):
        return _mul_dag(Ut[:, :, t - 1 if t else T - 1], v) if dagger else _mul(Ut[:, :, t], v)

    eye = torch.eye(3, dtype=torch.complex128, device="cuda").reshape(3, 3, 1, 1, 1)
    c, G = None, eye.expand(3, 3, *eta.shape[3:])  # G[column][row]
    for t in order:
        c = eta[:, :, t] / mu if c is None else (eta[:, :, t] + step(t, c)) / mu
        G = step(t, G) / mu
    K = (eye - bc * G).permute(2, 3, 4, 1, 0)
    v = torch.linalg.solve(K, c.permute(2, 3, 4, 1, 0)).permute(4, 3, 0, 1, 2)  # the last value in order
    out, e = [None] * T, bc * v
    for t in order:
        e = (eta[:, :, t] + step(t, e)) / mu
        out[t] = e
    return torch.stack(out, 2)


def _schur(U, x, mu, gf):
    """M-hat on a full field that is zero on the even sites."""
    v = torch.cat([_Tinv(U, x[:2], mu, True), x[2:]])
    v = _hop_space(U, v)
    v = torch.cat([_Tinv(U, v[:2], mu, True), _Tinv(U, v[2:], mu, False)])
    v = _hop_space(U, v)
    return x - torch.cat([v[:2], _Tinv(U, v[2:], mu, False)]) / gf ** 2


def _odd_sites(L):
    z, y, xh = torch.meshgrid(torch.arange(L), torch.arange(L), torch.arange(L // 2), indexing="ij")
    x = 2 * xh + (y + z + 1) % 2
    return (x + L * (y + L * z)).reshape(-1).cuda()


def _from_odd(half, L):  # [t][k][spin][colour] -> [spin][colour][t][z][y][x], zero on even sites
    T = half.shape[0]
    full = torch.zeros(4, 3, T, L ** 3, dtype=torch.complex128, device="cuda")
    full[..., _odd_sites(L)] = half.permute(2, 3, 0, 1)
    return full.reshape(4, 3, T, L, L, L)


def _to_odd(full, L):
    T = full.shape[2]
    return full.reshape(4, 3, T, L ** 3)[..., _odd_sites(L)].permute(2, 3, 0, 1)


def _dot(a, b):
    return (a.conj() * b).sum()


def _cg(A, b, tol, most=4000):
    """A x = b for a hermitian positive A."""
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), float(_dot(r, r).real)
    stop = tol * tol * rr
    for _ in range(most):
        if rr <= stop:
            break
        q = A(p)
        a = rr / float(_dot(p, q).real)
        x += a * p
        r -= a * q
        new = float(_dot(r, r).real)
        p = r + (new / rr) * p
        rr = new
    return x


def _clover(U, c_s, c_t):
    """A = -[(c_t / 2) sum_i sigma_i0 F_i0 + (c_s / 2) sum_{i<j} sigma_ij F_ij] as [spin][colour][spin][colour]."""
    sig = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128, device="cuda")
    g = torch.zeros(4, 4, 4, dtype=torch.complex128, device="cuda")
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * sig[k], 1j * sig[k]
    g[3] = torch.diag(torch.tensor([1.0, 1.0, -1.0, -1.0]).to(g))

    def mm(a, b):
        return (a[:, :, None] * b[None]).sum(1)

    def dg(a):
        return a.conj().transpose(0, 1)

    def at(f, mu, step):  # f(x + step mu)
        return torch.roll(f, -step, _AXIS[mu])

    A = 0.0
    for a, b in ((0, 1), (0, 2), (1, 2), (0, 3), (1, 3), (2, 3)):
        Ua, Ub = U[a], U[b]
        Q = mm(mm(Ua, at(Ub, a, 1)), dg(mm(Ub, at(Ua, b, 1))))
        Uam, Ubm = at(Ua, a, -1), at(Ub, a, -1)
        Q = Q + mm(mm(Ub, dg(at(Uam, b, 1))), mm(dg(Ubm), Uam))
        Uamm = at(Uam, b, -1)
        Q = Q + mm(mm(dg(Uam), dg(at(Ubm, b, -1))), mm(Uamm, at(Ub, b, -1)))
        Ubn = at(Ub, b, -1)
        Q = Q + mm(mm(dg(Ubn), at(Ua, b, -1)), mm(at(Ubn, a, 1), dg(Ua)))
        F = (Q - dg(Q)) / 8.0
        eye = torch.eye(3, dtype=torch.float64, device="cuda").reshape(3, 3, 1, 1, 1, 1)
        F = F - eye * (F[0, 0] + F[1, 1] + F[2, 2]) / 3.0
        s = 0.5 * (g[a] @ g[b] - g[b] @ g[a])
        A = A - (0.5 * (c_t if b == 3 else c_s)) * torch.einsum("ab,cdtzyx->acbdtzyx", s, F)
    return A


def _exact_solve(case, U, src):
    mu, gf = 1.0 / (2.0 * _kappas(case)[1]), case["xi"]
    A = _clover(U, *CLOVER) if _is_clover(case) else None

    def M(v):
        return _M(U, v, mu, gf, A)

    def MdM(v):
        return _g5(M(_g5(M(v))))

    out = []
    for eta in src:
        b = eta.permute(4, 5, 0, 1, 2, 3).contiguous()
        x = 0.0
        for _ in range(2):  # the second round corrects what rounding left of the first
            r = b - M(x) if torch.is_tensor(x) else b
            x = x + _cg(MdM, _g5(M(_g5(r))), 1e-13)
        out.append(x.permute(2, 3, 4, 5, 0, 1))
    return torch.stack(out)


def _gell_mann():
    lam = torch.zeros(8, 3, 3, dtype=torch.complex128, device="cuda")
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        lam[a, i, j] = lam[a, j, i] = 1.0
        lam[a + 1, i, j], lam[a + 1, j, i] = -1j, 1j
    lam[2, 0, 0], lam[2, 1, 1] = 1.0, -1.0
    lam[7] = torch.diag(torch.tensor([1.0, 1.0, -2.0], dtype=torch.float64).cuda()) / math.sqrt(3.0)
    return lam


def _link_force(f, U):
    """d f / d eps for U_mu(x) -> exp(i eps lambda_a / 2) U_mu(x), as [t][z][y][x][mu][a]."""
    V = [u.detach().clone().requires_grad_(True) for u in U]
    g = torch.autograd.grad(f(V), V, allow_unused=True)
    out = []
    for u, d in zip(U, g):
        if d is None:
            d = torch.zeros_like(u)
        W = (u[:, None] * d.conj()[None, :]).sum(2)  # sum_c U_ac conj(G)_bc: f' = Re sum conj(G) (i T U)
        out.append(torch.einsum("kba,abtzyx->tzyxk", 0.5j * _gell_mann(), W).real)
    return torch.stack(out, -2)


def _exact_md(case, U, src):
    L, T = case["L"], case["T"]
    mu, gf = 1.0 / (2.0 * _kappas(case)[1]), case["xi"]
    phi = _from_odd(src[0], L)

    def S(v):
        return _schur(U, v, mu, gf)

    X = _cg(lambda v: _g5(S(_g5(S(v)))), phi, 1e-14)
    Y = S(X)
    F = _link_force(lambda V: -2.0 * _dot(Y, _schur(V, X, mu, gf)).real, U)

    def logdet(V):
        P = V[3][:, :, 0]
        for t in range(1, T):
            P = (P[:, :, None] * V[3][:, :, t][None]).sum(1)
        eye = torch.eye(3, dtype=torch.float64, device="cuda").reshape(3, 3, 1, 1, 1)
        K = (mu ** T * eye + P).permute(2, 3, 4, 0, 1)
        return 4.0 * torch.linalg.det(K).abs().log().sum()

    return {"action": float(_dot(Y, Y).real), "force": F, "logdet": float(logdet(U)), "logdet_force": _link_force(logdet, U)}


def exact(case, seed):
    L, n = case["L"], case.get("nrhs", 1)
    V = L ** 3 * case["T"]
    if case["kind"] == "solve" and n * V > 16 ** 3 * 128:
        return None  # more than about 20 seconds
    U, src = _inputs(case, seed)
    U = _fields(U)
    if case["kind"] == "md":
        return _exact_md(case, U, src)
    if case["kind"] == "solve":
        return _exact_solve(case, U, src)
    mu, gf = 1.0 / (2.0 * _kappas(case)[1]), case["xi"]
    out = torch.empty_like(src)
    for k in range(n):
        if case["op"] == "schur":
            v = _from_odd(src[k], L)
            v = _g5(_schur(U, _g5(v), mu, gf)) if case["dagger"] else _schur(U, v, mu, gf)
            out[k] = _to_odd(v, L)
            continue
        v = src[k].permute(4, 5, 0, 1, 2, 3)
        if case["op"] == "M":
            v = _g5(_M(U, _g5(v), mu, gf)) if case["dagger"] else _M(U, v, mu, gf)
        else:
            v = _Tinv(U, v, mu, case["dagger"])
        out[k] = v.permute(2, 3, 4, 5, 0, 1)
    return out.to(torch.complex64) if case["f32"] else out
