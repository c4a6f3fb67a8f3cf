"""Measured workloads of the library: whole calls through its public Python entry points.

Sizes are those of the repository's own workloads (48, 400, 800 and 1200 atomic orbitals, the
uneven batch, the embedded fragment problem) and ragged ones between them.  The values follow the
seeded inputs of the tests and the benchmark: packed Cholesky vectors N(0,1) exp(-|mu-nu|/8)
exp(-L/naux), a one-electron matrix with the same band decay, orthogonal MO coefficients, and
fragment RDMs of ensembles of determinants in rotated orbitals (dense, N-representable).
"""
import math

import torch

from paper_2505_03755_gb300 import LasDF
from paper_2505_03755_gb300.las import energy_grad_batched, las_energy, split_gemm

DEV = "cuda"


def listed():
    return [
        # the smallest problem anybody runs (the 48-orbital workload): launches and latency count
        dict(name="energy-grad-48", kind="energy_grad", precision="split_packed", nao=48, naux=160,
             nmo=48, ncore=10, frags="2,2", gorb=True),
        # native FP64, a ragged size of the batch's range: the mode that checks the others
        dict(name="energy-grad-237-fp64", kind="energy_grad", precision="fp64", nao=237, naux=948,
             nmo=237, ncore=29, frags="4,3,5", gorb=True),
        # the ordinary evaluation of an orbital optimisation step (the 400-orbital workload)
        dict(name="energy-grad-400", kind="energy_grad", precision="split", nao=400, naux=1600,
             nmo=400, ncore=60, frags="4,4,4,4", gorb=True),
        # the differentiable energy, forward and backward (the 800-orbital workload)
        dict(name="autograd-800", kind="autograd", precision="split_packed", nao=800, naux=3200,
             nmo=800, ncore=100, frags="6,6,6,6"),
        # one of two ranks' block of auxiliary rows of the 1200-orbital workload
        dict(name="energy-grad-1200-shard", kind="energy_grad", precision="split_packed", nao=1200,
             naux=2400, nmo=1200, ncore=150, frags="8,8,8,8,8", gorb=False),
        # Coulomb and exchange matrices of the core density (every SCF-like step)
        dict(name="jk-800", kind="jk", precision="split_packed", nao=800, naux=1600, nmo=800,
             ncore=100, frags="6,6,6,6"),
        # embedding potentials of an open-shell state: general densities of both spins
        dict(name="veff-400", kind="veff", precision="split", nao=400, naux=1600, nmo=400,
             ncore=60, frags="4,4,4,4"),
        # half- and full-transformed Cholesky vectors of the active orbitals over all MOs
        dict(name="transform-400", kind="transform", precision="split", nao=400, naux=1600,
             nmo=400, ncore=60, frags="4,4,4,4", p0=0, p1=400),
        # a fragment's embedded integrals, 2 (4 + 100) embedded orbitals of the 400-orbital system
        dict(name="ao2mo-208", kind="ao2mo", precision="split_packed", nao=208, naux=1600, nmo=208,
             ncore=50, frags="4"),
        # orbital Hessian-vector product (second-order optimisation)
        dict(name="hvp-400", kind="hvp", precision="split", nao=400, naux=1600, nmo=400, ncore=60,
             frags="4,4,4,4"),
        # many uneven systems at once under one graph
        dict(name="batch-8", kind="batch", precision="split",
             systems="100:12:2,3;131:16:4,4,2;163:20:8,2;209:26:5,3,7;250:31:2,8,4,6;303:37:6,6;"
                     "347:43:3,7,2,5,4;400:50:8,8,3"),
        # the emulated-FP64 product by itself, ragged
        dict(name="gemm-2999", kind="gemm", m=2999, k=1201, n=187),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _frags(rng, most):
    out, left = [], most
    for _ in range(rng.randint(1, 5)):
        m = rng.randint(2, 8)
        if m > left:
            break
        out.append(m)
        left -= m
    return out or [1]


def draw(rng):
    kind = rng.choice(["energy_grad", "energy_grad", "energy_grad", "autograd", "jk", "veff",
                       "transform", "ao2mo", "hvp", "batch", "gemm"])
    if kind == "gemm":
        return dict(kind=kind, m=_log_int(rng, 40, 20000), k=_log_int(rng, 16, 3000),
                    n=_log_int(rng, 8, 600))
    if kind == "batch":
        rows = []
        for _ in range(rng.randint(3, 10)):
            n = _log_int(rng, 60, 350)
            rows.append("%d:%d:%s" % (n, n // 8, ",".join(map(str, _frags(rng, n // 4)))))
        return dict(kind=kind, precision=rng.choice(["split", "split", "split_packed"]),
                    systems=";".join(rows))
    if kind == "ao2mo":
        n = _log_int(rng, 40, 320)
        m = rng.randint(2, 8)
        return dict(kind=kind, precision=rng.choice(["split", "split_packed"]), nao=n,
                    naux=_log_int(rng, 2 * n, 1600), nmo=n, ncore=n // 4, frags=str(m))
    fp64 = kind in ("energy_grad", "jk") and rng.random() < 0.2
    top = {"energy_grad": 1200, "autograd": 800, "jk": 800, "veff": 600, "transform": 500,
           "hvp": 600}[kind]
    n = _log_int(rng, 24, 200 if fp64 else top)
    frags = _frags(rng, n // 4)
    c = max(1, n // 8 + rng.randint(-2, 2))
    case = dict(kind=kind, precision="fp64" if fp64 else rng.choice(["split", "split_packed"]),
                nao=n, naux=min(2400, max(16, int(n * rng.uniform(1.5, 4.5)))),
                nmo=n - rng.choice([0, 0, 1, n // 10]), ncore=c,
                frags=",".join(map(str, frags)))
    if kind == "energy_grad":
        case["gorb"] = rng.random() < 0.5
    if kind == "transform":
        p0 = rng.choice([0, 0, c])
        case.update(p0=p0, p1=rng.randint(p0 + 1, case["nmo"]))
    return case


# ----------------------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _packed_B(g, n, naux):
    mu, nu = torch.tril_indices(n, n, device=DEV)
    decay = torch.exp(-(mu - nu).to(torch.float64) / 8)
    B = torch.empty(naux, n * (n + 1) // 2, device=DEV, dtype=torch.float64)
    B.normal_(generator=g)
    B *= decay
    B *= torch.exp(-torch.arange(naux, device=DEV, dtype=torch.float64) / naux)[:, None]
    return B


def _fragment_rdms(g, m):
    """(gamma_alpha, gamma_beta) and the spin-summed Gamma_pqrs = <p+ r+ s q> of an ensemble of
    three determinants in rotated orbitals: 2 floor(m/2) electrons, one more alpha than beta in
    one of them."""
    dm1, dm2 = torch.zeros(2, m, m, dtype=torch.float64), torch.zeros(m, m, m, m, dtype=torch.float64)
    for k, w in enumerate((0.6, 0.3, 0.1)):
        q, _ = torch.linalg.qr(_normal(g, m, m).cpu())
        na = nb = m // 2
        if k == 1 and na < m and nb > 0:
            na, nb = na + 1, nb - 1
        gs = [q[:, :x] @ q[:, :x].T for x in (na, nb)]
        D = gs[0] + gs[1]
        dm1 += w * torch.stack(gs)
        dm2 += w * torch.einsum("pq,rs->pqrs", D, D)
        for s in gs:
            dm2 -= w * torch.einsum("ps,rq->pqrs", s, s)
    return dm1.to(DEV), dm2.to(DEV)


def _frag_list(case):
    return [int(x) for x in case["frags"].split(",")]


def _system(case, seed):
    """All inputs of one problem, from the seed alone."""
    g = _gen(seed)
    n, nmo = case["nao"], case["nmo"]
    s = dict(B=_packed_B(g, n, case["naux"]))
    mu, nu = torch.tril_indices(n, n, device=DEV)
    h = torch.zeros(n, n, device=DEV, dtype=torch.float64)
    h[mu, nu] = _normal(g, mu.numel()) * torch.exp(-(mu - nu).to(torch.float64) / 8)
    s["h"] = torch.tril(h) + torch.tril(h, -1).T
    q, _ = torch.linalg.qr(_normal(g, n, n))
    s["C"] = q[:, :nmo].contiguous()
    s["nact"] = _frag_list(case)
    rdms = [_fragment_rdms(g, m) for m in s["nact"]]
    s["dm1s"] = torch.cat([a.reshape(-1) for a, _ in rdms])
    s["dm2"] = torch.cat([b.reshape(-1) for _, b in rdms])
    s["rdms"] = rdms
    x = _normal(g, nmo, nmo)
    x = x - x.T
    s["X"] = x / x.norm()
    return s


def _context(case, s):
    return LasDF(s["B"], case["nao"], case["naux"], case["nmo"], case["ncore"], s["nact"],
                 precision=case["precision"])


def _spin_density(case, s, sigma):
    """Factored spin density of the LAS state: core and natural active orbitals, and weights."""
    c, cols, w = case["ncore"], [], []
    cols.append(s["C"][:, :c])
    w.append(torch.ones(c, device=DEV, dtype=torch.float64))
    o = c
    for (dm1, _), m in zip(s["rdms"], s["nact"]):
        e, v = torch.linalg.eigh(dm1[sigma])
        cols.append(s["C"][:, o:o + m] @ v)
        w.append(e)
        o += m
    return torch.cat(cols, 1).contiguous(), torch.cat(w)


def _batch_cases(case):
    out = []
    for row in case["systems"].split(";"):
        n, c, fr = row.split(":")
        out.append(dict(nao=int(n), naux=4 * int(n), nmo=int(n), ncore=int(c), frags=fr,
                        precision=case["precision"]))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        g = _gen(seed)
        A = _normal(g, case["m"], case["k"]) * torch.exp(2 * _normal(g, case["m"], 1))
        B = _normal(g, case["k"], case["n"]) * torch.exp(2 * _normal(g, 1, case["n"]))
        return dict(kind=kind, A=A, B=B)
    if kind == "batch":
        st = dict(kind=kind, las=[], items=[])
        for i, c in enumerate(_batch_cases(case)):
            s = _system(c, seed * 1000 + i)
            las = _context(c, s)
            las.release_packed_B()
            st["las"].append(las)
            st["items"].append((s["C"], s["h"], s["dm1s"], s["dm2"],
                                torch.empty((), device=DEV, dtype=torch.float64),
                                torch.empty(c["nao"], c["nmo"], device=DEV, dtype=torch.float64)))
        return st
    s = _system(case, seed)
    st = dict(kind=kind, case=case, las=_context(case, s), C=s["C"], h=s["h"], dm1s=s["dm1s"],
              dm2=s["dm2"])
    if kind == "hvp":
        st["X"] = s["X"]
    if kind == "veff":
        st["spin"] = _spin_density(case, s, 0) + _spin_density(case, s, 1)
    return st


def run(state):
    kind = state["kind"]
    if kind == "gemm":
        return split_gemm(state["A"], state["B"])
    if kind == "batch":
        energy_grad_batched(state["las"], state["items"])
        return [(E, G) for *_, E, G in state["items"]]
    las, C = state["las"], state["C"]
    args = (C, state["h"], state["dm1s"], state["dm2"])
    if kind == "energy_grad":
        return las.energy_grad(*args, want_gorb=state["case"]["gorb"])
    if kind == "autograd":
        x = C.detach().requires_grad_(True)
        E = las_energy(x, las, *args[1:])
        E.backward()
        return E.detach(), x.grad
    if kind == "jk":
        return las.df_jk(C)
    if kind == "veff":
        return las.veff(*state["spin"])
    if kind == "transform":
        return las.df_transform(C, state["case"]["p0"], state["case"]["p1"])
    if kind == "ao2mo":
        return las.frag_ao2mo(C, state["case"]["ncore"], _frag_list(state["case"])[0])
    return las.orbital_hvp(*args, state["X"])


# ----------------------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, k, n = case["m"], case["k"], case["n"]
        return dict(bytes=8 * (m * k + k * n + m * n), flops=2 * m * n * k)
    if kind == "batch":
        each = [work(dict(c, kind="energy_grad", gorb=False)) for c in _batch_cases(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n, X, nmo, c = case["nao"], case["naux"], case["nmo"], case["ncore"]
    fr = _frag_list(case)
    a = sum(fr)
    o = c + a
    B = 8 * X * (n * (n + 1) // 2)
    state = 8 * (n * nmo + n * n + sum(2 * m * m + m ** 4 for m in fr))
    one = 2 * n * n * o + 2 * n * o * o                      # h in the occupied space
    grad = 2 * X * n * n * o + 4 * X * n * o * o + one       # half, full transform, projection
    if kind in ("energy_grad", "autograd"):
        g = kind == "energy_grad" and case["gorb"]
        return dict(bytes=B + state + 8 * (1 + n * nmo + (nmo * nmo if g else 0)),
                    flops=grad + (2 * n * nmo * o if g else 0))
    if kind == "hvp":
        tangent = 2 * X * n * n * o + 6 * X * n * o * o + 2 * n * n * o
        return dict(bytes=B + state + 8 * (2 * nmo * nmo + n * nmo),
                    flops=grad + tangent + 2 * n * nmo * nmo + 4 * n * nmo * o)

    def jk(r):   # traces, half transform, J, and the lower triangle of K
        return 2 * X * n * n * r + 2 * X * n * r + X * n * (n + 1) + X * n * n * r
    if kind == "jk":
        return dict(bytes=B + 8 * (n * c + 2 * n * n), flops=jk(c))
    if kind == "veff":
        return dict(bytes=B + 8 * (2 * n * o + 2 * n * n), flops=2 * jk(o))
    if kind == "transform":
        np_ = case["p1"] - case["p0"]
        return dict(bytes=B + 8 * (n * nmo + X * a * (n + np_)),
                    flops=2 * X * n * n * a + 2 * X * n * np_ * a)
    m = fr[0]
    return dict(bytes=B + 8 * (n * nmo + 2 * (nmo * m) ** 2),
                flops=2 * X * (n * n * nmo + n * nmo * nmo) + 2 * X * nmo * nmo * m * m
                + X * (nmo * m) ** 2)


# ----------------------------------------------------------------------------------------
# The same results in plain 64-bit torch
# ----------------------------------------------------------------------------------------
def _blocks(B, n):
    """(first row, symmetric squares) of the packed Cholesky vectors, block by block."""
    mu, nu = torch.tril_indices(n, n, device=DEV)
    step = max(1, (1 << 27) // (n * n))
    for l0 in range(0, B.shape[0], step):
        rows = B[l0:l0 + step]
        b = torch.zeros(rows.shape[0], n, n, device=DEV, dtype=torch.float64)
        b[:, mu, nu] = rows
        b[:, nu, mu] = rows
        yield l0, b


def _active_rdms(s):
    """Block-product D and Gamma of the whole active space from the fragments' RDMs."""
    a, off = sum(s["nact"]), [0]
    for m in s["nact"]:
        off.append(off[-1] + m)
    gs = torch.zeros(2, a, a, device=DEV, dtype=torch.float64)
    for K, (dm1, _) in enumerate(s["rdms"]):
        gs[:, off[K]:off[K + 1], off[K]:off[K + 1]] = dm1
    D = gs[0] + gs[1]
    G = torch.einsum("pq,rs->pqrs", D, D)
    for x in gs:
        G -= torch.einsum("ps,rq->pqrs", x, x)
    for K, (_, dm2) in enumerate(s["rdms"]):
        r = slice(off[K], off[K + 1])
        G[r, r, r, r] = dm2
    return D, G


def _per_aux(T, c, D, G):
    """The matrices W_L (linear in T_L) with dE/dC = one-electron part + sum_L H_L W_L, and the
    energy terms eps_L."""
    a = D.shape[0]
    Tc, Ta, Tca = T[:, :c, :c], T[:, c:, c:], T[:, :c, c:]
    vc = 2 * torch.einsum("lii->l", Tc)
    va = torch.einsum("luv,uv->l", Ta, D)
    Y = (Ta.reshape(-1, a * a) @ G.reshape(a * a, a * a).T).reshape(-1, a, a)
    Z = Tca @ D
    W = torch.zeros_like(T)
    W[:, :c, :c] = -4 * Tc
    W[:, range(c), range(c)] += 4 * (vc + va)[:, None]
    W[:, c:, :c] = -2 * Z.transpose(1, 2)
    W[:, :c, c:] = -2 * Z
    W[:, c:, c:] = 2 * vc[:, None, None] * D + 2 * Y.transpose(1, 2)
    eps = (vc * vc / 2 - (Tc * Tc).sum((1, 2)) + vc * va - (Z * Tca).sum((1, 2))
           + (Ta * Y).sum((1, 2)) / 2)
    return W, eps


def _one_electron_grad(hC, c, D, n, nmo):
    G = torch.zeros(n, nmo, device=DEV, dtype=torch.float64)
    o = c + D.shape[0]
    G[:, :c] = 4 * hC[:, :c]
    G[:, c:o] = 2 * hC[:, c:] @ D
    return G


def _exact_energy_grad(case, s, X=None):
    """E, dE/dC and the rotation gradient; with X also their derivatives along C X."""
    n, nmo, c = case["nao"], case["nmo"], case["ncore"]
    D, Gam = _active_rdms(s)
    o = c + D.shape[0]
    C = s["C"]
    Co = C[:, :o]
    hC = s["h"] @ Co
    E = 2 * torch.einsum("mi,mi->", Co[:, :c], hC[:, :c])
    E = E + torch.einsum("mu,mv,uv->", Co[:, c:], hC[:, c:], D)
    G = _one_electron_grad(hC, c, D, n, nmo)
    if X is not None:
        dC = C @ X
        dCo = dC[:, :o]
        dG = _one_electron_grad(s["h"] @ dCo, c, D, n, nmo)
    terms = []
    for _, b in _blocks(s["B"], n):
        H = b @ Co
        T = Co.T @ H
        W, eps = _per_aux(T, c, D, Gam)
        terms.append(eps)
        flat = H.permute(1, 0, 2).reshape(n, -1)
        G[:, :o] += flat @ W.reshape(-1, o)
        if X is not None:
            dH = b @ dCo
            x = H.transpose(1, 2) @ dCo
            dW, _ = _per_aux(x + x.transpose(1, 2), c, D, Gam)
            dG[:, :o] += dH.permute(1, 0, 2).reshape(n, -1) @ W.reshape(-1, o)
            dG[:, :o] += flat @ dW.reshape(-1, o)
    E = E + math.fsum(torch.cat(terms).tolist())
    if X is not None:
        M = dC.T @ G + C.T @ dG
        return dG, M - M.T
    M = C.T @ G
    return E, G, M - M.T


def _exact_jk(B, n, factors, w):
    """J and K of the density factors diag(w) factors^T."""
    J = torch.zeros(n, n, device=DEV, dtype=torch.float64)
    K = torch.zeros_like(J)
    dens = (factors * w) @ factors.T
    for _, b in _blocks(B, n):
        v = b.reshape(-1, n * n) @ dens.reshape(-1)
        J += torch.einsum("l,lmn->mn", v, b)
        H = (b @ factors).permute(1, 0, 2)
        K += (H * w).reshape(n, -1) @ H.reshape(n, -1).T
    return J, K


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        s = prepare(case, seed)
        return s["A"] @ s["B"]
    if kind == "batch":
        out = []
        for i, c in enumerate(_batch_cases(case)):
            out.append(_exact_energy_grad(c, _system(c, seed * 1000 + i))[:2])
        return out
    s = _system(case, seed)
    n, c = case["nao"], case["ncore"]
    if kind in ("energy_grad", "autograd"):
        E, G, g = _exact_energy_grad(case, s)
        return (E, G, g) if kind == "energy_grad" and case["gorb"] else (E, G)
    if kind == "hvp":
        return _exact_energy_grad(case, s, s["X"])
    if kind == "jk":
        w = torch.full((c,), 2.0, device=DEV, dtype=torch.float64)
        return _exact_jk(s["B"], n, s["C"][:, :c], w)
    if kind == "veff":
        (Ja, Ka), (Jb, Kb) = (_exact_jk(s["B"], n, *_spin_density(case, s, x)) for x in (0, 1))
        return Ja + Jb - Ka, Ja + Jb - Kb
    if kind == "transform":
        act = s["C"][:, c:c + sum(s["nact"])]
        P = s["C"][:, case["p0"]:case["p1"]]
        lmu = torch.cat([b @ act for _, b in _blocks(s["B"], n)])
        return lmu, torch.einsum("mp,lmu->lpu", P, lmu)
    m = s["nact"][0]
    T = torch.cat([s["C"].T @ (b @ s["C"]) for _, b in _blocks(s["B"], n)])
    X, nmo = T.shape[0], case["nmo"]
    aa = T[:, c:c + m, c:c + m].reshape(X, -1)
    pa = T[:, :, c:c + m].reshape(X, -1)
    ppaa = (T.reshape(X, -1).T @ aa).reshape(nmo, nmo, m, m)
    return ppaa, (pa.T @ pa).reshape(nmo, m, nmo, m)
