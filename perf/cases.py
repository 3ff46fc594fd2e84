"""The workloads whose speed is watched: single steps and whole calls of the public entry points.

Real use of this framework is: build the double layer of an iPEPS tensor, run CTMRG moves (FP64, or
TF32x3 with the subspace eigensolver) or HOTRG steps, read observables off the environment, and
differentiate them. Each kind below is one of those calls; the sizes are those of the workloads in
inputs.py, of the tests and of the benchmark, and draw() spreads over the ranges between them.
"""
import math

import numpy as np
import torch

from paper_2410_11596_gb300 import _lib as L
from paper_2410_11596_gb300 import inputs
from paper_2410_11596_gb300 import api

DEV = "cuda:0"


# ---- the cases ---------------------------------------------------------------------------------


def listed():
    return [
        # the smallest whole call: a D=2 run from the tensor to the bond's density matrix, launch-bound
        dict(name="run_f64_d2_chi16", kind="run", D=2, chi=16, moves=6),
        # building and rotating the largest double layer of the batched workload, both separate calls
        dict(name="double_layer_d7", kind="double_layer", D=7),
        # one accurate (FP64) move of an ordinary environment
        dict(name="move_f64_d4_chi64", kind="move", D=4, chi=64, warm=4),
        # the headline tensor size in mixed precision: from the tensor through its first moves, where the
        # environment still turns and every move takes several rounds of the warm-started projector
        dict(name="env_tf32x3_d6_chi144", kind="env", D=6, chi=144, moves=8),
        # a HOTRG run of a tensor without lattice symmetry, from the tensor to ln Z
        dict(name="hotrg_f64_d4_chi32", kind="hotrg", D=4, chi=32, steps=3),
        # bond density matrix of the headline environment: the largest observable
        dict(name="rdm2_d6_chi144", kind="rdm2", D=6, chi=144, warm=2),
        # one-site environment of Eq. (4), the symmetry-error diagnostic
        dict(name="one_site_env_d5_chi100", kind="one_site", D=5, chi=100, warm=2),
        # variational step with the environment held fixed: energy and its gradient, real
        dict(name="bond_grad_d4_chi64", kind="bond_grad", D=4, chi=64, warm=2, complex=False),
        # the same of the complex workload
        dict(name="bond_grad_complex_d5_chi100", kind="bond_grad", D=5, chi=100, warm=2, complex=True),
        # energy of a whole run and its gradient through every move
        dict(name="run_grad_d3_chi27", kind="run_grad", D=3, chi=27, moves=5),
        # the block GEMM primitive at the shape of the headline's largest block product, FP64 and mixed
        dict(name="gemm_f64_block", kind="gemm", M=10368, N=666, K=666, precision="f64"),
        dict(name="gemm_tf32x3_block", kind="gemm", M=10368, N=666, K=666, precision="tf32x3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "double_layer", "move", "env", "hotrg", "rdm2", "one_site", "bond_grad",
                       "bond_grad_complex", "run_grad", "gemm", "gemm", "gemm"])
    if kind == "run":
        D = rng.randint(2, 3)
        return dict(kind="run", D=D, chi=rng.randint(6, 8 * D), moves=rng.randint(3, 8))
    if kind == "double_layer":
        return dict(kind="double_layer", D=rng.randint(2, 7), seed_offset=rng.randint(0, 99))
    if kind == "move":
        D = rng.randint(2, 5)
        return dict(kind="move", D=D, chi=rng.randint(D * D, 4 * D * D), warm=3)
    if kind == "env":
        D = rng.randint(3, 6)
        return dict(kind="env", D=D, chi=rng.randint(2 * D * D, 4 * D * D), moves=rng.randint(4, 8))
    if kind == "hotrg":
        D = rng.randint(2, 4)
        return dict(kind="hotrg", D=D, chi=_log_int(rng, 8, 32), steps=rng.randint(2, 3))
    if kind == "rdm2":
        D = rng.randint(2, 6)
        return dict(kind="rdm2", D=D, chi=rng.randint(D * D, 4 * D * D), warm=2)
    if kind == "one_site":
        D = rng.randint(2, 6)
        return dict(kind="one_site", D=D, chi=rng.randint(D * D, 4 * D * D), warm=2)
    if kind in ("bond_grad", "bond_grad_complex"):
        cplx = kind.endswith("complex")
        D = rng.randint(2, 4 if cplx else 5)
        return dict(kind="bond_grad", D=D, chi=rng.randint(D * D, 4 * D * D), warm=2, complex=cplx)
    if kind == "run_grad":
        D = rng.randint(2, 3)
        return dict(kind="run_grad", D=D, chi=rng.randint(2 * D, 4 * D * D), moves=rng.randint(2, 5))
    # GEMM blocks: narrow subspace products, tall corner and edge products, square ones
    M, N, K = _log_int(rng, 20, 12000), _log_int(rng, 20, 2600), _log_int(rng, 16, 2600)
    while 2.0 * M * N * K > 4e10:
        M = max(20, M // 2)
    return dict(kind="gemm", M=M, N=N, K=K, precision=rng.choice(["f64", "f64", "tf32x3", "bf16x3"]))


# ---- what a program has in hand ------------------------------------------------------------------


def _tensor(case, seed):
    """The iPEPS tensor of a case (host): C4v-symmetric as the CTMRG assumes, generic for HOTRG."""
    seed = 7919 * int(seed) + case.get("seed_offset", 0)
    if case["kind"] == "hotrg":
        return inputs.asymmetric_ipeps(2, case["D"], seed)
    return inputs.random_ipeps(2, case["D"], seed, bool(case.get("complex", False)))


def _gemm_operands(case, seed):
    """Operands like a corner product's: the contraction index runs over boundary states of falling
    weight, two decades over the range."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    M, N, K = case["M"], case["N"], case["K"]
    w = torch.logspace(0, -1, K, dtype=torch.float64, device=DEV)
    A = torch.randn(M, K, dtype=torch.float64, device=DEV, generator=g) * w
    B = torch.randn(N, K, dtype=torch.float64, device=DEV, generator=g) * w
    return A, B


def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case, ctx=api.Context(0), h=inputs.heisenberg_bond())
    if k == "gemm":
        s["A"], s["B"] = _gemm_operands(case, seed)
        s["C"] = torch.empty(case["M"], case["N"], dtype=torch.float64, device=DEV)
        return s
    A = _tensor(case, seed)
    if k in ("run", "env", "hotrg", "run_grad", "double_layer"):
        s["A"] = api.to_device(A)
        if k == "double_layer":
            D, q = case["D"], case["D"] ** 2
            s["a"] = torch.empty(q, q, q, q, dtype=torch.float64, device=DEV)
            s["blocks"] = torch.empty(L.hs_z2_tensor_bytes(D, L.HS_BASIS_HERMITIAN, L.HS_F64) // 8,
                                      dtype=torch.float64, device=DEV)
        return s
    # an environment a few moves from the traced boundary, at the full boundary dimension
    c = api.CTMRG(s["ctx"], A, case["chi"])
    c.run(case["warm"])
    s["ctm"] = c
    if k == "bond_grad":
        s["A"] = torch.from_numpy(A).to(DEV).requires_grad_(True)
        s["h"] = torch.from_numpy(s["h"]).to(DEV)
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "gemm":
        L.hs_gemm(s["ctx"].handle, api.PRECISION[case["precision"]], s["A"], s["B"], s["C"])
        return s["C"]
    if k == "double_layer":
        h, D = s["ctx"].handle, case["D"]
        L.hs_make_double_layer(h, s["A"], 2, D, L.HS_F64, s["a"])
        L.hs_to_hermitian_basis(h, s["a"], D, L.HS_F64, 1e-10, s["blocks"])
        ne, no = D * (D + 1) // 2, D * (D - 1) // 2
        r0, r1 = ne * ne + no * no, 2 * ne * no
        return {"a": s["a"], "blocks": s["blocks"][: r0 * r0 + r1 * r1]}
    if k == "run":
        c = api.CTMRG(s["ctx"], s["A"], case["chi"])
        c.run(case["moves"])
        rho, tr, trh = c.rdm2(s["h"])
        C, T = c.dense_env()
        return {"rho": rho, "tr": tr, "trh": trh, "spectrum": c.corner_spectrum(), "C": C, "T": T}
    if k == "env":
        c = api.CTMRG(s["ctx"], s["A"], case["chi"], precision="tf32x3", eig="subspace")
        c.run(case["moves"])
        C, T = c.dense_env()
        return {"C": C, "T": T}
    if k == "move":
        s["ctm"].move()
        C, T = s["ctm"].dense_env()
        return {"C": C, "T": T}
    if k == "hotrg":
        t = api.HOTRG(s["ctx"], s["A"], case["chi"])
        t.run(case["steps"])
        v, w = (t.t.v_even, t.t.v_odd), (t.t.h_even, t.t.h_odd)
        r0, r1 = v[0] * w[0] + v[1] * w[1], v[0] * w[1] + v[1] * w[0]
        # the sizes of the two parity blocks follow from the tensor's values: zeros after them keep one shape
        T = torch.nn.functional.pad(t.t_buf[: r0 * r0 + r1 * r1], (0, t.t_buf.numel() - r0 * r0 - r1 * r1))
        return {"log_z": t.log_z_per_site(), "log_norms": np.array(t.log_norms), "T": T}
    if k == "rdm2":
        rho, tr, trh = s["ctm"].rdm2(s["h"])
        return {"rho": rho, "tr": tr, "trh": trh}
    if k == "one_site":
        return s["ctm"].one_site_env()
    if k == "bond_grad":
        E = api.bond_energy(s["ctm"], s["A"], s["h"])
        (g,) = torch.autograd.grad(E, s["A"])
        return {"E": E, "dA": g}
    A = s["A"].detach().requires_grad_(True)
    E = api.ctmrg_energy(s["ctx"], A, case["chi"], case["moves"], s["h"])
    (g,) = torch.autograd.grad(E, A)
    return {"E": E, "dA": g}


# ---- what a pass cannot do without -----------------------------------------------------------------


def _move_work(D, c0, c):
    """Contractions of one move, and one product of the enlarged corner with the kept vectors; two parity
    blocks of half the size in each index do a quarter of the plain work."""
    q = D * D
    f = 2.0 * (c0 ** 3 * q + c0 ** 3 * q * q + c0 ** 2 * q ** 4)
    f += 2.0 * (c * c0 ** 2 * q * q + c * c0 * q ** 4 + c * c * c0 * q * q) + 2.0 * (c0 * q) ** 2 * c
    return f / 4.0


def _rho_work(D, c, z):
    """Half rings, then each site's ket and bra tensors one after the other; z real products a product."""
    q = D * D
    f = 2.0 * (2 * c ** 3 * q + c ** 3 * q * q)
    f += 2 * (2.0 * c * c * q * q * 2 * q + 2.0 * c * c * 2 * q * q * 2 * q + 2.0 * c ** 3 * 4 * q * q)
    return z * f


def work(case):
    k = case["kind"]
    if k == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=8.0 * (M * K + N * K + M * N), flops=2.0 * M * N * K)
    D = case["D"]
    q, chi = D * D, case.get("chi", 0)
    nA = 2 * D ** 4
    env = 8.0 * (chi * chi + chi * chi * q)
    if k == "double_layer":
        return dict(bytes=8.0 * (nA + 2 * q ** 4 + q ** 4 / 2), flops=2.0 * 2 * q ** 4 + 16.0 * q ** 4)
    if k in ("run", "env", "run_grad"):
        f, c = 0.0, q
        for _ in range(case["moves"]):
            f += _move_work(D, c, min(chi, c * q))
            c = min(chi, c * q)
        f += 0.0 if k == "env" else _rho_work(D, c, 1)
        grad = k == "run_grad"
        return dict(bytes=8.0 * nA * (2 if grad else 1) + (0 if grad else env), flops=f * (3 if grad else 1))
    if k == "move":
        return dict(bytes=env + 8.0 * q ** 4 / 2, flops=_move_work(D, chi, chi))
    if k == "hotrg":
        f, v, h = 0.0, q, q
        for i in range(case["steps"]):
            if i % 2:
                v, h = h, v
            hn = min(chi, h * h)
            f += 2.0 * (h * v * h * v * v * h + h ** 4 * v * v + v * v * h ** 4 * v + v * v * h ** 4 * hn
                        + v * v * h * h * hn * hn) / 2
            h = hn
            if i % 2:
                v, h = h, v
        return dict(bytes=8.0 * (nA + v * v * h * h / 2), flops=f)
    if k == "rdm2":
        return dict(bytes=env + 8.0 * nA, flops=_rho_work(D, chi, 1))
    if k == "one_site":
        return dict(bytes=env + 8.0 * q ** 4, flops=2.0 * (2 * chi ** 3 * q + 2 * chi ** 3 * q * q + q ** 4 * chi ** 2))
    z = 4 if case["complex"] else 1
    return dict(bytes=(2 if case["complex"] else 1) * (env + 16.0 * nA), flops=3 * _rho_work(D, chi, z))


# ---- the same in 64 bits, plain torch ----------------------------------------------------------------


def _u(D):
    """Eigenbasis of the bra-ket swap on one combined leg x = ket + D bra (columns; even states first)."""
    U = torch.zeros(D * D, D * D, dtype=torch.float64, device=DEV)
    j = 0
    for k in range(D):
        U[k + D * k, j] = 1.0
        j += 1
    for sign in (1.0, -1.0):
        for k in range(D):
            for m in range(k + 1, D):
                U[k + D * m, j] = 0.5 ** 0.5
                U[m + D * k, j] = sign * 0.5 ** 0.5
                j += 1
    return U


def _double_layer(A):
    """a[u, l, d, r], combined index ket + D bra."""
    D = A.shape[1]
    a = torch.einsum("puldr,pabcf->aublcdfr", A, A.conj())
    return a.reshape((D * D,) * 4)


def _rotate(a, U):
    return torch.einsum("uldr,ua,lb,dc,re->abce", a, U, U, U, U)


def _parity(D):
    ne = D * (D + 1) // 2
    return torch.tensor([0] * ne + [1] * (D * D - ne), device=DEV)


def _ctmrg(A, chi, moves):
    """C4v CTMRG in the Hermitian basis, plain tensors; boundary states even first. Returns (C, T)."""
    D = A.shape[1]
    U, pq = _u(D), _parity(D)
    a = _rotate(_double_layer(A), U)
    v = torch.zeros(D * D, dtype=torch.float64, device=DEV)
    v[:D] = 1.0
    C = torch.einsum("uldr,u,l->dr", a, v, v)
    T = torch.einsum("uldr,l->dru", a, v)
    C, T = C / C.detach().abs().max(), T / T.detach().abs().max()
    pc = pq
    for _ in range(moves):
        c, q = T.shape[0], T.shape[1]
        X = torch.tensordot(T, C, dims=([2], [1]))
        X = torch.tensordot(X, T, dims=([2], [2])).permute(0, 2, 3, 1)           # (a, e, y, x)
        X = torch.tensordot(X, a, dims=([2, 3], [2, 3]))                         # (a, e, u, l)
        Cp = X.permute(0, 2, 1, 3).reshape(c * q, c * q)
        p = (pc[:, None] ^ pq[None, :]).reshape(-1)
        w, V, blk = [], [], []
        for b in (0, 1):
            i = torch.nonzero(p == b)[:, 0]
            if len(i) == 0:
                continue
            M = Cp[i][:, i]
            wb, Vb = torch.linalg.eigh(0.5 * (M + M.T))
            full = torch.zeros(c * q, len(i), dtype=Cp.dtype, device=DEV).index_put((i,), Vb)
            w.append(wb)
            V.append(full)
            blk += [b] * len(i)
        w, V, blk = torch.cat(w), torch.cat(V, 1), torch.tensor(blk, device=DEV)
        order = torch.argsort(-w.detach().abs(), stable=True)[: min(chi, c * q)]
        order = torch.cat([order[blk[order] == 0], order[blk[order] == 1]])
        P = V[:, order].reshape(c, q, -1)
        C = torch.diag(w[order])
        Y = torch.einsum("adk,bxa->kbdx", P, T)
        Z = torch.tensordot(Y, a, dims=([2, 3], [2, 3]))                         # (k, b, u, r)
        T = torch.einsum("kbur,bum->krm", Z, P)
        C, T = C / C.detach().abs().max(), T / T.detach().abs().max()
        pc = blk[order]
    return C, torch.einsum("axb,yx->ayb", T, U)


def _ctmrg_complex(A, chi, moves):
    """Complex CTMRG in the plain basis: clockwise boundary tensors, isometries from the left singular
    vectors of the enlarged corner."""
    D = A.shape[1]
    a = _double_layer(A)
    v = torch.zeros(D * D, dtype=a.dtype, device=DEV)
    v[torch.arange(D, device=DEV) * (D + 1)] = 1.0
    C = torch.einsum("uldr,u,l->dr", a, v, v)
    T = torch.einsum("uldr,l->dru", a, v)
    for _ in range(moves):
        c, q = T.shape[0], T.shape[1]
        X = torch.tensordot(torch.tensordot(T, C, dims=([2], [0])), T, dims=([2], [0]))
        X = torch.tensordot(X, a, dims=([1, 2], [1, 0]))
        Cp = X.permute(0, 2, 1, 3).reshape(c * q, c * q)
        w, V = torch.linalg.eigh(Cp @ Cp.conj().T)
        P = V[:, -min(chi, c * q):]
        C = P.conj().T @ Cp @ P
        P = P.reshape(c, q, -1)
        Y = torch.tensordot(P.conj(), T, dims=([0], [0]))
        Z = torch.tensordot(Y, a, dims=([0, 2], [2, 1]))
        T = torch.tensordot(Z, P, dims=([1, 2], [0, 1]))
        C, T = C / C.abs().max(), T / T.abs().max()
    return C, T


def _site(X, A, B, T):
    """Half of the two-site network: X[t, b, x1, x2] closed with the ket tensor A[s, k1, k2, k3, m] and the
    bra tensor B (the same legs) over x1, x2, then with the edge T[b, x3, e] over b and x3:
    out[t, e, s, s', m]."""
    D = A.shape[1]
    t, b = X.shape[:2]
    X = X.reshape(t, b, D, D, D, D)                                              # bra, ket of each leg
    Y = torch.einsum("tbiujv,suvwm->tbijswm", X, A)
    Y = torch.einsum("tbijswm,zijkn->tsmznbkw", Y, B)
    Y = Y.reshape(t, 4 * D * D, b * D * D)
    Y = torch.matmul(Y, T.reshape(b * D * D, -1)).reshape(t, 2, D, 2, D, -1)
    return Y.permute(0, 5, 1, 3, 4, 2).reshape(t, -1, 2, 2, D * D)


def _rho(C, T, A):
    """Two-site density matrix (not normalised) as the C4v network has it: rho[(s1 s2), (t1 t2)]."""
    E = torch.einsum("ta,alc,cb->tlb", C, T, C)
    X = torch.einsum("tlb,tuz->zblu", E, T)                                      # [t', b, l, u]
    left = _site(X, A.permute(0, 2, 1, 3, 4), A.permute(0, 2, 1, 3, 4).conj(), T)
    right = _site(X, A.permute(0, 4, 1, 3, 2), A.permute(0, 4, 1, 3, 2).conj(), T)
    return torch.einsum("tezym,tewxm->zwyx", left, right).reshape(4, 4)


def _rho_complex(C, T, A):
    """The same on the clockwise ring of a complex environment."""
    H = torch.einsum("ac,cxe,eb->axb", C, T, C)
    # left chain from b to t: T[b, d1, c] H[c, l1, e] T[e, u1, t]; right chain T[t, u2, c] H[c, r2, e] T[e, d2, b]
    X = torch.einsum("bdc,cle->bedl", T, H)
    left = _site(X, A.permute(0, 3, 2, 1, 4), A.permute(0, 3, 2, 1, 4).conj(), T)                     # [b, t, ...]
    X = torch.einsum("tuc,cre->teur", T, H)
    right = _site(X, A.permute(0, 1, 4, 3, 2), A.permute(0, 1, 4, 3, 2).conj(), T)                    # [t, b, ...]
    return torch.einsum("btzym,tbwxm->zwyx", left, right).reshape(4, 4)


def _energy(rho, h):
    return torch.real(torch.trace(rho @ h.to(rho.dtype)) / torch.trace(rho))


def _fso_blocks(a, ne):
    """The even-total blocks of a[u, l, d, r]: pairs of legs grouped by parity, row-major inside."""
    q = a.shape[0]
    e, o = range(ne), range(ne, q)
    pairs = {0: [(i, j) for i in e for j in e] + [(i, j) for i in o for j in o],
             1: [(i, j) for i in e for j in o] + [(i, j) for i in o for j in e]}
    m = a.reshape(q * q, q * q)
    out = []
    for b in (0, 1):
        ix = torch.tensor([i * q + j for i, j in pairs[b]], dtype=torch.int64, device=DEV)
        if len(ix):
            out.append(m[ix][:, ix].reshape(-1))
    return torch.cat(out)


def _hotrg(A, chi, steps):
    """(ln Z per site, log norms) of a HOTRG run in the Hermitian basis."""
    a = _rotate(_double_layer(A), _u(A.shape[1]))
    logs = [torch.log(a.abs().max()).item()]
    T = a / a.abs().max()
    for k in range(steps):
        R = T.permute(3, 0, 1, 2) if k % 2 else T
        best = None
        for side in (0, 1):
            S = R.permute(0, 3, 2, 1) if side else R
            u, l, d, r = S.shape
            A1 = torch.einsum("ulkr,umnr->lmkn", S, S).reshape(l * l, -1)
            A2 = torch.einsum("kldr,nmdr->lmkn", S, S).reshape(l * l, -1)
            G = (A1 @ A2.T).reshape(l, l, l, l).permute(0, 2, 1, 3).reshape(l * l, l * l)
            w, V = torch.linalg.eigh(0.5 * (G + G.T))
            keep = min(chi, l * l)
            order = torch.argsort(-w.abs(), stable=True)
            gone = w[order[keep:]].abs().sum().item()
            if best is None or gone < best[0]:
                best = (gone, V[:, order[:keep]])
        V = best[1].reshape(l, l, -1)
        Y = torch.einsum("abL,uakr->Lbukr", V, R)
        Y = torch.einsum("Lbukr,kbds->Ludrs", Y, R)
        Tn = torch.einsum("Ludrs,rsM->uLdM", Y, V)
        logs.append(torch.log(Tn.abs().max()).item())
        Tn = Tn / Tn.abs().max()
        T = Tn.permute(1, 2, 3, 0) if k % 2 else Tn
    tr = torch.einsum("ulul->", T).item()
    ln = logs[0] + sum(logs[k] / 2.0 ** k for k in range(1, steps + 1)) + math.log(tr) / 2.0 ** steps
    return ln, np.array(logs)


def exact(case, seed):
    k = case["kind"]
    if k == "gemm":
        A, B = _gemm_operands(case, seed)
        return A @ B.T
    A = torch.from_numpy(_tensor(case, seed)).to(DEV)
    h = torch.from_numpy(inputs.heisenberg_bond()).to(DEV)
    if k == "double_layer":
        a = _double_layer(A)
        D = case["D"]
        return {"a": a, "blocks": _fso_blocks(_rotate(a, _u(D)), D * (D + 1) // 2)}
    if k == "hotrg":
        # the tensor itself is given up to the sign of each kept state
        log_z, logs = _hotrg(A, case["chi"], case["steps"])
        return {"log_z": log_z, "log_norms": logs, "T": None}
    if k == "run":
        C, T = _ctmrg(A, case["chi"], case["moves"])
        rho = _rho(C, T, A)
        sv = torch.linalg.svdvals(C)
        # T is given up to the sign of each boundary state
        return {"rho": rho, "tr": torch.trace(rho).item(), "trh": torch.trace(rho @ h).item(),
                "spectrum": sv / sv[0], "C": C, "T": None}
    if k == "env":
        return None     # the mixed-precision corner is a projection whose gauge is the solver's own
    if k == "move":
        return {"C": _ctmrg(A, case["chi"], case["warm"] + 1)[0], "T": None}
    if k == "run_grad":
        A = A.requires_grad_(True)
        E = _energy(_rho(*_ctmrg(A, case["chi"], case["moves"]), A), h)
        return {"E": E.detach(), "dA": torch.autograd.grad(E, A)[0]}
    with torch.no_grad():
        C, T = (_ctmrg_complex if case.get("complex") else _ctmrg)(A, case["chi"], case["warm"])
    if k == "rdm2":
        rho = _rho(C, T, A)
        return {"rho": rho, "tr": torch.trace(rho).item(), "trh": torch.trace(rho @ h).item()}
    if k == "one_site":
        H = torch.einsum("ac,cxe,eb->axb", C, T, C)
        up = torch.einsum("aub,brc->acur", H, T)
        down = torch.einsum("cde,ela->acdl", H, T)
        q = T.shape[1]
        eps = up.reshape(-1, q * q).T @ down.reshape(-1, q * q)
        return eps.reshape(q, q, q, q).permute(0, 3, 2, 1)                       # u, r, d, l -> u, l, d, r
    A = A.requires_grad_(True)
    E = _energy((_rho_complex if case["complex"] else _rho)(C, T, A), h)
    return {"E": E.detach(), "dA": torch.autograd.grad(E, A)[0]}
