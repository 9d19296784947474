"""Timed cases of the residual engine: what a user has it compute, through Engine.

Each case builds a synthetic Hamiltonian on the GPU (the recipe of the synth package: orbital
energies, Z2 labels, DF factors and Fock noise, seeded) and calls one public entry point:

  residual     Engine.residual    one evaluation of the amplitude equations
  iterations   Engine.solve       a few Jacobi + DIIS iterations from T = 0
  solve        Engine.solve       a converged solve
  vjp          Engine.vjp         reverse mode with respect to T, the DF factors and the Fock matrices

exact() evaluates the same equations with plain torch in 64 bits.
"""
import itertools
import math

import torch

import paper_2401_11935_gb300 as P

METHOD = {"ccsd": 0, "dcsd": 1}
PREC = {"fp64": P.PREC_FP64, "bf16": P.PREC_BF16, "bf16x3": P.PREC_BF16X3, "bf16x6": P.PREC_BF16X6,
        "mixed": P.PREC_MIXED}


def _case(name, call, prec, dims, method="dcsd", ref=0):
    c = {"call": call, "prec": prec, "n_c": dims[0], "n_v": dims[1], "naux": dims[2], "method": method, "ref": ref}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small molecule in a minimal basis, other reference: every launch counts
        _case("residual_fp64_tiny", "residual", "fp64", (2, 5, 12), "ccsd", 1),
        # the smallest named workload, one residual and a whole converged solve
        _case("residual_fp64_c1", "residual", "fp64", (4, 20, 60)),
        _case("solve_fp64_c1", "solve", "fp64", (4, 20, 60)),
        # odd sizes between the first two workloads, CCSD (the exchange rings too)
        _case("residual_fp64_odd", "residual", "fp64", (7, 53, 131), "ccsd"),
        # the second workload in the default precision
        _case("residual_fp64_c2", "residual", "fp64", (10, 120, 360)),
        # gradients in the default precision at a size of the gradient tests
        _case("vjp_fp64", "vjp", "fp64", (6, 60, 120)),
        # a converged mixed-precision solve (BF16, BF16X6, FP64 defect correction)
        _case("solve_mixed", "solve", "mixed", (8, 90, 270)),
        # the refinement precision at the adjoint workload: residual and gradients
        _case("residual_bf16x6_c4", "residual", "bf16x6", (12, 160, 480)),
        _case("vjp_bf16x6_c4", "vjp", "bf16x6", (12, 160, 480)),
        # split precision at odd sizes
        _case("residual_bf16x3_odd", "residual", "bf16x3", (13, 251, 703), "ccsd"),
        # solver iterations of the third workload (update and DIIS included)
        _case("iterations_bf16_c3", "iterations", "bf16", (20, 300, 900)),
        # the benchmark workload: one residual
        _case("residual_bf16_c5", "residual", "bf16", (30, 500, 1500)),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    call, prec = rng.choice([("residual", "fp64"), ("residual", "fp64"), ("residual", "bf16"),
                             ("residual", "bf16x3"), ("residual", "bf16x6"), ("iterations", "bf16"),
                             ("solve", "fp64"), ("solve", "mixed"), ("vjp", "fp64"), ("vjp", "bf16x6")])
    lo, hi = {("residual", "fp64"): (5, 120), ("residual", "bf16"): (40, 450), ("residual", "bf16x3"): (40, 260),
              ("residual", "bf16x6"): (40, 200), ("iterations", "bf16"): (40, 280), ("solve", "fp64"): (5, 30),
              ("solve", "mixed"): (30, 90), ("vjp", "fp64"): (5, 60), ("vjp", "bf16x6"): (40, 150)}[call, prec]
    n_v = _log_int(rng, lo, hi)
    n_c = max(1, min(28, round(n_v * rng.uniform(0.05, 0.2))))
    if n_v > 200:
        n_c = min(n_c, 26)
    if prec == "fp64" or call == "solve":
        n_c = min(n_c, 10)
    naux = max(8, round((n_c + n_v) * rng.uniform(1.8, 2.9)))
    return _case(None, call, prec, (n_c, n_v, naux), rng.choice(["dcsd", "dcsd", "ccsd"]), rng.choice([0, 0, 1]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _system(case, seed):
    """(B, fock_a, fock_b, parity, generator) on the GPU."""
    nc, nv, X = case["n_c"], case["n_v"], case["naux"]
    n, dev = nc + 2 + nv, "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(1000003 * (seed + 1) + 97 * n + X)
    f64 = {"dtype": torch.float64, "device": dev}
    par = torch.randint(0, 2, (n,), generator=g, device=dev)
    par[nc], par[nc + 1] = 0, 1
    aux = torch.randint(0, 2, (X,), generator=g, device=dev)
    eps = torch.empty(n, **f64)
    eps[:nc] = torch.sort(-1.5 + 1.2 * torch.rand(nc, generator=g, **f64)).values
    eps[nc], eps[nc + 1] = -0.2, -0.1
    eps[nc + 2:] = torch.sort(0.2 + 2.8 * torch.rand(nv, generator=g, **f64)).values
    pq = par[:, None] ^ par[None, :]

    def noise():
        x = torch.triu(0.005 * torch.randn(n, n, generator=g, **f64), 1)
        return torch.diag(eps) + (x + x.T) * (pq == 0)

    fa, fb = noise(), noise()
    sigma = 0.05 * min(1.0, (60.0 * 21.0 ** 2 / (X * float(nv + 1) ** 2)) ** 0.25)
    B = torch.randn(X, n, n, generator=g, **f64).mul_(sigma)
    for lo in range(0, X, 64):
        u = torch.triu(B[lo:lo + 64])
        B[lo:lo + 64] = (u + torch.triu(u, 1).transpose(1, 2)) * (pq[None] == aux[lo:lo + 64, None, None])
    return B, fa, fb, par, g


def _orbitals(case, ref):
    """Occupied and virtual orbitals of each spin, in the amplitude layout's order."""
    nc, n = case["n_c"], case["n_c"] + 2 + case["n_v"]
    core, t, u, ext = list(range(nc)), nc, nc + 1, list(range(nc + 2, n))
    act = (t, u) if ref == 0 else (u, t)
    return [core + [act[0]], core + [act[1]]], [[act[1]] + ext, [act[0]] + ext]


def _amplitudes(case, par, g, scale):
    """Symmetry-respecting random amplitudes (the A->B double zero)."""
    occ, vir = _orbitals(case, case["ref"])
    po = [par[torch.tensor(x, device=par.device)].to(torch.int8) for x in occ]
    pv = [par[torch.tensor(x, device=par.device)].to(torch.int8) for x in vir]
    o, v = len(occ[0]), len(vir[0])
    f64 = {"dtype": torch.float64, "device": par.device}
    out = [scale * torch.randn(o, v, generator=g, **f64) * (po[s][:, None] == pv[s][None, :]) for s in (0, 1)]
    for s1, s2 in ((0, 0), (1, 1), (0, 1)):
        x = torch.randn(o, o, v, v, generator=g, **f64).mul_(scale)
        if s1 == s2:
            x = x - x.transpose(0, 1)
            x = x - x.transpose(2, 3)
        x *= (po[s1][:, None, None, None] ^ po[s2][None, :, None, None] ^ pv[s1][None, None, :, None]
              ^ pv[s2][None, None, None, :]) == 0
        if s1 != s2:
            x[o - 1, o - 1, 0, 0] = 0.0
        out.append(x.contiguous())
    return tuple(out)


def prepare(case, seed):
    B, fa, fb, par, g = _system(case, seed)
    s = {"case": case, "T": None, "Rbar": None}
    if case["call"] in ("residual", "vjp"):
        s["T"] = _amplitudes(case, par, g, 1e-3)
    if case["call"] == "vjp":
        s["Rbar"] = _amplitudes(case, par, g, 0.02)
    s["eng"] = P.Engine(case["n_c"], case["n_v"], case["naux"], fa.cpu().numpy(), fb.cpu().numpy(), B.cpu().numpy())
    return s


def run(s):
    c, eng = s["case"], s["eng"]
    method, ref, prec = METHOD[c["method"]], c["ref"], PREC[c["prec"]]
    if c["call"] == "residual":
        return eng.residual(s["T"], ref=ref, method=method, precision=prec)
    if c["call"] == "vjp":
        return eng.vjp(s["T"], Rbar=s["Rbar"], Ebar=1.0, Wbar=0.5, ref=ref, method=method, want_B=True,
                       want_fock=True, precision=prec)
    if c["call"] == "iterations":
        T, r = eng.solve(method=method, ref=ref, precision=prec, tol=1e-30, maxiter=4)
        return T, r.dEA, r.W
    T, r = eng.solve(method=method, ref=ref, precision=prec, tol=1e-10 if c["prec"] == "fp64" else 1e-8, maxiter=80)
    return T, r.E_S, r.E_T


def work(case):
    """Amplitudes and DF factors read once, results written once; the contractions of one residual over
    the independent elements: ladder with symmetric / antisymmetric pairs and its integrals, rings, the
    integrals' other uses.  A converged solve is counted as 15 residuals, a gradient as three."""
    o, v, X = case["n_c"] + 1.0, case["n_v"] + 1.0, float(case["naux"])
    n = o + v + 1
    amp = 8 * (2 * o * v + 3 * o * o * v * v)
    ladder = 2 * o * o * v ** 4 / 2 + 4 * (o * (o - 1) / 2) * (v * (v - 1) / 2) ** 2 + 2 * X * v ** 4 / 4
    ring = (8 if case["method"] == "ccsd" else 6) * 2 * (o * v) ** 3 + 10 * 2 * X * (o * v) ** 2
    small = 3 * 2 * o ** 4 * v * v * 2 + 3 * 2 * 2 * o * o * v ** 3 + 8 * 2 * X * n * n * o
    flops, nbytes = ladder + ring + small, 2 * amp + 8 * X * n * n
    k = {"residual": 1, "iterations": 4, "solve": 15, "vjp": 3}[case["call"]]
    if case["call"] == "vjp":
        nbytes = 3 * amp + 16 * X * n * n
    return {"bytes": nbytes, "flops": k * flops}


# ---------------------------------------------------------------------------
# the equations in plain torch, 64 bits
# ---------------------------------------------------------------------------
# Amplitudes live on spin-free index spaces: occ = (core, t, u), vir = (t, u, ext), zero where an
# orbital is not occupied / virtual for that spin; t2 holds the blocks alpha-alpha, beta-beta, alpha-beta.

def _union_index(case, ref):
    nc = case["n_c"]
    occ, vir = _orbitals(case, ref)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    return ([torch.tensor(x, device=dev) for x in occ], [torch.tensor([p - nc for p in x], device=dev) for x in vir])


def _spread(case, ref, T):
    O, V = case["n_c"] + 2, case["n_v"] + 2
    io, iv = _union_index(case, ref)
    t1 = [torch.zeros(O, V, dtype=torch.float64, device=T[0].device).index_put((io[s][:, None], iv[s][None, :]), T[s])
          for s in (0, 1)]
    t2 = []
    for b, (p, q) in enumerate(((0, 0), (1, 1), (0, 1))):
        ix = (io[p][:, None, None, None], io[q][None, :, None, None], iv[p][None, None, :, None],
              iv[q][None, None, None, :])
        t2.append(torch.zeros(O, O, V, V, dtype=torch.float64, device=T[0].device).index_put(ix, T[2 + b]))
    return t1, t2


def _gather(case, ref, R1, R2):
    io, iv = _union_index(case, ref)
    out = [R1[s][io[s][:, None], iv[s][None, :]] for s in (0, 1)]
    for b, (p, q) in enumerate(((0, 0), (1, 1), (0, 1))):
        out.append(R2[b][io[p][:, None, None, None], io[q][None, :, None, None], iv[p][None, None, :, None],
                         iv[q][None, None, None, :]])
    return out


E = torch.einsum


def _single_reference(case, ref, method, t1, t2, B, fock):
    """Connected CCSD / DCSD residual in the T1-transformed Hamiltonian, and the energy."""
    nc, O = case["n_c"], case["n_c"] + 2
    x, y = (1.0, 1.0) if method == "ccsd" else (0.0, 0.5)
    f = fock if ref == 0 else fock[::-1]
    act = (nc, nc + 1) if ref == 0 else (nc + 1, nc)
    Bov, Bvv = B[:, :O, nc:], B[:, nc:, nc:]
    n = B.shape[1]
    Bd, fd = [], []
    jv = E("Lka,ka->L", Bov, t1[0] + t1[1])
    Jt = E("Lpq,L->pq", B, jv)
    for s in (0, 1):
        tau = torch.zeros(n, n, dtype=B.dtype, device=B.device)
        tau = torch.cat([tau[:nc], torch.cat([t1[s].T, tau[nc:, O:]], 1)], 0)
        one = torch.eye(n, dtype=B.dtype, device=B.device)
        Bd.append((one - tau) @ (B @ (one + tau)))
        occ = list(range(nc)) + [act[s]]
        K = E("Lpk,Lkq->pq", B[:, :, occ], B[:, occ, :])
        Kd = E("Lpk,Lkq->pq", Bd[s][:, :, occ], Bd[s][:, occ, :])
        fd.append((one - tau) @ (f[s] + K + Jt) @ (one + tau) - Kd)
    VO = [b[:, nc:, :O] for b in Bd]
    OO = [b[:, :O, :O] for b in Bd]
    VV = [b[:, nc:, nc:] for b in Bd]
    t2ba = t2[2].permute(1, 0, 3, 2)
    amp = [[t2[0], t2[2]], [t2ba, t2[1]]]
    Z = [E("ikac,Lkc->Lia", amp[s][0], Bov) + E("ikac,Lkc->Lia", amp[s][1], Bov) for s in (0, 1)]
    J = E("Lkc,Lld->klcd", Bov, Bov)
    Foc = [fd[s][:O, :O] + y * E("Lme,Lje->mj", Bov, Z[s]) for s in (0, 1)]
    Fvi = [fd[s][nc:, nc:] - y * E("Lme,Lmb->be", Bov, Z[s]) for s in (0, 1)]
    V = Bvv.shape[1]
    # ladder over the undressed (ac|bd), chunks of a, and its T1 corrections
    stack = torch.stack([t2[0], t2[1], t2[2], t2[2].transpose(2, 3)]).reshape(4 * O * O, V * V)
    step = max(1, int(6e8 // V ** 3))
    lad = [(stack[:3 * O * O] @ E("Lac,Lbd->cdab", Bvv[:, a:a + step], Bvv).reshape(V * V, -1)).reshape(3, O, O, -1, V)
           for a in range(0, V, step)]
    lad = torch.cat(lad, 3)
    G = [(stack @ E("Lkc,Lbd->cdkb", Bov[:, k:k + step], Bvv).reshape(V * V, -1)).reshape(4, O, O, -1, V)
         for k in range(0, O, step)]
    G = torch.cat(G, 3)
    R2 = []
    for b, (p, q) in enumerate(((0, 0), (1, 1), (0, 1))):
        same = p == q
        r = E("Lai,Lbj->ijab", VO[p], VO[q]) + lad[b]
        if same:
            r = r - E("Laj,Lbi->ijab", VO[p], VO[p])
        r = r + E("bc,ijac->ijab", Fvi[q], t2[b]) + E("ac,ijcb->ijab", Fvi[p], t2[b])
        H = E("kmcd,ijcd->ijkm", J, t2[b])
        r = r - E("ka,ijkb->ijab", t1[p], G[b])
        r = r + E("mb,ijma->ijab", t1[q], G[b]) if same else r - E("mb,ijma->ijab", t1[q], G[3])
        r = r + E("ka,ijkb->ijab", t1[p], E("ijkm,mb->ijkb", H, t1[q]))
        Wo = E("Lki,Llj->klij", OO[p], OO[q]) + (0.5 if same else 1.0) * H.permute(2, 3, 0, 1)
        r = r + E("klij,klab->ijab", Wo, t2[b])
        r = r - E("lj,ilab->ijab", Foc[q], t2[b]) - E("ki,kjab->ijab", Foc[p], t2[b])
        R2.append(r)
    # rings
    Jx = J.permute(0, 1, 3, 2)
    U = [E("Lkj,Lbc->kcjb", OO[s], VV[s]) for s in (0, 1)]
    for p in (0, 1):
        for q in (0, 1):
            r = E("Lia,Ljb->iajb", Z[p], VO[q].transpose(1, 2) + 0.5 * Z[q])
            for t in (0, 1):
                if t == q:
                    r = r - E("ikac,kcjb->iajb", amp[p][t], U[t])
                if x:
                    r = r - 0.5 * x * E("ikac,kcjb->iajb", amp[p][t], E("klcd,jlbd->kcjb", Jx, amp[q][t]))
            r = r.permute(0, 2, 1, 3)
            if p == q:
                r = r - r.transpose(0, 1)
                R2[p] = R2[p] + r - r.transpose(2, 3)
            else:
                R2[2] = R2[2] + (r if p == 0 else r.permute(1, 0, 3, 2))
    M1 = -E("Lki,Lbc->kcib", OO[0], VV[1])
    M2 = -E("Lkj,Lac->kcja", OO[1], VV[0])
    if x:
        M1 = M1 + 0.5 * x * E("kldc,ildb->kcib", J, t2[2])
        M2 = M2 + 0.5 * x * E("kldc,ljad->kcja", J, t2[2])
    R2[2] = R2[2] + E("kjac,kcib->ijab", t2[2], M1) + E("ikcb,kcja->ijab", t2[2], M2)
    R1 = []
    for s in (0, 1):
        r = fd[s][nc:, :O].T + E("Lac,Lic->ia", VV[s], Z[s]) - E("Lki,Lka->ia", OO[s], Z[s])
        for t in (0, 1):
            r = r + E("kc,ikac->ia", fd[t][:O, nc:], amp[s][t])
        R1.append(r)
    e = sum((f[s][:O, nc:] * t1[s]).sum() for s in (0, 1)) + (J * t2[2]).sum()
    e = e + E("ijab,ia,jb->", J, t1[0], t1[1])
    for s in (0, 1):
        e = e + 0.5 * ((J * t2[s]).sum() + E("ijab,ia,jb->", J, t1[s], t1[s]) - E("ijab,ib,ja->", J, t1[s], t1[s]))
    return R1, R2, e


def _clusters(I, A):
    """Terms (sign, factors) of <E_I^A Phi| exp(T1 + T2) |Phi>."""
    if not I:
        return [(1, [])]
    out = []
    for p in range(len(A)):
        out += [((-1) ** p * s, [(I[:1], A[p:p + 1])] + f) for s, f in _clusters(I[1:], A[:p] + A[p + 1:])]
    for q in range(1, len(I)):
        for p, r in itertools.combinations(range(len(A)), 2):
            rest = [A[k] for k in range(len(A)) if k not in (p, r)]
            out += [((-1) ** (p + r + q) * s, [([I[0], I[q]], [A[p], A[r]])] + f)
                    for s, f in _clusters(I[1:q] + I[q + 1:], rest)]
    return out


def _excite(det, holes, parts):
    """a+_A1 .. a+_Ak a_Ik .. a_I1 on a sorted tuple of spin orbitals: (determinant, sign), or None."""
    sign = 1
    for h in holes:
        if h not in det:
            return None
        k = det.index(h)
        sign, det = sign * (-1) ** k, det[:k] + det[k + 1:]
    for a in reversed(parts):
        if a in det:
            return None
        k = sum(d < a for d in det)
        sign, det = sign * (-1) ** k, det[:k] + (a,) + det[k:]
    return det, sign


def _coupling(case, ref, t1, t2):
    """c_q = <this determinant excited by q| exp(T_other) |other determinant> for singles and doubles."""
    nc, nv = case["n_c"], case["n_v"]
    n, O, V = nc + 2 + nv, nc + 2, nv + 2
    o1 = [t1[1], t1[0]]                                   # T_other: the spins exchanged
    o2 = [t2[1], t2[0], t2[2].permute(1, 0, 3, 2)]
    occ, vir = _orbitals(case, ref)
    this = tuple(sorted([p for p in occ[0]] + [n + p for p in occ[1]]))
    occ_b, _ = _orbitals(case, 1 - ref)
    other = tuple(sorted([p for p in occ_b[0]] + [n + p for p in occ_b[1]]))
    core, ext = slice(0, nc), slice(2, V)

    def sel(x, kinds):  # one index after the other: a slice or one position
        for d in reversed(range(len(kinds))):
            x = x[(slice(None),) * d + (kinds[d],)]
        return x

    def factor(I, A):
        """(values, letters) of t1 or t2 of the other frame; tokens are (spin, index or slice, letter)."""
        sp = [z[0] for z in I], [z[0] for z in A]
        if sorted(sp[0]) != sorted(sp[1]):
            return None
        if len(I) == 1:
            return sel(o1[sp[0][0]], [I[0][1], A[0][1]]), I[0][2] + A[0][2], 1
        sign = 1
        if sp[0] == [1, 0]:
            I, sign = I[::-1], -sign
        if sp[0][0] != sp[0][1] and sp[1] == [1, 0]:
            A, sign = A[::-1], -sign
        x = o2[2] if sp[0][0] != sp[0][1] else o2[sp[0][0]]
        toks = I + A
        return sel(x, [z[1] for z in toks]), "".join(z[2] for z in toks), sign

    def value(spins, kinds, letters, n_holes):
        """kinds: 'act' or 'free' per index; the coefficient over the free indices."""
        toks, reps, used = [], [], {}
        for k, (s, kind, ch) in enumerate(zip(spins, kinds, letters)):
            hole = k < n_holes
            if kind == "act":
                p = occ[s][nc] if hole else vir[s][0]
                toks.append((s, p if hole else p - nc, ""))
            else:
                m = used.get((s, hole), 0)
                used[s, hole] = m + 1
                if m >= (nc if hole else nv):
                    return None
                p = m if hole else nc + 2 + m
                toks.append((s, core if hole else ext, ch))
            reps.append(s * n + p)
        made = _excite(this, reps[:n_holes], reps[n_holes:])
        det, s1 = made
        I = [g for g in other if g not in det]
        A = [g for g in det if g not in other]
        _, s2 = _excite(other, I, A)
        tok_of = {}
        for r, z in zip(reps, toks):
            tok_of[r] = z

        def tok(g, hole):
            if g in tok_of and tok_of[g][2]:
                return tok_of[g]
            return (g // n, g % n if hole else g % n - nc, "")

        It, At = [tok(g, True) for g in I], [tok(g, False) for g in A]
        total = 0.0
        out = "".join(z[2] for z in toks)
        for sg, facs in _clusters(It, At):
            got = [factor(*f) for f in facs]
            if any(x is None for x in got):
                continue
            for x in got:
                sg *= x[2]
            term = sg if not got else sg * E(",".join(x[1] for x in got) + "->" + out, *[x[0] for x in got])
            total = total + term
        return s1 * s2 * total

    def place(target, spins, kinds, val, n_holes):
        ix = []
        for k, (s, kind) in enumerate(zip(spins, kinds)):
            if k < n_holes:
                ix.append(core if kind == "free" else occ[s][nc])
            else:
                ix.append(ext if kind == "free" else vir[s][0] - nc)
        view = target
        for d in reversed(range(len(ix))):
            view = view[(slice(None),) * d + (ix[d],)]
        view.copy_(val) if torch.is_tensor(val) else view.fill_(val)

    f64 = {"dtype": torch.float64, "device": t1[0].device}
    c1 = [torch.zeros(O, V, **f64) for _ in (0, 1)]
    c2 = [torch.zeros(O, O, V, V, **f64) for _ in range(3)]
    for s in (0, 1):
        for kinds in itertools.product(("act", "free"), repeat=2):
            val = value((s, s), kinds, "ia", 1)
            if val is not None:
                place(c1[s], (s, s), kinds, val, 1)
    for b, (p, q) in enumerate(((0, 0), (1, 1), (0, 1))):
        for kinds in itertools.product(("act", "free"), repeat=4):
            if p == q and ("act", "act") in (kinds[:2], kinds[2:]):
                continue
            val = value((p, q, p, q), kinds, "ijab", 2)
            if val is not None:
                place(c2[b], (p, q, p, q), kinds, val, 2)
        if p == q:
            torch.diagonal(c2[b], dim1=0, dim2=1).zero_()
            torch.diagonal(c2[b], dim1=2, dim2=3).zero_()
    return c1, c2


def _residual(case, T, B, fock):
    """(R in the amplitude layout, W, dE) of the two-determinant equations, differentiable."""
    ref, nc = case["ref"], case["n_c"]
    t1, t2 = _spread(case, ref, T)
    i, j = (nc, nc + 1) if ref == 0 else (nc + 1, nc)
    a, b = (1, 0) if ref == 0 else (0, 1)
    keep = torch.ones_like(t2[2])
    keep[i, j, a, b] = 0.0
    fixed = -t1[0][i, a] * t1[1][j, b]
    t2[2] = t2[2] * keep + (1.0 - keep) * fixed
    R1, R2, e = _single_reference(case, ref, case["method"], t1, t2, B, fock)
    W = R2[2][i, j, a, b] + t1[0][i, a] * R1[1][j, b] + t1[1][j, b] * R1[0][i, a]
    c1, c2 = _coupling(case, ref, t1, t2)
    for k, (p, q) in enumerate(((0, 0), (1, 1), (0, 1))):
        x = E("ia,jb->ijab", t1[p], c1[q])
        if p == q:
            x = x - x.transpose(0, 1)
            x = x - x.transpose(2, 3)
        else:
            x = x + E("ia,jb->ijab", c1[p], t1[q])
        R2[k] = R2[k] - W * (c2[k] - x)
    R1 = [R1[s] - W * c1[s] for s in (0, 1)]
    R2[2] = R2[2] * keep
    return _gather(case, ref, R1, R2), W, e


def _converge(case, B, fock, tol, iters=200):
    """Jacobi steps with DIIS to max|R| <= tol."""
    occ, vir = _orbitals(case, case["ref"])
    f = fock if case["ref"] == 0 else fock[::-1]
    d = [f[s].diagonal() for s in (0, 1)]
    o = [d[s][torch.tensor(occ[s], device=B.device)] for s in (0, 1)]
    v = [d[s][torch.tensor(vir[s], device=B.device)] for s in (0, 1)]
    D = [v[s][None, :] - o[s][:, None] for s in (0, 1)]
    for p, q in ((0, 0), (1, 1), (0, 1)):
        D.append(v[p][None, None, :, None] + v[q] - o[p][:, None, None, None] - o[q][None, :, None, None])
    sizes = [x.numel() for x in D]
    D = [x.expand(y) for x, y in zip(D, [x.shape for x in D])]
    T = [torch.zeros_like(x) for x in D]
    hist_t, hist_e = [], []
    for _ in range(iters):
        R, W, e = _residual(case, T, B, fock)
        if max(float(r.abs().max()) for r in R) <= tol:
            break
        step = torch.cat([(-r / x).reshape(-1) for r, x in zip(R, D)])
        hist_t.append(torch.cat([t.reshape(-1) for t in T]) + step)
        hist_e.append(step)
        hist_t, hist_e = hist_t[-8:], hist_e[-8:]
        m = len(hist_e)
        A = torch.zeros(m + 1, m + 1, dtype=torch.float64)
        for x in range(m):
            for y in range(m):
                A[x, y] = float(torch.dot(hist_e[x], hist_e[y]))
        A[:m, :m] /= max(float(A[:m, :m].abs().max()), 1e-300)
        A[m, :m] = A[:m, m] = -1.0
        rhs = torch.zeros(m + 1, dtype=torch.float64)
        rhs[m] = -1.0
        coef = torch.linalg.solve(A, rhs)[:m] if m > 1 else torch.ones(1, dtype=torch.float64)
        flat = sum(float(k) * t for k, t in zip(coef, hist_t))
        T = [x.reshape(y.shape) for x, y in zip(torch.split(flat, sizes), D)]
    return T, W, e


def exact(case, seed):
    # the FP64 CUDA cores need minutes for one residual of the larger systems
    if case["n_v"] * (case["n_c"] + 2) > 4600 or case["call"] == "iterations":
        return None
    B, fa, fb, par, g = _system(case, seed)
    fock = [fa, fb]
    if case["call"] == "solve":
        T, W, e = _converge(case, B, fock, 1e-12)
        return tuple(T), float(e + W), float(e - W)
    T = _amplitudes(case, par, g, 1e-3)
    if case["call"] == "residual":
        R, W, e = _residual(case, T, B, fock)
        return tuple(R), float(W), float(e)
    Rbar = _amplitudes(case, par, g, 0.02)
    leaves = [x.requires_grad_(True) for x in (*T, B, fa, fb)]
    R, W, e = _residual(case, T, B, fock)
    phi = sum((r * x).sum() for r, x in zip(R, Rbar)) + e + 0.5 * W
    grads = torch.autograd.grad(phi, leaves)
    # the same-spin doubles are redundant (antisymmetric): their gradient as stored is a convention
    return (grads[0], grads[1], None, None, grads[4]), grads[5], grads[6], grads[7]
