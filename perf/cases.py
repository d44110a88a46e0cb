"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one pass of a program that computes (X)MS-CASPT2 energies, densities or derivatives
at one geometry: new orbitals, integrals and reference densities go in (caspt2_set_inputs),
the amplitudes of all classes are solved, and the results come out.  The sizes are those of
this repository's workloads, tests and serving stream (nclosed 4-42, nact 0-8, nvirt 20-350,
1-4 states).  Inputs are synthetic and seeded, made on the GPU: DF factors with a decaying
singular spectrum, canonical orbital energies, and reference states that are the lowest
singlets of the active-space Hamiltonian, with their spin-free 1- to 4-RDMs.  Orbital
energies and shifts are those of a calculation whose active space is well chosen (no
intruder states), so that every result is determined to the digits that are compared.

`exact` forms the same results in 64 bits from explicit active-space vectors: the class
functions E_Omega|N> become products of active creation and annihilation operators on the
CI vectors, overlaps, Fock matrices and sources their inner products.
"""
import ctypes
import itertools
import math
import types

import numpy as np
import torch

import paper_1606_01273_gb300 as cp

DEV = "cuda"
F8 = torch.float64
CLASSES = "ABCDEFGH"


# ------------------------------------------------------------------------- the cases
def _case(name, call, c, a, v, X, n, **kw):
    """call: what is asked for beside the energies ('energies', 'densities', 'gradient',
    'orbital', 'oneshot', 'serve').  nel: active electrons; form: 'fp64' or 'bf16x' (the
    precision form, 7 slices); canonical: whether the closed and virtual orbitals come as
    eigenvectors of their Fock blocks; ovl: the cut on overlap eigenvalues (larger active spaces
    have nearly dependent class functions, which a calculation drops to keep its digits)."""
    d = {"name": name, "call": call, "nclosed": c, "nact": a, "nvirt": v, "naux": X,
         "nstate": n, "nel": a - a % 2, "form": "fp64", "xms": 1, "scheme": "msmr",
         "shift": 0.2, "target": 0, "canonical": True, "requests": 1,
         "ovl": 1e-6 if a >= 6 else 1e-9}
    d.update(kw)
    return d


def listed():
    return [
        # the smallest solve, as a script's one call on host arrays: context, inputs, solve,
        # densities to host arrays
        _case("oneshot_c4a4v20", "oneshot", 4, 4, 20, 84, 2),
        # one step of a small molecule's optimisation or scan, context and buffers kept
        _case("step_c4a4v20", "densities", 4, 4, 20, 84, 2),
        # odd sizes, three states in the state-specific contraction, precision form, energies
        # only (a single point)
        _case("odd_c5a3v70", "energies", 5, 3, 70, 137, 3, nel=2, scheme="sssr", form="bf16x",
              shift=0.1, target=-1),
        # one state, six active orbitals, densities for a property calculation
        _case("prop_c9a6v83", "densities", 9, 6, 83, 293, 1, shift=0.25),
        # two-state MS gradient with respect to f and B (the autograd form's two calls)
        _case("grad_c12a4v90", "gradient", 12, 4, 90, 318, 2, xms=0),
        # source of the Z-vector equation: orbital derivative with every block of d2
        _case("orb_c6a5v41", "orbital", 6, 5, 41, 157, 2, target=1),
        # localised (non-canonical) closed and virtual orbitals, three states
        _case("local_c8a4v61", "densities", 8, 4, 61, 219, 3, canonical=False, form="bf16x"),
        # a closed-shell molecule: class H alone, plain double precision
        _case("closed_c30v300", "energies", 30, 0, 300, 990, 1, shift=0.0),
        # six different requests at a server of four slots (the serving form)
        _case("serve_6", "serve", 24, 6, 120, 450, 3, requests=6),
        # the 20/8/200 workload, three states: precision form with densities (an optimisation
        # step of a medium molecule), and plain double precision, energies only
        _case("step_c20a8v200", "densities", 20, 8, 200, 700, 3, form="bf16x"),
        _case("fp64_c20a8v200", "energies", 20, 8, 200, 700, 3, target=-1),
        # the largest orbital spaces of the serving range, four states, precision form
        _case("large_c42a6v350", "energies", 42, 6, 350, 1194, 4, form="bf16x", shift=0.3),
    ]


def draw(rng):
    def logi(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["energies", "energies", "densities", "densities", "gradient", "orbital"])
    a = rng.choice([2, 3, 4, 4, 5, 6, 6, 7])
    big = call in ("energies", "densities")
    n = rng.randint(1, 4 if a < 7 else 2)
    if a <= 3:
        n = min(n, 3)
    if a == 2:
        n = min(n, 2)
    c = logi(4, 30 if big else 12)
    v = logi(20, 240 if big else 70)
    d = _case("", call, c, a, v, 3 * (c + a + v) - rng.randint(0, 5), n,
              form=rng.choice(["fp64", "bf16x"]), xms=0 if call == "gradient" else rng.randint(0, 1),
              scheme=rng.choice(["msmr", "msmr", "sssr"]), shift=rng.choice([0.15, 0.2, 0.3]),
              target=rng.randint(0, n - 1), canonical=rng.random() < 0.8)
    if a in (3, 5, 7) and rng.random() < 0.5:
        d["nel"] = a + 1
    d.pop("name")
    return d


# ------------------------------------------------- active-space vectors (inputs, exact)
def _strings(norb, nel):
    return sorted(sum(1 << o for o in occ) for occ in itertools.combinations(range(norb), nel))


_ANN = {}


def _ann(norb, nel, dev):
    """a_p on one spin's strings: [norb, strings(nel - 1), strings(nel)] of 0, +1, -1."""
    key = (norb, nel, str(dev))
    if key not in _ANN:
        src, dst = _strings(norb, nel), {s: i for i, s in enumerate(_strings(norb, nel - 1))}
        A = np.zeros((norb, max(1, len(dst)) if nel > 0 else 0, len(src)))
        for i, s in enumerate(src):
            for p in range(norb):
                if s >> p & 1:
                    A[p, dst[s ^ (1 << p)], i] = (-1.0) ** bin(s & ((1 << p) - 1)).count("1")
        _ANN[key] = torch.tensor(A, dtype=F8, device=dev)
    return _ANN[key]


def _excite(norb, nel, dev):
    """e_pq = a+_p a_q on one spin's strings: [norb, norb, ns, ns]."""
    if nel == 0:
        return torch.zeros(norb, norb, 1, 1, dtype=F8, device=dev)
    A = _ann(norb, nel, dev)
    return torch.einsum("pki,qkj->pqij", A, A)


def _casci(norb, nel, h1, eri, nstate, dev):
    """The lowest singlets (Sz = 0 vectors X[state, alpha, beta], symmetric in alpha, beta)."""
    na = nel // 2
    e = _excite(norb, na, dev)
    ns = e.shape[-1]
    em = e.reshape(norb * norb, ns * ns)
    k = h1 - 0.5 * torch.einsum("rsst->rt", eri)
    one = torch.einsum("pq,pqij->ij", k, e)
    ee = torch.einsum("xy,xik->yik", eri.reshape(norb * norb, -1), e.reshape(-1, ns, ns))
    one = one + 0.5 * torch.einsum("yik,ykj->ij", ee, e.reshape(-1, ns, ns))
    swap = torch.arange(norb * norb, device=dev).reshape(norb, norb).T.reshape(-1)
    two = em.T @ (eri.reshape(norb * norb, -1) @ em - 10.0 * em[swap])   # + 10 S^2
    H = two.reshape(ns, ns, ns, ns).permute(0, 2, 1, 3).reshape(ns * ns, ns * ns).contiguous()
    eye = torch.eye(ns, dtype=F8, device=dev)
    H += torch.kron(one, eye) + torch.kron(eye, one)
    H.diagonal().add_(10.0 * na)
    m = ns * ns
    if m <= 500:
        X = torch.linalg.eigh(H)[1][:, :nstate]
    else:
        # block Davidson from the lowest determinants
        d = H.diagonal().clone()
        V = torch.zeros(m, 4 * nstate, dtype=F8, device=dev)
        lo = torch.argsort(d)[:4 * nstate]
        V[lo, torch.arange(4 * nstate, device=dev)] = 1.0
        for _ in range(60):
            V = torch.linalg.qr(V)[0]
            HV = H @ V
            w, y = torch.linalg.eigh((V.T @ HV).cpu())
            y = y[:, :nstate].to(dev)
            X, R = V @ y, HV @ y
            R -= X * w[:nstate].to(dev)
            if R.norm(dim=0).max() < 1e-11:
                break
            den = d[:, None] - w[:nstate].to(dev)
            den = torch.where(den.abs() < 1e-2, torch.full_like(den, 1e-2), den)
            keep = V if V.shape[1] < 24 * nstate else torch.cat([X, V @ _rest(V, HV, nstate)], 1)
            V = torch.cat([keep, R / den], 1)
    at = X.abs().argmax(0)
    X = X * torch.sign(X[at, torch.arange(nstate, device=dev)])
    X = X.T.reshape(nstate, ns, ns)
    X = 0.5 * (X + X.transpose(1, 2))
    return torch.linalg.qr(X.reshape(nstate, -1).T)[0].T.reshape(X.shape)


def _rest(V, HV, nstate):
    """Ritz vectors nstate .. 2 nstate of a Davidson space (kept at a restart)."""
    w, y = torch.linalg.eigh((V.T @ HV).cpu())
    return y[:, nstate:2 * nstate].to(V.device)


def _tuples(norb, nel, k, dev):
    """a_qk .. a_q1 on one spin's strings for canonical q (q1 < .. < qk): matrices, and for
    every ordered tuple the canonical index and the sign (0 where an orbital repeats)."""
    combos = list(itertools.combinations(range(norb), k))
    M = []
    for q in combos:
        A = torch.eye(len(_strings(norb, nel)), dtype=F8, device=dev)
        for s, p in enumerate(q):
            A = _ann(norb, nel - s, dev)[p] @ A
        M.append(A)
    where = {q: i for i, q in enumerate(combos)}
    idx, sgn = [], []
    for t in itertools.product(range(norb), repeat=k):
        s = tuple(sorted(t))
        if len(set(t)) < k or not combos:
            idx.append(0)
            sgn.append(0.0)
            continue
        inv = sum(1 for x in range(k) for y in range(x + 1, k) if t[x] > t[y])
        idx.append(where[s])
        sgn.append((-1.0) ** inv)
    return (torch.stack(M), torch.tensor(idx, device=dev),
            torch.tensor(sgn, dtype=F8, device=dev))


def _rdm(X, norb, nel, k):
    """Spin-free k-RDMs between the states X: [n, n, p1, q1, .. pk, qk]."""
    n, dev, na = X.shape[0], X.device, nel // 2
    out = torch.zeros((n, n) + (norb,) * (2 * k), dtype=F8, device=dev)
    pairs = [x for j in range(k) for x in (2 + j, 2 + k + j)]
    for ka in range((k + 1) // 2, k + 1):          # alpha operators; the mirror is equal
        kb = k - ka
        if ka > na or kb > na:
            continue
        Ma, ia, sa = _tuples(norb, na, ka, dev)
        Mb, ib, sb = _tuples(norb, na, kb, dev)
        v = torch.einsum("xij,njk->nxik", Ma, X)
        v = torch.einsum("ykj,nxij->nxyik", Mb, v)
        nx, ny = v.shape[1], v.shape[2]
        v = v.reshape(n * nx * ny, -1)
        G = v @ v.T
        idx = (ia[:, None] * ny + ib[None, :]).reshape(-1)
        sg = (sa[:, None] * sb[None, :]).reshape(-1)
        st = torch.arange(n, device=dev)[:, None] * (nx * ny)
        full, s2 = (st + idx).reshape(-1), sg.repeat(n)
        G = G[full] * s2[:, None]
        G = G[:, full]
        G *= s2
        G = G.reshape((n,) + (norb,) * k + (n,) + (norb,) * k)
        G = G.permute(0, k + 1, *range(1, k + 1), *range(k + 2, 2 * k + 2))  # n n p.. q..
        for S in itertools.combinations(range(k), ka):
            order = list(S) + [j for j in range(k) if j not in S]   # position of base slot
            inv = [order.index(j) for j in range(k)]
            g = G.permute(0, 1, *[2 + j for j in inv], *[2 + k + j for j in inv])
            out += (2.0 if ka != kb else 1.0) * g.permute(0, 1, *pairs)
        del G
    return out


def _inputs(case, seed, dev=DEV):
    """Seeded f, B, reference vectors and RDMs of one molecule-like problem."""
    c, a, v, X, n = (case[k] for k in ("nclosed", "nact", "nvirt", "naux", "nstate"))
    nmo = c + a + v
    g = torch.Generator(device="cpu").manual_seed(int(seed) * 7919 + c * 131 + a * 17 + v)
    gd = torch.Generator(device=dev).manual_seed(int(seed) * 104729 + nmo)
    K = min(X, 160)                                    # exp(-k/10) beyond is below 1e-7
    sig = torch.exp(-torch.arange(K, dtype=F8, device=dev) / 10.0)
    alpha = math.sqrt(0.175 / (X * float((sig ** 2).sum())))
    W = torch.randn(K, nmo, nmo, dtype=F8, device=dev, generator=gd)
    W = 0.5 * (W + W.transpose(1, 2))
    # closed and virtual charge distributions are less compact than the active ones
    s = torch.ones(nmo, dtype=F8, device=dev)
    s[:c], s[c + a:] = 0.6, 0.3
    W *= s[:, None] * s[None, :]
    U = torch.randn(X, K, dtype=F8, device=dev, generator=gd) * sig
    B = (alpha * (U @ W.reshape(K, -1))).reshape(X, nmo, nmo)
    del W
    u = lambda k: torch.rand(k, dtype=F8, generator=g).to(dev)  # noqa: E731
    f = torch.zeros(nmo, nmo, dtype=F8, device=dev)
    f.diagonal()[:c] = torch.sort(-2.5 + 1.8 * u(c))[0]
    f.diagonal()[c + a:] = torch.sort(torch.exp(math.log(0.4) + math.log(10.0) * u(v)))[0]
    ci, rdm = None, [torch.zeros(n, n, 1, dtype=F8, device=dev)] * 4   # read for nact > 0 only
    if a > 0:
        act = slice(c, c + a)
        Ba = B[:, act, act].reshape(X, a * a)
        eri = (Ba.T @ Ba).reshape(a, a, a, a)
        t = (0.105 * u(a * a) - 0.0525).reshape(a, a)
        t = torch.triu(t) + torch.triu(t, 1).T
        mean = lambda d: (torch.einsum("rstu,tu->rs", eri, d)  # noqa: E731
                          - 0.5 * torch.einsum("ruts,tu->rs", eri, d))
        fc = t - mean((case["nel"] / a) * torch.eye(a, dtype=F8, device=dev))
        ci = _casci(a, case["nel"], fc, eri, n, dev)
        rdm = [_rdm(ci, a, case["nel"], k).reshape(n, n, -1) for k in (1, 2, 3, 4)]
        dsa = rdm[0].reshape(n, n, a, a).diagonal(dim1=0, dim2=1).mean(-1)
        f[act, act] = fc + mean(dsa)
        f[act, act] = 0.5 * (f[act, act] + f[act, act].T.clone())
    if not case["canonical"]:
        Q = torch.eye(nmo, dtype=F8, device=dev)
        for lo, hi in ((0, c), (c + a, nmo)):
            Q[lo:hi, lo:hi] = torch.linalg.qr(
                torch.randn(hi - lo, hi - lo, dtype=F8, device=dev, generator=gd))[0]
        f = Q.T @ f @ Q
        f[:c, c:] = f[c:c + a, :c] = f[c:c + a, c + a:] = f[c + a:, :c + a] = 0.0
        f = 0.5 * (f + f.T)
        B = Q.T @ B @ Q
    B = 0.5 * (B + B.transpose(1, 2))
    return f.contiguous(), B.contiguous(), ci, rdm


def _requests(case, seed):
    """The requests of a serving pass: sizes spread below the case's own."""
    c, a, v, n = case["nclosed"], case["nact"], case["nvirt"], case["nstate"]
    out = []
    for k in range(case["requests"]):
        q = dict(case, call="energies" if k % 2 else "densities", nclosed=max(4, c - 4 * k),
                 nact=a - k % 3, nvirt=max(20, v - 17 * k), nstate=1 + (n + k) % n,
                 form="bf16x" if k % 3 == 0 else "fp64")
        q["naux"] = 3 * (q["nclosed"] + q["nact"] + q["nvirt"])
        q["nel"] = q["nact"] - q["nact"] % 2
        q["ovl"] = 1e-6 if q["nact"] >= 6 else 1e-9
        out.append((q, seed * 31 + k))
    return out


def _options(case):
    o = dict(xms=case["xms"], scheme=cp.MSMR if case["scheme"] == "msmr" else cp.SSSR,
             shift=case["shift"], target_state=case["target"], ovl_thresh=case["ovl"])
    if case["form"] == "bf16x":
        o.update(precision=cp.BF16X, slices=7)
    if case["call"] == "orbital":
        o.update(dens_offdiag=1)
    return o


def _problem(case, seed):
    """The same inputs as host arrays, in the form that solve_problem and Server.submit take."""
    f, B, _, rdm = _inputs(case, seed)
    return types.SimpleNamespace(
        nclosed=case["nclosed"], nact=case["nact"], nvirt=case["nvirt"], naux=case["naux"],
        nstate=case["nstate"], nmo=f.shape[0], f=f.cpu().numpy(), B=B.cpu().numpy(),
        rdm={k + 1: r.cpu().numpy() for k, r in enumerate(rdm)})


def prepare(case, seed):
    """What a program holds before a pass: the inputs (device tensors, or host arrays where
    the call takes those) and its context or server."""
    if case["call"] == "oneshot":
        return {"case": case, "prob": _problem(case, seed)}
    if case["call"] == "serve":
        req = _requests(case, seed)
        return {"case": case, "req": [(q, _problem(q, s)) for q, s in req],
                "server": cp.Server(budget_bytes=32 << 30, slots=4)}
    f, B, _, rdm = _inputs(case, seed)
    ctx = cp.Context(case["nclosed"], case["nact"], case["nvirt"], case["naux"], case["nstate"],
                     **_options(case))
    return {"case": case, "ctx": ctx, "inputs": (f, B, *rdm)}


# ------------------------------------------------------------------------- one pass
def _energies(case, r):
    out = {"U": r.U, "E0": r.E0, "Href": r.Href, "Heff": r.Heff, "Ems": r.Ems, "R": r.R,
           "Ecore": np.array(r.Ecore), "e": r.e_class, "norm": r.norm_class}
    if case["target"] >= 0:
        out.update(NL=r.lam_NL, lv=r.lam_lv)
    return out


def _device_call(fn, ctx, shapes, *mid):
    """A C-ABI getter with device outputs, as a program that keeps its data on the GPU calls it."""
    outs = [torch.empty(s, dtype=F8, device=DEV) if s else None for s in shapes]
    ptr = [None if t is None else ctypes.c_void_p(t.data_ptr()) for t in outs]
    st = fn(ctx._h, cp.MEM_DEVICE, *ptr, *mid)
    if st < 0:
        raise cp.CASPT2Error(st, fn.__name__)
    return [t for t in outs if t is not None]


def run(state):
    case = state["case"]
    if case["call"] == "oneshot":
        r = cp.solve_problem(state["prob"], densities=True, **_options(case))
        return {**_energies(case, r), "d1": r.d1, "d2": r.d2, "gdf": r.gdf}
    if case["call"] == "serve":
        srv = state["server"]
        tickets = [srv.submit(p, densities=q["call"] == "densities", **_options(q))
                   for q, p in state["req"]]
        keep = ("Ems", "R", "Heff", "d1", "d2", "gdf")
        done = [srv.wait(t) for t in tickets]
        return {str(k): {x: r[x] for x in keep if x in r} for k, r in enumerate(done)}
    ctx = state["ctx"]
    ctx.set_inputs(*state["inputs"])
    out = _energies(case, ctx.result(ctx.solve()))
    nmo, X = case["nclosed"] + case["nact"] + case["nvirt"], case["naux"]
    L = cp.lib()
    if case["call"] == "densities":
        ctx.compute_densities()
        out["d1"], out["d2"], out["gdf"] = _device_call(
            L.caspt2_get_densities, ctx, [(nmo, nmo), (nmo, nmo), None, (X, nmo, nmo)])
    elif case["call"] == "gradient":
        out["gf"], out["gB"] = _device_call(L.caspt2_gradient, ctx,
                                            [(nmo, nmo), (X, nmo, nmo)], None)
    elif case["call"] == "orbital":
        out["Y"], = _device_call(L.caspt2_orbital_derivative, ctx, [(nmo, nmo)], None)
    return out


# ------------------------------------------------------------------------- its least work
def work(case):
    """Bytes: f, B and the RDMs read once, the results written once.  Flops: the class-H pair
    integrals K_ij (i <= j), the integral blocks of the other classes, each sector's two
    eigenproblems (4/3 m^3 for the reduction and 2 m^3 for the vectors) and its transform, the
    n^2 shifted sums (about 8 a term); densities and derivatives cost about twice their
    energies' contractions again."""
    if case["call"] == "serve":
        w = [work(q) for q, _ in _requests(case, 0)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    c, a, v, X, n = (case[k] for k in ("nclosed", "nact", "nvirt", "naux", "nstate"))
    nmo = c + a + v
    el = nmo ** 2 + X * nmo ** 2 + sum(n * n * a ** (2 * k) for k in (1, 2, 3, 4) if a)
    if case["call"] in ("densities", "oneshot"):
        el += (X + 2) * nmo ** 2
    elif case["call"] == "gradient":
        el += (X + 1) * nmo ** 2
    elif case["call"] == "orbital":
        el += nmo ** 2
    one = case["scheme"] == "sssr"
    pairs, vv, cc = c * (c + 1) / 2, v * (v + 1) / 2, c * (c + 1) / 2
    fl = 2.0 * pairs * v * v * X + 8.0 * pairs * v * v * (1 if one else n * n)
    if a:
        ints = (a * a * a * (c + v) + 2 * a * a * c * v + a * a * (cc + vv) + a * c * c * v
                + a * c * v * v)
        fl += 2.0 * X * ints
        rows = {"A": (a ** 3, c), "B": (a * a, cc), "C": (a ** 3, v), "D": (2 * a * a, c * v),
                "E": (2 * a, cc * v), "F": (a * a, vv), "G": (2 * a, vv * c)}
        for m, nt in rows.values():
            ms, reps = (m, n) if one else (m * n, 1)
            fl += reps * (20.0 / 3.0 * ms ** 3 + 2.0 * ms * ms * nt * n + 8.0 * ms * nt * n * n)
    if case["call"] not in ("energies",):
        fl *= 3.0
    return {"bytes": 8.0 * el, "flops": fl}


# ------------------------------------------------------------------------- 64-bit results
def _apply(ops, x, spin):
    """One-spin operator matrices ops[..., i, j] on the vectors x[n, alpha, beta]: the result
    has the operator indices first, then n, alpha, beta (beta operators pass no alpha here: a
    class uses them at one alpha electron number only, where their sign is common)."""
    if spin == 0:
        return torch.einsum("...ij,njk->...nik", ops, x)
    return torch.einsum("...kj,nij->...nik", ops, x)


def _fock(fact, norb, na, nb, x):
    """f_act on vectors x[..., alpha, beta] with na alpha and nb beta electrons."""
    Fa = torch.einsum("pq,pqij->ij", fact, _excite(norb, na, x.device))
    Fb = torch.einsum("pq,pqij->ij", fact, _excite(norb, nb, x.device))
    return Fa @ x + x @ Fb.T


class _Vectors:
    """Active parts of the class functions of the states X, per class: a list of (weight,
    alpha electrons, beta electrons, vectors [rows, n, alpha, beta])."""

    def __init__(self, X, a, nel):
        dev, na = X.device, nel // 2
        n = X.shape[0]
        self.a, self.n = a, n
        A = _ann(a, na, dev)
        Ap = _ann(a, na + 1, dev).transpose(1, 2) if na < a else torch.zeros(
            a, 1, A.shape[2], dtype=F8, device=dev)
        e = _excite(a, na, dev)
        EX = _apply(e, X, 0) + _apply(e, X, 1)                       # [s, t, n, i, k]
        flat = lambda t, k: t.reshape((a ** k,) + t.shape[k:])  # noqa: E731
        lift = lambda M, T: torch.einsum("rij,stnjk->rstnik", M, T)  # noqa: E731
        d = torch.eye(a, dtype=F8, device=dev)
        rX = _apply(A, X, 0)                                         # a_r alpha
        cX = _apply(Ap, X, 0)                                        # a+_r alpha
        wC = lift(A, EX) - torch.einsum("rs,tnik->rstnik", d, rX)
        self.v = {"A": [(2.0, na + 1, na, flat(lift(Ap, EX), 3))],
                  "C": [(2.0, na - 1, na, flat(wC, 3))],
                  "E": [(2.0, na + 1, na, cX)], "G": [(2.0, na - 1, na, rX)]}
        # D: E_ai,rs = sum a+ i E_rs, E_ar,si = -sum a+ i s+ r (spins: equal, opposite)
        dn = -_apply(e.transpose(0, 1), X, 0)
        same = torch.cat([flat(EX, 2), flat(dn, 2)])
        mixed = torch.einsum("rij,skl,njl->rsnik", A, Ap, X)          # r alpha, s+ beta
        mixed = torch.cat([torch.zeros_like(flat(mixed, 2)), flat(mixed, 2)])
        self.v["D"] = [(2.0, na, na, same), (2.0, na - 1, na + 1, mixed)]
        # B, F: distinct holes (particles), and the pair on one orbital
        for k, O, s in (("B", Ap, 1), ("F", A, -1)):
            nn = na + s
            if s > 0:
                O2 = (_ann(a, na + 2, dev).transpose(1, 2) if na + 2 <= a else
                      torch.zeros(a, 1, O.shape[1], dtype=F8, device=dev))
                two = torch.einsum("rij,sjk->rsik", O2, O)
            else:
                O2 = _ann(a, na - 1, dev) if na >= 2 else torch.zeros(
                    a, 1, O.shape[1], dtype=F8, device=dev)
                two = torch.einsum("sij,rjk->rsik", O2, O)
            ab = torch.einsum("rij,skl,njl->rsnik", O, O, X)
            lst = [(2.0, nn, nn, flat(ab, 2))]
            if 0 <= na + 2 * s <= a:
                lst.append((2.0, na + 2 * s, na, flat(_apply(two, X, 0), 2)))
            self.v[k] = lst
            self.v[k + "="] = [(1.0, nn, nn, flat(ab + ab.transpose(0, 1), 2))]

    def matrices(self, key, fact, states=None):
        """S and F_act of a class, rows (function, state); F differentiable in fact."""
        S = F = 0.0
        for w, na, nb, x in self.v[key]:
            if states is not None:
                x = x[:, states]
            m = x.reshape(x.shape[0] * x.shape[1], -1)
            S = S + w * (m @ m.T)
            F = F + w * (m @ _fock(fact, self.a, na, nb, x).reshape(m.shape).T)
        return S, 0.5 * (F + F.T)


def _resolvent_sums(S, A_of, ext, cf, E0, shift, n, one, thresh):
    """Moment sums of one class block over its external tuples: M1[L,N,L'], M2[L,N], M3[L].
    S [rows n, rows n] (rows slowest); A_of(states) the differentiable F; ext [tuples]; cf
    [tuples, rows] the integral coefficients.  The values come from the eigenvectors, held
    fixed, inserted into functionals that are stationary in the solutions, so that derivatives
    with respect to f, ext, E0 and cf are those of the exact sums."""
    R = S.shape[0] // n
    S4 = S.reshape(R, n, R, n)
    M1, M2, M3 = [], [], []
    groups = [[L] for L in range(n)] if one else [list(range(n))]
    done = {}
    for L in range(n):
        grp = [L] if one else groups[0]
        if tuple(grp) not in done:
            Sg = S4[:, grp][:, :, :, grp].reshape(R * len(grp), -1)
            s, Q = torch.linalg.eigh(Sg)
            X = (Q / s.clamp_min(1e-300).sqrt())[:, s >= thresh]
            A = X.T @ A_of(grp) @ X
            A = 0.5 * (A + A.T)
            om, P = torch.linalg.eigh(A.detach())
            A = P.T @ A @ P
            # Z[mu, L', row']: the source of coefficient row' on reference L'
            Z = torch.einsum("xm,xrl->mlr", X @ P, S4[:, grp].reshape(R * len(grp), R, n))
            done[tuple(grp)] = (A, om, torch.einsum("mlr,tr->lmt", Z, cf))
        A, om, b = done[tuple(grp)]
        sh = ext - E0[L] + shift
        bd = b.detach()
        inv = 1.0 / (om[:, None] + sh.detach()[None, :])
        y, z = bd * inv, bd * inv * inv
        Ay = torch.einsum("mk,lkt->lmt", A, y) + y * sh
        M1.append(torch.einsum("amt,bmt->ab", y, b) + torch.einsum("amt,bmt->ab", b, y)
                  - torch.einsum("amt,bmt->ab", y, Ay))
        r = b - Ay                                        # zero in value
        M2.append(torch.einsum("amt,mt->a", y, y[L]) + torch.einsum("mt,amt->a", z[L], r)
                  + torch.einsum("amt,mt->a", z, r[L]))
        M3.append((y[L] * z[L]).sum())
    return torch.stack(M1), torch.stack(M2), torch.stack(M3)


def _moments(case, V, f, h, B, E0, Ftil):
    """Moments of every class, differentiable in the Fock matrix f (denominators), the
    one-electron operator h and B (sources) and E0; closed and virtual orbitals canonical."""
    c, a, v, n = (case[k] for k in ("nclosed", "nact", "nvirt", "nstate"))
    one, Es = case["scheme"] == "sssr", case["shift"]
    C, T, W = slice(0, c), slice(c, c + a), slice(c + a, None)
    eps = f.diagonal()
    ec, ev = eps[C], eps[W]
    mo = {}
    Bv = {k: B[:, x, y].reshape(B.shape[0], -1) for k, x, y in
          (("ca", C, T), ("aa", T, T), ("va", W, T), ("vc", W, C))}
    dim = {"ca": (c, a), "aa": (a, a), "va": (v, a), "vc": (v, c)}

    def eri(x, y):
        return (Bv[x].T @ Bv[y]).reshape(dim[x] + dim[y])

    if a > 0:
        bs = torch.einsum("Pii->P", B[:, C, C])
        fc = h + 2.0 * torch.einsum("P,Pxy->xy", bs, B)
        fc = fc - torch.einsum("Pxj,Pjy->xy", B[:, :, C], B[:, C, :])
        fact, nel = f[T, T], case["nel"]
        d = torch.eye(a, dtype=F8, device=B.device)
        cfA = eri("ca", "aa") + torch.einsum("ir,st->irst", fc[C, T], d) / nel
        cfC = eri("va", "aa") + torch.einsum("ar,st->arst", fc[W, T], d) / (nel - 1)
        D1 = eri("vc", "aa") + torch.einsum("ai,rs->airs", fc[W, C], d) / nel
        D2 = eri("va", "ca").permute(0, 2, 1, 3)                      # (ar|is) -> [a, i, r, s]
        cfD = torch.cat([D1.reshape(v * c, -1), D2.reshape(v * c, -1)], 1)
        jobs = [("A", "A", cfA.reshape(c, -1), -ec),
                ("C", "C", cfC.reshape(v, -1), ev),
                ("D", "D", cfD, (ev[:, None] - ec[None, :]).reshape(-1))]
        for k, pair, e in (("B", "ca", -ec), ("F", "va", ev)):
            g = eri(pair, pair).permute(0, 2, 1, 3)
            g = g.reshape(g.shape[0], g.shape[1], -1)                 # (i r | j s)
            i, j = torch.triu_indices(g.shape[0], g.shape[0], 1, device=B.device)
            q = torch.arange(g.shape[0], device=B.device)
            jobs += [(k, k, g[i, j], e[i] + e[j]), (k, k + "=", 0.5 * g[q, q], 2.0 * e)]
        # E: functions (ai, rj) and (aj, ri): S = g(2, -1), sums with 1 and 3 times g;
        # G: (ar, bi) and (br, ai) likewise
        for k, g in (("E", eri("vc", "ca").permute(1, 2, 0, 3)),      # (ai|rj) -> [i, j, a, r]
                     ("G", eri("va", "vc").permute(0, 2, 3, 1))):     # (ar|bi) -> [a, b, i, r]
            N = g.shape[0]
            i, j = torch.triu_indices(N, N, 1, device=B.device)
            q = torch.arange(N, device=B.device)
            eo, ep, shp = (-ec, ev, v) if k == "E" else (ev, -ec, c)
            x = (eo[i] + eo[j])[:, None] + ep[None, :]
            jobs += [(k, (k, 1.0), ((g[i, j] + g[j, i]) * math.sqrt(0.5)).reshape(-1, a),
                      x.reshape(-1)),
                     (k, (k, 1.0), g[q, q].reshape(-1, a),
                      (2.0 * eo[:, None] + ep[None, :]).reshape(-1)),
                     (k, (k, 3.0), ((g[i, j] - g[j, i]) * math.sqrt(0.5)).reshape(-1, a),
                      x.reshape(-1))]
        for cls, key, cf, ext in jobs:
            sc, vk = (key[1], key[0]) if isinstance(key, tuple) else (1.0, key)
            S, _ = V.matrices(vk, fact.detach())
            part = None
            for lo in range(0, max(1, len(ext)), 1 << 17):
                m = _resolvent_sums(sc * S, lambda st: sc * V.matrices(vk, fact, st)[1],
                                    ext[lo:lo + (1 << 17)], cf[lo:lo + (1 << 17)], E0, Es, n, one,
                                    case["ovl"])
                part = m if part is None else tuple(x + y for x, y in zip(part, m))
            mo[cls] = part if cls not in mo else tuple(x + y for x, y in zip(mo[cls], part))
    # class H: shifted closed-shell pair sums in the eigenbasis of Ftil
    dev = B.device
    om, P = torch.linalg.eigh(Ftil.detach())
    Om = P.T @ Ftil @ P                                               # differentiable, diagonal
    cfh = Bv["vc"]
    M1 = torch.zeros(n, n, n, dtype=F8, device=dev)
    M2, M3 = torch.zeros(n, n, dtype=F8, device=dev), torch.zeros(n, dtype=F8, device=dev)
    cols = cfh.reshape(-1, v, c)
    for i in range(c):
        Ki = (cols[:, :, i].T @ cfh).reshape(v, v, c).permute(2, 0, 1)  # [j, a, b] = (ai|bj)
        k2 = 2.0 * Ki - Ki.transpose(1, 2)
        ext = ev[None, :, None] + ev[None, None, :] - ec[i] - ec[:, None, None]
        for L in range(n):
            if one:
                x = 1.0 / (ext + Es).detach()
                num, xe = (Ki * k2), ext + Es
                M1[L, L, L] = M1[L, L, L] + (num * (2 * x - x * x * xe)).sum()
                M2[L, L] = M2[L, L] + (num * (3 * x * x - 2 * x ** 3 * xe)).sum()
                M3[L] = M3[L] + (num.detach() * x ** 3).sum()
                continue
            xs = [1.0 / (ext.detach() + om[k] - E0[L].detach() + Es) for k in range(n)]
            num, nd = Ki * k2, (Ki * k2).detach()
            xe = ext - E0[L] + Es
            # resolvent of (ext + Om): diagonal and first-order off-diagonal elements
            G1 = torch.zeros(n, n, dtype=F8, device=dev)
            G2 = torch.zeros(n, n, dtype=F8, device=dev)
            for p in range(n):
                xp = xs[p]
                off = xp - xp * xp * (xe + Om[p, p])      # zero in value
                G1[p, p] = G1[p, p] + (num * xp + nd * off).sum()
                G2[p, p] = G2[p, p] + (num * xp * xp + 2 * nd * xp * off).sum()
                for q in range(n):
                    if q != p:
                        xq = xs[q]
                        G1[p, q] = G1[p, q] - (nd * xp * xq).sum() * (Om[p, q] - Om[p, q].detach())
                        G2[p, q] = G2[p, q] - (nd * xp * xq * (xp + xq)).sum() * (
                            Om[p, q] - Om[p, q].detach())
            M1[L] = M1[L] + P @ G1 @ P.T
            M2[L] = M2[L] + (P @ G2 @ P.T)[L]
            M3[L] = M3[L] + sum((P[L, p] ** 2) * (nd * xs[p] ** 3).sum() for p in range(n))
    mo["H"] = (M1, M2, M3)
    z = (torch.zeros_like(M1), torch.zeros_like(M2), torch.zeros_like(M3))
    return {k: mo.get(k, z) for k in CLASSES}


def _canonical(f, c, a):
    """Eigenvectors of the closed and the virtual block of f (differentiable in f)."""
    blocks = [torch.linalg.eigh(0.5 * (f[:c, :c] + f[:c, :c].T))[1],
              torch.eye(a, dtype=F8, device=f.device),
              torch.linalg.eigh(0.5 * (f[c + a:, c + a:] + f[c + a:, c + a:].T))[1]]
    return torch.block_diag(*[b for b in blocks if b.shape[0]])


def _mean_field(B, dact, c, a):
    Ba = B[:, :, c:c + a]
    J = torch.einsum("P,Pxy->xy", torch.einsum("Prs,rs->P", Ba[:, c:c + a], dact), B)
    return J - 0.5 * torch.einsum("Pxt,tu,Pyu->xy", Ba, dact, Ba)


def _signed(M):
    at = M.abs().argmax(0)
    return M * torch.sign(M[at, torch.arange(M.shape[1], device=M.device)])


def exact(case, seed):
    if case["call"] in ("serve", "oneshot"):
        req = [(case, seed)] if case["call"] == "oneshot" else _requests(case, seed)
        outs = [_exact_one(dict(q, call="densities" if case["call"] == "oneshot" else q["call"]), s)
                for q, s in req]
        if case["call"] == "oneshot":
            return outs[0]
        keep = ("Ems", "R", "Heff", "d1", "d2", "gdf")
        return {str(k): {x: o[x] for x in keep if x in o} for k, o in enumerate(outs)}
    return _exact_one(case, seed)


def _exact_one(case, seed, dev=DEV):
    c, a, n = case["nclosed"], case["nact"], case["nstate"]
    f, B, ci, rdm = _inputs(case, seed, dev)
    T = slice(c, c + a)
    P = case["target"]
    want = case["call"]
    if a > 0:
        g1 = rdm[0].reshape(n, n, a, a)
        dsa = g1.diagonal(dim1=0, dim2=1).mean(-1)
        fref = torch.einsum("rs,mnrs->mn", f[T, T], g1)
        U = _signed(torch.linalg.eigh(0.5 * (fref + fref.T))[1]) if case["xms"] else \
            torch.eye(n, dtype=F8, device=dev)
        V = _Vectors(torch.einsum("mn,mik->nik", U, ci), a, case["nel"])
        g1 = torch.einsum("km,ln,klrs->mnrs", U, U, g1)
        g2 = torch.einsum("km,ln,kle->mne", U, U, rdm[1]).reshape((n, n) + (a,) * 4)
    else:
        U, V = torch.eye(n, dtype=F8, device=dev), None
        dsa = torch.zeros(0, 0, dtype=F8, device=dev)
        g1 = torch.zeros(n, n, 0, 0, dtype=F8, device=dev)
        g2 = torch.zeros(n, n, 0, 0, 0, 0, dtype=F8, device=dev)

    def reference(h, B):
        """Core energy and H^ref from h and B."""
        Bc = B[:, :c, :c]
        bs = torch.einsum("Pii->P", Bc)
        J = torch.einsum("P,Pxy->xy", bs, B)
        K = torch.einsum("Pxj,Pjy->xy", B[:, :, :c], B[:, :c, :])
        fc = h + 2.0 * J - K
        core = (h + fc).diagonal()[:c].sum()
        Ba = B[:, T, T].reshape(B.shape[0], -1)
        eri = (Ba.T @ Ba).reshape((a,) * 4)
        H = torch.einsum("rs,mnrs->mn", fc[T, T], g1) + 0.5 * torch.einsum(
            "rstu,mnrstu->mn", eri, g2)
        return core, H + core * torch.eye(n, dtype=F8, device=dev)

    def second(f, h, B):
        """Class moments with the zeroth-order operator f and sources from h and B."""
        C = _canonical(f, c, a)
        fr, hr, Br = C.T @ f @ C, C.T @ h @ C, C.T @ B @ C
        Ft = torch.einsum("rs,mnrs->mn", f[T, T], g1)
        Ft = 0.5 * (Ft + Ft.T)
        return _moments(case, V, fr, hr, Br, Ft.diagonal(), Ft)

    def one_electron(f, B):
        bs = torch.einsum("Pii->P", B[:, :c, :c])
        core = 2.0 * torch.einsum("P,Pxy->xy", bs, B) - torch.einsum(
            "Pxj,Pjy->xy", B[:, :, :c], B[:, :c, :])
        return f - core - (_mean_field(B, dsa, c, a) if a > 0 else 0.0)

    with torch.no_grad():
        h = one_electron(f, B)
        core, Href = reference(h, B)
        mo = second(f, h, B)
    e = {k: -torch.stack([m[0][L, L] for L in range(n)]) for k, m in mo.items()}
    nr = {k: m[1].diagonal() for k, m in mo.items()}
    Heff = Href + sum(0.5 * (x + x.T) for x in e.values())
    Heff = Heff - case["shift"] * torch.diag(sum(nr.values()))
    w, R = torch.linalg.eigh(0.5 * (Heff + Heff.T))
    R = _signed(R)
    E0 = torch.einsum("rs,nnrs->n", f[T, T], g1)
    out = {"U": U, "E0": E0, "Href": Href, "Heff": Heff, "Ems": w, "R": R, "Ecore": core,
           "e": e, "norm": nr}
    if P >= 0:
        r, Es = R[:, P], case["shift"]
        out["NL"] = {k: r * (m[1] @ r) + 2 * Es * r * r * m[2] for k, m in mo.items()}
        out["lv"] = {k: -r[:, None] * torch.einsum("lnk,n->lk", m[0], r)
                     - 2 * Es * (r * r)[:, None] * m[1] for k, m in mo.items()}
    size = case["nvirt"] * case["nclosed"] * max(1, n)
    if want in ("densities", "gradient") and size <= 9000:
        x = [t.clone().requires_grad_(True) for t in (f, h, B)]
        # the energy of state P as a function of (f, h, B); the gradient ties h to f and B
        hh = one_electron(x[0], x[2]) if want == "gradient" else x[1]
        m2 = second(x[0], hh, x[2])
        E = 0.0
        for M1, M2, _ in m2.values():
            ee = -torch.stack([M1[L, L] for L in range(n)])
            E = E + R[:, P] @ ee @ R[:, P] - case["shift"] * (R[:, P] ** 2 * M2.diagonal()).sum()
        sym = lambda t: 0.5 * (t + t.transpose(-1, -2))  # noqa: E731
        if want == "gradient":
            E = E + R[:, P] @ reference(hh, x[2])[1] @ R[:, P]
            gf, gB = torch.autograd.grad(E, [x[0], x[2]])
            mask = torch.block_diag(*[torch.ones(k, k, dtype=F8, device=dev) for k in
                                      (c, a, case["nvirt"]) if k])
            out["gf"], out["gB"] = sym(gf) * mask, sym(gB)
        else:
            g = torch.autograd.grad(E, x, allow_unused=True)
            g = [torch.zeros_like(t) if y is None else y for t, y in zip(x, g)]
            mask = torch.block_diag(*[torch.ones(k, k, dtype=F8, device=dev) for k in
                                      (c, a, case["nvirt"]) if k])
            out["d2"], out["d1"], out["gdf"] = sym(g[0]) * mask, sym(g[1]), sym(g[2])
    return out
