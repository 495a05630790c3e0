"""Performance cases of the generalized Kohn-Sham eigensolver, through its public calls.

Each case is one call (or one forward and backward) that a program using this package makes:
`Context.solve` for the spin modes, precisions and partial spectra, `Context.solve_batched`
for independent systems of uneven order, `Context.occupy` for the density matrices after
eigenvalues were gathered, `GKSSolve` for gradients, `Context.gemm` for one FP64-accurate
product.  Orders are 13 basis functions per atom, from 8 atoms to 384.

Inputs are localized-basis pencils: atoms on a jittered lattice, on-site levels of 13
functions per atom, and random hopping and overlap elements that decay with the distance of
the two atoms, so that entries range over many decades as in a real basis.  The overlaps are
scaled to condition numbers near 10, which keeps every output (eigenvectors among them)
determined to about 1e-12.  Four electrons per atom, kT 0.01 Ha.
"""
import math

import torch

from paper_2606_09058_gb300 import gks

PER_ATOM = 13


def listed():
    return [
        # the smallest cell: eight atoms at the Gamma point; launches and latency
        {"name": "gamma8", "kind": "solve", "n": 104, "nk": 1, "spin": "collinear", "complex": False},
        # a 64-atom supercell at the Gamma point
        {"name": "gamma64", "kind": "solve", "n": 832, "nk": 1, "spin": "collinear", "complex": False},
        # the same supercell on a 2 x 2 x 2 k mesh, all k-points in one call
        {"name": "kbatch64", "kind": "solve", "n": 832, "nk": 8, "spin": "collinear", "complex": True},
        # two spin channels of an odd-sized system with a shared chemical potential
        {"name": "spin83", "kind": "solve", "n": 1079, "nk": 1, "spin": "spin_polarized", "complex": False},
        # spinor eigenproblem of order 2 n (noncollinear magnetism)
        {"name": "spinor96", "kind": "solve", "n": 1248, "nk": 1, "spin": "noncollinear", "complex": True},
        # only the lowest part of the spectrum at four k-points (ragged order)
        {"name": "partial125", "kind": "solve", "n": 1625, "nk": 4, "spin": "collinear", "complex": True, "n_ev": 700},
        # single-precision start and refinement sweeps
        {"name": "mixed108", "kind": "solve", "n": 1404, "nk": 1, "spin": "collinear", "complex": False,
         "precision": "mixed"},
        # one k-point of a 384-atom supercell
        {"name": "kpoint384", "kind": "solve", "n": 4992, "nk": 1, "spin": "collinear", "complex": True},
        # a 216-atom cluster with gradients with respect to H and S
        {"name": "grad216", "kind": "grad", "n": 2808, "nk": 1, "spin": "collinear", "complex": False, "kT": 0.02},
        # eight independent systems of 16 to 88 atoms in one captured batch, two of them spinors
        {"name": "uneven8", "kind": "batch", "n": 208, "n_max": 1144, "count": 8, "spinors": 2},
        # shared chemical potential, density and energy-density matrices from gathered eigenvalues
        {"name": "occupy128", "kind": "occupy", "n": 1664, "nk": 4, "spin": "collinear", "complex": True},
        # one FP64-accurate complex product
        {"name": "product4096", "kind": "gemm", "m": 4096, "n": 4096, "k": 4096, "complex": True, "opA": "N",
         "opB": "C"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "grad", "batch", "occupy", "gemm"])
    if kind == "solve":
        spin = rng.choice(["collinear", "collinear", "spin_polarized", "noncollinear"])
        cx = spin == "noncollinear" or rng.random() < 0.5
        nk = rng.choice([1, 1, 2, 4, 8]) if spin == "collinear" else 1
        top = {1: 3600, 2: 2600, 4: 1700, 8: 1100}[nk]
        n = _log(rng, 104, top // 2 if spin == "noncollinear" else min(top, 2200) if spin == "spin_polarized" else top)
        case = {"kind": kind, "n": n, "nk": nk, "spin": spin, "complex": cx}
        if n >= 208 and spin == "collinear":
            option = rng.choice(["none", "none", "partial", "mixed"])
            if option == "partial":
                case["n_ev"] = int(n * rng.uniform(0.25, 0.5)) + 1
            elif option == "mixed" and n <= 2200:
                case["precision"] = "mixed"
        return case
    if kind == "grad":
        cx = rng.random() < 0.5
        return {"kind": kind, "n": _log(rng, 104, 2000 if cx else 2808), "nk": 1, "spin": "collinear", "complex": cx,
                "kT": 0.02}
    if kind == "batch":
        return {"kind": kind, "n": _log(rng, 104, 300), "n_max": _log(rng, 600, 1144), "count": rng.randint(3, 8),
                "spinors": rng.randint(0, 2)}
    if kind == "occupy":
        return {"kind": kind, "n": _log(rng, 208, 2500), "nk": rng.choice([1, 2, 4]), "spin": "collinear",
                "complex": rng.random() < 0.7}
    return {"kind": kind, "m": _log(rng, 256, 4096), "n": _log(rng, 256, 4096), "k": _log(rng, 256, 4096),
            "complex": rng.random() < 0.5, "opA": rng.choice(["N", "C"]), "opB": rng.choice(["N", "C"])}


# ----------------------------------------------------------------------------- inputs

def _generator(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + 7919 * salt) % (1 << 62))


def _decay(n, g):
    """exp(-distance / 4 bohr) between the atoms of every pair of basis functions."""
    natoms = -(-n // PER_ATOM)
    side = math.ceil(natoms ** (1 / 3))
    i = torch.arange(natoms, device="cuda")
    grid = torch.stack([i // (side * side), i // side % side, i % side], 1).double()
    pos = 4.6 * grid + 0.4 * (torch.rand(natoms, 3, dtype=torch.float64, device="cuda", generator=g) - 0.5)
    w = torch.exp(-torch.cdist(pos, pos) / 4.0)
    atom = torch.arange(n, device="cuda") // PER_ATOM
    return w[atom][:, atom], atom


def _noise(lead, n, cx, g):
    a = torch.randn(*lead, n, n, dtype=torch.float64, device="cuda", generator=g)
    if cx:
        a = torch.complex(a, torch.randn(*lead, n, n, dtype=torch.float64, device="cuda", generator=g)) * 0.5 ** 0.5
    return (a + a.mH) * 0.5 ** 0.5


def _pencil(n, nk, spin, cx, seed, salt=0):
    g = _generator(seed, salt)
    w, atom = _decay(n, g)
    far = torch.where(atom[:, None] == atom[None, :], torch.zeros_like(w), w)
    width = 2.0 * far.square().sum(1).max().sqrt().clamp_min(1e-3)  # 2-norm of far * noise
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    S = eye + 0.8 / width * far * _noise((nk,), n, cx, g)
    level = torch.linspace(-0.6, 1.5, PER_ATOM, dtype=torch.float64, device="cuda")[torch.arange(n, device="cuda") % PER_ATOM]
    H = torch.diag(level) + 0.6 / width * w * _noise((nk, 2) if spin == "spin_polarized" else (nk,), n, cx, g)
    if spin == "noncollinear":
        mix = 0.2 / width * w.repeat(2, 2) * _noise((nk,), 2 * n, True, g)
        H = torch.block_diag(*([torch.zeros(n, n, dtype=H.dtype, device="cuda")] * 2)) + mix + torch.stack(
            [torch.block_diag(h, h) for h in H])
    return H.contiguous(), S.contiguous()


def _electrons(n):
    return 4.0 * n / PER_ATOM


def _batch_sizes(case):
    lo, hi, c = case["n"], case["n_max"], case["count"]
    return [int(round(lo * (hi / lo) ** (b / (c - 1)))) for b in range(c)]


def _batch_spins(case):
    # the spinors are the second and third smallest systems (their order is 2 n)
    return ["noncollinear" if 1 <= b <= case["spinors"] else "collinear" for b in range(case["count"])]


def prepare(case, seed):
    kind = case["kind"]
    kT = case.get("kT", 0.01)
    if kind == "gemm":
        g = _generator(seed)
        dt = torch.complex128 if case["complex"] else torch.float64
        sa = (case["m"], case["k"]) if case["opA"] == "N" else (case["k"], case["m"])
        sb = (case["k"], case["n"]) if case["opB"] == "N" else (case["n"], case["k"])
        A, B = (torch.randn(*s, dtype=dt, device="cuda", generator=g) for s in (sa, sb))
        return {"case": case, "ctx": gks.Context(), "A": A, "B": B,
                "out": torch.empty(case["m"], case["n"], dtype=dt, device="cuda")}
    if kind == "batch":
        problems = []
        for b, (n, spin) in enumerate(zip(_batch_sizes(case), _batch_spins(case))):
            H, S = _pencil(n, 1, spin, spin == "noncollinear", seed, b + 1)
            problems.append({"H": H, "S": S, "kT": kT, "n_elec": _electrons(n), "spin": spin})
        stream = torch.cuda.Stream()  # a batch is captured on a stream of its own
        stream.wait_stream(torch.cuda.current_stream())
        return {"case": case, "ctx": gks.Context(graph=True, stream=stream), "problems": problems, "out": None}
    n, nk, spin, cx = case["n"], case["nk"], case["spin"], case["complex"]
    if kind == "occupy":
        g = _generator(seed)
        # the eigenvalues of all k-points and this process's eigenvectors
        eps = torch.sort(-0.8 + 2.5 * torch.rand(nk, n, dtype=torch.float64, device="cuda", generator=g), dim=1).values
        C = torch.randn(nk, n, n, dtype=torch.complex128 if cx else torch.float64, device="cuda", generator=g)
        return {"case": case, "ctx": gks.Context(), "eps": eps, "C": C / n ** 0.5, "kT": kT, "ne": _electrons(n)}
    H, S = _pencil(n, nk, spin, cx, seed)
    if kind == "grad":
        target = _pencil(n, nk, spin, cx, seed, 1)[1] * (2.0 * 2.0 / PER_ATOM)
        return {"case": case, "H": H.requires_grad_(), "S": S.requires_grad_(), "target": target, "kT": kT,
                "ne": _electrons(n)}
    ctx = gks.Context(precision=case.get("precision", "fp64"), n_ev=case.get("n_ev", 0))
    return {"case": case, "ctx": ctx, "H": H, "S": S, "kT": kT, "ne": _electrons(n)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        return state["ctx"].gemm(state["A"], state["B"], state["out"], case["opA"], case["opB"])
    if kind == "batch":
        # the outputs of the first pass are used again, so that the captured batch is replayed
        state["out"] = state["ctx"].solve_batched(state["problems"], out=state["out"])
        return [_solution(s) for s in state["out"]]
    if kind == "occupy":
        mu, rho, eb, edm = state["ctx"].occupy(state["eps"], state["C"], state["kT"], state["ne"], spin=case["spin"],
                                               edm=True)
        return {"mu": mu, "rho": rho, "e_band": eb, "edm": edm}
    if kind == "grad":
        H, S = state["H"], state["S"]
        eps, rho, eb, mu = gks.GKSSolve.apply(H, S, state["kT"], state["ne"], case["spin"])
        d = rho - state["target"]
        loss = eb.sum() + (d * d.conj()).real.sum()
        gH, gS = torch.autograd.grad(loss, (H, S))
        return {"eps": eps.detach(), "rho": rho.detach(), "e_band": eb.detach(), "mu": mu, "grad_H": gH, "grad_S": gS}
    return _solution(state["ctx"].solve(state["H"], state["S"], state["kT"], state["ne"], case["spin"]))


def _solution(s):
    return {"eps": s.eps, "C": s.C, "mu": s.mu, "rho": s.rho, "e_band": s.e_band}


# ----------------------------------------------------------------------------- work

def _solve_work(n, nk, spin, cx, n_ev=0):
    M = 2 * n if spin == "noncollinear" else n
    items = 2 * nk if spin == "spin_polarized" else nk
    ev = n_ev or M
    occ = 4.0 * n / PER_ATOM / (1 if spin == "noncollinear" else 2)
    es, f = (16, 4.0) if cx else (8, 1.0)
    # Cholesky, reduction, tridiagonalization, merges (real), two back-transforms, density
    flops = nk * f * n ** 3 / 3 + items * (f * (M ** 3 + 4 / 3 * M ** 3 + 3.0 * M * M * ev + M * M * occ) + 4 / 3 * M ** 3)
    bytes_ = es * (nk * n * n + items * (2.0 * M * M + M * ev)) + 8.0 * items * M
    return bytes_, flops


def work(case):
    kind = case["kind"]
    es, f = (16, 4.0) if case.get("complex") else (8, 1.0)
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": es * (m * k + k * n + m * n), "flops": f * 2.0 * m * n * k}
    if kind == "batch":
        w = [_solve_work(n, 1, s, s == "noncollinear") for n, s in zip(_batch_sizes(case), _batch_spins(case))]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    n, nk = case["n"], case["nk"]
    if kind == "occupy":
        return {"bytes": nk * (es * 3.0 * n * n + 8.0 * n), "flops": nk * f * 2.0 * n * n * (2.0 * n / PER_ATOM)}
    b, fl = _solve_work(n, nk, case["spin"], case["complex"], case.get("n_ev", 0))
    if kind == "grad":  # rho_bar in, C^H rho_bar C and two products C B C^H, both gradients out
        b, fl = b + es * 4.0 * n * n, fl + f * 12.0 * n ** 3
    return {"bytes": b, "flops": fl}


# ----------------------------------------------------------------------------- 64-bit values

def _fermi(eps, kT, ne, gs):
    """mu, f for eps (nk, M) with weights 1 / nk, by bisection to the last bits."""
    wt = gs / eps.shape[0]
    lo, hi = float(eps.min()) - 1.0, float(eps.max()) + 1.0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if wt * float(torch.special.expit((mid - eps) / kT).sum()) < ne:
            lo = mid
        else:
            hi = mid
    mu = 0.5 * (lo + hi)
    return mu, torch.special.expit((mu - eps) / kT)


def _eigen(H, S):
    """eps, C of one pencil with the largest entry of each column real and positive."""
    L = torch.linalg.cholesky(S)
    A = torch.linalg.solve_triangular(L, H, upper=False)
    A = torch.linalg.solve_triangular(L, A.mH, upper=False).mH
    eps, X = torch.linalg.eigh(0.5 * (A + A.mH))
    C = torch.linalg.solve_triangular(L.mH, X, upper=True)
    top = torch.gather(C, 0, C.abs().argmax(0, keepdim=True))
    return eps, C * (top.conj() / top.abs())


def _exact_solve(H, S, spin, kT, ne, n_ev=0):
    nk, M = H.shape[0], H.shape[-1]
    sp = spin == "spin_polarized"
    pairs = [(H[k, s], S[k]) for k in range(nk) for s in range(2)] if sp else [
        (H[k], torch.block_diag(S[k], S[k]) if spin == "noncollinear" else S[k]) for k in range(nk)]
    e, C = zip(*(_eigen(*p) for p in pairs))
    e, C = torch.stack(e), torch.stack(C)
    gs = 2.0 if spin == "collinear" else 1.0
    # spin-polarized: both channels of a k-point carry its whole weight
    mu, f = _fermi(e, kT, ne, 2.0 * gs if sp else gs)
    w = 1.0 / nk
    f = torch.where(f >= 1e-16, f, torch.zeros_like(f))
    rho = (C * (gs * f)[:, None, :]) @ C.mH
    eb = w * gs * (f * e).sum()
    ev = n_ev or M
    lead = (nk, 2) if sp else (nk,)
    return {"eps": e.reshape(*lead, M), "C": C[:, :, :ev].reshape(*lead, M, ev).contiguous(),
            "mu": torch.tensor([mu], dtype=torch.float64), "rho": rho.reshape(*lead, M, M), "e_band": eb.reshape(1)}


def _exact_grad(state):
    H, S, kT = state["H"].detach(), state["S"].detach(), state["kT"]
    r = _exact_solve(H, S, "collinear", kT, state["ne"])
    e, C, mu, rho = r["eps"][0], r["C"][0], float(r["mu"]), r["rho"][0]
    gs = 2.0
    W = C.mH @ (2.0 * (rho - state["target"][0])) @ C
    x = (e - mu) / kT
    f = torch.special.expit(-x)
    fp = -f * torch.special.expit(x) / kT
    a = 0.5 * x
    d = a[:, None] - a[None, :]
    sinhc = torch.where(d.abs() < 1e-4, 1.0 + d * d / 6.0, torch.sinh(d) / torch.where(d == 0, torch.ones_like(d), d))
    D = -sinhc / (4.0 * kT) / torch.cosh(a)[:, None] / torch.cosh(a)[None, :]        # (f_i - f_j) / (e_i - e_j)
    E = 0.5 * (f[:, None] + f[None, :]) + 0.5 * (e[:, None] + e[None, :]) * D        # the same of e f
    g = gs * (f + e * fp)
    dmu = -(gs * fp * W.diagonal().real).sum() - (gs * e * fp).sum()
    g = g + dmu * fp / fp.sum()
    gH = C @ (gs * W * D + torch.diag(g)) @ C.mH
    gS = -C @ (gs * W * E + torch.diag(g * e)) @ C.mH
    return {"eps": r["eps"], "rho": r["rho"], "e_band": r["e_band"], "mu": r["mu"],
            "grad_H": 0.5 * (gH + gH.mH)[None], "grad_S": 0.5 * (gS + gS.mH)[None]}


def exact(case, seed):
    kind = case["kind"]
    st = prepare(case, seed)
    if kind == "gemm":
        A, B = (x if op == "N" else x.mH for x, op in ((st["A"], case["opA"]), (st["B"], case["opB"])))
        return A @ B
    if kind == "occupy":
        e, C = st["eps"], st["C"]
        mu, f = _fermi(e, st["kT"], st["ne"], 2.0)
        f = torch.where(f >= 1e-16, 2.0 * f, torch.zeros_like(f))
        return {"mu": torch.tensor([mu], dtype=torch.float64), "rho": (C * f[:, None, :]) @ C.mH,
                "e_band": (f * e).sum().reshape(1) / e.shape[0], "edm": (C * (f * e)[:, None, :]) @ C.mH}
    if kind == "batch":
        return [_exact_solve(p["H"], p["S"], p["spin"], p["kT"], p["n_elec"]) for p in st["problems"]]
    if work(case)["flops"] > 2.5e12:  # too long on the FP64 units
        return None
    if kind == "grad":
        return _exact_grad(st)
    return _exact_solve(st["H"], st["S"], case["spin"], st["kT"], st["ne"], case.get("n_ev", 0))
