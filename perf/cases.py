"""Performance cases of the CTM library: what a user's program asks of it.

Each case is one pass through the public Python entry points (``CTM``,
``Batch``) on synthetic tensors of the sizes that the repository's own
workloads use: the 2x2 ruby cell of d = 8 block sites at D = 2 .. 6 and
chi = 16 .. 144, in the arithmetic forms that those workloads run in.

Kinds of a case:

step      one CTM iteration with its readout: the tensors uploaded and the
          double layers rebuilt, ``sweeps`` sweeps, the two-site RDMs
converge  a coupling point from scratch: ``reset_env``, ``converge`` for at most
          ``sweeps`` sweeps (its corner spectra after each), the one-site RDMs
spectra   one iteration of a monitored convergence: a sweep and the spectra
kappa     a sweep of the mixed network of two neighbouring states of a coupling
          line and its kappa (fidelity)
scan      a batch of instances of uneven D and chi: sweeps, the bond RDMs of all
cylinder  a sweep at a cylinder's bond dimension and its leading spectrum
boundary  dense boundary spectrum and Renyi-2 entropy of a given environment
leading   leading boundary spectrum (Lanczos) of a given environment

The state goes on from pass to pass where a user's program iterates (step,
spectra, kappa, scan, cylinder), after ``warm`` sweeps that the program has
already done; converge starts over each time.  Corner
spectra are read where the contractions are FP64-accurate; the environment
tensors themselves are defined up to a gauge and are not compared.

Numbers of the FP64 forms come back as float64 / complex128.  The BF16 forms
multiply in FP32-class arithmetic (24 significand bits, FP32 accumulation), so
their readouts come back as float32 / complex64, the type of that arithmetic.
"""
import math

import numpy as np
import torch

from paper_1711_04798_gb300 import CTM, Batch

PHYS = 8  # three spins of a triangle block site
NOISE = 0.1
FP64_FORMS = ("fp64", "fp64tc")
CUTOFF = {"fp64": 1e-8, "fp64tc": 1e-8, "bf16x6": 1e-6}


def _case(name, kind, D, chi, prec, sweeps=1, warm=0, lx=2, ly=2, corners=4, nv=0, k=0, real=False, tune=False,
          instances=0, shift=0):
    return {"name": name, "kind": kind, "D": D, "chi": chi, "prec": prec, "sweeps": sweeps, "warm": warm, "lx": lx, "ly": ly,
            "corners": corners, "nv": nv, "k": k, "real": real, "tune": tune, "instances": instances, "shift": shift}


def listed():
    return [
        # the repository's smallest workload (real iid tensors, D = 2, chi = 16): launches and latency
        _case("step_fp64_D2_chi16", "step", 2, 16, "fp64", warm=2, real=True),
        # small convergence in plain FP64, a size between the tuned ones
        _case("converge_fp64_D3_chi27", "converge", 3, 27, "fp64", sweeps=4),
        # an iteration of the FP64 convergence of the D = 4, chi = 64 workload
        _case("spectra_fp64_D4_chi64", "spectra", 4, 64, "fp64"),
        # its fidelity part: the mixed network of two states in the FP64-accurate form
        _case("kappa_fp64tc_D4_chi64", "kappa", 4, 64, "fp64tc", warm=3),
        # ordinary precision-form convergence of one coupling point
        _case("converge_bf16x6_D4_chi64", "converge", 4, 64, "bf16x6", sweeps=5),
        # one-row cell, two-corner projectors, odd chi: single-lane moves
        _case("step_bf16x6_D4_chi53_2x1", "step", 4, 53, "bf16x6", warm=2, lx=2, ly=1, corners=2),
        # the main workload: D = 5, chi = 100, tuned, one iteration with its readout
        _case("step_bf16x6_D5_chi100", "step", 5, 100, "bf16x6", warm=3, tune=True),
        # the same size in the FP64-accurate form: an iteration of the final convergence
        _case("spectra_fp64tc_D5_chi100", "spectra", 5, 100, "fp64tc"),
        # the phase-diagram scan: D in {3, 4, 5} and chi in {32, 48, 64, 100} round robin
        _case("scan_bf16x6_12", "scan", 5, 100, "bf16x6", warm=2, instances=12),
        # the cylinder workload's size, the largest: D = 6, chi = 144
        _case("cylinder_bf16x6_D6_chi144", "cylinder", 6, 144, "bf16x6", warm=1, nv=2, k=8),
        # dense boundary spectrum of a D = 4 cylinder of four block sites
        _case("boundary_fp64tc_D4_chi40", "boundary", 4, 40, "fp64tc", warm=2, nv=4),
        # leading boundary spectrum of a cylinder of six block sites
        _case("leading_bf16x6_D4_chi48", "leading", 4, 48, "bf16x6", warm=2, nv=6, k=24),
    ]


def draw(rng):
    """One more case of the same ranges: the kinds, cells and forms above at
    other D and at chi spread over its logarithm (odd sizes among them)."""
    kind = rng.choice(["step", "step", "step", "converge", "converge", "spectra", "spectra", "kappa", "scan",
                       "boundary", "leading"])
    prec = rng.choice(["fp64", "fp64tc", "fp64tc", "bf16x6", "bf16x6", "bf16x6", "bf16x6"])
    if kind in ("spectra", "kappa"):
        prec = rng.choice(FP64_FORMS)
    if kind == "boundary":
        prec = rng.choice(["fp64tc", "fp64"])
    if kind == "scan":
        prec = "bf16x6"
    top = {"fp64": 64, "fp64tc": 90, "bf16x6": 110}[prec]
    D = rng.choice([2, 3, 4] if prec == "fp64" else [2, 3, 4, 5])
    if kind in ("boundary", "leading"):
        D, top = rng.choice([2, 3, 4]), 48
    if kind == "scan":
        D = rng.choice([3, 4])
    if kind == "converge":
        D, top = min(D, 4), min(top, 72)
    low = max(D * D, 12)
    chi = int(round(math.exp(rng.uniform(math.log(low), math.log(top)))))
    lx, ly = rng.choice([(2, 2), (2, 2), (2, 2), (1, 1), (2, 1), (1, 2)]) if kind in ("step", "converge") else (2, 2)
    nv = {"boundary": 4, "leading": 6}.get(kind, 0)
    k = rng.randint(4, 24) if kind == "leading" else 0
    case = _case("", kind, D, chi, prec, sweeps=rng.randint(2, 4) if kind == "converge" else 1,
                 warm={"converge": 0, "spectra": 0, "kappa": 3}.get(kind, 2), lx=lx, ly=ly,
                 corners=rng.choice([4, 4, 2]) if kind == "step" else 4, nv=nv, k=k,
                 instances=rng.randint(2, 5) if kind == "scan" else 0, shift=rng.randint(0, 999))
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _state_tensors(case, seed, count, D, salt=0, angle=0.0):
    """Site tensors A[p,u,l,d,r]: iid real normals over their largest, or the
    all-up product state plus complex normal noise, at ``angle`` of the line
    cos N1 + sin N2 between two draws of the noise."""
    g = np.random.default_rng([seed, case["shift"], salt, D])
    shape = (PHYS, D, D, D, D)
    out = []
    for _ in range(count):
        if case["real"]:
            A = g.standard_normal(shape)
            out.append(A / np.abs(A).max())
        else:
            n1, n2 = (g.standard_normal(shape) + 1j * g.standard_normal(shape) for _ in range(2))
            A = NOISE * math.sqrt(0.5) * (math.cos(angle) * n1 + math.sin(angle) * n2)
            A[0, 0, 0, 0, 0] += 1.0
            out.append(A)
    return out


def _pattern(lx, ly):
    return [[y * lx + x for x in range(lx)] for y in range(ly)]


def _scan_sizes(case):
    """(D, chi) of each instance: the scan's round robin, largest first, or for
    a drawn scan sizes around the case's own."""
    n = case["instances"]
    if case["D"] == 5 and case["chi"] == 100:
        return [((3, 4, 5)[i % 3], (32, 48, 64, 100)[i % 4]) for i in range(n)]
    return [(case["D"] - i % 2, max(case["D"] ** 2, case["chi"] - 5 * i)) for i in range(n)]


def _inputs(case, seed):
    n = case["lx"] * case["ly"]
    if case["kind"] == "scan":
        return [{"tensors": _state_tensors(case, seed, n, D, i), "pattern": _pattern(case["lx"], case["ly"]),
                 "chi": chi} for i, (D, chi) in enumerate(_scan_sizes(case))]
    ket = _state_tensors(case, seed, n, case["D"])
    bra = _state_tensors(case, seed, n, case["D"], angle=math.pi / 8) if case["kind"] == "kappa" else None
    return {"ket": ket, "bra": bra}


def prepare(case, seed):
    inp = _inputs(case, seed)
    state = {"case": case}
    if case["kind"] == "scan":
        state["batch"] = Batch(inp, tune=False, prec=case["prec"])
        state["batch"].sweep(case["warm"])
        return state
    state["tensors"] = inp["ket"]
    state["ctm"] = CTM(inp["ket"], _pattern(case["lx"], case["ly"]), case["chi"], prec=case["prec"], bra=inp["bra"],
                       corners=case["corners"])
    if case["tune"]:
        state["ctm"].autotune()
    if case["warm"]:
        state["ctm"].sweep(case["warm"])
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _as_form(case, v):
    """A readout in the type of the case's arithmetic."""
    if case["prec"] in FP64_FORMS:
        return v
    if isinstance(v, dict):
        return {k: _as_form(case, x) for k, x in v.items()}
    return v.astype(np.complex64 if np.iscomplexobj(v) else np.float32)


def run(state):
    case = state["case"]
    kind, n = case["kind"], case["sweeps"]
    if kind == "scan":
        b = state["batch"]
        b.sweep(n)
        return [_as_form(case, b.instance(i).rdms()) for i in range(b.n)]
    g = state["ctm"]
    if kind == "step":
        g.set_tensors(state["tensors"])
        g.sweep(n)
        return _as_form(case, g.rdms())
    if kind == "converge":
        g.reset_env()
        done, _, _ = g.converge(1e-13, n)  # below any form's floor: the sweep count is the limit
        return {"sweeps": done, "rho": _as_form(case, g.site_rdms())}
    if kind == "spectra":
        g.sweep(n)
        return g.spectra()
    if kind == "kappa":
        g.sweep(n)
        k = g.kappa()
        return np.array([k.real, k.imag])
    if kind == "cylinder":
        g.sweep(n)
        lam, _, _, _ = g.boundary_rho_topk(0, case["nv"], case["k"], max_iter=36)
        return {"lam": _as_form(case, lam), "rho": _as_form(case, g.site_rdms())}
    if kind == "boundary":
        lam, ent = g.boundary_rho(0, case["nv"])
        s2, purity = g.boundary_renyi2(0, case["nv"])
        return {"lam": lam, "scalars": np.array([ent, s2, purity])}
    lam, ent, rest, _ = g.boundary_rho_topk(0, case["nv"], case["k"])
    return {"lam": _as_form(case, lam), "scalars": _as_form(case, np.array([ent, rest]))}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _sweep_flops(D, chi, lx, ly, corners):
    """Real flops of a sweep: the enlarged corners, the range finder (k = chi +
    16, two subspace iterations) and projectors of each cut, the absorption."""
    D2, N, k = D * D, chi * D * D, chi + 16
    corner = chi ** 3 * D2 + chi ** 3 * D2 ** 2 + chi ** 2 * D2 ** 4
    absorb = 4 * chi ** 3 * D2 + 2 * chi ** 3 * D2 ** 2 + chi ** 2 * D2 ** 4
    cut = corners * corner + 6 * corners * N * N * k + corners * N * N * chi + absorb
    return 8.0 * 4 * lx * ly * cut


def _rdm_flops(D, chi, bonds):
    half = (chi ** 3 * D ** 2 + chi ** 3 * D ** 4 + 2 * PHYS * chi ** 2 * D ** 6 + PHYS * chi ** 3 * D ** 5
            + PHYS ** 2 * chi ** 2 * D ** 4)
    return 8.0 * bonds * (2 * half + PHYS ** 4 * chi ** 2 * D ** 2)


def _site_flops(D, chi, sites):
    return 8.0 * sites * (2 * chi ** 3 * D ** 2 + 2 * chi ** 3 * D ** 4 + chi ** 2 * D ** 6
                          + PHYS * D ** 8 + PHYS ** 2 * D ** 4)


def _env_bytes(D, chi, sites):
    return 16.0 * sites * 4 * (chi * chi + chi * chi * D * D) + 16.0 * sites * PHYS * D ** 4


def work(case):
    D, chi, sites = case["D"], case["chi"], case["lx"] * case["ly"]
    kind, n = case["kind"], case["sweeps"]
    if kind == "scan":
        b = f = 0.0
        for Di, ci in _scan_sizes(case):
            b += 2 * _env_bytes(Di, ci, sites)
            f += n * _sweep_flops(Di, ci, case["lx"], case["ly"], case["corners"]) + _rdm_flops(Di, ci, 2 * sites)
        return {"bytes": b, "flops": f}
    b = 2 * _env_bytes(D, chi, sites)
    f = n * _sweep_flops(D, chi, case["lx"], case["ly"], case["corners"])
    if kind == "step":
        f += _rdm_flops(D, chi, 2 * sites)
    elif kind == "converge":
        f += _site_flops(D, chi, sites)
    elif kind == "kappa":
        f += 8.0 * 2 * (chi * D * D) ** 3
    elif kind == "cylinder":
        f += _site_flops(D, chi, sites)
    elif kind in ("boundary", "leading"):
        v = D ** case["nv"]
        b = 16.0 * 2 * chi * chi * D * D + 8.0 * (case["k"] or v)
        f = 8.0 * 2 * v * v * chi * chi  # both rings
        if kind == "boundary":
            f += 8.0 * 3 * v ** 3
        else:
            f += 8.0 * 2 * v * v * case["k"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same numbers in plain 64-bit torch: the directional CTM with the truncated
# SVD of each cut's ring of enlarged corners
# ---------------------------------------------------------------------------
_E = torch.einsum


def _unit(t):
    return t / torch.linalg.vector_norm(t)


def _pad(t, shape):
    out = torch.zeros(shape, dtype=t.dtype, device=t.device)
    out[tuple(slice(0, s) for s in t.shape)] = t
    return out


class _Net:
    """Network and environment: a, A, C, T as [y][x] (C, T by role first)."""

    def __init__(self, kets, bras, lx, ly, D, chi):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.lx, self.ly, self.D, self.chi = lx, ly, D, chi
        A = [torch.tensor(np.asarray(t, dtype=np.complex128), device=dev) for t in kets]
        B = A if bras is None else [torch.tensor(np.asarray(t, dtype=np.complex128), device=dev) for t in bras]
        self.A = [[A[y * lx + x] for x in range(lx)] for y in range(ly)]
        self.a = [[_E("pulsr,pULSR->uUlLsSrR", A[y * lx + x], B[y * lx + x].conj()).reshape([D * D] * 4)
                   for x in range(lx)] for y in range(ly)]
        # each C / T starts as the neighbouring site with its outward legs traced ket against bra
        off = [(-1, -1, "iijjdr->dr"), (1, -1, "iildjj->ld"), (1, 1, "uliijj->ul"), (-1, 1, "uiijjr->ru"),
               (0, -1, "iildr->ldr"), (1, 0, "uldii->uld"), (0, 1, "uliir->rul"), (-1, 0, "uiidr->dru")]
        traced = ["ul", "ur", "dr", "ld", "u", "r", "d", "l"]
        env = []
        for (dx, dy, spec), legs in zip(off, traced):
            rows = []
            for y in range(ly):
                row = []
                for x in range(lx):
                    s = self.a[(y + dy) % ly][(x + dx) % lx]
                    s = s.reshape([v for q in "uldr" for v in ([D, D] if q in legs else [D * D])])
                    t = _E(spec, s)
                    row.append(_unit(_pad(t, (chi, chi) if t.ndim == 2 else (chi, D * D, chi))))
                rows.append(row)
            env.append(rows)
        self.C, self.T = env[:4], env[4:]

    def turned(self):
        """The network rotated by 90 degrees counter-clockwise: legs relabelled."""
        r = object.__new__(_Net)
        r.lx, r.ly, r.D, r.chi = self.ly, self.lx, self.D, self.chi

        def at(rows, f=lambda t: t):
            return [[f(rows[xp % self.ly][(-yp) % self.lx]) for xp in range(r.lx)] for yp in range(r.ly)]

        r.a = at(self.a, lambda t: t.permute(3, 0, 1, 2).contiguous())
        r.A = at(self.A, lambda t: t.permute(0, 4, 1, 2, 3).contiguous())
        r.C = [at(self.C[(j + 1) % 4]) for j in range(4)]
        r.T = [at(self.T[(j + 1) % 4]) for j in range(4)]
        return r


def _turn(net, k):
    for _ in range(k % 4):
        net = net.turned()
    return net


def _corners(s, x, y, which=(0, 1, 2, 3)):
    x1, y1 = (x + 1) % s.lx, (y + 1) % s.ly
    C, T, a, N = s.C, s.T, s.a, s.chi * s.D ** 2
    Q = [None] * 4
    if 0 in which:
        t = _E("dea,acr->decr", T[3][y][x], _E("ab,bcr->acr", C[0][y][x], T[0][y][x]))
        Q[0] = _E("decr,ceDR->dDrR", t, a[y][x]).reshape(N, N)
    if 1 in which:
        t = _E("Lth,hmE->LtmE", _E("Ltg,gh->Lth", T[0][y][x1], C[1][y][x1]), T[1][y][x1])
        Q[1] = _E("LtmE,tKem->LKEe", t, a[y][x1]).reshape(N, N)
    if 2 in which:
        t = _E("Umg,gtL->UmtL", _E("Umh,hg->Umg", T[1][y1][x1], C[2][y1][x1]), T[2][y1][x1])
        Q[2] = _E("UmtL,uKtm->UuLK", t, a[y1][x1]).reshape(N, N)
    if 3 in which:
        t = _E("gmU,Rtg->mUtR", _E("gh,hmU->gmU", C[3][y1][x], T[3][y1][x]), T[2][y1][x])
        Q[3] = _E("mUtR,umtr->UuRr", t, a[y1][x]).reshape(N, N)
    return Q


def _leading_svd(up, dn, count):
    """Leading singular triplets of X = up^T dn, given as lists of factors."""
    def mul(fs, v):
        for f in reversed(fs):
            v = f @ v
        return v

    X = [f.T for f in reversed(up)] + dn
    XH = [f.conj().T for f in reversed(X)]
    n = X[0].shape[0]
    if n <= 320:
        M = X[0]
        for f in X[1:]:
            M = M @ f
        U, s, Vh = torch.linalg.svd(M.cpu())
        return U.to(M.device), s.to(M.device), Vh.conj().T.to(M.device)
    k = min(n, count + 64)
    gen = torch.Generator().manual_seed(1)
    V = torch.randn(n, k, dtype=torch.complex128, generator=gen).to(X[0].device)
    for _ in range(6):
        V = torch.linalg.qr(mul(XH, torch.linalg.qr(mul(X, V))[0]))[0]
    U, R = torch.linalg.qr(mul(X, V))
    u, s, vh = torch.linalg.svd(R.cpu())
    u, s, vh = (t.to(R.device) for t in (u, s, vh))
    return U @ u, s, V @ vh.conj().T


def _projectors(s, x, y, corners, cutoff):
    Q = _corners(s, x, y, (0, 3) if corners == 2 else (0, 1, 2, 3))
    up, dn = ([Q[0]], [Q[3]]) if corners == 2 else ([Q[0], Q[1]], [Q[3], Q[2].T])
    U, sv, V = _leading_svd(up, dn, s.chi)
    keep = int(min(s.chi, (sv > cutoff * sv[0]).sum()))
    isq = sv[:keep].rsqrt()
    P, Pt = V[:, :keep], U[:, :keep].conj()
    for f in reversed(dn):
        P = f @ P
    for f in reversed(up):
        Pt = f @ Pt
    n = s.chi * s.D ** 2
    shape = (s.chi, s.D ** 2, s.chi)
    P = _pad(P * isq[None, :], (n, s.chi)).reshape(shape)
    return P, _pad((Pt * isq[None, :]).T, (s.chi, n)).reshape(s.chi, s.chi, s.D ** 2)


def _left_move(s, corners, cutoff):
    for x in range(s.lx):
        proj = [_projectors(s, x, y, corners, cutoff) for y in range(s.ly)]
        new = []
        for y in range(s.ly):
            Pm, Ptm = proj[(y - 1) % s.ly]
            P, Pt = proj[y]
            c1 = _E("asr,asn->nr", _E("ab,bsr->asr", s.C[0][y][x], s.T[0][y][x]), Pm)
            t4 = _E("mfhb,gmhr->fbgr", _E("emf,ehb->mfhb", s.T[3][y][x], P), s.a[y][x])
            t4 = _E("fbgr,afg->bra", t4, Ptm)
            c4 = _E("rsu,aus->ra", _E("gu,rsg->rsu", s.C[3][y][x], s.T[2][y][x]), Pt)
            new.append((_unit(c1), _unit(t4), _unit(c4)))
        for y in range(s.ly):
            s.C[0][y][(x + 1) % s.lx], s.T[3][y][(x + 1) % s.lx], s.C[3][y][(x + 1) % s.lx] = new[y]
    return s


def _sweeps(s, n, corners, cutoff):
    for _ in range(n):
        for turn in (0, 2, 1, 3):  # left, right, up, down
            s = _turn(_left_move(_turn(s, turn), corners, cutoff), 4 - turn)
    return s


def _bond(s, x, y):
    D, c, d, x1 = s.D, s.chi, PHYS, (x + 1) % s.lx
    A, B = s.A[y][x], s.A[y][x1]

    def t(j, xx):
        return s.T[j][y][xx].reshape(c, D, D, c)

    L = _E("eLMa,aUVh->eLMUVh", t(3, x), _E("ab,bUVh->aUVh", s.C[0][y][x], t(0, x)))
    L = _E("eLMUVh,pULSr->eMVhpSr", L, A)
    L = _E("eMVhpSr,ekST->MVhprkT", L, _E("ge,kSTg->ekST", s.C[3][y][x], t(2, x)))
    L = _E("MVhprkT,qVMTs->hrskpq", L, A.conj())
    R = _E("hUVf,fRSg->hUVRSg", _E("hUVc,cf->hUVf", t(0, x1), s.C[1][y][x1]), t(1, x1))
    R = _E("hUVRSg,pUlXR->hVSgplX", R, B)
    R = _E("hVSgplX,gXYk->hVSplYk", R, _E("gi,iXYk->gXYk", s.C[2][y][x1], t(2, x1)))
    R = _E("hVSplYk,qVmYS->hlmkpq", R, B.conj())
    rho = _E("hrskpq,hrskPQ->pPqQ", L, R).reshape(d * d, d * d)
    return rho / torch.trace(rho)


def _bonds(s):
    r = s.turned()
    h = [[_bond(s, x, y) for x in range(s.lx)] for y in range(s.ly)]
    v = [[_bond(r, y % r.lx, (-x) % r.ly) for x in range(s.lx)] for y in range(s.ly)]
    return {"h": np.array([[m.cpu().numpy() for m in row] for row in h]),
            "v": np.array([[m.cpu().numpy() for m in row] for row in v])}


def _sites(s):
    out = np.zeros((s.ly, s.lx, PHYS, PHYS), dtype=np.complex128)
    D = s.D
    for y in range(s.ly):
        for x in range(s.lx):
            C, T = [s.C[j][y][x] for j in range(4)], [s.T[j][y][x] for j in range(4)]
            top = _E("aUc,ce->aUe", _E("ab,bUc->aUc", C[0], T[0]), C[1])
            bot = _E("fVi,gi->fVg", _E("hf,iVh->fVi", C[3], T[2]), C[2])
            ring = _E("UefL,eRg->UfLRg", _E("aUe,fLa->UefL", top, T[3]), T[1])
            ring = _E("UfLRg,fVg->ULVR", ring, bot).reshape([D] * 8)
            rho = _E("pULSR,qULSR->pq", _E("uUlLsSrR,pulsr->pULSR", ring, s.A[y][x]), s.A[y][x].conj())
            out[y, x] = (rho / torch.trace(rho)).cpu().numpy()
    return out


def _spectra(s):
    out = np.zeros((4, s.ly, s.lx, s.chi))
    for j in range(4):
        for y in range(s.ly):
            for x in range(s.lx):
                v = np.linalg.svd(s.C[j][y][x].cpu().numpy(), compute_uv=False)
                out[j, y, x] = v / v[0]
    return out


def _kappa(s):
    Q = _corners(s, 0, 0)
    window = ((Q[0] @ Q[1]) * (Q[3] @ Q[2].T)).sum()
    xr, yb = 1 % s.lx, 1 % s.ly
    C = [s.C[0][0][0], s.C[1][0][xr], s.C[2][yb][xr], s.C[3][yb][0]]
    corners = torch.trace(C[0] @ C[1] @ C[2] @ C[3])
    top = _E("aub,bvc->auvc", s.T[0][0][0], s.T[0][0][xr])
    bot = _E("cvb,bua->cvua", s.T[2][yb][xr], s.T[2][yb][0])
    cols = _E("auvc,cvua->", _E("xa,auvc->xuvc", C[0], top), _E("cd,dvue,ex->cvux", C[1] @ C[2], bot, C[3]))
    # T4 [d,r,u] on the left, T2 [u,l,d] on the right
    left = _E("drc,cse->drse", s.T[3][yb][0], s.T[3][0][0])
    right = _E("aub,bvc->auvc", s.T[1][0][xr], s.T[1][yb][xr])
    rows = _E("drse,esrf->df", left, _E("ea,asrc,cf->esrf", C[0] @ C[1], right, C[2] @ C[3]))
    rows = torch.trace(rows)
    k = complex(window * corners / (cols * rows))
    return np.array([k.real, k.imag])


def _rings(s, nv):
    def ring(role, x):
        D, c = s.D, s.chi
        r = None
        for i in range(nv):
            t = s.T[role][i % s.ly][x].reshape(c, D, D, c)
            t = t if role == 1 else t.permute(3, 1, 2, 0)
            if r is None:
                r = t
            elif i < nv - 1:
                r = _E("aKBm,mkbc->aKkBbc", r, t).reshape(c, r.shape[1] * D, r.shape[2] * D, c)
            else:
                r = _E("aKBm,mkba->KkBb", r, t).reshape(r.shape[1] * D, r.shape[2] * D)
        r = r * torch.exp(-1j * torch.angle(torch.trace(r)))
        return (0.5 * (r + r.conj().T)).cpu().numpy()

    return ring(3, 1 % s.lx), ring(1, 0)


def exact(case, seed):
    kind, cut = case["kind"], CUTOFF[case["prec"]]
    done = case["warm"] + (0 if kind in ("boundary", "leading") else case["sweeps"])
    if done * (case["D"] ** 2 * case["chi"] / 2500.0) ** 1.5 > 1.5 or kind == "cylinder":
        return None  # over 20 seconds in 64 bits
    inp = _inputs(case, seed)
    if kind == "scan":
        out = []
        for (D, chi), i in zip(_scan_sizes(case), inp):
            s = _Net(i["tensors"], None, case["lx"], case["ly"], D, chi)
            out.append(_bonds(_sweeps(s, done, case["corners"], cut)))
        return out
    s = _Net(inp["ket"], inp["bra"], case["lx"], case["ly"], case["D"], case["chi"])
    s = _sweeps(s, done, case["corners"], cut)
    if kind == "step":
        return _bonds(s)
    if kind == "converge":
        return {"sweeps": None, "rho": _sites(s)}
    if kind == "spectra":
        return _spectra(s)
    if kind == "kappa":
        return _kappa(s)
    sl, sr = _rings(s, case["nv"])
    if kind == "boundary":
        _, sv, vh = np.linalg.svd(sl.T)
        w = (vh.conj().T * np.sqrt(sv)[None, :]) @ vh
        lam = np.linalg.svd(w @ sr @ w, compute_uv=False)
        lam = lam / lam.sum()
        m = sl.T @ sr
        purity = float(np.real(np.trace(m @ m)) / np.real(np.trace(m)) ** 2)
        p = lam[lam > 0]
        return {"lam": lam, "scalars": np.array([-np.sum(p * np.log(p)), -math.log(purity), purity])}
    return None
