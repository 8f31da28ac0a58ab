"""Performance cases of the GSE-TDVP1 library: the calls a user's program makes, through the
public binding (paper_2005_06104_gb300.gse_tdvp), over the sizes the method meets.

Families
  heff     one H_eff apply on caller operands (gse_tdvp.heff_contract)
  site     the FP64 contractions around one site: both environment updates and the bond
           operator (env_contract, keff_contract)
  expm     one local exponential (expm_contract): the Lanczos run of every site update
  observe  the local S^z profile of a state, which walks the orthogonality centre over the
           whole chain (GseTdvp.expect_local)
  sweep    one real-time TDVP1 sweep of a kept handle, its state read back, its energy
  step     a script's whole GSE-TDVP1 step from host tensors: create, expand, sweep, read out
  tdvp2    the same with a two-site TDVP step
  batch    a step of several random-field chains on one GPU (GseTdvpBatch), read out
A step that extends or truncates the bases fixes its tensors only up to a gauge: what is read out
of it are the numbers a run records (energy, norm, bond dimensions, S^z profile).  A real-time
sweep cuts nothing, so its tensors come back whole.

Lattices are those of workloads.py; "chain" (MPO bond dimension 5), "ladder" (8), "cylinder"
(up to 14) and "oat" (3).  States are seeded random MPS: charge-conserving (u1) as every
Heisenberg run from a Neel state is, or dense, with bond weights spread over decades the way
evolved states are.
"""
import math

import numpy as np
import torch

from paper_2005_06104_gb300 import gse_tdvp as g
from paper_2005_06104_gb300 import workloads as wl

PREC = {"fp64": g.PREC_FP64, "bf16x10": g.PREC_BF16X10, "bf16x6": g.PREC_BF16X6}
LATTICE_W = {"chain": 5, "oat": 3, "ladder": 8, "cylinder": 14}
ITERATIONS = 8  # Krylov vectors of a local exponential at the time steps in use


def listed():
    return [
        # a local operator of a small chain (10-site chain, chi <= 16): latency and launches
        dict(name="heff_fp64_chain16", family="heff", precision="fp64", lattice="chain", ml=16, mr=16),
        # the default precision's site update on the 2 x L ladder, ragged sizes just past one tile
        dict(name="expm_fp64_ladder129", family="expm", precision="fp64", lattice="ladder", ml=129, mr=127, u1=False,
             kind="real"),
        # environment updates and bond operator of a wide cylinder at an odd bond dimension
        dict(name="site_fp64_cyl_300x277", family="site", lattice="cylinder", ml=300, mr=277),
        # one FP64 apply at the ladder workload's cap on the widest MPO
        dict(name="heff_fp64_cyl512", family="heff", precision="fp64", lattice="cylinder", ml=512, mr=512),
        # the precision form on operands without a conserved charge, environments new on every call
        dict(name="heff_bf16x10_cyl1024", family="heff", precision="bf16x10", lattice="cylinder", ml=1024, mr=1024),
        # the site update of the cylinder benchmark at its cap: charge-conserving environments
        dict(name="expm_bf16x10_u1_cyl1024", family="expm", precision="bf16x10", lattice="cylinder", ml=1024, mr=1024,
             u1=True, kind="real"),
        # reading the magnetisation profile of a large state: gauge moves over the whole chain
        dict(name="observe_cyl24_chi384", family="observe", lattice="cylinder", sites=24, chi=384, u1=True),
        # a production sweep in the precision form
        dict(name="sweep_bf16x10_cyl24_chi256", family="sweep", precision="bf16x10", lattice="cylinder", sites=24,
             chi=256, u1=True),
        # a whole step with the benchmark's settings (Krylov vectors in BF16X6), ends of the chain growing
        dict(name="step_bf16x10_cyl20_chi128", family="step", precision="bf16x10", krylov="bf16x6",
             lattice="cylinder", sites=20, chi=128, u1=True, kind="real", k=3),
        # imaginary time with the default precision, dense blocks, truncating SVDs
        dict(name="step_fp64_imag_ladder20_chi40", family="step", precision="fp64", krylov="fp64", lattice="ladder",
             sites=20, chi=40, u1=False, kind="imag", k=3),
        # the two-site integrator on the ladder, charge-conserving
        dict(name="tdvp2_fp64_ladder16_chi64", family="tdvp2", precision="fp64", lattice="ladder", sites=16, chi=64,
             u1=True, kind="real"),
        # disorder realisations: short chains at the bond dimensions such a batch reaches
        dict(name="batch_fp64_4chains_chi16", family="batch", precision="fp64", chains=4, shortest=12, longest=20,
             chi=16, k=2),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["heff", "heff", "site", "expm", "expm", "observe", "sweep", "step", "tdvp2", "batch"])
    lattice = rng.choice(["chain", "ladder", "cylinder"])
    if family == "heff":
        precision = rng.choice(["fp64", "fp64", "bf16x10", "bf16x6"])
        lattice = rng.choice(["chain", "oat", "ladder", "cylinder"])
        top = 512 if precision == "fp64" else 1024
        m = log(8, top)
        return dict(family=family, precision=precision, lattice=lattice, ml=m, mr=min(top, log(max(4, m / 2), 2 * m)))
    if family == "site":
        m = log(8, 300)
        return dict(family=family, lattice=lattice, ml=m, mr=min(300, log(max(4, m / 2), 2 * m)))
    if family == "expm":
        precision = rng.choice(["fp64", "bf16x10"])
        u1 = rng.random() < 0.5
        top = (1024 if u1 else 640) if precision != "fp64" else 160
        m = log(8 if precision == "fp64" else 96, top)
        return dict(family=family, precision=precision, lattice=lattice, ml=m, mr=min(top, log(max(4, m / 1.5), 1.5 * m)),
                    u1=u1, kind=rng.choice(["real", "imag"]))
    if family == "batch":
        a = rng.randint(8, 14)
        return dict(family=family, precision="fp64", chains=rng.randint(2, 4), shortest=a, longest=a + rng.randint(1, 6),
                    chi=log(4, 16), k=rng.choice([2, 3]))
    sites = 4 * rng.randint(3, 5) if lattice == "cylinder" else 2 * rng.randint(5, 10)
    if family == "observe":
        return dict(family=family, lattice=lattice, sites=sites, chi=log(16, 320), u1=rng.random() < 0.7)
    if family == "sweep":
        p = rng.choice(["fp64", "bf16x10"])
        return dict(family=family, precision=p, lattice=lattice, sites=sites, chi=log(12, 56 if p == "fp64" else 200),
                    u1=True)
    kind = rng.choice(["real", "imag"])
    if family == "tdvp2":
        return dict(family=family, precision="fp64", lattice=lattice, sites=min(sites, 16), chi=log(8, 48), u1=True,
                    kind=kind)
    p = rng.choice(["fp64", "bf16x10"])
    return dict(family=family, precision=p, krylov="fp64" if p == "fp64" else "bf16x6", lattice=lattice,
                sites=min(sites, 16), chi=log(8, 32 if p == "fp64" else 96), u1=kind == "real", kind=kind,
                k=rng.choice([2, 3]))


# ---------------------------------------------------------------- inputs
def _lattice(name, sites):
    if name == "cylinder":
        return wl.cylinder_snake(sites // 4, 4)
    return wl.zigzag_ladder(sites // 2, 1.0, 1.0) if name == "ladder" else wl.chain(sites)


def _mpo_site(name):
    """The widest site tensor of the lattice's MPO and the charges of its channels (2 S^z)."""
    W = wl.oat_mpo(8) if name == "oat" else wl.heisenberg_mpo(_lattice(name, 24))
    i = max(range(len(W)), key=lambda k: (W[k].shape[0] * W[k].shape[3], -abs(k - len(W) // 2)))
    ch = wl.mpo_channel_charges(W)
    return W[i], ch[i], ch[i + 1]


def _randn(gen, *shape):
    re, im = (torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64) for _ in range(2))
    return torch.complex(re, im)


def _site_operands(case, seed):
    """Dense Gaussian environments, site tensor and bond matrix, normalised as in the tests."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    W, _, _ = _mpo_site(case["lattice"])
    ml, mr, d = case["ml"], case["mr"], W.shape[1]

    def rnd(*shape):
        return _randn(gen, *shape) / math.sqrt(shape[-1])
    return W, rnd(ml, W.shape[0], ml), rnd(mr, W.shape[3], mr), rnd(ml, d, mr), rnd(ml, mr)


def _bond_charges(m, parity):
    """m charges of one parity in contiguous sectors, binomial sizes (widest at charge ~0)."""
    q = np.arange(-8 + parity, 9, 2)
    p = np.exp(-0.18 * q.astype(float) ** 2)
    n = np.maximum((m * p / p.sum()).astype(int), 1 if m >= len(q) else 0)
    while n.sum() > m:
        n[np.argmax(n)] -= 1
    n[len(q) // 2] += m - n.sum()
    return torch.from_numpy(np.repeat(q, n)).cuda()


def _environment(gen, q, charges, identity, block):
    """A Hermitian set of channel matrices E[a, w, a'] like those of a canonical MPS: the identity
    channel, the finished terms (norm about 6) and spin operators (norm about 1/2) whose S^+ and
    S^- channels are each other's adjoints; nonzero where q_a = q_a' + c_w when charges are kept."""
    m, w = q.numel(), len(charges)
    E = torch.zeros(m, w, m, dtype=torch.complex128, device="cuda")

    def mat(c, scale):
        x = _randn(gen, m, m) * (scale / math.sqrt(2.0 * m))
        return x * (q[:, None] == q[None, :] + c) if block else x
    E[:, identity, :] = torch.eye(m, dtype=torch.complex128, device="cuda")
    x = mat(0, 3.0)
    E[:, w - 1 - identity, :] = x + x.conj().T
    for k in range(1, w - 1, 3):
        z = mat(0, 0.25)
        E[:, k, :] = z + z.conj().T
        p = mat(int(charges[k + 1]), 0.25)
        E[:, k + 1, :] = p
        E[:, k + 2, :] = p.conj().T
    return E


def _expm_operands(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    W, cl, cr = _mpo_site(case["lattice"])
    ml, mr, d = case["ml"], case["mr"], W.shape[1]
    ql, qr = _bond_charges(ml, 0), _bond_charges(mr, 1)
    L = _environment(gen, ql, cl, 0, case["u1"])
    R = _environment(gen, qr, cr, W.shape[3] - 1, case["u1"])
    x = _randn(gen, ml, d, mr)
    if case["u1"]:
        ph = torch.tensor(wl.SZ2, device="cuda")
        x = x * (qr[None, None, :] == ql[:, None, None] + ph[None, :, None])
    return W, L, R, x / torch.linalg.norm(x)


def _state(n, chi, seed, u1):
    """A normalisable random MPS with bond weights spread over half a decade (u1) or a decade."""
    mps = wl.random_u1_mps(n, chi, seed, shuffle=False) if u1 else wl.random_isometric_mps(n, chi, seed)
    rng = np.random.default_rng([seed, 1])
    for a in mps[:-1]:
        a *= 10.0 ** (-(0.5 if u1 else 1.0) * rng.random(a.shape[2]))
    psi = np.ones((1, 1), dtype=np.complex128)  # <psi|psi>, to normalise
    for a in mps:
        t = np.tensordot(psi, a, axes=([1], [0]))
        psi = np.tensordot(a.conj(), t, axes=([0, 1], [0, 1]))
    mps[-1] = mps[-1] / math.sqrt(psi[0, 0].real)
    return mps


def _step_options(case, lat):
    real = case.get("kind", "real") == "real"
    return dict(tau=0.1 if real else -1j / wl.lambda_top(lat), eps_k=1e-8 if real else 1e-12, eps_m=1e-8,
                eps=(1e-10 if not real else 1e-9 if case["family"] == "tdvp2" else 0.0), chi_max=case["chi"],
                precision=PREC[case.get("precision", "fp64")])


def prepare(case, seed):
    f = case["family"]
    s = dict(case=case)
    if f in ("heff", "site"):
        W, L, R, x, c = _site_operands(case, seed)
        s.update(W=W, L=L, R=R, x=x, c=c, y=torch.empty_like(x))
        if f == "site":
            s.update(Lo=torch.empty(case["mr"], W.shape[3], case["mr"], dtype=torch.complex128, device="cuda"),
                     Ro=torch.empty(case["ml"], W.shape[0], case["ml"], dtype=torch.complex128, device="cuda"),
                     yc=torch.empty_like(c),
                     # the bond operator's two environments share one channel count
                     Rb=_randn(torch.Generator(device="cuda").manual_seed(seed + 7), case["mr"], W.shape[0],
                               case["mr"]) / math.sqrt(case["mr"]))
    elif f == "expm":
        W, L, R, x = _expm_operands(case, seed)
        s.update(W=W, L=L, R=R, x=x, y=torch.empty_like(x))
    elif f == "batch":
        rng = np.random.default_rng([seed, 2])
        s["chains"] = []
        for i in range(case["chains"]):
            n = 2 * (int(rng.integers(case["shortest"], case["longest"] + 1)) // 2)
            lat = wl.chain(n, 1.0, fields=rng.uniform(-2.0, 2.0, size=n))
            s["chains"].append((_state(n, case["chi"], seed + 100 + i, True), wl.heisenberg_mpo(lat),
                                dict(tau=0.05, chi_max=2 * case["chi"], eps_k=1e-8, eps_m=1e-8,
                                     precision=PREC[case["precision"]])))
    else:
        lat = _lattice(case["lattice"], case["sites"])
        s.update(mpo=wl.heisenberg_mpo(lat), mps=_state(case["sites"], case["chi"], seed, case["u1"]),
                 opts=_step_options(case, lat))
        if f in ("observe", "sweep"):
            s["handle"] = g.GseTdvp(s["mps"], s["mpo"], **s["opts"])
    return s


def run(s):
    case = s["case"]
    f = case["family"]
    if f == "heff":
        g.heff_contract(s["L"], s["W"], s["R"], s["x"], s["y"], precision=PREC[case["precision"]])
        return s["y"]
    if f == "site":
        g.env_contract(0, s["L"], s["W"], s["x"], s["Lo"])
        g.env_contract(1, s["R"], s["W"], s["x"], s["Ro"])
        g.keff_contract(s["L"], s["Rb"], s["c"], s["yc"])
        return dict(left=s["Lo"], right=s["Ro"], bond=s["yc"])
    if f == "expm":
        real = case["kind"] == "real"
        it = g.expm_contract(s["L"], s["W"], s["R"], s["x"], s["y"], 0.05, kind=g.REAL if real else g.IMAG,
                             precision=PREC[case["precision"]])
        return dict(y=s["y"], iterations=it)
    if f == "observe":
        h = s["handle"]
        return np.array([h.expect_local(wl.SZ, i) for i in range(case["sites"])])
    if f == "sweep":
        h = s["handle"]
        h.sweep(0.1, g.REAL)
        return dict(energy=h.energy(), mps=h.get_mps())
    if f == "batch":
        b = g.GseTdvpBatch(s["chains"])
        b.step(0.05, g.REAL, case["k"])
        out = dict(energies=np.array(b.energies()), norms=np.array(b.norms()),
                   sz=np.array([b.chain(i).expect_local(wl.SZ, 0) for i in range(case["chains"])]))
        b.close()
        return out
    h = g.GseTdvp(s["mps"], s["mpo"], **s["opts"])
    kind = g.REAL if case["kind"] == "real" else g.IMAG
    if f == "tdvp2":
        h.sweep2(0.1, kind)
    else:
        h.krylov_precision(PREC[case["krylov"]])
        h.step(0.1, kind, case["k"])
    out = dict(energy=h.energy(), norm=h.norm(), bonds=np.array(h.bond_dims()),
               sz=np.array([h.expect_local(wl.SZ, i) for i in range(case["sites"])]))
    h.close()
    return out


# ---------------------------------------------------------------- work
def _heff_flops(ml, mr, wl_, wr, nnz, d=2):
    return 8.0 * (ml * d * mr * (ml * wl_ + mr * wr) + ml * mr * nnz)


def work(case):
    f = case["family"]
    if f in ("heff", "site", "expm"):
        W, cl, cr = _mpo_site(case["lattice"])
        ml, mr, a, b = case["ml"], case["mr"], W.shape[0], W.shape[3]
        nnz, env, vec = int(np.count_nonzero(W)), 16.0 * (ml * ml * a + mr * mr * b), 16.0 * 2 * ml * mr
        flops = _heff_flops(ml, mr, a, b, nnz)
        if f == "heff":
            return dict(bytes=env + 2 * vec, flops=flops)
        if f == "site":
            return dict(bytes=2 * env + vec + 16.0 * (mr * mr * a + 2 * ml * mr),
                        flops=2 * flops + 8.0 * a * ml * mr * (ml + mr))
        if case["u1"]:
            ql, qr = _bond_charges(ml, 0).tolist(), _bond_charges(mr, 1).tolist()
            flops = wl.heff_flops_u1(ql, qr, W, cl, cr)
        return dict(bytes=env + 2 * vec, flops=ITERATIONS * flops)
    if f == "batch":
        n, chi, w, chains = (case["shortest"] + case["longest"]) // 2, case["chi"], 5, case["chains"]
    else:
        n, chi, w, chains = case["sites"], case["chi"], LATTICE_W[case["lattice"]], 1
    dims = wl.full_bond_dims(n, chi)
    state = sum(16.0 * dims[i] * 2 * dims[i + 1] for i in range(n))
    # a conserved charge leaves about one entry in four of the local blocks
    share = 0.25 if case.get("u1", f == "batch") else 1.0
    cubes = sum(2.0 * dims[i] * dims[i + 1] * (dims[i] + dims[i + 1]) for i in range(n))
    moves = 8.0 * share * cubes
    if f == "observe":
        return dict(bytes=2 * state, flops=2 * moves)
    site = 8.0 * share * w * cubes
    flops = 2 * ITERATIONS * site * (2 if f == "tdvp2" else 1) + 4 * site + 2 * moves
    if f in ("step", "batch"):
        flops += case["k"] * w * site
    return dict(bytes=chains * 2 * state, flops=chains * flops)


# ---------------------------------------------------------------- exact values (64 bits, torch)
def _heff(L, W, R, x):
    ml, a, _ = L.shape
    mr, b, _ = R.shape
    d = W.shape[1]
    t = (L.reshape(ml * a, ml) @ x.reshape(ml, d * mr)).reshape(ml, a, d, mr)
    t = torch.einsum("wstv,awtb->asvb", W, t)
    return (t.reshape(ml * d, b * mr) @ R.reshape(mr, b * mr).T).reshape(ml, d, mr)


def _keff(L, R, c):
    ml, a, _ = L.shape
    mr = R.shape[0]
    t = L.reshape(ml * a, ml) @ c
    return t.reshape(ml, a * mr) @ R.reshape(mr, a * mr).T


def _env_left(E, W, A):
    ml, d, mr = A.shape
    a, b = W.shape[0], W.shape[3]
    t = (E.reshape(ml * a, ml) @ A.reshape(ml, d * mr)).reshape(ml, a, d, mr)
    t = torch.einsum("wstv,awtb->asvb", W, t).reshape(ml * d, b * mr)
    return (A.reshape(ml * d, mr).conj().T @ t).reshape(mr, b, mr)


def _env_right(E, W, A):
    ml, d, mr = A.shape
    a, b = W.shape[0], W.shape[3]
    t = (E.reshape(mr * b, mr) @ A.reshape(ml * d, mr).T).reshape(mr, b, ml, d)
    t = torch.einsum("wstv,bvat->sbwa", W, t).reshape(d * mr, a * ml)
    return (A.reshape(ml, d * mr).conj() @ t).reshape(ml, a, ml)


def _expm(op, x, delta, kind):
    """exp(-i delta op) x or exp(-delta op) x: Lanczos, re-orthogonalised twice, past convergence."""
    V, alpha, beta = [x / torch.linalg.norm(x)], [], []
    n = x.numel()
    f = -1j * delta if kind == "real" else -delta
    for j in range(min(n, 40)):
        w = op(V[-1])
        alpha.append(torch.vdot(V[-1].reshape(-1), w.reshape(-1)).real.item())
        M = torch.stack([v.reshape(-1) for v in V])
        for _ in range(2):
            w = w - (M.T @ (M.conj() @ w.reshape(-1))).reshape(w.shape)
        b = torch.linalg.norm(w).item()
        e, u = np.linalg.eigh(np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1))
        y = u @ (np.exp(f * e) * u[0].conj())
        if b * abs(y[-1]) < 1e-15 or b < 1e-13:
            break
        beta.append(b)
        V.append(w / b)
    out = sum(complex(c) * v for c, v in zip(y, V))
    return out * torch.linalg.norm(x)


def _qr(M):
    return torch.linalg.qr(M)


def _sweep(mps, mpo, dt):
    """One symmetric real-time TDVP1 sweep (nothing truncated); the energy of the result."""
    A = [torch.from_numpy(a).cuda() for a in mps]
    W = [torch.from_numpy(w).cuda() for w in mpo]
    n = len(A)
    one = torch.ones(1, 1, 1, dtype=torch.complex128, device="cuda")
    R = [None] * n
    R[-1] = one
    for i in range(n - 1, 0, -1):
        l, d, r = A[i].shape
        q, c = _qr(A[i].reshape(l, d * r).conj().T)
        A[i] = q.conj().T.reshape(-1, d, r)
        A[i - 1] = torch.tensordot(A[i - 1], c.conj().T, 1)
        R[i - 1] = _env_right(R[i], W[i], A[i])
    L = [None] * n
    L[0] = one
    for i in range(n):
        x = _expm(lambda v: _heff(L[i], W[i], R[i], v), A[i], dt / 2, "real")
        if i == n - 1:
            A[i] = x
            break
        l, d, r = x.shape
        q, c = _qr(x.reshape(l * d, r))
        A[i] = q.reshape(l, d, -1)
        L[i + 1] = _env_left(L[i], W[i], A[i])
        c = _expm(lambda v: _keff(L[i + 1], R[i], v), c, -dt / 2, "real")
        A[i + 1] = torch.tensordot(c, A[i + 1], 1)
    for i in range(n - 1, -1, -1):
        x = _expm(lambda v: _heff(L[i], W[i], R[i], v), A[i], dt / 2, "real")
        if i == 0:
            A[0] = x
            break
        l, d, r = x.shape
        q, c = _qr(x.reshape(l, d * r).conj().T)
        A[i] = q.conj().T.reshape(-1, d, r)
        R[i - 1] = _env_right(R[i], W[i], A[i])
        c = _expm(lambda v: _keff(L[i], R[i - 1], v), c.conj().T, -dt / 2, "real")
        A[i - 1] = torch.tensordot(A[i - 1], c, 1)
    x = A[0]
    h = _heff(L[0], W[0], R[0], x)
    return (torch.vdot(x.reshape(-1), h.reshape(-1)).real / torch.linalg.norm(x) ** 2).item()


def exact(case, seed):
    f = case["family"]
    if f == "heff":
        W, L, R, x, _ = _site_operands(case, seed)
        return _heff(L, torch.from_numpy(W).cuda(), R, x)
    if f == "site":
        s = prepare(case, seed)
        W = torch.from_numpy(s["W"]).cuda()
        return dict(left=_env_left(s["L"], W, s["x"]), right=_env_right(s["R"], W, s["x"]),
                    bond=_keff(s["L"], s["Rb"], s["c"]))
    if f == "expm":
        W, L, R, x = _expm_operands(case, seed)
        Wd = torch.from_numpy(W).cuda()
        return dict(y=_expm(lambda v: _heff(L, Wd, R, v), x, 0.05, case["kind"]), iterations=None)
    if f == "observe":
        mps = _state(case["sites"], case["chi"], seed, case["u1"])
        A = [torch.from_numpy(a).cuda() for a in mps]
        sz = torch.from_numpy(wl.SZ).cuda()
        left = [torch.ones(1, 1, dtype=torch.complex128, device="cuda")]
        for a in A:
            left.append(torch.einsum("asb,asd->bd", a.conj(), torch.tensordot(left[-1], a, 1)))
        right = torch.ones(1, 1, dtype=torch.complex128, device="cuda")
        out = np.zeros(len(A), dtype=np.complex128)
        for i in range(len(A) - 1, -1, -1):
            t = torch.tensordot(torch.tensordot(left[i], A[i], 1), right, 1)
            num = torch.einsum("asb,st,atb->", A[i].conj(), sz, t)
            out[i] = (num / left[-1][0, 0]).item()
            right = torch.einsum("asb,csb->ac", torch.tensordot(A[i], right, 1), A[i].conj())
        return out
    if f == "sweep":
        mps = _state(case["sites"], case["chi"], seed, case["u1"])
        lat = _lattice(case["lattice"], case["sites"])
        return dict(energy=_sweep(mps, wl.heisenberg_mpo(lat), 0.1), mps=[None] * case["sites"])
    return None
