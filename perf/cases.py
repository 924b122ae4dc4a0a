"""Performance cases of the framework: what its users have it do, at the sizes they run.

One pass of a molecular-dynamics case is one call cycle of a production run, as the README
shows it: advance by a block of steps, read the observable record, read the state reached (a
trajectory frame).  Mixed-precision runs hand their results on in 32 bits, the width the
library holds them in; FP64 runs in 64.  Systems are the seeded rock-salt crystals of
``workloads.py``, shifted by a quarter of the lattice constant so that no lattice site lies on
a cell face (a wrapped coordinate there would flip between the two faces).
"""
import math

import numpy as np
import torch

from paper_1905_02521_gb300 import qtb, workloads as W

HBAR = 0.6582119569             # eV fs
COULOMB = 14.3996454784         # eV A
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# --- the cases ------------------------------------------------------------------

def _md(crystal, ncell, **kw):
    lih = crystal == "lih"
    case = dict(kind="md", crystal=crystal, ncell=ncell, removed=0, beads=1, T=50.0 if lih else 100.0,
                dt=0.25 if lih else 1.0, noise="qtb", taps=2049, omega_max=0.6 if lih else 0.3, precision="mixed",
                filter="bf16", segment_blocks=0, npt=False, steps=256)
    case.update(kw)
    return case


def listed():
    return [
        # the small FP64 reference run (64-ion MgO, 513 taps): parity checks, equilibration tests
        dict(_md("mgo", 2, T=300.0, taps=513, precision="fp64"), name="mgo64_qtb_fp64"),
        # FP64 production at medium size: the form results are checked against
        dict(_md("mgo", 6, precision="fp64"), name="mgo1728_qtb_fp64"),
        # the smallest crystal of the heat-capacity sweep, run alone: latency of a step
        dict(_md("mgo", 3), name="mgo216_qtb"),
        # the flagship workload: 8000-ion MgO, QTB-MD, tensor-core noise filter
        dict(_md("mgo", 10), name="mgo8000_qtb"),
        # QTB-PIMD of LiH, 8 beads (kappa_P spectrum)
        dict(_md("lih", 6, beads=8, noise="qtb_pimd"), name="lih1728_qtbpimd_p8"),
        # standard PIMD of LiH, 32 beads, white bath
        dict(_md("lih", 6, beads=32, noise="white"), name="lih1728_pimd_p32"),
        # the largest: 64000 ions x 32 beads (2.05 M bead-atoms)
        dict(_md("lih", 20, beads=32, noise="white"), name="lih64000_pimd_p32"),
        # LiH at zero pressure, isotropic Langevin cell: every step needs the virial
        dict(_md("lih", 6, npt=True), name="lih1728_qtb_npt"),
        # heat-capacity sweep: 64 MgO systems of 216-4096 ions, 10-1500 K, one context
        dict(kind="sweep", systems=64, filter="bf16", steps=256, name="sweep64_qtb"),
        # zero-point-leakage study: 32769 double wells, QTB-PIMD, default FP32 filter, a record every 8 steps
        dict(kind="wells", atoms=10923, beads=8, noise="qtb_pimd", taps=2049, precision="mixed", filter="fp32",
             steps=256, stride=8, name="wells32769_qtbpimd_p8"),
        # forces and energies of configurations made elsewhere (minimisers, force matching, lattice dynamics)
        dict(kind="forces", crystal="mgo", ncell=8, removed=0, beads=1, precision="mixed", name="mgo4096_forces"),
        # set-up of a kappa_P study: the Eq. 10 solves of four bead counts and the training of their learned model
        dict(kind="training", beads="2,4,8,32", samples=3200, iters=200, name="kappa_model_training"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "pimd", "pimd", "fp64", "npt", "sweep", "wells", "forces", "forces", "kappa"])
    crystal = rng.choice(["mgo", "lih"])
    T = round(math.exp(rng.uniform(math.log(20.0), math.log(400.0))), 2)
    removed = 2 * rng.randint(0, 7)
    taps = 2 * _spread(rng, 100, 1100) + 1
    if kind == "md":
        return _md(crystal, _spread(rng, 2, 20), removed=removed, T=T, taps=taps, filter=rng.choice(["bf16", "bf16", "fp32"]),
                   segment_blocks=rng.choice([0, 0, 0, 1]), steps=rng.choice([256, 256, 100, 300]))
    if kind == "pimd":
        P = rng.choice([2, 3, 4, 5, 6, 8, 16, 32])
        return _md(crystal, _spread(rng, 2, int((250000 / (8 * P)) ** (1 / 3))), removed=removed, beads=P, T=T, taps=taps,
                   noise=rng.choice(["white", "qtb_pimd"]), steps=rng.choice([256, 256, 100]))
    if kind == "fp64":
        return _md(crystal, _spread(rng, 2, 7), removed=removed, T=T, taps=taps, precision="fp64",
                   steps=rng.choice([256, 100]))
    if kind == "npt":
        P = rng.choice([1, 1, 4, 8])
        return _md(crystal, _spread(rng, 3, 8), removed=removed, beads=P, T=T, taps=taps, npt=True,
                   noise="qtb" if P == 1 else "qtb_pimd")
    if kind == "sweep":
        return dict(kind="sweep", systems=rng.randint(3, 60), filter="bf16", steps=256)
    if kind == "wells":
        P = rng.choice([1, 2, 4, 8, 16, 32])
        return dict(kind="wells", atoms=_spread(rng, 1, 160000 // P), beads=P, noise="qtb" if P == 1 else
                    rng.choice(["white", "qtb_pimd"]), taps=taps, precision=rng.choice(["mixed", "mixed", "fp64"]) if
                    P <= 8 else "mixed", filter="fp32", steps=rng.choice([256, 300]), stride=rng.choice([1, 8, 64]))
    if kind == "forces":
        P = rng.choice([1, 1, 4])
        return dict(kind="forces", crystal=crystal, ncell=_spread(rng, 2, 16 if P == 1 else 8), removed=removed, beads=P,
                    precision=rng.choice(["mixed", "mixed", "fp64"]))
    return dict(kind="kappa", beads=rng.randint(2, 32), nodes=_spread(rng, 128, 1024))


# --- inputs ----------------------------------------------------------------------

def _crystal(case, seed):
    """One system dict and its potential: a perturbed rock-salt crystal, `removed` ions (half of
    each kind) taken out."""
    make, a = (W.mgo_system, 4.21) if case["crystal"] == "mgo" else (W.lih_system, 4.08)
    s, pot = make(case["ncell"], case.get("T", 300.0), gamma=1e-3, n_beads=case["beads"], seed=seed, vel_seed=seed + 1)
    s["pos"] = np.mod(s["pos"] + a / 4, s["box"])
    if case["removed"]:
        rng = np.random.default_rng(seed + 2)
        keep = np.ones(len(s["types"]), bool)
        for t in (0, 1):
            keep[rng.choice(np.flatnonzero(s["types"] == t), case["removed"] // 2, replace=False)] = False
        s["pos"], s["vel"], s["types"] = s["pos"][:, keep].copy(), s["vel"][:, keep].copy(), s["types"][keep].copy()
    return s, pot


def _params(pot, case, seed, dt, **kw):
    p = {k: pot[k] for k in ("mass", "charge", "buck_A", "buck_rho", "buck_C")}
    p.update(dsf_alpha=pot["dsf_alpha"], r_cut=pot["r_cut"], dt=dt, seed=seed,
             precision=qtb.FP64 if case.get("precision") == "fp64" else qtb.MIXED,
             filter_prec=qtb.FILTER_BF16 if case.get("filter") == "bf16" else qtb.FILTER_FP32)
    p.update(kw)
    return p


def _npt(s):
    """Cell of a ~300 fs volume period at a bulk modulus of ~1 eV/A^3, zero pressure."""
    return dict(npt=1, pressure=0.0, cell_mass=9.0 * float(np.prod(s["box"])) / (2 * np.pi / 300.0) ** 2, cell_gamma=4e-3)


MODES = {"white": qtb.NOISE_WHITE, "qtb": qtb.NOISE_QTB, "qtb_pimd": qtb.NOISE_QTB_PIMD}


class _Run:
    """What a program keeps of one run: the context (freed with it) and pinned buffers for the frames."""

    def __init__(self, case, ctx, systems):
        self.case, self.ctx, self.systems = case, ctx, systems
        shapes = [x["pos"].shape for x in systems]
        pin = (lambda sh: torch.empty(sh, dtype=torch.float64, pin_memory=True)) if DEV == "cuda" else torch.empty
        self.pos, self.vel = [pin(sh) for sh in shapes], [pin(sh) for sh in shapes]

    def __del__(self):
        qtb.qtb_destroy(self.ctx)


class _Model:
    """A learned-kappa_P model and the weights its training starts from."""

    def __init__(self, case, seed):
        self.case, self.weights, self.handle = case, _weights(seed), qtb.qtb_kappa_model_create(1 + seed)

    def __del__(self):
        qtb.qtb_kappa_model_destroy(self.handle)


def _weights(seed):
    rng = np.random.default_rng(seed)
    parts = [rng.uniform(-1, 1, n) * a for n, a in ((128, 3 ** .5), (64, 0.0), (4096, (6 / 64) ** .5), (64, 0.0), (64, (6 / 64) ** .5))]
    return np.concatenate(parts + [[0.7]]).astype(np.float32)


def _sweep(case, seed):
    systems, pot = W.sweep_systems(case["systems"], gamma=1e-3)
    for k, s in enumerate(systems):
        rng = np.random.default_rng(seed + k)
        s["pos"] = np.mod(s["pos"] + 4.21 / 4 + rng.normal(0.0, 0.005, s["pos"].shape), s["box"])
    return systems, pot


def _y0(seed):
    """Where the collocation grid turns from linear to logarithmic."""
    return 1.0 + (seed % 997) / 4000.0


def prepare(case, seed):
    kind = case["kind"]
    if kind == "kappa":
        return dict(P=case["beads"], n=case["nodes"], y_max=1000.0, y0=_y0(seed))
    if kind == "training":
        return _Model(case, seed)
    with torch.cuda.stream(torch.cuda.Stream()):  # a run is issued on a stream of its own (its block graphs are captured there)
        if kind == "sweep":
            systems, pot = _sweep(case, seed)
            ctx = qtb.qtb_init(systems, _params(pot, case, seed, 1.0, obs_stride=case["steps"], max_records=64))
            qtb.qtb_set_filter(ctx, -1, qtb.NOISE_QTB, 2049, 0.3)
        elif kind == "wells":
            s, pot = W.oscillators(case["atoms"], 100.0, 0.004, n_beads=case["beads"], x0=0.5, spread=0.05, seed=seed,
                                   vel_seed=seed + 1)
            systems = [s]
            ctx = qtb.qtb_init(systems, _params(pot, case, seed, 0.5, potential=qtb.POT_DOUBLEWELL, ext_V0=0.1, ext_a=0.5,
                                                obs_stride=case["stride"], max_records=case["steps"]))
            if case["noise"] != "white":
                qtb.qtb_set_filter(ctx, 0, MODES[case["noise"]], case["taps"], 0.6)
        elif kind == "forces":
            s, pot = _crystal(case, seed)
            other, _ = _crystal(case, seed + 5)  # the context exists; the configurations come later
            systems = [s]
            ctx = qtb.qtb_init([other], _params(pot, case, seed, 1.0))
        else:
            s, pot = _crystal(case, seed)
            systems = [s]
            kw = _npt(s) if case["npt"] else {}
            ctx = qtb.qtb_init(systems, _params(pot, case, seed, case["dt"], obs_stride=case["steps"], max_records=64, **kw))
            if case["noise"] != "white":
                qtb.qtb_set_filter(ctx, 0, MODES[case["noise"]], case["taps"], case["omega_max"])
            if case["segment_blocks"]:
                qtb.qtb_set_generator(ctx, qtb.GEN_FOURIER, case["segment_blocks"])
        return _Run(case, ctx, systems)


def run(state):
    if isinstance(state, dict):
        return qtb.qtb_kappa_solve(**state)
    case = state.case
    kind = case["kind"]
    if kind == "training":
        qtb.qtb_kappa_model_set_weights(state.handle, state.weights)
        qtb.qtb_kappa_model_train(state.handle, [int(p) for p in case["beads"].split(",")], case["samples"], case["iters"])
        return qtb.qtb_kappa_model_get_weights(state.handle)
    ctx = state.ctx
    # the mixed form holds its results in 32 bits
    out = (lambda a: a) if case.get("precision") == "fp64" else (lambda a: torch.as_tensor(a).to(torch.float32))
    if kind == "forces":
        s = state.systems[0]
        qtb.qtb_set_state(ctx, 0, s["pos"], s["vel"])
        f = qtb.qtb_get_forces(ctx, 0, *s["pos"].shape[:2])
        return {"forces": out(f), "record": out(qtb.qtb_observables(ctx, 0))}
    qtb.qtb_step_n(ctx, case["steps"])
    if kind == "wells":
        rec = [qtb.qtb_get_series(ctx, 0, case["steps"] // case["stride"])]
    else:
        rec = [qtb.qtb_observables(ctx, k) for k in range(len(state.systems))]
    for k in range(len(state.systems)):
        qtb.qtb_get_state_into(ctx, k, state.pos[k].numpy(), state.vel[k].numpy())
    if kind == "sweep":  # one tensor each for the whole batch
        return {"record": out(np.stack(rec)), "pos": out(torch.cat([x.reshape(-1) for x in state.pos])),
                "vel": out(torch.cat([x.reshape(-1) for x in state.vel]))}
    res = {"record": out(rec[0]), "pos": out(state.pos[0]), "vel": out(state.vel[0])}
    if case.get("npt"):
        box, p_e = qtb.qtb_get_cell(ctx, 0)
        res["cell"] = out(np.append(box, p_e))
    return res


def work(case):
    kind = case["kind"]
    if kind == "kappa":  # 2P entries in each of 2n - 1 rows; normal equations, factorisation, solves
        n, P = case["nodes"], case["beads"]
        return {"bytes": 8.0 * n, "flops": 4.0 * P * P * 2 * (2 * n - 1) + n ** 3 / 3.0 + 8.0 * n * n}
    if kind == "training":
        Ps = [int(p) for p in case["beads"].split(",")]
        n, fwd = len(Ps) * case["samples"], 2.0 * (64 * 2 + 64 * 64 + 64)
        solve = sum(work(dict(kind="kappa", nodes=1024, beads=p))["flops"] for p in Ps)
        return {"bytes": 2 * 4.0 * 4417, "flops": 3.0 * fwd * n * case["iters"] + solve}
    size = 8 if case.get("precision") == "fp64" else 4
    if kind == "sweep":
        parts = [(8 * (3 + k % 6) ** 3, 1, 0.1072) for k in range(case["systems"])]
        taps, steps = 2049, case["steps"]
    elif kind == "wells":
        parts, taps, steps = [(case["atoms"], case["beads"], 0.0)], case["taps"], case["steps"]
    else:
        a = 4.21 if case["crystal"] == "mgo" else 4.08
        parts = [(8 * case["ncell"] ** 3 - case["removed"], case["beads"], 8 / a ** 3)]
        taps, steps = case.get("taps", 1), case.get("steps", 1)
    nbytes = flops = 0.0
    for n, P, rho in parts:
        # 64 flops per ordered pair within 8 A, the coloured noise (fast convolution), two fast mode
        # transforms each way, the step itself
        pairs = 64.0 * rho * 4 / 3 * math.pi * 512
        noise = 0.0 if case.get("noise") == "white" or kind == "forces" else 3 * min(2.0 * taps, 4 * 2.5 * math.log2(512 + taps))
        modes = 3 * 4 * 2.5 * math.log2(P)
        flops += steps * n * P * (pairs + noise + modes + 60)
        nbytes += n * P * 3 * size * (2.0 if kind == "forces" else 4.0)
    return {"bytes": nbytes + 23 * 8, "flops": flops}


# --- the same results in 64 bits, plain torch ----------------------------------------

def _mulhilo(m, x):
    lo, hi = m * (x & 0xFFFF), m * (x >> 16)
    hi = hi + (lo >> 16)
    return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)


def _normals(seed, dofs, n0, n, stream=0):
    """White noise [dofs, n] of steps n0 .. n0 + n - 1: Philox4x32-10, Box-Muller pairs."""
    q0, q1 = n0 // 4, -((-(n0 + n)) // 4)
    q = torch.arange(q0, q1, dtype=torch.int64, device=DEV)[None, :]
    d = torch.as_tensor(dofs, dtype=torch.int64, device=DEV)[:, None]
    q, d = torch.broadcast_tensors(q, d)
    c = [q & 0xFFFFFFFF, d, torch.full_like(q, stream), (q >> 32) & 0xFFFFFFFF]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    z = []
    for a, b in ((c[0], c[1]), (c[2], c[3])):
        r = torch.sqrt(-2.0 * torch.log((a.double() + 1.0) * 2.0 ** -32))
        ph = 2.0 * math.pi * b.double() * 2.0 ** -32
        z += [r * torch.cos(ph), r * torch.sin(ph)]
    z = torch.stack(z, -1).reshape(d.shape[0], -1)
    return z[:, n0 - 4 * q0:n0 - 4 * q0 + n]


def _fth(x):
    x = np.abs(np.asarray(x, np.float64))
    s = np.where(x < 1e-6, 1.0, x)
    return np.where(x < 1e-6, 1.0 + x * x / 12.0, s * (0.5 + 1.0 / np.expm1(np.minimum(s, 700.0))))


def _tail(P, y):
    return _fth(math.sqrt(P) * y) / P + math.sqrt(P) / (2.0 * y)


def _kappa(P, n, y_max=1000.0, y0=1.0):
    """F_P of Eq. 10 at the nodes y0 sinh(i t): least squares over nodes and midpoints."""
    t = math.asinh(y_max / y0) / (n - 1)
    nodes = y0 * np.sinh(np.arange(n) * t)
    y = y0 * np.sinh(0.5 * t * np.arange(2 * n - 1))
    A, rhs = np.zeros((2 * n - 1, n)), _fth(math.sqrt(P) * y)
    for k in range(P):
        yk2 = y * y + 4.0 * P * math.sin(math.pi * k / P) ** 2
        w = np.ones_like(y) if k == 0 else y * y / yk2
        yk = np.sqrt(yk2)
        inn = np.flatnonzero((yk <= y_max) & (w > 0))
        out = np.flatnonzero((yk > y_max) & (w > 0))
        i = np.minimum((np.arcsinh(yk[inn] / y0) / t).astype(int), n - 2)
        lam = (yk[inn] - nodes[i]) / (nodes[i + 1] - nodes[i])
        np.add.at(A, (inn, i), w[inn] * (1.0 - lam))
        np.add.at(A, (inn, i + 1), w[inn] * lam)
        rhs[out] -= w[out] * _tail(P, yk[out])
    sc = 1.0 / _fth(math.sqrt(P) * y)
    return np.linalg.lstsq(A * sc[:, None], rhs * sc, rcond=None)[0], nodes


def _kappa_at(P, F, nodes, y):
    out = np.interp(y, nodes, F)
    far = y > nodes[-1]
    return np.where(far, _tail(P, np.where(far, y, 1.0)), out)


def _coloured(s, case, seed, dt, n_taps, omega_max, n0, n, sysid=0):
    """eta [steps, dofs] of steps n0 .. n0 + n - 1."""
    P, N = s["pos"].shape[:2]
    kT = W.KB * s["T"]
    D = 3 * N * P
    key = (seed & 0xFFFFFFFF) | (((seed >> 32) ^ sysid) << 32)
    K = 0 if case["noise"] == "white" else (n_taps - 1) // 2
    if K or case["noise"] != "white":
        L = 2 * K + 1
        w = 2.0 * math.pi * np.arange(K + 1) / (L * dt)
        if case["noise"] == "qtb":
            S = kT * _fth(HBAR * w / kT)
        else:
            S = kT * _kappa_at(P, *_kappa(P, 1024), HBAR * w / kT)
        S = np.sqrt(S / (1.0 + np.exp(np.minimum((w - omega_max) / (omega_max / 50.0), 700.0))))
        k = np.arange(K + 1)
        h = np.array([(S[0] + 2.0 * np.sum(S[1:] * np.cos(2.0 * math.pi * ((k[1:] * kk) % L) / L))) / L for kk in k])
    else:
        h = np.array([math.sqrt(kT)])
    full = torch.as_tensor(np.concatenate([h[:0:-1], h]), device=DEV)
    M = n + 2 * K
    F = 1 << (M + len(full)).bit_length()
    Hf = torch.fft.rfft(full, F)
    eta = torch.empty(n, D, dtype=torch.float64, device=DEV)
    for d0 in range(0, D, 32768):
        x = _normals(key, range(d0, min(D, d0 + 32768)), n0 - K, M)
        eta[:, d0:d0 + 32768] = torch.fft.irfft(torch.fft.rfft(x, F) * Hf, F)[:, 2 * K:2 * K + n].T
    return eta


class _Pairs:
    """Forces, energy and virial of periodic replicas from a list of ordered pairs."""

    def __init__(self, s, pot, margin=2.0):
        self.rc, self.al, self.margin = pot["r_cut"], pot["dsf_alpha"], margin
        self.box = torch.as_tensor(s["box"], device=DEV)
        self.t = torch.as_tensor(s["types"].astype(np.int64), device=DEV)
        self.nt = len(pot["mass"])
        flat = lambda k: torch.as_tensor(np.asarray(pot[k], np.float64).reshape(-1), device=DEV)  # noqa: E731
        self.A, self.rho, self.C, self.q = flat("buck_A"), flat("buck_rho"), flat("buck_C"), flat("charge")
        self.ref = None

    def build(self, x):  # x [P, N, 3], beads within a bond of bead 0
        R, L, x0 = self.rc + self.margin, self.box, x[0]
        m = [int(math.ceil(R / float(b) - 0.5)) if float(b) < 2 * R else 0 for b in L]
        sh = torch.cartesian_prod(*[torch.arange(-k, k + 1, device=DEV, dtype=torch.float64) for k in m]).reshape(-1, 3) * L
        ii, jj, ss = [], [], []
        step = max(1, 40_000_000 // (x0.shape[0] * sh.shape[0]))
        for i0 in range(0, x0.shape[0], step):
            d = x0[None, :, :] - x0[i0:i0 + step, None, :]
            base = -L * torch.round(d / L)
            e = d + base
            r2 = ((e[:, :, None, :] + sh) ** 2).sum(-1)
            a, b, k = torch.nonzero((r2 < R * R) & (r2 > 1e-12), as_tuple=True)
            ii.append(a + i0), jj.append(b), ss.append(base[a, b] + sh[k])
        self.i, self.j, self.s = torch.cat(ii), torch.cat(jj), torch.cat(ss)
        p = self.t[self.i] * self.nt + self.t[self.j]
        self.pA, self.pr, self.pC, self.pq = self.A[p], 1.0 / self.rho[p], self.C[p], COULOMB * self.q[self.t[self.i]] * self.q[self.t[self.j]]
        self.ref = x.clone()
        rc, al = self.rc, self.al
        self.es = self.pA * torch.exp(-rc * self.pr) - self.pC / rc ** 6
        self.e0 = math.erfc(al * rc) / rc
        self.fs = self.e0 / rc + 2 * al / math.sqrt(math.pi) * math.exp(-(al * rc) ** 2) / rc

    def __call__(self, x, lam=1.0):
        if self.ref is None or float((x - self.ref).abs().max()) > 0.2 * self.margin:
            self.build(x)
        f, E, Wv = torch.zeros_like(x), 0.0, torch.zeros(3, 3, dtype=torch.float64, device=DEV)
        for b in range(x.shape[0]):
            d = (x[b][self.j] - x[b][self.i] + self.s) * lam
            r2 = (d * d).sum(1)
            inn = r2 < self.rc ** 2
            r2 = torch.where(inn, r2, torch.ones_like(r2))
            r = torch.sqrt(r2)
            ex, er = self.pA * torch.exp(-r * self.pr), torch.erfc(self.al * r) / r
            gg = 2 * self.al / math.sqrt(math.pi) * torch.exp(-self.al ** 2 * r2)
            fr = (ex * self.pr - 6 * self.pC / r2 ** 3 / r + self.pq * ((er + gg) / r - self.fs)) / r * inn
            en = (ex - self.pC / r2 ** 3 - self.es + self.pq * (er - self.e0 + self.fs * (r - self.rc))) * inn
            fd = fr[:, None] * d
            f[b].index_add_(0, self.i, -fd)
            E = E + 0.5 * en.sum()
            Wv = Wv + 0.5 * fd.T @ d
        P = x.shape[0]
        return f / P, float(E) / P, Wv.cpu().numpy() / P


class _Wells:
    def __init__(self, V0=0.1, a=0.5):
        self.V0, self.a2 = V0, a * a

    def __call__(self, x, lam=1.0):
        P, u = x.shape[0], x * x / self.a2 - 1.0
        f = -4.0 * self.V0 * u * x / self.a2
        vir = np.diag((x * f).sum((0, 1)).cpu().numpy()) / P
        return f / P, float((self.V0 * u * u).sum()) / P, vir


def _record(step, s, x, v, f, V, vir, m, lam, wells):
    P, N = x.shape[:2]
    kT = W.KB * s["T"]
    mv = (m * W.MVV2E)[None, :, None]
    L = torch.as_tensor(s["box"], device=DEV)
    d = x - x[:1]
    if not wells:
        d = d - L * torch.round(d / L)
    d = d * lam
    K = float(0.5 * (mv * v * v).sum())
    spr = float(0.5 * P * (kT / HBAR) ** 2 * (mv * (d - torch.roll(d, -1, 0)) ** 2).sum()) if P > 1 else 0.0
    vb = v.mean(0, keepdim=True)
    K0 = float(0.5 * P * (mv * vb * vb).sum())
    cv = float(((d - d.mean(0, keepdim=True)) * f).sum())
    mom = (m[None, :, None] * v).sum((0, 1)).cpu().numpy()
    x2 = float((x * x).sum()) / P if wells else 0.0
    vol = float(np.prod(s["box"])) * lam ** 3
    return np.concatenate([[step, K, V, spr, K - spr + V], vir.reshape(-1), mom,
                           [x2, 1.5 * N * kT - 0.5 * cv, K0 - 0.5 * cv, vol, K0, np.trace(vir) - cv]])


def _trajectory(s, pot, case, seed, dt, steps, stride, n_taps, omega_max, force, npt=None):
    """BAOAB in normal modes (one bead also in a Langevin cell): records every `stride` steps, final state."""
    wells = isinstance(force, _Wells)
    x, v = (torch.as_tensor(s[k], dtype=torch.float64, device=DEV).clone() for k in ("pos", "vel"))
    P, N = x.shape[:2]
    m = torch.as_tensor(pot["mass"][s["types"]], device=DEV)
    h = 0.5 * dt
    hm = (h / (m * W.MVV2E))[None, :, None]
    kT, c1 = W.KB * s["T"], math.exp(-s["gamma"] * dt)
    sig = torch.sqrt((1 - c1 * c1) / (m * W.MVV2E))[None, :, None]
    C = np.zeros((P, P))
    for b in range(P):
        for k in range(P):
            ang = 2 * math.pi * ((b * k) % P) / P
            C[b, k] = (1 / math.sqrt(P) if k == 0 else math.sqrt(2 / P) * math.cos(ang) if 2 * k < P else
                       (-1) ** b / math.sqrt(P) if 2 * k == P else math.sqrt(2 / P) * math.sin(ang))
    C = torch.as_tensor(C, device=DEV)
    w = 2 * math.sqrt(P) * kT / HBAR * np.sin(math.pi * np.arange(P) / P)
    col = lambda a: torch.as_tensor(a, device=DEV)[:, None, None]  # noqa: E731
    cs, ws = col(np.cos(h * w)), col(-w * np.sin(h * w))
    sw = col(np.array([h if k == 0 else math.sin(h * w[k]) / w[k] for k in range(P)]))
    eta = _coloured(s, case, seed, dt, n_taps, omega_max, 0, steps)
    to_modes = lambda a: torch.tensordot(C.T, a, 1)  # noqa: E731
    L = torch.as_tensor(s["box"], device=DEV)
    lam, pe, pending = 1.0, 0.0, False
    f, V, vir = force(x, lam)
    recs = []
    K = float(0.5 * ((m * W.MVV2E)[None, :, None] * v * v).sum())
    if npt:
        al, Wc = 1 + 1 / N, npt["cell_mass"]
        ce = math.exp(-npt["cell_gamma"] * dt)
        xi = _normals(seed, [0], 0, steps, stream=1)[0].cpu().numpy()
    for n in range(steps):
        noise = eta[n].reshape(P, 3, N).transpose(1, 2) * sig
        if npt:  # displacements of the reference cell; one bead
            G = 2 * al * K + np.trace(vir) - 3 * float(np.prod(s["box"])) * lam ** 3 * npt["pressure"]
            pe += h * G * (2 if pending else 1)
            pending = True
            y = pe / Wc * h
            v = v * math.exp(-al * y) + hm * f * (-math.expm1(-al * y) / (al * y) if y else 1.0)
            lam *= math.exp(y)
            x = x + v * (h * (math.expm1(y) / y if y else 1.0) / lam)
            pe = ce * pe + math.sqrt((1 - ce * ce) * Wc * kT) * xi[n]
            v = c1 * v + noise
            y = pe / Wc * h
            lam *= math.exp(y)
            x = x + v * (h * (math.expm1(y) / y if y else 1.0) / lam)
            f, V, vir = force(x, lam)
            v = v * math.exp(-al * y) + hm * f * (-math.expm1(-al * y) / (al * y) if y else 1.0)
            K = float(0.5 * ((m * W.MVV2E)[None, :, None] * v * v).sum())
        else:
            d = x - x[:1]
            if not wells:
                d = d - L * torch.round(d / L)
            q, p = to_modes(d), to_modes(v + hm * f)
            q, p = q * cs + p * sw, q * ws + p * cs
            p = c1 * p + noise
            q, p = q * cs + p * sw, q * ws + p * cs
            x = x + torch.tensordot(C, q, 1) - d
            v = torch.tensordot(C, p, 1)
            f, V, vir = force(x)
            v = v + hm * f
        if (n + 1) % stride == 0:
            recs.append(_record(n + 1, s, x, v, f, V, vir, m, lam, wells))
    if not wells:
        x = x - L * torch.floor(x / L)
    cell = np.append(s["box"] * lam, pe)
    return np.array(recs), (x * lam).cpu().numpy(), v.cpu().numpy(), cell


def _training(case, w0):
    dt = dict(dtype=torch.float64, device=DEV)
    xs, ts = [], []
    n = case["samples"]
    y = np.sinh(math.asinh(1000.0) * (np.arange(n) + 0.5) / n)
    for P in [int(p) for p in case["beads"].split(",")]:
        ratio = _kappa_at(P, *_kappa(P, 1024), y) / _fth(y)
        xs.append(np.stack([np.arcsinh(y) / math.asinh(1000.0), np.full(n, math.log(P / 2) / math.log(16))], 1))
        ts.append(ratio)
    x, t = torch.as_tensor(np.concatenate(xs), **dt), torch.as_tensor(np.concatenate(ts), **dt)
    w = torch.as_tensor(w0.astype(np.float64), **dt).requires_grad_()
    m, v, it = torch.zeros_like(w), torch.zeros_like(w), case["iters"]
    silu = torch.nn.functional.silu
    for k in range(it):
        a = silu(x @ w[:128].reshape(64, 2).T + w[128:192])
        a = silu(a @ w[192:4288].reshape(64, 64).T + w[4288:4352])
        loss = ((a @ w[4352:4416] + w[4416] - t) ** 2).mean()
        (g,) = torch.autograd.grad(loss, w)
        with torch.no_grad():
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            lr = 3e-3 * 3e-3 ** (k / it)
            w -= lr * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)
    return w.detach().cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "kappa":
        return _kappa(case["beads"], case["nodes"], 1000.0, _y0(seed))[0]
    if kind == "training":
        return _training(case, _weights(seed))
    if kind == "sweep":
        return None  # too many trajectories
    if kind == "forces":
        s, pot = _crystal(case, seed)
        x, v = (torch.as_tensor(s[k], dtype=torch.float64, device=DEV) for k in ("pos", "vel"))
        f, V, vir = _Pairs(s, pot, margin=0.1)(x)
        m = torch.as_tensor(pot["mass"][s["types"]], device=DEV)
        return {"forces": f.cpu().numpy(), "record": _record(0, s, x, v, f, V, vir, m, 1.0, False)}
    if kind == "wells":
        s, pot = W.oscillators(case["atoms"], 100.0, 0.004, n_beads=case["beads"], x0=0.5, spread=0.05, seed=seed,
                               vel_seed=seed + 1)
        rec, x, v, _ = _trajectory(s, pot, case, seed, 0.5, case["steps"], case["stride"], case["taps"], 0.6, _Wells())
        return {"record": rec, "pos": x, "vel": v}
    # the noise of Fourier segments, a cell on ring polymers, and sizes that take too long: no value
    if case["segment_blocks"] or (case["npt"] and case["beads"] > 1) or 8 * case["ncell"] ** 3 * case["beads"] > 60000:
        return None
    s, pot = _crystal(case, seed)
    npt = _npt(s) if case["npt"] else None
    rec, x, v, cell = _trajectory(s, pot, case, seed, case["dt"], case["steps"], case["steps"], case["taps"],
                                  case["omega_max"], _Pairs(s, pot), npt)
    res = {"record": rec[-1], "pos": x, "vel": v}
    if npt:
        res["cell"] = cell
    return res
