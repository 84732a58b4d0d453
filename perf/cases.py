"""Performance cases of the library: what a program that uses it has it do, over the real range.

Every case goes through the public entry points of `paper_1904_08756_gb300.epsr`. Sizes come from
the test systems of `synth` (the 900-atom and the paper-scale water box, the paper-scale silica
box, the 64 uneven replicas, the flexible water, the 1.5e6-atom row of the atom-count sweep) and
the ranges between them.

  listed()            the cases
  draw(rng)           one more case of the same ranges (rng: random.Random)
  prepare(case, seed) inputs, handles and plans that a program holds before the call
  run(state)          one pass
  work(case)          bytes and operations that the pass cannot do without
  exact(case, seed)   the pass in 64 bits, in plain torch and numpy (None where there is no such value)

Boxes are liquid-like and made from the seed: one molecule or atom per site of a cubic lattice,
displaced at random up to the least separation the random sequential placement of `synth` keeps
(O-O 2.3 A, silica 1.5 A), water in random orientations redrawn until no two atoms of different
molecules are closer than 1 A.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1904_08756_gb300 import epsr, synth

DEV = "cuda"
SQ_MODES = {"fp32": epsr.SQ_FP32, "tf32x3": epsr.SQ_TF32X3, "bf16x3": epsr.SQ_BF16X3, "bf16x6": epsr.SQ_BF16X6}


# ---- cases -----------------------------------------------------------------------------------------

def listed():
    return [
        # the whole step (moves, g(r), S(Q)) on the smallest shipped box: launches and latency
        dict(name="step_water_900", kind="step", system="water", atoms=900, moves=1000, r_lj=0.0, ep=False),
        # the step of a production run: the paper's 99,999-atom water box
        dict(name="step_water_99999", kind="step", system="water", atoms=99999, moves=10000, r_lj=0.0, ep=False),
        # atom moves of the paper's silica box under an empirical potential, as after the first refinement pass
        dict(name="sweep_silica_ep_99000", kind="sweep", system="silica", atoms=99000, moves=5000, r_lj=0.0, ep=True,
             log=False),
        # the cutoff form of the energy change: Lennard-Jones truncated at the Coulomb cutoff
        dict(name="sweep_water_cutoff_99999", kind="sweep", system="water", atoms=99999, moves=5000, r_lj=9.0,
             ep=False, log=False),
        # flexible molecules under an empirical potential, every move logged (a run that is replayed later)
        dict(name="sweep_flexible_ep_12000", kind="sweep", system="flexible", atoms=12000, moves=4000, r_lj=0.0,
             ep=True, log=True),
        # a large box, whose partners do not fit in shared memory
        dict(name="sweep_water_1500000", kind="sweep", system="water", atoms=1500000, moves=400, r_lj=0.0, ep=False,
             log=False),
        # g(r) of a stored configuration
        dict(name="gr_silica_99000", kind="gr", system="silica", atoms=99000, cells=False),
        # g(r) of a large box through the cell-list entry point
        dict(name="gr_cells_water_300000", kind="gr", system="water", atoms=300000, cells=True),
        # the differentiable form: chi^2 of the smeared g(r) and its gradient for every coordinate
        dict(name="smeared_water_99999", kind="smeared", system="water", atoms=99999, sigma=0.05),
        # S(Q) of 64 replicas' partial g(r) in one contraction
        dict(name="sq_bf16x3_192", kind="sq", mode="bf16x3", nq=2000, bins=600, cols=192, cols_per_set=3),
        # one pass of the refinement loop against three isotopic datasets
        dict(name="refine_water_9999", kind="refine", system="water", atoms=9999, moves=2000, data=3),
        # 64 uneven replicas, water and silica, advanced, binned and transformed together
        dict(name="replicas_64", kind="replicas", boxes=64, lo=2000, hi=60000, moves=250),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "sweep", "sweep", "sweep", "gr", "gr", "smeared", "sq", "refine", "replicas"])
    system = rng.choice(["water", "silica"])
    if kind in ("step", "sweep"):
        if kind == "sweep":
            system = rng.choice(["water", "silica", "flexible"])
        n = _log_uniform(rng, 900, 100000 if kind == "step" or system == "silica" else 600000) // 3 * 3
        moves = min(_log_uniform(rng, 200, 6000), 300000000 // n)
        case = dict(kind=kind, system=system, atoms=n, moves=moves, r_lj=rng.choice([0.0, 0.0, 9.0]),
                    ep=rng.random() < 0.5)
        return case if kind == "step" else dict(case, log=rng.random() < 0.25)
    if kind == "gr":
        return dict(kind=kind, system=system, atoms=_log_uniform(rng, 900, 150000) // 3 * 3, cells=rng.random() < 0.4)
    if kind == "smeared":
        return dict(kind=kind, system=system, atoms=_log_uniform(rng, 900, 99999) // 3 * 3,
                    sigma=rng.choice([0.03, 0.05, 0.08]))
    if kind == "sq":
        sets = _log_uniform(rng, 1, 64)
        return dict(kind=kind, mode=rng.choice(["fp32", "tf32x3", "bf16x3", "bf16x6"]), nq=_log_uniform(rng, 200, 2000),
                    bins=_log_uniform(rng, 200, 600), cols=3 * sets, cols_per_set=3)
    if kind == "refine":
        return dict(kind=kind, system="water", atoms=_log_uniform(rng, 900, 30000) // 3 * 3,
                    moves=_log_uniform(rng, 200, 2000), data=rng.choice([1, 3]))
    return dict(kind=kind, boxes=rng.randrange(4, 33), lo=2000, hi=_log_uniform(rng, 6000, 30000),
                moves=rng.randrange(100, 250))


# ---- inputs ----------------------------------------------------------------------------------------

def _sites(n, spacing_min, L_fx, rng):
    """n sites of a cubic lattice (in random order), displaced so that none come closer than spacing_min."""
    k = 1
    while k ** 3 < n:
        k += 1
    a = L_fx / k / synth.SCALE
    at = rng.permutation(k ** 3)[:n]
    grid = np.stack([at % k, at // k % k, at // (k * k)], axis=1)
    jitter = max(0.0, 0.5 * (a - spacing_min))
    return k, grid, (grid + 0.5) * a + rng.uniform(-jitter, jitter, (n, 3))


def _orient(rng, n):
    q = rng.normal(size=(n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                  1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                  1 - 2 * (x * x + y * y)], axis=1).reshape(n, 3, 3)
    return np.einsum("nij,kj->nki", R, synth.water_geometry_A())


def _water_xyz(n_mol, L_fx, rng):
    k, grid, centre = _sites(n_mol, 2.3, L_fx, rng)
    off = _orient(rng, n_mol)
    ids = torch.full((k, k, k), -1, dtype=torch.int64, device=DEV)
    g = torch.from_numpy(grid).to(DEV)
    ids[g[:, 0], g[:, 1], g[:, 2]] = torch.arange(n_mol, device=DEV)
    L = L_fx / synth.SCALE
    shifts = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if (a, b, c) > (0, 0, 0)]
    for _ in range(40):
        pos = torch.from_numpy(centre[:, None] + off).to(DEV)
        bad = torch.zeros(n_mol, dtype=torch.bool, device=DEV)
        for s in shifts:
            nb = ids[(g[:, 0] + s[0]) % k, (g[:, 1] + s[1]) % k, (g[:, 2] + s[2]) % k]
            d = pos[:, :, None] - pos[nb.clamp(min=0)][:, None]
            d = d - L * torch.round(d / L)
            bad |= (nb >= 0) & (d.square().sum(-1).flatten(1).min(1).values < 1.0)
        at = bad.nonzero()[:, 0].cpu().numpy()
        if not len(at):
            break
        off[at] = _orient(rng, len(at))
    return (np.rint((centre[:, None] + off) * synth.SCALE).astype(np.int64) % L_fx).reshape(-1, 3)


def _system(name, n, seed, r_lj=0.0, bins=None):
    """A box of n atoms: the force field, bins and Q grid of `synth`'s box of that name."""
    rng = np.random.default_rng(seed)
    base = {"water": synth.water_box, "flexible": synth.flexible_water_box, "silica": synth.silica_box}[name](
        4, seed=0, **({} if name == "silica" else {"L_A": 20.8}))
    more = {}
    if name == "silica":
        L_fx = synth.box_side_fx(n, 0.0662)
        _, _, x = _sites(n, 1.5, L_fx, rng)
        xyz = np.rint(x * synth.SCALE).astype(np.int64) % L_fx
        typ = (np.arange(n) >= n // 3).astype(np.int32)
        start = np.arange(n + 1, dtype=np.int64)
    else:
        L_fx = synth.box_side_fx(n, 0.1)
        xyz = _water_xyz(n // 3, L_fx, rng)
        typ = np.tile(np.array([0, 1, 1], np.int32), n // 3)
        start = np.arange(0, n + 1, 3, dtype=np.int64)
    if bins:
        more = dict(n_bins=bins[0], bin_p=bins[1], bin_q=bins[2], Q=bins[3])
    return synth.System(**{**base.__dict__, "L_fx": L_fx, "xyz": xyz.astype(np.int32), "type": typ,
                           "mol_start": start, "seed": seed, "r_lj": r_lj, **more})


def _ep_table(s, seed):
    """An empirical potential of the size a refinement leaves: smooth, a few tenths of kJ/mol."""
    rng = np.random.default_rng(seed + 7)
    r = (np.arange(s.n_bins) + 0.5) * s.dr
    P = s.n_types * (s.n_types + 1) // 2
    amp, k, ph = rng.uniform(0.1, 0.4, (P, 1)), rng.uniform(1.0, 2.5, (P, 1)), rng.uniform(0, 6.28, (P, 1))
    return (amp * np.cos(k * r + ph) * np.exp(-r / 4.0)).astype(np.float32)


def _replica_systems(case, seed):
    rng = np.random.default_rng(3)               # the sizes belong to the case, the configurations to the seed
    sizes = [int(case["lo"] * (case["hi"] / case["lo"]) ** u) // 3 * 3 for u in rng.random(case["boxes"])]
    bins = (600, 2, 100, 0.3 + np.arange(2000) * (39.7 / 1999.0))
    return [_system("water" if i < case["boxes"] // 2 else "silica", n, seed * 1000 + i, bins=bins)
            for i, n in enumerate(sizes)]


def _datasets(s, n_data):
    """Eq. (1) weights (2 - delta) c_a c_b b_a b_b and flat parts of n_data isotopic samples, and target S(Q)."""
    c = np.bincount(s.type, minlength=s.n_types) / s.n_atoms
    w, flat = [], []
    for b_h in (-3.739, 6.671, 1.466)[:n_data]:
        b = 0.1 * np.array([s.b[0], b_h])
        w.append([(1 if i == j else 2) * c[i] * c[j] * b[i] * b[j] for i in range(2) for j in range(i, 2)])
        flat.append((c * b * b).sum())
    Q = s.Q.astype(np.float32).astype(np.float64)
    target = np.array(flat)[:, None] + 0.03 * np.sin(np.outer([1.0, 1.3, 0.8][:n_data], Q)) * np.exp(-Q / 6)
    return np.array(w), np.array(flat), target.astype(np.float32)


def _g_columns(case, seed):
    """Columns like a liquid's g(r): zero inside the core, damped oscillations about 1 beyond it."""
    rng = np.random.default_rng(seed)
    r = (np.arange(case["bins"]) + 0.5) * (12.0 / case["bins"])
    n = case["cols"]
    core, k, ph = rng.uniform(0.9, 2.6, (n, 1)), rng.uniform(1.8, 2.8, (n, 1)), rng.uniform(0, 6.28, (n, 1))
    g = (r > core) * (1.0 + np.exp(-r / 2.5) * np.cos(k * r + ph) * 1.5)
    Q = 0.3 + np.arange(case["nq"]) * (39.7 / max(1, case["nq"] - 1))
    return g.astype(np.float32), Q, rng.uniform(-0.3, 0.5, n), rng.uniform(0.2, 0.4, n // case["cols_per_set"])


def prepare(case, seed):
    st = {"case": case, "seed": seed, "move0": 0, "configs": 0}
    kind = case["kind"]
    if kind == "sq":
        g, Q, st["w"], st["flat"] = _g_columns(case, seed)
        st["g"] = torch.from_numpy(g).to(DEV)
        st["plan"] = epsr.SqPlan(Q, case["bins"], 12.0 / case["bins"], SQ_MODES[case["mode"]], max_cols=case["cols"])
        st["Sp"] = torch.zeros((case["cols"], case["nq"]), dtype=torch.float32, device=DEV)
        st["S"] = torch.zeros((case["cols"] // case["cols_per_set"], case["nq"]), dtype=torch.float32, device=DEV)
        return st
    systems = _replica_systems(case, seed) if kind == "replicas" else \
        [_system(case["system"], case["atoms"], seed, case.get("r_lj", 0.0))]
    s = systems[0]
    box = st["box"] = epsr.Box(systems)
    if case.get("ep"):
        box.epsr_box_set_ep(0, _ep_table(s, seed))
    P = s.n_types * (s.n_types + 1) // 2
    if kind in ("step", "sweep", "replicas"):
        st["xyz"] = torch.zeros((box.n_atoms, 3), dtype=torch.int32, device=DEV)
    if kind == "sweep" and case["log"]:
        st["log"] = torch.zeros(case["moves"] * epsr.MOVE_LOG_DTYPE.itemsize, dtype=torch.uint8, device=DEV)
    if kind in ("step", "gr", "replicas", "refine"):
        st["H"] = torch.zeros(box.hist_len, dtype=torch.int64, device=DEV)
        st["g"] = torch.zeros(box.hist_len, dtype=torch.float32, device=DEV)
    if kind in ("step", "gr", "replicas"):
        ws = [box.epsr_sq_weights(b) for b in range(box.n_boxes)]
        st["w"], st["flat"] = np.concatenate([w for w, _ in ws]), np.array([f for _, f in ws])
        st["plan"] = epsr.SqPlan(s.Q, s.n_bins, s.dr, epsr.SQ_BF16X3 if kind == "replicas" else epsr.SQ_FP32,
                                 max_cols=P * box.n_boxes)
        st["S"] = torch.zeros((box.n_boxes, len(s.Q)), dtype=torch.float32, device=DEV)
    if kind == "smeared":
        w_cols, flat = box.epsr_sq_weights(0)
        rho = s.n_atoms / s.L ** 3
        _, _, target, C_ = _smeared_inputs(case, s, seed)
        st["plan"] = epsr.SqPlan(s.Q, s.n_bins, s.dr, epsr.SQ_FP32, max_cols=P)
        st["pos"] = torch.from_numpy(s.xyz / synth.SCALE).float().to(DEV).requires_grad_(True)
        st["fn"] = epsr.smeared_chi2_function()
        st["args"] = (torch.from_numpy(C_).to(DEV), box, st["plan"], case["sigma"], w_cols / (4 * math.pi * rho),
                      w_cols, flat, torch.from_numpy(target).to(DEV), 0.5, rho)
    if kind == "refine":
        w, flat, target = _datasets(s, case["data"])
        st["plan"] = epsr.SqPlan(s.Q, s.n_bins, s.dr, epsr.SQ_FP32, max_cols=case["data"] * P)
        st["refiner"] = epsr.Refiner(box, st["plan"], torch.from_numpy(target).to(DEV), w, flat, s.Q,
                                     moves_per_pass=case["moves"], seed=seed, accumulate=True, n_basis=20, s_basis=0.5,
                                     gamma=0.0 if case["data"] == P else 0.01, alpha=0.1)
        st["S"] = torch.zeros((case["data"], len(s.Q)), dtype=torch.float32, device=DEV)
        st["dS"] = torch.zeros_like(st["S"])
        st["P"] = P
    return st


# ---- one pass --------------------------------------------------------------------------------------

def run(st):
    return globals()["_run_" + st["case"]["kind"]](st)


def _moves(st):
    case, box = st["case"], st["box"]
    stats = box.epsr_mc_sweep(case["moves"], st["seed"], st["move0"], log=st.get("log"))
    st["move0"] += case["moves"]
    box.epsr_box_get_coords_device(st["xyz"])
    return stats


def _run_sweep(st):
    out = {"stats": _moves(st), "xyz": st["xyz"]}
    if "log" in st:
        rec = st["log"].view(-1, epsr.MOVE_LOG_DTYPE.itemsize)
        out["dU"] = rec.view(torch.float32)[:, 2]
        out["moves"] = rec.view(torch.int32)[:, :2]
        out["trial"] = rec.view(torch.int32)[:, 6:30]
    return out


def _run_step(st):
    box = st["box"]
    out = {"stats": _moves(st), "xyz": st["xyz"]}
    st["configs"] += 1
    box.epsr_partial_gr(st["H"], st["g"], st["configs"])
    st["plan"].epsr_sq_exec(st["g"].view(len(st["w"]), -1), st["w"], len(st["w"]), st["flat"], None, st["S"])
    return dict(out, H=st["H"], g=st["g"], S=st["S"])


def _run_gr(st):
    box = st["box"]
    st["H"].zero_()
    (box.epsr_partial_gr_cells if st["case"]["cells"] else box.epsr_partial_gr)(st["H"], st["g"], 1)
    st["plan"].epsr_sq_exec(st["g"].view(len(st["w"]), -1), st["w"], len(st["w"]), st["flat"], None, st["S"])
    return {"H": st["H"], "g": st["g"], "S": st["S"]}


def _run_smeared(st):
    # one gradient step's worth: the loss is read back, as a minimiser does to judge its step
    st["pos"].grad = None
    chi2 = st["fn"].apply(st["pos"], *st["args"])
    chi2.backward()
    return {"chi2": chi2.item(), "grad": st["pos"].grad}


def _run_sq(st):
    st["plan"].epsr_sq_exec(st["g"], st["w"], st["case"]["cols_per_set"], st["flat"], st["Sp"], st["S"])
    return {"S_partial": st["Sp"], "S": st["S"]}


def _run_refine(st):
    # the pass, then what a run stores of it; the fitted coefficients are left to the table they
    # make: the basis is nearly collinear (condition 1e10), so they are not determined to 64 bits
    box, ref = st["box"], st["refiner"]
    out = ref.step()
    ref.get(hist=st["H"], g=st["g"], S=st["S"], dS=st["dS"])
    return dict(out, H=st["H"], g=st["g"], S=st["S"], dS=st["dS"],
                ep=box.epsr_box_get_ep(0, (st["P"], box.systems[0].n_bins)))


def _run_replicas(st):
    case, box = st["case"], st["box"]
    box.epsr_mc_sweep_async(case["moves"], st["seed"], st["move0"])
    st["move0"] += case["moves"]
    st["H"].zero_()
    box.epsr_partial_gr(st["H"], st["g"], 1)
    st["plan"].epsr_sq_exec(st["g"].view(len(st["w"]), -1), st["w"], 3, st["flat"], None, st["S"])
    box.epsr_box_get_coords_device(st["xyz"])
    return {"xyz": st["xyz"], "H": st["H"], "g": st["g"], "S": st["S"]}


# ---- work ------------------------------------------------------------------------------------------

def _sweep_work(system, n, moves, r_lj, ep, r_ep):
    """Moved atoms against their partners, old and new position: Lennard-Jones (20 operations) with every
    partner of a type that has one, or inside r_lj; Coulomb or the table (20) inside their range."""
    rho, m, lj_own, lj_all = (0.1, 3, 1, n // 3) if system != "silica" else (0.0662, 1, 1, n)
    near = min(n, rho * 4.19 * (r_ep if ep else 9.0) ** 3)
    far = min(lj_all, near * lj_all / n) if r_lj else lj_all
    return moves * 2 * 20.0 * (lj_own * far + m * near)


def work(case):
    kind = case["kind"]
    if kind == "sq":
        k, q, c = case["bins"], case["nq"], case["cols"]
        return {"bytes": 4.0 * (k * q + c * k + c * q + c * q / case["cols_per_set"]), "flops": 2.0 * k * q * c}
    if kind == "replicas":
        sizes = [case["lo"] * (case["hi"] / case["lo"]) ** ((i + 0.5) / case["boxes"]) for i in range(case["boxes"])]
        fl = sum(_sweep_work("water" if i < case["boxes"] // 2 else "silica", n, case["moves"], 0, False, 12.0) +
                 10.0 * _in_range("water" if i < case["boxes"] // 2 else "silica", n, 12.0) for i, n in enumerate(sizes))
        return {"bytes": 28.0 * sum(sizes) + case["boxes"] * (3 * 600 * 12 + 2000 * 4.0) + 4.8e6,
                "flops": fl + 2.0 * 600 * 2000 * 3 * case["boxes"]}
    n, silica = case["atoms"], case["system"] == "silica"
    r_max, n_bins, nq = (12.0, 600, 2000) if silica else (10.0, 333, 1000)
    out = {"bytes": 28.0 * n, "flops": 0.0}
    if "moves" in case:
        out["flops"] += _sweep_work(case["system"], n, case["moves"], case.get("r_lj", 0.0), case.get("ep", False), r_max)
        out["bytes"] += 128.0 * case["moves"] if case.get("log") else 0.0
    if kind in ("step", "gr", "refine"):
        sets = case.get("data", 1)
        out["flops"] += 10.0 * _in_range(case["system"], n, r_max) + 2.0 * 3 * n_bins * nq * sets
        out["bytes"] += 3.0 * n_bins * 12 + 4.0 * nq * sets * 2 + 4.0 * n_bins * nq
    if kind == "smeared":
        spread = 10.0 * case["sigma"] / (r_max / n_bins)
        out["flops"] += 2 * 10.0 * spread * _in_range(case["system"], n, r_max)
        out["bytes"] += 12.0 * n + 4.0 * n_bins * nq
    return out


def _in_range(system, n, r_max):
    return 0.5 * n * min(n, (0.0662 if system == "silica" else 0.1) * 4.19 * r_max ** 3)


# ---- the same in 64 bits -----------------------------------------------------------------------------

def _philox(c, key):
    """Philox4x32-10 of counters c [4][n] (uint64 holding 32-bit words)."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [x.astype(np.uint64) for x in c]
    k0, k1 = np.uint64(key & 0xFFFFFFFF), np.uint64(key >> 32)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
    return c


class _Chain:
    """The Metropolis chain of one box in 64 bits, one move after the other."""

    def __init__(self, s, box_index=0, ep=None):
        self.s, self.b = s, box_index
        self.X = torch.from_numpy(s.xyz.astype(np.int64)).to(DEV)
        self.h = s.xyz.astype(np.int64)
        self.typ = torch.from_numpy(s.type.astype(np.int64)).to(DEV)
        nt = s.n_types
        ke = (1.602176634e-19 ** 2) * 6.02214076e23 / (4 * math.pi * 8.8541878128e-12) * 1e7
        self.c12, self.c6, self.kqq = (torch.zeros((nt, nt), dtype=torch.float64, device=DEV) for _ in range(3))
        pair = np.zeros((nt, nt), np.int64)
        p = 0
        for a in range(nt):
            for b in range(a, nt):
                e, sg = math.sqrt(s.eps[a] * s.eps[b]), 0.5 * (s.sigma[a] + s.sigma[b])
                for i, j in ((a, b), (b, a)):
                    self.c12[i, j], self.c6[i, j], self.kqq[i, j] = 4 * e * sg ** 12, 4 * e * sg ** 6, ke * s.q[a] * s.q[b]
                    pair[i, j] = p
                p += 1
        S = synth.SCALE
        self.rc2 = round(s.r_coul * S) ** 2
        self.rl2 = round(s.r_lj * S) ** 2 if s.r_lj > 0 else None
        self.ep = None if ep is None else torch.from_numpy(ep.astype(np.float64)).to(DEV)
        self.pair, self.T = torch.from_numpy(pair).to(DEV), torch.from_numpy(_thresholds(s)).to(DEV)
        self.sum_dU = 0.0

    def _u(self, pos, typ, keep):
        L = self.s.L_fx
        d = (self.X[None] - pos[:, None]).abs()
        d2 = torch.minimum(d, L - d).square().sum(-1)
        r2 = d2.double() * (1.0 / synth.SCALE ** 2)
        c12, c6, kqq = (t[typ][:, self.typ] for t in (self.c12, self.c6, self.kqq))
        s6 = r2 ** -3
        lj = (c12 * s6 - c6) * s6
        if self.rl2 is not None:
            lj = torch.where(d2 < self.rl2, lj, 0.0)
        u = lj + torch.where(d2 < self.rc2, kqq * r2.rsqrt(), 0.0)
        if self.ep is not None:
            row, k = self.pair[typ][:, self.typ], torch.bucketize(d2, self.T, right=True) - 1
            u = u + torch.where(d2 < self.T[-1], self.ep[row, k.clamp(max=self.s.n_bins - 1)], 0.0)
        return torch.where(keep, u, 0.0)

    def _springs(self, pos, typ):
        e, S, L = 0.0, synth.SCALE, self.s.L_fx
        for i in range(len(pos)):
            for j in range(i + 1, len(pos)):
                d = np.abs(pos[i] - pos[j])
                r = math.sqrt(float((np.minimum(d, L - d).astype(np.float64) ** 2).sum())) / S
                e += self.s.bond_k[typ[i]][typ[j]] * (r - self.s.bond_d[typ[i]][typ[j]]) ** 2
        return e

    def run(self, n_moves, seed):
        s, L, S = self.s, self.s.L_fx, synth.SCALE
        t = np.arange(n_moves, dtype=np.uint64)
        z = np.zeros_like(t)
        w = sum((_philox([t, z, z + np.uint64(self.b), z + np.uint64(lane)], seed) for lane in range(4)), [])
        u53 = [((w[i] >> np.uint64(5)) * 67108864.0 + (w[i + 1] >> np.uint64(6))) * 2.0 ** -53 for i in (4, 6, 8, 10)]
        mol = (w[0] * np.uint64(s.n_mol)) >> np.uint64(32)
        M = round(s.max_translation * S)
        shift = np.stack([(w[1 + a] % np.uint64(2 * M + 1)).astype(np.int64) - M for a in range(3)], 1)
        h = math.tan(0.5 * s.max_rotation_deg * math.pi / 180.0) / math.sqrt(3.0)
        v = [h * (2.0 * u - 1.0) for u in u53[:3]]
        nn = np.sqrt(((1.0 + v[0] * v[0]) + v[1] * v[1]) + v[2] * v[2])
        qw, qx, qy, qz = 1.0 / nn, v[0] / nn, v[1] / nn, v[2] / nn
        R = np.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                      2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                      2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)], 1)
        R = np.rint(R * 1073741824.0).astype(np.int64).reshape(-1, 3, 3)
        kT = 1.380649e-23 * 6.02214076e23 * 1e-3 * s.temperature
        dU = np.zeros(n_moves)
        idx = torch.arange(s.n_atoms, device=DEV)
        for k in range(n_moves):
            a0, a1 = int(s.mol_start[int(mol[k])]), int(s.mol_start[int(mol[k]) + 1])
            old, m, typ = self.h[a0:a1], a1 - a0, s.type[a0:a1]
            kind = int(w[12][k] % np.uint64(3)) if s.flexible else (1 if s.rigid_molecules else 0)
            if kind == 1:
                o = old - old[0]
                o = np.where(2 * o > L, o - L, np.where(2 * o <= -L, o + L, o))
                sm = o.sum(0)
                num = sm * 1073741824 + (m * o - sm) @ R[k].T
                new = old[0] + ((num + m * 536870912) >> 30) // m + (0 if s.flexible else shift[k])
            elif kind == 0:
                new = old + shift[k]
            else:
                new = old.copy()
                new[int(w[13][k] % np.uint64(m))] += shift[k]
            new = new % L
            keep = ((idx < a0) | (idx >= a1))[None]
            tt = self.typ[a0:a1]
            pos = torch.from_numpy(np.concatenate([new, old])).to(DEV)
            du = float((self._u(pos[:m], tt, keep) - self._u(pos[m:], tt, keep)).sum())
            if s.flexible:
                du += self._springs(new, typ) - self._springs(old, typ)
            dU[k] = du
            if du <= 0 or (u53[3][k] > 0 and du < -kT * math.log(u53[3][k])) or u53[3][k] == 0:
                self.sum_dU += du
                self.h[a0:a1] = new
                self.X[a0:a1] = pos[:m]
        return dU


def _thresholds(s):
    return np.array([-(-(k * s.bin_p) ** 2 * (1 << 40) // s.bin_q ** 2) for k in range(s.n_bins + 1)], np.int64)


def _pairs(X, L, d2_max):
    """Chunks (i, j, d2) of the pairs i < j with d2 < d2_max."""
    n = len(X)
    rows = max(1, 16000000 // n)
    for i0 in range(0, n, rows):
        xi = X[i0:i0 + rows]
        d2 = torch.zeros((len(xi), n - i0), dtype=torch.int64, device=X.device)
        for a in range(3):
            d = (xi[:, None, a] - X[None, i0:, a]).abs()
            d2 += torch.minimum(d, L - d).square()
        keep = (d2 < d2_max).triu(1)
        i, j = keep.nonzero(as_tuple=True)
        yield i + i0, j + i0, d2[i, j]


def _pair_table(s):
    nt = s.n_types
    t = torch.zeros((nt, nt), dtype=torch.int64, device=DEV)
    order = [(a, b) for a in range(nt) for b in range(a, nt)]
    for p, (a, b) in enumerate(order):
        t[a, b] = t[b, a] = p
    c = np.bincount(s.type, minlength=nt).astype(np.float64)
    return t, np.array([0.5 * c[a] * (c[a] - 1) if a == b else c[a] * c[b] for a, b in order])


def _norm(s):
    k = np.arange(s.n_bins + 1) * s.dr
    return s.L ** 3 / (_pair_table(s)[1][:, None] * (4 * math.pi / 3) * np.diff(k ** 3)[None])


def _g_exact(s, X):
    tab, _ = _pair_table(s)
    T = torch.from_numpy(_thresholds(s)).to(DEV)
    typ = torch.from_numpy(s.type.astype(np.int64)).to(DEV)
    H = torch.zeros(tab.max().item() * s.n_bins + s.n_bins, dtype=torch.int64, device=DEV)
    for i, j, d2 in _pairs(X, s.L_fx, int(T[-1])):
        H += torch.bincount(tab[typ[i], typ[j]] * s.n_bins + torch.bucketize(d2, T, right=True) - 1, minlength=len(H))
    return H.cpu().numpy().reshape(-1, s.n_bins) * _norm(s)


def _sine(Q, bins, dr):
    q, r = np.asarray(Q, np.float32).astype(np.float64), (np.arange(bins) + 0.5) * dr
    return r * dr * np.sin(np.outer(q, r)) / q[:, None]


def _weights(s):
    c, b = np.bincount(s.type, minlength=s.n_types) / s.n_atoms, 0.1 * np.array(s.b[:s.n_types])
    rho = s.n_atoms / s.L ** 3
    w = [4 * math.pi * rho * (1 if i == j else 2) * c[i] * c[j] * b[i] * b[j]
         for i in range(s.n_types) for j in range(i, s.n_types)]
    return np.array(w), (c * b * b).sum()


def _sq_exact(s, g):
    w, flat = _weights(s)
    return flat + w @ ((g - 1.0) @ _sine(s.Q, s.n_bins, s.dr).T)


def _poisson_F(n_basis, sb, Q, rho):
    Q = np.asarray(Q, np.float32).astype(np.float64)
    F = []
    for n in range(1, n_basis + 1):
        m = n + 2
        log_c = n - n * math.log(n * sb) + math.lgamma(m) + m * math.log(sb)
        F.append(4 * math.pi * rho / Q * np.exp(log_c - 0.5 * m * np.log1p((Q * sb) ** 2)) * np.sin(m * np.arctan(Q * sb)))
    return np.stack(F)


def _smeared_inputs(case, s, seed):
    rng = np.random.default_rng(seed + 3)
    w, flat = _weights(s)
    Q = s.Q.astype(np.float32).astype(np.float64)
    target = flat + 0.05 * np.sin(1.3 * Q) * np.exp(-Q / 8) + rng.normal(size=len(Q)) * 0.005
    return w, flat, target.astype(np.float32), rng.normal(size=(len(w), 20)) * 0.001


def _smeared_exact(case, s, seed):
    w, flat, target, C_ = _smeared_inputs(case, s, seed)
    rho, sg, nb, dr = s.n_atoms / s.L ** 3, case["sigma"], s.n_bins, s.dr
    X = torch.from_numpy(s.xyz.astype(np.int64)).to(DEV)
    typ = torch.from_numpy(s.type.astype(np.int64)).to(DEV)
    tab, _ = _pair_table(s)
    reach = (nb * dr + 5 * sg) * synth.SCALE
    span = int(10 * sg / dr) + 2

    def bins(r):
        k0 = torch.floor((r - 5 * sg) / dr).long()
        for o in range(span):
            k = k0 + o
            lo, hi = (k.double() * dr - r) / sg, ((k + 1).double() * dr - r) / sg
            yield k.clamp(0, nb - 1), (k >= 0) & (k < nb), lo, hi

    P = len(w)
    H = torch.zeros(P * nb, dtype=torch.float64, device=DEV)
    for i, j, d2 in _pairs(X, s.L_fx, int(reach * reach)):
        r, p = d2.double().sqrt() / synth.SCALE, tab[typ[i], typ[j]]
        for k, ok, lo, hi in bins(r):
            a, b = (0.5 * torch.erf(t.clamp(-5, 5) * math.sqrt(0.5)) for t in (lo, hi))
            H.index_add_(0, p * nb + k, torch.where(ok, b - a, 0.0))
    norm = _norm(s)
    K, F = _sine(s.Q, nb, dr), _poisson_F(20, 0.5, s.Q, rho)
    res = flat + w @ ((H.cpu().numpy().reshape(P, nb) * norm - 1.0) @ K.T) + (w / (4 * math.pi * rho)) @ (C_ @ F) - target
    lam = torch.from_numpy((2 * w[:, None] * (res @ K)[None] * norm).reshape(-1)).to(DEV)
    grad = torch.zeros((s.n_atoms, 3), dtype=torch.float64, device=DEV)
    for i, j, d2 in _pairs(X, s.L_fx, int(reach * reach)):
        r, p = d2.double().sqrt() / synth.SCALE, tab[typ[i], typ[j]]
        f = torch.zeros_like(r)
        for k, ok, lo, hi in bins(r):
            a, b = (torch.where(t.abs() < 5, torch.exp(-0.5 * t * t), 0.0) for t in (lo, hi))
            f += torch.where(ok, lam[p * nb + k] * (a - b), 0.0)
        f *= 1.0 / (math.sqrt(2 * math.pi) * sg) / r
        d = X[i] - X[j]
        d = torch.where(2 * d > s.L_fx, d - s.L_fx, torch.where(2 * d <= -s.L_fx, d + s.L_fx, d)).double() / synth.SCALE
        grad.index_add_(0, i, f[:, None] * d)
        grad.index_add_(0, j, -f[:, None] * d)
    return {"chi2": float((res * res).sum()), "grad": grad}


def _refine_exact(case, s, seed):
    chain = _Chain(s)
    chain.run(case["moves"], seed)
    g = _g_exact(s, chain.X)
    w, flat, target = _datasets(s, case["data"])
    rho, P = s.n_atoms / s.L ** 3, len(w[0])
    S = flat[:, None] + 4 * math.pi * rho * w @ ((g - 1.0) @ _sine(s.Q, s.n_bins, s.dr).T)
    dS = target - S
    gamma = 0.0 if case["data"] == P else 0.01
    A, rhs = np.vstack([w, gamma * np.eye(P)]), np.vstack([dS, np.zeros((P, dS.shape[1]))])
    F = _poisson_F(20, 0.5, s.Q, rho)
    C_ = np.linalg.lstsq(F.T, np.linalg.lstsq(A, rhs, rcond=None)[0].T, rcond=None)[0].T
    r = (np.arange(s.n_bins) + 0.5) * s.dr
    p = np.stack([np.exp(n * np.log(r / (n * 0.5)) + n - r / 0.5) for n in range(1, 21)])
    ep = -0.1 * 1.380649e-23 * 6.02214076e23 * 1e-3 * s.temperature * (C_ @ p)
    return {"chi2": float((dS * dS).sum()), "ep_change_max": float(np.abs(ep).max()), "g": g.reshape(-1), "S": S,
            "dS": dS, "ep": ep}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sq":
        g, Q, w, flat = _g_columns(case, seed)
        Sp = w[:, None] * ((g.astype(np.float64) - 1.0) @ _sine(Q, case["bins"], 12.0 / case["bins"]).T)
        return {"S_partial": Sp, "S": flat[:, None] + Sp.reshape(len(flat), -1, len(Q)).sum(1)}
    if kind == "replicas":
        if case["boxes"] * case["moves"] > 20000:
            return None
        out = []
        for b, s in enumerate(_replica_systems(case, seed)):
            chain = _Chain(s, b)
            chain.run(case["moves"], seed)
            g = _g_exact(s, chain.X)
            out.append((g.reshape(-1), _sq_exact(s, g)))
        return {"g": np.concatenate([g for g, _ in out]), "S": np.stack([S for _, S in out])}
    s = _system(case["system"], case["atoms"], seed, case.get("r_lj", 0.0))
    if kind == "smeared":
        return _smeared_exact(case, s, seed)
    if kind == "refine":
        return _refine_exact(case, s, seed)
    if kind == "gr" and case["atoms"] > 150000:
        return None
    X, out = torch.from_numpy(s.xyz.astype(np.int64)).to(DEV), {}
    if kind in ("step", "sweep"):
        chain = _Chain(s, ep=_ep_table(s, seed) if case["ep"] else None)
        dU = chain.run(case["moves"], seed)
        out["stats"] = [[None, None, None, chain.sum_dU]]
        if case.get("log"):
            out["dU"] = dU
        X = chain.X
    if kind != "sweep":
        g = _g_exact(s, X)
        out.update(g=g.reshape(-1), S=_sq_exact(s, g)[None])
    return out
