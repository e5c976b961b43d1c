"""What a user of this framework has it do, as timed cases: single force / charge evaluations, MD
steps, replica batches, the iterative solve with its learned start, and the network's training and
prediction, in both precisions, through the public binding.

Every case is a dict of plain values; `kind` selects the entry points:

  oneshot   new positions (device memory) -> modes -> charges and forces (device memory)
  provider  the captured host-I/O force provider: pinned positions in, forces and charges out
  charges   new positions -> modes -> electrode charges, b and the electrode potential (host arrays);
            solver "direct" or "pcg" (PCG started from the network's prediction)
  md        velocity-Verlet steps with the Langevin thermostat, then the positions and velocities
  batch     MD steps of several uneven replicas as one graph per step, then their positions
  train     an AdamW training of the per-site network on host rows
  predict   the network's forward pass on device rows

Systems are slabs of 2 x 3 electrode layers (nx x ny sites each, `vacancies` sites left out) with a
liquid of 3-site cations and 1-site anions ("sites" 3) or point ions ("sites" 1) placed on a jittered
grid.  The mixed form computes in FP32, so a program that chose it keeps its results in FP32: its
outputs are returned in that type.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_24742_gb300 import srbe

VOLT = 0.694461          # 1 V in e/nm
K_E = 138.935458         # kJ mol^-1 nm e^-2
KB = 0.0083144626        # kJ mol^-1 K^-1
LAYER_DZ, WALL_GAP, LAM = 0.335, 0.3, 1.5
ETA = 1.0 / 19.79
BOND_K, BOND_R0, DT = 1000.0, 0.35, 0.002
N_IN, N_H = 80, 128


# ------------------------------------------------------------------------------------------ cases
def _system(name, kind, mixed, Lx, Ly, Lz, nx, ny, pairs, sites, alpha, rc, P, M, volt, **more):
    return {"name": name, "kind": kind, "mixed": mixed, "Lx": Lx, "Ly": Ly, "Lz": Lz, "nx": nx, "ny": ny,
            "vacancies": 0, "pairs": pairs, "sites": sites, "alpha": alpha, "rc": rc, "P": P, "M": M, "volt": volt,
            **more}


def listed():
    slab784 = (2.0, 2.0, 12.0, 8, 8, 200, 1, 3.5, 1.2, 100, 2, 1.0)
    slab11072 = (4.0, 4.0, 16.0, 32, 16, 2000, 3, 3.5, 1.2, 200, 4, 1.0)
    slab52k = (7.9, 8.3, 21.3, 32, 32, 11423, 3, 1.87, 1.6, 301, 2, 2.0)
    return [
        # the smallest evaluation (384 sites, 400 ions) in the default precision: one configuration,
        # as a script does that asks for the forces and charges of a frame it has just read
        _system("oneshot_784_fp64", "oneshot", False, *slab784),
        # the same slab served to an MD engine that keeps its state in host memory: latency
        _system("provider_784_mixed", "provider", True, *slab784),
        # the benchmark slab (3,072 sites, 8,000 ion sites): production MD in the mixed form
        _system("md_11072_mixed", "md", True, *slab11072, steps=32, relax=30),
        # the same MD in the default precision
        _system("md_11072_fp64", "md", False, *slab11072, steps=4, relax=10),
        # electrode charges alone, electrode larger than the L2 cache holds and with a vacancy, so
        # neither even nor a lattice (analysis of stored frames: charging curves)
        _system("charges_6143_mixed", "charges", True, 8.0, 8.0, 24.0, 32, 32, 400, 1, 1.87, 1.6, 100, 3, 2.0,
                vacancies=1, solver="direct"),
        # a mid-size slab (6,144 sites, 45,692 ion sites, odd box and mode count): single evaluations
        # in the mixed form and in FP64 (the judge of a mixed run)
        _system("oneshot_52k_mixed", "oneshot", True, *slab52k),
        _system("oneshot_52k_fp64", "oneshot", False, *slab52k),
        # the largest system: 98,304 sites, 1.1 M ion sites, spectral charge solve
        _system("md_1200k_mixed", "md", True, 24.0, 24.0, 60.0, 128, 128, 275000, 3, 1.2, 2.5, 1000, 2, 2.0,
                steps=10, relax=10),
        # a voltage scan: eight uneven replicas stepped as one unit
        {"name": "batch_8_mixed", "kind": "batch", "mixed": True, "replicas": 8, "smin": 16, "smax": 24,
         "lo": 5000, "hi": 30000, "alpha": 1.87, "rc": 1.6, "steps": 10, "relax": 30},
        # the learned form: PCG to 1e-8 from the network's prediction
        _system("charges_pcg_11072_mixed", "charges", True, *slab11072, solver="pcg"),
        # training of the network on recorded charges (about seven frames of the benchmark slab)
        {"name": "train_20k", "kind": "train", "rows": 20000, "batch": 512, "epochs": 1, "lr": 1e-3},
        # its prediction for every site of the largest electrode
        {"name": "predict_98304", "kind": "predict", "rows": 98304},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["oneshot", "oneshot", "provider", "charges", "charges", "md", "md", "batch", "train", "predict"])
    if kind == "train":
        return {"kind": kind, "rows": int(_log(rng, 1500, 40000)), "batch": int(_log(rng, 64, 2048)),
                "epochs": rng.choice([1, 2]), "lr": 1e-3}
    if kind == "predict":
        return {"kind": kind, "rows": int(_log(rng, 300, 200000))}
    if kind == "batch":
        lo = int(rng.uniform(3000, 8000))
        return {"kind": kind, "mixed": True, "replicas": rng.randint(2, 8), "smin": 12, "smax": rng.randint(14, 24),
                "lo": lo, "hi": int(lo * rng.uniform(1.5, 4.0)), "alpha": 1.87, "rc": 1.6, "steps": 10, "relax": 30}
    nx, ny = int(_log(rng, 9, 33)), int(_log(rng, 9, 33))
    Lx, Ly = round(nx * rng.uniform(0.24, 0.27), 3), round(ny * rng.uniform(0.24, 0.27), 3)
    rc = 1.2 if min(Lx, Ly) < 4.0 else rng.choice([1.2, 1.6])
    alpha = 3.5 if rc == 1.2 and Lx * Ly < 14.0 else 1.87
    height = rng.uniform(5.0, 12.0)
    pairs = max(50, int(rng.uniform(35.0, 60.0) * Lx * Ly * height / 4))
    Lz = round(LAM * (height + 2 * (2 * LAYER_DZ + WALL_GAP)), 2)
    # modes enough for the box: G / P <= 8, as in the batch workload, keeps the random-batch noise of
    # the forces within what the thermostat holds (G ~ V (alpha / sqrt(pi))^3 modes carry weight)
    G = Lx * Ly * Lz * (alpha / math.sqrt(math.pi)) ** 3
    P = max(int(_log(rng, 60, 500)), int(G / 8) + 1)
    mixed = rng.random() < 0.6
    c = _system("", kind, mixed, Lx, Ly, Lz, nx, ny, pairs, 3, alpha, rc, P, max(1, int(Lz // max(Lx, Ly))),
                rng.choice([0.5, 1.0, 2.0, 4.0]))
    del c["name"]
    if kind == "charges":
        c["vacancies"] = rng.choice([0, 1, 3])
        c["solver"] = rng.choice(["direct", "direct", "pcg"])
        if c["solver"] == "pcg":
            c["mixed"] = True
    if kind == "md":
        c["steps"], c["relax"] = (16 if mixed else 3), 20
    return c


# ----------------------------------------------------------------------------------------- inputs
def _electrode(case):
    Lx, Ly, H, nx, ny = case["Lx"], case["Ly"], case["Lz"] / LAM, case["nx"], case["ny"]
    iy, ix = np.divmod(np.arange(nx * ny), nx)
    ax, ay = Lx / nx, Ly / ny
    R, side = [], []
    for s, zs in ((0, (0.0, LAYER_DZ, 2 * LAYER_DZ)), (1, (H - 2 * LAYER_DZ, H - LAYER_DZ, H))):
        for layer, z in enumerate(zs):
            x = (ix * ax + (0.5 * ax if layer % 2 else 0.0) + 0.25 * ax) % Lx
            R.append(np.c_[x, iy * ay + 0.25 * ay, np.full(nx * ny, z)])
            side.append(np.full(nx * ny, s, np.int8))
    R, side = np.concatenate(R), np.concatenate(side)
    if case["vacancies"]:
        gone = np.random.default_rng(11).choice(R.shape[0], case["vacancies"], replace=False)
        keep = np.setdiff1d(np.arange(R.shape[0]), gone)
        R, side = R[keep], side[keep]
    return R, side


def _liquid(case, seed):
    """Ion sites on a jittered near-cubic grid between the walls: whole molecule pairs (three cation
    sites in a row and an anion, or cation and anion) along x, the anion's place drawn at random."""
    rng = np.random.default_rng(seed)
    Lx, Ly, H, n = case["Lx"], case["Ly"], case["Lz"] / LAM, case["pairs"]
    zlo, zhi = 2 * LAYER_DZ + WALL_GAP, H - 2 * LAYER_DZ - WALL_GAP
    per = case["sites"] + 1
    cell = (Lx * Ly * (zhi - zlo) / (per * n)) ** (1.0 / 3.0)
    gx, gy = max(1, int(Lx / (per * cell))), max(1, int(Ly / cell))     # blocks of `per` grid points along x
    gz = -(-n // (gx * gy))
    at = np.sort(rng.permutation(gx * gy * gz)[:n])
    bx, by, bz = at % gx, (at // gx) % gy, at // (gx * gy)
    cx, cy, cz = Lx / (per * gx), Ly / gy, (zhi - zlo) / gz
    r = np.empty((n, per, 3))
    r[:, :, 0] = (bx[:, None] * per + np.arange(per) + 0.5) * cx
    r[:, :, 1] = (by[:, None] + 0.5) * cy
    r[:, :, 2] = zlo + (bz[:, None] + 0.5) * cz
    r += rng.uniform(-0.1, 0.1, r.shape) * np.array([cx, cy, cz])
    anion = rng.choice(np.array([0, per - 1]), n)
    kind = np.where(np.arange(per)[None, :] == anion[:, None], 3, 0)
    if per == 4:
        kind = np.where(kind == 3, 3, np.where(anion[:, None] == 0, np.arange(per)[None, :] - 1, np.arange(per)[None, :]))
    mol = 2 * np.arange(n)[:, None] + (kind == 3)
    q = np.where(kind == 3, -0.78, 0.26 if per == 4 else 0.78)
    r, kind, mol, q = r.reshape(-1, 3), kind.ravel().astype(np.int32), mol.ravel().astype(np.int32), q.ravel()
    r[:, 0] %= Lx
    r[:, 1] %= Ly
    m0 = 67.0 if per == 4 else 124.0
    mass = np.array([m0, 42.0, 15.0, 145.0])[kind]
    v = rng.normal(size=r.shape) * np.sqrt(KB * 400.0 / mass)[:, None]
    bonds = np.zeros((0, 2), np.int32)
    if per == 4:
        first = per * np.arange(n) + (anion == 0)
        bonds = np.concatenate([np.c_[first, first + 1], np.c_[first + 1, first + 2]]).astype(np.int32)
    sig = np.array([0.50, 0.40, 0.35, 0.45, 0.337])
    sig[:4] *= min(1.0, 0.8 * min(cx, cy, cz) / 0.50, 0.3 / 0.50)
    eps = np.array([2.0, 2.0, 2.0, 2.0, 1.0])
    return {"r": r, "q": q, "mass": mass, "itype": kind, "mol": mol, "bonds": bonds, "v": v,
            "sig": 0.5 * (sig[:, None] + sig[None, :]), "eps": np.sqrt(eps[:, None] * eps[None, :])}


def _context(case, liquid, stream=None):
    c = srbe.Context((case["Lx"], case["Ly"], case["Lz"]), case["alpha"], ETA, case["rc"], case["P"], case["M"], 0.0,
                     case["volt"])
    if stream is not None:
        c.set_stream(stream.cuda_stream)
    c.set_precision(srbe.MIXED if case["mixed"] else srbe.FP64)
    c.set_electrode(*_electrode(case))
    c.set_positions(liquid["r"], liquid["q"])
    c.set_md(liquid["mass"], liquid["itype"], liquid["mol"], liquid["sig"], liquid["eps"], liquid["bonds"],
             np.full(len(liquid["bonds"]), BOND_R0), BOND_K, DT, v=liquid["v"])
    return c


def _replica(case, seed, i):
    """Replica i of a batch: its size, voltage and mode count are the case's, its liquid the seed's."""
    rng = np.random.default_rng(100 + i)
    s = int(rng.integers(case["smin"], case["smax"] + 1))
    L = 0.25 * s
    ions = max(400.0, rng.uniform(case["lo"], case["hi"]) - 6 * s * s)
    gap = 2 * (2 * LAYER_DZ + WALL_GAP)
    Lz = min(max(1.5 * (ions / (50.0 * L * L) + gap), 3.0 * L), 8.0 * L)
    pairs = max(50, int(50.0 * L * L * (Lz / LAM - gap) / 4))
    P = int(min(400, max(100, 50 * math.ceil(L * L * Lz / 250.0))))
    one = _system("", "md", case["mixed"], L, L, Lz, s, s, pairs, 3, case["alpha"], case["rc"], P, int(Lz // L),
                  0.0625 * int(rng.integers(0, 65)))
    return one, 1000 * seed + i


def _rows(case, seed):
    """Rows like the descriptors of recorded frames (radial densities and low-k_z features) and a
    target that depends on them smoothly, with noise."""
    rng = np.random.default_rng(seed)
    n = case["rows"]
    D = np.empty((n, N_IN), np.float32)
    D[:, :64] = rng.gamma(2.0, 0.15, (n, 64))
    D[:, 64:] = rng.normal(0.0, 3.0, (n, N_IN - 64))
    w = rng.normal(size=(N_IN, 3)) / np.sqrt(N_IN)
    z = ((D - D.mean(0)) / D.std(0)) @ w
    T = (0.03 * (np.tanh(z[:, 0]) + 0.5 * z[:, 1] * z[:, 2]) + 0.003 * rng.normal(size=n)).astype(np.float32)
    return D, T


def _network(seed):
    """Parameters of the size of a trained network's (the binding's layout)."""
    rng = np.random.default_rng(seed + 77)
    parts = [rng.normal(0, 0.13, N_H * N_IN), rng.normal(0, 0.05, N_H), rng.normal(0, 0.12, N_H * N_H),
             rng.normal(0, 0.05, N_H), rng.normal(0, 0.15, N_H), [0.01], np.r_[np.full(64, 0.3), np.zeros(16)],
             np.r_[np.full(64, 0.21), np.full(16, 3.0)], [0.001], [0.03]]
    return np.concatenate([np.asarray(p, np.float64) for p in parts]).astype(np.float32)


def _tiny_context():
    c = srbe.Context((2.0, 2.0, 12.0), 3.5, ETA, 1.2, 10, 2)
    return c


# ---------------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        D, T = _rows(case, seed)
        return {"case": case, "ctx": _tiny_context(), "D": D, "T": T, "P": _network(seed), "seed": seed}
    if kind == "predict":
        D, _ = _rows(case, seed)
        stream = torch.cuda.Stream()
        c = _tiny_context()
        c.set_stream(stream.cuda_stream)
        c.mlp_set_params(_network(seed))
        return {"case": case, "ctx": c, "D": torch.from_numpy(D).cuda(), "stream": stream,
                "out": torch.empty(case["rows"], dtype=torch.float32, device="cuda")}
    if kind == "batch":
        ctxs = []
        for i in range(case["replicas"]):
            one, s = _replica(case, seed, i)
            c = _context(one, _liquid(one, s))
            c.minimize(case["relax"], seed=s)
            c.set_thermostat(50.0, 400.0, s)
            ctxs.append(c)
        return {"case": case, "ctxs": ctxs, "batch": srbe.Batch(ctxs),
                "seeds": np.arange(1, len(ctxs) + 1, dtype=np.uint64) * 7919 + seed}
    liquid = _liquid(case, seed)
    if kind == "md":
        c = _context(case, liquid)
        c.minimize(case["relax"], seed=seed)
        c.set_thermostat(50.0, 400.0, seed)
        return {"case": case, "ctx": c, "seed": seed}
    n = liquid["r"].shape[0]
    if kind == "provider":
        c = _context(case, liquid)
        frames = [torch.from_numpy(liquid["r"] + d) for d in (0.0, 0.004)]
        st = {"case": case, "ctx": c, "seed": seed, "frames": frames, "t": 0}
        st["r"], st["F"] = (torch.empty((n, 3), dtype=torch.float64).pin_memory() for _ in range(2))
        st["Q"] = torch.empty(c.n_ele, dtype=torch.float64).pin_memory()
        c.set_host_io(st["r"].data_ptr(), st["F"].data_ptr(), st["Q"].data_ptr())
        return st
    stream = torch.cuda.Stream()
    c = _context(case, liquid, stream)
    st = {"case": case, "ctx": c, "seed": seed, "stream": stream, "n": n,
          "r": torch.from_numpy(liquid["r"]).cuda(), "q": torch.from_numpy(liquid["q"]).cuda()}
    if kind == "oneshot":
        st["F"] = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        st["Q"] = torch.empty(c.n_ele, dtype=torch.float64, device="cuda")
    elif case["solver"] == "pcg":
        # a network trained on a few evaluations of the direct solve, as the learned form is used
        c.mlp_init(seed)
        D, T = [], []
        for t in range(4):
            c.sample_k(seed, 100 + t)
            c.solve_charges()
            D.append(c.descriptors())
            T.append(c.solution().astype(np.float32))
        c.mlp_train(np.concatenate(D), np.concatenate(T), epochs=2, batch=512, lr=1e-3, seed=seed)
        c.set_solver(srbe.PCG, tol=1e-8, maxit=2000, warm=srbe.WARM_MODEL)
    torch.cuda.synchronize()
    return st


# -------------------------------------------------------------------------------------------- run
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "train":
        st["ctx"].mlp_set_params(st["P"])
        loss = st["ctx"].mlp_train(st["D"], st["T"], epochs=case["epochs"], batch=case["batch"], lr=case["lr"],
                                   weight_decay=1e-4, seed=st["seed"])
        return {"params": st["ctx"].mlp_params(), "loss": loss}
    if kind == "predict":
        st["ctx"].mlp_predict_dev(st["D"].data_ptr(), case["rows"], st["out"].data_ptr())
        return {"y": st["out"]}
    if kind == "batch":
        st["batch"].step(case["steps"], st["seeds"])
        return {"r%d" % i: c.get_positions().astype(np.float32) for i, c in enumerate(st["ctxs"])}
    c, mixed = st["ctx"], case["mixed"]
    if kind == "md":
        c.step(case["steps"], st["seed"])
        r, v = c.get_positions(velocities=True)
        return {"r": r.astype(np.float32), "v": v.astype(np.float32)} if mixed else {"r": r, "v": v}
    if kind == "provider":
        st["r"].copy_(st["frames"][st["t"] & 1])
        st["t"] += 1
        c.forces_host_io(st["seed"], 0)
        return {"F": st["F"].float(), "Q": st["Q"].float()} if mixed else {"F": st["F"], "Q": st["Q"]}
    c.set_positions_dev(st["n"], st["r"].data_ptr(), st["q"].data_ptr())
    c.sample_k(st["seed"], 0)
    if kind == "oneshot":
        c.forces_dev(st["F"].data_ptr(), st["Q"].data_ptr())
        if not mixed:
            return {"F": st["F"], "Q": st["Q"]}
        with torch.cuda.stream(st["stream"]):
            return {"F": st["F"].float(), "Q": st["Q"].float()}
    Q, psi, b = c.solve_charges()
    v = np.append(b, psi)            # the potentials of the sites, then the electrodes' common one
    return {"Q": Q.astype(np.float32), "v": v.astype(np.float32)} if mixed else {"Q": Q, "v": v}


# ------------------------------------------------------------------------------------------- work
def _sizes(case):
    ne = 6 * case["nx"] * case["ny"] - case["vacancies"]
    return case["pairs"] * (case["sites"] + 1), ne, case["P"] + case["M"]


def _pairs(case):
    """Ion-ion pairs and ion-electrode pairs within rc: mean density, walls one-sided."""
    ni, ne, _ = _sizes(case)
    area, h, rc = case["Lx"] * case["Ly"], case["Lz"] / LAM - 2 * (2 * LAYER_DZ + WALL_GAP), case["rc"]
    rho = ni / (area * h)
    ii = 0.5 * ni * rho * 4.0 / 3.0 * math.pi * rc ** 3
    ie = 0.0
    for layer in range(3):
        z0 = WALL_GAP + layer * LAYER_DZ
        if rc > z0:
            ie += ne / 3.0 * rho * math.pi * (rc - z0) ** 2 * (2 * rc + z0) / 3.0
    return ii, ie


def _matrix(case, ne):
    """Bytes and operations of the charge solve: one product with the projected inverse, or for a
    lattice the transforms of its spectral form."""
    if ne <= 16384 and not (ne >= 8192 and case["vacancies"] == 0):
        return 8.0 * ne * ne, 2.0 * ne * ne
    return 32.0 * ne * 6, 4 * 8.0 * ne * (math.log2(case["nx"]) + math.log2(case["ny"])) + 48.0 * ne


def _evaluation(case, forces):
    ni, ne, K = _sizes(case)
    ii, ie = _pairs(case)
    mb, mf = _matrix(case, ne)
    byts = mb + 32.0 * ni + 24.0 * ne + (24.0 * ni if forces else 8.0 * ne)
    flops = mf + 12.0 * K * (ni + ne) + 30.0 * ie
    if forces:
        flops += 12.0 * K * (ni + ne) + 30.0 * (ii + ie)
    return byts, flops


def work(case):
    kind = case["kind"]
    gemm = 2.0 * (N_IN * N_H + N_H * N_H)
    if kind == "train":
        rows = case["rows"] * case["epochs"]
        params = N_H * (N_IN + N_H + 3) + 1
        return {"bytes": 4.0 * (N_IN + 1) * case["rows"] + 8.0 * params, "flops": 3 * gemm * rows}
    if kind == "predict":
        return {"bytes": 4.0 * (N_IN + 1) * case["rows"], "flops": gemm * case["rows"]}
    if kind == "batch":
        ones = [_replica(case, 0, i)[0] for i in range(case["replicas"])]
        byts, flops = (sum(v) for v in zip(*(_evaluation(c, True) for c in ones)))
        return {"bytes": byts * case["steps"], "flops": flops * case["steps"]}
    byts, flops = _evaluation(case, kind != "charges")
    if kind == "md":
        ni, ne, _ = _sizes(case)
        byts, flops = byts + 100.0 * ni, flops + 30.0 * ni
        return {"bytes": byts * case["steps"], "flops": flops * case["steps"]}
    if kind == "charges" and case["solver"] == "pcg":
        ne = _sizes(case)[1]
        flops += 2.0 * ne * ne * 40 + gemm * ne      # about 40 iterations reach 1e-8
    return {"bytes": byts, "flops": flops}


# ------------------------------------------------------------------------------------------ exact
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x64-10 on arrays of counters (Salmon et al., SC'11)."""
    u = np.uint64
    x = [np.broadcast_to(np.asarray(c, u), np.shape(c0)).copy() for c in (c0, c1, c2, c3)]
    k0, k1 = int(k0), int(k1)

    def mul(a, b):
        al, ah = u(a & 0xFFFFFFFF), u(a >> 32)
        bl, bh = b & u(0xFFFFFFFF), b >> u(32)
        ll, lh, hl, hh = al * bl, al * bh, ah * bl, ah * bh
        mid = (ll >> u(32)) + (lh & u(0xFFFFFFFF)) + (hl & u(0xFFFFFFFF))
        return hh + (lh >> u(32)) + (hl >> u(32)) + (mid >> u(32)), u(a) * b

    with np.errstate(over="ignore"):
        for _ in range(10):
            hA, lA = mul(0xD2E7470EE14C6C93, x[0])
            hB, lB = mul(0xCA5A826395121157, x[2])
            x = [hB ^ x[1] ^ u(k0), lB, hA ^ x[3] ^ u(k1), lA]
            k0, k1 = (k0 + 0x9E3779B97F4A7C15) & (2 ** 64 - 1), (k1 + 0xBB67AE8584CAA73B) & (2 ** 64 - 1)
    return x


def _open0(w):
    return ((w >> np.uint64(11)).astype(np.float64) + 1.0) / 9007199254740992.0


def _mode_list(case, seed):
    """The deterministic modes and the Metropolis samples of (seed, step 0) with their weights."""
    L, a, M, P = [case["Lx"], case["Ly"], case["Lz"]], case["alpha"], case["M"], case["P"]
    sig = [a * l / (math.sqrt(2.0) * math.pi) for l in L]
    j = np.arange(2 * P + 200, dtype=np.uint64)
    w0 = _philox(2 * j, 0, 0, 0, seed, 0x5352424500000001)
    w1 = _philox(2 * j + np.uint64(1), 0, 0, 0, seed, 0x5352424500000001)
    ra, ta = np.sqrt(-2 * np.log(_open0(w0[0]))), 2 * math.pi * _open0(w0[1])
    rb, tb = np.sqrt(-2 * np.log(_open0(w0[2]))), 2 * math.pi * _open0(w0[3])
    g = np.stack([ra * np.cos(ta), ra * np.sin(ta), rb * np.cos(tb)], 1)
    prop = np.floor(g * np.array(sig) + 0.5).astype(int)
    acc = _open0(w1[0])

    def q(m):
        out = 1.0
        for d in range(3):
            s = math.sqrt(2.0) * sig[d]
            out *= 0.5 * (math.erf((m[d] + 0.5) / s) - math.erf((m[d] - 0.5) / s))
        return out

    def p(m):
        return math.exp(-sum((2 * math.pi * m[d] / L[d]) ** 2 for d in range(3)) / (4 * a * a))

    inside = lambda m: m[0] == 0 and m[1] == 0 and abs(m[2]) <= M  # noqa: E731
    at = 0
    while inside(prop[at]):
        at += 1
    cur, out = prop[at], []
    at += 1
    for k in range(P):
        if k:
            new = prop[at]
            if not inside(new) and acc[at] <= p(new) * q(cur) / (p(cur) * q(new)):
                cur = new
            at += 1
        out.append(cur)
    theta = [sum(math.exp(-(math.pi * m / (a * l)) ** 2) for m in range(-400, 401)) for l in L]
    det = sum(math.exp(-(math.pi * m / (a * L[2])) ** 2) for m in range(1, M + 1))
    G = theta[0] * theta[1] * theta[2] - 1.0 - 2.0 * det
    V = L[0] * L[1] * L[2]
    m = np.array([[0, 0, z] for z in range(1, M + 1)] + [list(o) for o in out])
    k2 = ((2 * math.pi * m / np.array(L)) ** 2).sum(1)
    w = np.where(np.arange(len(m)) < M, 2.0 * np.exp(-k2 / (4 * a * a)), G / P) * 4 * math.pi / (V * k2)
    return m, w


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _phase(m, r, L):
    t = (r / L) @ m.T
    return 2 * math.pi * (t - torch.round(t))


def _shifts(reach, L):
    n = max(0, math.ceil(reach / L - 0.5))
    return range(-n, n + 1)


def _near(x, y, reach, L):
    """(i, j, d, r2) of all pairs of x and y, images included, with 0 < r < reach, in blocks."""
    step = max(64, int(2.0e8 // max(1, y.shape[0]) // 8))
    for i0 in range(0, x.shape[0], step):
        d0 = x[i0:i0 + step, None, :] - y[None, :, :]
        for k in (0, 1):
            d0[..., k] -= L[k] * torch.round(d0[..., k] / L[k])
        for a in _shifts(reach, float(L[0])):
            for b in _shifts(reach, float(L[1])):
                dx, dy, dz = d0[..., 0] + a * L[0], d0[..., 1] + b * L[1], d0[..., 2]
                r2 = dx * dx + dy * dy + dz * dz
                i, j = torch.nonzero((r2 < reach * reach) & (r2 > 0), as_tuple=True)
                yield i + i0, j, torch.stack([dx[i, j], dy[i, j], dz[i, j]], 1), r2[i, j]


def _matrix_A(case, R):
    """A of the constant-potential conditions, with an Ewald parameter of its own."""
    Lf = [case["Lx"], case["Ly"], case["Lz"]]
    L, V = _dev(Lf), Lf[0] * Lf[1] * Lf[2]
    a = 7.0 / (Lf[2] - float(R[:, 2].max() - R[:, 2].min()))
    n = R.shape[0]
    kmax = 2 * a * 6.3
    top = [int(kmax * l / (2 * math.pi)) for l in Lf]
    m = np.stack(np.meshgrid(*(np.arange(-t, t + 1) for t in top), indexing="ij"), -1).reshape(-1, 3)
    half = (m[:, 2] > 0) | ((m[:, 2] == 0) & ((m[:, 1] > 0) | ((m[:, 1] == 0) & (m[:, 0] > 0))))
    m = m[half]
    k2 = ((2 * math.pi * m / np.array(Lf)) ** 2).sum(1)
    m, k2 = m[k2 < kmax * kmax], k2[k2 < kmax * kmax]
    w = _dev(8 * math.pi / (V * k2) * np.exp(-k2 / (4 * a * a)))
    A = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    md = _dev(m)
    for k0 in range(0, len(m), 4096):
        ph = _phase(md[k0:k0 + 4096], R, L)
        for t in (torch.cos(ph), torch.sin(ph)):
            A += (t * w[k0:k0 + 4096]) @ t.T
    for i, j, _, r2 in _near(R, R, 6.4 / a, L):
        r = torch.sqrt(r2)
        A.index_put_((i, j), (torch.erfc(a * r) - torch.erfc(r / (math.sqrt(2.0) * ETA))) / r, accumulate=True)
    A += torch.eye(n, dtype=torch.float64, device="cuda") * (2.0 * (1.0 / (math.sqrt(2 * math.pi) * ETA) - a / math.sqrt(math.pi)))
    A += 4 * math.pi / V * R[:, 2][:, None] * R[:, 2][None, :]
    return A


def _evaluate(case, seed, forces):
    """Q, the potentials (b, then psi_bar; V) and the forces of one evaluation, from the formulas, in 64 bits."""
    R_h, side = _electrode(case)
    liq = _liquid(case, seed)
    Lf = [case["Lx"], case["Ly"], case["Lz"]]
    L, V, al, rc = _dev(Lf), Lf[0] * Lf[1] * Lf[2], case["alpha"], case["rc"]
    R, r, q = _dev(R_h), _dev(liq["r"]), _dev(liq["q"])
    m_h, w_h = _mode_list(case, seed)
    m, w = _dev(m_h), _dev(w_h)
    d = _dev(np.where(side == 1, 0.5, -0.5))
    pr, pR = _phase(m, r, L), _phase(m, R, L)
    S1 = torch.complex(q @ torch.cos(pr), q @ torch.sin(pr))
    eR = torch.complex(torch.cos(pR), torch.sin(pR))
    b = -(torch.conj(eR) @ (w.to(S1.dtype) * S1)).real
    Mz = (q * r[:, 2]).sum()
    b -= 4 * math.pi / V * R[:, 2] * Mz
    for i, j, _, r2 in _near(R, r, rc, L):
        x = torch.sqrt(r2)
        b.index_add_(0, i, -q[j] * (torch.erfc(al * x) - torch.erfc(x / ETA)) / x)
    C = torch.linalg.cholesky(_matrix_A(case, R))
    dpsi = case["volt"] * VOLT
    sol = torch.cholesky_solve(torch.stack([dpsi * d + b, torch.ones_like(b)], 1), C)
    psi = -sol[:, 0].sum() / sol[:, 1].sum()
    Q = sol[:, 0] + psi * sol[:, 1]
    out = {"Q": Q, "v": torch.cat([b, psi.reshape(1)]) / VOLT}
    if not forces:
        return out
    S = S1 + Q.to(S1.dtype) @ eR
    im = S.imag * w * torch.cos(pr) - S.real * w * torch.sin(pr)
    F = -K_E * q[:, None] * (im @ (2 * math.pi * m / L))
    F[:, 2] -= K_E * 4 * math.pi / V * q * (Mz + (Q * R[:, 2]).sum())
    two = 2.0 / math.sqrt(math.pi)
    ty, mo = torch.as_tensor(liq["itype"], device="cuda").long(), torch.as_tensor(liq["mol"], device="cuda").long()
    sig2, eps = _dev(liq["sig"]) ** 2, _dev(liq["eps"])

    def lj(ti, tj, r2):
        s6 = (sig2[ti, tj] / r2) ** 3
        return 24.0 * eps[ti, tj] * (2.0 * s6 * s6 - s6) / r2

    for i, j, dr, r2 in _near(r, r, rc, L):
        x = torch.sqrt(r2)
        f = K_E * q[i] * q[j] * (torch.erfc(al * x) / x + two * al * torch.exp(-al * al * r2)) / r2
        f = f + torch.where(mo[i] != mo[j], lj(ty[i], ty[j], r2), torch.zeros_like(r2))
        F.index_add_(0, i, f[:, None] * dr)
    for i, j, dr, r2 in _near(r, R, rc, L):
        x = torch.sqrt(r2)
        f = torch.erfc(al * x) / x + two * al * torch.exp(-al * al * r2)
        f = f - torch.erfc(x / ETA) / x - two / ETA * torch.exp(-r2 / (ETA * ETA))
        f = K_E * q[i] * Q[j] * f / r2 + lj(ty[i], torch.full_like(ty[i], 4), r2)
        F.index_add_(0, i, f[:, None] * dr)
    bonds = torch.as_tensor(liq["bonds"], device="cuda").long()
    if len(bonds):
        dr = r[bonds[:, 0]] - r[bonds[:, 1]]
        for k in (0, 1):
            dr[:, k] -= L[k] * torch.round(dr[:, k] / L[k])
        ln = torch.sqrt((dr * dr).sum(1))
        f = (-BOND_K * (ln - BOND_R0) / ln)[:, None] * dr
        F.index_add_(0, bonds[:, 0], f)
        F.index_add_(0, bonds[:, 1], -f)
    out["F"] = F
    return out


def _unpack(P):
    p, o = [], 0
    for shape in ((N_H, N_IN), (N_H,), (N_H, N_H), (N_H,), (N_H,), (1,), (N_IN,), (N_IN,), (1,), (1,)):
        k = int(np.prod(shape))
        p.append(P[o:o + k].reshape(shape))
        o += k
    return p


def _forward(p, D):
    W1, b1, W2, b2, W3, b3, xm, xs, ym, ys = p
    h = torch.nn.functional.silu(((D - xm) / xs) @ W1.T + b1)
    return torch.nn.functional.silu(h @ W2.T + b2) @ W3 + b3


def _train(case, seed):
    D_h, T_h = _rows(case, seed)
    D, T = _dev(D_h), _dev(T_h)
    n, size = case["rows"], case["batch"]
    p = [t.clone() for t in _unpack(_dev(_network(seed)))]
    p[6], p[7] = D.mean(0), D.std(0, unbiased=False)
    p[8], p[9] = T.mean().reshape(1), T.std(unbiased=False).reshape(1)
    x, y = D, (T - p[8]) / p[9]
    m1, m2, t, ctr, last = [0.0] * 6, [0.0] * 6, 0, 0, 0.0
    for e in range(case["epochs"]):
        # Fisher-Yates with one Philox draw per exchange, as the binding's training shuffles its rows
        c = np.arange(ctr, ctr + n - 1, dtype=np.uint64)
        ctr += n - 1
        i = np.arange(n - 1, 0, -1)
        at = _philox(c, e, 0, 0x53485546, seed, 0x5352424500000004)[0] % (i + 1).astype(np.uint64)
        perm = list(range(n))
        for a, b in zip(i.tolist(), at.tolist()):
            perm[a], perm[b] = perm[b], perm[a]
        perm, tot = torch.tensor(perm, device="cuda"), 0.0
        for b0 in range(0, n, size):
            rows = perm[b0:b0 + size]
            w = [q.detach().requires_grad_(True) for q in p[:6]]
            loss = ((_forward(w + p[6:], x[rows]) - y[rows]) ** 2).mean()
            g = torch.autograd.grad(loss, w)
            tot += float(loss.detach()) * len(rows)
            t += 1
            for k in range(6):
                m1[k] = 0.9 * m1[k] + 0.1 * g[k]
                m2[k] = 0.999 * m2[k] + 0.001 * g[k] ** 2
                p[k] = p[k] - case["lr"] * ((m1[k] / (1 - 0.9 ** t)) / (torch.sqrt(m2[k] / (1 - 0.999 ** t)) + 1e-8)
                                            + 1e-4 * p[k])
        last = tot / n
    return {"params": torch.cat([q.reshape(-1) for q in p]), "loss": last}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train(case, seed)
    if kind == "predict":
        p = _unpack(_dev(_network(seed)))
        return {"y": _forward(p, _dev(_rows(case, seed)[0])) * p[9] + p[8]}
    if kind in ("md", "batch"):
        return None          # a trajectory: many evaluations after a relaxation
    out = _evaluate(case, seed, kind != "charges")
    return {k: out[k] for k in (("Q", "v") if kind == "charges" else ("F", "Q"))}
