"""What is timed: the periodic FMM's public calls over the range of systems they are used on.

Every case is one call that a simulation program makes per step (or per batch of frames), on a box of
ions in rigid three-site water or of random charges, through FMMPlan, FMMBatch or FmmEnergy:

  kind "step"   FMMPlan.evaluate: energy terms, forces and/or the solute-solvent energy
  kind "host"   the same with NumPy arrays in host memory (the copies are part of the call)
  kind "grad"   FmmEnergy forward and backward, the model's positions and charges in FP32
  kind "batch"  FMMBatch.lambda_energies on boxes of uneven size (coupling windows, trajectory frames)

The mixed path computes its fields in FP32 and only reduces in FP64; programs that run it keep FP32
force arrays, so its forces come back as FP32.  FP64 plans return FP64 forces.  The solute-solvent energy
and its parts, which cancel in it, come back as one FP32 row, as a program logs them per step.
"""
import math

import numpy as np
import torch

from paper_2003_13218_gb300.fmm import FmmEnergy, FMMBatch, FMMPlan

DENSITY = 0.0334  # water molecules per cubic Angstrom
Q_O, Q_H, R_OH, HOH = -0.834, 0.417, 0.9572, math.radians(104.52)


def listed():
    return [
        # a small cell of point charges in the default (FP64) precision: Madelung-type checks, unit tests of a force field
        dict(name="charges_700_fp64", kind="step", system="charges", n=700, depth=3, p=8, precision="fp64", ws=1, forces=False, solute=0, boundary="conducting"),
        # one Mg2+ in 999 waters, the small end of the ion-in-water boxes, with everything asked for, in both precisions
        dict(name="mg_3k", kind="step", system="water", n=999, depth=3, p=8, precision="mixed", ws=1, forces=True, solute=1, boundary="conducting"),
        dict(name="mg_3k_fp64", kind="step", system="water", n=999, depth=3, p=8, precision="fp64", ws=1, forces=True, solute=1, boundary="conducting"),
        # a polarisable or learned-charge model: energy with gradients for positions and charges
        dict(name="grad_12k", kind="grad", system="water", n=4001, depth=4, p=10, precision="mixed", ws=1, boundary="conducting"),
        # an MD step of the 100,000-charge box (energy and forces), and the same from a program whose arrays live on the host
        dict(name="cl_100k", kind="step", system="water", n=33333, depth=5, p=12, precision="mixed", ws=1, forces=True, solute=0, boundary="conducting"),
        dict(name="cl_100k_host", kind="host", system="water", n=33333, depth=5, p=12, precision="mixed", ws=1, forces=True, solute=1, boundary="conducting"),
        # the FP64 reference evaluation of that box, which a user takes to validate a mixed-precision run
        dict(name="cl_100k_fp64", kind="step", system="water", n=33333, depth=5, p=12, precision="fp64", ws=1, forces=True, solute=1, boundary="conducting"),
        # second-nearest-neighbour near field at a lower order, the paper's own setting
        dict(name="ws2_100k", kind="step", system="water", n=33333, depth=5, p=8, precision="mixed", ws=2, forces=True, solute=1, boundary="conducting"),
        # a molecular solute of 210 charges in a box of ragged size: forces and solute-solvent energy, vacuum boundary
        dict(name="solute_210_61k", kind="step", system="water", n=20411, depth=4, p=10, precision="mixed", ws=1, forces=True, solute=210, boundary="vacuum"),
        # sixteen coupling windows of uneven size, evaluated together
        dict(name="windows_16", kind="batch", boxes=16, n_lo=3400, n_hi=40000, p=12, precision="mixed"),
        # the one-million-charge box with everything asked for, and the largest one: ten million charges, energy and forces
        dict(name="na_1m", kind="step", system="water", n=333333, depth=6, p=12, precision="mixed", ws=1, forces=True, solute=1, boundary="conducting"),
        dict(name="mg_10m", kind="step", system="water", n=3333333, depth=7, p=10, precision="mixed", ws=1, forces=True, solute=0, boundary="conducting"),
    ]


def depth_for(n, rng, shallow=True):
    """The depth that gives about four charges a leaf, or one level less (denser leaves, fewer levels)."""
    d = round(math.log(max(n / 3.8, 1.0), 8))
    if shallow and rng.random() < 0.4:
        d -= 1
    return max(2, min(7, d))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "fp64", "fp64", "ws2", "host", "grad", "batch"])

    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    c = dict(kind=kind, system="water", precision="mixed", ws=1, boundary=rng.choice(["conducting", "conducting", "vacuum"]))
    if kind == "batch":
        lo = size(1200, 9000)
        return dict(kind="batch", boxes=rng.randint(3, 20), n_lo=lo, n_hi=min(lo * rng.randint(2, 9), 45000), p=rng.choice([8, 10, 12]), precision="mixed")
    if kind == "fp64":
        c.update(kind="step", precision="fp64", n=size(80, 28000), p=rng.choice([5, 6, 8, 10, 12]), system=rng.choice(["water", "water", "charges"]))
    elif kind == "ws2":
        c.update(kind="step", ws=2, n=size(1500, 33000), p=rng.choice([6, 8]))
    elif kind == "host":
        c.update(n=size(300, 60000), p=rng.choice([6, 8, 10, 12]))
    elif kind == "grad":
        c.update(n=size(150, 60000), p=rng.choice([6, 8, 10, 12]))
    else:
        c.update(n=size(120, 700000), p=rng.choice([4, 6, 7, 8, 10, 11, 12]))
    atoms = c["n"] if c["system"] == "charges" else 3 * c["n"] + 1
    c["depth"] = depth_for(atoms, rng)
    if c["precision"] == "fp64":
        c["depth"] = min(c["depth"], 5 if c["p"] <= 10 else 4)
    if c["ws"] == 2:
        c["depth"] = min(5, max(3, c["depth"]))
    if c["kind"] != "grad":
        c["forces"] = rng.random() < 0.6
        c["solute"] = rng.choice([0, 1, 1, rng.randint(2, 64), rng.randint(65, 400)]) if atoms > 2000 else rng.choice([0, 1])
        if not c["forces"] and c["solute"] == 0:
            c["forces"] = True
    return c


# ---------------------------------------------------------------- inputs
def device():
    return torch.device("cuda")


def water_box(n_waters, solute, seed):
    """One ion at the centre and n_waters rigid waters on jittered lattice sites in random orientations.  The
    solute is the ion and, with solute > 1, the atoms nearest to it, one whole molecule after another."""
    dev = device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def u(*shape):
        return torch.rand(*shape, generator=g, device=dev, dtype=torch.float64)

    box = (n_waters / DENSITY) ** (1.0 / 3.0)
    n = 1
    while n ** 3 < n_waters + 1:
        n += 1
    centre = n // 2
    mid = centre + n * (centre + n * centre)
    site = torch.randperm(n ** 3 - 1, generator=g, device=dev)[:n_waters]
    site = site + (site >= mid)
    off = 0.5 * (n % 2)
    grid = torch.stack([site % n, (site // n) % n, site // (n * n)], dim=1).double()
    o = (grid + off) * (box / n) + (u(n_waters, 3) * 2.0 - 1.0) * 0.3
    a = u(3, n_waters)
    r1, r2 = torch.sqrt(1.0 - a[0]), torch.sqrt(a[0])
    w, x = r1 * torch.sin(2 * math.pi * a[1]), r1 * torch.cos(2 * math.pi * a[1])
    y, z = r2 * torch.sin(2 * math.pi * a[2]), r2 * torch.cos(2 * math.pi * a[2])
    e1 = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)], dim=1)
    e3 = torch.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], dim=1)
    s, c = R_OH * math.sin(HOH / 2), R_OH * math.cos(HOH / 2)
    mol = torch.stack([o, o + s * e1 + c * e3, o - s * e1 + c * e3], dim=1)
    pos = torch.empty(1 + 3 * n_waters, 3, dtype=torch.float64, device=dev)
    pos[0] = (centre + off) * (box / n)
    q = torch.empty(1 + 3 * n_waters, dtype=torch.float64, device=dev)
    q[0] = float(2 - seed % 2)  # Mg2+ or Na+
    sol = torch.zeros(1 + 3 * n_waters, dtype=torch.uint8, device=dev)
    if solute > 1:
        mol = mol[torch.argsort(((mol[:, 0] - pos[0]) ** 2).sum(1), stable=True)]
    pos[1:] = mol.reshape(-1, 3)
    q[1::3], q[2::3], q[3::3] = Q_O, Q_H, Q_H
    sol[:max(solute, 1)] = 1
    pos = pos - box * torch.floor(pos / box)
    return box, pos.contiguous(), q, sol


def charge_box(n, seed):
    """Uniform random charges at a density of 0.1 per cubic Angstrom."""
    dev = device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    box = (n / 0.1) ** (1.0 / 3.0)
    pos = torch.rand(n, 3, generator=g, device=dev, dtype=torch.float64) * box
    q = torch.rand(n, generator=g, device=dev, dtype=torch.float64) * 2.0 - 1.0
    sol = torch.zeros(n, dtype=torch.uint8, device=dev)
    sol[0] = 1
    return box, pos, q, sol


def system(case, seed):
    if case["system"] == "charges":
        return charge_box(case["n"], seed)
    return water_box(case["n"], case.get("solute", 1), seed)


def window_sizes(case):
    """Molecules per box: spread evenly between n_lo and n_hi in a mixed order, no two alike."""
    k = case["boxes"]
    step = (case["n_hi"] - case["n_lo"]) / max(k - 1, 1)
    return [case["n_lo"] + int(step * ((7 * i) % k if k % 7 else i)) for i in range(k)]


def window_depth(n_waters):
    """The shallower tree that suits many boxes at once: 6 to 50 charges a leaf."""
    return 3 if 3 * n_waters < 25000 else 4


def prepare(case, seed):
    if case["kind"] == "batch":
        sizes = window_sizes(case)
        parts = [water_box(n, 1, 1000 * (seed % 1000003) + i) for i, n in enumerate(sizes)]
        batch = FMMBatch([b for b, _, _, _ in parts], [q.numel() for _, _, q, _ in parts], [window_depth(n) for n in sizes],
                         [case["p"]] * len(sizes), precision=case["precision"])
        lam = np.arange(len(sizes)) % 16 / 15.0
        return dict(case=case, batch=batch, pos=[p for _, p, _, _ in parts], q=[q for _, _, q, _ in parts],
                    sol=[s for _, _, _, s in parts], lam=lam)
    box, pos, q, sol = system(case, seed)
    plan = FMMPlan(box, q.numel(), case["depth"], case["p"], precision=case["precision"], ws=case["ws"],
                   boundary=case["boundary"])
    s = dict(case=case, box=box, plan=plan)
    if case["kind"] == "grad":
        s.update(pos=pos.float().requires_grad_(True), q=q.float().requires_grad_(True))
        return s
    s.update(pos=pos, q=q, sol=sol if case["solute"] else None, forces=torch.empty_like(pos) if case["forces"] else None)
    if case["kind"] == "host":
        for k in ("pos", "q", "sol", "forces"):
            s[k] = None if s[k] is None else s[k].cpu().numpy()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "batch":
        out = s["batch"].lambda_energies(s["pos"], s["q"], s["sol"], s["lam"])
        return {k: v.astype(np.float32) for k, v in out.items()}
    if case["kind"] == "grad":
        s["pos"].grad = s["q"].grad = None
        e = FmmEnergy.apply(s["pos"].double(), s["q"].double(), s["plan"])
        e.backward()
        return {"energy": e.detach().float(), "dpos": s["pos"].grad, "dq": s["q"].grad}
    terms, uv = s["plan"].evaluate(s["pos"], s["q"], s["sol"], forces=s["forces"])
    out = {"terms": terms}
    if uv is not None:
        out["uv"] = np.array([uv[k] for k in ("e_uv", "W", "A", "B", "C", "nf_uv", "bc_cross")], dtype=np.float32)
    f = s["forces"]
    if f is not None and case["precision"] == "mixed":
        f = f.astype(np.float32) if case["kind"] == "host" else f.float()
    if f is not None:
        out["forces"] = f
    return out


# ---------------------------------------------------------------- work
def n_il(ws):
    return (4 * ws + 2) ** 3 - (2 * ws + 1) ** 3


def fmm_work(n, depth, p, ws, forces, solute):
    """Arithmetic of the method at its order: dense M2L and L2L per cell, M2M, P2M and L2P (with the gradient),
    and the near-field pairs at the mean leaf occupancy; inputs read once, results written once."""
    c = (p + 1) ** 2
    cells = sum(8 ** l for l in range(1, depth + 1))
    flops = 2.0 * c * c * (n_il(ws) + 2) * cells
    flops += n * c * (10 + (30 if forces else 10))
    flops += 20.0 * n * (n / 8.0 ** depth) * (2 * ws + 1) ** 3
    nbytes = 32.0 * n + (24.0 * n if forces else 0) + (n if solute else 0)
    return {"bytes": nbytes + 200, "flops": flops}


def work(case):
    if case["kind"] == "batch":
        parts = [fmm_work(3 * n + 1, window_depth(n), case["p"], 1, False, 1) for n in window_sizes(case)]
        return {k: sum(x[k] for x in parts) for k in ("bytes", "flops")}
    n = case["n"] if case["system"] == "charges" else 3 * case["n"] + 1
    if case["kind"] == "grad":
        w = fmm_work(n, case["depth"], case["p"], case["ws"], True, 0)
        return {"bytes": 16.0 * n + 16.0 * n + 4, "flops": w["flops"]}
    w = fmm_work(n, case["depth"], case["p"], case["ws"], case["forces"], case["solute"])
    if case["precision"] == "mixed" and case["forces"]:
        w["bytes"] -= 12.0 * n  # FP32 forces
    return w


# ---------------------------------------------------------------- the definition in 64 bits
A_EWALD = 12.0  # splitting parameter times the box: erfc(6) < 3e-17 at half a box
K_EWALD = 24    # reciprocal vectors |n_i| <= 24: exp(-(24 pi / 12)^2) < 1e-17
N_EXACT = 130000


def structure(pos, q, box):
    """sum_j q_j e^{i k r_j} on the grid n_x, n_y in [-K, K], n_z in [0, K], and the three phase tables."""
    kx = torch.arange(-K_EWALD, K_EWALD + 1, device=pos.device, dtype=torch.float64) * (2 * math.pi / box)
    e = [torch.polar(torch.ones(1, 1, device=pos.device, dtype=torch.float64), kx[:, None] * pos[None, :, a]) for a in range(3)]
    return torch.stack([(e[0] * (q * e[2][K_EWALD + z])) @ e[1].T for z in range(K_EWALD + 1)], dim=2), e


def weights(box, dev):
    n = torch.arange(-K_EWALD, K_EWALD + 1, device=dev, dtype=torch.float64)
    n2 = n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, K_EWALD:] ** 2
    k2 = n2 * (2 * math.pi / box) ** 2
    w = torch.where(n2 > 0, 4 * math.pi / box ** 3 * torch.exp(-k2 * (box / A_EWALD) ** 2 / 4) / k2.clamp(min=1e-300), 0.0)
    w[:, :, 1:] *= 2  # the half space n_z < 0
    return w, n * (2 * math.pi / box)


def real_space(pos, q, box, targets, want_field):
    """sum_j q_j erfc(a r)/r over the nearest images (and the field) at pos[targets]; the target itself left out."""
    a = A_EWALD / box
    phi = torch.zeros(targets.numel(), dtype=torch.float64, device=pos.device)
    fld = torch.zeros(targets.numel(), 3, dtype=torch.float64, device=pos.device) if want_field else None
    step = max(1, 40_000_000 // q.numel())
    for b in range(0, targets.numel(), step):
        t = targets[b:b + step]
        d = pos[t][:, None, :] - pos[None, :, :]
        d -= box * torch.round(d / box)
        r2 = (d * d).sum(2)
        r2[torch.arange(t.numel(), device=t.device), t] = math.inf
        ir = torch.rsqrt(r2)
        r = torch.where(torch.isinf(r2), 1.0, r2 * ir)
        v = torch.special.erfc(a * r) * ir
        phi[b:b + step] = v @ q
        if want_field:
            f = (v + 2 * a / math.sqrt(math.pi) * torch.exp(-(a * r) ** 2) * (ir > 0)) * ir * ir
            fld[b:b + step] = torch.einsum("ij,j,ijk->ik", f, q, d)
    return phi, fld


def ewald_exact(box, pos, q, want_field, want_phi, vacuum):
    """The Ewald sum of the point charges and their uniform neutralising background (conducting boundary): phi_i =
    dE/dq_i, E = 1/2 sum q phi, forces; with the vacuum boundary the dipole surface term is added on wrapped coordinates."""
    a = A_EWALD / box
    phi, fld = real_space(pos, q, box, torch.arange(q.numel(), device=pos.device), want_field)
    s, e = structure(pos, q, box)
    w, k = weights(box, pos.device)
    ws = w * s.conj()
    rec = torch.zeros_like(phi)
    grad = torch.zeros_like(pos) if want_field else None
    for z in range(K_EWALD + 1):
        t = (ws[:, :, z].T @ e[0])  # [ny, N]
        x = (t * e[1]).sum(0) * e[2][K_EWALD + z]
        rec += x.real
        if want_field:
            tx = ((ws[:, :, z] * k[:, None]).T @ e[0] * e[1]).sum(0) * e[2][K_EWALD + z]
            ty = (t * e[1] * k[:, None]).sum(0) * e[2][K_EWALD + z]
            grad[:, 0] -= tx.imag
            grad[:, 1] -= ty.imag
            grad[:, 2] -= (x * k[K_EWALD + z]).imag
    total = q.sum()
    phi = phi + rec - 2 * a / math.sqrt(math.pi) * q - math.pi * total / (box ** 3 * a * a)
    field = fld - grad if want_field else None
    if vacuum:
        c = 4 * math.pi / (3 * box ** 3)
        mu = (q[:, None] * pos).sum(0)
        phi = phi + c * (pos @ mu)
        if want_field:
            field = field - c * mu
    return 0.5 * (q * phi).sum(), phi if want_phi else None, q[:, None] * field if want_field else None


def exact(case, seed):
    if case["kind"] == "batch":
        sizes = window_sizes(case)
        if sum((3 * n + 1) ** 2 for n in sizes) > 2e10:
            return None
        keys = ("e_total", "e_uv", "v_lambda", "dv_dlambda")
        out = {k: np.zeros(len(sizes)) for k in keys}
        for i, n in enumerate(sizes):
            box, pos, q, sol = water_box(n, 1, 1000 * (seed % 1000003) + i)
            e = float(ewald_exact(box, pos, q, False, False, False)[0])
            uv = float(solute_exact(box, pos, q, sol, False))
            lam = i % 16 / 15.0
            for k, v in zip(keys, (e, uv, e - lam * uv, -uv)):
                out[k][i] = v
        return out
    n = case["n"] if case["system"] == "charges" else 3 * case["n"] + 1
    if n > N_EXACT:
        return None
    box, pos, q, sol = system(case, seed)
    vacuum = case["boundary"] == "vacuum"
    if case["kind"] == "grad":
        pos, q = pos.float().double(), q.float().double()
        e, phi, f = ewald_exact(box, wrapped(pos, box), q, True, True, vacuum)
        return {"energy": e, "dpos": -f, "dq": phi}
    e, _, f = ewald_exact(box, pos, q, case["forces"], False, vacuum)
    volume, total = box ** 3, float(q.sum())
    mu = (q[:, None] * pos).sum(0)
    kappa = 2.0 / box
    terms = {"near": None, "far": None, "charged": -math.pi * total ** 2 / (2 * volume * kappa ** 2),
             "quad_surface": 2 * math.pi / (3 * volume) * total * float((q * (pos * pos).sum(1)).sum()),
             "dipole_surface": 0.0 if vacuum else -2 * math.pi / (3 * volume) * float(mu @ mu), "total": float(e)}
    out = {"terms": terms}
    if case["solute"]:
        out["uv"] = None  # its parts belong to this method's decomposition
    if f is not None:
        out["forces"] = f.cpu().numpy() if case["kind"] == "host" else f
    return out


def wrapped(pos, box):
    return pos - box * torch.floor(pos / box)


def solute_exact(box, pos, q, sol, vacuum):
    """E(u + v) - E(u) - E(v): the solute charges and their background in the field of the solvent's."""
    a = A_EWALD / box
    u = torch.nonzero(sol).flatten()
    qu, qv = torch.where(sol == 1, q, 0.0), torch.where(sol == 1, 0.0, q)
    phi, _ = real_space(pos, qv, box, u, False)
    w, _ = weights(box, pos.device)
    su, sv = structure(pos, qu, box)[0], structure(pos, qv, box)[0]
    e = (q[u] * phi).sum() + (w * (su * sv.conj()).real).sum() - math.pi * qu.sum() * qv.sum() / (box ** 3 * a * a)
    if vacuum:
        e = e + 4 * math.pi / (3 * box ** 3) * ((qu[:, None] * pos).sum(0) @ (qv[:, None] * pos).sum(0))
    return e
