"""The workloads this library is measured on, through its public Python API.

Four kinds of call cover what a user has the library do:

  efv      energies, forces and virials of one configuration (NEP.compute, or
           compute_efv_static, the form without device allocations)
  md       a block of molecular-dynamics steps from a stored snapshot (MD.step)
  snes     the population losses of a training set (Dataset.evaluate), or a
           block of training generations (SNES.run)
  grad     the force loss of a training set and its gradient (force_loss)

Inputs are the shapes of `inputs.py`: diamond cells of a Si-like crystal with
Gaussian displacements and optional vacancies, PbTe-like rocksalt cells with
two species, and training sets of small cells of uneven size and density.
`exact` is the method of the paper in plain FP64 torch: pair list by cells,
the angular sums of Eq. 13 through the moment tensors of the unit vectors
(P_l(u.v) is a polynomial in u.v, and (u.v)^k contracts two rank-k moments),
forces by automatic differentiation with respect to the pair vectors.
"""
import itertools
import math

import numpy as np
import torch

from paper_2107_08119_gb300 import nep
from paper_2107_08119_gb300.inputs import A_PBTE, A_SI, AMU_A2_FS2_EV, KB_EV, MASS_PBTE, MASS_SI, PBTE_HYPER, Z_PB, Z_TE

HYPER = {"si": nep.Hyper(), "pbte": nep.Hyper(**PBTE_HYPER)}
MASS = {"si": MASS_SI, "pbte": MASS_PBTE}
SITES = {
    "si": ([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0],
            [.25, .25, .25], [.25, .75, .75], [.75, .25, .75], [.75, .75, .25]], A_SI),
    "pbte": ([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0],
              [.5, 0, 0], [.5, .5, .5], [0, 0, .5], [0, .5, 0]], A_PBTE),
}
DRIVE = (2e-3, -1e-3, 5e-4)  # HNEMD driving force (1/A)
TARGET_K, COUPLING_FS = 300.0, 100.0


def _efv(name, model, n1, n2, n3, vacancy=0.0, static=False, sync=False):
    return dict(name=name, kind="efv", model=model, n1=n1, n2=n2, n3=n3, vacancy=vacancy, static=static, sync=sync)


def _md(name, model, n1, n2, n3, steps, vacancy=0.0, heat=True, drive=False):
    return dict(name=name, kind="md", model=model, n1=n1, n2=n2, n3=n3, steps=steps, vacancy=vacancy, heat=heat,
                drive=drive)


def _snes(name, structures, population, precision, generations):
    return dict(name=name, kind="snes", structures=structures, population=population, precision=precision,
                generations=generations)


def listed():
    return [
        # one training cell, labelled or checked by itself: the smallest call,
        # its box too small for a cell grid (all pairs and images); the caller
        # waits for the answer
        _efv("efv_cell_96", "si", 2, 2, 3, sync=True),
        # the 512-atom single-configuration call of the benchmark, waited for
        _efv("efv_si_512", "si", 4, 4, 4, sync=True),
        # an allocator-free host program's call, uneven box with vacancies
        _efv("efv_static_1800", "si", 6, 6, 7, vacancy=0.1, static=True),
        # one configuration of the MD headline's size, in a host program's stream
        _efv("efv_si_125k", "si", 25, 25, 25),
        # two species with split cutoffs and 41 descriptors, uneven box
        _efv("efv_pbte_64k", "pbte", 20, 19, 21),
        # a small production run (the paper's benchmark has about this many atoms)
        _md("md_si_4k", "si", 8, 8, 8, 50, heat=False),
        # the MD headline
        _md("md_si_125k", "si", 25, 25, 25, 20),
        # heat transport in a large box with vacancies, J every step
        _md("md_vacancy_922k", "si", 40, 40, 80, 5, vacancy=0.1),
        # driven (HNEMD) and thermostatted run for a conductivity
        _md("md_hnemd_14k", "si", 12, 12, 12, 20, drive=True),
        # losses of one population in full precision (validation, restarts)
        _snes("snes_fp32_eval", 200, 50, "fp32", 0),
        # a block of training generations, tensor-core precision
        _snes("snes_bf16_20gen", 200, 50, "bf16", 20),
        # gradient-based refinement: one loss and its gradient
        dict(name="force_loss_grad", kind="grad", structures=200),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(rng, lo, hi, least):
    """Cells per direction of a box of about lo..hi atoms, each at least `least`."""
    edge = (math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8.0) ** (1.0 / 3.0)
    return [max(least, int(round(edge * rng.uniform(0.75, 1.3)))) for _ in range(3)]


def draw(rng):
    kind = rng.choice(["efv", "efv", "efv", "md", "md", "snes", "grad"])
    vacancy = rng.choice([0.0, round(rng.uniform(0.02, 0.1), 3)])
    if kind == "efv":
        form = rng.choice(["static", "si", "si", "pbte"])
        if form == "static":
            return _unnamed(_efv("", "si", *_cells(rng, 216, 2000, 2), vacancy=vacancy, static=True))
        cells = _cells(rng, 64, 250_000, 2) if form == "si" else _cells(rng, 512, 64_000, 3)
        return _unnamed(_efv("", form, *cells, vacancy=vacancy, sync=math.prod(cells) < 500))
    if kind == "md":
        form = rng.choice(["si", "si", "pbte"])
        cells = _cells(rng, 512, 250_000 if form == "si" else 64_000, 3 if form == "si" else 4)
        return _unnamed(_md("", form, *cells, max(5, min(50, 1_500_000 // (8 * math.prod(cells)))), vacancy=vacancy,
                            heat=rng.random() < 0.7, drive=rng.random() < 0.3))
    structures = _log_int(rng, 10, 200)
    if kind == "grad":
        return dict(kind="grad", structures=structures)
    return _unnamed(_snes("", structures, rng.randint(10, 64), rng.choice(["fp32", "bf16"]), rng.choice([0, 5, 20])))


def _unnamed(case):
    del case["name"]
    return case


# ------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed, device):
    return torch.Generator(device=device).manual_seed(1_000_003 * seed + 17)


def _weights(model, seed):
    """U(-1/2, 1/2); for the weighted two-species descriptors the input
    columns are scaled to their size, as a trained potential's are."""
    h = HYPER[model]
    z = np.random.default_rng([seed, 1]).uniform(-0.5, 0.5, h.n_par)
    if model == "pbte":
        zbar = math.sqrt(Z_PB * Z_TE)
        w1 = z[:h.n_neu * h.n_des].reshape(h.n_neu, h.n_des)
        w1[:, :h.n_max_R + 1] /= zbar
        w1[:, h.n_max_R + 1:] /= zbar ** 2
    return z.astype(np.float32)


def _configuration(case, seed):
    """Positions (3, n) FP64 in A, box lengths, species numbers or None."""
    dev = _device()
    gen = _generator(seed, dev)
    basis, a = SITES[case["model"]]
    cells = [case["n1"], case["n2"], case["n3"]]
    grid = torch.cartesian_prod(*[torch.arange(c, dtype=torch.float64, device=dev) for c in cells]).reshape(-1, 3)
    pos = ((grid[:, None, :] + torch.tensor(basis, dtype=torch.float64, device=dev)) * a).reshape(-1, 3)
    species = torch.tensor([Z_PB] * 4 + [Z_TE] * 4, dtype=torch.float64, device=dev).repeat(len(grid))
    sigma = 0.15 if case["vacancy"] else 0.1
    n_keep = len(pos) - int(round(case["vacancy"] * len(pos)))
    keep = torch.randperm(len(pos), generator=gen, device=dev)[:n_keep].sort().values
    pos, species = pos[keep], species[keep]
    pos = pos + sigma * torch.randn(pos.shape, generator=gen, dtype=torch.float64, device=dev)
    return pos.T.contiguous(), np.array([c * a for c in cells]), species if case["model"] == "pbte" else None


def _velocities(n, mass, seed):
    dev = _device()
    v = torch.randn(3, n, generator=_generator(seed + 1, dev), dtype=torch.float64, device=dev)
    v = (v - v.mean(dim=1, keepdim=True)) * math.sqrt(KB_EV * 300.0 / (mass * AMU_A2_FS2_EV))
    return v.contiguous()


def _training_set(n_struct, seed):
    """Cells of 32 to 256 atoms, density +-10 %, displacements 0.1 to 0.3 A,
    labels of the size of DFT energies, forces and virials."""
    rng = np.random.default_rng([seed, 2])
    shapes = [s for s in itertools.product(range(1, 5), repeat=3) if 4 <= math.prod(s) <= 32]
    basis = np.array(SITES["si"][0])
    structures = []
    for _ in range(n_struct):
        cells = np.array(shapes[rng.integers(len(shapes))])
        a = A_SI * (1.0 + rng.uniform(-0.1, 0.1)) ** (-1.0 / 3.0)
        grid = np.stack(np.meshgrid(*[np.arange(c) for c in cells], indexing="ij"), -1).reshape(-1, 1, 3)
        pos = ((grid + basis) * a).reshape(-1, 3)
        structures.append({"pos": pos + rng.normal(0.0, rng.uniform(0.1, 0.3), pos.shape), "box": np.diag(cells * a)})
    count = np.array([len(s["pos"]) for s in structures])
    e = count * rng.normal(-3.0, 0.1, n_struct)
    f = rng.normal(0.0, 1.0, (count.sum(), 3))
    w = count[:, None] * rng.normal(0.0, 0.5, (n_struct, 6))
    return structures, e, f, w


def _population(n_pop, seed):
    return np.random.default_rng([seed, 3]).normal(0.0, 0.1, (n_pop, HYPER["si"].n_par)).astype(np.float32)


PRECISION = {"fp32": nep.PREC_FP32, "bf16": nep.PREC_BF16}


def prepare(case, seed):
    dev = _device()
    s = {"case": case}
    if case["kind"] in ("efv", "md"):
        pos, box, species = _configuration(case, seed)
        s.update(pos=pos, box=np.diag(box))
        z = _weights(case["model"], seed)
        if case.get("static"):
            s["z"] = torch.tensor(z, device=dev)
            return s
        s["model"] = nep.NEP(z, HYPER[case["model"]])
        if species is not None:
            s["model"].set_species(species.cpu().numpy())
        if case["kind"] == "md":
            n, steps = pos.shape[1], case["steps"]
            s["md"] = nep.MD(s["model"], n, s["box"], MASS[case["model"]])
            if case["drive"]:
                s["md"].set_hnemd(DRIVE)
                s["md"].set_thermostat(TARGET_K, COUPLING_FS)
            s.update(pos0=pos, vel0=_velocities(n, MASS[case["model"]], seed), pos=pos.clone(), vel=torch.empty_like(pos),
                     thermo=torch.empty(steps, nep.THERMO_COLS, dtype=torch.float64, device=dev),
                     heat=torch.empty(steps, 3, dtype=torch.float64, device=dev) if case["heat"] else None)
        return s
    s["model"] = nep.NEP(_weights("si", seed))
    s["set"] = nep.Dataset(s["model"], *_training_set(case["structures"], seed))
    if case["kind"] == "grad":
        s["z"] = torch.tensor(_weights("si", seed + 1), device=dev, requires_grad=True)
        return s
    # the launch shape the library's tuner settles on for sets of these sizes
    # (given here, so that every measurement runs the same one)
    tensor = int(case["precision"] == "bf16")
    s["set"].set_shape(fused=0, discard=1, recv_unroll=1, mlp_threads=256 if tensor else 128, owner_tc=tensor,
                       pop_pipe=tensor)
    if case["generations"]:
        n_par = HYPER["si"].n_par
        mean = np.random.default_rng([seed, 4]).uniform(-0.5, 0.5, n_par)
        s["snes"] = nep.SNES(s["model"], case["population"], mean, np.full(n_par, 0.1), seed)
    else:
        s["z"] = torch.tensor(_population(case["population"], seed), device=dev)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "efv":
        if case["static"]:
            return nep.compute_efv_static(s["z"], s["pos"], s["box"])
        return s["model"].compute(s["pos"], s["box"], sync=case["sync"])
    if case["kind"] == "md":
        # the snapshot is restored, as at a restart, and the block of steps run
        s["pos"].copy_(s["pos0"])
        s["vel"].copy_(s["vel0"])
        s["md"].invalidate()
        s["md"].step(s["pos"], s["vel"], case["steps"], 1.0, s["thermo"], s["heat"])
        out = {"pos": s["pos"], "vel": s["vel"], "thermo": s["thermo"]}
        return dict(out, heat=s["heat"]) if case["heat"] else out
    if case["kind"] == "grad":
        s["z"].grad = None
        loss = nep.force_loss(s["z"], s["set"])
        loss.backward()
        return {"loss": loss, "grad": s["z"].grad}
    if case["generations"]:
        history = s["snes"].run(s["set"], case["generations"], PRECISION[case["precision"]], history=True)
        mean, sigma, _, order = s["snes"].state()
        return {"loss": history, "mean": mean, "sigma": sigma, "order": order}
    return s["set"].evaluate(s["z"], PRECISION[case["precision"]])


# --------------------------------------------------------------------- work
def _site_flops(model, n, volume):
    """Per atom: 134 per radial pair, 250 x orders per angular pair, the
    network and its input gradient; pairs from the mean density."""
    h = HYPER[model]
    ball = 4.0 / 3.0 * math.pi * n / volume
    return n * ((50.0 + 10.5 * (h.n_max_R + 1)) * ball * h.rc_R ** 3 + 250.0 * (h.n_max_A + 1) * ball * h.rc_A ** 3
                + 4.0 * h.n_neu * h.n_des + 10.0 * h.n_neu)


def work(case):
    if case["kind"] in ("efv", "md"):
        a = SITES[case["model"]][1]
        cells = case["n1"] * case["n2"] * case["n3"]
        n = 8 * cells - int(round(case["vacancy"] * 8 * cells))
        one = _site_flops(case["model"], n, cells * a ** 3)
        if case["kind"] == "efv":  # FP64 positions in; FP64 energies, FP32 forces and virials out
            return {"bytes": n * (24.0 + 8 + 12 + 36), "flops": one}
        return {"bytes": n * 96.0 * case["steps"], "flops": one * case["steps"]}
    # a training set's mean cell has about 13 lattice cells
    n = 104.0 * case["structures"]
    pairs, angular = 27.7 * n, 12.7 * n
    members = 1 if case["kind"] == "grad" else case["population"]
    set_bytes = n * (32 * 4 + 96 * 4 + 12) + pairs * 48.0 + angular * 288.0
    flops = members * (4.0 * 32 * 30 * n + 31.0 * pairs + 144.0 * angular + 192.0 * n)
    if case["kind"] == "grad":  # positions and labels in, loss and gradient out; forward and backward site passes
        return {"bytes": n * 36.0 + HYPER["si"].n_par * 8.0, "flops": 3.0 * 29_700.0 * n}
    per = {"bytes": set_bytes, "flops": flops}
    return {k: v * max(1, case["generations"]) for k, v in per.items()}


# -------------------------------------------------------------------- exact
def _pairs(pos, box, rc):
    """i, j and r_j + shift - r_i of every pair within rc, all images.
    pos (n, 3) FP64, box (3,) lengths."""
    dev, n = pos.device, len(pos)
    L = torch.tensor(box, dtype=torch.float64, device=dev)
    x = pos - L * torch.floor(pos / L)
    nc = np.maximum(1, np.floor(box / rc).astype(int))
    reach = np.ceil(rc / (box / nc) - 1e-12).astype(int)
    nct = torch.tensor(nc, device=dev)
    c = torch.minimum((x / L * nct).long(), nct - 1)
    cid = (c[:, 0] * int(nc[1]) + c[:, 1]) * int(nc[2]) + c[:, 2]
    order = torch.argsort(cid, stable=True)
    count = torch.bincount(cid, minlength=int(nc.prod()))
    start = torch.cumsum(count, 0) - count
    table = torch.full((int(nc.prod()), int(count.max())), -1, device=dev)
    table[cid[order], torch.arange(n, device=dev) - start[cid[order]]] = order
    xp = torch.cat([x, torch.full((1, 3), 1e9, dtype=torch.float64, device=dev)])  # row -1: an empty place
    cell = torch.cartesian_prod(*[torch.arange(int(m), device=dev) for m in nc]).reshape(-1, 3)
    out = []
    for o in itertools.product(*[range(-int(r), int(r) + 1) for r in reach]):
        to = cell + torch.tensor(o, device=dev)
        shift = torch.div(to, nct, rounding_mode="floor")
        to = to - shift * nct
        other = table[(to[:, 0] * int(nc[1]) + to[:, 1]) * int(nc[2]) + to[:, 2]]
        r = (xp[other] + (shift * L)[:, None, :])[:, None, :, :] - xp[table][:, :, None, :]
        d2 = (r * r).sum(-1)
        ok = (d2 < rc * rc) & (table[:, :, None] >= 0) & (other[:, None, :] >= 0) & (d2 > 0)
        at = ok.nonzero(as_tuple=True)
        out.append((table[at[0], at[1]], other[at[0], at[2]], r[at]))
    i, j, r = (torch.cat(v) for v in zip(*out))
    by = torch.argsort(i, stable=True)
    return i[by], j[by], r[by]


def _radial(d, rc, orders, weight):
    fc = 0.5 * (1.0 + torch.cos(math.pi * d / rc)) * weight
    x = 2.0 * (d / rc - 1.0) ** 2 - 1.0
    T = [torch.ones_like(x), x]
    while len(T) < orders:
        T.append(2.0 * x * T[-1] - T[-2])
    return [fc if n == 0 else 0.5 * (T[n] + 1.0) * fc for n in range(orders)]


# monomials x^a y^b z^c of degree 0..4, their degree and multinomial weight
_MONO = [(a, b, k - a - b) for k in range(5) for a in range(k, -1, -1) for b in range(k - a, -1, -1)]
_MULT = [math.factorial(sum(m)) / math.prod(math.factorial(v) for v in m) for m in _MONO]


def _descriptors(h, n, i, r, weight):
    """q (n, N_des) of the atoms i counts from 0."""
    d = r.norm(dim=1)
    near = (d < h.rc_R).nonzero()[:, 0]
    g = torch.stack(_radial(d[near], h.rc_R, h.n_max_R + 1, weight[near]), 1)
    q = [torch.zeros(n, h.n_max_R + 1, dtype=r.dtype, device=r.device).index_add(0, i[near], g)]
    near = (d < h.rc_A).nonzero()[:, 0]
    u = r[near] / d[near, None]
    power = [[torch.ones_like(u[:, c])] for c in range(3)]
    for c in range(3):
        for _ in range(4):
            power[c].append(power[c][-1] * u[:, c])
    mono = torch.stack([power[0][a] * power[1][b] * power[2][c] for a, b, c in _MONO], 1)
    degree = torch.tensor([sum(m) for m in _MONO], device=r.device)
    mult = torch.tensor(_MULT, dtype=r.dtype, device=r.device)
    for gn in _radial(d[near], h.rc_A, h.n_max_A + 1, weight[near]):
        S = torch.zeros(n, len(_MONO), dtype=r.dtype, device=r.device).index_add(0, i[near], gn[:, None] * mono)
        s = torch.zeros(n, 5, dtype=r.dtype, device=r.device).index_add(1, degree, mult * S * S)  # sum g g (u.v)^k
        q.append(torch.stack([s[:, 1], (3 * s[:, 2] - s[:, 0]) / 2, (5 * s[:, 3] - 3 * s[:, 1]) / 2,
                              (35 * s[:, 4] - 30 * s[:, 2] + 3 * s[:, 0]) / 8], 1))
    return torch.cat(q, 1)


def _split(h, z):
    m = h.n_neu * h.n_des
    return z[:m].reshape(h.n_neu, h.n_des), z[m:m + h.n_neu], z[m + h.n_neu:m + 2 * h.n_neu], z[-1]


def _network(h, z, q):
    w1, b1, w2, b2 = _split(h, z)
    return torch.tanh(q @ w1.T - b1) @ w2 - b2


def _weight(species, i, j):
    return torch.ones(len(i), dtype=torch.float64, device=i.device) if species is None else (species[i] * species[j]).sqrt()


def _exact_efv(h, z, pos, box, species):
    """U (n,), F (3, n), W (9, n) for positions (3, n)."""
    n = pos.shape[1]
    i, j, r = _pairs(pos.T, box, max(h.rc_R, h.rc_A))
    U = torch.empty(n, dtype=torch.float64, device=pos.device)
    p = torch.empty_like(r)
    ends = torch.searchsorted(i, torch.arange(0, n + 16384, 16384, device=i.device).clamp(max=n)).tolist()
    for b, (e0, e1) in enumerate(zip(ends[:-1], ends[1:])):
        a0 = b * 16384
        a1 = min(n, a0 + 16384)
        if a0 >= a1:
            break
        rb = r[e0:e1].clone().requires_grad_(True)
        q = _descriptors(h, a1 - a0, i[e0:e1] - a0, rb, _weight(species, i[e0:e1], j[e0:e1]))
        u = _network(h, z, q)
        p[e0:e1] = torch.autograd.grad(u.sum(), rb)[0]
        U[a0:a1] = u.detach()
    F = torch.zeros(n, 3, dtype=torch.float64, device=pos.device).index_add(0, i, p).index_add(0, j, -p)
    # W_j = sum over pairs (i, j): r_ji (x) p_ij with r_ji = -r_ij
    W = torch.zeros(n, 9, dtype=torch.float64, device=pos.device)
    W.index_add_(0, j, -(r[:, :, None] * p[:, None, :]).reshape(-1, 9))
    return U, F.T.contiguous(), W.T.contiguous()


def _exact_md(case, h, z, pos, box, species, vel):
    n, dt, m = pos.shape[1], 1.0, MASS[case["model"]] * AMU_A2_FS2_EV
    L = torch.tensor(box, dtype=torch.float64, device=pos.device)[:, None]
    pos = pos - L * torch.floor(pos / L)
    built = pos.clone()
    thermo, heat = [], []

    def forces():
        U, F, W = _exact_efv(h, z, pos, box, species)
        if case["drive"]:
            fe = torch.tensor(DRIVE, dtype=torch.float64, device=pos.device)
            ext = (fe[:, None, None] * W.reshape(3, 3, n)).sum(0)
            F = F + ext - ext.mean(dim=1, keepdim=True)
        return U, F, W

    F = forces()[1]
    for _ in range(case["steps"]):
        vel = vel + 0.5 * dt / m * F
        pos = pos + dt * vel
        if ((pos - built) ** 2).sum(0).max() > (0.5 * h.skin) ** 2:  # positions are wrapped at each list build
            pos = pos - L * torch.floor(pos / L)
            built = pos.clone()
        U, F, W = forces()
        vel = vel + 0.5 * dt / m * F
        heat.append((W.reshape(3, 3, n) * vel[None]).sum((1, 2)))
        kinetic = 0.5 * m * (vel * vel).sum()
        if case["drive"]:
            scale2 = 1.0 + dt / COUPLING_FS * (TARGET_K / (2.0 * kinetic / ((3 * n - 3) * KB_EV)) - 1.0)
            vel, kinetic = vel * scale2.sqrt(), kinetic * scale2
        W = W.sum(1)
        thermo.append(torch.stack([U.sum(), kinetic, W[0], W[4], W[8], W[1], W[5], W[6]]))
    out = {"pos": pos, "vel": vel, "thermo": torch.stack(thermo)}
    return dict(out, heat=torch.stack(heat)) if case["heat"] else out


def _set_pairs(h, structures):
    dev, off, parts = _device(), 0, []
    for s in structures:
        i, j, r = _pairs(torch.tensor(s["pos"], device=dev), np.diag(s["box"]), max(h.rc_R, h.rc_A))
        parts.append((i + off, j + off, r))
        off += len(s["pos"])
    i, j, r = (torch.cat(v) for v in zip(*parts))
    return off, i, j, r


def _exact_losses(case, seed):
    h, dev = HYPER["si"], _device()
    structures, e_tar, f_tar, w_tar = _training_set(case["structures"], seed)
    n, i, j, r = _set_pairs(h, structures)
    count = torch.tensor([len(s["pos"]) for s in structures], device=dev)
    of = torch.repeat_interleave(torch.arange(len(count), device=dev), count)
    e_tar, f_tar, w_tar = (torch.tensor(v, device=dev) for v in (e_tar, f_tar, w_tar))
    r.requires_grad_(True)
    q = _descriptors(h, n, i, r, _weight(None, i, j))
    voigt = torch.tensor([[0, 0], [1, 1], [2, 2], [0, 1], [1, 2], [2, 0]], device=dev)
    rows = []
    for zk in _population(case["population"], seed):
        z = torch.tensor(zk, device=dev).double()
        qk = q.detach().requires_grad_(True)
        U = _network(h, z, qk)
        p = torch.autograd.grad(q, r, torch.autograd.grad(U.sum(), qk)[0], retain_graph=True)[0]
        F = torch.zeros(n, 3, dtype=torch.float64, device=dev).index_add(0, i, p).index_add(0, j, -p)
        w = -r.detach()[:, voigt[:, 0]] * p[:, voigt[:, 1]]
        W = torch.zeros(len(count), 6, dtype=torch.float64, device=dev).index_add(0, of[j], w)
        E = torch.zeros(len(count), dtype=torch.float64, device=dev).index_add(0, of, U.detach())
        terms = [(((E - e_tar) / count) ** 2).mean().sqrt(), ((F - f_tar) ** 2).mean().sqrt(),
                 (((W - w_tar) / count[:, None]) ** 2).mean().sqrt(), z.abs().mean(), (z * z).mean().sqrt()]
        rows.append(torch.stack([terms[0] + terms[1] + terms[2] + 0.05 * (terms[3] + terms[4])] + terms))
    return torch.stack(rows)


def _exact_gradient(case, seed):
    h, dev = HYPER["si"], _device()
    structures, _, f_tar, _ = _training_set(case["structures"], seed)
    n, i, j, r = _set_pairs(h, structures)
    z = torch.tensor(_weights("si", seed + 1), device=dev).double().requires_grad_(True)
    r.requires_grad_(True)
    q = _descriptors(h, n, i, r, _weight(None, i, j))
    w1, b1, w2, _ = _split(h, z)
    x = torch.tanh(q.detach() @ w1.T - b1)
    G = (w2 * (1.0 - x * x)) @ w1
    p = torch.autograd.grad(q, r, G.detach(), retain_graph=True)[0]
    F = torch.zeros(n, 3, dtype=torch.float64, device=dev).index_add(0, i, p).index_add(0, j, -p)
    res = F - torch.tensor(f_tar, device=dev)
    loss = (res * res).mean().sqrt()
    # dL/dG_i = sum_j dq_i/dr_ij . (delta_i - delta_j): the product of the
    # Jacobian with the pair differences, by differentiating its transpose
    delta = res / (res.numel() * loss)
    v = torch.zeros_like(q, requires_grad=True)
    back = torch.autograd.grad(q, r, v, create_graph=True)[0]
    dG = torch.autograd.grad(back, v, delta[i] - delta[j])[0]
    return {"loss": loss, "grad": torch.autograd.grad(G, z, dG, allow_unused=True)[0]}


def exact(case, seed):
    if case["kind"] == "grad":
        return _exact_gradient(case, seed)
    if case["kind"] == "snes":
        # a block of generations is up to a thousand evaluations: over 20 s
        return None if case["generations"] else _exact_losses(case, seed)
    h = HYPER[case["model"]]
    pos, box, species = _configuration(case, seed)
    n = pos.shape[1]
    z = torch.tensor(_weights(case["model"], seed), device=pos.device).double()
    if case["kind"] == "md":
        if n * case["steps"] * (4 if case["model"] == "pbte" else 1) > 4_000_000:
            return None  # over 20 s
        return _exact_md(case, h, z, pos, box, species, _velocities(n, MASS[case["model"]], seed))
    U, F, W = _exact_efv(h, z, pos, box, species)
    out = {"e_total": U.sum().reshape(1), "e_atom": U, "force": F, "virial_atom": W, "virial_total": W.sum(1)}
    return dict(out, err=None) if case["static"] else out
