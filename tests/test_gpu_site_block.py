"""Kernels at the edges of their tiles, blocks and variants: the site pass (32
atoms per block, 16 list slots per shared tile and 32 own slots per word and
thread: atom counts around the block, slot counts around the tile and every
capacity class against the oracle, at the bars of the force path: 1e-6 eV,
1e-4 eV/A), the list by direct tests and by cells, the cell offsets, the FP32
population network, the adjoint, dependent launches back to back, the split of
the positions, and the step sums of driven and plain MD."""
import numpy as np
import pytest

from gpu_util import aos, f32_exact, soa, virial_aos
from paper_2107_08119_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,edge,capacity,n_neu", [
    (1, 5.43, 96, 30),      # no neighbour: no tile at all
    (31, 5.43, 96, 30),
    (32, 5.43, 16, 30),     # clusters of few neighbours
    (33, 5.43, 96, 1),      # fewer neurons than warps
    (65, 4.6, 96, 7),
    (512, 4.3, 128, 30),    # 60 neighbours; the last capacity of one word per thread
    (512, 4.3, 129, 30),    # three words, no in-cutoff masks
    (500, 4.0, 384, 64),
])
def test_block_edges(orc, n, edge, capacity, n_neu):
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n + capacity)
    pos, box = inputs.diamond(4, 4, 4, edge)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    hyper = nep.Hyper(max_neighbors=capacity, n_neu=n_neu)
    z = inputs.random_z(hyper.n_par, rng)
    model = nep.NEP(z, hyper)
    out = model.compute(soa(pos), box)
    U, F, W = orc.efv(orc.NepHyper(n_neu=n_neu), f32_exact(z), pos, box)
    assert np.abs(out["e_atom"].cpu().numpy() - U).max() <= 1e-6 * max(1.0, n_neu / 30)
    assert np.abs(aos(out["force"]) - F).max() <= 1e-4
    assert np.abs(virial_aos(out["virial_atom"]) - W).max() <= 1e-4
    assert abs(out["e_total"].item() - U.sum()) <= 1e-6 * n * max(1.0, n_neu / 30)
    model.close()


@pytest.mark.parametrize("n", [6080, 6081, 12160, 12161, 12193])
def test_atoms_per_block(orc, n):
    """The last size of 8 atoms per block, the range of 16, and 32 with ragged
    tails: the first and last atoms and a sample, on a cut-open crystal."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n)
    pos, box = inputs.diamond(12, 12, 12)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    z = inputs.random_z(1021, rng)
    model = nep.NEP(z)
    out = model.compute(soa(pos), box)
    idx = np.unique(np.concatenate([np.arange(40), np.arange(n - 40, n), rng.integers(0, n, 100)]))
    U, F, W = orc.efv_sample(orc.NepHyper(), f32_exact(z), pos, box, idx)
    assert np.abs(out["e_atom"].cpu().numpy()[idx] - U).max() <= 1e-6
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4
    assert np.abs(virial_aos(out["virial_atom"])[idx] - W).max() <= 1e-4
    # the totals are the sums of the per-atom outputs (FP64 sums, so 1e-9 of the largest terms' sum)
    e, w = out["e_atom"].sum().item(), out["virial_atom"].double().sum(dim=1)
    assert abs(out["e_total"].item() - e) <= 1e-9 * n
    assert (out["virial_total"] - w).abs().max().item() <= 1e-9 * n * 10
    model.close()


@pytest.mark.parametrize("cells,n", [
    ((1, 1, 1), 8),      # every pair through several images
    ((2, 2, 2), 63),     # no cell grid, odd count
    ((2, 3, 5), 240),    # no cell grid in one direction only
    ((4, 4, 4), 511),    # grid box, nearest images
    ((7, 7, 7), 2500),   # the last count of the direct list
    ((7, 7, 7), 2501),   # the first of the cells path
])
def test_list_by_direct_tests(orc, cells, n):
    """The list built by testing every atom: the same neighbours, distances
    ascending, as the oracle's brute-force list, and the forces from it."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n)
    pos, box = inputs.diamond(*cells)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    z = inputs.random_z(1021, rng)
    model = nep.NEP(z)
    out = model.compute(soa(pos), box)
    cnt, nbr = (t.cpu().numpy() for t in model.neighbors(n))
    _, F, _ = orc.efv_sample(orc.NepHyper(), f32_exact(z), pos, box, np.arange(min(n, 200)))
    assert np.abs(aos(out["force"])[:200] - F).max() <= 1e-4
    L = np.diag(box)
    x = pos - L * np.floor(pos / L)
    for i in range(0, n, max(1, n // 50)):
        v = nbr[:cnt[i], i]
        code = v >> 24
        shift = np.stack([code // 25 - 2, code // 5 % 5 - 2, code % 5 - 2], 1)
        r = np.linalg.norm(x[v & 0xFFFFFF] + shift * L - x[i], axis=1)
        assert np.all(np.diff(r) >= -1e-5) and r.max() < 5.0 + 1e-5
        assert len(set(v.tolist())) == len(v)
        img = np.stack(np.meshgrid(*[np.arange(-2, 3)] * 3, indexing="ij"), -1).reshape(-1, 1, 3) * L
        d = np.linalg.norm(x[None] + img - x[i], axis=2)
        assert abs(int(np.sum((d < 5.0) & (d > 1e-9))) - len(v)) <= int(np.sum(np.abs(d - 5.0) < 1e-5))
    model.close()


@pytest.mark.parametrize("n_struct,n_pop,n_neu,threads", [
    (1, 1, 30, 128),     # one member, one ragged tile of atoms
    (1, 2, 1, 256),
    (3, 5, 30, 128),     # a partial member group
    (3, 9, 30, 256),
    (2, 64, 64, 256),    # the largest network and population: four members per block
])
def test_population_network_shapes(orc, n_struct, n_pop, n_neu, threads):
    """The FP32 population network around its tiles (128 atoms, 4 or 8
    members): every loss term of every member against the oracle.  FP32 sums of
    ~100 terms per force: 3e-4, the bar of the population tests."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n_pop)
    hyper = nep.Hyper(n_neu=n_neu)
    structures = inputs.training_structures(n_struct, seed_stream=n_pop)
    n = sum(len(s["pos"]) for s in structures)
    e = rng.normal(-3.0, 0.1, n_struct) * [len(s["pos"]) for s in structures]
    f, w = rng.normal(0.0, 1.0, (n, 3)), rng.normal(0.0, 1.0, (n_struct, 6))
    pop = rng.normal(0.0, 0.1, (n_pop, hyper.n_par)).astype(np.float32)
    model = nep.NEP(pop[0], hyper)
    ds = nep.Dataset(model, structures, e, f, w)
    ds.set_shape(fused=0, mlp_threads=threads)
    got = ds.evaluate(torch.tensor(pop, device="cuda")).cpu().numpy()
    for k in {0, n_pop // 2, n_pop - 1}:
        want = orc.loss(orc.NepHyper(n_neu=n_neu), f32_exact(pop[k]), structures, e, f, w)
        assert np.abs(got[k] - want).max() <= 3e-4, (k, got[k], want)
    ds.close()
    model.close()


@pytest.mark.parametrize("n_struct", [1, 40, 110, 140])
def test_adjoint_by_atoms_per_block(orc, n_struct):
    """The force loss and its gradient with 8 atoms per block (1 and 40
    structures), 16 and 32, and ragged tails: against the oracle for the small
    set, and by a central difference of the loss along the gradient for all
    (the loss is smooth: step 1e-3 |z| leaves ~1e-6 relative, FP32 forces
    ~1e-4 of the difference)."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n_struct)
    structures = inputs.training_structures(n_struct, seed_stream=77)
    n = sum(len(s["pos"]) for s in structures)
    f = rng.normal(0.0, 1.0, (n, 3))
    z = inputs.random_z(1021, rng).astype(np.float32)
    model = nep.NEP(z)
    ds = nep.Dataset(model, structures, np.zeros(n_struct), f, np.zeros((n_struct, 6)))
    t = torch.tensor(z, device="cuda", requires_grad=True)
    loss = nep.force_loss(t, ds)
    loss.backward()
    g = t.grad.double()
    if n_struct == 1:
        want, lf = orc.force_loss_grad(orc.NepHyper(), f32_exact(z), structures, f)
        assert abs(loss.item() - lf) <= 1e-6 * lf
        assert np.abs(g.cpu().numpy() - want).max() <= 1e-5 * np.abs(want).max()
    d = g / g.norm()
    h = 1e-3 * float(t.detach().norm())
    up, dn = ((t.detach().double() + s * h * d).float() for s in (1.0, -1.0))
    fd = (ds.force_loss(up) - ds.force_loss(dn)).item() / float(((up - dn).double() * d).sum())
    assert abs(fd - float(g.norm())) <= 2e-3 * float(g.norm()), (fd, float(g.norm()))
    ds.close()
    model.close()


@pytest.mark.parametrize("kind", ["dense spot", "thin grid", "few large cells", "split model"])
def test_cells_path_search(orc, kind):
    """The half-shell search per cell: a cell with more candidates than its
    shared buffer (a dense cluster in a large box), a grid of three cells in one
    direction, eight warps per cell, and the 8 A cells of the split model.
    Counts and forces of a sample against the oracle."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(len(kind))
    hyper, oh = nep.Hyper(max_neighbors=384), orc.NepHyper()
    if kind == "dense spot":      # 3000 atoms at 2.4 A spacing in one corner of a 400 A box
        g = np.stack(np.meshgrid(*[np.arange(15)] * 3, indexing="ij"), -1).reshape(-1, 3)[:3000] * 2.4
        pos, box = g + rng.normal(0.0, 0.1, (3000, 3)), np.diag([400.0] * 3)
    elif kind == "thin grid":
        pos, box = inputs.diamond(3, 12, 11)
        pos = inputs.displace(pos, 0.1, rng)
    elif kind == "few large cells":
        pos, box = inputs.diamond(7, 7, 8)
        pos = inputs.displace(pos, 0.1, rng)
    else:
        pos, _, box, z, _ = inputs.config_pbte((7, 7, 8))
        hyper = nep.Hyper(**inputs.PBTE_HYPER)
        oh = orc.NepHyper(12, 6, 4, 40, 8.0, 4.0)
    assert len(pos) > 2500
    if kind != "split model":
        z = inputs.random_z(hyper.n_par, rng)
    model = nep.NEP(z, hyper)
    out = model.compute(soa(pos), box)
    cnt, _ = model.neighbors(len(pos))
    idx = np.unique(rng.integers(0, len(pos), 150))
    U, F, _ = orc.efv_sample(oh, f32_exact(z), pos, box, idx)
    assert np.abs(out["e_atom"].cpu().numpy()[idx] - U).max() <= 1e-6
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4
    rc, L = hyper.rc_R, np.diag(box)
    for i in idx[:40]:
        d = pos - pos[i]
        r = np.linalg.norm(d - L * np.round(d / L), axis=1)
        near = int(np.sum(np.abs(r - rc) < 1e-5))
        assert abs(int(cnt[i]) - int(np.sum((r < rc) & (r > 0)))) <= near
    model.close()


@pytest.mark.parametrize("cells", [(1, 1, 1), (4, 4, 4), (7, 7, 7), (12, 12, 12), (20, 20, 20)])
def test_calls_back_to_back(cells):
    """The kernels of a call are set up while their predecessors still run: calls
    enqueued without a wait between them give the bits of calls that were waited
    for (the summation orders are fixed, so equality)."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(5)
    pos, box = inputs.diamond(*cells)
    states = [soa(inputs.displace(pos, 0.1, rng)) for _ in range(6)]
    model = nep.NEP(inputs.random_z(1021, rng))
    waited = []
    for x in states:
        waited.append({k: v.clone() for k, v in model.compute(x, box).items()})
        torch.cuda.synchronize()
    queued = [{k: v.clone() for k, v in model.compute(x, box).items()} for x in states]
    torch.cuda.synchronize()
    for a, b in zip(waited, queued):
        for k in a:
            assert torch.equal(a[k], b[k]), k
    model.close()


@pytest.mark.parametrize("value", [0.0, -0.0, 1e-310, -1e-40, 2.0 ** -101, 2.0 ** -102, 1e-20, 5.5, 1.0 + 2.0 ** -24,
                                   1.0 + 3 * 2.0 ** -24, np.nextafter(2.0, 0.0), -3.0 + 2.0 ** -40])
def test_position_split(orc, value):
    """Positions are split into two FP32 words by integer operations: zeros,
    denormals, the ends of that range, halves of the last place and carries into
    the next binade as coordinates of one atom."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(11)
    pos, box = inputs.diamond(3, 3, 3)
    pos = inputs.displace(pos, 0.1, rng)
    pos -= pos[5]
    pos[5] = value  # all other coordinates moved with it
    pos[:5] += value
    pos[6:] += value
    z = inputs.random_z(1021, rng)
    model = nep.NEP(z)
    out = model.compute(soa(pos), box)
    U, F, W = orc.efv(orc.NepHyper(), f32_exact(z), pos, box)
    assert np.abs(out["e_atom"].cpu().numpy() - U).max() <= 1e-6
    assert np.abs(aos(out["force"]) - F).max() <= 1e-4
    model.close()


@pytest.mark.parametrize("n", [63, 65, 38912, 38913])
def test_driven_step_sums(n):
    """The per-atom step kernels run in blocks of 64 atoms up to 38,912 and of
    256 above: E_kin of the last step is that of the velocities (FP64 sums of
    n terms: 1e-12 relative), and the drive keeps the total momentum (FP32
    forces: each of n steps of dt F / m rounds at 2^-24 of at most 10 eV/A)."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n)
    pos, box = inputs.diamond(17, 17, 17) if n > 1000 else inputs.diamond(2, 2, 3)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    vel = rng.normal(0.0, 1e-3, (n, 3))
    vel -= vel.mean(axis=0)
    model = nep.NEP(inputs.random_z(1021, rng))
    mass, dt = 28.085, 1.0
    md = nep.MD(model, n, box, mass)
    md.set_hnemd([1e-4, 0.0, -2e-4])
    x, v = soa(pos), soa(vel)
    thermo = torch.zeros((3, 8), dtype=torch.float64, device="cuda")
    md.step(x, v, 3, dt, thermo=thermo)
    unit = 1.66053906660e-27 * 1.0e10 / 1.602176634e-19  # amu A^2 / fs^2 in eV
    ekin = 0.5 * mass * unit * (v * v).sum().item()
    assert abs(thermo[2, 1].item() - ekin) <= 1e-12 * ekin
    assert v.sum(dim=1).abs().max().item() <= n * 3 * dt * 10 * 2.0 ** -24 / (mass * unit)
    md.close()
    model.close()


@pytest.mark.parametrize("n,drive,tau", [(512, False, 0.0), (512, True, 0.0), (38913, False, 0.0), (512, False, 20.0),
                                         (512, True, 20.0)])
def test_step_sums_inside_the_next_kick(n, drive, tau):
    """The sums of a step are added up by the next step's first kernel where one
    follows in the same graph and by a kernel of their own where none does: the
    rows, J and states of one run of 12 steps (graphs of five, five, one and one)
    have the bits of twelve runs of one step (the same order of sums).  With a
    thermostat the next kick applies the factor to the velocities instead: the
    product is rounded in both forms."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n)
    pos, box = inputs.diamond(17, 17, 17) if n > 1000 else inputs.diamond(4, 4, 4)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    vel = rng.normal(0.0, 1e-3, (n, 3))
    model = nep.NEP(inputs.random_z(1021, rng))
    got = []
    for chunk in (12, 1):
        md = nep.MD(model, n, box, 28.085)
        if drive:
            md.set_hnemd([1e-4, 0.0, -2e-4])
        if tau:
            md.set_thermostat(300.0, tau)
        x, v = soa(pos), soa(vel)
        thermo = torch.zeros((12, 8), dtype=torch.float64, device="cuda")
        heat = torch.zeros((12, 3), dtype=torch.float64, device="cuda")
        for s in range(0, 12, chunk):
            md.step(x, v, chunk, 1.0, thermo=thermo[s:s + chunk], heat=heat[s:s + chunk])
        torch.cuda.synchronize()
        got.append((x, v, thermo, heat))
        md.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert got[0][2][:, 1].min().item() > 0.0 and got[0][3].abs().min().item() > 0.0
    model.close()


@pytest.mark.parametrize("nc", [(32, 16, 16), (33, 16, 16), (48, 32, 16), (110, 110, 110)])
def test_cell_offsets_by_slices(orc, nc):
    """Cell offsets scanned in slices of 8192 cells (one, one and a rest, three,
    and with 1.3 million cells two rounds per slice): 1500 pairs of atoms spread
    over the box find their partners, twice (the counts are zero after a build)."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(sum(nc))
    L = 5.0 * np.array(nc) + 0.5
    m = np.array([20, 10, 10])
    g = np.stack(np.meshgrid(*[np.arange(k) for k in m], indexing="ij"), -1).reshape(-1, 3)
    a = (g[rng.permutation(len(g))[:1500]] + 0.5) * (L / m)  # centres at least 8 A apart
    d = rng.normal(size=(1500, 3))
    d *= (rng.uniform(1.0, 1.25, 1500) / np.linalg.norm(d, axis=1))[:, None]
    pos, box = np.concatenate([a - d, a + d]), np.diag(L)
    z = inputs.random_z(1021, rng)
    model = nep.NEP(z)
    idx = np.unique(rng.integers(0, 3000, 100))
    U, F, _ = orc.efv_sample(orc.NepHyper(), f32_exact(z), pos, box, idx)
    for _ in range(2):
        out = model.compute(soa(pos), box)
        cnt, _ = model.neighbors(3000)
        assert int(cnt.min()) >= 1
        assert np.abs(out["e_atom"].cpu().numpy()[idx] - U).max() <= 1e-6
        assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4
    model.close()
