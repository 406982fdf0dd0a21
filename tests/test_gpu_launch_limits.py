"""Calls at the limits of what a kernel takes: the default shared memory (48 KB, of
which a kernel's static part counts too), and the 96 slots of the in-cutoff masks."""
import numpy as np
import pytest

from gpu_util import aos, f32_exact, soa
from paper_2107_08119_gb300 import inputs

pytestmark = pytest.mark.gpu


def _split_model(n_neu, rng):
    """Hyperparameters and parameters of the split model at another width, the
    input columns scaled to the weighted descriptors."""
    from paper_2107_08119_gb300 import nep
    hyper = nep.Hyper(**dict(inputs.PBTE_HYPER, n_neu=n_neu))
    z = inputs.random_z(hyper.n_par, rng)
    n_r = hyper.n_max_R + 1
    n_des = hyper.n_par // n_neu - 2
    zbar = np.sqrt(inputs.Z_PB * inputs.Z_TE)
    w1 = z[:n_neu * n_des].reshape(n_neu, n_des)
    w1[:, :n_r] /= zbar
    w1[:, n_r:] /= zbar ** 2
    return hyper, z


@pytest.mark.parametrize("n_neu", [49, 50, 51, 52, 64])
@pytest.mark.parametrize("n", [12160, 12161])
def test_split_model_widths(orc, n, n_neu):
    """The site pass of the split model with 16 and 32 atoms per block around the
    width at which the latter needs more than the default shared memory (50 and 51
    only together with the static part): a sample against the oracle, at the bars
    of the force path for wider networks."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n_neu)
    pos, _, box = inputs.rocksalt(12, 12, 11)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    hyper, z = _split_model(n_neu, rng)
    model = nep.NEP(z, hyper)
    out = model.compute(soa(pos), box)
    idx = np.unique(rng.integers(0, n, 60))
    U, F, _ = orc.efv_sample(orc.NepHyper(12, 6, 4, n_neu, 8.0, 4.0), f32_exact(z), pos, box, idx)
    assert np.abs(out["e_atom"].cpu().numpy()[idx] - U).max() <= 1e-6 * n_neu / 30
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4
    model.close()


@pytest.mark.parametrize("capacity,edge", [(128, 3.3), (129, 3.3), (185, 3.0), (186, 3.0), (187, 3.0), (384, 3.0)])
def test_list_capacities(orc, capacity, edge):
    """The row sort of the cells path around the capacity at which its shared tile
    no longer fits (116 and 155 neighbours per atom): the rows are the atoms within
    the cutoff, distances ascending, and the forces those of the oracle (1e-4 eV/A
    at forces of 10 eV/A; here they are larger, and FP32 is relative)."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(capacity)
    pos, box = inputs.diamond(6, 8, 7, edge)
    pos = inputs.displace(pos, 0.05, rng)
    n = len(pos)
    hyper = nep.Hyper(max_neighbors=capacity)
    z = inputs.random_z(hyper.n_par, rng)
    model = nep.NEP(z, hyper)
    out = model.compute(soa(pos), box)
    cnt, nbr = (t.cpu().numpy() for t in model.neighbors(n))
    idx = np.unique(rng.integers(0, n, 40))
    _, F, _ = orc.efv_sample(orc.NepHyper(), f32_exact(z), pos, box, idx)
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4 * max(1.0, np.abs(F).max() / 10)
    L = np.diag(box)
    for i in idx:
        d = pos - pos[i]
        r = np.linalg.norm(d - L * np.round(d / L), axis=1)
        row = r[nbr[:cnt[i], i] & 0xFFFFFF]
        assert abs(int(cnt[i]) - int(np.sum((r < 5.0) & (r > 0)))) <= int(np.sum(np.abs(r - 5.0) < 1e-5))
        assert row.max() < 5.0 + 1e-5 and np.all(np.diff(row) >= -1e-5)
        assert len(set((nbr[:cnt[i], i] & 0xFFFFFF).tolist())) == cnt[i]
    model.close()


def test_more_than_96_slots_in_a_large_box(orc):
    """The assembly by atoms (above 60,000 of them) without slot masks: a cluster
    whose atoms have more than 96 neighbours beside a sparse crystal, net force
    and a sample of the cluster against the oracle (1e-4 eV/A at forces of
    10 eV/A)."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(3)
    pos, box = inputs.diamond(20, 20, 20)
    pos = inputs.displace(pos, 0.1, rng)
    far = np.linalg.norm(pos - np.diag(box) / 2, axis=1) > 12.0
    spot, edges = inputs.diamond(5, 5, 5, 3.2)
    spot = inputs.displace(spot, 0.05, rng) - np.diag(edges) / 2 + np.diag(box) / 2
    pos = np.concatenate([pos[far], spot])
    n = len(pos)
    assert n > 60000
    hyper = nep.Hyper(max_neighbors=256)
    z = inputs.random_z(hyper.n_par, rng)
    model = nep.NEP(z, hyper)
    out = model.compute(soa(pos), box)
    cnt, _ = model.neighbors(n)
    assert int(cnt.max()) > 96 and float(cnt.double().mean()) < 45
    idx = np.argsort(cnt.cpu().numpy())[-40:]
    U, F, _ = orc.efv_sample(orc.NepHyper(), f32_exact(z), pos, box, idx)
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4 * max(1.0, np.abs(F).max() / 10)
    model.close()


def _training(n_neu, cells, seed):
    """A training set of two cells and a model of n_neu neurons, and a population."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(seed)
    hyper = nep.Hyper(n_neu=n_neu)
    pos, box = inputs.diamond(*cells)
    structures = [{"pos": inputs.displace(pos, 0.1, rng), "box": box} for _ in range(2)]
    n = 2 * len(pos)
    model = nep.NEP(inputs.random_z(hyper.n_par, rng), hyper)
    ds = nep.Dataset(model, structures, np.zeros(2), rng.normal(0.0, 1.0, (n, 3)), np.zeros((2, 6)))
    pop = torch.tensor(rng.normal(0.0, 0.1, (16, hyper.n_par)).astype(np.float32), device="cuda")
    return model, ds, pop


@pytest.mark.parametrize("fused", [0, 8])
def test_training_sets_of_two_widths_in_two_threads(fused):
    """Kernels' shared-memory limits belong to the kernels, not to a training set:
    two host threads that evaluate sets of networks of 4 and 64 neurons, with 32
    and 256 atoms per structure, do not lower them for one another.  Every loss has
    the bits of the same evaluation alone."""
    import threading

    import torch
    sets = [_training(4, (1, 2, 2), 1), _training(64, (4, 4, 2), 2)]
    want = []
    for _, ds, pop in sets:
        ds.set_shape(fused=fused, mlp_threads=256)
        want.append(ds.evaluate(pop).clone())
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            _, ds, pop = sets[k]
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(400):
                    got = ds.evaluate(pop)
                torch.cuda.current_stream().synchronize()
                assert torch.equal(got, want[k])
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for model, ds, _ in sets:
        ds.close()
        model.close()


@pytest.mark.parametrize("change", ["rows", "target temperature"])
def test_step_graphs_outlive_their_rows(change):
    """A block of steps that writes its rows elsewhere, or has another target
    temperature, runs from the graphs of the block before: the states and rows of
    the same run by single steps, and no time for new graphs (twice the block's own
    time when they were captured again; a factor of 1.5 leaves room for noise)."""
    import statistics
    import time

    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(8)
    pos, box = inputs.diamond(4, 4, 4)
    pos = inputs.displace(pos, 0.05, rng)
    n, steps, blocks = len(pos), 5, 40
    vel = rng.normal(0.0, 1e-3, (n, 3))
    model = nep.NEP(inputs.random_z(1021, rng))

    def run(fresh, ramp, chunk):
        """Blocks with rows of their own (fresh) or in one buffer, in calls of `chunk` steps."""
        md = nep.MD(model, n, box, 28.085)
        x, v = soa(pos), soa(vel)
        thermo = torch.zeros((blocks * steps, 8), dtype=torch.float64, device="cuda")
        heat = torch.zeros((blocks * steps, 3), dtype=torch.float64, device="cuda")
        one, two = thermo[:chunk].clone(), heat[:chunk].clone()
        times = []
        for s in range(0, blocks * steps, chunk):
            md.set_thermostat(300.0 + (5.0 * (s // steps) if ramp else 0.0), 100.0)
            torch.cuda.synchronize()
            t = time.perf_counter()
            if fresh:
                md.step(x, v, chunk, 1.0, thermo=thermo[s:s + chunk], heat=heat[s:s + chunk])
            else:
                md.step(x, v, chunk, 1.0, thermo=one, heat=two)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
            if not fresh:
                thermo[s:s + chunk].copy_(one)
                heat[s:s + chunk].copy_(two)
        md.close()
        return statistics.median(times[len(times) // 2:]), x, v, thermo, heat

    ramp = change != "rows"
    base, *same = run(False, False, steps)
    other, *got = run(not ramp, ramp, steps)
    _, *want = run(False, ramp, 1)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert torch.equal(got[2], same[2]) != ramp
    assert other <= 1.5 * base, (other, base)
    model.close()


def test_short_blocks_with_a_new_time_step():
    """Few steps with a new time step do not pay for a graph of several steps: a
    block of five with a new time step takes at most 1.6 times as long as the same
    block again (1.26 times with the capture of one step, 1.93 with that of five)."""
    import time

    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(9)
    pos, box = inputs.diamond(2, 2, 2)
    pos = inputs.displace(pos, 0.05, rng)
    model = nep.NEP(inputs.random_z(1021, rng))
    md = nep.MD(model, len(pos), box, 28.085)
    x, v = soa(pos), soa(rng.normal(0.0, 1e-3, (len(pos), 3)))

    def block(dt):
        torch.cuda.synchronize()
        t = time.perf_counter()
        md.step(x, v, 5, dt)
        torch.cuda.synchronize()
        return time.perf_counter() - t

    times = np.array([[block(1.0 + 1e-4 * k), block(1.0 + 1e-4 * k)] for k in range(80)])
    new, again = np.median(times[40:], axis=0)
    assert new <= 1.6 * again, (new, again)
    md.close()
    model.close()


def test_short_runs_with_new_loss_weights():
    """Few generations with new weights of the loss terms do not pay for a graph of
    several generations: six take at most 1.45 times as long as the same six again
    (1.25 times with the capture of one generation, 1.6 with both graphs); and runs
    of 6, 40 and 14 generations, through both graphs, have the states of one run of
    60."""
    import time

    import torch
    from paper_2107_08119_gb300 import nep
    model, ds, _ = _training(30, (1, 2, 2), 6)
    mean = np.random.default_rng(6).uniform(-0.5, 0.5, model.hyper.n_par)
    ds.set_shape(fused=0, mlp_threads=256, owner_tc=1, pop_pipe=1)

    def fresh():
        return nep.SNES(model, 16, mean, np.full(len(mean), 0.1), 3)

    snes = fresh()

    def run(weight):
        torch.cuda.synchronize()
        t = time.perf_counter()
        snes.run(ds, 6, nep.PREC_BF16, lambdas=[weight, 1.0, 1.0, 0.05, 0.05])
        torch.cuda.synchronize()
        return time.perf_counter() - t

    times = np.array([[run(1.0 + 1e-4 * k), run(1.0 + 1e-4 * k)] for k in range(80)])
    new, again = np.median(times[40:], axis=0)
    assert new <= 1.45 * again, (new, again)
    snes.close()
    states = []
    for blocks in ((60,), (6, 40, 14)):
        snes = fresh()
        for g in blocks:
            snes.run(ds, g, nep.PREC_BF16)
        states.append([t.clone() for t in snes.state()[:2]])
        snes.close()
    for a, b in zip(*states):
        assert torch.equal(a, b)
    ds.close()
    model.close()


@pytest.mark.parametrize("nc", [(17, 17, 17), (18, 18, 18), (60, 9, 10), (100, 100, 100)])
def test_sparse_boxes(orc, nc):
    """The cells path below and above two cells per atom, where the search goes by
    atoms: 2600 atoms in close pairs and triples, one cell with forty of them, all
    counts against brute force and a sample against the oracle; and MD with the
    list built behind a gate (spectral heat current) and without, same bits."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(sum(nc))
    L = 6.0 * np.array(nc) + 0.5  # cells of the list radius of MD
    a = rng.uniform(0.0, L, (1300, 3))
    d = rng.normal(size=(1300, 3))
    pos = np.concatenate([a, a + d * (rng.uniform(1.5, 4.0, 1300) / np.linalg.norm(d, axis=1))[:, None]])
    g = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3)[:40]
    pos[:40] = 6.2 + 1.3 * g + rng.normal(0.0, 0.05, (40, 3))
    box, n = np.diag(L), len(pos)
    z = inputs.random_z(1021, rng)
    model = nep.NEP(z)
    out = model.compute(soa(pos), box)
    cnt = model.neighbors(n)[0].cpu().numpy()
    for i in range(n):
        r = pos - pos[i]
        r = np.linalg.norm(r - L * np.round(r / L), axis=1)
        near = int(np.sum(np.abs(r - 5.0) < 1e-5))
        assert abs(int(cnt[i]) - int(np.sum((r < 5.0) & (r > 0)))) <= near
    idx = np.unique(np.concatenate([np.arange(40), rng.integers(0, n, 100)]))
    U, F, _ = orc.efv_sample(orc.NepHyper(), f32_exact(z), pos, box, idx)
    assert np.abs(out["e_atom"].cpu().numpy()[idx] - U).max() <= 1e-6
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4
    got = []
    for shc in (False, True):
        md = nep.MD(model, n, box, 28.085)
        if shc:
            md.set_shc(4, 2)
        x, v = soa(pos), soa(np.full((n, 3), 0.05))
        md.step(x, v, 12, 1.0)
        torch.cuda.synchronize()
        assert md.rebuild_count() > 0
        got.append((x, v))
        md.close()
    for s, t in zip(*got):
        assert torch.equal(s, t)
    model.close()


def test_empty_cells_cost_little():
    """3,000 atoms in a box of 512,000 cells take at most twice as long as in one of
    8,000 (five times as long when every empty cell had a block)."""
    import time

    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(2)
    model = nep.NEP(inputs.random_z(1021, rng))

    def call(edge):
        x, box = soa(rng.uniform(0.0, edge, (3000, 3))), np.diag([edge] * 3)
        times = []
        for _ in range(30):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(5):
                model.compute(x, box, sync=False)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
        return np.median(times[10:])

    small, large = call(100.0), call(400.0)
    assert large <= 2.0 * small, (large, small)
    model.close()


@pytest.mark.parametrize("profile", [False, True])
def test_rows_and_targets_in_turn(profile):
    """One-step calls whose rows and target temperature stay or change, and with no
    rows between: every row and state of the same steps with rows of their own, and
    no row written that its call did not name."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(4)
    pos, box = inputs.diamond(3, 3, 3)
    pos = inputs.displace(pos, 0.05, rng)
    n = len(pos)
    vel = rng.normal(0.0, 1e-3, (n, 3))
    model = nep.NEP(inputs.random_z(1021, rng))
    model.profile(profile)
    # (buffer of the rows or None, target temperature or None)
    calls = [(0, None), (0, None), (1, None), (0, None), (None, None), (0, None), (0, 300.0), (0, 300.0), (0, 500.0),
             (1, 500.0), (1, 300.0), (None, 300.0), (1, None), (1, None), (0, None)]

    def run(shared):
        md = nep.MD(model, n, box, 28.085)
        x, v = soa(pos), soa(vel)
        rows = [torch.zeros(11, dtype=torch.float64, device="cuda") for _ in range(2)]
        out = []
        for b, target in calls:
            md.set_thermostat(target or 0.0, 100.0 if target else 0.0)
            if not shared:
                rows = [torch.zeros(11, dtype=torch.float64, device="cuda") for _ in range(2)]
            for r in rows:
                r.fill_(-1.0)
            if b is None:
                md.step(x, v, 1, 1.0)
            else:
                md.step(x, v, 1, 1.0, thermo=rows[b][:8], heat=rows[b][8:])
            out.append(torch.stack(rows + [torch.cat([x.sum(1), v.sum(1), x[:, 0], v[:, 0]])[:11]]))
        md.close()
        return torch.stack(out)

    got, want = run(True), run(False)
    assert torch.equal(got, want)
    for (b, _), g in zip(calls, got):
        for k in range(2):
            assert bool((g[k] == -1.0).all()) != (k == b)
    model.profile(False)
    model.close()


@pytest.mark.parametrize("cells,steps", [((15, 15, 16), 12), ((15, 16, 16), 5), ((15, 16, 16), 12)])
def test_first_steps_of_a_new_state(cells, steps):
    """The first call on a new state below and above 30,000 atoms, where its graph of
    five steps is captured behind the starting forces: states and rows of the same
    steps one by one."""
    import torch
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(6)
    pos, box = inputs.diamond(*cells)
    pos = inputs.displace(pos, 0.05, rng)
    n = len(pos)
    vel = rng.normal(0.0, 1e-3, (n, 3))
    model = nep.NEP(inputs.random_z(1021, rng))
    got = []
    for chunk in (steps, 1):
        md = nep.MD(model, n, box, 28.085)
        x, v = soa(pos), soa(vel)
        rows = torch.zeros((steps, 8), dtype=torch.float64, device="cuda")
        for s in range(0, steps, chunk):
            md.step(x, v, chunk, 1.0, thermo=rows[s:s + chunk])
        torch.cuda.synchronize()
        got.append((x, v, rows))
        md.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    model.close()
