"""The one-kernel step (a warp per cell, all groups) against the general batched
sequence: the same bits in every particle array, counter and status, over cells
that hold none, one or many of each species, both pairing cases, both sides of
the permutation's size limit, every lane-group class, unequal ion weights, odd
region starts, positions, several materials and steps; eager and from a graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

DEFAULT_POLLS = 1 << 22


@pytest.fixture(scope="module")
def pcc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    return pcc


def workload(law, n_cells, seed, with_x):
    rng = np.random.default_rng(seed)
    if law == "mixed":       # sizes around the classes' and the permutation's edges
        pick = np.array([0, 1, 2, 3, 5, 16, 31, 32, 33, 63, 64, 65, 127, 200, 383, 513, 1025])
        ne, ni, ng, npos = (rng.choice(pick, n_cells) for _ in range(4))
        npos //= 8
    elif law == "ions":      # N_p < N_t everywhere
        ne, ni, ng = rng.integers(0, 40, n_cells), rng.integers(20, 300, n_cells), rng.integers(0, 30, n_cells)
        npos = rng.integers(0, 3, n_cells)
    else:                    # N_p >> N_t
        ne, ni, ng = rng.integers(500, 2500, n_cells), rng.integers(1, 9, n_cells), rng.integers(50, 700, n_cells)
        npos = rng.integers(0, 20, n_cells)
    wl = W.solid_cu(n_cells=n_cells, e_per_cell=ne, i_per_cell=ni, photons_per_cell=ng, seed=seed, dt=0.5e-15, T_mev=20.0)
    pos = W.solid_cu(n_cells=n_cells, e_per_cell=npos, i_per_cell=1, seed=seed + 1, T_mev=20.0).species["em"]
    wl.species["ep"] = pos
    if law != "ions":        # unequal weights in some cells
        ion = wl.species["ion"]
        odd = ion["cell"] % 3 == 0
        ion["w"] = np.where(odd, ion["w"] * rng.uniform(0.5, 1.5, len(odd)), ion["w"]).astype(np.float32)
    em = wl.species["em"]
    em["w"] = (em["w"] * 10.0 ** rng.uniform(-2, 1, len(em["w"]))).astype(np.float32)
    if with_x:
        for d in wl.species.values():
            d["x"] = rng.uniform(0, 1, len(d["w"])).astype(np.float32)
    return wl


def run(pcc, wl, law, with_x, fused, graph, mask, steps):
    ctx = pcc.Context(0)
    mats = [pcc.material(29, 5.0, 8.5e28, 100.0), pcc.material(79, 20.0, 5.9e28, 1000.0)]
    ctx.tables_build(mats, pcc.table_spec(n_rows=63, n_cols=65))
    dev = {}
    for name, d in wl.species.items():
        sp = pcc.DeviceSpecies.empty(wl.n_cells, 2 * len(d["w"]) + 130 * wl.n_cells, with_x=with_x)
        pcc.bin(ctx, pcc.particles_to_device(d), wl.n_cells, sp, slack_abs=121, slack_rel=0.5)
        dev[name] = sp
    mat = torch.as_tensor((np.arange(wl.n_cells) % 2).astype(np.int32), device="cuda")
    ledger = torch.zeros((wl.n_cells, 4), dtype=torch.float32, device="cuda")
    ctx.read_status()
    if not fused:
        ctx.set_wait_limit(DEFAULT_POLLS - 1)     # a context with a wait limit of its own keeps the staged sequence
    n0 = pcc.launch_count()
    args = (wl.n_cells, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, 77)
    if graph:
        ctx.steps_capture(*args, 3, steps, mask=mask, ledger=ledger)
        ctx.steps_launch()
    else:
        for s in range(steps):
            pcc.collide(ctx, *args, 3 + s, mask=mask, ledger=ledger)
            for k in ("em", "ep", "ph"):
                pcc.append_secondaries(ctx, wl.n_cells, dev[k])
    n = pcc.launch_count() - n0
    status, stats = ctx.read_status()
    out = {k: {f: getattr(dev[k], f).cpu().numpy() for f in ("ux", "uy", "uz", "w", "pid", "cell_start", "cell_count",
                                                            "cell_added")} for k in ("em", "ep", "ph")}
    if with_x:
        for k in out:
            out[k]["x"] = dev[k].x.cpu().numpy()
    led = ledger.cpu().numpy().astype(np.float64)
    ctx.close()
    return n, status, stats, out, led


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("law,n_cells,with_x", [("mixed", 1500, True), ("mixed", 33, False), ("ions", 700, False),
                                                ("dense", 64, True)])
@pytest.mark.parametrize("groups", [0, 0x100, 0x200 | 0x400])
def test_same_bits_as_the_general_sequence(pcc, law, n_cells, with_x, graph, groups):
    wl = workload(law, n_cells, 5 + n_cells, with_x)
    mask = 7 | groups
    steps = 2
    na, st_a, a_stats, a, la = run(pcc, wl, law, with_x, True, graph, mask, steps)
    nb, st_b, b_stats, b, lb = run(pcc, wl, law, with_x, False, graph, mask, steps)
    assert na < nb                                   # the two paths really differ
    assert st_a == st_b and not st_a & pcc.ST_CAPACITY   # (what an overflow drops depends on the order of atomics)
    assert sum(b_stats["created"]) > (5 if groups != 0x600 else -1)
    for f in ("pairs", "accepted", "created", "candidates"):
        assert a_stats[f] == b_stats[f], f
    # sums over events in FP64 in another order
    np.testing.assert_allclose(a_stats["energy_change"], b_stats["energy_change"], rtol=1e-9)
    for k in a:
        for f in a[k]:
            assert np.array_equal(a[k][f], b[k][f]), (k, f)
    for c in (0, 2):                                 # a cell's events are added in FP32 in another order
        np.testing.assert_allclose(la[:, c] - la[:, c + 1], lb[:, c] - lb[:, c + 1], rtol=1e-5)
