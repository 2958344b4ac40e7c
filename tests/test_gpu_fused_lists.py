"""The one-kernel step where candidates are many: more than a warp stages in shared
memory, and long lists in cells with N_p < N_t, which the block works off together
or a second kernel spreads over the chip; few projectiles with many pairs each; and
slots beyond what a staged candidate can name.  The same bits as the general
sequence."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

DEFAULT_POLLS = 1 << 22
FIELDS = ("ux", "uy", "uz", "w", "x", "pid", "cell_count", "cell_added")


@pytest.fixture(scope="module")
def pcc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    return pcc


def workload(law, n):
    rng = np.random.default_rng(len(law) + n)
    if law == "many":        # N_p >= N_t, thousands of candidates a cell
        ne, ni, ng, npos = (rng.integers(lo, hi, n) for lo, hi in ((3000, 9000), (10, 200), (1500, 6000), (500, 2500)))
    elif law == "ions":      # N_p < N_t, from one projectile to thousands
        ne, ng, npos = rng.integers(1, 3000, n), rng.integers(1, 1500, n), rng.integers(1, 40, n)
        ni = rng.integers(3000, 6000, n)
    else:                    # list lengths on both sides of every limit
        ne, ni, ng, npos = (rng.choice([0, 1, 7, 33, 64, 129, 500, 1024, 4100], n) for _ in range(4))
    wl = W.solid_cu(n_cells=n, e_per_cell=ne, i_per_cell=ni, photons_per_cell=ng, seed=n, dt=2e-13, T_mev=20.0)
    wl.species["ep"] = W.solid_cu(n_cells=n, e_per_cell=npos, i_per_cell=1, seed=n + 1, T_mev=20.0).species["em"]
    em = wl.species["em"]
    em["w"] = (em["w"] * 10.0 ** rng.uniform(-1, 1, len(em["w"]))).astype(np.float32)
    for d in wl.species.values():
        d["x"] = rng.uniform(0, 1, len(d["w"])).astype(np.float32)
    return wl


def run(pcc, wl, fused, graph):
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(29, 5.0, 8.5e28, 100.0)], pcc.table_spec(n_rows=63, n_cols=65))
    dev = {}
    for name, d in wl.species.items():
        sp = pcc.DeviceSpecies.empty(wl.n_cells, 2 * len(d["w"]) + 6001 * wl.n_cells, with_x=True)
        pcc.bin(ctx, pcc.particles_to_device(d), wl.n_cells, sp, slack_abs=6000, slack_rel=0.5)
        dev[name] = sp
    mat = torch.zeros(wl.n_cells, dtype=torch.int32, device="cuda")
    ctx.read_status()
    if not fused:
        ctx.set_wait_limit(DEFAULT_POLLS - 1)     # a context with a wait limit of its own keeps the staged sequence
    n0 = pcc.launch_count()
    args = (wl.n_cells, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, 77)
    if graph:
        ctx.steps_capture(*args, 3, 2)
        ctx.steps_launch()
    else:
        for s in range(2):
            pcc.collide(ctx, *args, 3 + s)
            for k in ("em", "ep", "ph"):
                pcc.append_secondaries(ctx, wl.n_cells, dev[k])
    n = pcc.launch_count() - n0
    status, stats = ctx.read_status()
    out = {k: {f: getattr(dev[k], f).cpu().numpy() for f in FIELDS} for k in ("em", "ep", "ph")}
    ctx.close()
    return n, status, stats, out


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("law,n_cells", [("many", 40), ("ions", 40), ("edges", 70), ("many", 17), ("ions", 31),
                                         ("many", 100), ("ions", 120), ("edges", 900)])
def test_long_lists(pcc, law, n_cells, graph):
    wl = workload(law, n_cells)
    na, st_a, a_stats, a = run(pcc, wl, True, graph)
    nb, st_b, b_stats, b = run(pcc, wl, False, graph)
    # beyond a cell for every other SM the long lists are left to a second kernel
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert na == (2 if 2 * n_cells <= sms else 4) + (0 if graph else 6) < nb and st_a == st_b and not st_a & pcc.ST_CAPACITY
    for f in ("pairs", "accepted", "created", "candidates"):
        assert a_stats[f] == b_stats[f], f
    assert min(a_stats["candidates"]) > 1000 and min(a_stats["created"][0], a_stats["created"][4]) > 20
    for k in a:
        for f in FIELDS:
            assert np.array_equal(a[k][f], b[k][f]), (k, f)


@pytest.mark.parametrize("blocks_per_sm", [1, 2])
def test_grid_cap(pcc, blocks_per_sm):
    """pcc_set_schedule's cap on the grid: warps take more cells each, in several batches; the same bits."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 8 * 8 * sms + 77                            # more than a batch of eight cells for each warp of one block per SM
    wl = W.solid_cu(n_cells=n, e_per_cell=30, i_per_cell=7, photons_per_cell=9, seed=3, dt=1e-15, T_mev=20.0)
    out = []
    for cap in (0, blocks_per_sm):
        ctx = pcc.Context(0)
        ctx.tables_build([pcc.material(29, 5.0, 8.5e28, 100.0)], pcc.table_spec(n_rows=63, n_cols=65))
        ctx.set_schedule(4, cap)
        dev = {}
        for name, d in wl.species.items():
            dev[name] = pcc.DeviceSpecies.empty(n, len(d["w"]) + 31 * n)
            pcc.bin(ctx, pcc.particles_to_device(d), n, dev[name], slack_abs=30, slack_rel=0.0)
        mat = torch.zeros(n, dtype=torch.int32, device="cuda")
        n0 = pcc.launch_count()
        ctx.steps_capture(n, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, 5, 0, 3)
        ctx.steps_launch()
        _, stats = ctx.read_status()
        assert pcc.launch_count() - n0 == 3 and stats["created"][0] > 50
        out.append((stats, {k: [getattr(dev[k], f) for f in FIELDS if f != "x"] for k in ("em", "ep", "ph")}))
        ctx.close()
    for f in ("pairs", "accepted", "created", "candidates"):
        assert out[0][0][f] == out[1][0][f]
    for k in ("em", "ep", "ph"):
        assert all(torch.equal(x, y) for x, y in zip(out[0][1][k], out[1][1][k])), k


def test_slots_beyond_a_staged_candidate(pcc):
    """A cell of 2^27 + 2^25 electrons: the same electrons change on both paths."""
    n_cells, big = 33, (1 << 27) + (1 << 25)
    ne = np.full(n_cells, 50)
    ne[5] = big
    start = np.concatenate([[0], np.cumsum(ne)]).astype(np.int32)
    gen = torch.Generator(device="cuda")

    def species(counts, room, scale, w):
        cap = int(counts.sum() + room * n_cells)
        sp = pcc.DeviceSpecies.empty(n_cells, cap)
        st = torch.as_tensor(np.concatenate([[0], np.cumsum(counts + room)]).astype(np.int32), device="cuda")
        sp.cell_start.copy_(st)
        sp.cell_count.copy_(torch.as_tensor(counts.astype(np.int32), device="cuda"))
        gen.manual_seed(3)
        for f in ("ux", "uy", "uz"):
            getattr(sp, f).copy_(torch.randn(cap, device="cuda", generator=gen) * scale)
        sp.w.fill_(w)
        torch.arange(cap, out=sp.pid)
        return sp

    res = []
    for fused in (True, False):
        ctx = pcc.Context(0)
        ctx.tables_build([pcc.material(29, 5.0, 8.5e28, 100.0)], pcc.table_spec(n_rows=32, n_cols=32))
        if not fused:
            ctx.set_wait_limit(DEFAULT_POLLS - 1)
        none = np.zeros(n_cells, np.int64)
        em, ion = species(ne, 0, 10.0, 1e20), species(np.full(n_cells, 8), 0, 1e-3, 8.5e28 / 8)
        ep, ph = species(none, 4, 0.0, 0.0), species(none, 200000, 0.0, 0.0)
        pcc.collide(ctx, n_cells, torch.zeros(n_cells, dtype=torch.int32, device="cuda"), W.MASS_CU, em, ep, ph, ion, 3e-16, 5, 0,
                    mask=pcc.BREMS)
        status, stats = ctx.read_status()
        assert not status & pcc.ST_CAPACITY and stats["created"][0] > 1000
        res.append((stats["candidates"], stats["accepted"], em.ux, em.uz))
        ctx.close()
    assert res[0][:2] == res[1][:2]
    gen.manual_seed(3)
    before = torch.randn(res[0][2].numel(), device="cuda", generator=gen) * 10.0
    assert int((res[0][2] != before)[int(start[5]) + (1 << 27):].sum()) > 100
    assert torch.equal(res[0][2], res[1][2]) and torch.equal(res[0][3], res[1][3])
