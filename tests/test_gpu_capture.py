"""Calls inside a caller's stream capture, where the library cannot allocate: after a
warm call that went the other way (one kernel or the general sequence), on
fewer or more cells, on a stream that joins another; a graph's buffers stay when a
later call goes the other way; binning a growing species allocates once."""
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


def context(pcc):
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(29, 5.0, 8.5e28, 100.0)], pcc.table_spec(n_rows=32, n_cols=32))
    return ctx


def cells(pcc, ctx, n):
    wl = W.solid_cu(n_cells=n, e_per_cell=200, i_per_cell=40, photons_per_cell=50, seed=5, dt=2e-15, T_mev=10.0)
    dev = {}
    for name, d in wl.species.items():
        sp = pcc.DeviceSpecies.empty(n, len(d["w"]) + 200 * n)
        pcc.bin(ctx, pcc.particles_to_device(d), n, sp, slack_abs=200, slack_rel=0.0)
        dev[name] = sp
    return wl, dev, torch.zeros(n, dtype=torch.int32, device="cuda")


def collide(pcc, ctx, wl, dev, mat, step=0, **kw):
    pcc.collide(ctx, wl.n_cells, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, 7, step, **kw)


def capture(work):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        work()
    return g


def used():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("how", ["fewer cells", "wait limit"])
def test_collide_captured_after_the_other_way(pcc, how):
    ctx, ref = context(pcc), context(pcc)
    warm = cells(pcc, ctx, 64)
    n = 16 if how == "fewer cells" else 64
    wl, dev, mat = cells(pcc, ctx, n)
    rl, rdev, rmat = cells(pcc, ref, n)
    n0 = pcc.launch_count()
    collide(pcc, ctx, *warm)
    assert pcc.launch_count() - n0 == 1                     # one kernel
    if how == "wait limit":
        ctx.set_wait_limit(DEFAULT_POLLS - 1)
    n0 = pcc.launch_count()
    g = capture(lambda: collide(pcc, ctx, wl, dev, mat))
    assert pcc.launch_count() - n0 == 15                    # the general sequence
    g.replay()
    collide(pcc, ref, rl, rdev, rmat)
    torch.cuda.synchronize()
    for k in ("em", "ep", "ph"):
        assert torch.equal(dev[k].cell_added, rdev[k].cell_added)
    assert torch.equal(dev["em"].ux, rdev["em"].ux) and int(dev["ph"].cell_added.sum()) > 0
    ctx.close()
    ref.close()


def test_totals_captured_on_more_cells(pcc):
    ctx, ctx2 = context(pcc), context(pcc)
    _, small, _ = cells(pcc, ctx2, 8)                       # binned elsewhere: this context has no scratch yet
    _, big, _ = cells(pcc, ctx2, 4000)
    pcc.totals(ctx, 8, small["em"])
    out = []
    g = capture(lambda: out.append(pcc.totals(ctx, 4000, big["em"])))
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out[0].cpu().numpy(), pcc.totals(ctx2, 4000, big["em"]).cpu().numpy())
    ctx.close()
    ctx2.close()


def test_chained_kernels_after_a_join(pcc):
    """The captured stream has just joined another one, so that the first kernel depends on two."""
    ctx, ref = context(pcc), context(pcc)
    (wl, dev, mat), (rl, rdev, rmat) = cells(pcc, ctx, 20), cells(pcc, ref, 20)
    pcc.totals(ctx, 20, dev["em"])
    x = torch.zeros(1 << 20, device="cuda")
    y = torch.zeros(8, device="cuda")
    side, out = torch.cuda.Stream(), []

    def work():
        main = torch.cuda.current_stream()
        x.add_(1.0)
        for call in (lambda: collide(pcc, ctx, wl, dev, mat, precision=pcc.FP64_PLAIN),
                     lambda: [pcc.append_secondaries(ctx, 20, dev[k]) for k in ("em", "ep", "ph")],
                     lambda: out.append(pcc.totals(ctx, 20, dev["ph"], is_photon=True))):
            side.wait_stream(main)
            with torch.cuda.stream(side):
                x.mul_(2.0)
            y.add_(1.0)
            main.wait_stream(side)
            call()

    g = capture(work)
    g.replay()
    collide(pcc, ref, rl, rdev, rmat, precision=pcc.FP64_PLAIN)
    for k in ("em", "ep", "ph"):
        pcc.append_secondaries(ref, 20, rdev[k])
    want = pcc.totals(ref, 20, rdev["ph"], is_photon=True)
    torch.cuda.synchronize()
    assert float(x[5]) == 8.0 and torch.equal(dev["em"].ux, rdev["em"].ux) and torch.equal(dev["ph"].pid, rdev["ph"].pid)
    np.testing.assert_array_equal(out[0].cpu().numpy(), want.cpu().numpy())
    ctx.close()
    ref.close()


def test_graph_keeps_its_buffers_when_a_call_goes_the_other_way(pcc):
    ctx = context(pcc)
    wl, dev, mat = cells(pcc, ctx, 64)
    args = (64, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, 7)
    ctx.steps_capture(*args, 0, 2, timing=True)             # the general sequence
    before = used()
    collide(pcc, ctx, wl, dev, mat, 9)                      # one kernel
    assert used() == before                                 # nothing was freed or made
    ctx.steps_launch()
    status, stats = ctx.read_status()
    assert not status & pcc.ST_CAPACITY and sum(stats["created"]) > 0
    ctx.close()


def test_binning_a_growing_species_allocates_once(pcc):
    ctx = context(pcc)
    n_cells, cap = 500, 4_000_000
    sp = pcc.DeviceSpecies.empty(n_cells, cap)
    rng = np.random.default_rng(2)
    parts = []
    for n in (1000, 200_000, 1_000_000, 2_500_000):
        f = rng.normal(size=n).astype(np.float32)
        parts.append(pcc.particles_to_device({"ux": f, "uy": f, "uz": f, "w": np.ones(n, np.float32), "x": None,
                                              "pid": np.arange(n, dtype=np.uint64), "cell": rng.integers(0, n_cells, n).astype(np.int32)}))
    pcc.bin(ctx, parts[0], n_cells, sp, slack_abs=1, slack_rel=0.0)
    before = used()
    for p in parts[1:]:
        pcc.bin(ctx, p, n_cells, sp, slack_abs=1, slack_rel=0.0)
        assert used() == before
    ctx.close()
