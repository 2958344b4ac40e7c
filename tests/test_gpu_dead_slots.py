"""The whole photon arrays after a step, slots behind the live particles
included: photons are removed and emitted in the same cells, and what the removal
leaves behind the live records (absorbed and moved photons, then copies of the
emitted ones in id order) follows from the state alone, on all three paths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

FIELDS = ("ux", "uy", "uz", "w", "x", "pid")


def arrays(sp):
    return {f: getattr(sp, f).cpu().numpy() for f in FIELDS}


def expected(before, start, count, after, new_count):
    """The photon arrays that one step leaves, from the live records it leaves."""
    out = {f: v.copy() for f, v in before.items()}
    both = 0
    for c in range(len(count)):
        a, n, m = start[c], count[c], new_count[c]
        made = ~np.isin(after["pid"][a:a + m], before["pid"][a:a + n])
        kept = int(m - made.sum())
        new = {f: after[f][a + kept:a + m] for f in FIELDS}
        assert not made[:kept].any() and np.all(np.diff(new["pid"]) > 0)
        gone = ~np.isin(before["pid"][a:a + n], after["pid"][a:a + kept])
        assert gone.sum() == n - kept
        both += bool(gone.any() and len(new["pid"]) > 1)
        out["w"][a:a + n][gone] = 0.0
        for f in FIELDS:
            out[f][a + n:a + n + len(new["pid"])] = new[f]     # emitted, in id order
            live = np.concatenate([before[f][a:a + n][~gone], new[f]])
            out[f][a:a + m] = live                              # moved down; what lies behind stays
    return out, both


@pytest.mark.parametrize("n_cells,precision", [(16, "fp32"), (64, "fp32"), (40, "fp64")])
def test_photon_slots_follow_from_the_state(n_cells, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    rng = np.random.default_rng(3)
    ne = rng.integers(200, 900, n_cells)
    wl = W.solid_cu(n_cells=n_cells, e_per_cell=ne, i_per_cell=rng.integers(20, 400, n_cells),
                    photons_per_cell=rng.integers(100, 600, n_cells), seed=9, dt=1e-12, T_mev=30.0)
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(29, 5.0, 8.5e28, 100.0)], pcc.table_spec(n_rows=48, n_cols=48))
    dev = {}
    for name, d in wl.species.items():
        d["x"] = rng.uniform(0, 1, len(d["w"])).astype(np.float32)
        sp = pcc.DeviceSpecies.empty(n_cells, len(d["w"]) + 2500 * n_cells, with_x=True)
        pcc.bin(ctx, pcc.particles_to_device(d), n_cells, sp, slack_abs=2000, slack_rel=0.0)
        dev[name] = sp
    mat = torch.as_tensor(wl.material_of_cell, device="cuda")
    ctx.read_status()
    both = 0
    for step in range(3):
        before, count = arrays(dev["ph"]), dev["ph"].cell_count.cpu().numpy()
        pcc.collide(ctx, n_cells, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, wl.seed, step,
                    precision=pcc.FP64_PLAIN if precision == "fp64" else pcc.FP32_BATCHED)
        for k in ("em", "ep", "ph"):
            pcc.append_secondaries(ctx, n_cells, dev[k])
        status, _ = ctx.read_status()
        assert not status & pcc.ST_CAPACITY
        after = arrays(dev["ph"])
        want, n = expected(before, dev["ph"].cell_start.cpu().numpy(), count, after, dev["ph"].cell_count.cpu().numpy())
        both += n
        for f in FIELDS:
            assert np.array_equal(after[f], want[f]), (step, f)
    assert both >= 20                                           # cells that removed photons and emitted several
    ctx.close()
