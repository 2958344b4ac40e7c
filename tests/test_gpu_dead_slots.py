"""The whole photon arrays after a step, slots behind the live particles
included: photons are removed and emitted in the same cells, and what the removal
leaves behind the live records (absorbed and moved photons, then copies of the last
emitted ones, in the order in which the scan marks their pairs, of more than 32 in
id order) follows from the state alone, on all three paths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

FIELDS = ("ux", "uy", "uz", "w", "x", "pid")


def arrays(sp):
    return {f: getattr(sp, f).cpu().numpy() for f in FIELDS}


def lane_group(thr, n):
    """Lanes that scan a cell of n pairs: its size class, two per octave, against the thresholds."""
    b = n.bit_length()
    cls = 0 if b < 2 else 2 * (b - 1) + (n >= 3 << (b - 2))
    return next((g for g, t in zip((32, 16, 8, 4), thr) if cls >= t), 2)


def scan_order(pid, n_p, n_t, slot_of_pair, thr, plain):
    """Sort key of an emitted photon: its projectile group, then its pair's place in the scan."""
    ep, j = (pid >> 41) & 7, (pid >> 1) & 0xFFFF
    n_p, G = n_p[ep], lane_group(thr[ep], max(n_p[ep], n_t))
    if n_p < n_t:
        m, s = divmod(j, n_p)
        i = m * -(-n_p // 4) + s // 4
        return ep, j if plain else (i // G, s % 4, i % G)
    s = slot_of_pair[ep][j]
    it = s // (4 * G)
    return ep, s if plain else (it // 8, s // 4 % G, it % 8, s % 4)


def expected(before, start, count, after, new_count, key):
    """The photon arrays that one step leaves, from the live records it leaves."""
    out = {f: v.copy() for f, v in before.items()}
    both = [0, 0]
    for c in range(len(count)):
        a, n, m = start[c], count[c], new_count[c]
        made = ~np.isin(after["pid"][a:a + m], before["pid"][a:a + n])
        kept = int(m - made.sum())
        new = {f: after[f][a + kept:a + m] for f in FIELDS}
        assert not made[:kept].any() and np.all(np.diff(new["pid"]) > 0)
        gone = ~np.isin(before["pid"][a:a + n], after["pid"][a:a + kept])
        assert gone.sum() == n - kept
        k = len(new["pid"])
        if gone.any() and k > 1:
            both[k > 32] += 1
        order = range(k) if k > 32 else sorted(range(k), key=lambda q: key(c, int(new["pid"][q])))
        out["w"][a:a + n][gone] = 0.0
        for f in FIELDS:
            out[f][a + n:a + n + k] = new[f][list(order)]      # emitted
            out[f][a:a + m] = np.concatenate([before[f][a:a + n][~gone], new[f]])   # moved down; what lies behind stays
    return out, np.array(both)


@pytest.mark.parametrize("electrons,photons", [((200, 900), (100, 600)), ((5, 40), (1000, 3000))])
@pytest.mark.parametrize("n_cells,precision", [(16, "fp32"), (64, "fp32"), (40, "fp64")])
def test_photon_slots_follow_from_the_state(n_cells, precision, electrons, photons):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    rng = np.random.default_rng(3)
    wl = W.solid_cu(n_cells=n_cells, e_per_cell=rng.integers(*electrons, n_cells), i_per_cell=rng.integers(2, 400, n_cells),
                    photons_per_cell=rng.integers(*photons, n_cells), seed=9, dt=1e-12, T_mev=30.0)
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(29, 5.0, 8.5e28, 100.0)], pcc.table_spec(n_rows=48, n_cols=48))
    dev = {}
    for name, d in wl.species.items():
        d["x"] = rng.uniform(0, 1, len(d["w"])).astype(np.float32)
        sp = pcc.DeviceSpecies.empty(n_cells, len(d["w"]) + 2500 * n_cells, with_x=True)
        pcc.bin(ctx, pcc.particles_to_device(d), n_cells, sp, slack_abs=2000, slack_rel=0.0)
        dev[name] = sp
    mat = torch.as_tensor(wl.material_of_cell, device="cuda")
    thr = [ctx.scan_classes(0), ctx.scan_classes(1)]
    n_t = dev["ion"].cell_count.cpu().numpy()
    ctx.read_status()
    both = 0
    for step in range(3):
        before, count = arrays(dev["ph"]), dev["ph"].cell_count.cpu().numpy()
        lept = []
        for g, k in enumerate(("em", "ep")):
            j = pcc.pairing(ctx, n_cells, dev[k], dev["ion"], g, wl.seed, step)[0].cpu().numpy()
            lept.append((dev[k].cell_start.cpu().numpy(), dev[k].cell_count.cpu().numpy(), j))

        def key(c, pid):
            n_p = [int(l[1][c]) for l in lept]
            inv = [dict(zip(l[2][l[0][c]:l[0][c] + l[1][c]].tolist(), range(l[1][c]))) for l in lept]
            return scan_order(pid, n_p, int(n_t[c]), inv, thr, precision == "fp64")

        pcc.collide(ctx, n_cells, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, wl.seed, step,
                    precision=pcc.FP64_PLAIN if precision == "fp64" else pcc.FP32_BATCHED)
        for k in ("em", "ep", "ph"):
            pcc.append_secondaries(ctx, n_cells, dev[k])
        status, _ = ctx.read_status()
        assert not status & pcc.ST_CAPACITY
        after = arrays(dev["ph"])
        want, n = expected(before, dev["ph"].cell_start.cpu().numpy(), count, after, dev["ph"].cell_count.cpu().numpy(), key)
        both = both + n
        for f in FIELDS:
            assert np.array_equal(after[f], want[f]), (step, f)
    assert both.sum() >= 20                                     # cells that removed photons and emitted several
    ctx.close()
