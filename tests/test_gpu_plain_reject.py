"""The plain FP64 path evaluates a pair in full only where its accept digit or
its energy can matter: the same events, counters and status bits as the oracle,
which evaluates every pair, for energies on both sides of the table's end, ions
at rest, fast and relativistic, both pairing cases and steps from far too short
for an event to long enough that every pair collides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

SPEC = dict(n_rows=48, n_cols=48, gamma_max=300.0)


@pytest.fixture(scope="module")
def pcc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    return pcc


@pytest.mark.parametrize("dt", [1e-20, 2e-16, 1e-14, 1e-9])
@pytest.mark.parametrize("ion_u", [0.0, 0.3, 4.0])
@pytest.mark.parametrize("ne,ni", [(70, 20), (9, 40)])
def test_same_as_evaluating_every_pair(pcc, orc, dt, ion_u, ne, ni):
    # mean kinetic energies around the end of the tables / the boost of fast ions
    wl = W.solid_cu(n_cells=12, e_per_cell=ne, i_per_cell=ni, photons_per_cell=ne // 2, seed=31, dt=dt,
                    T_mev=60.0 / (1.0 + 6.0 * ion_u))
    rng = np.random.default_rng(8)
    ion = wl.species["ion"]
    v = rng.normal(size=(3, len(ion["w"])))
    v *= ion_u / np.sqrt((v ** 2).sum(0))
    for k, x in zip(("ux", "uy", "uz"), v):
        ion[k] = x.astype(np.float32)
    for k in ("em", "ph"):                    # one cell far above the tables, one clearly below
        d = wl.species[k]
        for c in ("ux", "uy", "uz"):
            d[c] = np.where(d["cell"] == 3, d[c] * 20, np.where(d["cell"] == 4, d[c] * 0.05, d[c])).astype(np.float32)
    m = wl.materials[0]
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(m.Z, m.Zstar, m.n_i, m.T_e)], pcc.table_spec(**SPEC))
    dev = {}
    for name, d in wl.species.items():
        sp = pcc.DeviceSpecies.empty(wl.n_cells, len(d["w"]) + 800 * wl.n_cells)
        pcc.bin(ctx, pcc.particles_to_device(d), wl.n_cells, sp, slack_abs=700, slack_rel=0.0)
        dev[name] = sp
    mat = torch.as_tensor(wl.material_of_cell, device="cuda")
    pcc.collide(ctx, wl.n_cells, mat, wl.ion_mass, dev["em"], dev["ep"], dev["ph"], dev["ion"], wl.dt, wl.seed, 0,
                precision=pcc.FP64_PLAIN)
    for k in ("em", "ep", "ph"):
        pcc.append_secondaries(ctx, wl.n_cells, dev[k])
    status, stats = ctx.read_status()
    T = orc.OracleTables([orc.material(m.Z, m.Zstar, m.n_i, m.T_e)], orc.table_spec(**SPEC))
    sp = {k: orc.OracleSpecies(v, cap=len(v["w"]) + 20000) for k, v in wl.species.items()}
    _, ost = orc.step(T, wl.n_cells, wl.material_of_cell, sp["em"], sp["ep"], sp["ph"], sp["ion"], wl.ion_mass, wl.dt,
                      wl.seed, 0)
    assert status == int(ost["status"])
    assert stats["pairs"] == [int(x) for x in ost["pairs"]]
    assert stats["accepted"] == [int(x) for x in ost["accepted"]]
    assert stats["created"] == [int(x) for x in ost["created"]]
    for k in ("em", "ep", "ph"):
        g, o = dev[k].live_host(), sp[k].canonical()
        assert np.array_equal(g["pid"], o["pid"]) and np.array_equal(g["cell"], o["cell"]), k
        np.testing.assert_allclose(g["ux"], o["ux"], rtol=1e-5, atol=1e-6)
    ctx.close()
