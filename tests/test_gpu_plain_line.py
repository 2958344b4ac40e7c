"""The plain FP64 path on both sides of the cell count from which it takes blocks of 64
threads: the oracle's events, counters, momenta and ledger over cells whose lists end
at, before and behind a warp or a block, with uniform and with uneven ion weights."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

SPEC = dict(n_rows=48, n_cols=48)
SIZES = np.array([0, 1, 5, 31, 32, 33, 63, 64, 65, 127, 128, 129, 300])


@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("uneven", [False, True])
def test_block_sizes_at_the_line(orc, more, uneven):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    n = 96 * torch.cuda.get_device_properties(0).multi_processor_count + more
    rng = np.random.default_rng(5)
    e, i = rng.integers(0, 6, n), rng.integers(0, 4, n)
    e[:600], i[:600] = rng.choice(SIZES, 600), rng.choice(SIZES, 600)
    wl = W.solid_cu(n_cells=n, e_per_cell=e, i_per_cell=i, photons_per_cell=e[::-1] // 2 + 1, seed=37, dt=3e-14, T_mev=20.0)
    if uneven:
        ion = wl.species["ion"]
        ion["w"] = (ion["w"] * rng.choice([0.5, 1.0, 2.0], len(ion["w"]))).astype(np.float32)
    m = wl.materials[0]
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(m.Z, m.Zstar, m.n_i, m.T_e)], pcc.table_spec(**SPEC))
    dev = {}
    for name, d in wl.species.items():
        sp = pcc.DeviceSpecies.empty(n, len(d["w"]) + 150 * n)
        pcc.bin(ctx, pcc.particles_to_device(d), n, sp, slack_abs=150, slack_rel=0.0)
        dev[name] = sp
    ledger = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
    pcc.collide(ctx, n, torch.as_tensor(wl.material_of_cell, device="cuda"), wl.ion_mass, dev["em"], dev["ep"], dev["ph"],
                dev["ion"], wl.dt, wl.seed, 0, precision=pcc.FP64_PLAIN, ledger=ledger)
    for k in ("em", "ep", "ph"):
        pcc.append_secondaries(ctx, n, dev[k])
    status, stats = ctx.read_status()
    T = orc.OracleTables([orc.material(m.Z, m.Zstar, m.n_i, m.T_e)], orc.table_spec(**SPEC))
    sp = {k: orc.OracleSpecies(v, cap=len(v["w"]) + 200000) for k, v in wl.species.items()}
    ol = np.zeros((n, 2))
    _, ost = orc.step(T, n, wl.material_of_cell, sp["em"], sp["ep"], sp["ph"], sp["ion"], wl.ion_mass, wl.dt, wl.seed, 0, 7, ol)
    assert status == int(ost["status"]) and sum(stats["created"]) > 50
    for k in ("pairs", "accepted", "created"):
        assert stats[k] == [int(x) for x in ost[k]]
    for k in ("em", "ep", "ph"):
        g, o = dev[k].live_host(), sp[k].canonical()
        assert np.array_equal(g["pid"], o["pid"]) and np.array_equal(g["cell"], o["cell"]), k
        assert np.array_equal(g["w"], o["w"]), k
        for f in ("ux", "uy", "uz"):   # float32 storage
            np.testing.assert_allclose(g[f], o[f], rtol=2e-6, atol=1e-6, err_msg=k)
    led = ledger.cpu().numpy().astype(np.float64)
    for q in (0, 1):                   # float32 contributions of a cell, added in float32
        np.testing.assert_allclose(led[:, 2 * q] - led[:, 2 * q + 1], ol[:, q], rtol=2e-6, atol=1e-30)
    ctx.close()
