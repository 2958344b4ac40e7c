"""Unequal ion weights in cells of fewer ions than a scan's lane group: the positron
and photon groups of a call (which may take the ion sums from the electron scan)
against the oracle, on the general sequence and on the one-kernel step, with
enough events in each group to see a wrong coefficient."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1907_02814_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

DEFAULT_POLLS = 1 << 22
SPEC = dict(n_rows=64, n_cols=64)


def workload():
    n, rng = 75, np.random.default_rng(17)
    wl = W.solid_cu(n_cells=n, e_per_cell=rng.integers(1, 500, n), i_per_cell=rng.integers(2, 9, n),
                    photons_per_cell=rng.integers(20, 400, n), seed=41, dt=2e-12, T_mev=30.0)
    wl.species["ep"] = W.solid_cu(n_cells=n, e_per_cell=rng.integers(20, 300, n), i_per_cell=1, seed=42, T_mev=30.0).species["em"]
    ion = wl.species["ion"]
    ion["w"] = (ion["w"] * 10.0 ** rng.uniform(-1, 1, len(ion["w"]))).astype(np.float32)
    for k in ("em", "ep", "ph"):
        d = wl.species[k]
        d["w"] = (d["w"] * rng.uniform(0.3, 3.0, len(d["w"]))).astype(np.float32)
    return wl


@pytest.mark.parametrize("general", [True, False])
def test_coefficients_of_all_groups(orc, general):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    wl = workload()
    n, m = wl.n_cells, wl.materials[0]
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(m.Z, m.Zstar, m.n_i, m.T_e)], pcc.table_spec(**SPEC))
    if general:
        ctx.set_wait_limit(DEFAULT_POLLS - 1)     # a context with a wait limit of its own keeps the staged sequence
    dev = {}
    for name, d in wl.species.items():
        sp = pcc.DeviceSpecies.empty(n, len(d["w"]) + 2000 * n)
        pcc.bin(ctx, pcc.particles_to_device(d), n, sp, slack_abs=2000, slack_rel=0.0)
        dev[name] = sp
    ctx.read_status()
    n0 = pcc.launch_count()
    pcc.collide(ctx, n, torch.as_tensor(wl.material_of_cell, device="cuda"), wl.ion_mass, dev["em"], dev["ep"], dev["ph"],
                dev["ion"], wl.dt, wl.seed, 0)
    assert (pcc.launch_count() - n0 > 1) == general
    for k in ("em", "ep", "ph"):
        pcc.append_secondaries(ctx, n, dev[k])
    status, stats = ctx.read_status()
    T = orc.OracleTables([orc.material(m.Z, m.Zstar, m.n_i, m.T_e)], orc.table_spec(**SPEC))
    sp = {k: orc.OracleSpecies(v, cap=len(v["w"]) + 400000) for k, v in wl.species.items()}
    _, st = orc.step(T, n, wl.material_of_cell, sp["em"], sp["ep"], sp["ph"], sp["ion"], wl.ion_mass, wl.dt, wl.seed, 0)
    assert status & (pcc.ST_CAPACITY | pcc.ST_NONFINITE) == 0
    assert stats["pairs"] == [int(v) for v in st["pairs"]]
    created = [int(v) for v in st["created"]]
    assert created[1] > 100 and created[4] > 100              # positron Bremsstrahlung, Bethe-Heitler
    # decisions within FP32 rounding of their threshold, as in the batched path's other comparisons
    mism = sum(len(set(dev[k].live_host()["pid"].tolist()) ^ set(sp[k].canonical()["pid"].tolist())) for k in ("em", "ep", "ph"))
    assert mism <= max(2, 1e-5 * sum(stats["pairs"])), (mism, stats["created"], created)
    ctx.close()
