"""FP64 path, cells of one electron and two ions that move against each other: after
radiating against the first ion the electron can have more energy in the
simulation frame than before, and its second pair lies above the tables.  The
status word equals the oracle's, which evaluates every pair."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SPEC = dict(n_rows=48, n_cols=48, gamma_max=41.0)
N, MASS, DT = 200000, 196.97 * 1822.9, 5e-16


def species():
    f = lambda v: np.asarray(v, np.float32)
    def make(ux, uy, w, cell):
        n = len(cell)
        return {"ux": f(ux), "uy": f(uy), "uz": np.zeros(n, np.float32), "w": f(w), "pid": np.arange(n, dtype=np.uint64),
                "cell": np.asarray(cell, np.int32)}
    em = make(np.full(N, 1.73), np.zeros(N), np.full(N, 1e28), np.arange(N))
    ion = make(np.tile([10.0, -10.0], N), np.zeros(2 * N), np.full(2 * N, 2.95e28), np.repeat(np.arange(N), 2))
    none = make([], [], [], [])
    return {"em": em, "ep": none, "ph": none, "ion": ion}


def test_status_after_a_gain_of_energy(orc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(79, 20.0, 5.9e28, 1000.0)], pcc.table_spec(**SPEC))
    T = orc.OracleTables([orc.material(79, 20.0, 5.9e28, 1000.0)], orc.table_spec(**SPEC))
    mat = torch.zeros(N, dtype=torch.int32, device="cuda")
    seen = 0
    for seed in range(1, 13):
        dev = {}
        for name, d in species().items():
            sp = pcc.DeviceSpecies.empty(N, len(d["w"]) + 8 * N)
            pcc.bin(ctx, pcc.particles_to_device(d), N, sp, slack_abs=8, slack_rel=0.0)
            dev[name] = sp
        ctx.read_status()
        pcc.collide(ctx, N, mat, MASS, dev["em"], dev["ep"], dev["ph"], dev["ion"], DT, seed, 0, mask=pcc.BREMS,
                    precision=pcc.FP64_PLAIN)
        status, stats = ctx.read_status()
        sp = {k: orc.OracleSpecies(v, cap=len(v["w"]) + 4 * N) for k, v in species().items()}
        _, st = orc.step(T, N, np.zeros(N, np.int32), sp["em"], sp["ep"], sp["ph"], sp["ion"], MASS, DT, seed, 0, 1)
        assert stats["accepted"] == [int(v) for v in st["accepted"]]
        assert status == int(st["status"]), seed
        seen += bool(status & pcc.ST_TABLE_RANGE)
    assert 0 < seen < 12        # with and without such a pair
    ctx.close()
