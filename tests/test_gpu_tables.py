"""Table rows over the shapes of the quadrature: node counts on both sides of the
lane-group widths, the fewest columns, odd and even column counts (the mirrored
half), more materials than a block takes, both screenings and momentum-transfer
bounds, mixed elements, and Thomas-Fermi and Debye lengths that nearly agree."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# both sides are FP64; the oracle's printed form of I2 cancels terms of size (L delta)^2
RTOL = 1e-7


def bethe_heitler_total(T, L, cols, nodes):
    """The Bethe-Heitler total for Z = 1 by the table's panels and nodes, the printed forms in 40 digits."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    L, T, N = mp.mpf(float(L)), mp.mpf(float(T)), cols - 1
    x, w = np.polynomial.legendre.leggauss(nodes)
    k, L2 = 2 + T, L * L

    def f(y):
        gp = 1 + y * T
        gm = k - gp
        d = k / (2 * gp * gm)
        at, ln = mp.atan(L * d) - mp.atan(L), mp.log((1 + L2) / (1 + L2 * d * d))
        i1 = L * d * at - L2 * (1 - d) ** 2 / (2 * (1 + L2)) + ln / 2
        i2 = (4 * L2 * L * d ** 3 * at + (1 + 3 * L2 * d * d) * ln + 6 * L2 * L2 * d * d / (1 + L2) * mp.log(d)
              + L2 * (d - 1) * (d + 1 - 4 * L2 * d * d) / (1 + L2)) / 2
        return ((gp * gp + gm * gm) * (i1 + 1) + 2 * gp * gm / 3 * (i2 + mp.mpf(5) / 6)) * T / k ** 3

    tot = mp.mpf(0)
    for c in range(N):
        a, b = mp.mpf(c) / N, mp.mpf(c + 1) / N
        g = [(b - a) * mp.mpf(4) ** -i for i in range(1, 13)]
        cuts = [a] + [b - v for v in g] + [b] if c == N - 1 else [a] + [a + v for v in reversed(g)] + [b] if c == 0 else [a, b]
        for lo, hi in zip(cuts[:-1], cuts[1:]):
            tot += (hi - lo) / 2 * sum(mp.mpf(v) * f((lo + hi) / 2 + (hi - lo) / 2 * mp.mpf(u)) for u, v in zip(x, w))
    return float(4 * mp.mpf("2.8179403262e-15") ** 2 * mp.mpf("7.2973525693e-3") * tot)


@pytest.mark.parametrize("rows,cols,nodes,kw", [
    (5, 3, 1, {}), (4, 4, 3, {}), (6, 5, 8, {}), (7, 33, 5, {}), (9, 64, 16, {}), (3, 130, 32, {}), (8, 40, 8, {"nr_qbounds": 1}),
    (6, 21, 8, {"screening": 1}), (5, 30, 4, {"screening": 1, "cutoff_exp": 20}), (4, 16, 6, {"gamma_max": 5.0}),
    (4, 16, 6, {"gamma_min": 3.0, "gamma_max": 1e6})])
def test_tables_against_the_oracle(orc, rows, cols, nodes, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    mats = [(29, 5.0, 8.5e28, 100.0), (79, 30.0, 5.9e28, 1000.0), (13, 0.0, 6e28, 10.0), (1, 1.0, 1e25, 10.0)]
    mats += [(73, float(z), 5.55e28, 10.0 ** (1 + z / 20)) for z in range(1, 7)]      # ten: two chunks
    scr = orc.screening(orc.material(29, 2.0, 1e28, 100.0)).as_dict()
    for off in (1e-8, 1e-3):         # Debye lengths shrunk to nearly the Thomas-Fermi length
        mats.append((29, 2.0, 1e28, 100.0, 1.0, scr["LTF"] / scr["LD"] * (1.0 + off)))
    ctx = pcc.Context(0)
    ctx.tables_build([pcc.material(*m) for m in mats], pcc.table_spec(n_rows=rows, n_cols=cols, quad_nodes=nodes, **kw))
    got = ctx.tables_read()
    ctx.close()
    ref = orc.OracleTables([orc.material(*m) for m in mats],
                           orc.table_spec(n_rows=rows, n_cols=cols, quad_nodes=nodes, **kw))
    # the printed form of I2 loses (L delta)^3 2^-53: where that exceeds the
    # tolerance (one material here, 1e-4) the oracle says nothing, and the
    # Bethe-Heitler totals are compared with the same rule in 40 digits
    L = got["screening"][:, 5]
    good = L ** 3 * 2.0 ** -53 < 0.1 * RTOL
    assert list(np.flatnonzero(~good)) == [3]
    for k in ("brems_sigma", "brems_cdf", "bh_sigma", "bh_cdf", "tri_gp_cdf", "tri_split_cdf"):
        r = np.asarray(getattr(ref, k)).reshape(got[k].shape)
        sel = slice(None) if k.startswith("tri") else good
        np.testing.assert_allclose(got[k][sel], r[sel], rtol=RTOL, atol=1e-12 * np.abs(r).max(), err_msg=k)
        if k.endswith("cdf"):
            assert np.all(np.diff(got[k], axis=-1) >= 0.0) and np.all(got[k][..., -1] == 1.0)
    if not kw and cols * nodes <= 200:
        want = [bethe_heitler_total(T, L[3], cols, nodes) for T in 0.002 * (1999.0 / 0.002) ** (np.arange(rows) / (rows - 1))]
        np.testing.assert_allclose(got["bh_sigma"][3], want, rtol=1e-11)
