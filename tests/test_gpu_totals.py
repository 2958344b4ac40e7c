"""FP64 totals formed from split FP32 sums: against extended-precision sums at
the edges of a warp's tiles and of the range the split form covers (particles
at rest, momenta whose squares leave the float range, weights near its ends)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# terms are exact to 2^-60; a sum passes through at most about 30 FP64 additions
RTOL = 32 * 2.0 ** -53


def _species(pcc, counts, u, w):
    counts = np.asarray(counts, np.int32)
    start = np.concatenate([[0], np.cumsum(counts + 3)]).astype(np.int32)     # odd region starts
    slot = np.concatenate([start[c] + np.arange(n) for c, n in enumerate(counts)]) if counts.sum() else np.zeros(0, int)
    sp = pcc.DeviceSpecies.empty(len(counts), int(start[-1]) + 1)
    idx = torch.as_tensor(slot.astype(np.int64), device="cuda")
    for name, v in zip(("ux", "uy", "uz", "w"), (*u, w)):
        t = getattr(sp, name)
        t.fill_(7.0)                                                          # dead slots must not count
        t[idx] = torch.as_tensor(v, device="cuda")
    sp.cell_start.copy_(torch.as_tensor(start))
    sp.cell_count.copy_(torch.as_tensor(counts))
    return sp


@pytest.mark.parametrize("photon", [False, True])
@pytest.mark.parametrize("counts", [[1], [0, 31, 32, 33, 0, 127, 128, 129], [5] * 300, [4097, 0, 1]])
@pytest.mark.parametrize("scale", ["plain", "rest", "extreme"])
def test_totals_match_extended_precision(photon, counts, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    rng = np.random.default_rng(len(counts) + 2 * photon)
    n = int(np.sum(counts))
    u = (rng.normal(size=(3, n)) * 10.0 ** rng.uniform(-3, 3, n)).astype(np.float32)
    w = (1e27 * rng.uniform(0.1, 2.0, n)).astype(np.float32)
    if scale == "rest":
        u[:, ::2] = 0.0
        u[1:, 1::4] = 0.0
        w[::3] = 0.0
    if scale == "extreme":
        u *= (10.0 ** rng.uniform(-24, 18, n)).astype(np.float32)
        w = (10.0 ** rng.uniform(-30, 15, n)).astype(np.float32)
    sp = _species(pcc, counts, u, w)
    ctx = pcc.Context(0)
    got = pcc.totals(ctx, len(counts), sp, is_photon=photon).cpu().numpy()
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    pcc.totals_noalloc(len(counts), sp, out, is_photon=photon)
    L = np.longdouble
    k = np.sqrt((u.astype(L) ** 2).sum(0))
    W = w.astype(L)
    ref = np.array([W.sum(), (W * (k if photon else np.sqrt(1 + k * k))).sum(), (W * k).sum()], dtype=np.float64)
    np.testing.assert_allclose(got, ref, rtol=RTOL)
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=RTOL)
    ctx.close()


def test_totals_carry_non_finite_values():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    ctx = pcc.Context(0)
    u = np.ones((3, 40), np.float32)
    w = np.ones(40, np.float32)
    u[1, 17] = np.inf
    got = pcc.totals(ctx, 2, _species(pcc, [20, 20], u, w)).cpu().numpy()
    assert got[0] == 40.0 and np.isinf(got[1]) and np.isinf(got[2])
    u[1, 17] = np.nan
    got = pcc.totals(ctx, 2, _species(pcc, [20, 20], u, w)).cpu().numpy()
    assert got[0] == 40.0 and np.isnan(got[1]) and np.isnan(got[2])
    ctx.close()
