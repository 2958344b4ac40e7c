"""Binning at the edges of its sort classes (a warp's count, warp, block and
large-block radix sorts), of its pid ranges (storage numbers, wide secondary
ids, ids that differ in few high bits, input already in order) and on both
counting paths, against a lexicographic sort on the host."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build, pcc
    build.build()
    return pcc


def pids(rng, kind, n):
    if kind == "dense":
        return rng.permutation(n).astype(np.uint64)
    if kind == "ordered":
        return np.arange(n, dtype=np.uint64) * np.uint64(3)
    if kind == "high":        # differing bits far apart, the topmost among them
        v = rng.permutation(1 << int(np.ceil(np.log2(max(n, 2)))))[:n].astype(np.uint64)
        lo, hi = v & np.uint64(31), v >> np.uint64(5)
        return (hi << np.uint64(45)) | (lo << np.uint64(11)) | np.uint64(1 << 40)
    # primaries and secondaries: marker | step | channel | cell | pair | slot
    p = rng.permutation(n).astype(np.uint64)
    sec = rng.random(n) < 0.7
    step, ch = rng.integers(0, 5000, n).astype(np.uint64), rng.integers(0, 5, n).astype(np.uint64)
    s = np.uint64(1 << 63) | (step << np.uint64(44)) | (ch << np.uint64(41)) | p
    return np.where(sec, s, p)


def check(pcc, counts, kind, with_x, seed, invalid=0):
    rng = np.random.default_rng(seed)
    n_cells = len(counts)
    cell = np.repeat(np.arange(n_cells, dtype=np.int32), counts)
    n = len(cell)
    pid = pids(rng, kind, n)
    if kind != "ordered":
        perm = rng.permutation(n)
        cell, pid = cell[perm], pid[perm]
    f = {k: rng.normal(size=n).astype(np.float32) for k in ("ux", "uy", "uz", "w", "x")}
    if invalid:
        cell = np.concatenate([cell, np.full(invalid, n_cells, np.int32), np.full(invalid, -5, np.int32)])
        pid = np.concatenate([pid, np.arange(2 * invalid, dtype=np.uint64) + np.uint64(1 << 50)])
        f = {k: np.concatenate([v, np.ones(2 * invalid, np.float32)]) for k, v in f.items()}
    ctx = pcc.Context(0)
    d = dict(f, pid=pid, cell=cell)
    if not with_x:
        d["x"] = None
    sp = pcc.DeviceSpecies.empty(n_cells, int(1.25 * n) + 8 * n_cells + 8, with_x=with_x)
    pcc.bin(ctx, pcc.particles_to_device(d), n_cells, sp, slack_abs=7, slack_rel=0.2)
    counts = np.asarray(counts, np.int64)
    room = counts + np.maximum(7, np.ceil(0.2 * counts).astype(np.int64))
    start = np.concatenate([[0], np.cumsum(room)])
    assert np.array_equal(sp.cell_start.cpu().numpy(), start) and np.array_equal(sp.cell_count.cpu().numpy(), counts)
    assert not sp.cell_added.cpu().numpy().any()
    order = np.lexsort((pid[:n], cell[:n]))
    slot = start[cell[:n][order]] + np.arange(n) - np.repeat(np.cumsum(counts) - counts, counts)
    for k in ("ux", "uy", "uz", "w") + (("x",) if with_x else ()):
        ref = np.zeros(sp.capacity, np.float32)
        ref[slot] = f[k][:n][order]
        assert np.array_equal(getattr(sp, k).cpu().numpy(), ref), k
    ref = np.zeros(sp.capacity, np.uint64)
    ref[slot] = pid[:n][order]
    assert np.array_equal(sp.pid.cpu().numpy().view(np.uint64), ref)
    st, _ = ctx.read_status()
    assert bool(st & pcc.ST_NONFINITE) == (invalid > 0)
    ctx.close()


EDGES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 255, 256, 257, 511, 512, 513, 0, 1000, 2047, 2048, 2049, 5000, 8191, 8192, 8193, 0, 16383, 16384]


@pytest.mark.parametrize("kind", ["dense", "ordered", "high", "secondaries"])
@pytest.mark.parametrize("with_x", [False, True])
def test_bin_at_the_class_edges(pcc, kind, with_x):
    check(pcc, EDGES, kind, with_x, 1)


@pytest.mark.parametrize("counts", [[0], [1], [40], [0, 0, 3000], [2049], [0] * 1023 + [5] + [0] * 1024 + [600, 1]])
def test_bin_small_inputs(pcc, counts):
    check(pcc, counts, "secondaries", False, 2, invalid=3)


def test_bin_many_cells(pcc):
    rng = np.random.default_rng(3)
    check(pcc, np.minimum(np.rint(rng.lognormal(3.0, 1.5, 70001)), 9000).astype(np.int64), "dense", True, 4)


def test_bin_few_cells_count_in_shared_memory(pcc):
    rng = np.random.default_rng(5)
    check(pcc, rng.integers(0, 12000, 300), "dense", True, 6, invalid=100)


def test_bin_limits(pcc):
    ctx = pcc.Context(0)
    n = 16385
    d = {k: np.ones(n, np.float32) for k in ("ux", "uy", "uz", "w")}
    d.update(pid=np.arange(n, dtype=np.uint64), cell=np.zeros(n, np.int32), x=None)
    sp = pcc.DeviceSpecies.empty(2, 2 * n)
    with pytest.raises(pcc.PccError, match="16385 particles"):
        pcc.bin(ctx, pcc.particles_to_device(d), 2, sp, slack_abs=1, slack_rel=0.0)
    d["cell"][::2] = 1
    sp = pcc.DeviceSpecies.empty(2, n + 1)
    with pytest.raises(pcc.PccError, match=f"regions need {n + 2} slots"):
        pcc.bin(ctx, pcc.particles_to_device(d), 2, sp, slack_abs=1, slack_rel=0.0)
    assert not sp.ux.cpu().numpy().any()
    sp = pcc.DeviceSpecies.empty(2, n + 2)
    pcc.bin(ctx, pcc.particles_to_device(d), 2, sp, slack_abs=1, slack_rel=0.0)
    assert int(sp.cell_count.sum()) == n
    ctx.close()
