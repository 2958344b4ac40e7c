"""The autotuner's choice of a schedule from its timings: the fastest candidate, or the
default where the others differ from it by noise only."""
import pytest

pytest.importorskip("torch")

from paper_1907_02814_gb300 import tune  # noqa: E402


def test_noise_keeps_the_default():
    cands = ((4, 0), (5, 0), (2, 0))
    assert tune.pick(cands, {"4,0": 1.000, "5,0": 0.995, "2,0": 1.004}) == (4, 0)
    assert tune.pick(cands, {"4,0": 1.0, "5,0": 1.0, "2,0": 1.0}) == (4, 0)


def test_a_faster_candidate_is_taken():
    cands = ((4, 0), (5, 0), (2, 0))
    assert tune.pick(cands, {"4,0": 1.0, "5,0": 0.97, "2,0": 0.98}) == (5, 0)
