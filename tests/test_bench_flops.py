"""The bench's work model of the eigen phase where AUTO puts the polynomial transform before the split
eigensolve (k > 64, reported as SPLIT): it counts what the device counters say was done."""
import pytest

import bench
import synth


def _eig(k, schedule, counts):
    w = synth.WORKLOADS["turb256_k32"]
    return bench.kernel_work(w, k, 30720, 42.0, 2, 1024, 1, 100, schedule, counts)["eigen_update"][1]


@pytest.mark.parametrize("k", [65, 128])
def test_transformed_points_count_their_products(k):
    counts = {"cheb_points": 30000, "cheb_products": 400000, "cheb_handed_on": 720}
    want = 20.0 * k * k * 400000 + 36.0 * k * 30000 + 11.0 * k ** 3 * 720
    assert _eig(k, 2, counts) == pytest.approx(want / 1e12)


def test_plain_split_counts_the_eigensolve():
    none = {"cheb_points": 0, "cheb_products": 0, "cheb_handed_on": 0}
    for counts in (none, None):
        assert _eig(128, 2, counts) == pytest.approx(11.0 * 128 ** 3 * 30720 / 1e12)
    # k <= 64: SPLIT never has the transform before it
    some = {"cheb_points": 5, "cheb_products": 50, "cheb_handed_on": 0}
    assert _eig(64, 2, some) == pytest.approx(11.0 * 64 ** 3 * 30720 / 1e12)
