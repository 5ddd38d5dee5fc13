"""The form that the benchmark names as chosen is the fastest of those that converged."""
import bench


def test_fastest_form():
    assert bench.fastest({"plain": 2.8, "jacobi": 0.1, "unet": 0.2}) == "jacobi"
    assert bench.fastest({"plain": 2.8}) == "plain"
    assert bench.fastest({}) is None

