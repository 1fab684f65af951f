"""bench.py's sort rate: the bytes of the passes that ran, not of all digits."""
import pytest

import bench


class _A:
    n, d, bits, T = 3_000_000, 384, 8, 64


@pytest.mark.parametrize("passes,words", [(16.0, 1), (8.0, 1), (7.25, 2), (4.0, 2)])
def test_sort_bytes_follow_the_passes(passes, words):
    r = bench.keys_sort_hbm(_A, {"keys": 2.0, "sort": 25.0, "sort_passes": passes})["sort"]
    per = 16 + 24 * passes + (8 if passes < 16 else 0) + 4 + 16 * words
    assert r["bytes"] == pytest.approx(per * _A.n * _A.T)
    assert r["frac"] == pytest.approx(r["bytes"] / 25e-3 / 1e9 / bench.keys_sort_hbm(_A, {"keys": 2.0, "sort": 25.0})["peak"])
    assert r["all_digits"] == pytest.approx(_A.n * _A.T * 16 * 24 / 25e-3 / 1e9)
    assert r["passes_per_tree"] == passes


def test_one_word_keys():
    class A(_A):
        d, bits = 8, 8
    r = bench.keys_sort_hbm(A, {"keys": 1.0, "sort": 1.0, "sort_passes": 8.0})["sort"]
    assert r["bytes"] == pytest.approx((8 + 24 * 8) * A.n * A.T)
