"""The autotuner times the library's own choice among its candidates, so that a
tuned call is not slower than an untuned one (the group, tile and block kernels
alone leave out two half expansions and split tiles)."""
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,n,count", [(20, 10, 4096), (324, 18, 256), (12, 6, 1), (5, 30, 7)])
def test_default_choice_is_a_candidate(m, n, count):
    from paper_2204_00602_gb300 import PCV_ALGO_AUTO, autotune
    found = autotune.candidates(m, n, count)
    assert (PCV_ALGO_AUTO, 0) in found
    assert len(found) == len(set(found))
