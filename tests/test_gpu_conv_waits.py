"""The tensor-core layer's failure detection: each of its 13 warps (8 epilogue, 4 copy, 1 MMA) polls
and decides for itself, so a wait that runs out has to be counted whichever warp it was in.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2301_08911_gb300 import binding, build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return binding


@pytest.mark.parametrize("blocks", [1, 13, 40])
def test_a_wait_that_runs_out_in_any_one_warp_counts_its_cta_once(B, blocks):
    """CTA b lets the wait of warp b mod 13 run out and those of the other twelve complete."""
    B.nn_tc_timeouts()                                  # reset
    B.nn_tc_wait_probe(blocks)
    assert B.nn_tc_timeouts() == blocks
    assert B.nn_tc_timeouts() == 0
