"""Infinite values in the sums that run as FP32 pairs (TwoSum) on the GPU: they end as FP64 sums of
the same values do, infinite and not NaN.
"""
import numpy as np
import pytest

from synthetic import uniform_density, uniform_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2301_08911_gb300 import binding, build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return binding


def cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("n", [5, 8, 16])     # single values, 16-byte accesses, several blocks
@pytest.mark.parametrize("bad", [float("inf"), -float("inf")])
def test_oc_update_with_an_infinite_density(B, n, bad):
    """+inf makes the volume at the lower bounds infinite, above any target: everything goes to its
    lower bound; -inf the volume at the upper bounds -inf, below any: everything to its upper
    bound (there the multiplier is the largest hi / base, so base times it may round one unit
    below hi: two FP32 roundings, 2 x 6e-8). Without it the target lies between (mean 0.5)."""
    move = 0.1
    hom = B.Homogenization(n)
    r0 = uniform_density(n, 740 + n, 0.01, 1.0)
    r0[n ** 3 // 2] = bad
    rho, dc = cuda(r0), cuda(-uniform_field(n ** 3, 741, 1e-3, 1.0))
    hom.update(dc, rho, 0.5, move)
    got = rho.cpu().numpy()
    lo = np.maximum(np.float32(1e-3), r0 - np.float32(move))
    hi = np.minimum(np.float32(1.0), r0 + np.float32(move))
    want = np.minimum(lo if bad > 0 else hi, hi)
    keep = np.arange(n ** 3) != n ** 3 // 2
    np.testing.assert_allclose(got[keep], want[keep], rtol=0 if bad > 0 else 1.2e-7, atol=0)
    assert got[~keep][0] == (1.0 if bad > 0 else bad)
