"""Values past the FP32 range in the sums that run as FP32 pairs (TwoSum) on the GPU: they end as FP64 sums of
the same values do, infinite and not NaN. So does a sum that only passes FP32's largest value.
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


def _wgrad_of_spikes(B, cin, spikes):
    """dw, db of a 16^3 layer with x = 1 and dy zero but for channel 3 of some voxels: every tap's
    and input channel's sum over the 32 chunks (128 voxels each) is the sum of the spikes."""
    n = 16
    x = torch.ones((n ** 3, cin), dtype=torch.bfloat16, device="cuda")
    dy = torch.zeros((n ** 3, 32), dtype=torch.bfloat16, device="cuda")
    for chunk, value in spikes.items():
        dy[128 * chunk + 5, 3] = value
    dw, db = torch.empty((27, 32, cin), device="cuda"), torch.empty(32, device="cuda")
    B.nn_wgrad(n, cin, x, dy, dw, db, torch.empty(B.nn_wgrad_scratch(n, cin), device="cuda"))
    other = [o for o in range(32) if o != 3]
    assert not dw[:, other].any() and not db[other].any()
    return torch.cat([dw[:, 3].reshape(-1), db[3:4]])


@pytest.mark.parametrize("cin", [16, 32])
@pytest.mark.parametrize("bad", [float("inf"), -float("inf")])
def test_weight_gradient_with_an_infinite_voxel(B, cin, bad):
    assert (_wgrad_of_spikes(B, cin, {2: 1.0, 9: bad, 30: -2.0}) == bad).all()


@pytest.mark.parametrize("cin", [16, 32])
@pytest.mark.parametrize("chunks", [(0, 1, 2), (0, 8, 16), (7, 23, 31)])   # within and across the quarters
def test_weight_gradient_sum_that_leaves_the_fp32_range_on_the_way(B, cin, chunks):
    """b + b - b = b in FP64; b + b is past FP32's largest value."""
    b = torch.tensor(3e38, dtype=torch.bfloat16).float().item()
    got = _wgrad_of_spikes(B, cin, dict(zip(chunks, (b, b, -b))))
    assert (got == b).all()
