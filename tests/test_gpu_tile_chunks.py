"""The planes a block of the finest-level residual and Chebyshev kernels takes change with the cell: a
V-cycle of a cell shifted along z, whose block boundaries then fall on other planes, is the
shifted V-cycle, and the Chebyshev one (whose eigenvalue estimates do not shift) is symmetric.
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


@pytest.mark.parametrize("n,shift", [(24, 8), (48, 16), (64, 16), (80, 16), (96, 16), (112, 16), (160, 32)])
def test_vcycle_of_a_shifted_cell(B, n, shift):
    """The shift is a multiple of the coarsest cell, so every level shifts by whole cells (and
    colours). Only the coarsest inverse (FP64) pins another vertex. Rigid translations are outside
    the operator's range and removed. Bound 1e-4 of the largest entry, as for the V-cycle
    against the oracle; a plane read from the wrong place changes its entries by order one."""
    hom = B.Homogenization(n)
    assert shift % (n // hom.level_size(hom.num_levels - 1)) == 0
    rho = cuda(uniform_density(n, 980 + n, 0.2, 1.0)).view(n, n, n)
    r = uniform_field(18 * n ** 3, 981, -1, 1).reshape(18, -1)
    r = cuda(r - r.mean(axis=1, keepdims=True)).view(18, n, n, n)
    out = []
    for s in (0, shift):
        hom.set_density(torch.roll(rho, s, dims=0).contiguous().reshape(-1))
        z = torch.full((18 * n ** 3,), float("nan"), device="cuda")
        hom.vcycle(torch.roll(r, s, dims=1).contiguous().reshape(-1), z)
        z = torch.roll(z.view(18, n, n, n), -s, dims=1).double()
        out.append(z - z.mean(dim=(1, 2, 3), keepdim=True))
    torch.cuda.synchronize()
    assert torch.isfinite(out[0]).all()
    assert ((out[0] - out[1]).abs().max() / out[0].abs().max()).item() < 1e-4


@pytest.mark.parametrize("n", [24, 48, 80, 96, 160])
def test_chebyshev_vcycle_is_symmetric(B, n):
    """(a, M b) = (M a, b) for mean-free a and b; FP32 rounding leaves 1e-5 of |a| |M b|, a plane
    read from the wrong place order one."""
    hom = B.Homogenization(n, smoother="chebyshev")
    hom.set_density(cuda(uniform_density(n, 985 + n, 0.2, 1.0)))
    fields, images = [], []
    for seed in (986, 987):
        a = uniform_field(18 * n ** 3, seed, -1, 1).reshape(18, -1)
        fields.append(cuda(a - a.mean(axis=1, keepdims=True)).reshape(-1))
        z = torch.full_like(fields[-1], float("nan"))
        hom.vcycle(fields[-1], z)
        images.append(z)
    (a, b), (ma, mb) = [f.double() for f in fields], [f.double() for f in images]
    assert abs((a * mb).sum() - (ma * b).sum()) <= 1e-5 * a.norm() * mb.norm()
