"""The warm-start convolution and weight gradient at grid sizes that take the 32 x 11 x 1 tile or
leave its last tiles ragged, and at rows longer than a weight-gradient chunk, against the
oracle network on a GB300 (rounding contract and bounds as in test_gpu_learned.py)."""
import numpy as np
import pytest

from oracle import learned as L
from test_gpu_learned import _randn, acc_bound, bf16, check_bf16, f32, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2301_08911_gb300 import binding, build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return binding


@pytest.mark.parametrize("n,c_in", [(31, 16), (62, 32), (64, 32)])
def test_conv_tile_shapes(B, n, c_in):
    N = n ** 3
    x, xh = bf16(_randn((N, c_in), 1 + n))
    w, wh = bf16(_randn((27, 32, c_in), 2 + n, 0.1))
    b = _randn((32,), 3 + n, 0.2).astype(np.float32)
    res, resh = bf16(_randn((N, 32), 4 + n))
    out = torch.empty((N, 32), dtype=torch.bfloat16, device="cuda")
    B.nn_conv3d(n, c_in, x, w, bias=f32(b), res=res, epilogue="relu", out=out)
    want = L.conv3d(xh, wh, b.astype(np.float64), n)
    bound = acc_bound(xh, wh, n, b, resh)
    check_bf16(host(out), L.bf16_round(np.maximum(want + resh, 0.0)), bound)
    if c_in == 32:
        planes = torch.empty(18 * N, device="cuda")
        B.nn_conv3d(n, c_in, x, w, bias=f32(b), epilogue="planes", out_planes=planes, scale=np.ones(6))
        assert np.all(np.abs(host(planes).reshape(18, N) - want[:, :18].T) <= bound[:, :18].T)


@pytest.mark.parametrize("n,c_in", [(36, 16), (64, 32)])
def test_weight_gradient_of_long_rows(B, n, c_in):
    N = n ** 3
    x, xh = bf16(_randn((N, c_in), 21 + n))
    dy, dyh = bf16(_randn((N, 32), 22 + n))
    dw, db = torch.empty((27, 32, c_in), device="cuda"), torch.empty(32, device="cuda")
    scratch = torch.empty(B.nn_wgrad_scratch(n, c_in), device="cuda")
    B.nn_wgrad(n, c_in, x, dy, dw, db, scratch)
    want_w, want_b = L.conv3d_wgrad(xh, dyh, n)
    bw, bb = L.conv3d_wgrad(np.abs(xh), np.abs(dyh), n)
    assert np.all(np.abs(host(dw) - want_w) <= 1e-5 * bw + 1e-30)
    assert np.all(np.abs(host(db) - want_b) <= 1e-5 * bb + 1e-30)
