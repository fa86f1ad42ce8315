"""Kernels that are chosen by size or alignment, each against the form it replaces or the
operator it inverts, on a GB300: the finest level's one-launch sweep (n <= 16) against the
colour-pair launches (bitwise), fields that are not 8- or 16-byte aligned against aligned ones
(bitwise where the arithmetic is the same), and the blocked coarsest inverse at every size it
takes (K z = r).
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


def shifted(t):
    """The same values one float past a 16-byte boundary."""
    buf = torch.empty(t.numel() + 1, device="cuda", dtype=t.dtype)
    buf[1:].copy_(t)
    return buf[1:]


@pytest.mark.parametrize("n", [8, 10, 12, 14, 16])
def test_one_launch_fine_sweep_equals_pair_launches(B, n):
    hom = B.Homogenization(n)
    hom.set_density(cuda(uniform_density(n, 700 + n, 0.01, 1.0)))
    f, u0 = cuda(uniform_field(18 * n ** 3, 701, -1, 1)), cuda(uniform_field(18 * n ** 3, 702, -1, 1))
    r = uniform_field(18 * n ** 3, 703, -1, 1).reshape(18, -1)
    r = cuda(r + 0.25)                                   # plane means are not zero
    got = {}
    for form, sizes in {"one": (16, 32, 32), "pairs": (0, 32, 32)}.items():
        hom.set_coarse_smoother(*sizes)
        outs = []
        for reverse in (False, True):
            u = u0.clone()
            hom.smooth(0, reverse, f, u)
            outs.append(u)
        z = torch.full_like(u0, float("nan"))            # a sweep from zero must not read z
        hom.vcycle(r.reshape(-1), z)
        got[form] = outs + [z]
    torch.cuda.synchronize()
    assert torch.isfinite(got["one"][2]).all()
    for a, b in zip(got["one"], got["pairs"]):
        assert torch.equal(a, b), (a - b).abs().max().item()


@pytest.mark.parametrize("n", [16, 20, 56])
def test_unaligned_fields_give_the_aligned_results(B, n):
    hom = B.Homogenization(n)
    hom.set_density(cuda(uniform_density(n, 710 + n, 0.01, 1.0)))
    N = n ** 3
    f, u = cuda(uniform_field(18 * N, 711, -1, 1)), cuda(uniform_field(18 * N, 712, -1, 1))
    coarse = cuda(uniform_field(18 * (n // 2) ** 3, 713, -1, 1))
    res = []
    for move in (lambda t: t.clone(), shifted):
        fa, ua, wa, za = move(f), move(u), move(u), move(u)
        hom.smooth(0, False, fa, ua)
        hom.smooth(0, True, fa, ua)
        hom.prolong_add(0, coarse, wa)
        hom.vcycle(fa, za)
        res.append([ua.clone(), wa.clone(), za.clone()])
    torch.cuda.synchronize()
    for a, b in zip(*res):
        assert torch.equal(a, b), (a - b).abs().max().item()
    # the OC update sums in another order: where the move limit reaches the volume both meet it
    # and agree as closely as the bracket of the multiplier (16^-8 of its logarithm) and FP32
    # densities allow; at 0.4 it does not (mean 0.505, move 0.1) and every value is at its bound
    rho, dc = cuda(uniform_density(n, 714, 0.01, 1.0)), cuda(-uniform_field(N, 715, 1e-3, 1.0))
    for volfrac in (0.4, 0.5):
        out = []
        for move in (lambda t: t.clone(), shifted):
            r = move(rho)
            change = hom.update(move(dc), r, volfrac, 0.1)
            out.append((r.clone(), change))
            if volfrac == 0.4:
                assert torch.equal(r, torch.clamp(rho - 0.1, min=1e-3))
            else:
                assert abs(r.double().mean().item() - volfrac) < 1e-6
        assert (out[0][0] - out[1][0]).abs().max().item() <= 2e-6
        assert abs(out[0][1] - out[1][1]) <= 2e-6


@pytest.mark.parametrize("n", [4, 5, 6, 7, 8])
def test_blocked_coarsest_inverse_inverts_K(B, n):
    """A one-level cell's V-cycle is the coarsest solve: K z = r for a mean-free r. z is
    rounded to FP32 and K applied in FP32: 6e-8 of sum |A| |z|, whose ratio to |r| is below
    the operator's condition number (about 4 n^2 / pi^2 x 2 for moduli in [0.125, 1] x 8 < 1e3)."""
    hom = B.Homogenization(n, max_levels=1)
    assert hom.num_levels == 1
    hom.set_density(cuda(uniform_density(n, 720 + n, 0.5, 1.0)))
    r = uniform_field(18 * n ** 3, 721, -1, 1).reshape(18, -1)
    r = cuda(r - r.mean(axis=1, keepdims=True)).reshape(-1)
    z, back = torch.empty_like(r), torch.empty_like(r)
    hom.vcycle(r, z)
    hom.apply_K(z, back)
    torch.cuda.synchronize()
    assert ((back - r).norm() / r.norm()).item() < 6e-5
    assert z.reshape(18, -1).double().mean(dim=1).abs().max().item() < 1e-6 * z.abs().max().item()


def apply_stencil(st, u):
    """FP64 sum_d A_d u(v + d) of a level's stencil (z, y, x, 27, 9) on (6, 3, z, y, x) fields."""
    n = st.shape[0]
    out = torch.zeros_like(u)
    for d in range(27):
        s = (-(d // 9 - 1), -((d // 3) % 3 - 1), -(d % 3 - 1))
        A = st[..., d, :].double().view(n, n, n, 3, 3)
        out += torch.einsum("zyxrc,kczyx->krzyx", A, torch.roll(u, s, dims=(2, 3, 4)))
    return out


def bf16_stencil(st):
    """The stored BF16 stencil: each block averaged with its transposed counterpart, then rounded."""
    n, out = st.shape[0], torch.empty_like(st)
    for d in range(27):
        s = (-(d // 9 - 1), -((d // 3) % 3 - 1), -(d % 3 - 1))
        other = torch.roll(st[..., 26 - d, :], s, dims=(0, 1, 2)).view(n, n, n, 3, 3).transpose(-1, -2)
        out[..., d, :] = (0.5 * (st[..., d, :] + other.reshape(n, n, n, 9))).bfloat16().float()
    return out


@pytest.mark.parametrize("n,level", [(40, 1), (48, 1), (56, 1), (112, 2), (224, 1)])
def test_staged_coarse_sweep_matches_its_stencil(B, n, level):
    """Levels 20, 24, 28 and 112: stencil rows of one tile and a ragged one, shorter than a warp's
    vertices and both tile splits (<= 96 and above), both stencil precisions and colour
    orders, two sweeps in a row (the second chained to the first), against an FP64 sweep with the
    same stencil. Bound 2e-6 a sweep, as for one sweep of any coarse form against the oracle."""
    nl = n >> level
    rho = cuda(uniform_density(n, 730 + n, 0.05, 1.0))
    f, u0 = cuda(uniform_field(18 * nl ** 3, 731, -1, 1)), cuda(uniform_field(18 * nl ** 3, 732, -1, 1))
    hom = B.Homogenization(n)
    hom.set_density(rho)
    st = torch.empty(nl ** 3 * 243, device="cuda")
    hom.get_stencil(level, st)
    st = st.view(nl, nl, nl, 27, 9)
    ax = torch.arange(nl, device="cuda") & 1
    colour = ax[None, None, :] + 2 * ax[None, :, None] + 4 * ax[:, None, None]
    for precision in ("fp32", "mixed"):
        if precision == "mixed":
            hom = B.Homogenization(n, precision=precision)
            hom.set_density(rho)
            st = bf16_stencil(st)
        Sinv = torch.linalg.inv(st[..., 13, :].double().view(nl, nl, nl, 3, 3))
        for reverse in (False, True):
            u = u0.clone()
            for _ in range(2):
                hom.smooth(level, reverse, f, u)
            ref = u0.double().view(6, 3, nl, nl, nl).clone()
            fd = f.double().view_as(ref)
            for _ in range(2):
                for k in range(8):
                    r = fd - apply_stencil(st, ref)
                    du = torch.einsum("zyxrc,kczyx->krzyx", Sinv, r)
                    ref += du * (colour == (7 - k if reverse else k))
            err = u.double().view_as(ref) - ref
            assert (err.norm() / ref.norm()).item() < 4e-6, (precision, reverse)
            assert (err.abs().max() / ref.abs().max()).item() < 4e-6, (precision, reverse)


@pytest.mark.parametrize("n", [4, 16, 20, 40, 80, 112])
def test_product_over_chunk_sizes(B, n):
    """One and two planes a block, ragged tiles in x and y, against the level's own stencil in
    FP64: 2e-6 of the terms each output sums, as against the oracle."""
    hom = B.Homogenization(n)
    hom.set_density(cuda(uniform_density(n, 740 + n, 0.05, 1.0)))
    u = cuda(uniform_field(18 * n ** 3, 741, -1, 1))
    out = torch.empty_like(u)
    hom.apply_K(u, out)
    st = torch.empty(n ** 3 * 243, device="cuda")
    hom.get_stencil(0, st)
    st = st.view(n, n, n, 27, 9)
    ud = u.double().view(6, 3, n, n, n)
    err = (out.double().view_as(ud) - apply_stencil(st, ud)).abs()
    assert torch.all(err <= 2e-6 * apply_stencil(st.abs(), ud.abs()))
