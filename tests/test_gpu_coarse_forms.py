"""Which kernel form the sizes of homo_set_coarse_smoother select, seen from the launches it takes,
and every form that can run a level above 16 cells per axis against the others, bitwise: the
staged one (no size covers the level, or the default sizes), a thread per (vertex, case), and the
clusters through L2.
"""
import numpy as np
import pytest

from synthetic import smoothed_threshold_density, uniform_density, uniform_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STAGED, ITEM, CLUSTER = (0, 0, 0), (0, 0, 1024), (0, 1024, 0)


@pytest.fixture(scope="module")
def B():
    from paper_2301_08911_gb300 import binding, build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    return binding


def cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
def test_the_sizes_select_the_form(B, precision):
    """A cluster form takes one launch a sweep, the others one a colour. n = 64: levels 32, 16, 8."""
    n = 64
    hom = B.Homogenization(n, precision=precision)
    hom.set_density(cuda(uniform_density(n, 950, 0.05, 1.0)))
    clusters, resident = hom.coarse_smoother()[3] > 0, hom.coarse_smoother()[4] == 16
    for sizes, form32, form16, form8 in [((16, 32, 32), "colour", "resident", "resident"),     # the defaults
                                         ((8, 32, 32), "colour", "cluster", "resident"),
                                         ((0, 32, 0), "cluster", "cluster", "cluster"),
                                         ((16, 32, 0), "cluster", "resident", "resident"),
                                         ((0, 16, 32), "colour", "cluster", "cluster"),
                                         (CLUSTER, "cluster", "cluster", "cluster"),
                                         (ITEM, "colour", "colour", "colour"),
                                         (STAGED, "colour", "colour", "colour")]:
        hom.set_coarse_smoother(*sizes)
        for level, form in ((1, form32), (2, form16), (3, form8)):
            nl = n >> level
            f, u = cuda(uniform_field(18 * nl ** 3, 951, -1, 1)), cuda(uniform_field(18 * nl ** 3, 952, -1, 1))
            hom.smooth(level, False, f, u)               # builds the hierarchy the first time
            before = hom.launch_count
            hom.smooth(level, False, f, u)
            one = (form == "cluster" and clusters) or (form == "resident" and (resident or (nl < 16 and clusters)))
            assert hom.launch_count - before == (1 if one else 8), (sizes, level)


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("n,level", [(40, 1), (64, 1), (224, 1), (224, 2)])
def test_forms_above_16_are_bitwise_equal(B, n, level, precision):
    """Levels 20 (a ragged last tile), 32, 112 (three cases per thread) and 56: two sweeps in each
    colour order, and the V-cycle whose pre-smoothing starts from zero."""
    nl = n >> level
    hom = B.Homogenization(n, precision=precision)
    hom.set_density(cuda(uniform_density(n, 960 + n, 0.05, 1.0)))
    f, u0 = cuda(uniform_field(18 * nl ** 3, 961, -1, 1)), cuda(uniform_field(18 * nl ** 3, 962, -1, 1))
    r = uniform_field(18 * n ** 3, 963, -1, 1).reshape(18, -1)
    r = cuda(r - r.mean(axis=1, keepdims=True)).reshape(-1)
    default = hom.coarse_smoother()[:3]
    want = None
    for sizes in (default, STAGED, ITEM, CLUSTER):
        hom.set_coarse_smoother(*sizes)
        outs = []
        for reverse in (False, True):
            u = u0.clone()
            hom.smooth(level, reverse, f, u)
            hom.smooth(level, reverse, f, u)
            outs.append(u)
        z = torch.full_like(r, float("nan"))
        hom.vcycle(r, z)
        torch.cuda.synchronize()
        outs.append(z)
        if want is None:
            want = outs
            assert all(torch.isfinite(o).all() for o in outs) and not torch.equal(outs[0], u0)
        for a, b in zip(want, outs):
            assert torch.equal(a, b), (sizes, (a - b).abs().max().item())


def test_autotuner_times_the_forms_it_names(B):
    """Launches of one timing run: per level two smoothing phases of 3^(level - 1) sweeps, once
    untimed and four times (once above 32^3) timed, in each form it reports."""
    n = 128
    hom = B.Homogenization(n)
    hom.set_density(cuda(smoothed_threshold_density(n, 0.3, 6)))
    hom.autotune_coarse(retime=True)
    before = hom.launch_count
    _, times = hom.autotune_coarse(retime=True)
    got = hom.launch_count - before
    want = 0
    for level, row in times.items():
        sweeps, reps = 3 ** (level - 1), 5 if n >> level <= 32 else 2
        assert {"vertex", "item"} <= set(row)
        for form in row:
            want += reps * 2 * (1 if form in ("cluster", "resident") else 8 * sweeps)
    assert sorted(times) == [1, 2, 3, 4] and got == want


@pytest.mark.parametrize("n", [8, 16, 24])
def test_fine_autotuner_times_its_variants_on_small_cells_too(B, n):
    """Per variant five sweeps of four launches; a cell of at most 16 would take one launch a sweep."""
    hom = B.Homogenization(n)
    hom.set_density(cuda(uniform_density(n, 970, 0.05, 1.0)))
    hom.autotune(retime=True)
    before = hom.launch_count
    choice, times = hom.autotune(retime=True)
    assert hom.launch_count - before == 4 * 5 * 4
    assert len(times) == 4 and times[choice] == min(times.values())
