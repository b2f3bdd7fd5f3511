"""Grids with odd axes (GPU): every axis is halved level by level, the last
cell of an odd axis made of three, down to a dense coarsest level, and the
solve lands on the oracle's solution."""
import numpy as np
import pytest

import oracle
import paris_inputs as pi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, W = pi.PERIODIC, pi.WALL
# odd finest axes, axes that turn odd after one and two halvings, long thin boxes, periodic odd axes
GRIDS = [pi.Grid(45, 31, 27, 1 / 45, (W, W, W)), pi.Grid(50, 26, 34, 1 / 50, (W, P, W)),
         pi.Grid(33, 33, 33, 1 / 33, (P, P, P)), pi.Grid(36, 20, 44, 1 / 44, (P, W, P)),
         pi.Grid(5, 6, 203, 1 / 203, (W, W, W)), pi.Grid(131, 3, 9, 1 / 131, (P, W, W))]
ids = lambda g: f"{g.nx}x{g.ny}x{g.nz}_{''.join('pw'[b] for b in g.bc)}"


@pytest.fixture(scope="module")
def paris():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2012_11744_gb300 as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("grid", GRIDS, ids=ids)
def test_odd_axes_match_oracle(paris, grid, precision):
    """p and u to 1e-8 of the oracle's (the parity bar of the other grids),
    without falling back to the other precision."""
    pr = pi.random_problem(grid, seed=41, rho1=1000.0)
    ref = oracle.projection_step(grid, pr.C, pr.rho1, pr.rho2, pr.dt, pr.u, pr.v, pr.w)
    with paris.Context(grid, opts=paris.default_opts(precision=getattr(paris, precision))) as ctx:
        u, p = [dev(x) for x in (pr.u, pr.v, pr.w)], torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
        st = ctx.projection_step(dev(pr.C), pr.rho1, pr.rho2, pr.dt, *u, p)
    assert st["converged"] == 1 and st["fell_back"] == 0, st
    assert np.abs(p.cpu().numpy() - ref.p).max() <= 1e-8 * np.abs(ref.p).max()
    umax = max(np.abs(x).max() for x in (pr.u, pr.v, pr.w))
    for a in range(3):
        assert np.abs(u[a].cpu().numpy() - ref.u[a]).max() <= 1e-8 * umax


@pytest.mark.parametrize("grid", [GRIDS[0], GRIDS[4], pi.Grid(41, 48, 57, 1 / 57, (W, P, W))], ids=ids)
def test_tail_and_fused_sweep_bit_identical_on_odd_levels(paris, grid):
    """The single-block tail and the fused sweep do the arithmetic of the
    per-level kernels on levels with odd axes too (periodic axes even on
    every smoothed level, where a colour pass has one result)."""
    pr = pi.random_problem(grid, seed=43, rho1=1000.0)
    out = []
    for kw in ({"coarse_tail": 1}, {"coarse_tail": 0}, {"smoother": paris.SMOOTH_RBGS}):
        with paris.Context(grid, opts=paris.default_opts(level0_density=0, **kw)) as ctx:
            u, p = [dev(x) for x in (pr.u, pr.v, pr.w)], torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
            ctx.projection_step(dev(pr.C), pr.rho1, pr.rho2, pr.dt, *u, p)
            out.append(p.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])


@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("nu", [(2, 2), (1, 2), (2, 1)], ids=lambda n: f"nu{n[0]}{n[1]}")
@pytest.mark.parametrize("grid", [pi.Grid(130, 4, 90, 1 / 130, (W, P, W)), pi.Grid(46, 58, 34, 1 / 58, (W, W, W)),
                                  pi.Grid(40, 64, 36, 1 / 64, (P, P, W)), pi.Grid(64, 64, 64, 1 / 64, (P, P, P))],
                         ids=ids)
def test_box_levels_bit_identical(paris, grid, nu, precision):
    """A small level's half of the V-cycle in one launch and by its passes,
    restriction and prolongation: the same arithmetic in the same order
    (boxes cut off by walls and odd axes, an axis shorter than the halo, one
    that is not halved, one and two sweeps; conjugate gradients may run out of
    iterations where the numbers of sweeps differ, the V-cycle then being
    unsymmetric, in both forms alike)."""
    pr = pi.random_problem(grid, seed=47, rho1=1000.0)
    out = []
    for tail in (0, 1):
        opts = paris.default_opts(precision=getattr(paris, precision), coarse_tail=tail, nu1=nu[0], nu2=nu[1])
        with paris.Context(grid, opts=opts) as ctx:
            u, p = [dev(x) for x in (pr.u, pr.v, pr.w)], torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
            try:
                ran_out = 0
                ctx.projection_step(dev(pr.C), pr.rho1, pr.rho2, pr.dt, *u, p)
            except paris.ParisError as e:
                assert e.status == 3 and nu[0] != nu[1]
                ran_out = 1
            out.append([np.array(ran_out)] + [x.cpu().numpy() for x in (p, *u)])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("grid", [pi.Grid(58, 7, 45, 1 / 58, (W, W, W)), pi.Grid(22, 55, 6, 1 / 55, (W, W, W)),
                                  pi.Grid(31, 111, 50, 1 / 111, (W, W, W)), pi.Grid(52, 9, 75, 1 / 75, (W, W, W))],
                         ids=ids)
def test_tail_of_mixed_factors_bit_identical(paris, grid, precision):
    """Tails whose coarse cells have one, two and three children along
    different axes (an axis no longer halved beside an odd one)."""
    pr = pi.random_problem(grid, seed=53, rho1=1000.0)
    out = []
    for tail in (0, 1):
        opts = paris.default_opts(precision=getattr(paris, precision), coarse_tail=tail)
        with paris.Context(grid, opts=opts) as ctx:
            u, p = [dev(x) for x in (pr.u, pr.v, pr.w)], torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
            st = ctx.projection_step(dev(pr.C), pr.rho1, pr.rho2, pr.dt, *u, p)
            assert st["converged"] == 1 and st["fell_back"] == 0, (tail, st)
            out.append([x.cpu().numpy() for x in (p, *u)])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("grid", [pi.Grid(31, 111, 50, 1 / 111, (W, W, P)), pi.Grid(50, 31, 60, 1 / 60, (P, W, P)),
                                  pi.Grid(100, 6, 100, 1 / 100, (P, W, P))], ids=ids)
def test_tail_with_odd_periodic_levels_converges(paris, grid, precision):
    """Levels whose periodic axes turn odd inside the tail (cells of one
    colour meet across the seam): the V-cycle stays symmetric enough for
    conjugate gradients, within twice the iterations (and five) of the
    levels' own kernels."""
    pr = pi.random_problem(grid, seed=82, rho1=234.0)
    its = []
    for tail in (0, 1):
        opts = paris.default_opts(precision=getattr(paris, precision), coarse_tail=tail)
        with paris.Context(grid, opts=opts) as ctx:
            u, p = [dev(x) for x in (pr.u, pr.v, pr.w)], torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
            st = ctx.projection_step(dev(pr.C), pr.rho1, pr.rho2, pr.dt, *u, p)
            assert st["converged"] == 1 and st["fell_back"] == 0, (tail, st)
            its.append(st["iters"])
    assert its[1] <= 2 * its[0] + 5, its


@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("density", [0, 1])
@pytest.mark.parametrize("grid", [pi.Grid(33, 33, 33, 1 / 33, (P, P, P)), pi.Grid(50, 26, 34, 1 / 50, (W, P, P)),
                                  pi.Grid(132, 33, 20, 1 / 132, (P, P, W)), pi.Grid(264, 66, 18, 1 / 264, (P, P, P)),
                                  pi.Grid(9, 30, 75, 1 / 75, (P, W, P))], ids=ids)
def test_odd_periodic_axes_bit_identical(paris, grid, density, precision):
    """Where a periodic axis has an odd number of cells, cells of one colour
    meet across its seam.  Every form of the colour passes takes them as they
    were before the pass: run twice, with the small levels in one launch or by
    their own kernels, slab by slab and as the fused sweep (which writes to a
    second array) the result is the same.  Rows of at least a warp's vectors,
    pairs, FP16 level 1, levels of more than 512 cells."""
    pr = pi.random_problem(grid, seed=59, rho1=1000.0)
    forms = [{}, {}, {"coarse_tail": 0}, {"slab_planes": 3}]
    if not density or precision == "FP64":
        forms.append({"smoother": paris.SMOOTH_RBGS})
    out = []
    for kw in forms:
        opts = paris.default_opts(precision=getattr(paris, precision), level0_density=density, **kw)
        with paris.Context(grid, opts=opts) as ctx:
            u, p = [dev(x) for x in (pr.u, pr.v, pr.w)], torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
            st = ctx.projection_step(dev(pr.C), pr.rho1, pr.rho2, pr.dt, *u, p)
            assert st["converged"] == 1 and st["fell_back"] == 0, (kw, st)
            out.append([x.cpu().numpy() for x in (p, *u)])
    for kw, o in zip(forms, out):
        for a, b in zip(out[0], o):
            np.testing.assert_array_equal(a, b, err_msg=str(kw))
