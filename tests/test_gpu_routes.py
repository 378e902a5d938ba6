"""What rides on the map's last pass, its modes on ragged and persistent tiles,
and its capture into a graph, over the grids that the paired kernels serve:
against the FP64 oracle, element by element."""
import numpy as np
import pytest

import microstructure as ms
from oracle import rpm_oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5      # one map, relative L2 (float32 fields)


@pytest.fixture(scope="module")
def rpm():
    from paper_2003_07720_gb300 import rpm as r
    return r


def _cell(shape, phases, seed):
    """Voxel-wise random phases of different Poisson ratios."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lam, mu = zip(*[ms.lame(e, nu) for e, nu in ((1.0, 0.3), (10.0, 0.2), (0.3, 0.4))[:phases]])
    l0, m0 = ms.lame(2.0, 0.3)
    return ms.Cell(phase=rng.integers(0, phases, shape).astype(np.uint8), lam=np.array(lam),
                   mu=np.array(mu), lam0=l0, mu0=m0)


def _field(shape, E, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return (np.reshape(E, (6, 1, 1, 1)) + 0.2 * rng.standard_normal((6,) + shape)).astype(np.float32)


def _err(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("shape,plane", [
    # the post-step in clusters of one-warp blocks (single-step lengths), of two warps
    ((1, 16, 16), 0), ((2, 4, 4), 0), ((6, 6, 6), 0), ((4, 8, 8), 0), ((16, 12, 12), 0),
    ((24, 24, 24), 0), ((3, 32, 32), 0),
    # 96^2 in blocks of 128 threads (more than 50 planes)
    ((64, 96, 96), 0),
    # the post-step as a kernel of its own: unequal sides, 256^2, forced variants
    ((12, 16, 8), 0), ((4, 24, 96), 0), ((1, 256, 256), 0), ((8, 24, 24), 1), ((16, 48, 48), 2)])
@pytest.mark.parametrize("phases", [2, 3])
def test_polarization_map_on_every_route(rpm, shape, plane, phases):
    """One step of Algorithm 3 from a given field."""
    cell = _cell(shape, phases, 10 * shape[0] + shape[2])
    E = np.array([0.3, -0.2, 0.1, 0.05, -0.04, 0.07])
    x = _field(shape, E, 5)
    out = torch.full((6,) + shape, float("nan"), device="cuda")
    opts = rpm.rpm_default_options(scheme=rpm.RPM_SCHEME_POLARIZATION, alpha=1.5, beta=1.2,
                                   max_iters=1, tol=0.0, p_max=0, plane_variant=plane)
    with rpm.Context(cell, opts) as ctx:
        st, info = ctx.solve(E, eps0=torch.from_numpy(x).cuda(), eps_out=out, raise_on_failure=False)
    assert st == rpm.RPM_ERR_NOT_CONVERGED and info["iters"] == 1
    ref = o.apply_F_polarization(o.Problem.from_cell(cell), x.astype(np.float64), E, 1.5, 1.2)
    assert _err(out.cpu().numpy().astype(np.float64), ref) < TOL


@pytest.mark.parametrize("shape,plane", [
    # five passes, the last row block ragged: one- and two-step rows, small and large blocks
    ((2, 6, 12), 0), ((4, 12, 16), 0), ((64, 48, 16), 0), ((2, 12, 48), 0), ((16, 48, 64), 0),
    ((32, 32, 32), 2),
    # three passes, and the addition as a kernel of its own
    ((8, 24, 24), 0), ((16, 48, 48), 0), ((16, 48, 48), 1)])
def test_the_defect_of_a_recentred_iterate_is_added(rpm, shape, plane):
    """Plain iteration at contrast 100 gains less than a half in 8 steps, so with
    n_max = 1 it is re-centred again and again and every later map adds the
    defect; what it stops at has to be a fixed point of the oracle's map (to the
    stopping test, 1e-5, and one map's rounding)."""
    phase = ms.random_two_phase(shape, 3, 0.4)
    (l1, m1), (l2, m2), (l0, m0) = ms.lame(1.0, 0.3), ms.lame(100.0, 0.3), ms.lame(50.5, 0.3)
    cell = ms.Cell(phase=phase, lam=np.array([l1, l2]), mu=np.array([m1, m2]), lam0=l0, mu0=m0)
    E = np.array([0.6, -0.3, 0.2, 0.3, -0.2, 0.4])
    out = torch.full((6,) + shape, float("nan"), device="cuda")
    opts = rpm.rpm_default_options(tol=1e-5, p_max=0, n_max=1, plane_variant=plane)
    with rpm.Context(cell, opts) as ctx:
        res, _ = ctx.trace()
        st, info = ctx.solve(E, eps_out=out)
    r = res[np.isfinite(res)]          # read every fourth step
    assert np.sum(r[2:] > 0.5 * r[:-2]) >= 2, "no stall: nothing was re-centred"
    prob = o.Problem.from_cell(cell)
    eps = out.cpu().numpy().astype(np.float64)
    assert o.residual(prob, o.apply_F(prob, eps, E), eps, E) < 2e-5


@pytest.mark.parametrize("shape", [
    # two-step and single-step planes, the persistent z pass, few planes, ragged rows and columns
    (12, 96, 96), (256, 24, 24), (1, 128, 128), (256, 48, 12), (1, 256, 256), (64, 128, 32),
    (2, 8, 4), (16, 96, 24), (6, 12, 48)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_two_phase_map_in_every_mode(rpm, shape, mode):
    cell = _cell(shape, 2, shape[0] + shape[1])
    E = np.array([0.3, -0.2, 0.1, 0.05, -0.04, 0.07])
    x = _field(shape, E, 7)
    out = torch.full((6,) + shape, float("nan"), device="cuda")
    with rpm.Context(cell, rpm.rpm_default_options(p_max=0)) as ctx:
        ctx.apply_gamma(torch.from_numpy(x).cuda(), E, out, mode)
    prob, xx = o.Problem.from_cell(cell), x.astype(np.float64)
    ref = (o.apply_F(prob, xx, E) if mode == 0 else
           o.apply_F_linear(prob, xx) if mode == 1 else o.apply_gamma_raw(prob, xx))
    assert _err(out.cpu().numpy().astype(np.float64), ref) < TOL


@pytest.mark.parametrize("shape", [(4, 4, 4), (16, 16, 16), (32, 32, 32), (48, 48, 48),
                                   (1, 256, 256), (24, 96, 48), (8, 12, 6)])
def test_maps_captured_into_a_graph(rpm, shape):
    """Three chained maps, launched early one after the other, captured once and
    replayed on new inputs: bitwise the maps called one at a time."""
    cell = _cell(shape, 3, 4)
    E = ms.unit_strain(0)
    stream = torch.cuda.Stream()
    a, b, c, d = (torch.empty((6,) + shape, device="cuda") for _ in range(4))
    xs = [torch.from_numpy(_field(shape, E, 20 + k)).cuda() for k in range(3)]
    with rpm.Context(cell, rpm.rpm_default_options(p_max=0), stream=stream) as ctx:
        want = []
        for x in xs:
            a.copy_(x)
            for s, t in ((a, b), (b, c), (c, d)):
                torch.cuda.synchronize()
                ctx.apply_gamma(s, E, t)
            torch.cuda.synchronize()
            want.append(d.clone())
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            ctx.apply_gamma(a, E, b)
            ctx.apply_gamma(b, E, c)
            ctx.apply_gamma(c, E, d)
        for x, w in zip(xs, want):
            a.copy_(x)
            b.zero_(), c.zero_(), d.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(d, w)
