"""The paired kernels (square planes of side up to 128, and the five-pass form on
any grid) against the FP64 oracle over the z lengths and options their z pass distinguishes: single-step and
two-step lengths, each number of pencils per block, a ragged last block,
non-unit cell lengths, a material table of more than two phases."""
import numpy as np
import pytest

import microstructure as ms
from oracle import rpm_oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5      # single Gamma0-apply, relative L2 (float32 fields)


def _cell(shape, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    lam, mu = zip(*(ms.lame(e, 0.3) for e in (1.0, 10.0, 0.1)))
    l0, m0 = ms.lame(5.0, 0.3)
    return ms.Cell(phase=rng.integers(0, 3, shape).astype(np.uint8), lam=np.array(lam),
                   mu=np.array(mu), lam0=l0, mu0=m0)


def _check(shape, pencil, plane):
    from paper_2003_07720_gb300 import rpm
    nz, ny, nx = shape
    cell = _cell(shape, 100 * nz + nx)
    lengths = (0.7, 1.0, 1.3)
    E = np.array([0.3, -0.2, 0.1, 0.05, -0.04, 0.07])
    x = np.random.Generator(np.random.PCG64(nz)).standard_normal((6,) + shape).astype(np.float32)
    out = torch.full((6,) + shape, float("nan"), device="cuda")
    opts = rpm.rpm_default_options(p_max=0, pencil_variant=pencil, plane_variant=plane)
    with rpm.Context(cell, opts, lengths=lengths) as ctx:
        assert rpm.rpm_plane_variant(ctx.handle) == plane
        ctx.apply_gamma(torch.from_numpy(x).cuda(), E, out)
    got = out.cpu().numpy().astype(np.float64)
    prob = o.Problem(cell.phase, cell.lam, cell.mu, cell.lam0, cell.mu0, lengths=lengths)
    ref = o.apply_F(prob, x.astype(np.float64), E)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < TOL


@pytest.mark.parametrize("nz,n", [(1, 128), (2, 64), (3, 96), (4, 48), (6, 64), (8, 48), (12, 96),
                                  (16, 64), (24, 48), (32, 48), (48, 96), (64, 48), (96, 48),
                                  (128, 96), (256, 64),
                                  # one-warp planes
                                  (32, 32), (24, 24), (16, 16), (6, 12), (8, 8), (6, 6), (3, 4),
                                  (128, 32), (1, 16), (256, 24)])
@pytest.mark.parametrize("pencil", [0, 1, 2])
def test_paired_map_matches_oracle(nz, n, pencil):
    _check((nz, n, n), pencil, 0)


@pytest.mark.parametrize("shape", [
    # every x length with few and with many rows; ragged last row and column blocks
    (2, 8, 4), (64, 256, 4), (3, 4, 6), (12, 16, 8), (6, 6, 12), (4, 24, 16), (16, 96, 24),
    (64, 128, 32), (24, 96, 48), (8, 12, 64), (48, 64, 96), (4, 96, 128), (1, 256, 256),
    # every y length; nz = 256, whose z pass is persistent, with a ragged last tile
    (32, 4, 48), (128, 6, 16), (96, 8, 24), (24, 32, 8), (256, 48, 12), (256, 64, 128)])
@pytest.mark.parametrize("pencil", [0, 2])
def test_five_passes_match_oracle(shape, pencil):
    _check(shape, pencil, 2)


@pytest.mark.parametrize("n,contrast,p_max", [(16, 1e3, 44), (16, 10.0, 12), (48, 10.0, 6)])
def test_reductions_of_every_basis_size(n, contrast, p_max):
    """RPM solves whose reductions take each form of the dot kernels: two and
    more float4 a thread, both differences of a growth at once, results polled
    by the host, and above 32 vectors the chunked launches (16^3 at contrast
    1e3 fills its 44).  The stopping test leaves at most some 100 x 1e-6."""
    from paper_2003_07720_gb300 import rpm
    phase = ms.random_two_phase((n, n, n), 3, 0.3) if n < 48 else ms.centred_sphere(n)
    (l1, m1), (l2, m2) = ms.lame(1.0, 0.3), ms.lame(contrast, 0.3)
    l0, m0 = ms.lame(0.5 * (1.0 + contrast), 0.3)
    cell = ms.Cell(phase=phase, lam=np.array([l1, l2]), mu=np.array([m1, m2]), lam0=l0, mu0=m0)
    E = ms.unit_strain(0)
    ref = o.rpm_solve(o.Problem.from_cell(cell), E,
                      o.Options(tol=1e-8, p_max=p_max, n_max=5, max_iters=3000))
    opts = rpm.rpm_default_options(tol=1e-6, p_max=p_max, n_max=5, max_iters=3000)
    with rpm.Context(cell, opts) as ctx:
        st, info = ctx.solve(E)
    assert ref.converged and info["converged"]
    assert p_max < 44 or info["basis_size"] > 32
    got = np.array(info["mean_stress"])
    assert np.max(np.abs(got - ref.mean_stress)) < 1e-4 * np.max(np.abs(ref.mean_stress))
