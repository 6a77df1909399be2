"""The float64 path's moments: where they are the sums of the CUDA-core kernels to the last bit
(mp_moments_noalloc runs those kernels), and how near the oracle's they are elsewhere."""
import numpy as np
import pytest

from gpu_helpers import edge_term_errors, gpu_solve, moment_term_errors, oracle_solve, term_scales
from paper_2602_02507_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()


def cuda_core_moments(w):
    """Angular moments [n_r][K_L] as the CUDA-core kernels sum them."""
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    m = w.mesh
    rho = torch.from_numpy(np.ascontiguousarray(w.rho)).cuda().reshape(-1)
    out = torch.empty(m.shape[0] * m.KL, dtype=torch.float64, device="cuda")
    with mpl.Mesh(m.r, m.theta, m.phi, m.L, m.G, precision="fp64") as mesh:
        mesh.moments_noalloc(rho, out)
        mesh.synchronize()
    return out.cpu().numpy().reshape(m.shape[0], m.KL)


@pytest.mark.parametrize("shape,L", [((260, 24, 32), 50), ((260, 40, 150), 64), ((260, 24, 8), 56)])
def test_moments_whose_squares_overflow_are_the_cuda_core_sums(shape, L):
    """Over five decades of r the edge moments of these degrees have no norm (M^R reaches 1e150
    and more): two solutions can be compared by equality alone, so the order of their sums stays."""
    w = W.presn(n_r=shape[0], n_theta=shape[1], n_phi=shape[2], L=L)
    w.rho *= 0.5 + np.random.default_rng(L).random(w.rho.shape)
    got = gpu_solve(w, "fp64")
    assert np.array_equal(got["A"], cuda_core_moments(w))
    assert np.all(np.isfinite(got["MR"])) and np.all(np.isfinite(got["MI"]))


@pytest.mark.parametrize("L,center,width", [(8, 0.15, 0.05), (32, 0.15, 0.05), (32, 3.0, 0.02), (40, 0.4, 0.1), (71, 0.3, 0.1)])
def test_every_moment_of_a_clump_near_the_pole(L, center, width):
    """A clump beside the axis: its cells meet the smallest entries of the polar tables (sin^m
    theta).  Every A_lm, M^R and M^I is within the float64 path's 1e-12 of the sum of the magnitudes
    of its own terms; float64 sums of 128 + 256 terms stay below 400 * 2^-53 = 5e-14 of it."""
    w = W.random_small((20, 128, 256), L, seed=L, r0=0.5, r1=1.0)
    thc, phc = (0.5 * (e[1:] + e[:-1]) for e in (w.mesh.theta, w.mesh.phi))
    w.rho *= np.exp(-((thc[:, None] - center) / width) ** 2 - ((phc[None, :] - 1.0) / 0.5) ** 2)[None]
    ref, got = oracle_solve(w), gpu_solve(w, "fp64")
    S = term_scales(w.rho, ref["tables"], w.mesh.G)
    assert max(moment_term_errors(got["A"], ref["A"], S, L)) <= 1e-12
    for key, errs in edge_term_errors(got, ref, S).items():
        assert max(errs) <= 1e-12, key


def test_theta_rows_are_summed_as_the_cuda_core_kernels_do():
    """With few azimuthal cells both steps of the moments run on CUDA cores: blocks of 16 and 32
    shells, 32 degrees and 32 polar cells, each with a remainder, equal k64_theta to the last bit."""
    for shape, L in (((33, 33, 3), 33), ((17, 64, 2), 40), ((1, 1, 1), 0), ((40, 31, 15), 64), ((16, 70, 1), 31)):
        w = W.random_small(shape, L, seed=5, r0=0.9, r1=1.0, uneven=True)
        assert np.array_equal(gpu_solve(w, "fp64")["A"], cuda_core_moments(w)), (shape, L)


@pytest.mark.parametrize("n_phi", [128, 500, 2048])
def test_small_cells_beside_a_large_one_are_rounded_both_ways(n_phi):
    """One cell of each ring is 2^30 times the others: their last bits do not fit the ring's fixed
    point.  Truncated, they would take n_phi 2^-56 off the monopole; rounded to nearest they leave
    sqrt(n_phi) 2^-57, below the rounding of the 16 polar terms and their table (16 * 2^-53) and
    of the sums of the chains of 128 cells (2^-50 of the hot cell for 2048): 5e-15 holds both."""
    w = W.random_small((4, 16, n_phi), 2, seed=n_phi, r0=0.5, r1=1.0)
    rng = np.random.default_rng(n_phi)
    w.rho *= 2.0 ** -30
    hot = rng.integers(0, n_phi, (4, 16))
    np.put_along_axis(w.rho, hot[:, :, None], 1.0, axis=2)
    m = w.mesh
    LD = np.longdouble
    polar = -np.diff(np.cos(m.theta.astype(LD)))
    ring = (w.rho.astype(LD) * np.diff(m.phi.astype(LD))).sum(axis=2)
    exact = (ring * polar).sum(axis=1) * np.sqrt(4 * np.arccos(LD(-1)))
    got = gpu_solve(w, "fp64")["A"][:, 0]
    assert np.max(np.abs(got - exact) / exact) <= 5e-15


@pytest.mark.parametrize("ratio", [1e-6, 0.04, 0.7])
def test_a_large_density_in_a_narrow_azimuthal_cell(ratio):
    """The other cells of the ring keep their bits beside a hot cell that is narrow: within 1e-13 of
    the sum of the terms' magnitudes (float64 sums of 32 + 64 terms: 96 * 2^-53 = 1.1e-14, and
    tables that agree to a few 1e-14)."""
    w = W.random_small((8, 32, 64), 12, seed=3, r0=0.5, r1=1.0)
    width = np.ones(64)
    width[10] = ratio
    edges = np.concatenate([[0.0], np.cumsum(width)])
    w.mesh.phi[:] = edges / edges[-1] * 2.0 * np.pi
    w.rho[:] = 1e-6
    w.rho[:, :, 10] = np.exp(0.5 * (w.mesh.r[1:] + w.mesh.r[:-1]))[:, None]
    ref, got = oracle_solve(w), gpu_solve(w, "fp64")
    S = term_scales(w.rho, ref["tables"], w.mesh.G)
    assert max(moment_term_errors(got["A"], ref["A"], S, 12)) <= 1e-13
    assert np.max(np.abs(got["phi"] - ref["phi"]) / np.abs(ref["phi"])) <= 1e-12
