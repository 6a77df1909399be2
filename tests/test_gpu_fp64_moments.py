"""The float64 path's moments: where they are the sums of the CUDA-core kernels to the last bit
(mp_moments_noalloc runs those kernels), and how near the oracle's they are elsewhere."""
import numpy as np
import pytest

from gpu_helpers import gpu_solve
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
