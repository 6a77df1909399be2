"""The m = 0 kernels beside the tensor-core theta stages, at the edges of their tiles (16 to 80
degrees and 8 shells of the contraction; groups of 8 degrees, 4 or 8 shells and up to 128 polar
cells of the synthesis), against the oracle within the split path's bars: 1e-6 of Phi, and for the
m = 0 moments the bar of the error model relative to the sum of the magnitudes of their terms."""
import pytest

from gpu_helpers import gpu_solve, moment_term_errors, oracle_solve, phi_rel_err, split_moment_bar, term_scales
from paper_2602_02507_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()


# n_r, n_theta, n_phi, l_max: one to five groups of 16 degrees, each full and one degree more; two
# blocks of degrees; one and two tiles of polar cells; ragged last shells; eight shells a thread
@pytest.mark.parametrize("shape,L", [((1, 129, 32), 1), ((9, 32, 32), 15), ((7, 31, 48), 16), ((5, 130, 64), 31),
                                     ((8, 127, 80), 32), ((6, 97, 112), 48), ((3, 140, 144), 64), ((3, 161, 176), 79),
                                     ((4, 170, 176), 80), ((2435, 33, 32), 7)])
def test_m0_columns_match_the_oracle(shape, L):
    w = W.random_small(shape, L, seed=L, r0=1.0, r1=1.0 + 0.001 * shape[0], uneven=True)
    ref = oracle_solve(w)
    got = gpu_solve(w, "bf16x3", engine="tensor")
    assert got["info"]["effective_precision"] == 1 and got["info"]["theta_tensor_cores"] == 1
    assert phi_rel_err(got["phi"], ref["phi"]) <= 1e-6
    err = moment_term_errors(got["A"], ref["A"], term_scales(w.rho, ref["tables"], w.mesh.G), L)
    assert max(err) <= split_moment_bar(w.mesh, "bf16x3"), err
