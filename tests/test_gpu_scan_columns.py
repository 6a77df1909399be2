"""The radial recurrences with four moment columns a block, at 4, 8 and 16 shells a thread (the
warps' sums go one way below 16 and another at 16), a ragged last chunk and a last block of one
column: against the oracle within the float64 path's 1e-12 (pointwise in Phi; moments per degree)."""
import pytest

from gpu_helpers import edge_moment_errors, gpu_solve, oracle_solve, phi_rel_err
from paper_2602_02507_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()


# (L + 1)^2 columns: 625 (one over a multiple of four) and 676
@pytest.mark.parametrize("n_r,L", [(3, 24), (511, 24), (513, 25), (1023, 24), (1025, 24)])
def test_four_columns_a_block_match_the_oracle(n_r, L):
    w = W.random_small((n_r, 40, 60), L, seed=n_r, r0=1.0, r1=1.0 + 0.0005 * n_r)
    ref, got = oracle_solve(w), gpu_solve(w, "fp64")
    assert phi_rel_err(got["phi"], ref["phi"]) <= 1e-12
    for key, errs in edge_moment_errors(got, ref).items():
        assert max(errs) <= 1e-12, (key, errs)
