"""The float64 path's tensor-core contractions at the sizes where their tiles, passes and chains
change: against the oracle within the float64 path's 1e-12 (pointwise in Phi; moments per
degree), and against themselves under exact scalings of the density."""
import numpy as np
import pytest

from gpu_helpers import edge_moment_errors, gpu_solve, oracle_solve, per_l_errors, phi_rel_err
from paper_2602_02507_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()


def _thin(n_r, n_theta, n_phi, L, **kw):
    return W.presn(n_r=n_r, n_theta=n_theta, n_phi=n_phi, L=L, r_lo=1e7, r_hi=1.02e7 + 2e4 * n_r, **kw)


CASES = {
    # the column m = 0 in a block of its own; three chains of azimuthal cells, the last one short;
    # a ragged last tile of rows
    "own_m0_chains_5x70x300_L32": lambda: _thin(5, 70, 300, 32),
    # one accumulator set too wide for a second one; an odd number of azimuthal cells (8-byte loads)
    "odd_phi_7x40x141_L20": lambda: W.random_small((7, 40, 141), 20, seed=11, r0=0.5, r1=0.7, uneven=True),
    # two passes over the density; both chunks of a long expansion
    "two_passes_3x90x200_L40": lambda: _thin(3, 90, 200, 40),
    "two_chunks_3x100x130_L50": lambda: _thin(3, 100, 130, 50),
    # more than 64 degrees: orders with a second set of columns; the last l_max served, and the
    # first one beyond
    "extra_set_3x140x150_L64": lambda: _thin(3, 140, 150, 64),
    "largest_2x150x146_L71": lambda: _thin(2, 150, 146, 71),
    "beyond_2x150x146_L72": lambda: _thin(2, 150, 146, 72),
    # the fewest azimuthal cells of the tensor-core phi stages, and one fewer
    "phi16_40x9x16_L4": lambda: W.random_small((40, 9, 16), 4, seed=12, r0=0.5, r1=1.0),
    "phi15_40x9x15_L4": lambda: W.random_small((40, 9, 15), 4, seed=13, r0=0.5, r1=1.0),
    # shells past one group of 64 and one of 128; polar cells past one chain
    "groups_130x131x32_L3": lambda: W.random_small((130, 131, 32), 3, seed=14, r0=1.0, r1=2.0),
    "monopole_200x3x24_L0": lambda: W.random_small((200, 3, 24), 0, seed=15, r0=1.0, r1=2.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tile_edges_match_the_oracle(name):
    w = CASES[name]()
    ref, got = oracle_solve(w), gpu_solve(w, "fp64")
    assert phi_rel_err(got["phi"], ref["phi"]) <= 1e-12
    assert max(per_l_errors(got["A"], ref["A"], w.mesh.L)) <= 1e-12
    for key, errs in edge_moment_errors(got, ref).items():
        assert max(errs) <= 1e-12, (key, errs)


def test_cells_of_one_row_far_apart_in_size():
    """Each chain takes its own scale: rows whose cells, and whose chains of 128 cells, differ
    by many orders of magnitude (and in sign)."""
    w = W.random_small((6, 20, 400), 10, seed=16, r0=0.5, r1=0.8)
    rng = np.random.default_rng(16)
    w.rho *= 10.0 ** rng.uniform(-12, 0, w.rho.shape) * 10.0 ** (-(np.arange(400) // 100) * 3.0)
    w.rho[:, :, ::7] *= -0.5
    ref, got = oracle_solve(w), gpu_solve(w, "fp64")
    scale = np.abs(ref["phi"]).max(axis=(1, 2), keepdims=True)
    assert np.max(np.abs(got["phi"] - ref["phi"]) / scale) <= 1e-12


@pytest.mark.parametrize("power", [-1000, -850, 900])
def test_power_of_two_scalings_of_the_density(power):
    """The potential is linear in the density: a scaling by 2^power, down to the bottom of the
    float64 range, scales it exactly (up to what denormal intermediates lose)."""
    w = W.random_small((9, 24, 48), 6, seed=17, r0=0.5, r1=1.0)
    base = gpu_solve(w, "fp64", want_moments=False)["phi"]
    w.rho = np.ldexp(w.rho, power)
    got = np.ldexp(gpu_solve(w, "fp64", want_moments=False)["phi"], -power)
    assert phi_rel_err(got, base) <= 1e-13


def test_buffers_on_8_byte_boundaries():
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    w = W.random_small((6, 30, 64), 8, seed=18, r0=0.5, r1=1.0)
    m = w.mesh
    ref = gpu_solve(w, "fp64", want_moments=False)["phi"]
    rho = torch.empty(w.rho.size + 1, dtype=torch.float64, device="cuda")
    phi = torch.empty_like(rho)
    rho[1:] = torch.from_numpy(w.rho.reshape(-1)).cuda()
    with mpl.Mesh(m.r, m.theta, m.phi, m.L, m.G, precision="fp64") as mesh:
        mesh.set_density(rho[1:])
        mesh.set_phi_output(phi[1:])
        mesh.solve()
        mesh.synchronize()
    assert np.array_equal(phi[1:].cpu().numpy().reshape(ref.shape), ref)


def test_waits_that_run_out_are_reported_and_the_mesh_stays_usable():
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    w = W.random_small((40, 32, 64), 8, seed=19, r0=0.5, r1=1.0)
    m = w.mesh
    ref = gpu_solve(w, "fp64", want_moments=False)["phi"]
    rho = torch.from_numpy(w.rho).cuda()
    phi = torch.empty_like(rho)
    with mpl.Mesh(m.r, m.theta, m.phi, m.L, m.G, precision="fp64") as mesh:
        mesh.set_density(rho)
        mesh.set_phi_output(phi)
        mesh.set_wait_budget(1)
        mesh.solve()
        with pytest.raises(mpl.MultipoleError) as ei:
            mesh.synchronize()
        assert ei.value.name == "MP_ERR_TIMEOUT"
        mesh.set_wait_budget(0)
        mesh.solve()
        mesh.synchronize()
    assert np.array_equal(phi.cpu().numpy(), ref)
