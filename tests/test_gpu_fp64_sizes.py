"""The float64 path on either side of its size rules: small meshes take the CUDA-core kernels, and
the tensor-core kernels at the edges of their tiles, passes and chains on meshes large enough
for them, within the float64 path's 1e-12 of the oracle (Phi pointwise; moments per degree)."""
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


@pytest.mark.parametrize("shape,L", [((4, 4, 16), 2), ((16, 8, 16), 4), ((32, 16, 32), 6), ((40, 24, 17), 8), ((512, 1, 64), 8)])
def test_small_meshes_are_summed_on_cuda_cores(shape, L):
    """A tile of a tensor-core kernel costs more than these meshes' whole sums: their moments are
    those of mp_moments_noalloc, which runs the CUDA-core kernels, to the last bit."""
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    w = W.random_small(shape, L, seed=21, r0=0.9, r1=1.1)
    m = w.mesh
    out = torch.empty(m.shape[0] * m.KL, dtype=torch.float64, device="cuda")
    with mpl.Mesh(m.r, m.theta, m.phi, m.L, m.G, precision="fp64") as mesh:
        mesh.moments_noalloc(torch.from_numpy(w.rho).cuda().reshape(-1), out)
        mesh.synchronize()
    assert np.array_equal(gpu_solve(w, "fp64")["A"], out.cpu().numpy().reshape(m.shape[0], m.KL))


@pytest.mark.parametrize("shape,L", [
    ((40, 40, 141), 20),    # odd azimuthal cells: 8-byte loads, plain stores
    ((6, 90, 200), 40),     # two passes over the density, an expansion in two pieces
    ((2000, 30, 16), 8),    # the fewest azimuthal cells; the column m = 0 in a block of its own
    ((700, 41, 17), 12),    # one more, polar rows that are no multiple of four
    ((130, 131, 64), 5),    # shells past one group of 64 and one of 128
    ((2000, 130, 24), 0),   # the monopole alone
    ((1000, 65, 48), 1),
    ((3000, 3, 64), 16),    # three polar cells
    ((3, 140, 300), 64),    # three chains, the last one short
])
def test_tensor_core_sizes_match_the_oracle(shape, L):
    w = W.random_small(shape, L, seed=L, r0=1.0, r1=1.0 + 0.002 * shape[0] + 0.01, uneven=True)
    ref, got = oracle_solve(w), gpu_solve(w, "fp64")
    assert phi_rel_err(got["phi"], ref["phi"]) <= 1e-12
    assert max(per_l_errors(got["A"], ref["A"], L)) <= 1e-12
    for key, errs in edge_moment_errors(got, ref).items():
        assert max(errs) <= 1e-12, key


@pytest.mark.parametrize("power", [-1000, -850, 900])
def test_power_of_two_scalings_on_a_larger_mesh(power):
    """As for the small mesh: exact, up to what denormal intermediates lose."""
    w = W.random_small((60, 48, 96), 10, seed=17, r0=0.5, r1=1.0)
    base = gpu_solve(w, "fp64", want_moments=False)["phi"]
    w.rho = np.ldexp(w.rho, power)
    got = np.ldexp(gpu_solve(w, "fp64", want_moments=False)["phi"], -power)
    assert phi_rel_err(got, base) <= 1e-13


def test_buffers_on_8_byte_boundaries_of_a_larger_mesh():
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    w = W.random_small((60, 48, 96), 10, seed=18, r0=0.5, r1=1.0)
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


@pytest.mark.parametrize("shape,L", [((60, 48, 96), 10), ((60, 48, 96), 2), ((200, 64, 1), 20), ((400, 8, 32), 30)])
def test_nonfinite_densities_are_reported_by_every_route(shape, L):
    """Projection and synthesis may run on different units: a NaN in the last cell is reported."""
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    w = W.random_small(shape, L, seed=18, r0=0.5, r1=1.0)
    m = w.mesh
    rho = torch.from_numpy(w.rho).cuda()
    rho[-1, -1, -1] = float("nan")
    phi = torch.empty_like(rho)
    with mpl.Mesh(m.r, m.theta, m.phi, m.L, m.G, precision="fp64") as mesh:
        mesh.set_density(rho)
        mesh.set_phi_output(phi)
        mesh.solve()
        with pytest.raises(mpl.MultipoleError) as ei:
            mesh.synchronize()
        assert ei.value.name == "MP_ERR_NONFINITE"
