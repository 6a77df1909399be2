"""The gradients of the gravitational source terms where their integer form has its edges: the
float64 expression (Phi[hi] - Phi[lo]) * w is met within one unit in the last place (both round to
nearest; the integer form takes ties away from zero), and zeros, sign changes, denormals,
infinities and NaN go the float64 way exactly."""
import numpy as np
import pytest

from oracle import gravity as OG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__ as g
    g.build()


def _potential(kind, shape):
    rng = np.random.default_rng(7)
    smooth = -1e19 / (1.0 + np.arange(shape[0])[:, None, None] * 0.01) * (1.0 + 1e-3 * rng.standard_normal(shape))
    if kind == "smooth":
        return smooth
    if kind == "nearly_equal":  # differences of a few units in the last place, and none
        return smooth[0, 0, 0] * (1.0 + 2.0 ** -52 * rng.integers(0, 3, shape))
    if kind == "sign_changes":
        return rng.standard_normal(shape)
    if kind == "far_apart":
        return -(2.0 ** rng.uniform(-14, 14, shape))
    if kind == "range_ends":  # down to denormals, up to where differences overflow
        return np.ldexp(-1.0 - rng.random(shape), rng.choice([-1073, -1030, -1000, 0, 1000, 1023], shape))
    p = smooth.copy()
    p.flat[rng.integers(0, p.size, p.size // 7)] = 0.0
    p.flat[rng.integers(0, p.size, p.size // 9)] = np.inf
    p.flat[rng.integers(0, p.size, p.size // 11)] = np.nan
    return p


@pytest.mark.parametrize("kind", ["smooth", "nearly_equal", "sign_changes", "far_apart", "range_ends", "special"])
@pytest.mark.parametrize("shape", [(5, 4, 33), (4, 3, 64), (3, 5, 66), (2, 2, 190), (3, 1, 1), (1, 4, 130)])
def test_gradient_matches_the_float64_expression(kind, shape):
    import torch
    from paper_2602_02507_gb300 import multipole as mpl
    n_r, n_t, n_p = shape
    r, th = np.linspace(0.5, 1.5, n_r + 1) ** 2, np.linspace(0.0, np.pi, n_t + 1)
    ph = np.linspace(0.0, 2.0 * np.pi, n_p + 1)
    phi = _potential(kind, shape)
    with np.errstate(all="ignore"):
        want = np.zeros((3,) + shape)
        for a, (edges, wraps) in enumerate(((r, False), (th, False), (ph, True))):
            lo, hi, dx = OG.stencil(edges, wraps)
            w = np.where(dx != 0.0, 1.0 / np.where(dx != 0.0, dx, 1.0), 0.0)
            want[a] = (phi.take(hi, axis=a) - phi.take(lo, axis=a)) * w.reshape([-1 if d == a else 1 for d in range(3)])
    grad = torch.empty(3 * phi.size, dtype=torch.float64, device="cuda")
    S = torch.empty_like(grad)
    with mpl.Mesh(r, th, ph, 2, 1.0, precision="fp64") as mesh:
        mesh.gravity_sources(phi=torch.from_numpy(phi).cuda().reshape(-1), rho=torch.ones(phi.size, dtype=torch.float64, device="cuda"),
                             grad=grad, S=S)
        mesh.synchronize()
    got = grad.cpu().numpy().reshape(want.shape)
    fine = np.isfinite(want)
    assert np.array_equal(np.isnan(want), np.isnan(got))
    assert np.array_equal(got[~fine & ~np.isnan(want)], want[~fine & ~np.isnan(want)])
    assert np.all(np.abs(got[fine] - want[fine]) <= 2.3e-16 * np.abs(want[fine]) + 5e-324)
    assert np.array_equal(S.cpu().numpy().reshape(want.shape)[fine], -got[fine])
