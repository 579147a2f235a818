"""Slopes of the advection sweep at the ends of the double range (csrc/kt_advect.cu half_slope)
and sweeps against the numpy reference for either sign of dt/dx."""
import numpy as np
import pytest

from oracle import advection as A
from paper_2504_04941_gb300 import inputs as I
from test_gpu_advect_windows import _network, kt  # noqa: F401

pytestmark = pytest.mark.gpu


def _sweep(kt, netw, n, rho, flux, dtdx, project):  # noqa: F811
    import torch
    return kt.advect_sweep(kt.Network(netw), *(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (n, rho, flux)),
                           0.37, dtdx, project=project).cpu().numpy()


@pytest.mark.parametrize("project", [False, True])
@pytest.mark.parametrize("low,high", [(1e-310, 1e-5), (5e-324, 1.0), (2.5e-308, 1.0), (4.2e-308, 3e-3), (1e-200, 1e-180),
                                      (1e-308, 2e-308)])
def test_small_abundances_between_ordinary_ones(kt, low, high, project):  # noqa: F811
    """Neighbours 0, low, high (and falling again): a slope limited by half a subnormal
    difference stays finite, the other species are not touched by it."""
    netw = _network(4, 2, 1)
    rng = np.random.default_rng(5)
    n = rng.uniform(0.1, 1.0, (4, 3, 40))
    n[1] = 0.0
    for at, v in enumerate((0.0, low, high, high, low, 0.0, low, high)):
        n[1, :, 5 + at] = v
    n[1, 1] = n[1, 1, ::-1]
    rho, flux = np.ones((3, 40)), np.concatenate([np.full((2, 40), 0.8), np.full((1, 40), -0.8)])
    ref = A.advect_step(n, rho, flux, 0.3, 0.37, A.element_projector(netw.counts) if project else None)
    got = _sweep(kt, netw, n, rho, flux, 0.3, project)
    assert np.all(np.isfinite(got))
    # without projection a species depends on itself only: 1e-12 of the largest of its stencil
    size = np.abs(n) if not project else np.broadcast_to(np.abs(n).max(0), n.shape)
    near = np.max([np.roll(size, k, -1) for k in (-2, -1, 0, 1, 2)], axis=0)
    assert np.all(np.abs(got - ref) <= 1e-12 * near + 1e-322)


def test_large_abundances(kt):  # noqa: F811
    """Differences whose reciprocal is subnormal."""
    netw = _network(2, 1, 3)
    rng = np.random.default_rng(6)
    n = rng.uniform(0.0, 1.0, (2, 2, 30)) * 1e308
    rho, flux = np.full((2, 30), 1.0), rng.uniform(-0.5, 0.5, (2, 30))
    got = _sweep(kt, netw, n, rho, flux, 0.3, False)
    # the same with everything scaled by 2^-40, where nothing is near the range's end
    ref = A.advect_step(n * 2.0 ** -40, rho, flux, 0.3, 0.37, None)
    assert np.all(np.abs(got * 2.0 ** -40 - ref) <= 1e-12 * 1e308 * 2.0 ** -40)


@pytest.mark.parametrize("project", [False, True])
@pytest.mark.parametrize("dtdx", [-0.3, 0.0, 0.3])
def test_upwind_side_follows_the_flux_for_either_sign_of_dtdx(kt, dtdx, project):  # noqa: F811
    netw = _network(5, 2, 4)
    rng = np.random.default_rng(8)
    n, rho, flux = rng.uniform(0.1, 1.0, (5, 4, 33)), rng.uniform(0.5, 2.0, (4, 33)), rng.uniform(-1.0, 1.0, (4, 33))
    ref = A.advect_step(n, rho, flux, dtdx, 0.37, A.element_projector(netw.counts) if project else None)
    got = _sweep(kt, netw, n, rho, flux, dtdx, project)
    assert np.all(np.abs(got - ref) <= 1e-12 * (n.max() + 0.6 * (n / rho[None]).max()))
