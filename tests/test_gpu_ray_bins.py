"""Ray tracing (csrc/kt_ray.cu) against the FP64 reference over what its exponential and its
register bins distinguish: one to eight bins, vacuum, optical depths per cell from 1e-20
(1 - e^-tau = tau to the last bit) over 1e-3 (where 1 - e^-tau would cancel) to beyond 700
(the general path), rays along the axes and rays that start outside."""
import numpy as np
import pytest

from oracle import raytrace as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_04941_gb300 import build, kt as ktm
    build.build()
    return ktm


@pytest.mark.parametrize("nb", [1, 2, 3, 4, 5, 8])
def test_bins_and_optical_depths(kt, nb):
    import torch
    rng = np.random.default_rng(nb)
    shape, h, dt = (7, 9, 5), (0.3, 0.45, 0.37), 0.2
    kappa = np.empty((nb,) + shape)
    for b in range(nb):
        lo, hi = [(-20, -1), (-4, 0), (-1, 1.5), (2.0, 4.5)][b % 4]
        kappa[b] = 10.0 ** rng.uniform(lo, hi, shape)
    kappa[:, 1] = 0.0
    src = np.array([3.4, 4.6, 2.3]) * h
    org, dirs, n0 = R.point_source_rays(src, [1.0 + b for b in range(nb)], dt, 300)
    axes = np.concatenate([np.eye(3), -np.eye(3)])
    org = np.concatenate([org, np.tile(src, (6, 1)), [[-1.0, 0.1, 0.1]]])
    dirs = np.concatenate([dirs, axes, [[1.0, 0.0, 0.0]]])
    n0 = np.concatenate([n0, np.ones((7, nb))])
    fo, ao, eo, _ = R.trace(shape, h, kappa, org, dirs, n0, dt)
    f, a, e = (t.cpu().numpy() for t in kt.raytrace(h, *(torch.from_numpy(np.ascontiguousarray(v)).cuda()
                                                         for v in (kappa, org, dirs, n0)), dt))
    for b in range(nb):
        assert np.allclose(f[b], fo[b], rtol=1e-11, atol=1e-13 * fo[b].max())
        # the reference sums N (1 - e^-tau), which cancels below tau ~ 1e-3: absolute there
        assert np.allclose(a[b], ao[b], rtol=1e-11, atol=1e-15 * n0[:, b].sum())
        assert np.allclose(e[:, b], eo[:, b], rtol=1e-11, atol=1e-14 * n0[:, b].max())
