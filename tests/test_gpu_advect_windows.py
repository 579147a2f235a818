"""Windows of the advection sweep (csrc/kt_advect.cu) against the numpy reference: every
window width, lines shorter than a window, lengths one off its multiples, odd lengths and an
odd base address (no 16-byte accesses), one species, the largest element rank, vacuum and
infinite abundances."""
import numpy as np
import pytest

from oracle import advection as A
from paper_2504_04941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_04941_gb300 import build, kt as ktm
    build.build()
    return ktm


def _network(ns, ne, seed):
    rng = np.random.default_rng(seed)
    counts = rng.integers(0, 4, (ns, ne))
    counts[:ne] += np.eye(min(ns, ne), ne, dtype=int)
    return I._irreversible("adv", [f"S{i}" for i in range(ns)], [f"E{i}" for i in range(ne)], np.ones(ns), np.zeros(ns),
                           np.ones(ns), counts, 0, 300.0, 10.0, 1e5, [((0,), (0,), 1.0, 0.0, 0.0, -1)])


@pytest.mark.parametrize("ns,ne,nl,L,odd", [(1, 1, 5, 3, 0), (3, 2, 9, 4, 0), (3, 2, 9, 5, 1), (10, 2, 7, 12, 0),
                                            (10, 2, 7, 13, 0), (10, 3, 6, 28, 1), (11, 3, 5, 29, 0), (32, 3, 4, 60, 0),
                                            (32, 3, 3, 61, 0), (40, 8, 3, 120, 1), (64, 4, 2, 122, 0), (250, 2, 1, 64, 0)])
def test_windows_match_reference(kt, ns, ne, nl, L, odd):
    import torch
    netw = _network(ns, ne, ns + L)
    rng = np.random.default_rng(L * 10 + ns)
    n = 10.0 ** rng.uniform(-8, 0, (ns, nl, L))
    n[0] = 0.0                                     # vacuum in one species
    rho, flux = rng.uniform(0.5, 2.0, (nl, L)), rng.uniform(-1.0, 1.0, (nl, L))
    base = 10.0 ** rng.uniform(-8, 0, n.shape)
    dx, dtdx = 0.37, 0.3
    P = A.element_projector(netw.counts)
    net = kt.Network(netw)

    def dev(a):                                    # an odd base address when asked for
        t = torch.empty(a.size + 1, dtype=torch.float64, device="cuda")[odd:odd + a.size].view(a.shape)
        t.copy_(torch.from_numpy(a))
        return t
    scale = np.abs(n) + dtdx * np.abs(n / rho[None]).max() * 2
    for project in (True, False):
        ref = A.advect_step(n, rho, flux, dtdx, dx, P if project else None)
        got = kt.advect_sweep(net, dev(n), dev(rho), dev(flux), dx, dtdx, project=project).cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-12 * scale)
        got = kt.advect_sweep(net, dev(n), dev(rho), dev(flux), dx, dtdx, alpha=0.5, n_base=dev(base),
                              project=project).cpu().numpy()
        assert np.all(np.abs(got - (0.5 * base + 0.5 * ref)) <= 1e-12 * (scale + base))


def test_non_finite_cells_stay_local(kt):
    """NaN and infinity reach the cells whose stencil holds them and no others."""
    import torch
    netw = _network(4, 2, 1)
    net = kt.Network(netw)
    rng = np.random.default_rng(2)
    n = rng.uniform(0.1, 1.0, (4, 2, 100))
    rho, flux = np.ones((2, 100)), rng.uniform(-1.0, 1.0, (2, 100))
    for bad in (np.nan, np.inf):
        m = n.copy()
        m[1, 0, 40] = bad
        got = kt.advect_sweep(net, *(torch.from_numpy(a).cuda() for a in (m, rho, flux)), 0.37, 0.3,
                              project=False).cpu().numpy()
        with np.errstate(all="ignore"):
            ref = A.advect_step(m, rho, flux, 0.3, 0.37, None)
        assert np.array_equal(np.isfinite(got), np.isfinite(ref))
        ok = np.isfinite(ref)
        assert np.allclose(got[ok], ref[ok], rtol=1e-12, atol=1e-12)
