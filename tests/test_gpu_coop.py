"""Several lanes per cell against one cell per lane (csrc/kt_coop.cuh, csrc/kt_lane.cuh).

kt_integrate_noalloc runs the lane-per-cell kernels, kt_integrate_ptrs the ones that split
a cell over a group of lanes; every output of a call must be the same bit for bit.  Sizes
cross the dispatch's lines (32, 16 and 8 lanes per cell on 152 SMs), leave groups and warps
partly empty and include one cell; networks of every size class, heat capacities
polynomial in T, three reactants and three products; both launch modes; in-place calls,
failing, reverted and non-finite cells.
"""
import numpy as np
import pytest

from paper_2504_04941_gb300 import inputs as I

pytestmark = pytest.mark.gpu

KEYS = ("y", "T", "status", "nsub", "nnewton")


@pytest.fixture(scope="module")
def kt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_04941_gb300 import build, kt as ktm
    build.build()
    return ktm


def _both(kt, netw, cells, dt, opts, in_place=False):
    import torch
    net = kt.Network(netw)
    n = cells.ncells
    res = []
    for call in (kt.integrate, kt.integrate_noalloc):
        y, T = torch.from_numpy(cells.y).cuda(), torch.from_numpy(cells.T).cuda()
        out = dict(y=y if in_place else torch.empty_like(y), T=T if in_place else torch.empty_like(T))
        for k in ("status", "nsub", "nnewton"):
            out[k] = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        r = call(net, y, T, dt, opts, out=out)
        torch.cuda.synchronize()
        res.append({k: r[k].cpu().numpy() for k in KEYS})
    return res


def _same(a, b):
    for k in KEYS:
        assert np.array_equal(a[k], b[k], equal_nan=k in ("y", "T")), k


FORMS = [dict(form=1, scheme=1), dict(form=0, scheme=1), dict(form=0, scheme=0), dict(form=0, scheme=0, guess=2)]


@pytest.mark.parametrize("n", [1, 3, 33, 609, 1300, 6081, 33000])
@pytest.mark.parametrize("form", FORMS[:3], ids=["fp32lu-tr", "fp64-tr", "fp64-be"])
def test_combustion_sizes(kt, n, form):
    wl = I.workload(2, n)
    _same(*_both(kt, wl.network, wl.cells, 3e-12 if n > 1000 else 1e-10, kt.options(wl.tol, persistent=1, **form)))


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("form", FORMS, ids=["fp32lu-tr", "fp64-tr", "fp64-be", "fp64-be-fullstep"])
def test_networks_and_launch_modes(kt, form, persistent):
    strom = I.stromgren_network(1e-3)
    rng = np.random.default_rng(3)
    n = 75
    x = rng.uniform(0.1, 0.9, n)
    scells = I.Cells(np.ascontiguousarray(np.stack([1 - x, x, x]) * 10.0), rng.uniform(5e3, 2e4, n), np.ones(n))
    small = I.combustion_network(seed=5, n_species=7, n_elements=2, n_reversible=6, name="comb7")
    iso = I.ism_network(seed=11, n_species=14, n_reactions=40)
    t1, t2, t3 = I.tolerances(1), I.tolerances(2), I.tolerances(3)
    cases = [(I.network(1), I.robertson_cells(n, 4), 10.0, t1), (strom, scells, 1e3, t1),
             (I.decay_chain_network(1.0, 30.0), I.robertson_cells(n, 5), 1.0, t1),
             (I.network(6), I.combustion_cells(I.network(6), n, 9), 1e-10, t2),
             (small, I.combustion_cells(small, n, 8), 1e-9, t2), (iso, I.ism_cells(iso, n, 7), 1e6, t3)]
    for netw, cells, dt, tol in cases:
        if form["scheme"] == 0:
            dt *= 1e-2
        a, b = _both(kt, netw, cells, dt, kt.options(tol, persistent=persistent, **form))
        _same(a, b)
        assert np.all(a["status"] <= 1)


@pytest.mark.parametrize("wid,dt", [(1, 10.0), (2, 1e-10)])
@pytest.mark.parametrize("form", FORMS[:3], ids=["fp32lu-tr", "fp64-tr", "fp64-be"])
def test_failing_and_non_finite_cells_in_place(kt, wid, dt, form):
    wl = I.workload(wid, 70)
    c = wl.cells
    c.y[0, 1] = np.nan
    c.T[2] = np.inf
    c.y[2, 3] = -1e-3 * abs(c.y[2, 3]) - 1e-12
    c.y[:, 5] = 0.0
    for kw in (dict(), dict(max_substeps=6), dict(max_substeps=6, retry=0), dict(max_newton=1), dict(max_newton=2)):
        o = kt.options(wl.tol, persistent=1, **form)
        for k, v in kw.items():
            setattr(o, k, v)
        a, b = _both(kt, wl.network, c, dt, o, in_place=True)
        _same(a, b)
        assert list(a["status"][1:3]) == [3, 3]
        if "max_substeps" in kw:
            assert np.any(a["status"] == 2)     # the reverting path ran
