"""Larger-network kernels (csrc/kt_warp.cuh) at their edges against the FP64 oracle: one
warp's last size and the team's first (32 and 33 unknowns), the sizes where a lane's rows
step up (64, 65), the oracle's largest (80) and
the largest (96, FP32-LU against FP64), and a network whose partials do not fit in shared
memory.  The comparison is the repository's parity rule (_parity.compare)."""
import os

import numpy as np
import pytest

from paper_2504_04941_gb300 import inputs as I
from _parity import atol_cells, compare, tight_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_04941_gb300 import build, kt as ktm
    build.build()
    return ktm


def _check(kt, oracle_mod, netw, cells, dt, tol, form, scheme):
    import torch
    net = kt.Network(netw)
    y, T = torch.from_numpy(cells.y).cuda(), torch.from_numpy(cells.T).cuda()
    r = kt.integrate(net, y, T, dt, kt.options(tol, form=form, scheme=scheme, persistent=1, cells_per_warp=1))
    kt.check_scratch(r["scratch"])
    g = {k: r[k].cpu().numpy() for k in ("y", "T", "status", "nsub", "nnewton")}
    nt = os.cpu_count() or 1
    o = oracle_mod.OracleNetwork(netw).integrate(cells, dt, oracle_mod.options(tol, scheme=scheme), nt)
    rep = compare(g, o, netw.energy, rtol=tol.rtol, tight=tight_oracle(oracle_mod, netw, cells, dt, tol, nt, scheme=scheme),
                  atol_cells=atol_cells(netw, cells, tol))
    assert rep.ok(), rep
    assert np.all(g["status"] == 0)


def _exchange_network(ns, seed):
    """ns isomers exchanging in random A + B <-> C + D pairs, with temperature."""
    rng = np.random.default_rng(seed)
    h = rng.uniform(-2e5, 2e5, ns)
    pairs = [((i, (i + 1) % ns), tuple(int(v) for v in rng.choice(ns, 2, replace=False))) for i in range(ns)]
    rx = I._reversible_pairs_to_entries(pairs, 10.0 ** rng.uniform(8, 13, ns), rng.uniform(-1, 1, ns),
                                        rng.uniform(0, 2e4, ns), h)
    return I._irreversible(f"x{ns}", [f"S{i}" for i in range(ns)], ["X"], np.full(ns, 20.0), h, np.full(ns, 25.0),
                           [[1]] * ns, 1, 1.0, 10.0, 1e5, rx)


@pytest.mark.parametrize("form,scheme", [(1, 1), (0, 1), (1, 0), (0, 0)])
@pytest.mark.parametrize("n_species", [1, 31, 32, 63, 64, 79])
def test_sizes(kt, oracle_mod, n_species, form, scheme):
    n = 9
    if n_species == 1:      # one species, no temperature: a photo-like decay into nothing it carries
        netw = I._irreversible("one", ["A"], ["X"], [1.0], [0.0], [0.0], [[0]], 0, 1.0, 1.0, 1e5,
                               [((0,), (), 3.0, 0.0, 0.0, -1)])
        cells, tol, dt = I.Cells(np.linspace(0.5, 1.0, n)[None].copy(), np.full(n, 300.0), np.ones(n)), I.tolerances(1), 0.3
    else:
        netw = I.combustion_network(seed=40 + n_species, n_species=n_species, n_elements=4,
                                    n_reversible=2 * n_species, name=f"c{n_species}") if n_species < 65 else \
            _exchange_network(n_species, 5)
        cells, tol, dt = I.combustion_cells(netw, n, seed=3), I.tolerances(5), 1e-11 if scheme else 1e-12
    _check(kt, oracle_mod, netw, cells, dt, tol, form, scheme)


def test_largest_size_agrees_across_forms(kt):
    import torch
    netw, tol = _exchange_network(95, 5), I.tolerances(5)
    cells, net, res = I.combustion_cells(netw, 9, seed=3), kt.Network(netw), []
    for form in (0, 1):
        r = kt.integrate(net, torch.from_numpy(cells.y).cuda(), torch.from_numpy(cells.T).cuda(), 1e-11,
                         kt.options(tol, form=form, scheme=1, persistent=1))
        kt.check_scratch(r["scratch"])
        res.append({k: r[k].cpu().numpy() for k in ("y", "T", "status", "nsub", "nnewton")})
    assert np.all(res[0]["status"] == 0) and compare(res[1], res[0], 1, rtol=tol.rtol).ok()


@pytest.mark.parametrize("form,scheme,n_reversible", [(0, 1, 1250), (1, 0, 1450)])
def test_networks_whose_partials_do_not_fit(kt, oracle_mod, form, scheme, n_reversible):
    netw = I.combustion_network(seed=77, n_species=64, n_elements=4, n_reversible=n_reversible, name="big64")
    _check(kt, oracle_mod, netw, I.combustion_cells(netw, 5, seed=4), 1e-12, I.tolerances(5), form, scheme)
