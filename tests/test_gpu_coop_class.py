"""Group kernels on the networks that share a compiled size's number of unknowns but not its
energy setting: two species with temperature (3 unknowns) and eleven isothermal species, bit
for bit against one cell per lane (csrc/kt_coop.cuh, csrc/kt_lane.cuh)."""
import dataclasses

import numpy as np
import pytest

from paper_2504_04941_gb300 import inputs as I
from test_gpu_coop import FORMS, _both, _same, kt  # noqa: F401

pytestmark = pytest.mark.gpu


def _two_species():
    """A <-> B and A + A <-> A + B with heats, one element."""
    rx = [((0,), (1,), 3.0e5, 0.5, 900.0, -1), ((1,), (0,), 2.0e5, 0.0, 2100.0, -1),
          ((0, 0), (0, 1), 4.0e6, 0.0, 1500.0, -1), ((1, 1), (0, 1), 1.0e6, 0.3, 2500.0, -1)]
    return I._irreversible("ab", ["A", "B"], ["X"], [0.02, 0.02], [0.0, 4.0e4], [30.0, 32.0], [[1], [1]], 1,
                           1.0, 200.0, 6000.0, rx)


@pytest.mark.parametrize("n", [1, 33, 700, 9000])
@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("form", FORMS, ids=["fp32lu-tr", "fp64-tr", "fp64-be", "fp64-be-fullstep"])
def test_other_energy_setting_of_the_compiled_sizes(kt, form, persistent, n):  # noqa: F811
    rng = np.random.default_rng(n)
    two = _two_species()
    iso = dataclasses.replace(I.combustion_network(seed=21, n_species=11, n_reversible=15, name="iso11"), energy=0)
    x = rng.uniform(0.05, 0.95, n)
    c2 = I.Cells(np.ascontiguousarray(np.stack([1 - x, x])), rng.uniform(400.0, 3000.0, n), np.ones(n))
    scale = 1e-2 if form["scheme"] == 0 else 1.0
    for netw, cells, dt, tol in ((two, c2, 1e-6, I.tolerances(2)), (iso, I.combustion_cells(iso, n, 7), 1e-9, I.tolerances(2))):
        assert netw.n in (3, 11)
        a, b = _both(kt, netw, cells, dt * scale, kt.options(tol, persistent=persistent, **form))
        _same(a, b)
        assert np.all(a["status"] <= 1) and a["nsub"].min() >= 1
