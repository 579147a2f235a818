"""Group kernels against one cell per lane, bit for bit, over intervals that reach equilibrium, where
the rates cancel and the last bit of a product decides: networks of any size with and without
temperature whose reactions are all A + B -> C + D (csrc/kt_lane.cuh reaction_pass)."""
import dataclasses

import pytest

from paper_2504_04941_gb300 import inputs as I
from test_gpu_coop import _both, _same, kt  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("energy", [0, 1])
@pytest.mark.parametrize("ns,nrev,dt", [(6, 4, 1e-9), (7, 6, 1e-9), (7, 10, 1e-9), (9, 20, 1e-10), (12, 6, 1e-9)])
def test_last_bits_at_equilibrium(kt, ns, nrev, dt, energy):  # noqa: F811
    netw = dataclasses.replace(I.combustion_network(seed=5, n_species=ns, n_elements=2, n_reversible=nrev, name="c"),
                               energy=energy)
    cells = I.combustion_cells(netw, 500, 7)
    for scheme in (1, 0):
        a, b = _both(kt, netw, cells, dt if scheme else 1e-2 * dt, kt.options(I.tolerances(2), persistent=1, form=0, scheme=scheme))
        _same(a, b)
