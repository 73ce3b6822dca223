"""Contexts of different models in one process, evaluated in turn."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells,force_mode", [(5, 0), (15, 0), (5, 1)])
def test_models_with_tables_of_different_sizes_take_turns(n_cells, force_mode):
    """Six species, one, six, eight (tables in global memory), two with 128 knots, one: each evaluates again after a smaller and after a larger one has.
    The kernels' shared-memory limit belongs to the process."""
    import paper_2608_16329_b200 as mlip
    pots = []
    for n_species, knots in ((6, 0), (1, 0), (8, 0), (2, 128)):
        a = 3.9
        box = np.full(3, a * n_cells)
        rng = np.random.default_rng(n_species)
        pos = wl.lattice_sites((n_cells,) * 3, a, wl._FCC_BASIS) + rng.uniform(0.0, 0.05, (4 * n_cells ** 3, 3))
        pos -= np.floor(pos / box) * box
        enc, head = wl.make_weights(n_species, 78, 0.05, 0.3)
        pot = mlip.Potential(n_species, 6.0, 0.5, enc, head, np.full(n_species, 50.0), table_knots=knots, force_mode=force_mode)
        pot.build_neighbors(pos, rng.integers(0, n_species, len(pos)).astype(np.int32), box)
        pots.append(pot)
    first = {}
    for q in (0, 1, 0, 2, 3, 1, 0, 3, 2, 1):
        e = float(pots[q].compute()["energy"].cpu())
        pots[q].sync_status()
        assert abs(e - first.setdefault(q, e)) <= 1e-9 * abs(e)   # (sums of the same terms in another order, in double)
