"""List builds in the forms that list_form picks, on both sides of its lines: the traversal that a later build takes is the single one, told by its
launches, and its lists are the oracle's."""
import numpy as np
import pytest

import oracle
import workloads as wl
from helpers import canonical_equal

pytestmark = pytest.mark.gpu


def build_twice(positions, n, box, list_format=0, C=3, seed=0):
    """Oracle's lists and context after two builds, the second of another configuration, in which the single traversal did not fall back to
    counting and filling: that takes a scan and a kernel more."""
    import paper_2608_16329_b200 as mlip
    rng = np.random.default_rng(n + seed)
    box = np.array(box)
    enc, head = wl.make_weights(C, seed=1, enc_hidden=8, enc_layers=1)
    pot = mlip.Potential(C, 6.0, 1.0, enc, head, np.ones(C), table_tol=1.0, enc_hidden=8, enc_layers=1, list_format=list_format)
    launches = [mlip.mlip_get_counters(pot.ctx)["launches"]]
    for trial in range(2):
        pos = positions(rng)
        pos -= np.floor(pos / box) * box
        pos[pos >= box] = 0.0
        pos = np.ascontiguousarray(pos)
        species = rng.integers(0, C, n).astype(np.int32)
        pot.build_neighbors(pos, species, box)
        launches.append(mlip.mlip_get_counters(pot.ctx)["launches"])
    assert launches[2] - launches[1] < launches[1] - launches[0]
    return oracle.neighbors(pos, species, C, box, 7.0), pot


@pytest.mark.parametrize("box,n", [((14.2, 60.0, 300.0), 18441), ((300.0, 14.2, 60.0), 18441), ((14.2, 60.3, 830.0), 50041)])
def test_grids_of_two_cells_across(box, n):
    nl, pot = build_twice(lambda rng: rng.uniform(0, 1, (n, 3)) * np.array(box), n, box)
    assert canonical_equal(nl, *pot.neighbors())
