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


# three cells across and more, two to four atoms to a cell: one atom to a warp, eight, and one to a lane
@pytest.mark.parametrize("box,n", [((400.0, 300.0, 21.5), 18063), ((300.0, 300.0, 21.5), 24063), ((170.0, 170.0, 170.0), 30011), ((280.0, 260.0, 240.0), 100003), ((240.0, 220.0, 210.0), 100003)])
@pytest.mark.parametrize("list_format", [0, 1])
def test_few_atoms_to_a_cell(box, n, list_format):
    nl, pot = build_twice(lambda rng: rng.uniform(0, 1, (n, 3)) * np.array(box), n, box, list_format)
    assert canonical_equal(nl, *pot.neighbors())


@pytest.mark.parametrize("n,edge,list_format", [(100003, 290.0, 0), (100003, 290.0, 1), (60011, 125.0, 0), (60011, 125.0, 1)])
def test_dense_clusters_among_few_atoms(n, edge, list_format):
    """A third of the atoms in a ball across the periodic boundary, lists of some hundred entries and more: eight to a warp, one to a lane."""
    def positions(rng):
        pos = rng.uniform(0, 1, (n, 3)) * edge
        pos[:n // 3] = rng.normal(0.0, 14.0, (n // 3, 3))
        return pos
    nl, pot = build_twice(positions, n, (edge, edge, edge), list_format)
    assert canonical_equal(nl, *pot.neighbors())
