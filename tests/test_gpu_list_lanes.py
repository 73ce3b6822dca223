"""List builds of tens of thousands of atoms, most of them with one central atom per lane: grids of three cells, columns that end inside a tile,
nearly empty cells, rows that are too short for their list, several tiles' remainders, both list formats, ghosts -- bit for bit against
the oracle's lists."""
import numpy as np
import pytest

import oracle
import workloads as wl
from helpers import canonical_equal

pytestmark = pytest.mark.gpu


def positions(rng, n, box, clustered):
    pos = rng.uniform(0, 1, (n, 3)) * box
    if clustered:   # a third of the atoms in a dense ball across the periodic boundary, the rest far apart
        m = n // 3
        ball = rng.normal(0.0, 7.0, (m, 3))
        pos[:m] = ball - np.floor(ball / box) * box
        pos[pos >= box] = 0.0
    return pos


@pytest.mark.parametrize("box,n,list_format,clustered", [((21.5, 21.5, 60.3), 18001, 0, False),       # 3 x 3 x 8 cells, some 130 atoms to a cell
                                                         ((66.1, 58.7, 50.2), 18000 + 31, 0, False), ((66.1, 58.7, 50.2), 18000 + 33, 1, False),
                                                         ((400.0, 300.0, 21.5), 18063, 0, False),     # a few atoms to a cell, columns of three cells: one atom to a warp,
                                                                                                      # as the clusters below; see test_gpu_list_forms for such with lanes
                                                         ((160.0, 160.0, 160.0), 18240, 1, True)])
def test_builds_equal_the_oracles_lists(box, n, list_format, clustered):
    import paper_2608_16329_b200 as mlip
    rng = np.random.default_rng(n)
    box = np.array(box)
    C = 3
    enc, head = wl.make_weights(C, seed=1, enc_hidden=8, enc_layers=1)
    pot = mlip.Potential(C, 6.0, 1.0, enc, head, np.ones(C), table_tol=1.0, enc_hidden=8, enc_layers=1, list_format=list_format)
    launches = [mlip.mlip_get_counters(pot.ctx)["launches"]]
    for trial in range(2):   # the first build has no array yet, the second takes the single traversal: no scan and no filling kernel behind it
        pos = positions(rng, n, box, clustered)
        species = rng.integers(0, C, n).astype(np.int32)
        pot.build_neighbors(pos, species, box)
        launches.append(mlip.mlip_get_counters(pot.ctx)["launches"])
    assert launches[2] - launches[1] < launches[1] - launches[0]
    nl = oracle.neighbors(pos, species, C, box, 7.0)
    assert canonical_equal(nl, *pot.neighbors())
    # a domain with ghosts: the last third has no lists of its own, and the others' stay what they are
    owned = 2 * n // 3
    before = mlip.mlip_get_counters(pot.ctx)["launches"]
    pot.build_neighbors(pos, species, box, n_owned=owned)
    assert mlip.mlip_get_counters(pot.ctx)["launches"] - before == launches[2] - launches[1]
    seg, nbr = pot.neighbors()
    seg, nbr = np.asarray(seg.cpu()), np.asarray(nbr.cpu())
    assert (seg[owned * C:] == seg[-1]).all()
    assert np.array_equal(seg[:owned * C + 1], nl.seg_ptr[:owned * C + 1]) and np.array_equal(nbr[:seg[-1]], nl.nbr[:seg[-1]])
