"""List build and canonical export at the edges of their kernels: grids with fewer than three cells in a dimension, cells of more than
one and of several dozen atoms, tile remainders, lists longer than the buffers -- first build (count and fill) and later ones
(single traversal) alike, both export entry points, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as wl
from helpers import canonical_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,n,list_format", [((14.1, 14.1, 14.1), 1, 0), ((14.1, 14.1, 14.1), 2, 0), ((14.1, 14.1, 14.1), 33, 0),
                                               ((14.2, 22.0, 30.0), 700, 0),         # 2 x 3 x 4 cells
                                               ((21.5, 21.5, 21.5), 257, 1), ((21.5, 22.0, 29.0), 1023, 0),
                                               ((21.5, 21.5, 21.5), 2300, 0),        # lists of about 330 entries, 85 atoms to a cell
                                               ((14.2, 21.5, 21.5), 1600, 0), ((21.5, 21.5, 21.5), 1800, 1)])
def test_builds_and_exports_equal_the_oracles_lists(box, n, list_format):
    import paper_2608_16329_b200 as mlip
    import torch
    rng = np.random.default_rng(n)
    box = np.array(box)
    C = 8
    enc, head = wl.make_weights(C, seed=1, enc_hidden=8, enc_layers=1)
    pot = mlip.Potential(C, 6.0, 1.0, enc, head, np.ones(C), table_tol=1.0, enc_hidden=8, enc_layers=1, list_format=list_format)
    for trial in range(3):   # other configurations in the same context
        pos = rng.uniform(0, 1, (n, 3)) * box
        species = rng.integers(0, C, n).astype(np.int32)
        pot.build_neighbors(pos, species, box)
        nl = oracle.neighbors(pos, species, C, box, 7.0, method="brute")
        assert canonical_equal(nl, *pot.neighbors())
        seg = torch.empty(n * C + 1, dtype=torch.int64, device=pot.device)
        nbr = torch.empty(max(nl.nbr.size, 1), dtype=torch.int32, device=pot.device)
        rc, total = mlip.mlip_get_neighbors_noalloc(pot.ctx, seg, nbr)
        assert rc == 0 and total == nl.nbr.size and canonical_equal(nl, seg, nbr[:total])
