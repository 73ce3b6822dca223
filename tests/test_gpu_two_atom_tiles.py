"""Tiles of 16 central atoms, two per warp: tile remainders, and neighborhoods around the room their shared pair queue has (256
pairs; the first atom keeps at most 160).  Tables too large for shared memory select this form at any system size."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,n_first,list_format", [(3.6, 1, 0), (3.6, 8, 0), (3.6, 9, 1), (3.6, 16, 0), (3.6, 17, 0),
                                                   (3.05, 31, 0), (3.02, 32, 1), (2.84, 33, 0), (2.8, 40, 1), (2.4, 23, 0)])
def test_tile_remainders_and_long_neighborhoods_match_the_oracle(a, n_first, list_format):
    """78 pairs per atom at a = 3.6 Angstrom, about 128 at 3.05 (two atoms fill the queue), 160 at 2.84 (the first atom's share), 265
    at 2.4 (neither fits).  n_first atoms are of the first species.  Tolerances: those of the order-one workloads, forces relative
    to their RMS where that exceeds 1 eV/Angstrom."""
    import paper_2608_16329_b200 as mlip
    rng = np.random.default_rng(n_first)
    n = int(np.ceil(21.5 / a))
    box = np.full(3, a * n)
    pos = wl.lattice_sites((n, n, n), a, wl._FCC_BASIS) + rng.normal(0.0, 0.03, (4 * n ** 3, 3))
    pos -= np.floor(pos / box) * box
    species = np.ones(len(pos), dtype=np.int32)
    species[rng.permutation(len(pos))[:n_first]] = 0
    enc, head = wl.make_weights(2, seed=77, enc_out_scale=0.05, head_out_scale=0.3)
    pot = mlip.Potential(2, 6.0, 0.5, enc, head, np.array([50.0, 60.0]), table_knots=512, list_format=list_format)
    pot.build_neighbors(pos, species, box)
    out = pot.compute(want_e_atom=True)
    pot.sync_status()
    ref = oracle.evaluate(oracle.Model(2, 6.0, enc, head), pos, species, box)
    scale = max(1.0, float(np.sqrt((ref["forces"] ** 2).sum(1).mean())))
    assert abs(float(out["energy"].cpu()) - ref["energy"]) <= 1e-6 * abs(ref["energy"])
    assert np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() <= 1e-4 * scale
    assert np.abs(out["e_atom"].cpu().numpy() - ref["e_atom"]).max() <= 2e-5 * max(1.0, np.abs(ref["e_atom"]).max())
