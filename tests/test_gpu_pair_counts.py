"""Fused kernel, atoms of every number of pairs: a lattice whose occupancy rises from none to all and falls again along the box gives each count from an
isolated atom's zero upwards, so that every remainder of the pair loops' steps (32, 16 and 8 pairs), both atoms of a warp sharing a batch, lists
beyond the prefetched three chunks and queues that overflow all occur, in small systems (one atom per warp) and larger ones (two)."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spacing,cells,list_format,force_mode", [(2.0, (40, 24, 24), 0, 0),    # 9,700 atoms: one per warp, up to 113 pairs
                                                                  (2.0, (80, 24, 24), 0, 0),    # 19,500 atoms: two per warp
                                                                  (2.0, (80, 24, 24), 1, 0), (2.0, (80, 24, 24), 0, 1),
                                                                  (1.6, (96, 24, 24), 0, 0)])   # up to 221 pairs: two atoms overflow their queue
def test_every_number_of_pairs_matches_the_oracle(spacing, cells, list_format, force_mode):
    """Tolerances: those of the order-one workloads, forces relative to their RMS where that exceeds 1 eV/Angstrom."""
    import paper_2608_16329_b200 as mlip
    rng = np.random.default_rng(sum(cells) + list_format)
    pos = wl.lattice_sites(cells, spacing, wl._SC_BASIS) + rng.normal(0.0, 0.03, (int(np.prod(cells)), 3))
    box = np.array(cells) * spacing
    pos -= np.floor(pos / box) * box
    pos[pos >= box] = 0.0
    occupied = rng.uniform(0.0, 1.0, len(pos)) < np.sin(np.pi * pos[:, 0] / box[0]) ** 3
    pos = np.ascontiguousarray(pos[occupied])
    species = rng.integers(0, 3, len(pos)).astype(np.int32)
    enc, head = wl.make_weights(3, seed=78, enc_out_scale=0.05, head_out_scale=0.3)
    pot = mlip.Potential(3, 6.0, 1.0, enc, head, np.array([50.0, 60.0, 70.0]), list_format=list_format, force_mode=force_mode)
    pot.build_neighbors(pos, species, box)
    out = pot.compute(want_e_atom=True)
    pot.sync_status()
    ref = oracle.evaluate(oracle.Model(3, 6.0, enc, head), pos, species, box)
    scale = max(1.0, float(np.sqrt((ref["forces"] ** 2).sum(1).mean())))
    assert abs(float(out["energy"].cpu()) - ref["energy"]) <= 1e-6 * abs(ref["energy"])
    assert np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() <= 1e-4 * scale
    assert np.abs(out["e_atom"].cpu().numpy() - ref["e_atom"]).max() <= 2e-5 * max(1.0, np.abs(ref["e_atom"]).max())
    assert np.abs(out["virial"].cpu().numpy().ravel() - np.asarray(ref["virial"]).ravel()).max() <= 1e-5 * np.abs(ref["virial"]).max()
