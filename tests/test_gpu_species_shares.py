"""Start of the fused kernel's CTAs on the species in proportion to their tiles: species with no atom, with one atom, with nearly all
of them; fewer tiles than SMs, and systems of two-atom tiles."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,counts", [(4, (0, 1, 0)), (4, (1, 0, 1)), (4, (8, 9, 0)), (5, (250, 0, 1)), (6, (1, 1, 1, 1, 1, 1, 1)),
                                          (7, (100, 0, 200, 0, 300, 0, 1)), (15, (1, 17, 12000)), (15, (0, 6000, 1))])
def test_uneven_species_match_the_oracle(cells, counts):
    """counts: atoms of the first species; the last one takes the rest.  Tolerances: those of the order-one workloads, forces
    relative to their RMS where that exceeds 1 eV/Angstrom."""
    import paper_2608_16329_b200 as mlip
    rng = np.random.default_rng(cells + len(counts))
    a, n_species = 3.9, len(counts) + 1
    box = np.full(3, a * cells)
    pos = wl.lattice_sites((cells, cells, cells), a, wl._FCC_BASIS) + rng.normal(0.0, 0.03, (4 * cells ** 3, 3))
    pos -= np.floor(pos / box) * box
    species = np.full(len(pos), n_species - 1, dtype=np.int32)
    species[rng.permutation(len(pos))[:sum(counts)]] = np.repeat(np.arange(len(counts)), counts)
    enc, head = wl.make_weights(n_species, seed=78, enc_out_scale=0.05, head_out_scale=0.3)
    pot = mlip.Potential(n_species, 6.0, 0.5, enc, head, np.full(n_species, 50.0))
    pot.build_neighbors(pos, species, box)
    out = pot.compute(want_e_atom=True)
    pot.sync_status()
    ref = oracle.evaluate(oracle.Model(n_species, 6.0, enc, head), pos, species, box)
    scale = max(1.0, float(np.sqrt((ref["forces"] ** 2).sum(1).mean())))
    assert abs(float(out["energy"].cpu()) - ref["energy"]) <= 1e-6 * abs(ref["energy"])
    assert np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() <= 1e-4 * scale
    assert np.abs(out["e_atom"].cpu().numpy() - ref["e_atom"]).max() <= 2e-5 * max(1.0, np.abs(ref["e_atom"]).max())


@pytest.mark.parametrize("counts", [(3000, 0, 1, 40000), (8000, 5000), (16, 17)])
def test_rare_species_of_a_large_system_match_the_double_precision_path(counts):
    """157,216 atoms, above 64 tiles of 16 atoms per CTA: the rare species' CTAs are rounded up.  The fp64 kernel deals its tiles out
    in its own way; tolerances as above."""
    import paper_2608_16329_b200 as mlip
    cells, a, n_species = 34, 3.9, len(counts) + 1
    rng = np.random.default_rng(n_species)
    box = np.full(3, a * cells)
    pos = wl.lattice_sites((cells, cells, cells), a, wl._FCC_BASIS) + rng.normal(0.0, 0.03, (4 * cells ** 3, 3))
    pos -= np.floor(pos / box) * box
    species = np.full(len(pos), n_species - 1, dtype=np.int32)
    species[rng.permutation(len(pos))[:sum(counts)]] = np.repeat(np.arange(len(counts)), counts)
    enc, head = wl.make_weights(n_species, seed=78, enc_out_scale=0.05, head_out_scale=0.3)
    got = []
    for precision in (0, 1):
        pot = mlip.Potential(n_species, 6.0, 0.5, enc, head, np.full(n_species, 50.0), precision=precision)
        pot.build_neighbors(pos, species, box)
        out = pot.compute(want_e_atom=True)
        pot.sync_status()
        got.append({key: np.asarray(out[key].cpu().numpy(), dtype=np.float64) for key in ("energy", "forces", "e_atom")})
        pot.close()
    one, ref = got
    scale = max(1.0, float(np.sqrt((ref["forces"] ** 2).sum(1).mean())))
    assert abs(one["energy"].item() - ref["energy"].item()) <= 1e-6 * abs(ref["energy"].item())
    assert np.abs(one["forces"] - ref["forces"]).max() <= 1e-4 * scale
    assert np.abs(one["e_atom"] - ref["e_atom"]).max() <= 2e-5 * max(1.0, np.abs(ref["e_atom"]).max())


@pytest.mark.parametrize("cells,counts", [(6, (200, 200, 0, 200)), (6, (0, 300, 0, 300, 0, 1, 100)), (10, (900, 0, 900, 900, 0, 900)), (15, (3000, 1, 0, 3000, 0))])
def test_species_passed_over_next_to_absent_ones(cells, counts):
    """A CTA's way through the species: one whose tiles are all claimed, then one without atoms, then another, in every rotation of that order.
    The decision to pass a species over must reach all warps of a CTA.  Tolerances as above, on each of eight evaluations."""
    import paper_2608_16329_b200 as mlip
    rng = np.random.default_rng(cells + len(counts))
    a, n_species = 3.9, len(counts) + 1
    box = np.full(3, a * cells)
    pos = wl.lattice_sites((cells, cells, cells), a, wl._FCC_BASIS) + rng.normal(0.0, 0.03, (4 * cells ** 3, 3))
    pos -= np.floor(pos / box) * box
    species = np.full(len(pos), n_species - 1, dtype=np.int32)
    species[rng.permutation(len(pos))[:sum(counts)]] = np.repeat(np.arange(len(counts)), counts)
    enc, head = wl.make_weights(n_species, seed=78, enc_out_scale=0.05, head_out_scale=0.3)
    pot = mlip.Potential(n_species, 6.0, 0.5, enc, head, np.full(n_species, 50.0))
    pot.build_neighbors(pos, species, box)
    ref = oracle.evaluate(oracle.Model(n_species, 6.0, enc, head), pos, species, box)
    scale = max(1.0, float(np.sqrt((ref["forces"] ** 2).sum(1).mean())))
    for _ in range(8):
        out = pot.compute()
        pot.sync_status()
        assert abs(float(out["energy"].cpu()) - ref["energy"]) <= 1e-6 * abs(ref["energy"])
        assert np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() <= 1e-4 * scale
