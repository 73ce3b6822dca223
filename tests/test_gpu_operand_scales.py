"""The fused kernel's contractions take fp16 hi + lo operand pairs whose exponent range is met by powers of two chosen per model
(weights, radial tables) and per atom (activations, W_i): networks far from order one must lose no accuracy."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("enc_scale,head_scale", [(1e-6, 1.0), (1e-3, 1e4), (0.1, 1e-6), (0.1, 1e6), (30.0, 1.0), (1e3, 1e-3)])
def test_networks_of_any_magnitude_match_the_oracle(enc_scale, head_scale):
    """Moments scale with the encoder's output (their squares reach 1e10 and 1e-12 here), energies with the head's.  The bounds are
    the ones of the order-one networks (forces 1e-4 at 1 eV/Angstrom RMS, E_i 2e-5 of its size) relative to the outputs' own size."""
    import paper_2608_16329_b200 as mlip
    w = wl.make_workload(5, n_cells=4)
    enc, head = wl.make_weights(6, 77, enc_scale, head_scale, e_ref=0.0)
    pot = mlip.Potential(6, w.r_cut, 1.0, enc, head, w.masses)
    pot.build_neighbors(w.pos, w.species, w.box)
    out = pot.compute(want_e_atom=True)
    pot.sync_status()
    ref = oracle.evaluate(oracle.Model(6, w.r_cut, enc, head), w.pos, w.species, w.box)
    df = np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() / np.sqrt((ref["forces"] ** 2).mean())
    de = np.abs(out["e_atom"].cpu().numpy() - ref["e_atom"]).max() / np.abs(ref["e_atom"]).max()
    print(f"encoder x {enc_scale:g}, head x {head_scale:g}: max|dF| / rms {df:.1e}, max|dE_i| / max {de:.1e}")
    assert df <= 1e-4 and de <= 2e-5
