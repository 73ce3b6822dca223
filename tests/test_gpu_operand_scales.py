"""The fused kernel's contractions take fp16 hi + lo operand pairs whose exponent range is met by powers of two chosen per model
(radial tables, weights) and per atom (activations, W_i): models whose parts are far from order one must lose no accuracy."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("enc_scale,spread,head_scale", [(1.0, 0, 1.0), (1e-6, 0, 1.0), (1e4, 0, 1e-6), (1.0, 3, 1e6), (1e-3, 5, 1.0), (1e5, 2, 1e4)])
def test_models_of_any_magnitude_match_the_oracle(enc_scale, spread, head_scale):
    """Channel c of every encoder is multiplied by f_c = enc_scale x 10^(+-spread) and the regression's first layer divided by f_c
    (l = 0) or f_c^2, so the function -- and with it its conditioning, the head's saturation included -- is that of the order-one
    model; the invariants' magnitudes spread over up to twenty decades.  head_scale multiplies E.  The bounds are those of the order-one
    model (forces 1e-4 at 1 eV/Angstrom RMS, E_i 2e-5 of its size), relative to the outputs' own size."""
    import paper_2608_16329_b200 as mlip
    w = wl.make_workload(5, n_cells=4)
    enc, head = wl.make_weights(6, 77, wl.ENC_OUT_SCALE[5], wl.HEAD_OUT_SCALE[5] * head_scale, e_ref=0.0)
    f = enc_scale * 10.0 ** np.random.default_rng(5).uniform(-spread, spread, 32)
    nets = enc.reshape(36, -1)
    nets[:, -32 * 128 - 32:-32] *= np.repeat(f, 128)
    nets[:, -32:] *= f
    first = head.reshape(6, -1)[:, :64 * 128].reshape(6, 64, 4, 32)
    first /= np.stack([f, f * f, f * f, f * f])
    pot = mlip.Potential(6, w.r_cut, 1.0, enc, head, w.masses)
    pot.build_neighbors(w.pos, w.species, w.box)
    out = pot.compute(want_e_atom=True)
    pot.sync_status()
    ref = oracle.evaluate(oracle.Model(6, w.r_cut, enc, head), w.pos, w.species, w.box)
    df = np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() / np.sqrt((ref["forces"] ** 2).mean())
    de = np.abs(out["e_atom"].cpu().numpy() - ref["e_atom"]).max() / np.abs(ref["e_atom"]).max()
    print(f"spread {spread}, encoder x {enc_scale:g}, head x {head_scale:g}: max|dF| / rms {df:.1e}, max|dE_i| / max {de:.1e}")
    assert df <= 1e-4 and de <= 2e-5


@pytest.mark.parametrize("first,hidden,shift", [(1.0, 10.0, 0.0), (0.03, 30.0, -14.0), (0.01, 100.0, -8.0), (0.003, 300.0, -14.0), (0.001, 1000.0, -10.0)])
def test_hidden_layers_far_from_their_norms_match_the_oracle(first, hidden, shift):
    """First layer x `first`, hidden weights x `hidden`, hidden biases + `shift`: activations and the reverse pass's operands lie up to 2^30
    below what the weights' row and column sums allow them to be (operands scaled to those sums lost 4 to 8 decades of the forces).
    Bounds as above."""
    import paper_2608_16329_b200 as mlip
    w = wl.make_workload(5, n_cells=4)
    enc, head = wl.make_weights(6, 70, wl.ENC_OUT_SCALE[5], wl.HEAD_OUT_SCALE[5], e_ref=0.0)
    nets = head.reshape(6, -1)
    nets[:, :64 * 128 + 64] *= first
    for layer in range(3):
        at = 64 * 129 + layer * 64 * 65
        nets[:, at:at + 64 * 64] *= hidden
        nets[:, at + 64 * 64:at + 64 * 65] += shift
    pot = mlip.Potential(6, w.r_cut, 1.0, enc, head, w.masses)
    pot.build_neighbors(w.pos, w.species, w.box)
    out = pot.compute(want_e_atom=True)
    pot.sync_status()
    ref = oracle.evaluate(oracle.Model(6, w.r_cut, enc, head), w.pos, w.species, w.box)
    df = np.abs(out["forces"].cpu().numpy() - ref["forces"]).max() / np.sqrt((ref["forces"] ** 2).mean())
    de = np.abs(out["e_atom"].cpu().numpy() - ref["e_atom"]).max() / np.abs(ref["e_atom"]).max()
    print(f"first x {first:g}, hidden x {hidden:g}, biases {shift:+g}: max|dF| / rms {df:.1e}, max|dE_i| / max {de:.1e}")
    assert df <= 1e-4 and de <= 2e-5
