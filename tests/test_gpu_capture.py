"""Calls captured into a CUDA graph and replayed, alone and in turn with ordinary calls, and calls that fail inside a capture."""
import numpy as np
import pytest
import torch

from helpers import make_pair

pytestmark = pytest.mark.gpu


def _same(got, want, exact, real):
    """exact: the integer sums of the deterministic mode; else sums in another order, 1e-6 of the forces' size in single precision
    (rounding of some 80 terms of order one) and 1e-12 in double."""
    tol = 0.0 if exact else 1e-12 if real == torch.float64 else 1e-6
    for key in ("energy", "virial", "forces"):
        a, b = got[key].double(), want[key].double()
        assert (a - b).abs().max() <= tol * max(1.0, float(b.abs().max())), key


@pytest.mark.parametrize("options", [dict(), dict(force_mode=1), dict(precision=1), dict(list_format=1)])
@pytest.mark.parametrize("cfg,n_cells", [(5, 6), (3, 15)])
def test_a_captured_evaluation_replays(cfg, n_cells, options):
    """864 and 13,500 atoms (tiles of 8 and 16): new positions through the captured arrays; ordinary evaluations of other positions before,
    between and after; then other species in the same lists' place."""
    w, _, pot = make_pair(cfg, n_cells, 1.0, **options)
    _, _, plain = make_pair(cfg, n_cells, 1.0, **options)
    rng = np.random.default_rng(3)
    exact, real = options.get("force_mode") == 1, torch.float64 if options.get("precision") == 1 else torch.float32
    for p in (pot, plain):
        p.build_neighbors(w.pos, w.species, w.box)

    def positions():
        x = w.pos + rng.uniform(-0.05, 0.05, w.pos.shape)
        return torch.as_tensor(np.where(x - np.floor(x / w.box) * w.box >= w.box, 0.0, x - np.floor(x / w.box) * w.box), device="cuda")

    def expected(x):
        plain.set_positions(x)
        return plain.compute()

    x = positions()
    pot.set_positions(x)
    _same(pot.compute(), expected(x), exact, real)
    static = positions()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        pot.set_positions(static)
        out = pot.compute()
    for turn in range(6):
        if turn in (2, 3, 5):
            x = positions()
            pot.set_positions(x)
            _same(pot.compute(), expected(x), exact, real)
            if turn == 3:
                pot.set_positions(x)   # leaves the forces to the next evaluation, whichever that is
        if turn == 4:
            species = rng.permutation(np.where(w.species == 0, 1, w.species)).astype(np.int32)
            for p in (pot, plain):
                p.build_neighbors(w.pos, species, w.box)
        static.copy_(positions())
        want = expected(static)
        graph.replay()
        torch.cuda.synchronize()
        _same(out, want, exact, real)
        assert pot.energies()[0].item() == out["energy"].item()
    assert pot.sync_status() == 0 and plain.sync_status() == 0


@pytest.mark.parametrize("ensemble", ["nve", "nvt"])
def test_captured_steps_replay(ensemble):
    states = []
    for replayed in (False, True):
        w, _, pot = make_pair(5, 6, 1.0, force_mode=1)
        pot.build_neighbors(w.pos, w.species, w.box)
        pot.set_velocities(w.vel)

        def run():
            pot.step(2, 1.0, 0) if ensemble == "nve" else pot.step_nvt(2, 1.0, 0, 300.0, 50.0)
        run()
        if replayed:
            graph = torch.cuda.CUDAGraph()
            torch.cuda.synchronize()
            with torch.cuda.graph(graph):
                run()
        for _ in range(3):
            graph.replay() if replayed else run()
        run()
        torch.cuda.synchronize()
        assert pot.sync_status() == 0
        states.append(b"".join(t.cpu().numpy().tobytes() for t in (*pot.state()[:2], pot.energies())))
    assert states[0] == states[1]


def test_a_call_that_fails_leaves_the_next_ones_alone():
    """A list build waits for the device, which a capture does not allow: the call is refused, and neither its error nor what it had
    noted for the next evaluation stays behind."""
    import paper_2608_16329_b200 as mlip
    from cuda.bindings import runtime
    w, _, pot = make_pair(5, 6, 1.0)
    _, _, other = make_pair(2, 6, 1.0)
    pot.build_neighbors(w.pos, w.species, w.box)
    want = pot.compute()
    pos, species = torch.as_tensor(w.pos, device="cuda"), torch.as_tensor(w.species, device="cuda")
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    assert runtime.cudaStreamBeginCapture(stream.cuda_stream, runtime.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)[0] == 0
    with pytest.raises(mlip.MlipError):
        mlip.mlip_build_neighbors(pot.ctx, pos, species, w.box, stream.cuda_stream)
    runtime.cudaStreamEndCapture(stream.cuda_stream)
    runtime.cudaGetLastError()
    wo, _, _ = make_pair(2, 6, 1.0)
    other.build_neighbors(wo.pos, wo.species, wo.box)
    other.compute()
    pot.build_neighbors(w.pos, w.species, w.box)
    _same(pot.compute(), want, False, torch.float32)
    assert pot.sync_status() == 0 and other.sync_status() == 0
