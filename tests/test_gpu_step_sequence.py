"""What the fused launch sequence of a step must keep: independence of how a run is cut into calls, the totals of the last evaluation,
the timing records."""
import numpy as np
import pytest

from helpers import make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ensemble", ["nve", "nvt"])
@pytest.mark.parametrize("cfg,n_cells,cuts", [(5, 6, (1, 4, 2)), (2, 16, (3, 3, 1)), (5, 15, (6, 1))])
def test_a_run_does_not_depend_on_how_it_is_cut_into_calls(cfg, n_cells, cuts, ensemble):
    """Bit for bit in the deterministic mode, with a rebuild on the way: the half kick that closes a step runs with the next step's drift
    inside a call and by itself at its end."""
    states = []
    for parts in ((sum(cuts),), cuts):
        w, _, pot = make_pair(cfg, n_cells, 1.0, force_mode=1)
        pot.build_neighbors(w.pos, w.species, w.box)
        pot.set_velocities(w.vel)
        for n in parts:
            pot.step(n, 1.0, 3) if ensemble == "nve" else pot.step_nvt(n, 1.0, 3, 300.0, 50.0)
        pot.sync_status()
        pos, vel, step = pot.state()
        states.append((pos.cpu().numpy().tobytes(), vel.cpu().numpy().tobytes(), pot.energies().cpu().numpy().tobytes(), step))
    assert states[0] == states[1]


def test_the_last_evaluations_totals_stay_until_the_next():
    import paper_2608_16329_b200 as mlip
    w, _, pot = make_pair(5, 6, 1.0)
    pot.build_neighbors(w.pos, w.species, w.box)
    for _ in range(3):
        e = float(pot.compute()["energy"].cpu())
        pairs = mlip.mlip_get_counters(pot.ctx)["pairs_in_cutoff"]
        pot.set_positions(w.pos)
        assert float(pot.energies()[0].cpu()) == e and mlip.mlip_get_counters(pot.ctx)["pairs_in_cutoff"] == pairs > 0


@pytest.mark.parametrize("n_cells", [6, 30])
def test_timing_records_keep_the_last_256_launches(n_cells):
    """Below and above the size where the kernels time themselves instead of events (864 and 108,000 atoms)."""
    import paper_2608_16329_b200 as mlip
    w, _, pot = make_pair(5, n_cells, 1.0)
    pot.build_neighbors(w.pos, w.species, w.box)
    pot.set_velocities(w.vel)
    pot.step(1, 0.01, 0)
    mlip.mlip_get_timings(pot.ctx, reset=True)
    for n, kept in ((20, 20), (300, 256), (900, 256)):
        pot.step(n, 0.001, 0)
        launches, ms = mlip.mlip_kernel_time(pot.ctx)
        build, kernel, integrate = mlip.mlip_get_timings(pot.ctx, reset=True)
        assert launches == kept and kernel == ms and build == 0.0
        assert 0.003 * kept < ms < 10.0 * kept and 0.0005 * kept < integrate < 1.0 * kept
    assert pot.sync_status() == 0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cfg,n_cells", [(5, 6), (5, 15)])
def test_every_evaluation_sees_the_positions_set_just_before_it(cfg, n_cells, precision):
    """Sixty times two configurations in turn without a wait between them: the fused kernel is resident while the positions are still
    being written.  Sums in another order: 1e-6 of the forces' size (1e-12 in double)."""
    import torch
    w, _, pot = make_pair(cfg, n_cells, 1.0, precision=precision)
    pot.build_neighbors(w.pos, w.species, w.box)
    moved = w.pos + np.random.default_rng(1).uniform(-0.1, 0.1, w.pos.shape)
    moved -= np.floor(moved / w.box) * w.box
    both = [torch.as_tensor(np.where(x >= w.box, 0.0, x), device="cuda") for x in (w.pos, moved)]
    want = []
    for x in both:
        pot.set_positions(x)
        torch.cuda.synchronize()
        want.append(pot.compute()["forces"].clone())
        torch.cuda.synchronize()
    got = []
    for turn in range(60):
        pot.set_positions(both[turn % 2])
        got.append(pot.compute()["forces"])
    tol = (1e-6, 1e-12)[precision]
    for turn, f in enumerate(got):
        assert (f - want[turn % 2]).abs().max() <= tol * want[turn % 2].abs().max(), turn
    assert pot.sync_status() == 0


def test_timing_records_outlive_the_streams_they_were_taken_on():
    import paper_2608_16329_b200 as mlip
    import torch
    from cuda.bindings import runtime
    w, _, pot = make_pair(5, 6, 1.0)
    pot.build_neighbors(w.pos, w.species, w.box)
    pot.compute()
    torch.cuda.synchronize()
    mlip.mlip_kernel_time(pot.ctx, reset=True)
    for _ in range(3):
        err, stream = runtime.cudaStreamCreate()
        assert err == 0
        mlip.mlip_compute(pot.ctx, stream=int(stream))
        assert runtime.cudaStreamSynchronize(stream)[0] == 0 and runtime.cudaStreamDestroy(stream)[0] == 0
    launches, ms = mlip.mlip_kernel_time(pot.ctx)
    assert launches == 3 and 0.003 < ms < 30.0
    pot.compute()
    assert pot.sync_status() == 0


def test_a_launch_that_overlaps_no_other_is_timed_from_its_begin():
    """The fused launch behind a list build stages its tables (215 KB per CTA, some 3 us) by itself; in a sequence of evaluations the kernel
    ahead hides that.  864 atoms, mean of 100 launches each."""
    import paper_2608_16329_b200 as mlip
    import torch
    w, _, pot = make_pair(5, 6, 1.0)
    mean = []
    for builds in (False, True):
        pot.build_neighbors(w.pos, w.species, w.box)
        pot.compute()
        torch.cuda.synchronize()
        mlip.mlip_kernel_time(pot.ctx, reset=True)
        for _ in range(100):
            if builds:
                pot.build_neighbors(w.pos, w.species, w.box)
            pot.compute()
        n, ms = mlip.mlip_kernel_time(pot.ctx)
        mean.append(1e3 * ms / n)
    print(f"fused kernel, 864 atoms: {mean[0]:.1f} us in a sequence, {mean[1]:.1f} us behind a build")
    assert mean[1] > mean[0] + 1.5   # (2.9 us here; the staging left out: 0.2)
