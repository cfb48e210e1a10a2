"""The binning of the build: the hits a candidate finds do not depend on the
grid they are binned in, so that builds with grids of every kind (one bin, bins
that no block slice divides evenly, the largest) are equal bit for bit, for
segments with fewer hits than a cluster has blocks, for empty ones, and for
more hits than the blocks keep azimuths of (65,536 in a segment); one, two and
three events of 14 layers take the three forms of the binning."""
import numpy as np
import pytest

from paper_1705_02876_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("events", [1, 2, 3])
@pytest.mark.parametrize("seeds,noise", [(3, 0), (40, 3), (700, 100)])
def test_grids_agree(oracle, events, seeds, noise):
    from paper_1705_02876_gb300 import build, kf
    build.build()
    ctx = kf.Context(0)
    ev = synth.make_build_events(71, events, seeds, noise_factor=noise)
    f = oracle.fit_seeds(ev)
    t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype=dt)
    args = (ev.hit_offsets, t(ev.hit_pos, torch.float32), t(ev.hit_cov, torch.float32), t(ev.seed_event, torch.int32),
            t(f["state"], torch.float32), t(f["cov"], torch.float32), t(ev.seed_fit.charge, torch.int8))
    off = ev.hit_offsets.copy()
    if seeds == 3:  # every layer of the last event but the first empty
        off[-1, 1:] = off[-1, 1]
    want = None
    for grid in ((256, 64), (1, 1), (3, 5), (7, 2), (1021, 3), (16384, 1), (1, 16384)):
        got = kf.build_tracks(ctx, kf.GeometryArgs.of(ev.build_geom), off, *args[1:],
                              opt=kf.options(n_phi_bins=grid[0], n_z_bins=grid[1]))
        got = {k: v.cpu().numpy() for k, v in got.items()}
        if want is None:
            want = got
            assert events == 1 and seeds == 3 or (got["nhits"][:, 0] > 0).any()
        for k in want:
            assert np.array_equal(got[k], want[k], equal_nan=True), (grid, k)
    ctx.close()
