"""Tracks put off to the second launch of a fit (those that need extended
precision: pT outside the bounds, ill-conditioned updates, hits that fail the
update) against the same tracks with it in line (KF_LAUNCH_FLAT): the same
arithmetic in another launch, so every output is equal bit for bit.  Sizes on
both sides of the one-launch limit (32,768 tracks), of the gathering blocks (256
tracks) and of what they gather in one pass (2 per SM), with every, some, and no
track put off."""
import numpy as np
import pytest

from paper_1705_02876_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.fixture(scope="module")
def kf():
    from paper_1705_02876_gb300 import build, kf as kf_
    build.build()
    return kf_


@pytest.mark.parametrize("n", [1, 255, 32767, 32768, 33025, 40_001])
def test_put_off_equals_in_line(kf, n):
    ctx = kf.Context(0)
    for lo, hi, share in ((260.0, 500.0, (0.9, 1.0)), (50.0, 500.0, (0.05, 0.95)), (1.0, 5.0, (0.0, 0.01))):
        b = synth.make_fit_batch(61, [n], pt_lo=lo, pt_hi=hi, pt_dist="loguniform")
        dev, geom = kf.to_device(b), kf.GeometryArgs.of(b.geom)
        want = kf.fit_tracks(ctx, geom, **dev, opt=kf.options(launch_mode=kf.LAUNCH_FLAT))
        routed = float(((want["flags"] & 16) != 0).float().mean())
        if n >= 32767:
            assert share[0] <= routed <= share[1], (lo, routed)
        for opt in (None, kf.options(tracks_per_block=64, reg_cap=96, hit_prefetch=1),
                    kf.options(tracks_per_block=128, reg_cap=128, hit_prefetch=4)):
            for _ in range(2):
                got = kf.fit_tracks(ctx, geom, **dev, opt=opt)
                for k in want:
                    assert np.array_equal(got[k].cpu().numpy(), want[k].cpu().numpy(), equal_nan=True), (lo, k)
    ctx.close()


@pytest.mark.parametrize("cond_max,share", [(1e4, (0.05, 0.3)), (10.0, (0.1, 0.5))])
def test_put_off_with_holes_stops_and_bad_hits(kf, cond_max, share):
    """More tracks than the gathering blocks take in one pass, sparsely put off, with
    hits missing, tracks that leave the barrel, hits and seeds that are not
    finite, and (cond_max 10) updates put off for their condition; every hit
    prefetch depth.  No mark of a track put off is left in the flags."""
    ctx, n = kf.Context(0), 160_001
    b = synth.make_fit_batch(66, [n], pt_lo=0.24, pt_hi=500.0, pt_dist="loguniform", eta_max=2.5, hit_eff=0.85,
                             sigma_rphi=0.001)
    rng = np.random.default_rng(1)
    bad = rng.choice(n, 300, replace=False)
    for k, t in enumerate(bad):  # the first used hit of some, a seed's value of others
        first = (int(b.hit_mask[t]) & -int(b.hit_mask[t])).bit_length() - 1
        if k % 3 == 0 and first >= 0:
            b.hit_pos[first, k % 2, t] = (np.nan, np.inf)[k % 2]
        elif k % 3 == 1 and first >= 0:
            b.hit_cov[first, (0, 2, 5)[k // 3 % 3], t] = (np.nan, np.inf, -1.0)[k // 9 % 3]
        else:
            b.seed_state[k % 6, t] = np.inf
    dev, geom = kf.to_device(b), kf.GeometryArgs.of(b.geom)
    want = kf.fit_tracks(ctx, geom, **dev, opt=kf.options(launch_mode=kf.LAUNCH_FLAT, cond_max=cond_max))
    flags = want["flags"].cpu().numpy()
    assert share[0] <= ((flags & 16) != 0).mean() <= share[1], ((flags & 16) != 0).mean()
    assert ((flags & 8) != 0).sum() >= 100 and ((flags & 2) != 0).sum() > 1000
    for shape in ({}, dict(tracks_per_block=32, reg_cap=96, hit_prefetch=2),
                  dict(tracks_per_block=256, reg_cap=128, hit_prefetch=4),
                  dict(tracks_per_block=64, reg_cap=80, hit_prefetch=1)):
        got = kf.fit_tracks(ctx, geom, **dev, opt=kf.options(cond_max=cond_max, **shape))
        assert (got["flags"] >= 0).all()  # bit 31 marks a track put off
        for k in want:
            assert np.array_equal(got[k].cpu().numpy(), want[k].cpu().numpy(), equal_nan=True), (shape, k)
    ctx.close()


@pytest.mark.parametrize("n", [300, 40_001])
@pytest.mark.parametrize("gain_max", [1.0, 100.0])
def test_float_float_gains_run_in_line(kf, n, gain_max):
    """With gain_max the plain kernel runs whatever the size and the shape: equal
    to KF_LAUNCH_FLAT bit for bit, and the shape reported is that kernel's."""
    ctx = kf.Context(0)
    b = synth.make_fit_batch(62, [n], pt_lo=0.24, pt_hi=500.0, pt_dist="loguniform", hit_eff=0.9)
    dev, geom = kf.to_device(b), kf.GeometryArgs.of(b.geom)
    want = kf.fit_tracks(ctx, geom, **dev, opt=kf.options(launch_mode=kf.LAUNCH_FLAT, gain_max=gain_max))
    assert float(((want["flags"] & 16) != 0).float().mean()) > 0.5
    for shape in ({}, dict(tracks_per_block=32, reg_cap=96, hit_prefetch=4)):
        got = kf.fit_tracks(ctx, geom, **dev, opt=kf.options(gain_max=gain_max, **shape))
        for k in want:
            assert np.array_equal(got[k].cpu().numpy(), want[k].cpu().numpy(), equal_nan=True), (shape, k)
        assert ctx.tuned_shape(b.geom.n_layers, n) == (64, 128, 1)
    ctx.close()


def test_new_context_behind_a_busy_default_stream(kf):
    """A context made while the default stream is busy, used at once on a stream
    that does not wait for it: what the context clears when it is made is cleared
    by then, so that no track put off is lost."""
    b = synth.make_fit_batch(63, [40_001], pt_lo=50.0, pt_hi=500.0, pt_dist="loguniform")
    dev, geom = kf.to_device(b), kf.GeometryArgs.of(b.geom)
    pinned = {k: v.cpu().pin_memory() for k, v in dev.items()}
    shape = dict(tracks_per_block=64, reg_cap=96, hit_prefetch=1)
    first = kf.Context(0)
    want = kf.fit_tracks(first, geom, **dev, opt=kf.options(launch_mode=kf.LAUNCH_FLAT))
    outs = [kf.fit_outputs(40_001, "cuda") for _ in range(100)]
    a = torch.randn(8192, 8192, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        a = (a @ a).clamp_(-1, 1)  # tens of ms on the default stream
    ctx = kf.Context(0)
    for out in outs:
        kf.fit_tracks(ctx, geom, **dev, out=out, opt=kf.options(**shape), stream=side)
    host = kf.fit_tracks_host(ctx, geom, **pinned)
    torch.cuda.synchronize()
    for out in outs + [host]:
        for k in want:
            assert np.array_equal(out[k].cpu().numpy(), want[k].cpu().numpy(), equal_nan=True), k
    ctx.close()
    first.close()


def test_replayed_fit_finds_its_own_tracks(kf):
    """A fit captured in a graph and replayed on batches with and without tracks to
    put off, other fits of the context in between: each replay's outputs are
    those of its own batch."""
    n, ctx, side = 40_001, kf.Context(0), torch.cuda.Stream()
    opt, flat = kf.options(tracks_per_block=64, reg_cap=96, hit_prefetch=1), kf.options(launch_mode=kf.LAUNCH_FLAT)
    batches = [synth.make_fit_batch(64, [n], pt_lo=50.0, pt_hi=500.0, pt_dist="loguniform"),
               synth.make_fit_batch(65, [n], pt_lo=1.0, pt_hi=5.0)]
    geom, dev = kf.GeometryArgs.of(batches[0].geom), [kf.to_device(b) for b in batches]
    want = [kf.fit_tracks(ctx, geom, **d, opt=flat) for d in dev]
    shares = [float(((w["flags"] & 16) != 0).float().mean()) for w in want]
    assert shares[0] > 0.05 and shares[1] == 0.0, shares
    buf, out, other = {k: v.clone() for k, v in dev[0].items()}, kf.fit_outputs(n, "cuda"), kf.fit_outputs(n, "cuda")
    kf.fit_tracks(ctx, geom, **buf, out=out, opt=opt)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        kf.fit_tracks(ctx, geom, **buf, out=out, opt=opt, stream=side)
    for i in (0, 1, 0, 0, 1, 1, 0):
        for k in buf:
            buf[k].copy_(dev[i][k])
        graph.replay()
        for k in out:
            assert np.array_equal(out[k].cpu().numpy(), want[i][k].cpu().numpy(), equal_nan=True), (i, k)
        kf.fit_tracks(ctx, geom, **dev[i ^ 1], out=other, opt=opt)
        assert all(np.array_equal(other[k].cpu().numpy(), want[i ^ 1][k].cpu().numpy(), equal_nan=True) for k in other)
    ctx.close()
