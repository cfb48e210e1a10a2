"""The library's per-track arithmetic (csrc/kf_math.cuh, fit_track of
csrc/kf_fit.cu) compiled for the host, against 64 bits."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1705_02876_gb300 import synth
from paper_1705_02876_gb300.build import nvcc

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
EPS = 2.0 ** -24  # half an ulp of FP32, relative
pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")


def _compile(name, tmp):
    so = str(tmp.mktemp("host") / (name + ".so"))
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-w",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1705_02876_gb300", "csrc"),
                    "-I", os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include"),
                    "-o", so, os.path.join(HERE, "host", name + ".cpp")], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return _compile("track_math", tmp_path_factory)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _opt(mode=1, cond_max=1e4, pt_lo=0.25, pt_hi=200.0, gain_max=0.0):
    return np.array([mode, cond_max, pt_lo, pt_hi, gain_max], np.float32)


def test_seed_covariance_on_the_first_layer(host, oracle):
    """What the first hit's t leaves of q2's variance, vv - vt^2 / tt, from a
    seed's covariance on the first layer: a small difference of terms of size vv
    (tt and vt^2 / tt are no larger in it), which the fit's covariance inherits.
    Each entry rounded once, by EPS / sqrt(3) of itself in the root mean square,
    puts it off by sqrt(1 + 4 + 1) EPS / sqrt(3) = sqrt(2) EPS vv; the sums' own
    roundings stay below that, in FP32 and further below in float-float (tracks
    outside the pT bounds)."""
    n = 3000
    b = synth.make_fit_batch(5, [n], pt_lo=0.24, pt_hi=500.0, pt_dist="loguniform", eta_max=1.5)
    g = b.geom
    r = float(np.float32(g.radii[0]))
    c, fl = {}, np.empty(n, np.uint32)
    for name, opt in (("float-float", _opt(pt_lo=1e3, pt_hi=2e3)), ("FP32", _opt(mode=0))):
        c[name] = np.empty((15, n), np.float32)
        host.host_enter(ctypes.c_int64(n), _p(b.seed_state), _p(b.seed_cov), _p(b.charge),
                        ctypes.c_float(0.00299792458 * g.bz), ctypes.c_float(r), ctypes.c_float(g.z_half), _p(opt),
                        _p(c[name]), _p(fl))
    rel = {k: [] for k in c}
    il = np.tril_indices(6)
    for t in np.nonzero(fl == 0)[0]:
        ok, x, J, _ = oracle.propagate(b.seed_state[:, t], int(b.charge[t]), float(np.float32(g.bz)), r)
        assert ok
        C = np.zeros((6, 6))
        C[il] = b.seed_cov[:, t]
        C = J @ (C + C.T - np.diag(np.diag(C))) @ J.T
        R, pt = np.hypot(x[0], x[1]), np.hypot(x[3], x[4])
        ut, uv = np.zeros(6), np.zeros(6)
        ut[:2] = -x[1] / R, x[0] / R
        uv[3:5] = -x[4] / pt, x[3] / pt
        tt, vt, vv = ut @ C @ ut, uv @ C @ ut, uv @ C @ uv
        for k in c:
            ctt, cvt, cvv = c[k][[0, 6, 9], t].astype(np.float64)
            rel[k].append((cvv - cvt ** 2 / ctt - (vv - vt ** 2 / tt)) / (EPS * vv))
    assert len(rel["FP32"]) > 0.9 * n
    rms = {k: float(np.sqrt(np.mean(np.square(v)))) for k, v in rel.items()}
    assert rms["FP32"] <= np.sqrt(2) and rms["float-float"] <= 0.9 * rms["FP32"], rms


def _updates(rng, n):
    """n local states, covariances and hits: x [6][n], c [15][n], n [2][n], m [3][n], v [6][n]."""
    A = rng.normal(size=(n, 5, 5)) * np.array([1e-2, 0.1, 1e-2, 1e-2, 0.1])[:, None]
    C = A @ A.transpose(0, 2, 1)
    il = np.tril_indices(5)
    phi = rng.uniform(0, 2 * np.pi, n)
    nrm = np.stack([np.cos(phi), np.sin(phi)])
    x = np.concatenate([4 * nrm, rng.normal(size=(1, n)), rng.normal(size=(3, n))])
    m = x[:3] + 0.01 * rng.normal(size=(3, n))
    v = np.zeros((6, n))
    v[0] = v[2] = 1e-4
    v[5] = 1e-2
    return [np.ascontiguousarray(a, dtype=np.float32) for a in (x, C[:, il[0], il[1]].T, nrm, m, v)]


def _slot_update(host, kind, x, c, nrm, m, v):
    n = x.shape[1]
    x, c, chi2, st = x.copy(), c.copy(), np.empty(n, np.float32), np.empty(n, np.int32)
    host.host_slot_update(kind, ctypes.c_int64(n), _p(x), _p(c), _p(nrm), _p(m), _p(v), _p(chi2), _p(st))
    return st, x, c, chi2


def test_float_float_update_tells_a_bad_s(host):
    """A hit covariance whose t pivot, C_tt + V_tt - V_nt^2 / V_nn, lies within
    some FP32 ulps of zero on either side (float-float resolves 2^-46 of its
    terms, here it is 2^-28 and more): the float-float update refuses what the
    FP64 one refuses, with the state and covariance left alone, and agrees with
    it on the rest."""
    n = 4000
    rng = np.random.default_rng(3)
    x, c, nrm, m, v = _updates(rng, n)
    nrm[0], nrm[1] = 1, 0
    c[[0, 1, 3, 6, 10]] = 0
    c[0] = (1e-9 * rng.uniform(1, 2, n)).astype(np.float32)
    a = rng.uniform(0.5, 1, n).astype(np.float32)
    v[0], v[1] = 1, a
    v[2] = (a.astype(np.float64) ** 2 * (1 + 2.0 ** -23 * rng.integers(-3, 4, n))).astype(np.float32)
    pivot = c[0].astype(np.float64) + v[2] - a.astype(np.float64) ** 2
    sel = np.abs(pivot) > 2.0 ** -28
    assert (pivot[sel] < 0).sum() > 500 and (pivot[sel] > 0).sum() > 500
    st2 = _slot_update(host, 2, x, c, nrm, m, v)[0]
    st3, x3, c3, _ = _slot_update(host, 3, x, c, nrm, m, v)
    assert (st2[sel] == np.where(pivot[sel] > 0, 2, 1)).all()
    assert np.array_equal(st3[sel], st2[sel])
    bad = st3 == 1
    assert np.array_equal(x3[:, bad], x[:, bad]) and np.array_equal(c3[:, bad], c[:, bad])


def test_update_outside_pt_bounds_keeps_a_precise_hit(host):
    """Predictions 2^6 to 2^26 times as wide as the hit, in t and z: the variances
    the update leaves, C V / (C + V) of an uncorrelated pair, against 64 bits.
    Half an ulp is EPS; the arithmetic adds 2^-45 C / V <= EPS / 2 of float-float
    below 2^20, and 2^-53 C / V of FP64 beyond."""
    n = 4000
    rng = np.random.default_rng(8)
    x, c, nrm, m, v = _updates(rng, n)
    nrm[0], nrm[1] = 1, 0
    c[[1, 3, 4, 6, 7, 10, 11]] = 0  # t and z uncorrelated with the rest
    c[0], c[2] = (2.0 ** rng.uniform(-10, 8, (2, n))).astype(np.float32)
    v[0] = v[2] = (c[0] * 2.0 ** rng.uniform(-26, -6, n)).astype(np.float32)
    v[5] = (c[2] * 2.0 ** rng.uniform(-26, -6, n)).astype(np.float32)
    m[:2] = x[:2]
    chi2, st = np.empty(n, np.float32), np.empty(n, np.int32)
    got = c.copy()
    host.host_update(ctypes.c_int64(n), _p(x.copy()), _p(got), _p(nrm), _p(m), _p(v),
                     _p(_opt(cond_max=1e30, pt_lo=1e3, pt_hi=2e3)), _p(chi2), _p(st))
    assert (st == 2).all()
    for i, j in ((0, 2), (2, 5)):
        want = c[i].astype(np.float64) * v[j] / (c[i].astype(np.float64) + v[j])
        rel = np.abs(got[i] / want - 1) / EPS
        assert rel.max() <= 1.5, (i, rel.max())


def test_fit_reads_no_absent_hit(tmp_path_factory, oracle):
    """The hits a fit reads are those of the mask, up to the layer where it stops;
    what the fit gives is the oracle's."""
    lib = _compile("fit_track", tmp_path_factory)
    n = 500
    b = synth.make_fit_batch(9, [n], geom=synth.toy_geometry(17), hit_eff=0.6, eta_max=2.0)
    g, L = b.geom, 17
    pad = np.zeros(3 * n * (32 - L), np.float32)  # hit_cov begins 32 layers after hit_pos
    block = np.concatenate([np.ravel(b.hit_pos).astype(np.float32), pad, np.ravel(b.hit_cov).astype(np.float32),
                            np.zeros(6 * n * (32 - L), np.float32)])
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    r, xx0 = f32(g.radii), f32(g.x_over_x0)
    mask = np.ascontiguousarray(b.hit_mask, dtype=np.uint32)
    out = [np.empty((6, n), np.float32), np.empty((21, n), np.float32), np.empty(n, np.float32), np.empty(n, np.int16),
           np.empty(n, np.uint32)]
    read = np.empty(n, np.uint32)
    lib.host_fit(L, _p(r), _p(xx0), ctypes.c_float(g.z_half), ctypes.c_float(0.00299792458 * g.bz), ctypes.c_int64(n),
                 _p(f32(b.seed_state)), _p(f32(b.seed_cov)), _p(b.charge), _p(block),
                 ctypes.c_void_p(block.ctypes.data + 4 * 3 * n * 32), _p(mask), *[_p(a) for a in out], _p(read))
    ref = oracle.fit_batch(b)
    stopped = (out[4] & 3) != 0
    assert np.array_equal(out[3], ref["ndof"]) and stopped.any()
    assert ((read & ~mask) == 0).all()
    assert (read[~stopped] == mask[~stopped]).all() and (mask != (1 << L) - 1).any()
    assert np.linalg.norm(out[0] - ref["state"]) < 1e-4 * np.linalg.norm(ref["state"])


def test_flop_count(tmp_path_factory):
    """The flops per track-layer and per track by which bench.py rates the fit and
    the build: counted on the kernels' source, the same for every track of the
    fit workload."""
    import bench
    lib = _compile("track_flops", tmp_path_factory)
    n, L = 100, 10
    b = synth.make_fit_batch(1, [n])
    g = b.geom
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    arrays = [f32(b.seed_state), f32(b.seed_cov), b.charge, f32(b.hit_pos), f32(b.hit_cov)]
    count = np.zeros(3, np.uint64)
    lib.host_count(L, _p(f32(g.radii)), _p(f32(g.x_over_x0)), ctypes.c_float(g.z_half),
                   ctypes.c_float(0.00299792458 * g.bz), ctypes.c_int64(n), *[_p(a) for a in arrays], _p(count))
    assert count[1] == n * (L - 1)
    assert count[0] == bench.FLOPS_PER_TRACK_LAYER * count[1] and count[2] == bench.FLOPS_PER_TRACK_ENDS * n
