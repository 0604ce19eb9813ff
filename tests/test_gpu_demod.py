"""Demodulation by nodes and the FP64 transform on chip against the oracle, at the edges of
their blocks and rules: series that end on the first, a middle and the last sample of a
block of 32 to 256 samples, the largest sampling interval that is taken by nodes and one
above it, every split of the FP64 transform with F on the band, on all bins and interbinned."""
import numpy as np
import pytest
import torch

from tests.helpers import F64_TOL
from oracle import earth
from oracle import fstat as ofs
from oracle import resample as ors
from paper_1003_0844_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1003_0844_gb300 import build, fstat
    build.build()
    fstat.load_library()
    return fstat


def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


# 256 samples per block at 2 s and below, 64 at 8 s, 32 at 16 s; every sample at 16.1 s
@pytest.mark.parametrize("dt,n", [(2.0, 4096), (2.0, 4097), (2.0, 4351), (2.0, 700), (0.5, 20001), (0.3, 9999),
                                  (3.0, 5000), (8.0, 10769), (16.0, 5377), (16.0, 5408), (16.1, 5377)])
def test_demodulated_series_matches_oracle(fs, dt, n):
    """Source times: the delay in double-float (1e-12 s) and its polynomial (1e-13 s), the
    oracle's own 1e-10 s; above 16 s the standing 2e-6 s of one Newton step in FP32.  The
    series: at most 40 roundings of FP32 (spline, amplitude, heterodyne) of the largest value,
    2.4e-6, or the parity tests' 2e-4 of its rms above 16 s.  The means: FP32 values, 1e-6."""
    det = W.Detector(lambda_e0=1.0)
    x = np.random.default_rng(n).standard_normal(n).astype(np.float32).astype(np.float64)
    ctx = fs.Context(det)
    seg = fs.Segment(ctx, _dev(x, torch.float32), dt, 1 << max(12, (n - 1).bit_length()), 435.1875, 2 * dt, t0=3e5)
    oseg = ors.Segment(x, dt)
    odet = earth.detector_at_epoch(det, 3e5)
    for alpha, delta in ((0.7, 0.4), (4.0, -1.3)):
        ya, yb, ts, ab = fs.demodulate(ctx, seg, alpha, delta)
        assert ctx.sync_status() == 0
        ref = ofs.demodulate(oseg, alpha, delta, 0.0, 435.1875, odet)
        assert np.max(np.abs(ts.cpu().numpy() - ref.t_src)) < (1e-9 if dt <= 16.0 else 2e-6)
        for got, want in ((ya, ref.ya), (yb, ref.yb)):
            err = np.max(np.abs(got.cpu().numpy() - want))
            assert err < (2.4e-6 * np.max(np.abs(want)) if dt <= 16.0 else 2e-4 * np.sqrt(np.mean(np.abs(want) ** 2)))
        a2, b2 = ab.cpu().numpy()
        assert abs(a2 / ref.a2 - 1) < 1e-6 and abs(b2 / ref.b2 - 1) < 1e-6


@pytest.mark.parametrize("p", range(12, 22))
@pytest.mark.parametrize("how", ["band", "all", "interbin"])
def test_fp64_transform_of_every_length(fs, p, how):
    nfft, n, dt, fl = 1 << p, 3001, 8.0, 435.1875
    det = W.Detector(lambda_e0=0.3)
    x = np.random.default_rng(p).standard_normal(n)
    f1 = np.array([-1e-8, -3e-9, 0.0])[:1 + p % 3]
    ctx = fs.Context(det)
    seg = fs.Segment(ctx, _dev(x), dt, nfft, fl, 2 * dt, precision="f64", interbin=how == "interbin")
    nb = nfft // 2 if how == "band" else nfft
    res = fs.search(ctx, seg, _dev([1.1]), _dev([0.2]), _dev(f1), 12.0, nbins=nb)
    assert ctx.sync_status() == 0
    F = res.F.cpu().numpy()
    oseg = ors.Segment(x, dt)
    for m in range(len(f1)):
        if how == "interbin":
            ref = ofs.fstat_interbinned(oseg, 1.1, 0.2, f1[m], fl, det, 2 * dt, nfft)
        else:
            ref = ofs.fstat(oseg, 1.1, 0.2, f1[m], fl, det, 2 * dt, nfft, nbins=nb)
        assert np.max(np.abs(F[m] - ref) / np.maximum(ref, 1.0)) <= F64_TOL
    sky, spin, k, Fc = res.candidates()
    assert len(k) == np.count_nonzero(F > 12.0) and np.allclose(F[spin, k], Fc, rtol=1e-6)


# The delay is up to 4e7 (1e8) half-samples here; the data holds sources whose delay stays
# within its 2.5 s (1 s), and reads nothing for the others.
@pytest.mark.parametrize("dt,n", [(2.5e-5, 100001), (1e-5, 100001)])
def test_short_sampling_intervals_match_oracle(fs, dt, n):
    """Bounds as at the other intervals (an error of 1e-12 s of the delay is 2e-7 half-samples
    at most), and the rounding of a and b themselves, sums of five FP32 terms of order one
    (2.4e-7): they are constant over so short a span, so it does not average out.  A source perpendicular to the Earth's position, one turned from there by a
    delay of 0.3 of the span (either way), and one whose delay exceeds the span."""
    det = W.Detector(lambda_e0=1.0)
    x = np.random.default_rng(n).standard_normal(n).astype(np.float32).astype(np.float64)
    ctx = fs.Context(det)
    seg = fs.Segment(ctx, _dev(x, torch.float32), dt, 1 << 17, 435.1875, 2 * dt)
    oseg = ors.Segment(x, dt)
    ce, se = np.cos(det.eps), np.sin(det.eps)
    for lon, lat in ((1.0 + np.pi / 2, 0.8), (1.0 + np.pi / 2 + 0.3 * n * dt / 499.0, 0.1),
                     (1.0 + np.pi / 2 - 0.3 * n * dt / 499.0, -0.1), (2.0, -0.5)):
        ec = np.array([np.cos(lat) * np.cos(lon), np.cos(lat) * np.sin(lon), np.sin(lat)])
        eq = np.array([ec[0], ce * ec[1] - se * ec[2], se * ec[1] + ce * ec[2]])
        alpha, delta = float(np.arctan2(eq[1], eq[0])), float(np.arcsin(eq[2]))
        ya, yb, ts, ab = fs.demodulate(ctx, seg, alpha, delta)
        assert ctx.sync_status() == 0
        ref = ofs.demodulate(oseg, alpha, delta, 0.0, 435.1875, det)
        assert np.max(np.abs(ts.cpu().numpy() - ref.t_src)) < 1e-9
        far = lon == 2.0
        assert far == (np.count_nonzero(ref.ya) == 0) and (far or np.count_nonzero(ref.ya) > n // 2)
        for got, want in ((ya, ref.ya), (yb, ref.yb)):
            assert np.max(np.abs(got.cpu().numpy() - want)) <= 2.4e-6 * np.max(np.abs(want)) + 2.4e-7 * np.max(np.abs(x)) * (not far)
        a2, b2 = ab.cpu().numpy()
        for got, want in ((a2, ref.a2), (b2, ref.b2)):
            assert abs(got / want - 1) < 1e-6 + 4.8e-7 / np.sqrt(want)


# Up to 16 sky positions, and two blocks of nodes per SM (4 positions of this series on 152
# SMs), the node kernel sets the search up itself.
@pytest.mark.parametrize("n,nfft,few,many", [(5000, 8192, 16, 17), (258492, 1 << 18, 4, 5), (258492, 1 << 18, 2, 17)])
def test_set_up_in_the_node_kernel_changes_nothing(fs, n, nfft, few, many):
    """The positions that two searches share have the same F and crossings, to the bit."""
    dt, rng = 2.0, np.random.default_rng(n + many)
    ctx = fs.Context(W.Detector(lambda_e0=1.0))
    seg = fs.Segment(ctx, _dev(rng.standard_normal(n), torch.float32), dt, nfft, 435.1875, 2 * dt)
    alpha, delta = _dev(rng.uniform(0, 2 * np.pi, many)), _dev(np.arcsin(rng.uniform(-1, 1, many)))
    f1 = _dev([-1e-8, -3e-9, 0.0])
    a = fs.search(ctx, seg, alpha[:few].contiguous(), delta[:few].contiguous(), f1, 14.0)
    assert ctx.sync_status() == 0
    Fa, ca = a.F.clone(), sorted(zip(*(v.tolist() for v in a.candidates())))
    b = fs.search(ctx, seg, alpha, delta, f1, 14.0)
    assert ctx.sync_status() == 0
    assert torch.equal(b.F[:3 * few], Fa)
    assert ca == sorted(c for c in zip(*(v.tolist() for v in b.candidates())) if c[0] < few)
    again = fs.search(ctx, seg, alpha[:few].contiguous(), delta[:few].contiguous(), f1, 14.0)  # the counters are zero again
    assert torch.equal(again.F, Fa)
