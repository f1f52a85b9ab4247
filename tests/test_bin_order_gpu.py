"""The ordered binning's final pass where bins are crowded: bins longer than a
warp takes at once, more hits in a bin than a place word holds, and its time
there."""
import numpy as np
import pytest

from paper_1605_05508_gb300 import synth as S
from fitutil import to_dev

pytestmark = pytest.mark.gpu


def _points(rng, n, dphi, deta):
    """n points at r = 16 cm, within dphi rad and deta of (0.3, 0.1)."""
    phi, eta = 0.3 + dphi * rng.uniform(-1, 1, n), 0.1 + deta * rng.uniform(-1, 1, n)
    return np.stack([16 * np.cos(phi), 16 * np.sin(phi), 16 * np.sinh(eta)]).astype(np.float32)


def _setup(ctx, kf, torch, xyz, offs):
    n, nseg = xyz.shape[1], len(offs) - 1
    lh = kf.LayerHits(to_dev(xyz), to_dev(np.asarray(offs, np.int64)), nseg, 1, 3)
    return lh, kf.HitBins(torch.empty((n, 4), device="cuda"),
                          torch.empty((nseg, kf.NBINS + 1), dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("sizes,dphi,deta", [
    ((129, 128, 4000), 0.0, 0.0),      # single bins, just past a run and far past it; 2 passes of the sort
    ((70_000, 3, 20_000), 0.05, 0.0),  # a few bins of thousands; 3 passes
    ((300_000,), 0.6, 0.3),            # hundreds of bins just around a run
    ((150_000,), 0.0, 0.0),            # more hits in one bin than a place word holds
    ((1_000_000,), 3.1, 1.4),          # a dense segment: the pass with few bins a warp
    ((3000,) * 27, 3.1, 1.4),          # many sparse segments: 128 bins a warp
    ((300,) * 30 + (60_000, 0, 1), 0.5, 0.5),  # the same with a crowded one
    ((30_000,) * 160, 3.1, 1.4),       # many segments of over a hit a bin: 64 bins a warp
    ((20,) * 60 + (160_000,), 0.0, 0.0),                   # large segments among many small ones: all in
    ((100,) * 200 + (100_000, 0, 70_000, 5), 3.1, 1.4),    # one bin; two of them, more segments than SMs;
    ((12_000,) * 155 + (1_000_000,) * 2, 1.0, 1.0),        # with 64 bins a warp
])
def test_crowded_bins_in_id_order(cuda_ctx_factory, sizes, dphi, deta):
    """Every hit once, with its own coordinates, ids ascending inside each bin,
    and the bins of the unordered binning."""
    import torch
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii)
    xyz = _points(np.random.default_rng(sizes[0]), sum(sizes), dphi, deta)
    offs = np.concatenate([[0], np.cumsum(sizes)])
    lh, b = _setup(ctx, kf, torch, xyz, offs)
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0, 1)
    kf.kf_bin_hits(ctx, lh, b)
    torch.cuda.synchronize()
    any_order, off = b.hits.cpu().numpy().copy(), b.bin_off.cpu().numpy().copy()
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0, 0)
    kf.kf_bin_hits(ctx, lh, b)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(b.bin_off.cpu().numpy(), off)
    hits = b.hits.cpu().numpy()
    for s, (p, e) in enumerate(zip(offs[:-1], offs[1:])):
        ids, ids0 = hits[p:e, 3].view(np.int32), any_order[p:e, 3].view(np.int32)
        np.testing.assert_array_equal(hits[p:e, :3], xyz[:, p + ids].T)
        bin_of = np.repeat(np.arange(kf.NBINS), np.diff(off[s]))
        np.testing.assert_array_equal(ids, ids0[np.lexsort((ids0, bin_of))])


def _best_us(ctx, kf, torch, sizes, dphi, deta, unordered, n=8):
    """The fastest of n timed calls."""
    offs = np.concatenate([[0], np.cumsum(sizes)])
    lh, b = _setup(ctx, kf, torch, _points(np.random.default_rng(3), offs[-1], dphi, deta), offs)
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0, unordered)
    us = []
    for _ in range(n):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        kf.kf_bin_hits(ctx, lh, b)
        t1.record()
        torch.cuda.synchronize()
        us.append(1e3 * t0.elapsed_time(t1))
    return min(us)


def test_crowded_bins_take_no_quadratic_time(cuda_ctx_factory):
    """60 000 hits in some 325 bins, ordered, in no more than the 1.1 ms that
    one thread a bin, sorting by insertion, took on a GB300."""
    import torch
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii)
    assert _best_us(ctx, kf, torch, [60_000], 0.3, 0.3, 0) < 1100


def test_one_large_segment_among_many_spreads_over_the_gpu(cuda_ctx_factory):
    """154 segments, one of 700 000 hits: ordered in no more than the 275 us that
    the passes over all points with a sort by a thread a bin took on a GB300 (one
    block for that segment: 1 072 us)."""
    import torch
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii)
    assert _best_us(ctx, kf, torch, [2000] * 70 + [700_000] + [2000] * 83, 3.1, 1.4, 0) < 275
