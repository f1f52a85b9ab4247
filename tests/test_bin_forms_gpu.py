"""The binning's two forms (passes over all points at once; one block per
segment) and the final order by id, where they can go wrong: empty and
one-hit segments, runs of 32 bins longer and shorter than a warp takes at
once, single bins beyond that, more hits in a bin than a place word holds.
The reference bins the same hits in pieces of at most 3 000 (one block each),
reads every hit's bin from that, and sorts by (bin, id) on the host."""
import numpy as np
import pytest

from paper_1605_05508_gb300 import synth as S
from fitutil import to_dev

pytestmark = pytest.mark.gpu


def _bin(ctx, kf, torch, xyz, offs, n_events, n_layers, unordered, fine):
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0, unordered)
    i32 = dict(dtype=torch.int32, device="cuda")
    n, nseg = xyz.shape[1], n_events * n_layers
    bins = kf.HitBins(torch.empty((n, 4), device="cuda"), torch.empty((nseg, kf.NBINS + 1), **i32),
                      fine_off=torch.empty((nseg, kf.NBINS_FINE + 1), **i32) if fine else None)
    kf.kf_bin_hits(ctx, kf.LayerHits(to_dev(xyz), to_dev(np.asarray(offs, np.int64)), n_events, n_layers, 3), bins)
    torch.cuda.synchronize()
    return bins.hits.cpu().numpy(), (bins.fine_off if fine else bins.bin_off).cpu().numpy(), bins.bin_off.cpu().numpy()


def _hit_bins(ctx, kf, torch, xyz, fine):
    """Every hit's (sub-)bin, from binning pieces of at most 3 000 hits."""
    n = xyz.shape[1]
    cuts = list(range(0, n, 3000)) + [n]
    hits, off, _ = _bin(ctx, kf, torch, xyz, cuts, len(cuts) - 1, 1, 1, fine)
    out = np.empty(n, np.int64)
    for k, (a, b) in enumerate(zip(cuts[:-1], cuts[1:])):
        out[a + hits[a:b, 3].view(np.int32)] = np.repeat(np.arange(off.shape[1] - 1), np.diff(off[k]))
    return out


def _points(rng, n, spread):
    """n points near r = 16 cm, within `spread` rad of phi = 0.3 and `spread` in eta."""
    phi, eta = 0.3 + spread * rng.uniform(-1, 1, n), 0.5 * spread * rng.uniform(-1, 1, n)
    r = 16.0 + 0.01 * rng.normal(size=n)
    return np.stack([r * np.cos(phi), r * np.sin(phi), r * np.sinh(eta)]).astype(np.float32)


@pytest.mark.parametrize("sizes,spread", [
    ((5000, 0, 1, 9001), 3.1),             # mostly lone hits: runs below a warp's
    ((4000, 1, 6000), 0.3),                # a few hundred hits in 32 bins
    ((3100, 3300), 0.02),                  # bins of hundreds of hits
    ((31, 0, 1, 3000), 0.3),               # small segments: one block each
])
@pytest.mark.parametrize("unordered,fine", [(0, False), (1, False), (1, True)])
def test_forms_sort_by_bin_and_id(cuda_ctx_factory, sizes, spread, unordered, fine):
    import torch
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii)
    rng = np.random.default_rng(len(sizes) + sizes[0])
    xyz = np.concatenate([_points(rng, n, spread) for n in sizes], axis=1)
    offs = np.concatenate([[0], np.cumsum(sizes)])
    hits, off, coarse = _bin(ctx, kf, torch, xyz, offs, len(sizes), 1, unordered, fine)
    bins = _hit_bins(ctx, kf, torch, xyz, fine)
    for s, (a, b) in enumerate(zip(offs[:-1], offs[1:])):
        ref = np.bincount(bins[a:b], minlength=off.shape[1] - 1)
        np.testing.assert_array_equal(off[s], np.concatenate([[0], np.cumsum(ref)]))
        np.testing.assert_array_equal(coarse[s], off[s][::2] if fine else off[s])
        ids = hits[a:b, 3].view(np.int32)
        np.testing.assert_array_equal(hits[a:b, :3], xyz[:, a + ids].T)
        order = np.argsort(bins[a:b], kind="stable")
        if unordered:  # the same hits in every bin
            ids = ids[np.lexsort((ids, bins[a + ids]))]
        np.testing.assert_array_equal(ids, order)


@pytest.mark.parametrize("fine", [False, True])
def test_more_hits_in_a_bin_than_a_place_word_holds(cuda_ctx_factory, fine):
    """150 000 hits of one segment in one bin (unordered form)."""
    import torch
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii)
    n = 150_000
    xyz = np.tile(_points(np.random.default_rng(1), 1, 0.0), (1, n))
    hits, off, _ = _bin(ctx, kf, torch, xyz, [0, n], 1, 1, 1, fine)
    assert np.count_nonzero(np.diff(off[0])) == 1 and off[0][-1] == n
    np.testing.assert_array_equal(np.sort(hits[:, 3].view(np.int32)), np.arange(n))
