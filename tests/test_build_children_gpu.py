"""The register-resident build's child lists against the grouped layout's
64-bit keys where they can go wrong: several copies of every hit (chi2 equal to
the last bit, so the hit id decides), windows of more hits than are staged at
a time, and more compatible children than a list holds.  Same bits, for every
number of lanes a seed, by bin and by sub-bin."""
import numpy as np
import pytest

from paper_1605_05508_gb300 import synth as S
from buildutil import gpu_build

pytestmark = pytest.mark.gpu

KEYS = ("par", "cov", "chi2", "nhits", "status", "hits", "n_cands", "cand_hits", "cand_chi2", "cand_nhits")


def _with_copies(batch, copies, seed):
    """Every segment's hits `copies` times over, in random order."""
    rng = np.random.default_rng(seed)
    segs = [batch.layer_xyz[:, a:b] for a, b in zip(batch.layer_off[:-1], batch.layer_off[1:])]
    segs = [np.tile(s, (1, copies))[:, rng.permutation(s.shape[1] * copies)] for s in segs]
    batch.layer_xyz = np.ascontiguousarray(np.concatenate(segs, axis=1))
    batch.layer_off = batch.layer_off * copies
    return batch


@pytest.mark.parametrize("copies", [1, 2, 5, 13])
@pytest.mark.parametrize("max_cands", [8, 6, 5, 4, 2, 1])
def test_tied_and_crowded_children(cuda_ctx_factory, copies, max_cands):
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii, max_cands=8)
    batch = _with_copies(S.make_build_batch(2100 + copies, 2, 130, noise_near=1, noise_near_sigma=0.02), copies, copies)
    kf.kf_set_tuning(ctx, 128, 0, 8, 0, 0, 0, 1)
    ref = gpu_build(ctx, batch, max_cands)
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0, 1)
    for fine in (False, True):
        got = gpu_build(ctx, batch, max_cands, fine=fine)
        for k in KEYS:
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"fine={fine} {k}")
    assert ref["nhits"].min() > 0
