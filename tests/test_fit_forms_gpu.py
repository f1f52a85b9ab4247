"""The fit in one launch and the staged launches per layer give the same bits
(batches whose layout the staged form takes, so that the two differ in every
launch), and what each asks of the context's device memory."""
import pytest

from paper_1605_05508_gb300 import synth as S
from fitutil import to_dev

pytestmark = pytest.mark.gpu


def _batch(n, seed=77):
    ev = S.make_fit_batch(seed, n, pt_range=(0.2, 10.0), keep_truth=False)
    valid = ev.hits.valid.copy()
    valid[3, ::7] = 0
    return ev, valid


def _run(ctx, fn, ev, valid, lo=True, status=True):
    import torch
    from paper_1605_05508_gb300 import kf
    n, L = ev.seeds.par.shape[1], ev.hits.xyz.shape[0]
    s = kf.Tracks(to_dev(ev.seeds.par), to_dev(ev.seeds.cov), to_dev(ev.seeds.charge))
    o = kf.Tracks(torch.empty((6, n), device="cuda"), torch.empty((21, n), device="cuda"), s.charge,
                  torch.empty((3, n), device="cuda") if lo else None)
    chi2, st = torch.empty((L, n), device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda") if status else None
    h = kf.TrackHits(to_dev(ev.hits.xyz), to_dev(valid))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    fn(ctx, s, h, o, chi2, st)
    torch.cuda.synchronize()
    return [t for t in (o.par, o.par_lo, o.cov, chi2, st) if t is not None], free - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("n,chunk", [(32, 0), (4096, 0), (40_000, 0), (300_032, 262144)])
def test_one_launch_equals_staged_launches(cuda_ctx_factory, n, chunk):
    import torch
    from paper_1605_05508_gb300 import kf
    ctx = cuda_ctx_factory(S.barrel().radii)
    ev, valid = _batch(n)
    kf.kf_set_tuning(ctx, 64, 0, 8, 4, chunk, 1)
    staged, _ = _run(ctx, kf.kf_fit, ev, valid)
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0)
    for fn in (kf.kf_fit, kf.kf_fit_fused, kf.kf_fit_noalloc)[:3 if n <= kf.NOALLOC_MAX_TRACKS else 2]:
        for a, b in zip(_run(ctx, fn, ev, valid)[0], staged):
            assert torch.equal(a, b)


def test_the_single_launch_takes_no_device_memory(cuda_ctx_factory):
    """In a context that may allocate nothing: kf_fit_noalloc, and kf_fit where
    it takes the single launch (by tuning, or for a layout that the staged form
    does not take), without status or low parts given; the staged form's scratch
    does not fit such a context."""
    from paper_1605_05508_gb300 import kf
    det = S.barrel()
    ctx = cuda_ctx_factory(det.radii, mem_budget_bytes=1)
    for n in (1001, kf.NOALLOC_MAX_TRACKS):
        ev, valid = _batch(n)
        for fn in (kf.kf_fit, kf.kf_fit_noalloc):
            _run(ctx, fn, ev, valid, False, False)  # loads the kernel
            assert _run(ctx, fn, ev, valid, False, False)[1] == 0
    kf.kf_set_tuning(ctx, 64, 0, 8, 4, 0, 1)
    _run(ctx, kf.kf_fit, *_batch(1001), False, False)
    with pytest.raises(kf.KfError) as e:
        _run(ctx, kf.kf_fit, *_batch(1024), False, False)
    assert e.value.code == kf.KF_ENOMEM
