"""The window of a candidate holds every hit with chi2 below the cut: kf_build
(one layer, one candidate) over binned hits against the same build over bins
that each hold every hit, so that whatever window is scanned sees all of them.
The hits lie just inside the chi2 cut, where its ellipsoid reaches farthest in
phi or in z, and within 1e-5 of an edge of a phi bin or an eta row."""
import numpy as np
import pytest

from paper_1605_05508_gb300 import synth as S
from fitutil import to_dev

pytestmark = pytest.mark.gpu
CUT, ETA_ROW = 30.0, 3.0 / 64


def _seeds(rng, n, R):
    """States at radius R with radial momentum, any phi and z; position
    covariance sigma^2 in x and y, so that a rotation or a shift in z changes
    nothing else."""
    phi, cot = rng.uniform(-np.pi, np.pi, n), rng.uniform(-1.2, 1.2, n)
    pt, sig, sz = rng.uniform(0.7, 8, n), 10 ** rng.uniform(-2.5, -0.3, n), 10 ** rng.uniform(-2, 0, n)
    z = R * cot + rng.uniform(-2, 2, n)
    cov = np.zeros((21, n))
    for i, v in enumerate((sig**2, sig**2, sz**2, 1e-8, 1e-8, 1e-8)):
        cov[i * (i + 1) // 2 + i] = v
    return phi, z, pt, cot, cov


def _state(phi, z, pt, cot, R):
    return np.stack([R * np.cos(phi), R * np.sin(phi), z, pt * np.cos(phi), pt * np.sin(phi), pt * cot])


@pytest.mark.parametrize("along", ["phi", "z"])
@pytest.mark.parametrize("fine", [False, True])
def test_no_compatible_hit_outside_the_window(cuda_ctx_factory, along, fine):
    import torch
    from paper_1605_05508_gb300 import kf
    det = S.barrel()
    ctx = cuda_ctx_factory(det.radii)
    kf.kf_set_tuning(ctx, 128, 0, 8, 4, 0, 0, 1)
    n, nb, nbf = 1200, kf.NBINS, kf.NBINS_FINE
    rng = np.random.default_rng(7 + fine)
    R0, R1 = float(det.radii[2]), float(det.radii[3])
    phi, z, pt, cot, cov = _seeds(rng, n, R0)
    sign, inside = np.where(rng.random(n) < 0.5, 1.0, -1.0), 1.0 - 10 ** rng.uniform(-4, -1, n)
    charge = torch.where(torch.rand(n, device="cuda") < 0.5, 1, -1).to(torch.int8)
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")

    def build(hits, seg_off, bin_off, fine_off):
        st = _state(phi, z, pt, cot, R0).astype(np.float32)
        out = kf.BuildResult(kf.Tracks(torch.empty((6, n), device="cuda"), torch.empty((21, n), device="cuda"), charge,
                                       torch.empty((3, n), device="cuda")),
                             torch.empty(n, device="cuda"), torch.empty(n, **i32), torch.empty(n, **i32),
                             torch.empty((1, n), **i32))
        bins = kf.HitBins(hits, bin_off, seg_off, n, 1, 3, fine_off)
        kf.kf_build(ctx, kf.Tracks(to_dev(st), to_dev(cov.astype(np.float32)), charge), off, bins, 1, out)
        torch.cuda.synchronize()
        return out

    def hits_at():
        """The hit of every seed: its prediction (a build over empty bins) plus the step to the cut."""
        o = build(torch.zeros((n, 4), device="cuda"), off, torch.zeros((n, nb + 1), **i32), None)
        p = (o.best.par[:3].double() + o.best.par_lo.double()).cpu().numpy()
        C = o.best.cov.double().cpu().numpy()
        S3 = np.array([[C[0], C[1], C[3]], [C[1], C[2], C[4]], [C[3], C[4], C[5]]]).transpose(2, 0, 1)
        S3 = S3 + np.diag([det.sigma_xy**2, det.sigma_xy**2, det.sigma_z**2])
        r = np.hypot(p[0], p[1])
        u = (np.stack([-p[1] / r, p[0] / r, 0 * r]) if along == "phi" else np.stack([0 * r, 0 * r, 1 + 0 * r])) * sign
        Su = np.einsum("nij,jn->in", S3, u)
        return p + Su * np.sqrt(CUT * inside / np.einsum("in,in->n", u, Su))

    # move every seed until its hit lies just beyond the next edge, seen from the prediction
    eps = rng.uniform(0, 1e-5, n) * sign
    for _ in range(3):
        h = hits_at()
        if along == "phi":
            width, at = 2 * np.pi / (2 * kf.BIN_PHI if fine else kf.BIN_PHI), np.arctan2(h[1], h[0])
            phi = phi + np.round((at + np.pi) / width) * width - np.pi + eps - at
        else:
            r, at = np.hypot(h[0], h[1]), np.arcsinh(h[2] / np.hypot(h[0], h[1]))
            z = z + r * np.sinh(np.round(at / ETA_ROW) * ETA_ROW + eps) - h[2]
    xyz = to_dev(hits_at().astype(np.float32))
    bins = kf.HitBins(torch.empty((n, 4), device="cuda"), torch.empty((n, nb + 1), **i32),
                      fine_off=torch.empty((n, nbf + 1), **i32) if fine else None)
    kf.kf_bin_hits(ctx, kf.LayerHits(xyz, off, n, 1, 3), bins)
    a = build(bins.hits, off, bins.bin_off, bins.fine_off)
    per = nbf if fine else nb  # every bin holds its event's hit
    one = torch.cat([xyz.T, torch.zeros((n, 1), device="cuda")], dim=1)
    b = build(one[:, None, :].expand(n, per, 4).reshape(-1, 4).contiguous(), off * per,
              torch.arange(0, per + 1, per // nb, **i32).expand(n, nb + 1).contiguous(),
              torch.arange(nbf + 1, **i32).expand(n, nbf + 1).contiguous() if fine else None)
    assert int(b.n_hits.sum()) > 0.9 * n  # nearly all are within the cut
    for x, y in ((a.n_hits, b.n_hits), (a.hit_idx, b.hit_idx), (a.chi2_tot, b.chi2_tot), (a.best.par, b.best.par),
                 (a.best.cov, b.best.cov), (a.status, b.status)):
        assert torch.equal(x, y)
