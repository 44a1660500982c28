"""The variance of a spectrum (float32 sums with their rounding errors kept, FP64
for values whose squares leave their range) against FP64 numpy: ordinary, large, tiny and mixed values, an
infinity and a NaN, on scans of one and of several rows per warp.

Bound: the reference's own sum of about 1e5 FP64 terms, 1e-12 relative.

Then against the exact sum, where the bound is the number of FP64 roundings on
the way from a lane's total to the result: 3 in the lane, 5 + 7 in the block,
5 + 7 over the blocks and the division, 28 of 2^-53 (and what FP64 leaves of the
lane's smaller sums, far below one).  Equal values are the hard
case: their float32 roundings all go the same way.
"""

import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def P():
    import paper_2104_06336_gb300 as P
    P.build()
    P.load()
    return P


@pytest.mark.parametrize("scan", [(2, 4), (30, 34), (512, 64)])
@pytest.mark.parametrize("kind", ["ordinary", "large", "tiny", "mixed", "inf", "nan"])
def test_variance_of_spectrum(P, scan, kind):
    ny, nx = scan
    rec = P.Reconstructor(synth.geometry(synth.workload(1, scan_ny=ny, scan_nx=nx)), n_cand=3)
    r = np.random.default_rng(7)
    H = (r.normal(size=(3, ny, nx // 2 + 1, 2)) * 1e3).astype(np.float32)
    mag = {"ordinary": 1.0, "large": 1e16, "tiny": 1e-25}.get(kind, 1.0)
    if kind == "mixed":
        H = (H * 10.0 ** r.uniform(-30, 14, size=H.shape)).astype(np.float32)
    H = (H * np.float32(mag)).astype(np.float32)
    H[:, :, :1, 1] = 0.0
    if kind in ("inf", "nan"):
        H[1, ny // 2, 1, 0] = np.inf if kind == "inf" else np.nan
    g0 = torch.tensor([1.0, 1.0], dtype=torch.float64, device="cuda")
    _, var = rec.image_from_spectrum(torch.view_as_complex(torch.from_numpy(H).cuda()), g0, phase=False)
    w = np.full(nx // 2 + 1, 2.0)
    w[0] = w[-1] = 1.0
    ref = (w * (H.astype(np.float64) ** 2).sum(-1)).sum((1, 2)) / (ny * nx) ** 2
    got = var.cpu().numpy()
    fine = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    assert np.all(np.abs(got[fine] - ref[fine]) <= 1e-12 * ref[fine]), (got, ref)


@pytest.mark.parametrize("scan,n", [((32, 32), 1), ((100, 150), 3), ((512, 512), 1), ((512, 512), 12)])
@pytest.mark.parametrize("kind", ["normal", "decay", "equal"])
def test_variance_to_the_last_bits_of_fp64(P, scan, n, kind):
    ny, nx = scan
    rec = P.Reconstructor(synth.geometry(synth.workload(1, scan_ny=ny, scan_nx=nx)), n_cand=n)
    r = np.random.default_rng(3)
    H = r.normal(size=(n, ny, nx // 2 + 1, 2)).astype(np.float32)
    if kind == "equal":
        H[:] = np.array([1.2345678, 0.3456789], dtype=np.float32)
    elif kind == "decay":
        H *= np.exp(-6.0 * r.random(size=H.shape[:3] + (1,))).astype(np.float32)
    g0 = torch.tensor([1.0, 1.0], dtype=torch.float64, device="cuda")
    _, var = rec.image_from_spectrum(torch.view_as_complex(torch.from_numpy(H).cuda()), g0, phase=False)
    w = np.full(nx // 2 + 1, 2.0)
    w[0] = w[-1] = 1.0
    for i in (0, n - 1):
        terms = w[None, :, None] * H[i].astype(np.float64) ** 2  # exact: squares of 24 bits
        ref = math.fsum(terms.reshape(-1).tolist()) / float(ny * nx) ** 2
        assert abs(float(var[i]) - ref) <= 28 * 2.0 ** -53 * ref, (i, float(var[i]), ref)
