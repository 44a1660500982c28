"""The shared-memory transform (scan sides that are no power of two) against
numpy in 64 bits: every radix it has a butterfly for, primes from 11 up first,
repeated and after one another, and tiles of scan rows that do not come out
even.

Bound: each of at most four stages of float32 butterflies rounds a value a few
times; G within 2e-6 of max|G| as for the other forms of the scan DFT, the
images within 1e-5 relative L2.
"""

import numpy as np
import pytest
import torch

import oracle as orc
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def P():
    import paper_2104_06336_gb300 as P
    P.build()
    P.load()
    return P


# sides and their stages: 6, 10, 12, 14, 18, 20, 22 = 11.2, 24, 26 = 13.2, 30 = 6.5, 36 = 6.6, 42 = 7.6, 44 = 11.4,
# 50 = 10.5, 54 = 9.6, 98 = 14.7, 112 = 14.8, 242 = 11.11.2, 286 = 11.13.2, 324 = 18.18, 336 = 21.16, 400 = 20.20,
# 480 = 24.20, 504 = 24.21
@pytest.mark.parametrize("scan", [(6, 10), (12, 14), (18, 20), (22, 24), (26, 30), (36, 42), (44, 50), (54, 98),
                                  (112, 6), (242, 2), (4, 286), (480, 16), (16, 480), (38, 64), (64, 46), (324, 4),
                                  (6, 336), (400, 2), (4, 504)])
def test_lengths_match_oracle(P, scan):
    w = synth.workload(5, scan_ny=scan[0], scan_nx=scan[1], e_per_frame=20.0)
    d = synth.generate(w, "cuda")
    geom = synth.geometry(w)
    rec = P.Reconstructor(geom)
    rec.load(d.idx, d.off)
    idx, off = d.numpy()
    G = orc.g_function(orc.densify(idx, off, geom), geom)
    nkx = scan[1] // 2 + 1
    got = rec.G_complex().cpu().numpy()[:, :rec.info["P"]].transpose(1, 2, 0)
    assert np.abs(got - G[:, :, :nkx]).max() <= 2e-6 * np.abs(G).max()
    th = (60.0, 10.0, -20.0, 3.0e3, 0.1)
    ph, _ = rec.reconstruct(torch.tensor(th))
    phi, V = orc.ssb_phase(G, geom, th)
    assert np.linalg.norm(ph[0].cpu().numpy() - phi) <= 1e-5 * np.linalg.norm(phi)
    _, com, dpc = rec.com_dpc(d.idx, d.off)
    sx, sy, n = orc.com_sums(idx, off, w.det_w, w.det_h)
    ref = orc.idpc(*orc.com_maps(sx, sy, n, *orc.pacbed_centre(sx, sy, n)), geom)
    assert np.linalg.norm(dpc.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
    u = np.random.default_rng(3).normal(size=scan).astype(np.float32)
    g = rec.grad(torch.tensor(th, dtype=torch.float64), torch.from_numpy(u).cuda()).cpu().numpy()
    gr = orc.ssb_grad(G, geom, th, u.astype(np.float64))
    scales = np.array([100.0, 50.0, 50.0, 1.0e4, 0.1])
    assert np.all(np.abs(g - gr) * scales <= 1e-4 * np.max(np.abs(gr) * scales))
    assert rec.check() == 0
