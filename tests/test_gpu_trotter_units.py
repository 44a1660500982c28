"""The trotter kernel's ways of taking a warp task, where they can go wrong:
whole or in segments, from the plan's lists or by the set tests, ragged and
Nyquist bins, both normalisations, G without 16-byte alignment.

Bounds: a phase is a sum of float32 terms, so two orders of summation differ
by a few times 1e-7 relative L2 (1e-6 allowed); against the FP64 oracle the
1e-5 of the other parity tests.
"""

import numpy as np
import pytest
import torch

import oracle as orc
import synth

pytestmark = pytest.mark.gpu

THETA = (70.0, -20.0, 15.0, 6.0e3, 0.0)


@pytest.fixture(scope="module", autouse=True)
def P():
    import paper_2104_06336_gb300 as P
    P.build()
    P.load()
    return P


def rel_l2(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _rec(P, ny, nx, norm=0, n_cand=1, cfg=1):
    w = synth.workload(cfg, scan_ny=ny, scan_nx=nx, e_per_frame=30.0)
    d = synth.generate(w, "cuda")
    rec = P.Reconstructor(synth.geometry(w), norm=norm, n_cand=n_cand)
    rec.load(d.idx, d.off)
    return w, d, rec


# one warp per column (2..32 rows), a ragged second warp, Nyquist bins inside
# and at the edge of a warp, the segment rule's largest and smaller splits
@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("scan", [(2, 4), (6, 2), (30, 34), (32, 32), (34, 30), (64, 16), (62, 66)])
def test_lists_set_tests_and_oracle_agree(P, scan, norm):
    w, d, rec = _rec(P, *scan, norm=norm)
    ph, var = rec.reconstruct(torch.tensor(THETA))
    # s = 1e-30: the same K' and the same sets, but the lists (rotation 0) do not apply
    ph_t, _ = rec.reconstruct(torch.tensor(THETA[:4] + (1e-30,), dtype=torch.float64))
    assert rel_l2(ph_t[0].cpu(), ph[0].cpu()) <= 1e-6
    geom = synth.geometry(w)
    G = orc.g_function(orc.densify(*d.numpy(), geom), geom)
    phi, V = orc.ssb_phase(G, geom, THETA, "area" if norm else "none")
    assert rel_l2(ph[0].cpu(), phi) <= 1e-5
    assert abs(float(var[0]) - V) <= 1e-5 * V
    Vg, g, _ = rec.variance_grad(torch.tensor(THETA))
    _, gr, _ = orc.ssb_value_and_grad_var(G, geom, THETA, "area" if norm else "none")
    scales = np.array([100.0, 50.0, 50.0, 1.0e4, 0.1])
    assert abs(float(Vg) - V) <= 1e-5 * V
    assert np.all(np.abs(g.cpu().numpy() - gr) * scales <= 1e-4 * np.max(np.abs(gr) * scales))
    assert rec.check() == 0


@pytest.mark.parametrize("scan,n", [((32, 32), 3), ((128, 128), 9), ((256, 256), 32)])
def test_whole_tasks_equal_segments_bit_for_bit(P, scan, n):
    """One candidate takes its tasks in segments; 32 candidates at 256x256
    take them whole (4 passes x 1032 tasks), 9 at 128x128 and 3 at 32x32 do
    not.  Same order of summation: the same bits."""
    _, _, rec = _rec(P, *scan, n_cand=n)
    cands = torch.zeros(n, 5, dtype=torch.float64)
    cands[:, 0] = torch.linspace(-150.0, 150.0, n)
    cands[:, 3] = 4.0e3
    ph, var = rec.reconstruct(cands)
    for i in (0, n // 2, n - 1):
        p1, v1 = rec.reconstruct(cands[i])
        assert torch.equal(p1[0], ph[i]), i
        assert abs(float(v1[0]) - float(var[i])) <= 1e-12 * float(v1[0])


def test_unaligned_spectrum_equals_aligned(P):
    """G at an 8-byte offset takes the 8-byte copies: the same values."""
    _, _, rec = _rec(P, 48, 64, cfg=2)
    ab = torch.tensor(THETA, dtype=torch.float64, device="cuda")
    ph, _ = rec.reconstruct(ab)
    buf = torch.empty(rec.G.numel() + 2, device="cuda")
    G = buf[2:]
    G.copy_(rec.G)
    assert G.data_ptr() % 16 == 8
    out = torch.empty_like(ph)
    P.ssb_reconstruct(rec.plan, G, ab, rec.scratch, out, None, status=rec.status)
    assert torch.equal(out, ph)
    assert rec.check() == 0
