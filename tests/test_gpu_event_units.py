"""Event kernels at the edges of their splits, whole numbers against the oracle:
run-length decoding (frame lengths about the 128-event chunk, frames per warp,
addresses off the 16-byte grid, sums out of range in the middle of frames), the
scatter (byte and 16-bit tiles side by side, frames per task, rows that do not
start on 16 bytes, several pixel chunks, windows cut by the detector's edge,
streamed ranges that start inside a tile) and the virtual detectors' counts.
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


def offsets(n):
    return np.concatenate([[0], np.cumsum(n)]).astype(np.int64)


def sums64(runs, off):
    """Running sums of each frame in 64 bits."""
    s = np.cumsum(runs.astype(np.uint64), dtype=np.uint64)
    first = np.repeat(off[:-1], np.diff(off))
    return s - np.where(first > 0, s[np.maximum(first, 1) - 1], 0).astype(np.uint64)


@pytest.mark.parametrize("shift", [(0, 0), (1, 1), (3, 3), (2, 1)])
@pytest.mark.parametrize("lengths", ["edges", "one", "long", "many"])
def test_rle_decode_units(P, lengths, shift):
    rng = np.random.default_rng(7)
    n = {"edges": np.array([0, 0, 1, 127, 128, 129, 0, 3, 4, 5, 255, 256, 257, 0, 1, 1, 1, 0]),
         "one": np.array([0, 3000, 0]),
         "long": rng.integers(0, 5000, 300),
         "many": rng.integers(0, 60, 240001)}[lengths]
    off = offsets(n)
    C = int(off[-1])
    runs = rng.integers(0, 700, C).astype(np.uint32)
    if lengths != "many":  # sums past 2^32: at a frame's end, in its middle, twice
        for k in rng.integers(0, C, 12):
            runs[k] = rng.integers(1 << 31, (1 << 32) - 1)
    ref = sums64(runs, off)
    big = ref > 0xFFFFFFFF
    ref = np.where(big, 0xFFFFFFFF, ref).astype(np.uint32)
    buf = torch.zeros(C + 4, dtype=torch.int32, device="cuda")
    out = torch.full((C + 4,), -7, dtype=torch.int32, device="cuda")
    src, dst = buf[shift[0]:shift[0] + C], out[shift[1]:shift[1] + C]
    src.copy_(torch.from_numpy(runs.view(np.int32)))
    st = torch.zeros(4, dtype=torch.int32, device="cuda")
    P.eer_decode_rle(src, torch.from_numpy(off).cuda(), idx=dst, status=st)
    np.testing.assert_array_equal(dst.cpu().numpy().view(np.uint32), ref)
    assert (P.status_code(st) != 0) == bool(big.any())
    o = out.cpu().numpy()
    assert (o[:shift[1]] == -7).all() and (o[shift[1] + C:] == -7).all()
    P.eer_decode_rle(src, torch.from_numpy(off).cuda(), idx=src, status=st)
    np.testing.assert_array_equal(src.cpu().numpy().view(np.uint32), ref)


def scan_events(geom, F, rng, heavy=()):
    """Events of F frames, most within the window; those of `heavy` exceed 255,
    several of them on the same pixel."""
    n = rng.integers(0, 90, F)
    n[rng.integers(0, F, F // 8)] = 0
    n[list(heavy)] = rng.integers(256, 3000, len(heavy))
    off = offsets(n)
    C = int(off[-1])
    idx = rng.integers(0, geom["det_w"] * geom["det_h"], C).astype(np.int64)
    for f in heavy:
        idx[off[f]:off[f] + 300] = idx[off[f]]
    return idx.astype(np.uint32).view(np.int32), off


GEOMS = {
    "disk": dict(),
    "edge": dict(crop_x0=-37, crop_y0=-20),
    "right": dict(crop_x0=300, crop_y0=350, bin=5),
    "large": dict(crop_px=48.0),
}


@pytest.mark.parametrize("geom", list(GEOMS))
@pytest.mark.parametrize("scan", [(6, 6), (10, 10), (16, 24), (34, 30)])
@pytest.mark.parametrize("tf", [0, 4, 8, 32, 128])
def test_scatter_units(P, geom, scan, tf):
    rng = np.random.default_rng(3)
    g = dict(synth.geometry(synth.workload(5, scan_ny=scan[0], scan_nx=scan[1])), **GEOMS[geom])
    F = scan[0] * scan[1]
    rec = P.Reconstructor(g)
    if tf:
        P.eer4d_set_tuning(rec.plan, dict(P.eer4d_get_tuning(rec.plan), scatter_tf=tf))
    idx, off = scan_events(g, F, rng, heavy=(1, F // 2 + 1))
    ref = orc.densify(idx.view(np.uint32), off, g)
    Pn, P_pad = rec.info["P"], rec.info["P_pad"]
    ti, to = torch.from_numpy(idx).cuda(), torch.from_numpy(off).cuda()
    for chunk in (None, F // 3 + 1):
        rec.counts.fill_(float("nan"))
        rec.load(ti, to, chunk_frames=chunk)
        got = rec.counts.reshape(P_pad, -1)
        np.testing.assert_array_equal(got[:Pn].float().cpu().numpy(), ref)
        assert not got[Pn:].any()
        assert rec.check() == 0
    sx, sy, sn = orc.com_sums(idx.view(np.uint32), off, g["det_w"], g["det_h"])
    sums = torch.empty(3, F, dtype=torch.int64, device="cuda")
    rec.totals.zero_()
    P.ssb_accumulate_com(rec.plan, ti, to, 0, rec.work, rec.G, True, sums, rec.totals, status=rec.status)
    np.testing.assert_array_equal(sums.cpu().numpy(), np.stack([sx, sy, sn]).reshape(3, F))
    np.testing.assert_array_equal(rec.totals.cpu().numpy(), [sx.sum(), sy.sum(), sn.sum()])
    np.testing.assert_array_equal(rec.counts.reshape(P_pad, -1)[:Pn].float().cpu().numpy(), ref)


@pytest.mark.parametrize("scan", [(2, 2), (10, 10), (34, 30)])
def test_ring_counts_units(P, scan):
    rng = np.random.default_rng(9)
    g = synth.geometry(synth.workload(5, scan_ny=scan[0], scan_nx=scan[1]))
    F = scan[0] * scan[1]
    rec = P.Reconstructor(g, alloc_counts=False)
    idx, off = scan_events(g, F, rng, heavy=(1, F // 2 + 1))
    radii = [0.0, 40.0, 97.5, 200.0]
    c = (g["det_w"] / 2 + 0.25, g["det_h"] / 2 - 3.5)
    got = rec.virtual_detectors(torch.from_numpy(idx).cuda(), torch.from_numpy(off).cuda(), radii,
                                use_totals=False, cx=c[0], cy=c[1])
    ref = orc.virtual_detector_counts(idx.view(np.uint32), off, g["det_w"], g["det_h"], radii, *c)
    np.testing.assert_array_equal(got.cpu().numpy().reshape(len(radii) - 1, F), ref)
    assert rec.check() == 0


@pytest.mark.parametrize("n", [1, 2, 31, 63, 64])
def test_ring_search(P, n):
    """The edges below a pixel, for odd and even numbers of them: equal edges
    (empty rings), the first at 0 and above it, the last past the detector and
    at infinity, edges on whole squared radii and between."""
    rng = np.random.default_rng(n)
    g = synth.geometry(synth.workload(5, scan_ny=10, scan_nx=10))
    F = 100
    rec = P.Reconstructor(g, alloc_counts=False)
    idx, off = scan_events(g, F, rng)
    ti, to = torch.from_numpy(idx).cuda(), torch.from_numpy(off).cuda()
    for last, first in ((250.0, 0.0), (5000.0, 3.5), (float("inf"), 0.0)):
        radii = np.sort(rng.uniform(0.0, 300.0, n + 1))
        radii[::3] = np.round(radii[::3])
        radii[1::4] = radii[:-1:4][:radii[1::4].size]
        radii = np.sort(radii)
        radii[0], radii[-1] = min(first, radii[0]), max(last, radii[-1])
        got = rec.virtual_detectors(ti, to, list(radii), use_totals=False, cx=287.0, cy=290.5)
        ref = orc.virtual_detector_counts(idx.view(np.uint32), off, g["det_w"], g["det_h"], list(radii), 287.0, 290.5)
        np.testing.assert_array_equal(got.cpu().numpy().reshape(n, F), ref)
    assert rec.check() == 0
