"""A workspace serves every call that asks for less than it was sized for: the
scratch of n candidates, calls with 1 .. n of them.  Tasks of few candidates
are split over warps, whose partial sums take memory that many candidates do
not need, so the largest need is not that of the largest call.
"""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

GUARD = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def P():
    import paper_2104_06336_gb300 as P
    P.build()
    P.load()
    return P


def _geometry(ny, nx):
    return synth.geometry(synth.workload(2, scan_ny=ny, scan_nx=nx))


def _guarded(nbytes):
    """A buffer of nbytes and the guard bytes behind it."""
    buf = torch.full((nbytes + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    return buf[:nbytes], buf[nbytes:]


@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("scan", [(2, 4), (32, 32), (128, 128), (128, 512), (256, 256), (336, 200), (1024, 512)])
def test_scratch_never_shrinks(P, scan, norm):
    plan = P.Plan(_geometry(*scan), norm=norm)
    n = list(range(1, 131)) + [255, 256, 257, 1023, 1024]
    size = [plan.workspace_bytes(i)[2] for i in n]
    assert all(a <= b for a, b in zip(size, size[1:]))


@pytest.mark.parametrize("scan,sized", [((256, 256), 64), ((128, 128), 121)])
def test_fewer_candidates_than_sized_for(P, scan, sized):
    w = synth.workload(2, scan_ny=scan[0], scan_nx=scan[1], e_per_frame=10.0)
    d = synth.generate(w, "cuda")
    rec = P.Reconstructor(synth.geometry(w))
    rec.load(d.idx, d.off)
    plan = rec.plan
    need = plan.workspace_bytes(sized)[2]
    cands = torch.zeros(sized, 5, dtype=torch.float64, device="cuda")
    cands[:, 0] = torch.linspace(-150.0, 150.0, sized)
    one = [rec.reconstruct(cands[i])[0][0].clone() for i in (0, 6, sized - 1)]
    scratch, guard = _guarded(need)
    for n in (1, 2, 7, 8, 16, 24, 25, 120, sized):
        if n > sized:
            continue
        assert plan.workspace_bytes(n)[2] <= need  # before anything is written
        ab = cands[-n:] if n == 1 else cands[:n].contiguous()
        ph = torch.empty(n, *scan, device="cuda")
        var = torch.empty(n, dtype=torch.float64, device="cuda")
        P.ssb_reconstruct(plan, rec.G, ab, scratch, ph, var, status=rec.status)
        H = torch.empty(n, scan[0], rec.info["nkx"], dtype=torch.complex64, device="cuda")
        g0 = torch.empty(2, dtype=torch.float64, device="cuda")
        P.ssb_spectrum_partial(plan, rec.G, ab, scratch, H, g0, status=rec.status)
        img = torch.empty_like(ph)
        P.ssb_image_from_spectrum(plan, H, g0, n, scratch, img, var)
        assert bool((guard == 0xA5).all()), n
        if n == 1:
            assert torch.equal(ph[0], one[2])
        else:
            assert torch.equal(ph[0], one[0]), n
            assert n < 7 or torch.equal(ph[6], one[1]), n
            assert n < sized or torch.equal(ph[-1], one[2]), n
        assert float((img - ph).norm() / ph.norm()) <= 1e-6
    # the same through the Reconstructor, which sizes its scratch once
    rec = P.Reconstructor(synth.geometry(w), n_cand=sized)
    rec.load(d.idx, d.off)
    for n in (16, 24):
        assert torch.equal(rec.reconstruct(cands[:n])[0][0], one[0])
        assert P.refocus.sweep(rec, cands[:n]).shape == (n,)
    assert rec.check() == 0


def test_batched_scratch_serves_any_of_its_datasets(P):
    """Sizes over nested lists (uneven sides, both norms, every order), then 16
    scans of 256x256 whose scratch is given to seven and to one of them."""
    sides = [(256, 256), (32, 32), (512, 512), (64, 96), (2, 4), (300, 100), (1024, 64), (256, 256)]
    plans = [P.Plan(_geometry(*s), norm=int(i == 3)) for i, s in enumerate(sides)] * 2
    for drop in range(len(plans)):
        size = [P.batched_scratch_bytes(plans[drop:drop + k]) for k in range(1, len(plans) - drop + 1)]
        assert all(a <= b for a, b in zip(size, size[1:])), drop
        rest = plans[:drop] + plans[drop + 1:]
        assert P.batched_scratch_bytes(rest) <= P.batched_scratch_bytes(plans), drop
        assert P.batched_scratch_bytes(rest[::-1]) == P.batched_scratch_bytes(rest)

    w = synth.workload(2, scan_ny=256, scan_nx=256, e_per_frame=5.0)
    d = synth.generate(w, "cuda")
    rec = P.Reconstructor(synth.geometry(w))
    rec.load(d.idx, d.off)
    recs = [rec] * 16
    need = P.batched_scratch_bytes([r.plan for r in recs])
    ab = torch.zeros(16, 5, dtype=torch.float64, device="cuda")
    ab[:, 0] = torch.linspace(-100.0, 100.0, 16)
    scratch, guard = _guarded(need)
    for n in (16, 8, 7, 1):
        assert P.batched_scratch_bytes([r.plan for r in recs[:n]]) <= need
        ph, _ = P.reconstruct_batched(recs[:n], ab[:n], scratch=scratch)
        assert bool((guard == 0xA5).all()), n
        for i in {0, n - 1}:
            assert torch.equal(ph[i], rec.reconstruct(ab[i])[0][0]), (n, i)
    assert rec.check() == 0
