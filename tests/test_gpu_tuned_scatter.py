"""The autotuner's largest scatter shape is the built-in one: its timed range
ends at three blocks per SM, where the kernel may fit more.  Launches of the
two are timed in turn, the shortest of 20 each: the same launch, so within 5 %
(three blocks instead of four took 12 % longer on these events).
"""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def test_three_blocks_mean_all_that_fit():
    import paper_2104_06336_gb300 as P
    P.build()
    P.load()
    w = synth.workload(5, scan_ny=1024, scan_nx=1024)
    g = synth.geometry(w)
    F = 1 << 20
    rec = P.Reconstructor(g)
    off = torch.arange(F + 1, dtype=torch.int64, device="cuda") * 50
    xy = torch.rand(2, 50 * F, device="cuda") * 0.6 + 0.2  # mostly kept pixels
    idx = (xy[0] * g["det_h"]).int() * g["det_w"] + (xy[1] * g["det_w"]).int()
    ev = [[torch.cuda.Event(enable_timing=True) for _ in P._lib.STAGES] for _ in range(2)]
    for e in ev[0] + ev[1]:
        e.record()
    P.eer4d_set_stage_events(rec.plan, *ev)
    at = P._lib.STAGES.index("scatter")
    base = dict(P.eer4d_get_tuning(rec.plan), scatter_tf=64)
    best = {0: 1e9, 3: 1e9}
    for _ in range(20):
        for cps in best:
            P.eer4d_set_tuning(rec.plan, dict(base, scatter_ctas_per_sm=cps))
            rec.accumulate(idx, off)
            torch.cuda.synchronize()
            best[cps] = min(best[cps], ev[0][at].elapsed_time(ev[1][at]))
    assert best[3] <= 1.05 * best[0], best
    assert rec.check() == 0
