"""Which receiver groups share a warp changes nothing.  The receiver side takes the work list in
fours from its start, so boxes laid before a box shift its groups against the fours; a box stepped
alone and behind others gives the same bits."""
import numpy as np
import pytest

from paper_1311_0182_gb300 import distributed as D
from paper_1311_0182_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TARGET = 4


def _batch(cones, shared, clock_limited, fp32):
    """Five boxes of odd sizes; two source bins (three frequencies, or two with a shared bin).  The
    source of the last box lies in a tight clump, so that its receivers run from one contribution to
    more than a warp takes at once and from a few edges to more than 64; with clock-limited steps
    packets wait in it."""
    dt = (0.004 if clock_limited else 0.1) * W.MYR
    wl = W.cfg4(n_boxes=5, n_min=150, n_max=400, n_rc=cones, n_tc=cones, n_ec=cones, n_freq_src=2,
                rec_shared_bin=shared, dt=dt, dt_em=dt, transport_fp32=fp32, cell_occupancy=2)
    wl["sigma"], wl["eps"] = np.array([6.3e-18, 1.6e-18]), np.array([1e-12, 1e-11])
    wl["src_ndot"] = np.repeat(wl["src_ndot"], 2) * 0.5
    lo = int(wl["box_off"][TARGET])
    rng = np.random.default_rng(cones)
    for k in ("x", "y", "z"):
        wl[k][lo:lo + 28] = float(wl["box_L"][0]) * (0.5 + rng.uniform(-0.01, 0.01, 28))
    wl["x_HI"][:] = 0.05
    return wl


@pytest.mark.parametrize("clock_limited", [False, True])
@pytest.mark.parametrize("barrier", [False, True])
@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("cones", [8, 32])
def test_groups_give_the_same_bits_whatever_they_share_a_warp_with(cones, shared, barrier,
                                                                   clock_limited):
    from paper_1311_0182_gb300 import rt
    for fp32 in (0, 1):
        wl = _batch(cones, shared, clock_limited, fp32)
        L = float(wl["box_L"][0])
        out = []
        for part in ([4], [0, 4], [1, 4], [2, 3, 4], [0, 1, 2, 3, 4]):
            sub = D.local_workload(wl, np.array(part))
            g = rt.context_for(sub)
            if barrier:
                g.set_barrier(len(part) - 1, 0, [0.55 * L, 0.5 * L, 0.5 * L], 0.2 * L)
            for step in range(3):
                g.step(step, allow_subcycle_limit=True)
            lo = int(sub["box_off"][-2])
            s, f, d = g.state(), g.slots(), g.deposits()
            out.append([s[k][lo:] for k in sorted(s)] + [f[:, lo:], g.budget()[-1]] +
                       [x[lo:] for x in d])
            st = g.stats()
            g.close()
        assert st["receiver_groups"] > 0 and st["staged_contrib"] > 0
        if clock_limited:
            assert out[0][-4][3] > 0          # packets in flight
        for o in out[1:]:
            assert all(np.array_equal(a, b) for a, b in zip(o, out[0]))
