"""Receivers of many staged contributions: a source cluster within one smoothing length sends a
packet of each source and cone to the same few neighbours."""
import numpy as np
import pytest

from paper_1311_0182_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cluster(wl, n_src, ndot):
    rng = np.random.default_rng(n_src)
    L = float(wl["box_L"][0])
    wl["src_box"] = np.zeros(n_src, np.int32)
    for k in ("src_x", "src_y", "src_z"):
        wl[k] = L * (0.5 + rng.uniform(-1e-3, 1e-3, n_src))
    wl["src_ndot"] = ndot * rng.uniform(0.5, 1.5, n_src) / n_src
    return wl


@pytest.mark.parametrize("cones", [8, 32])
@pytest.mark.parametrize("n_src", [1, 7, 8, 9, 31, 33, 64, 65, 130, 1025])
def test_segments_of_every_length(n_src, cones):
    """A neighbour of the cluster receives about one packet a source, so the segments run from one
    contribution over the edges of eight and 32 to many merge passes.  FP64 against the oracle
    (1e-9, the bar of every FP64 state check: a contribution lost or taken twice moves the state by
    the share of a packet); the same bits on both precisions for launch sizes that stage in another
    order."""
    import oracle
    from paper_1311_0182_gb300 import rt
    for fp32 in (0, 1):
        out = []
        for grid in ((0, 0, 0), (1, 1, 1), (7, 3, 40)):
            wl = _cluster(W.tiny(n=400, n_ngb=32, n_rc=cones, n_tc=cones, n_ec=cones, evolve_T=1,
                                 transport_fp32=fp32), n_src, 1e49)
            g = rt.context_for(wl, launch_grid=grid)
            for step in range(2):
                g.step(step, allow_subcycle_limit=True)
            b = g.budget()[0]
            assert abs(b[0] - b[1:].sum()) <= (1e-6 if fp32 else 1e-9) * b[0]
            out.append((g.state(), g.slots()))
            g.close()
        for s, f in out[1:]:
            assert all(np.array_equal(s[k], out[0][0][k]) for k in s)
            assert np.array_equal(f, out[0][1])
        if not fp32:
            o = oracle.Sim(wl)
            o.build_neighbours()
            for step in range(2):
                o.step(step)
            so = o.state()
            for k in ("x_HI", "T"):
                assert np.abs(out[0][0][k] / so[k] - 1).max() < 1e-9, k


def test_cost_of_a_source_cluster_is_not_quadratic():
    """Four times the sources of a cluster cost a step less than eight times as much: linear work
    would be four, comparing all pairs of a receiver's contributions sixteen."""
    import torch
    from paper_1311_0182_gb300 import rt
    ms = []
    for n_src in (4096, 16384):
        wl = _cluster(W.cfg1(24, transport_fp32=1), n_src, 5e48)
        wl["x_HI"][:] = 1e-3
        g = rt.context_for(wl)
        t = []
        for step in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            g.step(step, allow_subcycle_limit=True)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        ms.append(min(t[1:]))
        g.close()
    assert ms[1] < 8.0 * ms[0], ms
