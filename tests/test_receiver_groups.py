"""The receiver side's group batches at their edges: few and many contributions a group, more
than 64 reverse edges, waiting packets, both cone counts.  FP64 against the oracle, FP32 by its
photon budget and by repeating its bits."""
import numpy as np
import pytest

from paper_1311_0182_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _clustered(cones, clock_limited):
    """A tight clump of 28 particles among 172 others: its particles are neighbours of more than
    64 others, so their reverse lists take more than one block of edges."""
    dt = (0.0005 if clock_limited else 0.05) * W.MYR
    wl = W.tiny(n=200, n_ngb=32, n_rc=cones, n_tc=cones, n_ec=cones, dt=dt, dt_em=dt, evolve_T=1)
    rng = np.random.default_rng(3)
    L = float(wl["box_L"][0])
    for k in ("x", "y", "z"):
        wl[k][:28] = L * (0.5 + rng.uniform(-0.01, 0.01, 28))
    wl["x_HI"][:] = 0.05
    return wl


@pytest.mark.parametrize("clock_limited", [False, True])
@pytest.mark.parametrize("cones", [8, 32])
def test_groups_against_the_oracle(cones, clock_limited):
    import oracle
    from paper_1311_0182_gb300 import rt
    wl = _clustered(cones, clock_limited)
    g, o = rt.context_for(wl), oracle.Sim(wl)
    o.build_neighbours()
    assert np.bincount(o.neighbours()[0].ravel()).max() > 64
    for step in range(3):
        g.step(step, allow_subcycle_limit=True)
        o.step(step)
        # the transport is the same arithmetic on both sides; only the chemistry's exp and pow
        # round differently (1e-9 is the bar of every FP64 state check)
        sg, so = g.state(), o.state()
        for k in ("x_HI", "T"):
            assert np.abs(sg[k] / so[k] - 1).max() < 1e-9, k
    if clock_limited:
        assert g.budget()[0, 3] > 0      # packets wait at the end of the step


@pytest.mark.parametrize("clock_limited", [False, True])
@pytest.mark.parametrize("cones", [8, 32])
def test_groups_fp32_conserve_photons_and_repeat(cones, clock_limited):
    from paper_1311_0182_gb300 import rt
    out = []
    for occ in (1, 4):
        wl = _clustered(cones, clock_limited)
        g = rt.context_for(wl, transport_fp32=1, cell_occupancy=occ)
        for step in range(3):
            g.step(step, allow_subcycle_limit=True)
        b = g.budget()[0]
        assert abs(b[0] - b[1] - b[2] - b[3]) <= 1e-6 * b[0]
        out.append(g.state())
    for k in ("x_HI", "T", "N_rec"):
        assert np.array_equal(out[0][k], out[1][k]), k
