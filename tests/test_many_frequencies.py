"""More frequency bins than a warp has lanes: packets of every bin are sent."""
import numpy as np
import pytest

from paper_1311_0182_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _wl(n_freq, shared, cones):
    """A random box with n_freq source bins of a decade in cross-section, and recombination
    photons from the first step on."""
    wl = W.tiny(n=700, n_ngb=32, n_freq_src=n_freq, n_rc=cones, n_tc=cones, n_ec=cones, evolve_T=1,
                rec_shared_bin=shared)
    f = np.arange(n_freq)
    wl["sigma"] = 6.3e-18 * 10.0 ** (-f / n_freq)
    wl["eps"] = 1e-11 * (1.0 + f / n_freq)
    wl["src_ndot"] = np.full(n_freq, 1e48 / n_freq)
    return wl


@pytest.mark.parametrize("cones", [8, 32])
@pytest.mark.parametrize("n_freq,shared", [(31, 0), (32, 0), (33, 1), (64, 0)])
def test_bins_past_the_32nd_against_the_oracle(n_freq, shared, cones):
    """32, 33 and 65 bins: absorptions, state and sender counts on the FP64 path (the same
    arithmetic on both sides but for exp and pow: 1e-9, the bar of every FP64 state check), and
    the budget, to the bar of every FP64 budget check."""
    import oracle
    from paper_1311_0182_gb300 import rt
    wl = _wl(n_freq, shared, cones)
    g, o = rt.context_for(wl), oracle.Sim(wl)
    o.build_neighbours()
    for step in range(3):
        g.step(step, allow_subcycle_limit=True)
        o.step(step)
        ag, ao = g.deposits()[0], o.deposits()[0]
        assert np.allclose(ag, ao, rtol=1e-9, atol=1e-12 * ao.max())
        sg, so = g.state(), o.state()
        for k in ("x_HI", "T"):
            assert np.abs(sg[k] / so[k] - 1).max() < 1e-9, k
        b = g.budget()[0]
        assert abs(b[0] - b[1:].sum()) <= 1e-9 * b[0]
    assert (ao.sum(0) > 0).all()
    st = g.stats()
    assert st["senders"] <= st["hops"] * g.n


def test_bins_past_the_32nd_fp32_conserve_photons_and_step_alike():
    """The FP32 path at 34 bins: the budget closes, and graph and hop-by-hop steps give the same
    bits and the same counts."""
    from paper_1311_0182_gb300 import rt
    out = []
    for graph in (True, False):
        g = rt.context_for(_wl(33, 0, 32), transport_fp32=1)
        g.set_graph(graph)
        for step in range(3):
            g.step(step, allow_subcycle_limit=True)
        b = g.budget()[0]
        assert abs(b[0] - b[1:].sum()) <= 1e-6 * b[0]
        out.append((g.state(), g.stats()))
    assert all(np.array_equal(out[0][0][k], out[1][0][k]) for k in out[0][0])
    assert all(out[0][1][k] == out[1][1][k] for k in ("senders", "moving_packets", "gas_contrib"))


def test_cone_masks_of_bins_past_the_32nd():
    """Every held packet of 40 bins has its mask against the oracle's."""
    import oracle
    from paper_1311_0182_gb300 import rt
    wl = _wl(39, 0, 8)
    g, o = rt.context_for(wl), oracle.Sim(wl)
    o.build_neighbours()
    rng = np.random.default_rng(5)
    d = rng.normal(size=(3, g.n, g.S))
    d /= np.linalg.norm(d, axis=0)
    f = np.zeros((6, g.n, g.S))
    f[0] = np.where(rng.random((g.n, g.S)) < 0.3, 1e45, 0.0)
    f[1:4] = f[0] * d
    g.set_slots(f)
    o.set_slots(f)
    g.assign_cones(0)
    o.rotate(0)
    assert np.array_equal(g.cone_masks(), o.cone_masks())
