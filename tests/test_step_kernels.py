"""Kernels of a step at the sizes where they can go wrong: the chemistry's queue (fewer particles
than lanes, ragged counts), the budget's per-box sums with gated sources, the order
in which requests and staged contributions arrive."""
import numpy as np
import pytest

from paper_1311_0182_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("n", [33, 34, 127, 1025, 4099])
def test_chemistry_queue_against_the_oracle(n, fp32):
    """A dark, cooling region (no photons move): every particle's subcycles, whichever lane
    takes it.  FP64 to the bar of every FP64 state check; with FP32 rate fits, whose relative
    error is ~1e-6, over at most ~100 subcycles of a 10% change each."""
    import oracle
    from paper_1311_0182_gb300 import rt
    rng = np.random.default_rng(n)
    wl = W.tiny(n=n, n_ngb=32, evolve_T=1, rec_mode=W.REC_OTS_CASE_B, dt=2.0 * W.MYR, dt_em=2.0 * W.MYR)
    wl["n_H"] = 1e-2 * np.exp(rng.normal(0.0, 1.0, n))
    wl["x_HI"] = np.exp(rng.uniform(np.log(1e-4), 0.0, n))
    wl["T"] = np.exp(rng.uniform(np.log(3e3), np.log(6e4), n))
    wl["src_ndot"] = np.zeros_like(wl["src_ndot"])
    g, o = rt.context_for(wl, transport_fp32=fp32), oracle.Sim(wl)
    o.build_neighbours()
    g.step(0, allow_subcycle_limit=True)
    o.step(0)
    sg, so = g.state(), o.state()
    tol = 1e-4 if fp32 else 1e-9
    for k in ("x_HI", "T"):
        assert np.abs(sg[k] / so[k] - 1).max() < tol, k
    if not fp32:
        assert g.stats()["subcycles"] >= n


@pytest.mark.parametrize("n_src", [1, 255, 700])
def test_gated_sources_in_the_budget(n_src):
    """Three boxes; the emitted photons of a step are those of the open sources of each box (FP64
    sums of at most 700 terms in another order: 1e-13)."""
    from paper_1311_0182_gb300 import rt
    rng = np.random.default_rng(n_src)
    wl = W.cfg4(n_boxes=3, n_min=512, n_max=1500, transport_fp32=0)
    n = len(wl["x"])
    wl["x_HI"] = rng.choice([1e-3, 0.9], n)
    L = float(wl["box_L"][0])
    wl["src_box"] = rng.integers(0, 3, n_src).astype(np.int32)
    for k in ("src_x", "src_y", "src_z"):
        wl[k] = rng.uniform(0.0, L, n_src)
    wl["src_ndot"] = rng.uniform(1e47, 1e49, n_src)
    wl["src_gate"] = rng.integers(0, 2, n_src).astype(np.int32)
    g = rt.context_for(wl)
    snbr = g.neighbours()[2]
    on = (wl["src_gate"] == 0) | (wl["x_HI"][snbr[:, 0]] < 0.5)
    g.step(0, allow_subcycle_limit=True)
    want = np.bincount(wl["src_box"][on], wl["src_ndot"][on] * wl["params"]["dt_em"], minlength=3)
    assert np.allclose(g.budget()[:, 0], want, rtol=1e-13, atol=0.0)


@pytest.mark.parametrize("n_ntc", [2, 8, 32])
@pytest.mark.parametrize("n_side,n_freq", [(5, 1), (9, 8), (12, 3)])
def test_order_of_requests_and_staging_changes_nothing(n_side, n_freq, n_ntc):
    """Requests, staged contributions and receiver groups arrive in an order that depends on the
    launch; the results do not: the same bits for three launch sizes, on both precisions, at
    sizes that are no multiple of a warp's turn, from wide cones (every packet has many members)
    to narrow ones (most request a virtual particle), and with every particle's packets as free
    packets (emission-cone mode)."""
    from paper_1311_0182_gb300 import rt
    for mode in (W.REC_TRANSPORT, W.REC_EMISSION_CONES):
        for fp32 in (0, 1):
            wl = W.cfg2(n_side=n_side, n_freq_src=n_freq, n_tc=n_ntc, n_rc=8, n_ec=8, rec_mode=mode,
                        transport_fp32=fp32)
            wl["sigma"], wl["eps"] = wl["sigma"][:n_freq], wl["eps"][:n_freq]
            wl["src_ndot"] = wl["src_ndot"][:n_freq]
            out = []
            for grid in ((0, 0, 0), (1, 1, 1), (7, 3, 40)):
                g = rt.context_for(wl, launch_grid=grid)
                for step in range(3):
                    g.step(step, allow_subcycle_limit=True)
                out.append((g.state(), g.deposits(), g.slots(), g.stats()))
                g.close()
            for s, d, f, st in out[1:]:
                assert all(np.array_equal(s[k], out[0][0][k]) for k in s)
                assert all(np.array_equal(x, y) for x, y in zip(d, out[0][1]))
                assert np.array_equal(f, out[0][2])
                assert all(st[k] == out[0][3][k] for k in ("hops", "virtual", "gas_contrib",
                                                           "staged_contrib", "receiver_groups"))
