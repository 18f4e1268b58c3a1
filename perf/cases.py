"""Timed cases of the TRAPHIC transport sweep: whole RT steps through the public calls, over the
sizes, precisions and options that programs use, and the neighbour build of a moved particle set.

A step case is one time step of a radiation-hydrodynamics loop: the host code hands over the gas
state (rt_set_state), the library takes one RT step (rt_step), and the state and the photon
budget come back.  The gas state of every pass is the same, taken from a run that is already
under way, so the passes repeat the same step.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1311_0182_gb300 import rt
from paper_1311_0182_gb300 import workloads as W

MYR = W.MYR


def listed():
    return [
        # the smallest call: a test-sized box, where launches and latency are all there is
        dict(name="stromgren_12_f32", kind="stromgren", n_side=12, fp32=True, n_ngb=32, warm=12),
        # the paper's Sec. 3 sphere at its 16^3 size, all FP64: what a run of 200 steps repeats
        dict(name="stromgren_16_f64", kind="stromgren", n_side=16, fp32=False, n_ngb=32, warm=12),
        # a region whose source has gone out, on the spot: no photons move, so the step is the
        # chemistry and what a step costs anyway
        dict(name="fossil_80_f32", kind="fossil", n=80 ** 3, fp32=True, n_ngb=32, warm=0),
        # the benchmark's HII region: 32 cones, 8 source bins and the recombination bin
        dict(name="hii_64_f32", kind="hii", n_side=64, fp32=True, n_ngb=32, cones=32,
             rec_mode=W.REC_TRANSPORT, shared=False, warm=2),
        # the same on the FP64 path, the comparison path of every accuracy check
        dict(name="hii_32_f64", kind="hii", n_side=32, fp32=False, n_ngb=32, cones=32,
             rec_mode=W.REC_TRANSPORT, shared=False, warm=2),
        # an odd size with the recombination photons in the first source bin
        dict(name="hii_27_shared_f32", kind="hii", n_side=27, fp32=True, n_ngb=32, cones=32,
             rec_mode=W.REC_TRANSPORT, shared=True, warm=2),
        # without transported recombination radiation (case B on the spot): few packets
        dict(name="hii_64_ots_f32", kind="hii", n_side=64, fp32=True, n_ngb=32, cones=32,
             rec_mode=W.REC_OTS_CASE_B, shared=False, warm=2),
        # the dense clump behind a bright source at its full 128^3 particles, 8 cones
        dict(name="clump_2m_f32", kind="clump", n=128 ** 3, fp32=True, n_ngb=32,
             rec_mode=W.REC_TRANSPORT, warm=1),
        # many independent boxes of uneven size in the same launches
        dict(name="boxes_96_f32", kind="boxes", n_boxes=96, fp32=True, n_ngb=32, warm=1),
        # a clustered cosmological volume with many sources: packets travel a few hops a step
        dict(name="cosmo_128_f32", kind="cosmo", n_side=128, n_src=64, fp32=True, n_ngb=32, warm=1),
        # the shadow test: directed and gated emitters, a barrier, narrow cones, all FP64
        dict(name="shadow_32_f64", kind="shadow", n_side=32, n_front=100, n_bnd=50, fp32=False,
             n_ngb=32, warm=1),
        # new positions of the gas: particles and sources set, neighbours built
        dict(name="neighbours_300k", kind="neighbours", n=300007, fp32=True, n_ngb=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stromgren", "fossil", "hii", "hii", "hii", "clump", "clump", "boxes", "cosmo",
                       "shadow", "neighbours"])
    fp32 = rng.random() < 0.7
    c = dict(kind=kind, fp32=fp32, n_ngb=rng.choice([32, 32, 32, 27, 16]))
    if kind == "stromgren":
        c.update(n_side=rng.randint(8, 25), warm=rng.randint(4, 16))
    elif kind == "fossil":
        c.update(n=_log(rng, 3000, 600000), warm=0)
    elif kind == "hii":
        shared = rng.random() < 0.25
        mode = W.REC_TRANSPORT if shared else rng.choice(
            [W.REC_TRANSPORT, W.REC_TRANSPORT, W.REC_OTS_CASE_B, W.REC_CASE_A, W.REC_EMISSION_CONES])
        c.update(n_side=_log(rng, 12, 60 if fp32 else 36), cones=rng.choice([8, 32, 32]),
                 rec_mode=mode, shared=shared, warm=rng.randint(1, 3))
    elif kind == "clump":
        c.update(n=_log(rng, 15000, 1500000 if fp32 else 200000),
                 rec_mode=rng.choice([W.REC_TRANSPORT, W.REC_OTS_CASE_B]), warm=1)
    elif kind == "boxes":
        c.update(n_boxes=_log(rng, 3, 90 if fp32 else 12), warm=1)
    elif kind == "cosmo":
        c.update(n_side=_log(rng, 28, 120), n_src=_log(rng, 4, 256), warm=1)
    elif kind == "shadow":
        c.update(n_side=rng.randint(14, 34), n_front=rng.randint(20, 100), n_bnd=rng.randint(10, 50),
                 warm=1)
    else:
        c.update(n=_log(rng, 5000, 1200000), fp32=True)
    return c


# --- inputs ------------------------------------------------------------------------------------
def _particles(case):
    k = case["kind"]
    if k in ("stromgren", "hii", "shadow", "cosmo"):
        return case["n_side"] ** 3
    if k == "boxes":     # log-uniform in 512 .. 64000
        return int(case["n_boxes"] * (64000 - 512) / math.log(64000 / 512))
    return case["n"]


def _thin(wl, n, rng):
    """n particles of a one-box workload, in their order."""
    keep = np.sort(rng.permutation(len(wl["x"]))[:n])
    for k in ("x", "y", "z", "n_H", "N_H", "x_HI", "T"):
        wl[k] = np.ascontiguousarray(wl[k][keep])
    wl["N_H"] *= float(wl["box_off"][-1]) / n
    wl["box_off"] = np.array([0, n], np.int64)
    return wl


def _clump(case, seed, **p):
    # the generator's own count varies with its seed: a few per cent more, thinned to n
    wl = W.cfg3(n_total=int(1.04 * case["n"]) + 64, seed=seed, **p)
    return _thin(wl, case["n"], np.random.default_rng(seed + 1))


def _boxes(case, seed, **p):
    """The same boxes for every seed, each moved through itself periodically by its own offset."""
    wl, rng = W.cfg4(n_boxes=case["n_boxes"], **p), np.random.default_rng(seed)
    L, off = wl["box_L"], wl["box_off"]
    for b in range(case["n_boxes"]):
        part = slice(off[b], off[b + 1])
        for k in ("x", "y", "z"):
            wl[k][part] = np.minimum((wl[k][part] + rng.uniform(0.0, L[b])) % L[b], np.nextafter(L[b], 0.0))
    wl["params"]["seed"] = seed
    return wl


def _fossil(case, seed):
    """Gas of scattered density, ionisation and temperature around a source that is off."""
    n, rng = case["n"], np.random.default_rng(seed + 2)
    wl = W.cfg2(n_side=math.ceil(n ** (1.0 / 3.0) - 1e-9), seed=seed, rec_mode=W.REC_OTS_CASE_B,
                dt=2.5 * MYR, dt_em=2.5 * MYR)
    wl = _thin(wl, n, np.random.default_rng(seed + 1))
    L = float(wl["box_L"][0])
    wl["n_H"] = 3e-3 * np.exp(rng.normal(0.0, 1.0, n))
    wl["N_H"] = wl["n_H"] * L ** 3 / n
    wl["x_HI"] = np.exp(rng.uniform(math.log(1e-5), 0.0, n))
    wl["T"] = np.exp(rng.uniform(math.log(3e3), math.log(6e4), n))
    wl["src_ndot"] = np.zeros_like(wl["src_ndot"])
    return wl


def _workload(case, seed):
    k, p = case["kind"], dict(transport_fp32=int(case["fp32"]), n_ngb=case["n_ngb"])
    if k == "stromgren":
        wl = W.cfg1(n_side=case["n_side"], seed=seed, **p)
    elif k == "hii":
        c = case["cones"]
        wl = W.cfg2(n_side=case["n_side"], seed=seed, rec_mode=case["rec_mode"], n_rc=c, n_tc=c, n_ec=c,
                    rec_shared_bin=int(case["shared"]), **p)
    elif k == "clump":
        wl = _clump(case, seed, rec_mode=case["rec_mode"], **p)
    elif k == "boxes":
        wl = _boxes(case, seed, **p)
    elif k == "cosmo":
        wl = W.cfg5(n_side=case["n_side"], seed=seed, n_src=case["n_src"], **p)
    elif k == "shadow":
        wl = W.shadow(n_side=case["n_side"], seed=seed, n_front=case["n_front"], n_bnd=case["n_bnd"], **p)
    elif k == "fossil":
        wl = _fossil(case, seed)
        wl["params"].update(p)
    else:
        wl = _clump(case, seed, **p)
    return wl


def _gpu(a, dtype=np.float64):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def prepare(case, seed):
    wl = _workload(case, seed)
    ctx = rt.context_for(wl)
    if case["kind"] == "neighbours":
        n, kn = ctx.n, case["n_ngb"]
        return dict(
            case=case, ctx=ctx,
            gas=[_gpu(wl[k]) for k in ("x", "y", "z", "n_H", "N_H", "x_HI", "T")],
            src=[_gpu(wl["src_box"], np.int32)] + [
                _gpu(wl[k]) for k in ("src_x", "src_y", "src_z", "src_ndot", "sigma", "eps")],
            nbr=torch.zeros((n, kn), dtype=torch.int32, device="cuda"),
            h2=torch.zeros(n, dtype=torch.int64, device="cuda"),
            snbr=torch.zeros((ctx.ns, kn), dtype=torch.int32, device="cuda"),
            sh2=torch.zeros(ctx.ns, dtype=torch.int64, device="cuda"))
    for s in range(case["warm"]):
        ctx.step(s, allow_subcycle_limit=True)
    names = ("x_HI", "T", "N_rec", "eps_rec")
    gas = {k: torch.zeros(ctx.n, dtype=torch.float64, device="cuda") for k in names}
    ctx.get_state_into(**gas)
    # in nearly neutral gas rounding can leave the recombination photons or 1 - x_HI a last bit
    # below zero: nothing to emit, but refused as an input
    gas["N_rec"].clamp_(min=0.0)
    gas["x_HI"].clamp_(max=1.0)
    return dict(case=case, ctx=ctx, gas=gas, out={k: torch.zeros_like(v) for k, v in gas.items()})


def run(state):
    ctx = state["ctx"]
    if state["case"]["kind"] == "neighbours":
        ctx.set_particles(*state["gas"])
        ctx.set_sources(*state["src"])
        ctx.build_neighbours()
        out = [state[k] for k in ("nbr", "h2", "snbr", "sh2")]
        ctx._check(ctx.L.rt_get_neighbours(ctx.h, *[t.data_ptr() for t in out], rt.RT_DEVICE, ctx._s()),
                   "rt_get_neighbours")
        return out
    ctx.set_state(**state["gas"])
    ctx.step(state["case"]["warm"], allow_subcycle_limit=True)
    ctx.get_state_into(**state["out"])
    return dict(state["out"], budget=ctx.budget())


def work(case):
    n, kn = _particles(case), case["n_ngb"]
    if case["kind"] == "neighbours":
        # positions, atoms and state in; the neighbours and smoothing lengths out; a distance
        # (8 operations) for each neighbour found
        return dict(bytes=n * (56 + 4 * kn + 8), flops=8 * n * kn)
    # gas state in and out (4 doubles each), density and atoms, quantised position; the
    # neighbour list once, where photons travel; the rates and the update of one subcycle
    lists = 0 if case["kind"] == "fossil" else 4 * kn
    return dict(bytes=n * (64 + 16 + 12 + lists), flops=n * 200)


# --- 64-bit values --------------------------------------------------------------------------------
def _cooling_gas(wl):
    """x_HI and T after dt without photons: case-B recombination (Hui & Gnedin 1997), collisional
    ionisation, recombination and collisional-excitation cooling (Cen 1992), in subcycles of a 10%
    energy change with the electron density held in each."""
    kB, THI = 1.380649e-16, 157807.0
    p = wl["params"]
    x, T, nH = (np.array(wl[k], np.float64) for k in ("x_HI", "T", "n_H"))
    left = np.full(len(x), float(p["dt"]))
    on = np.arange(len(x))
    while len(on):
        xx, TT, nn, rest = x[on], T[on], nH[on], left[on]
        lam = 2.0 * THI / TT
        aB = 2.753e-14 * lam ** 1.5 / (1.0 + (lam / 2.74) ** 0.407) ** 2.242
        beta = 21.11 * TT ** -1.5 * np.exp(-lam / 2.0) * lam ** -1.089 / (1.0 + (lam / 0.354) ** 0.874) ** 1.101
        LB = 3.435e-30 * TT * lam ** 1.97 / (1.0 + (lam / 2.25) ** 0.376) ** 3.72
        Lce = 7.5e-19 * np.exp(-118348.0 / TT) / (1.0 + np.sqrt(TT / 1e5))
        ne = (1.0 - xx) * nn
        u = 1.5 * kB * TT * nn * (2.0 - xx)
        cool = ne * ((1.0 - xx) * nn) * LB + ne * (xx * nn) * Lce
        h = np.minimum(rest, np.where(cool > 0.0, 0.1 * u / np.where(cool > 0.0, cool, 1.0), rest))
        rate = (beta + aB) * ne
        eq = np.where(rate > 0.0, aB * ne / np.where(rate > 0.0, rate, 1.0), 0.0)
        xn = np.where(rate > 0.0, eq + (xx - eq) * np.exp(-rate * h), xx)
        x[on] = xn
        T[on] = np.maximum((u - h * cool) / (1.5 * kB * nn * (2.0 - xn)), p["T_floor"])
        left[on] = rest - h
        on = on[h < rest]
    return x, T, kB * T


def exact(case, seed):
    if case["kind"] != "fossil":
        # whole numbers (neighbours), or hops of packets whose every choice of a cone follows from
        # the last: minutes in plain arrays
        return None
    wl = _fossil(case, seed)
    x, T, eps = _cooling_gas(wl)
    return dict(x_HI=x, T=T, N_rec=np.zeros_like(x), eps_rec=eps, budget=np.zeros((1, 4)))
