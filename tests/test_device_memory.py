"""Device memory of a context: the library's capacity is the largest workload whose context fits the
GPU, so a context must not grow."""
import numpy as np
import pytest

from paper_1311_0182_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# MB that rt_create took on a GB300 before the hop kernels read particles and edges in packed pieces
# and staged contributions carried an order, for FP64 and FP32 packets
HELD = {
    "sphere": (2420, 1688),            # 64^3, 8 cones, 2 bins, default capacity of free packets
    "few_free_packets": (1120, 796),   # the same with room for 1000
    "few_neighbours": (1384, 868),     # the same with 4 neighbours a particle
    "emission_cones": (7510, 4786),
    "shared_bin": (2170, 1534),
    "no_source_bins": (2042, 1470),
    "hii_region": (12476, 6688),       # 64^3, 32 cones, 9 bins, room for 100,000
}


def _workload(name):
    if name == "hii_region":
        return W.cfg2(64, free_cap=100000)
    kw = {"few_free_packets": dict(free_cap=1000), "few_neighbours": dict(n_ngb=4),
          "emission_cones": dict(rec_mode=W.REC_EMISSION_CONES), "shared_bin": dict(rec_shared_bin=1),
          "no_source_bins": dict(n_freq_src=0)}.get(name, {})
    wl = W.cfg1(64, **kw)
    if name == "no_source_bins":
        wl.update(sigma=np.zeros(0), eps=np.zeros(0), src_ndot=np.zeros(0))
    return wl


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("name", sorted(HELD))
def test_a_context_holds_no_more_than(name, fp32):
    """The drop in free device memory over rt_create (allocations come in pieces of 2 MB)."""
    import torch
    from paper_1311_0182_gb300 import rt
    wl = _workload(name)
    rt.Context(wl, transport_fp32=fp32).close()      # what the first context loads, once
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    c = rt.Context(wl, transport_fp32=fp32)
    held = (before - torch.cuda.mem_get_info()[0]) / 2 ** 20
    c.close()
    assert held <= HELD[name][fp32] + 2
