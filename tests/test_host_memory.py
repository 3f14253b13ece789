"""A host allocation that fails inside the library comes back as SG_E_OOM: no C++
exception leaves the C ABI, and the simulator stays usable."""

import resource

import numpy as np
import pytest
import torch

from workloads.configs import base_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["sg_sim_get_clearance", "sg_sim_get_sector_skip"])
def test_plane_download_without_host_memory(entry):
    import ctypes as C

    from paper_2305_04180_gb300 import Sim, _lib

    side = 8192  # a plane of 67 MB: more than the allocator has at hand
    planes = 4 if entry == "sg_sim_get_sector_skip" else 1
    grid = np.ones((side, side), np.uint8)
    grid[4000:4003, 4000:4003] = 0
    s = Sim(base_params(march_sectors=planes), [grid], np.zeros(1, np.int32))
    get = getattr(s.L, entry)
    n = C.c_size_t(0)
    extra = [None] if entry == "sg_sim_get_clearance" else [None, None]
    assert get(s.handle, None, C.byref(n), *extra) == _lib.SG_OK and n.value == planes * side * side
    out = np.zeros(n.value, np.uint8)
    torch.cuda.synchronize()
    used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
    soft, hard = resource.getrlimit(resource.RLIMIT_AS)
    resource.setrlimit(resource.RLIMIT_AS, (used + (32 << 20), hard))
    try:
        rc = get(s.handle, out.ctypes.data, C.byref(n), *extra)
    finally:
        resource.setrlimit(resource.RLIMIT_AS, (soft, hard))
    assert rc == _lib.SG_E_OOM
    assert get(s.handle, out.ctypes.data, C.byref(n), *extra) == _lib.SG_OK
    assert out[4001 * side + 4001] > 0 and out[3999 * side + 4001] == 0
