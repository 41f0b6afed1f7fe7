"""Outputs that overwrite inputs: plain sweeping of small grids, which reads the caller's arrays directly, against the
same solve into arrays of its own, bitwise."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _problem(shape, dtype, seed):
    rng = np.random.default_rng(seed)
    r = torch.from_numpy(rng.uniform(0.5, 2.0, shape)).to(DEV, dtype)
    gamma = torch.zeros(shape, dtype=torch.uint8, device=DEV)
    g = torch.zeros(shape, dtype=dtype, device=DEV)
    for _ in range(3):
        at = tuple(int(rng.integers(0, s)) for s in shape)
        gamma[at], g[at] = 1, float(rng.uniform(0.0, 0.1))
    return r, gamma, g


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("into", ["r", "own g", "another g"])
def test_fsm_many_into_inputs(gpu, dtype, into):
    shape, k = (30, 33), 40
    r, gamma, g = _problem(shape, dtype, 9)
    gs = [g + 0.01 * i for i in range(k)]
    ref, _ = gpu.fsm_many(r, [gamma] * k, gs, 0.05)
    us = [torch.empty_like(r) for _ in range(k)]
    if into == "r":
        us[k // 2] = r
    elif into == "own g":
        us = gs
    else:
        us = gs[1:] + gs[:1]
    grid, lib, c = gpu.make_grid(r, 0.05), gpu.load(), gpu.ctypes
    ws = torch.empty(lib.eik_fsm_many_workspace_size(c.byref(grid), k) + 256, dtype=torch.uint8, device=DEV)
    wp, wn = gpu._aligned(ws)
    a = gpu._ptr_array
    rc = lib.eik_fsm_many(c.byref(grid), k, gpu._ptr(r), a([gamma] * k), a(gs), a(us), 1000, wp, wn, None,
                          gpu._stream(None))
    assert rc == 0
    for u, want in zip(us, ref):
        assert torch.equal(u, want)
