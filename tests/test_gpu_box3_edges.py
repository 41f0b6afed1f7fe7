"""3-D sweeps at the sizes where their schedules change, FP64 bitwise against the oracle: the tile form of the
plain sweeping (8 x 4 column tiles, chunks of 4 steps) and the hyperplane form that larger grids take, and the
subdomain boxes of the decomposition: partial tiles, more tiles than the warps hold, thin boxes without a border."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _problem(shape, seed, g0=0.0):
    rng = np.random.default_rng(seed)
    r = rng.uniform(0.5, 2.0, shape)
    gamma = np.zeros(shape, np.uint8)
    for _ in range(3):
        gamma[tuple(rng.integers(0, s) for s in shape)] = 1
    return r, gamma, g0 + rng.uniform(0.0, 0.1, shape)


def _dev(*arrs):
    return [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in arrs]


@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 4, 8), (4, 5, 9), (5, 3, 7), (8, 13, 17), (13, 8, 33), (29, 21, 16),
                                   (40, 9, 25), (3, 430, 420)])
def test_fsm3(gpu, shape):
    r, gamma, g = _problem(shape, sum(shape), g0=-1.0 if shape[0] == 5 else 0.0)
    u_ref, sweeps, _ = O.fsm(r, gamma, g, 0.05)
    u, st = gpu.fsm(*_dev(r, gamma, g), 0.05)
    np.testing.assert_array_equal(u.cpu().numpy(), u_ref)
    assert st["sweeps"] == sweeps and st["converged"] == 1


# tiles and cells per subdomain (x, y, z), coarse ratio
@pytest.mark.parametrize("tiles,cells,c", [((2, 2, 2), (4, 4, 4), 4), ((2, 1, 2), (8, 8, 8), 4), ((1, 2, 2), (10, 6, 4), 2),
                                           ((1, 1, 2), (64, 40, 4), 4), ((1, 1, 1), (2, 2, 2400), 2)])
def test_dd3_boxes(gpu, tiles, cells, c):
    shape = tuple(t * s + 1 for t, s in zip(reversed(tiles), reversed(cells)))
    r, gamma, g = _problem(shape, 17 + sum(shape))
    kw = dict(theta=0.2, max_iter=2, tol=0.0, max_coarse_sweeps=8)
    u_ref, s_ref, _ = O.dd(r, gamma, g, 0.05, tiles, c, **kw)
    u, st = gpu.dd_solve(*_dev(r, gamma, g), 0.05, tiles, c, **kw)
    assert st["iters"] == s_ref["iters"]
    np.testing.assert_array_equal(u.cpu().numpy(), u_ref)


def test_dd3_without_room_for_packed_boxes(gpu):
    """A problem that fits the library's static scratch only without the packed subdomains and the line flags: the
    same solve, bit for bit."""
    r, gamma, g = _problem((73, 73, 73), 3)
    r[20:40, 10:30, 33] = np.inf
    kw = dict(theta=0.2, max_iter=2, tol=0.0, max_coarse_sweeps=8)
    R, G, g_t = _dev(r, gamma, g)
    grid, p = gpu.make_grid(R, 0.05), gpu.dd_params((3, 3, 3), 4, **kw)
    assert gpu.eik_dd_workspace_size(grid, p) > 32 << 20
    u_ref, s_ref = gpu.dd_solve(R, G, g_t, 0.05, (3, 3, 3), 4, **kw)
    u = torch.empty_like(R)
    st = torch.zeros(gpu.ctypes.sizeof(gpu.DDStats), dtype=torch.uint8, device=DEV)
    gpu.eik_dd_solve_noalloc(grid, R, G, g_t, p, u, st)
    torch.cuda.synchronize()
    got = gpu.parse_dd_stats(st)
    assert torch.equal(u, u_ref)
    assert {k: v for k, v in got.items() if k != "launches"} == {k: v for k, v in s_ref.items() if k != "launches"}


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_fsm3_in_a_workspace_without_tiles(gpu, dtype):
    """A workspace with room for 8 bytes a node, which was once all that was asked for: the same solve."""
    r, gamma, g = _problem((17, 21, 30), 4)
    R, G, g_t = _dev(r, gamma, g)
    R, g_t = R.to(dtype), g_t.to(dtype)
    grid = gpu.make_grid(R, 0.05)
    u_ref, s_ref = gpu.fsm(R, G, g_t, 0.05)
    nbytes = (8 * R.numel() + 255) // 256 * 256 + 304
    assert gpu.eik_fsm_workspace_size(grid) > nbytes
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device=DEV)
    off = -ws.data_ptr() % 256
    u = torch.empty_like(R)
    st = torch.zeros(gpu.ctypes.sizeof(gpu.FsmStats), dtype=torch.uint8, device=DEV)
    gpu.eik_fsm(grid, R, G, g_t, u, 1000, ws[off:off + nbytes], st)
    torch.cuda.synchronize()
    got = gpu.FsmStats.from_buffer_copy(bytes(st.cpu().numpy()))
    assert torch.equal(u, u_ref)
    assert (got.sweeps, got.converged) == (s_ref["sweeps"], 1)
