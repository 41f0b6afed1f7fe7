"""Sweep engine at the sizes where its schedule changes, FP64 bitwise against the oracle: heights around the
8-row chunks and the 64-row ring, widths around the 32-column blocks, block counts around the switch from one
thread block to several, negative boundary values, and slownesses whose squares leave the FP64 range (where the
local solve takes the library square root)."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _problem(shape, seed, scale=1.0, g0=0.0):
    rng = np.random.default_rng(seed)
    r = scale * rng.uniform(0.5, 2.0, shape)
    gamma = np.zeros(shape, np.uint8)
    for _ in range(3):
        gamma[tuple(rng.integers(0, s) for s in shape)] = 1
    g = scale * (g0 + rng.uniform(0.0, 0.1, shape))
    return r, gamma, g


def _fsm(gpu, r, gamma, g, h, dtype=torch.float64):
    u, st = gpu.fsm(torch.from_numpy(r).to(DEV, dtype), torch.from_numpy(gamma).to(DEV),
                    torch.from_numpy(g).to(DEV, dtype), h)
    assert st["converged"] == 1
    return u.cpu().numpy(), st


@pytest.mark.parametrize("shape", [(2, 2), (7, 33), (8, 31), (9, 64), (24, 65), (32, 32), (33, 97), (63, 40), (64, 64),
                                   (65, 33), (71, 50), (72, 34), (73, 129), (95, 288), (40, 289), (66, 320), (41, 321),
                                   (130, 353)])
def test_heights_and_widths(gpu, shape):
    r, gamma, g = _problem(shape, 7 * shape[0] + shape[1])
    u_ref, sweeps, _ = O.fsm(r, gamma, g, 0.05)
    u, st = _fsm(gpu, r, gamma, g, 0.05)
    np.testing.assert_array_equal(u, u_ref)
    assert st["sweeps"] == sweeps


@pytest.mark.parametrize("scale,g0", [(1.0, -3.0), (1e-160, 0.0), (3e-154, 0.0), (1e150, 0.0), (1e-300, 0.0)])
def test_ranges(gpu, scale, g0):
    r, gamma, g = _problem((50, 70), 11, scale, g0)
    u_ref, _, _ = O.fsm(r, gamma, g, 0.05)
    u, _ = _fsm(gpu, r, gamma, g, 0.05)
    np.testing.assert_array_equal(u, u_ref)


# Small subdomains, which one warp sweeps with K columns a lane: widths around the 32 K edges, heights from the
# smallest to the largest that the form takes, and the first ones that go to the engine (FP32: 128 columns by 99
# rows; FP64: 36 columns).
@pytest.mark.parametrize("tiles,cells,c", [((1, 1), (2, 2), 1), ((3, 2), (2, 6), 2), ((2, 2), (30, 4), 2), ((2, 1), (31, 31), 31),
                                           ((1, 2), (32, 40), 4), ((2, 2), (62, 2), 2), ((1, 2), (63, 63), 21),
                                           ((2, 2), (64, 8), 8)])
def test_small_boxes(gpu, tiles, cells, c):
    shape = tuple(t * s + 1 for t, s in zip(reversed(tiles), reversed(cells)))
    r, gamma, g = _problem(shape, 5 + sum(shape), g0=-1.0 if cells[1] == 4 else 0.0)
    kw = dict(theta=0.2, max_iter=3, tol=0.0, max_coarse_sweeps=8)
    u_ref, s_ref, _ = O.dd(r, gamma, g, 0.05, tiles, c, **kw)
    u, st = gpu.dd_solve(*(torch.from_numpy(a).to(DEV) for a in (r, gamma, g)), 0.05, tiles, c, **kw)
    assert st["iters"] == s_ref["iters"]
    np.testing.assert_array_equal(u.cpu().numpy(), u_ref)


# FP32: a single subdomain has no inflow, so off the coarse lines it holds what plain sweeping gives
@pytest.mark.parametrize("nx,ny,c", [(3, 3, 2), (17, 9, 8), (32, 32, 31), (33, 5, 2), (64, 22, 21), (65, 129, 16), (96, 20, 19),
                                     (97, 33, 32), (127, 97, 6), (127, 100, 9), (129, 65, 32)])
def test_small_boxes_f32(gpu, nx, ny, c):
    r, gamma, g = _problem((ny, nx), nx + 3 * ny)
    u_ref, st_ref = _fsm(gpu, r, gamma, g, 0.05, torch.float32)
    u, st = gpu.dd_solve(torch.from_numpy(r).to(DEV, torch.float32), torch.from_numpy(gamma).to(DEV),
                         torch.from_numpy(g).to(DEV, torch.float32), 0.05, (1, 1), c, max_iter=2)
    off = (np.arange(ny)[:, None] % c != 0) & (np.arange(nx)[None, :] % c != 0)
    np.testing.assert_array_equal(u.cpu().numpy()[off], u_ref[off])
    assert st["fsm_sweeps_max"] == st_ref["sweeps"]


# ... and the same against the engine: the plain solve is made too wide for the one-warp form by a strip of Gamma nodes
# at +inf, which changes nothing
@pytest.mark.parametrize("nx,ny,c", [(3, 3, 2), (17, 9, 8), (32, 32, 31), (33, 5, 2), (64, 22, 21), (96, 20, 19), (97, 33, 32),
                                     (127, 97, 6)])
def test_small_boxes_f32_against_the_engine(gpu, nx, ny, c):
    r, gamma, g = _problem((ny, nx), nx + 3 * ny)
    wide = [np.concatenate([a, np.full((ny, 140), v, a.dtype)], 1) for a, v in ((r, 1.0), (gamma, 1), (g, np.inf))]
    u_ref, st_ref = _fsm(gpu, *wide, 0.05, torch.float32)
    u, st = gpu.dd_solve(torch.from_numpy(r).to(DEV, torch.float32), torch.from_numpy(gamma).to(DEV),
                         torch.from_numpy(g).to(DEV, torch.float32), 0.05, (1, 1), c, max_iter=2)
    off = (np.arange(ny)[:, None] % c != 0) & (np.arange(nx)[None, :] % c != 0)
    np.testing.assert_array_equal(u.cpu().numpy()[off], u_ref[:, :nx][off])
    assert st["fsm_sweeps_max"] == st_ref["sweeps"]


# plain sweeping of a small grid takes the one-warp form up to 128 (FP64: 36) columns while the box fits an SM; one by
# itself and several in a call, against the same nodes inside a grid too wide for it: a strip of Gamma nodes at +inf
# beside them changes nothing
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 200), (32, 33), (33, 17), (64, 190), (65, 40), (96, 31), (97, 101), (128, 190),
                                   (128, 205)])
def test_small_grids(gpu, nx, ny, dtype):
    r, gamma, g = _problem((ny, nx), 3 * nx + ny, g0=-0.5 if nx == 33 else 0.0)
    wide = [np.concatenate([a, np.full((ny, 140), v, a.dtype)], 1) for a, v in ((r, 1.0), (gamma, 1), (g, np.inf))]
    u_ref, st_ref = _fsm(gpu, *wide, 0.05, dtype)
    u, st = _fsm(gpu, r, gamma, g, 0.05, dtype)
    np.testing.assert_array_equal(u, u_ref[:, :nx])
    assert st["sweeps"] == st_ref["sweeps"]
    R = torch.from_numpy(r).to(DEV, dtype)
    gs = [torch.from_numpy(gamma).to(DEV)] * 3
    us, sts = gpu.fsm_many(R, gs, [torch.from_numpy(g + k).to(DEV, dtype) for k in range(3)], 0.05)
    np.testing.assert_array_equal(us[0].cpu().numpy(), u)
    assert sts[0]["sweeps"] == st["sweeps"] and all(s["converged"] == 1 for s in sts)


@pytest.mark.parametrize("shape", [(33, 30), (60, 150), (9, 8, 7)])
def test_g_is_read_at_gamma_only(gpu, shape):
    """The boundary values end behind the last Gamma node."""
    r, gamma, g = _problem(shape, 5)
    gamma[1:] = 0
    gamma[(0,) * len(shape)] = 1
    u_ref, _, _ = O.fsm(r, gamma, g, 0.05)
    R, G, first = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (r, gamma, g[0]))
    grid = gpu.make_grid(R, 0.05)
    ws = torch.empty(gpu.eik_fsm_workspace_size(grid) + 256, dtype=torch.uint8, device=DEV)
    u = torch.empty_like(R)
    gpu.eik_fsm(grid, R, G, first, u, 1000, ws, None)
    np.testing.assert_array_equal(u.cpu().numpy(), u_ref)


@pytest.mark.parametrize("shape", [(40, 300), (24, 1100)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_converged_in_the_last_sweep_allowed(gpu, shape, dtype):
    """Grids swept by several thread blocks, with exactly the sweeps that they need and with one less."""
    r, gamma, g = _problem(shape, 8)
    R, G, g_t = torch.from_numpy(r).to(DEV, dtype), torch.from_numpy(gamma).to(DEV), torch.from_numpy(g).to(DEV, dtype)
    u, st = gpu.fsm(R, G, g_t, 0.05)
    d = torch.ones_like(R)
    grad, ast = gpu.adjoint(R, G, u, d, 0.05)
    n, m = st["sweeps"], ast["sweeps"]
    many = [gpu.fsm_many(R, [G] * 3, [g_t] * 3, 0.05, max_sweeps=n + k)[1] for k in (-1, 0)]
    assert [[s["converged"] for s in q] for q in many] == [[0] * 3, [1] * 3]
    for _ in range(25):
        for k, conv in ((-1, 0), (0, 1)):
            s = gpu.fsm(R, G, g_t, 0.05, max_sweeps=n + k)[1]
            assert (s["sweeps"], s["converged"]) == (n + k, conv)
            s = gpu.adjoint(R, G, u, d, 0.05, max_sweeps=m + k)[1]
            assert (s["sweeps"], s["converged"]) == (m + k, conv)
