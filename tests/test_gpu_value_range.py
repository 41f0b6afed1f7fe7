"""Values at the ends of the FP64 range, signs of zero, boundary values that are no finite numbers.

Against plain serial sweeps of the same closed form in numpy: where (r h)^2 overflows the discriminant of the two-term branch is +inf or, if the difference squared overflows too,
NaN, which counts as 0; a NaN of the three-term branch leaves the node as it is."""
import itertools

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _solve(mins, rh):
    """The Godunov local solve from the minima of the two or three axes."""
    a = sorted(mins)
    d = a[0] - a[1]
    if not abs(d) < rh:
        return a[0] + rh
    u = (a[0] + a[1] + np.sqrt(np.fmax((2.0 * rh) * rh - d * d, 0.0))) * 0.5
    if len(a) == 3 and u > a[2]:
        d1, d2 = a[1] - a[0], a[2] - a[0]
        disc = (d1 + d2) * (d1 + d2) - 3.0 * ((d1 * d1 + d2 * d2) - rh * rh)
        u = a[0] + ((d1 + d2) + np.sqrt(0.0 if disc < 0.0 else disc)) / 3.0
    return u


def sweeps(r, gamma, g, h, most):
    """Serial sweeps in the 2^d orderings (the sign of x outermost, -1 first) until one changes nothing, `most` at
    most."""
    shape = r.shape
    u = np.full([s + 2 for s in shape], np.inf)
    core = tuple(slice(1, s + 1) for s in shape)
    u[core] = np.where(gamma != 0, g, np.inf)
    dim = len(shape)
    for k in range(most):
        changed = False
        signs = [(k >> a) & 1 for a in range(dim)]  # of the axes of the array: the last one, x, is the highest bit
        for at in itertools.product(*(range(s) if up else range(s - 1, -1, -1) for s, up in zip(shape, signs))):
            if gamma[at]:
                continue
            c = tuple(i + 1 for i in at)
            mins = []
            for a in range(dim):
                lo = c[:a] + (c[a] - 1,) + c[a + 1:]
                hi = c[:a] + (c[a] + 1,) + c[a + 1:]
                mins.append(np.fmin(u[lo], u[hi]))
            v = _solve(mins, r[at] * h)
            if v < u[c]:
                u[c] = v
                changed = True
        if not changed:
            return u[core], k + 1
    return u[core], most


def _dev(*arrs):
    return [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in arrs]


# one warp, one thread block and several in 2-D, tiles in 3-D
@pytest.mark.parametrize("shape", [(11, 9), (7, 40), (4, 300), (5, 6, 11)])
@pytest.mark.parametrize("scale", [1e153, 1e154, 1e155, 1e200, 1e300, 1.2e308])
def test_squares_above_the_range(gpu, shape, scale):
    rng = np.random.default_rng(sum(shape))
    r = scale * rng.choice([1.0, 0.75, 0.5], shape)
    gamma = np.zeros(shape, np.uint8)
    gamma[tuple(s // 2 for s in shape)] = gamma[(0,) * len(shape)] = 1
    g = np.zeros(shape)
    g[(0,) * len(shape)] = 0.125 * scale
    with np.errstate(all="ignore"):
        u_ref, n = sweeps(r, gamma, g, 1.0, 12)
    u, st = gpu.fsm(*_dev(r, gamma, g), 1.0, max_sweeps=12)
    np.testing.assert_array_equal(u.cpu().numpy(), u_ref)
    assert st["sweeps"] == n


# a node between two Gamma nodes at -0 and +0: a tie, which goes to the plus side
@pytest.mark.parametrize("tiles,cells,c", [((2, 2), 16, 8), ((1, 2), 60, 10), ((2, 2, 2), 8, 4)])
@pytest.mark.parametrize("z", [0.0, -0.0])
@pytest.mark.parametrize("step", ["fine", "coarse"])
def test_signs_of_zero(gpu, tiles, cells, c, z, step):
    shape = tuple(t * cells + 1 for t in reversed(tiles))
    rng = np.random.default_rng(len(shape) + cells)
    r = rng.uniform(0.5, 2.0, shape)
    gamma, g = np.zeros(shape, np.uint8), np.zeros(shape)
    w = 1 if step == "fine" else c  # neighbours of coarse node (c, c) on the fine grid or on its coarse grid
    for x, v in ((c - w, z), (c + w, -z)):
        at = (c,) * (len(shape) - 1) + (x,)
        gamma[at], g[at] = 1, v
    kw = dict(theta=0.2, max_iter=3, tol=0.0, max_coarse_sweeps=8)
    u_ref, s_ref, _, U_ref = O.dd(r, gamma, g, 0.05, tiles, c, return_coarse=True, **kw)
    u, st, *coarse = gpu.dd_solve(*_dev(r, gamma, g), 0.05, tiles, c, return_coarse=len(shape) == 2, **kw)
    np.testing.assert_array_equal(u.cpu().numpy(), u_ref)
    assert st["iters"] == s_ref["iters"]
    if coarse:
        U = coarse[0].cpu().numpy()
        on = ~np.isnan(U)
        np.testing.assert_array_equal(U[on], U_ref[on])
        if step == "fine":  # the x component of its wind: from the plus side
            assert int(coarse[1][c, c]) & 3 == 0


MINUS_NAN = np.array(0xfff8000000000000, np.uint64).view(np.float64)[()]  # what inf - inf is


def _special(shape, v):
    rng = np.random.default_rng(sum(shape))
    r = rng.uniform(0.5, 2.0, shape).astype(np.float32).astype(np.float64)
    gamma, g = np.zeros(shape, np.uint8), np.zeros(shape)
    for k, val in enumerate((v, 0.0, 0.0625)):
        at = tuple((s * (2 * k + 1)) // 7 for s in shape)
        gamma[at], g[at] = 1, val
    return r, gamma, g


# the nodes around a NaN do as if it were not there, and it stays; -inf reaches every node
@pytest.mark.parametrize("shape", [(11, 9), (7, 40), (4, 300), (5, 6, 11)])
@pytest.mark.parametrize("v", [np.nan, MINUS_NAN, -np.inf, np.inf])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_special_boundary_values(gpu, shape, v, dtype):
    r, gamma, g = _special(shape, v)
    R, G, g_t = _dev(r, gamma, g)
    u, st = gpu.fsm(R.to(dtype), G, g_t.to(dtype), 0.05)
    with np.errstate(all="ignore"):
        u_ref, n = sweeps(r, gamma, g, 0.05, 100)
    if dtype == torch.float64:
        np.testing.assert_array_equal(u.cpu().numpy(), u_ref)
        assert st["sweeps"] == n
    else:
        np.testing.assert_allclose(u.cpu().numpy(), u_ref, rtol=1e-5, equal_nan=True)


# subdomains of one warp and of several, 3-D boxes, the 1-D method in shared and in global memory
@pytest.mark.parametrize("tiles,cells,c", [((2, 2), 16, 8), ((1, 2), 60, 10), ((2, 2, 2), 8, 4), ((12,), 10, 10),
                                           ((2,), 20000, 20000)])
@pytest.mark.parametrize("v", [np.nan, MINUS_NAN])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_special_boundary_values_dd(gpu, tiles, cells, c, v, dtype):
    shape = tuple(t * cells + 1 for t in reversed(tiles))
    r, gamma, g = _special(shape, v)
    kw = dict(theta=0.2, max_iter=3, tol=0.0, max_coarse_sweeps=8)
    R, G, g_t = _dev(r, gamma, g)
    u, _ = gpu.dd_solve(R.to(dtype), G, g_t.to(dtype), 0.05, tiles, c, **kw)
    np.testing.assert_array_equal(np.isnan(u.cpu().numpy()), np.isnan(g))
