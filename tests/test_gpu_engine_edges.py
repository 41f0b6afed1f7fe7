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
