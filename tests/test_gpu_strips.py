"""The strip layout of the SET sweeps (chains of odd length, of more than 64
particles, and even ones under smart Monte Carlo that fill strips better than
tiles) against the oracle, with the tolerances of the paired kernels' tests:
chains of one particle up to the longest, chains that end inside a strip, at
its last lane and beyond it, several per strip, and items cut by the last
chain; both set orders, 16-bit fields and a grid with one cell on an axis."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import (MOVE_SMC, SET_ORDER_FIXED, SET_ORDER_RANDOM, System, SystemDesc,
                                    workloads)
from tests.conftest import oracle_system
from tests.test_gpu_parity import Runner
from tests.test_gpu_smc import compare_smc_cycle

pytestmark = pytest.mark.gpu

# (N, chains); U = N // 2 + 1 units per chain: 1, 2, 16, 17, 32, 33, 51, 128, 129
SHAPES = [(1, 700), (3, 501), (31, 97), (33, 130), (63, 65), (65, 64), (100, 37), (255, 5), (256, 9)]


def _desc(N, n, **kw):
    kw = dict(dict(f=0.4, box_Re=(2.0, 1.5, 1.0), grid=(12, 9, 6), chiN=25.0, kappaN=30.0, seed=17), **kw)
    return SystemDesc(n_chains=n, N=N, **kw)


@pytest.mark.parametrize("order", [SET_ORDER_RANDOM, SET_ORDER_FIXED])
@pytest.mark.parametrize("N,n", SHAPES)
def test_uniform_strips_match_oracle(cuda_device, N, n, order):
    r = Runner(_desc(N, n, set_order=order))
    live = True
    for _ in range(4):
        live = r.step(1)
        if not live:
            break
    if live:
        r.step(16)


def test_uniform_strips_with_one_cell_on_an_axis(cuda_device):
    r = Runner(_desc(33, 130, box_Re=(2.0, 1.0, 1.0 / 6.0), grid=(12, 6, 1)))
    for _ in range(3):
        if not r.step(1):
            break


@pytest.mark.parametrize("N,n", SHAPES + [(42, 100), (48, 81)])
def test_smart_monte_carlo_strips_match_oracle(cuda_device, N, n):
    for k, sweep in enumerate((0, 5)):
        d = _desc(N, n, move=MOVE_SMC, set_order=SET_ORDER_FIXED if k else SET_ORDER_RANDOM)
        moves, mism, acc = compare_smc_cycle(d, System(d), oracle_system(d),
                                             workloads.random_walk_positions(d, seed=60 + k), sweep)
        assert acc > 0.02 * moves and mism <= max(3, 1e-3 * moves)
