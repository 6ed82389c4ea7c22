"""Launch shapes of the one-block-per-SM sweeps at the edges of their rules: less
work than SMs, one unit a block, one round of warps exactly and one unit more (a
block then has fewer warps), the uniform strips' blocks of fewer than eight items
and more, the learned sweep's of four warps, five to eight and more, and chains of
one particle, which strips take in pairs.  One cycle against the oracle, and one call
of many cycles against as many of one."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import MOVE_SMC, MOVE_UNIFORM, System, SystemDesc, workloads as W
from tests.conftest import oracle_system
from tests.test_gpu_learned import test_learned_tensor_core_one_cycle_matches_bf16_oracle as learned_one_cycle
from tests.test_gpu_parity import Runner
from tests.test_gpu_smc import compare_smc_cycle

pytestmark = pytest.mark.gpu

BOX, GRID = (4.0, 3.0, 2.5), (24, 18, 15)
SMS = 152


def _compare(N, n, move):
    d = SystemDesc(n_chains=n, N=N, f=0.4, box_Re=BOX, grid=GRID, chiN=25.0, kappaN=30.0, seed=23, move=move)
    if move == MOVE_UNIFORM:
        Runner(d).step(1)
    else:
        moves, mism, acc = compare_smc_cycle(d, System(d), oracle_system(d), W.random_walk_positions(d, seed=31), 0)
        assert acc > 0.02 * moves and mism <= max(3, 1e-3 * moves)
    at_once, one_by_one = System(d), System(d)
    at_once.sweep(18)
    one_by_one.set_timing(True)    # two kernels a cycle
    for _ in range(18):
        one_by_one.sweep(1)
    np.testing.assert_array_equal(at_once.get_positions(), one_by_one.get_positions())
    np.testing.assert_array_equal(at_once.get_density(), one_by_one.get_density())
    assert at_once.observables()["accepted"] == one_by_one.observables()["accepted"]


# tiles of one chain of 64: fewer than SMs; one each; 28 (a round of force-biased moves) and
# 32 (of uniform ones) and one more; 65 (one call is then not one resident launch)
@pytest.mark.parametrize("tiles", [3, SMS, 28 * SMS, 28 * SMS + 1, 32 * SMS + 1, 65 * SMS])
@pytest.mark.parametrize("move", [MOVE_UNIFORM, MOVE_SMC])
def test_pair_tiles(cuda_device, move, tiles):
    _compare(64, tiles, move)


# chains of 63 take one strip each, of 200 four, of 5 three of 32 lanes
@pytest.mark.parametrize("N,n", [(63, 5), (63, SMS), (63, 7 * SMS), (63, 8 * SMS), (63, 33 * SMS), (200, 40),
                                 (200, 9 * SMS), (5, 70 * SMS), (129, 33 * SMS)])
@pytest.mark.parametrize("move", [MOVE_UNIFORM, MOVE_SMC])
def test_strips(cuda_device, move, N, n):
    _compare(N, n, move)


@pytest.mark.parametrize("tiles", [4 * SMS, 4 * SMS + 1, 8 * SMS + 1, 16 * SMS + 1])
def test_learned_tiles(cuda_device, tiles):
    learned_one_cycle(cuda_device, 64, tiles, GRID, BOX, 0)


# two single particles walk as one chain: an odd one left over, alone and past a strip
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 701, 64 * SMS + 1])
def test_single_particles(cuda_device, n):
    _compare(1, n, MOVE_UNIFORM)


@pytest.mark.parametrize("f", [0.4, 0.6])     # all B, all A
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 701, 64 * SMS + 1])
def test_single_particles_force_biased(cuda_device, n, f):
    """Against the architecture sweep of molecules of one particle."""
    d = SystemDesc(n_chains=n, N=1, f=f, box_Re=BOX, grid=GRID, chiN=25.0, kappaN=30.0, seed=23, move=MOVE_SMC)
    strips, molecules = System(d), System(d)
    molecules.set_architectures([int(f < 0.5)], np.zeros(n, np.uint8))
    for cycles in (1, 18):
        strips.sweep(cycles)
        molecules.sweep(cycles)
        np.testing.assert_array_equal(strips.get_positions(), molecules.get_positions())
        np.testing.assert_array_equal(strips.get_density(), molecules.get_density())
    assert 0 < strips.observables()["accepted"] == molecules.observables()["accepted"]
