"""The set-pair layout of the architecture sweep (architectures of at most two
sets whose pairs fill the lanes as the general kernel's tiles do) against the
oracle: hubs of more than three partners, several molecules per warp and one,
molecules shorter than their slots, monomers, ragged last tiles; both set
orders, uniform and smart Monte Carlo moves, two types and three."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import MOVE_SMC, System, SystemDesc, workloads
from tests.conftest import oracle_system
from tests.test_gpu_parity import _pos
from tests.test_gpu_topology import _cycles
from tests.test_gpu_topology_smc import _one_cycle
from tests.test_gpu_types import CHI3
from tests.test_gpu_types import _cycles as _type_cycles

pytestmark = pytest.mark.gpu

W = workloads
CASES = {
    "N32": (32, 601, [W.star_architecture(4, [8, 8, 8, 7]), *W.arch_large_molecules()]),
    "N32_lengths": (32, 333, [W.linear_architecture(32), W.linear_architecture(11, 0), ([0], [])]),
    "N12": (12, 1001, [W.linear_architecture(12), W.ring_architecture(12)]),
    "N64": (64, 129, [W.linear_architecture(64), W.ring_architecture(64)]),
}


def _setup(name, **over):
    N, n, mols = CASES[name]
    d = SystemDesc(n_chains=n, N=N, f=0.5, box_Re=(2.0, 1.5, 1.0), grid=(12, 9, 6), chiN=25.0,
                   kappaN=30.0, seed=7, **over)
    arch = np.random.default_rng(3).integers(0, len(mols), n).astype(np.uint8)
    words, starts = W.encode_architectures(mols)
    return d, arch, words, starts, W.architecture_positions(d, mols, arch, seed=50)


@pytest.mark.parametrize("set_order", [0, 1])
@pytest.mark.parametrize("name", CASES)
def test_uniform_cycles_match_oracle(cuda_device, name, set_order):
    d, arch, words, starts, pos0 = _setup(name, set_order=set_order)
    gpu = System(d)
    gpu.set_topology(words, starts, arch)
    gpu.set_positions(pos0)
    gpu.update_fields()
    orc = oracle_system(d)
    orc.set_topology(words, starts, arch)
    moves, mism, _ = _cycles(d, gpu, orc, _pos(pos0), 6)
    gpu.close()
    print(f"{name}: {moves} moves, tolerated mismatches {mism}")


@pytest.mark.parametrize("name", CASES)
def test_smart_monte_carlo_matches_oracle(cuda_device, name):
    d, arch, words, starts, pos0 = _setup(name, move=MOVE_SMC)
    moves, mism, acc = _one_cycle(d, words, starts, arch, pos0, 4)
    assert acc > 0.05 * moves and mism <= max(3, 1e-3 * moves)


def _abc(**over):
    d = SystemDesc(n_chains=500, N=32, f=0.5, box_Re=(2.0, 1.5, 1.0), grid=(12, 9, 6), kappaN=30.0, seed=7,
                   **over)
    mols = W.abc_molecules()
    arch = np.random.default_rng(3).integers(0, len(mols), d.n_chains).astype(np.uint8)
    words, starts = W.encode_architectures(mols)
    return d, arch, words, starts, W.architecture_positions(d, mols, arch, seed=51)


def test_three_types_match_oracle(cuda_device):
    d, arch, words, starts, pos0 = _abc()
    gpu, orc = System(d), oracle_system(d)
    gpu.set_types(3, CHI3)
    gpu.set_topology(words, starts, arch)
    gpu.set_positions(pos0)
    gpu.update_fields()
    orc.set_topology(words, starts, arch)
    orc.set_types(3, CHI3)
    _type_cycles(d, gpu, orc, _pos(pos0), 5, CHI3)
    gpu.close()
    d, arch, words, starts, pos0 = _abc(move=MOVE_SMC)
    moves, mism, acc = _one_cycle(d, words, starts, arch, pos0, 2, n_types=3, chi=CHI3)
    assert acc > 0.05 * moves and mism <= max(3, 1e-3 * moves)
