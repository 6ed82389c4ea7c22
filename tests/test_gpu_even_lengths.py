"""Even chain lengths N <= 64 that do not divide 64: a full tile of
floor(64/N) chains then fills only part of the 32 lanes, and the lanes past it
hold no pair.  Every sweep of the paired layout is compared with the oracle
(batches with the same systems run alone), with the tolerances of the tests
of the lengths that divide 64."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import (Batch, FLAG_LEARNED_UMMA, MOVE_SMC, System, SystemDesc, workloads)
from tests.conftest import oracle_system
from tests.test_gpu_batch import _compare
from tests.test_gpu_learned import test_learned_tensor_core_one_cycle_matches_bf16_oracle as learned_one_cycle
from tests.test_gpu_mixture import _sequences
from tests.test_gpu_parity import Runner
from tests.test_gpu_smc import compare_smc_cycle

pytestmark = pytest.mark.gpu

# (N, chains): one chain per tile (34, 48, 62), several (6, 10, 12, 24), ragged last tiles
SHAPES = [(6, 1003), (10, 1000), (12, 701), (24, 333), (34, 257), (48, 200), (62, 129)]


def _desc(N, n, **kw):
    return SystemDesc(n_chains=n, N=N, f=0.5, box_Re=(2.0, 1.5, 1.0), grid=(12, 9, 6), chiN=25.0,
                      kappaN=30.0, seed=13, **kw)


@pytest.mark.parametrize("N,n", SHAPES)
def test_uniform_sweeps_match_oracle(cuda_device, N, n):
    r = Runner(_desc(N, n))
    live = True
    for _ in range(4):
        live = r.step(1)
        if not live:
            break
    if live:
        r.step(16)
    print(f"N={N}: {r.moves} moves, tolerated mismatches {r.mismatch}")


@pytest.mark.parametrize("N,n", SHAPES)
def test_smart_monte_carlo_matches_oracle(cuda_device, N, n):
    d = _desc(N, n, move=MOVE_SMC)
    for k, sweep in enumerate((0, 7)):
        moves, mism, acc = compare_smc_cycle(d, System(d), oracle_system(d),
                                             workloads.random_walk_positions(d, seed=40 + k), sweep)
        assert acc > 0.05 * moves and mism <= max(3, 1e-3 * moves)


@pytest.mark.parametrize("flags", [0, FLAG_LEARNED_UMMA], ids=["mma_sync", "tcgen05"])
@pytest.mark.parametrize("N,n", [(12, 701), (48, 200)])
def test_learned_matches_oracle(cuda_device, N, n, flags):
    learned_one_cycle(cuda_device, N, n, (12, 9, 6), (2.0, 1.5, 1.0), flags)


def test_mixture_matches_oracle(cuda_device):
    d = _desc(12, 701)
    seq = _sequences(d.N)
    arch = np.random.default_rng(4).integers(0, len(seq), d.n_chains).astype(np.uint8)
    r = Runner(d)
    r.gpu.set_architectures(seq, arch)
    r.gpu.update_fields()
    r.orc.set_architectures(seq, arch)
    r.nA, r.nB = r.orc.histogram(r.p)
    r.wA, r.wB = r.orc.fields(r.nA, r.nB)
    for _ in range(4):
        if not r.step(1):
            break


def test_batch_members_match_single_systems(cuda_device):
    descs = [_desc(N, n, replica_id=i) for i, (N, n) in enumerate(SHAPES + [(32, 100)])]
    b = Batch(descs)
    singles = [System(d) for d in descs]
    b.sweep(18)
    for s in singles:
        s.sweep(18)
    _compare(b, singles)
    b.close()
