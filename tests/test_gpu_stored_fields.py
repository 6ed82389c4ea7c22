"""External fields, and the density of the description after architectures of
several lengths, take effect at the next field update (include/soma.h): a call
of many cycles right after setting them, which a small system makes in one
launch, leaves the bits of as many calls of one cycle and of the two kernels per
cycle that per-kernel timing takes."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import GRID_BF16, GRID_F32, System, SystemDesc, workloads as W

pytestmark = pytest.mark.gpu

# one cluster's shared memory; all SMs
SIZES = [(313, (1.5, 1.0, 1.0), (9, 6, 6)), (6000, (5.0, 4.0, 3.0), (30, 24, 18))]


def _external(d):
    rng = np.random.default_rng(3)
    return (rng.normal(0, 0.8, (2, d.cells)).astype(np.float32),
            (rng.random(d.cells) < 0.1).astype(np.uint8))


def _set_both(s):
    s.set_external(*_external(s.desc))


def _clear(s):
    s.set_external(*_external(s.desc))
    s.update_fields()
    s.set_external()


def _diblock_again(s):
    d = s.desc
    words, starts = W.encode_architectures([W.linear_architecture(d.N - 7), W.linear_architecture(d.N)])
    s.set_topology(words, starts, (np.arange(d.n_chains) % 2).astype(np.uint8))
    s.update_fields()
    s.set_architectures()


@pytest.mark.parametrize("dtype", [GRID_F32, GRID_BF16])
@pytest.mark.parametrize("change", [_set_both, _clear, _diblock_again])
@pytest.mark.parametrize("k", range(len(SIZES)))
@pytest.mark.parametrize("cycles", [4, 19])
def test_change_waits_for_the_next_field_update(cuda_device, k, change, dtype, cycles):
    n, box, grid = SIZES[k]
    d = SystemDesc(n_chains=n, N=32, f=0.4, box_Re=box, grid=grid, chiN=25.0, kappaN=40.0, seed=5,
                   grid_dtype=dtype)
    at_once, one_by_one, timed = System(d), System(d), System(d)
    for s in (at_once, one_by_one, timed):
        change(s)
    at_once.sweep(cycles)
    for _ in range(cycles):
        one_by_one.sweep(1)
    timed.set_timing(True)
    timed.sweep(cycles)
    for s in (one_by_one, timed):
        np.testing.assert_array_equal(at_once.get_positions(), s.get_positions())
        np.testing.assert_array_equal(at_once.get_density(), s.get_density())
        np.testing.assert_array_equal(at_once.get_fields(), s.get_fields())
