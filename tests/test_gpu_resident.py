"""Many cycles of a small system in one launch (csrc/resident.cu): single calls
of 1, 2, 3 and 16 cycles leave the state of the oracle's cycles, 40 cycles in
one call that of 40 calls with per-kernel timing on (which takes the two
kernels per cycle), for systems of one tile, fewer tiles than SMs, ragged last
tiles, more tiles than one per warp, several grid sizes against the threads,
16-bit fields, both interaction options, a mixture and closed cells; and the
counters and buffers stay usable by the calls that follow."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import GRID_BF16, GRID_F16, GRID_F32, System, SystemDesc, workloads
from tests.test_gpu_mixture import _sequences
from tests.test_gpu_parity import Runner

pytestmark = pytest.mark.gpu

# (N, chains, box, grid): 1 tile; 3 ragged; 63; 512; 6,000 tiles
SIZES = [(64, 1, (1.0, 1.0, 1.0), (6, 6, 6)), (16, 11, (1.0, 0.5, 0.5), (6, 3, 3)),
         (12, 313, (1.5, 1.0, 1.0), (9, 6, 6)), (32, 1024, (2.0, 2.0, 2.0), (12, 12, 12)),
         (32, 12000, (6.0, 4.0, 4.0), (36, 24, 24))]


def _desc(k, **kw):
    N, n, box, grid = SIZES[k]
    return SystemDesc(**dict(dict(n_chains=n, N=N, f=0.4, box_Re=box, grid=grid, chiN=25.0, kappaN=40.0, seed=9), **kw))


@pytest.mark.parametrize("k", range(4))
def test_calls_of_any_number_of_cycles_match_oracle(cuda_device, k):
    r = Runner(_desc(k))
    for n in (1, 2, 3, 16):
        if not r.step(n):
            break


@pytest.mark.parametrize("dtype", [GRID_F32, GRID_BF16, GRID_F16])
@pytest.mark.parametrize("ham", [0, 1])
@pytest.mark.parametrize("k", range(5))
def test_one_launch_equals_two_kernels_per_cycle(cuda_device, k, ham, dtype):
    d = _desc(k, hamiltonian=ham, grid_dtype=dtype)
    a, b = System(d), System(d)
    if k == 3:   # closed cells, a potential and a mixture
        rng = np.random.default_rng(1)
        ext, shut = rng.normal(0, 0.5, (2, d.cells)).astype(np.float32), rng.random(d.cells) < 0.1
        seq = _sequences(d.N)
        arch = rng.integers(0, len(seq), d.n_chains).astype(np.uint8)
        for s in (a, b):
            s.set_external(ext, shut.astype(np.uint8))
            s.set_architectures(seq, arch)
            s.update_fields()
    a.sweep(40)
    b.set_timing(True)
    b.sweep(40)
    b.set_timing(False)
    for _ in range(2):
        np.testing.assert_array_equal(a.get_positions(), b.get_positions())
        np.testing.assert_array_equal(a.get_density(), b.get_density())
        np.testing.assert_array_equal(a.get_fields(), b.get_fields())
        oa, ob = a.observables(), b.observables()
        assert (oa["accepted"], oa["sweeps"], oa["max_cell"]) == (ob["accepted"], ob["sweeps"], ob["max_cell"])
        a.set_sweep(7)   # the buffers by the new counter's parity
        b.set_sweep(7)
        a.sweep(3)
        b.set_timing(True)
        b.sweep(3)


def test_overflow_of_a_cell_is_reported(cuda_device):
    from paper_1711_03828_gb300 import SomaError, _abi
    d = SystemDesc(n_chains=4000, N=32, f=1.0, box_Re=(1.0, 1.0, 1.0), grid=(6, 6, 6), chiN=0.0, kappaN=0.0,
                   seed=2, a_Re=1e-3)
    s = System(d)
    pos = np.full((3, d.M), 0.5, np.float32)   # 128,000 particles in one cell
    s.set_positions(pos)
    with pytest.raises(SomaError) as e:
        s.sweep(2)
        s.sync()
    assert e.value.status == _abi.SOMA_EOVERFLOW
