"""Molecule-parallel systems of several chain lengths in one process: a system
goes on sweeping, eagerly and in its graph, after a shorter one of the same kernel
(lanes per chain, field type, linear or not) has been created."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import ITERATION_MOLECULE, System, SystemDesc, workloads as W

pytestmark = pytest.mark.gpu


def _system(N, n, architectures):
    d = SystemDesc(n_chains=n, N=N, f=0.5, box_Re=(3.0, 2.0, 1.5), grid=(18, 12, 9), chiN=20.0, kappaN=30.0,
                   seed=11, set_order=ITERATION_MOLECULE)
    s = System(d)
    if architectures:
        words, starts = W.encode_architectures([W.ring_architecture(N), W.linear_architecture(N)])
        s.set_topology(words, starts, (np.arange(n) % 2).astype(np.uint8))
        s.update_fields()
    return s


# four lanes per chain; two; one (chains enough for the lane rule, both above 48 KB a block)
@pytest.mark.parametrize("longer,shorter,n,architectures",
                         [(256, 130, 40, False), (256, 130, 20001, False), (44, 33, 20001, False),
                          (44, 34, 20001, True)])
def test_a_shorter_system_leaves_a_longer_one_alone(cuda_device, longer, shorter, n, architectures):
    alone = _system(longer, n, architectures)
    alone.sweep(19)
    want = alone.get_positions(), alone.get_density()
    alone.close()
    a = _system(longer, n, architectures)
    b = _system(shorter, n, architectures)
    for _ in range(3):
        a.sweep(1)
        b.sweep(1)
    a.sweep(16)
    b.sweep(16)
    np.testing.assert_array_equal(a.get_positions(), want[0])
    np.testing.assert_array_equal(a.get_density(), want[1])
    assert b.observables()["sweeps"] == 19
