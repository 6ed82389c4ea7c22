"""The molecule-parallel iteration with one, two and four lanes per chain (chosen
from the number of chains and their length) against the oracle: one cycle from
given positions, every chain without a near-tie bit for bit, for chains longer
than a warp's staging of the others, short ones (many attempts of a group on the
same or bonded particles), ragged groups, and molecules of other architectures."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import ITERATION_MOLECULE, System, SystemDesc, workloads
from tests.conftest import oracle_system
from tests.test_gpu_parity import TIE, _pos

pytestmark = pytest.mark.gpu

W = workloads
# (N, chains): 20,001 chains give one lane (N <= 44) or two; fewer chains four
SHAPES = [(3, 20001), (12, 20001), (46, 20001), (1, 33), (2, 1001), (5, 700), (64, 99), (65, 41), (100, 37),
          (256, 9)]


def _compare(d, s, orc, pos0):
    s.set_positions(pos0)
    s.update_fields()
    p = _pos(pos0)
    nA, nB = orc.histogram(p)
    wA, wB = orc.fields(nA, nB)
    _, margin, acc = orc.sweep(p, wA, wB, 0, want_margin=True, want_acc=True)
    s.sweep(1)
    g = s.get_positions()
    keep = ~(np.abs(margin.reshape(d.n_chains, d.N)) < TIE).any(axis=1)
    assert keep.mean() > 0.9
    G, P = g.reshape(3, d.n_chains, d.N)[:, keep], p.stacked().reshape(3, d.n_chains, d.N)[:, keep]
    np.testing.assert_array_equal(G, P)
    if keep.all():
        nA, nB = orc.histogram(p)
        n = s.get_density()
        np.testing.assert_array_equal(n & 0xFFFF, nA)
        np.testing.assert_array_equal(n >> 16, nB)
    s.close()


def _desc(N, n):
    return SystemDesc(n_chains=n, N=N, f=0.4, box_Re=(3.0, 2.0, 1.5), grid=(18, 12, 9), chiN=25.0, kappaN=30.0,
                      seed=19, set_order=ITERATION_MOLECULE)


@pytest.mark.parametrize("N,n", SHAPES)
def test_linear_chains_match_oracle(cuda_device, N, n):
    d = _desc(N, n)
    _compare(d, System(d), oracle_system(d), W.random_walk_positions(d, seed=70))


@pytest.mark.parametrize("N,n", [(16, 20001), (46, 20001), (16, 501)])
def test_architectures_match_oracle(cuda_device, N, n):
    d = _desc(N, n)
    mols = [W.star_architecture(5, (N - 1) // 5), W.ring_architecture(N), W.linear_architecture(N - 3)]
    arch = np.random.default_rng(2).integers(0, len(mols), n).astype(np.uint8)
    words, starts = W.encode_architectures(mols)
    s, orc = System(d), oracle_system(d)
    s.set_topology(words, starts, arch)
    orc.set_topology(words, starts, arch)
    _compare(d, s, orc, W.architecture_positions(d, mols, arch, seed=71))
