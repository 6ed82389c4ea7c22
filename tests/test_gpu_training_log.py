"""The training log (mean expected squared jump of the first and the last batch,
mean acceptance of the last), summed on the device: batches of one sample, at
the edges of a block's 256 and beyond one pass of the grid, against the means
over the same samples through soma_proposal_grad.

The samples and normals are redrawn here from the documented counters (purpose
5) with FP64 Box-Muller: the normals differ by a few FP32 roundings (2^-22
relative), J and the acceptance by some 1e-5, and a trial position within that
of a cell face may change a sample altogether (at most a few in 40,000)."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import MOVE_LEARNED, System, _abi, workloads

pytestmark = pytest.mark.gpu


def _draws(d, n, step):
    import torch
    ids = np.arange(n, dtype=np.uint64) + np.uint64(step * n)
    ctr = np.zeros((2, n, 4), np.uint32)
    ctr[:, :, 0] = ids & 0xFFFFFFFF
    ctr[:, :, 1] = ids >> 32
    ctr[1, :, 2] = 1
    ctr[:, :, 3] = (5 << 24) | d.replica_id
    key = np.tile(np.array([d.seed & 0xFFFFFFFF, d.seed >> 32], np.uint32), (2 * n, 1))
    c = torch.from_numpy(ctr.reshape(-1, 4).view(np.int32)).cuda()
    k = torch.from_numpy(key.view(np.int32)).cuda()
    o = torch.zeros_like(c)
    torch.cuda.synchronize()
    _abi.soma_philox(c.data_ptr(), k.data_ptr(), o.data_ptr(), 2 * n, None)
    torch.cuda.synchronize()
    r1, r2 = o.cpu().numpy().view(np.uint32).reshape(2, n, 4)
    chain = ((r1[:, 0].astype(np.uint64) << 32) | r1[:, 1]) % d.n_chains

    def radius(w):
        return np.sqrt(-2 * np.log(((w >> 8) + 0.5) * 2.0**-24))

    def angle(w):
        return 2 * np.pi * ((w >> 8) + 0.5) * 2.0**-24

    a, b = angle(r1[:, 3]), angle(r2[:, 1])
    xi = np.stack([radius(r1[:, 2]) * np.cos(a), radius(r1[:, 2]) * np.sin(a),
                   radius(r2[:, 0]) * np.cos(b)], 1)
    return np.stack([chain, r2[:, 3] % d.N], 1).astype(np.uint32), xi.astype(np.float32)


@pytest.mark.parametrize("n", [1, 255, 257, 40000])
def test_training_log_is_the_mean_over_the_batch(cuda_device, n):
    d = workloads.melt_small(n_chains=256, chiN=30.0, move=MOVE_LEARNED)
    s = System(d)
    s.sweep(3)
    W = (0.1 * workloads.random_mlp(11)).astype(np.float32)
    s.set_proposal_weights(W)
    log = s.train_proposal(steps=2, batch=n, sweeps_between=0, lr=0.0)
    J, alpha = [], []
    for step in (0, 1):
        samples, xi = _draws(d, n, step)
        _, j, la = s.proposal_grad(samples, xi, w=W)
        J.append(j.astype(np.float64).mean())
        alpha.append(np.minimum(1.0, np.exp(la.astype(np.float64))).mean())
    s.close()
    for got, want in ((log["mean_J_first"], J[0]), (log["mean_J_last"], J[1]),
                      (log["mean_alpha_last"], alpha[1])):
        assert got == pytest.approx(want, rel=1e-3), (got, want)
