"""soma_set_positions from device memory at any address: 16-byte and 4-byte
boundaries (read by the kernel that copies and checks) and others (copied first),
whole numbers of four particles and not; values out of range are refused from each."""
import ctypes

import numpy as np
import pytest

from paper_1711_03828_gb300 import SomaError, System, SystemDesc, _abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_chains", [64, 65])   # 384 particles; 390, not a multiple of four
@pytest.mark.parametrize("offset", [0, 4, 8, 1, 2, 6, 13])
def test_positions_from_any_device_address(cuda_device, n_chains, offset):
    import torch
    d = SystemDesc(n_chains=n_chains, N=6, box_Re=(1.0, 1.0, 1.0), grid=(6, 6, 6), seed=4)
    s = System(d)
    pos = np.random.default_rng(offset).uniform(-7, 13, (3, d.M)).astype(np.float32)
    buf = torch.zeros(16 + pos.nbytes, dtype=torch.uint8, device=cuda_device)
    buf[offset:offset + pos.nbytes] = torch.from_numpy(pos.reshape(-1).view(np.uint8)).to(cuda_device)
    torch.cuda.synchronize()
    src = ctypes.c_void_p(buf.data_ptr() + offset)
    _abi.soma_set_positions(s.h, src, 3 * d.M, 1)
    np.testing.assert_array_equal(s.get_positions(), pos)
    bad = pos.copy()
    bad[2, -1] = np.inf
    buf[offset:offset + pos.nbytes] = torch.from_numpy(bad.reshape(-1).view(np.uint8)).to(cuda_device)
    torch.cuda.synchronize()
    with pytest.raises(SomaError) as e:
        _abi.soma_set_positions(s.h, src, 3 * d.M, 1)
    assert e.value.status == _abi.SOMA_EINVAL
