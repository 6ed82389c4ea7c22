"""The batch's field update in its written roundings: fields of every storage type
and both interaction options equal the same operations in numpy, bit for bit, and
under K^1 those of the same systems alone."""
import numpy as np
import pytest

from paper_1711_03828_gb300 import GRID_BF16, GRID_F16, GRID_F32, Batch, System, SystemDesc

pytestmark = pytest.mark.gpu

f32 = np.float32


def _fma(a, b, c):
    """FP32 fused multiply-add: exact in extended precision, rounded once."""
    return (np.longdouble(a) * np.longdouble(b) + np.longdouble(c)).astype(f32)


def _descs(**kw):
    return [SystemDesc(n_chains=1500 + 130 * i, N=(16, 32, 64)[i % 3], f=0.4, box_Re=(4.0, 3.0, 2.0), grid=(24, 18, 12),
                       chiN=15.0 + 5 * i, kappaN=50.0 + i, seed=3, replica_id=i, **kw) for i in range(5)]


def _fields(d, density, rho_cell):
    inv, kappa0, half = f32(1.0 / rho_cell), f32(d.kappaN / d.N), f32(0.5 * d.chiN / d.N)
    phi = [((density & 0xFFFF).astype(f32) * inv).astype(f32), ((density >> 16).astype(f32) * inv).astype(f32)]
    comp = (kappa0 * ((phi[0] + phi[1]).astype(f32) - f32(1)).astype(f32)).astype(f32)
    if d.hamiltonian:
        chi0 = f32(2) * half
        return _fma(chi0, phi[1], comp), _fma(chi0, phi[0], comp)
    diff = (phi[0] - phi[1]).astype(f32)
    return _fma(-half, diff, comp), _fma(half, diff, comp)


def _stored(w, dtype):
    """w rounded once to the storage type, to nearest even."""
    if dtype == GRID_F32:
        return w
    import torch
    return torch.from_numpy(w).to(torch.bfloat16 if dtype == GRID_BF16 else torch.float16).float().numpy()


@pytest.mark.parametrize("dtype", [GRID_F32, GRID_BF16, GRID_F16])
@pytest.mark.parametrize("ham", [0, 1])
def test_fields_in_their_written_roundings(cuda_device, ham, dtype):
    b = Batch(_descs(hamiltonian=ham, grid_dtype=dtype))
    for cycles in (1, 16):
        b.sweep(cycles)
        for m in b.members:
            want = _fields(m.desc, m.get_density(), m.parameters()["rho_cell"])
            for got, w in zip(m.get_fields(), want):
                np.testing.assert_array_equal(got, _stored(w, dtype))
    b.close()


@pytest.mark.parametrize("dtype", [GRID_F32, GRID_BF16, GRID_F16])
def test_product_option_fields_are_those_of_the_systems_alone(cuda_device, dtype):
    descs = _descs(hamiltonian=1, grid_dtype=dtype)
    b = Batch(descs)
    alone = [System(d) for d in descs]
    for cycles in (1, 16):
        b.sweep(cycles)
        for m, s in zip(b.members, alone):
            s.sweep(cycles)
            np.testing.assert_array_equal(m.get_density(), s.get_density())
            np.testing.assert_array_equal(m.get_fields(), s.get_fields())
    b.close()
