"""Nuclear attraction over the whole range of T = zeta |P - C|^2 that finite
inputs reach: the Boys table below 64, the asymptotic form with and without an
FP32 seed above."""
import numpy as np
import pytest

import molgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required")
    import paper_2407_21445_gb300 as fk
    return torch, fk


@pytest.mark.parametrize("log10_r", [4, 9, 18.9, 19.2, 20, 30, 38.4, 40, 50, 70, 100, 150])
def test_far_nucleus(env, log10_r):
    """A charge at distance R acts as -Z/R on every product of functions, up to
    (size / R)^2 of it and, for products without overlap, size / R of it."""
    torch, fk = env
    rng = np.random.Generator(np.random.PCG64(42))
    bas = molgen.random_shells(rng, [0, 1, 2, 3], spread=1.0, kmax=3)
    r = 10.0 ** log10_r
    S, _, V = (x.cpu().numpy() for x in fk.fock_one_electron(bas, [3.0], [[r / 3, 2 * r / 3, -2 * r / 3]]))
    assert np.abs(V * r / 3.0 + S).max() <= 40.0 / r + 1e-13


def test_around_the_end_of_the_table(env):
    """Nuclei at distances on both sides of T = 64."""
    torch, fk = env
    bas = molgen.single_shell_basis([(l, np.zeros(3), [0.5], [1.0]) for l in (0, 1, 2, 3)])
    d = np.sqrt(64.0 * (1.0 + np.array([-1e-2, -1e-9, -1e-15, 0.0, 1e-15, 1e-9, 1e-2])))
    xyz = np.stack([d, 0 * d, 0 * d], axis=1)
    Z = np.arange(1.0, len(d) + 1)
    _, _, V = fk.fock_one_electron(bas, Z, xyz)
    assert np.abs(V.cpu().numpy() - oracle.nuclear(bas, Z, xyz)).max() < 1e-11


def test_little_device_memory(env):
    """A memory pool that ends at 32 MiB, set as the device's: the per-primitive
    values of 200 contracted d shells (five times that) go in small pieces."""
    import ctypes
    torch, fk = env

    class Props(ctypes.Structure):  # CUmemPoolProps
        _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("loc_type", ctypes.c_int),
                    ("loc_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                    ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]

    rng = np.random.Generator(np.random.PCG64(43))
    bas = molgen.single_shell_basis([(2, rng.uniform(-6, 6, 3), rng.uniform(0.2, 4.0, 8), rng.uniform(0.2, 1.0, 8))
                                     for _ in range(200)])
    nuclei = rng.uniform(-6, 6, (2, 3))
    ref = fk.fock_one_electron(bas, [1.0, 8.0], nuclei)
    assert 20100 * 64 * 36 * 3 * 8 > 5 * (32 << 20)
    cu = ctypes.CDLL("libcuda.so.1")
    pool, old = ctypes.c_void_p(), ctypes.c_void_p()
    dev = torch.cuda.current_device()
    props = Props(alloc_type=1, loc_type=1, loc_id=dev, max_size=32 << 20)
    torch.cuda.synchronize()
    assert cu.cuDeviceGetMemPool(ctypes.byref(old), dev) == 0
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(dev, pool) == 0
    try:
        out = fk.fock_one_electron(bas, [1.0, 8.0], nuclei)
        torch.cuda.synchronize()
    finally:
        assert cu.cuDeviceSetMemPool(dev, old) == 0
        assert cu.cuMemPoolDestroy(pool) == 0
    for a, b in zip(out, ref):
        assert float(b.abs().max()) > 0 and float((a - b).abs().max()) <= 1e-13 * float(b.abs().max())
