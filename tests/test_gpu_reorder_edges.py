"""The cloud reorder at its edges: tile and scan boundaries, clouds that share
one key or one digit, infinities, rows that start on no 16-byte boundary, and
the gather without packed records (taken when the scratch for them cannot be
had, here because the memory pool is capped)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TILE = 8192


def _keys(xyz):
    dim, n = xyz.shape
    key = np.zeros(n, dtype=np.int64)
    for d in range(dim):
        v = xyz[d]
        lo, hi = np.float32(np.nanmin(v)), np.float32(np.nanmax(v))
        with np.errstate(invalid="ignore", over="ignore"):
            ext = np.float32(hi - lo)
            scale = np.float32(1024.0) / ext if ext > 0 else np.float32(0.0)
            u = ((v - lo).astype(np.float32) * scale).astype(np.float32)
        q = np.where(u >= 0, np.minimum(u, np.float32(1023.0)), 0).astype(np.int64)
        for b in range(10):
            key |= ((q >> b) & 1) << (dim * b + d)
    return key


def _cloud(kind, n, dim):
    rng = np.random.default_rng([n, dim])
    x = rng.normal(size=(dim, n)).astype(np.float32)
    if kind == "one key":
        x[:] = 0.25
    elif kind == "two ends":                 # digits 0 and 1023 only
        x[:] = rng.integers(0, 2, (1, n)).astype(np.float32)
    elif kind == "sorted":
        x = x[:, np.argsort(_keys(x), kind="stable")]
    elif kind == "infinite":
        x[0, n // 2] = np.inf
        x[dim - 1, n // 3] = -np.inf
    return np.ascontiguousarray(x)


def _check(torch, cfs, x, offset=0, want_perm=True):
    dim, n = x.shape
    fn = (np.arange(n) % 251).astype(np.uint8)
    buf = torch.empty(dim * n + offset, dtype=torch.float32, device="cuda")
    d = buf[offset:].view(dim, n)
    d.copy_(torch.from_numpy(x))
    got = cfs.pointcloud_reorder(d, torch.from_numpy(fn).cuda(), want_perm=want_perm)
    torch.cuda.synchronize()
    order = np.argsort(_keys(x), kind="stable")
    assert np.array_equal(got[0].cpu().numpy(), x[:, order], equal_nan=True)
    assert np.array_equal(got[1].cpu().numpy(), fn[order])
    if want_perm:
        assert np.array_equal(got[2].cpu().numpy(), order)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("kind,n", [("random", 1), ("random", 2), ("random", 31),
                                    ("random", TILE - 1), ("random", TILE), ("random", TILE + 1),
                                    ("random", 33 * TILE + 5), ("one key", 3 * TILE + 7),
                                    ("two ends", 2 * TILE + 1), ("sorted", 70001),
                                    ("infinite", 20000)])
def test_reorder_equals_a_stable_sort(kind, n, dim):
    torch = pytest.importorskip("torch")
    from paper_2606_02226_gb300 import cfs
    _check(torch, cfs, _cloud(kind, n, dim), offset=n % 4, want_perm=n % 2 == 0)


class _PoolProps(ctypes.Structure):          # cudaMemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int),
                ("location_type", ctypes.c_int), ("location_id", ctypes.c_int),
                ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@pytest.mark.parametrize("dim", [2, 3])
def test_reorder_without_room_for_records(dim):
    torch = pytest.importorskip("torch")
    from paper_2606_02226_gb300 import cfs
    n = (1 << 23) + 3                        # records 134 MB, the rest 105 MB at most
    x = _cloud("random", n, dim)
    cfs.lib()
    rt = ctypes.CDLL("libcudart.so.13")
    dev = torch.cuda.current_device()
    torch.zeros(1, device="cuda")
    old, pool = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaDeviceGetMemPool(ctypes.byref(old), dev) == 0
    props = _PoolProps(1, 0, 1, dev, None, 112 << 20, 0)
    assert rt.cudaMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert rt.cudaDeviceSetMemPool(dev, pool) == 0
    try:
        p = ctypes.c_void_p()
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        # the cap holds: the records would not fit
        assert rt.cudaMallocAsync(ctypes.byref(p), ctypes.c_size_t(200 << 20), stream) == 2
        rt.cudaGetLastError()
        _check(torch, cfs, x)
        _check(torch, cfs, x, want_perm=False)
    finally:
        torch.cuda.synchronize()
        assert rt.cudaDeviceSetMemPool(dev, old) == 0
        rt.cudaMemPoolDestroy(pool)
