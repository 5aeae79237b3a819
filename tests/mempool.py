"""The device's stream-ordered memory pool, by the driver API: what the library's calls take from it."""
import contextlib
import ctypes

_USED, _USED_HIGH = 7, 8


class _Location(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("id", ctypes.c_int)]


class _Props(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location", _Location),
                ("win32", ctypes.c_void_p), ("max_size", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]


def _cu(name, *args):
    rc = getattr(ctypes.CDLL("libcuda.so.1"), name)(*args)
    assert rc == 0, (name, rc)


def _current():
    pool = ctypes.c_void_p()
    _cu("cuDeviceGetMemPool", ctypes.byref(pool), 0)
    return pool


def used():
    v = ctypes.c_uint64()
    _cu("cuMemPoolGetAttribute", _current(), _USED, ctypes.byref(v))
    return v.value


def reset_peak():
    _cu("cuMemPoolSetAttribute", _current(), _USED_HIGH, ctypes.byref(ctypes.c_uint64(0)))


def peak():
    v = ctypes.c_uint64()
    _cu("cuMemPoolGetAttribute", _current(), _USED_HIGH, ctypes.byref(v))
    return v.value


@contextlib.contextmanager
def limited(max_bytes):
    """Allocations inside come from a pool of their own that holds max_bytes at most (a request beyond it
    fails as on a full device); what was allocated before stays where it is."""
    props = _Props(alloc_type=1, location=_Location(1, 0), max_size=max_bytes)  # pinned, device 0
    pool, before = ctypes.c_void_p(), _current()
    _cu("cuMemPoolCreate", ctypes.byref(pool), ctypes.byref(props))
    _cu("cuDeviceSetMemPool", 0, pool)
    try:
        yield
    finally:
        _cu("cuDeviceSetMemPool", 0, before)
        _cu("cuMemPoolDestroy", pool)
