"""The records the binding packs whole hold what the ABI's fields say."""
import ctypes as C

import numpy as np
import pytest

from paper_2603_00839_gb300 import _lib as L
from paper_2603_00839_gb300 import api


def _fill(fields, start=1):
    """Distinct values for a struct's fields, flattened in declaration order."""
    out = []
    for name, ty in fields:
        if name == "pad":
            out.append(0)
        elif hasattr(ty, "_fields_"):
            out += _fill(ty._fields_, start + 100 + len(out))
        elif hasattr(ty, "_length_"):
            out += [start + len(out) + i for i in range(ty._length_)]
        else:
            out.append(start + len(out))
    return out


def _read(s):
    out = []
    for name, ty in s._fields_:
        v = getattr(s, name)
        if hasattr(ty, "_fields_"):
            out += _read(v)
        elif hasattr(ty, "_length_"):
            out += list(v)
        elif ty is C.c_void_p:
            out.append(v)
        elif hasattr(ty, "contents"):
            out.append(C.cast(v, C.c_void_p).value)
        else:
            out.append(v)
    return out


@pytest.mark.parametrize("fmt,cls", [(api._FACTOR, L.Factor), (api._OPTS, L.Opts), (api._PROBLEM, L.Problem),
                                     (api._INFO, L.Info)])
def test_record_formats_match_the_fields(fmt, cls):
    vals = _fill(cls._fields_)
    s = cls()
    fmt.pack_into(s, 0, *vals)
    assert _read(s) == vals
    assert list(fmt.unpack(s)) == vals


@pytest.mark.parametrize("big", [63, 65])   # 65 x 65 values: passed where they lie
def test_factor_arrays(big):
    rng = np.random.default_rng(big)
    M, N = rng.standard_normal((big, big)), rng.standard_normal((3, 3))
    A = [api.banded(1, 9, rng.standard_normal(5)), api.identity(2, 7), api.dense(4, M)]
    B = [api.banded(np.int64(2), np.int32(7), rng.standard_normal(1)), api.dense(3, N.T)]
    (a, none, b), keep = api._factor_arrays(A, (), B)
    assert none is None and len(a) == 3 and len(b) == 2
    for arr, fs in ((a, A), (b, B)):
        for r, f in zip(arr, fs):
            assert (r.mode, r.kind, r.n, r.radius) == (f.mode, f.kind, f.n, f.radius)
            assert bool(r.taps) == (f.taps is not None) and bool(r.dense) == (f.matrix is not None)
            if f.taps is not None:
                assert list(r.taps[:len(f.taps)]) == list(f.taps)
            if f.matrix is not None:
                assert list(r.dense[:f.n * f.n]) == list(f.matrix.ravel(order="F"))


@pytest.mark.parametrize("dims", [(5,), (4, 3), (1, 6, 2), (3, 0), (2, 3, 1, 4)])
def test_empty_is_column_major(dims):
    torch = pytest.importorskip("torch")
    t = api.empty(dims, torch.float64, "cpu")
    r = torch.empty(tuple(reversed(dims)), dtype=torch.float64).permute(*reversed(range(len(dims))))
    assert t.shape == r.shape and t.stride() == r.stride() and t.dtype == r.dtype
