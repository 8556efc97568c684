"""Edit lists in every memory layout reach the library as rows (op, tet, tet2), in order (no GPU: the
library is a stand-in that reads what the binding passes)."""
import ctypes as C

import numpy as np
import pytest

import paper_2605_11673_gb300 as P

H = 12345  # a handle that only the stand-in sees

ROWS = [np.array([[0, 5, -1], [0, 9, -1], [0, 2, -1]], np.int32), np.array([[1, 7, -1], [2, 1, 3]], np.int32)]


def _sliced(e):
    wide = np.zeros((2 * len(e), 5), np.int32)
    wide[::2, 1:4] = e
    return wide[::2, 1:4]


LAYOUTS = {
    "rows": lambda e: e,
    "columns": lambda e: np.array([e[:, 0], e[:, 1], e[:, 2]], np.int32).T,
    "fortran": np.asfortranarray,
    "sliced": _sliced,
    "reversed": lambda e: e[::-1].copy()[::-1],
    "columns reversed": lambda e: np.ascontiguousarray(e[:, ::-1])[:, ::-1],
    "int64": lambda e: e.astype(np.int64),
    "flat": lambda e: e.reshape(-1),
    "lists": lambda e: e.tolist(),
    "read-only": lambda e: np.frombuffer(e.tobytes(), np.int32).reshape(-1, 3),
}


class _Library:
    def __init__(self, k):
        self.k = k

    def _read(self, p, n):
        addr = p.value if isinstance(p, C.c_void_p) else p
        return np.array((C.c_int32 * (3 * n)).from_address(addr)).reshape(n, 3) if n else np.zeros((0, 3), np.int32)

    def sta_batch_apply_edits(self, h, counts, p, stream):
        assert h == H
        self.counts = list(counts[:self.k])
        self.got = self._read(p, sum(self.counts))
        return P.STA_OK

    def sta_apply_edits(self, h, p, n, stream):
        assert h == H
        self.got = self._read(p, n)
        return P.STA_OK


def _batch(monkeypatch, parts):
    lib = _Library(len(parts))
    monkeypatch.setattr(P, "load_library", lambda: lib)
    monkeypatch.setitem(P._fixed, H, {"k": len(parts)})
    P.sta_batch_apply_edits(H, parts, stream=0)
    return lib


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("lists", [ROWS, ROWS[:1], [ROWS[0], ROWS[0][:0], ROWS[1]]])
def test_batch_lists(monkeypatch, layout, lists):
    lib = _batch(monkeypatch, [LAYOUTS[layout](e) for e in lists])
    assert lib.counts == [len(e) for e in lists]
    assert np.array_equal(lib.got, np.concatenate(lists))


def test_batch_of_mixed_layouts(monkeypatch):
    parts = [LAYOUTS[name](ROWS[i % 2]) for i, name in enumerate(LAYOUTS)]
    lib = _batch(monkeypatch, parts)
    assert np.array_equal(lib.got, np.concatenate([ROWS[i % 2] for i in range(len(LAYOUTS))]))


@pytest.mark.parametrize("layout", LAYOUTS)
def test_single_list(monkeypatch, layout):
    lib = _Library(1)
    monkeypatch.setattr(P, "load_library", lambda: lib)
    P.sta_apply_edits(H, LAYOUTS[layout](ROWS[0]), stream=0)
    assert np.array_equal(lib.got, ROWS[0])


def test_pointer_of_columns_is_refused():
    with pytest.raises(ValueError):
        P._ptr(np.asfortranarray(ROWS[0]))
