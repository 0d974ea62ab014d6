"""ldl_load refuses files that are no checkpoint before it touches a GPU (CPU)."""
import ctypes
import os
import shutil
import struct

import pytest

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="needs nvcc")


def _file(path, n, level):
    """A one-level undirected checkpoint of n vertices; `level` gives the level's
    arrays as (count, bytes)."""
    from paper_2502_18497_gb300 import ldl
    p = ldl.make_params()
    out = b"LDLHIER1" + bytes(p) + struct.pack("<qi", n, 0) + struct.pack("<qqqQ", 0, 0, 0, 0)
    for count, width in ((n, 8), (0, 8), (n, 8)):
        out += struct.pack("<q", count) + bytes(count * width)
    for count, body in level:
        out += struct.pack("<q", count) + body
    path.write_bytes(out)


def _load(path):
    from paper_2502_18497_gb300 import ldl
    lib = ldl.load()
    h = ctypes.c_void_p()
    st = lib.ldl_load(os.fsencode(str(path)), None, ctypes.byref(h))
    assert not h.value
    return st, lib.ldl_last_error(None).decode()


@pytest.mark.parametrize("count", [3, 1 << 20, 1 << 39, 1 << 41, -1])
def test_counts_beyond_the_file(tmp_path, count):
    from paper_2502_18497_gb300 import ldl
    n = 4
    arrays = [(n, bytes(4 * n))] * 3 + [(n, bytes(8 * n)), (0, b""), (n, bytes(n)), (n + 1, bytes(8 * (n + 1)))]
    _file(tmp_path / "h", n, arrays + [(count, b"\0" * 8)])
    st, msg = _load(tmp_path / "h")
    assert st == ldl.LDL_E_INVALID and "truncated or corrupt" in msg


def test_rows_that_do_not_fit_their_table(tmp_path):
    from paper_2502_18497_gb300 import ldl
    n = 4
    arrays = [(n, bytes(4 * n))] * 3 + [(n, bytes(8 * n)), (0, b""), (n, bytes(n)), (n + 1, bytes(8 * (n + 1))),
                                        (2, bytes(8)), (2, bytes(16)), (0, b""), (0, b"")]
    _file(tmp_path / "h", n, arrays)
    st, msg = _load(tmp_path / "h")
    assert st == ldl.LDL_E_INVALID and "row table inconsistent" in msg


def test_no_checkpoint(tmp_path):
    from paper_2502_18497_gb300 import ldl
    (tmp_path / "h").write_bytes(b"")
    assert _load(tmp_path / "h")[0] == ldl.LDL_E_INVALID
    assert _load(tmp_path / "absent")[0] == ldl.LDL_E_INVALID
