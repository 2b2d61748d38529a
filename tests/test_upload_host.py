"""The surrogate's upload takes what a conversion by numpy takes: any dtype, order, stride,
byte order and alignment (here to host memory)."""
import numpy as np
import pytest

from paper_2507_12610_gb300 import surrogate


def _forms():
    rng = np.random.default_rng(1)
    a = rng.normal(size=(7, 3))
    rec = np.zeros(7, dtype=[("tag", "i1"), ("x", "f8", 3), ("r", "f4")])  # packed: unaligned
    rec["x"], rec["r"] = a, a[:, 0]
    odd = np.zeros(7, dtype=[("x", "f8", 3), ("r", "f4")])  # 28-byte rows
    odd["x"], odd["r"] = a, a[:, 0]
    frozen = a.copy()
    frozen.flags.writeable = False
    return {
        "f64": a, "f32": a.astype(np.float32), "f16": a.astype(np.float16),
        "int": (10 * a).astype(np.int64), "list": a.tolist(), "fortran": np.asfortranarray(a),
        "every_other": rng.normal(size=(14, 6))[::2, ::2], "reversed": a[::-1],
        "repeated": np.broadcast_to(a[0], (7, 3)), "big_endian": a.astype(">f8"),
        "read_only": frozen, "packed_field": rec["x"], "packed_column": rec["r"],
        "field_of_28_byte_rows": odd["x"], "column_of_28_byte_rows": odd["r"],
        "one": a[:1], "none": a[:0],
    }


@pytest.mark.parametrize("name", _forms().keys())
def test_upload_is_numpy_s_conversion(name):
    a = _forms()[name]
    want = np.ascontiguousarray(a, dtype=np.float32)
    first, got, last = surrogate._upload((np.ones(5), a, np.full(3, 2.0)), "cpu")
    assert np.array_equal(got.numpy(), want) and got.shape == want.shape
    assert got.data_ptr() % 16 == 0 or got.numel() == 0
    assert bool((first == 1).all()) and bool((last == 2).all())
