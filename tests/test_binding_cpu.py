"""The binding's int32 arguments: what numpy took is taken with the same values, what it refused is
refused (no GPU: the conversion alone)."""
import numpy as np
import pytest

import __graft_entry__ as g

g.build()
from paper_2607_17715_gb300 import c2kv  # noqa: E402


@pytest.mark.parametrize("x", [[0, 4], (1, 2, 3), [np.int64(3), np.int32(-4)], [True, 2], [1.0, 2.0], [[1, 2], [3, 4]], [],
                               [2 ** 31 - 1, -2 ** 31], np.arange(4), np.arange(6)[::2], np.array([5], dtype=np.int64)])
def test_i32_values(x):
    want = np.asarray(x, dtype=np.int32)
    keep, ptr = c2kv._i32(x)
    assert [ptr[i] for i in range(want.size)] == want.ravel().tolist()
    assert len(keep) == len(want)


@pytest.mark.parametrize("x", [[2 ** 31], (-2 ** 31 - 1,), [0, 2 ** 70]])
def test_i32_refuses_what_does_not_fit(x):
    with pytest.raises(OverflowError):
        c2kv._i32(x)


def test_i32_none():
    assert c2kv._i32(None) == (None, None)
