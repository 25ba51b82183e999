"""The memory a weight fit takes per row: the scaled counts and, per model, the row factors and
one array that holds beta and then the residuals."""
import ctypes

import pytest

from paper_1604_04997_gb300 import binding as B


@pytest.mark.parametrize("k", [1, 5, 12, 13, 31, 32])
@pytest.mark.parametrize("M", [1, 2, 3, 5, 8, 17, 64])
def test_scratch_per_row(k, M):
    import __graft_entry__
    __graft_entry__.build_library()
    f = B.lib().pmx_fit_scratch
    f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_int64, ctypes.c_int, ctypes.c_int]
    per_row = (f(3_000_000, k, M) - f(1_000_000, k, M)) / 2_000_000
    # float-float counts of k columns, four float-float values per model (24 bytes of padding
    # to 16-byte pieces are covered by what beta and the residuals share, from three models on)
    assert per_row <= 8 * k + 32 * M + (56 if M < 3 else 0)
