"""The FP32 tile factor's loads of diagonal-tile panels stay inside the matrix
(host arithmetic, no GPU): M has rows padded to 16 columns, a panel spans 32, so
for m mod 32 in 1 .. 16 the last panel is wider than the row.  No result can show
a load past the end (what it fetches lies above the diagonal), so the index
arithmetic is checked itself."""
import ctypes

import pytest


@pytest.mark.parametrize("first", range(1, 1058, 132))
def test_panel_loads_stay_inside_the_matrix(first):
    from paper_1502_03543_gb300 import build as B
    B.build()
    from paper_1502_03543_gb300 import _native as N
    row_end = ctypes.c_int64()
    for m in range(first, first + 132):
        ldm = (m + 15) // 16 * 16
        end = N.lib().pdas_chol_panel_extent(m, ldm, ctypes.byref(row_end))
        assert m <= row_end.value <= ldm and (m - 1) * ldm + m <= end <= m * ldm, m
