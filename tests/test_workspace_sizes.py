"""The work-memory sizes never decrease as the input grows: a buffer sized for the
largest input serves every smaller one, and the merge sorts its second-level
samples, whatever their number, in work memory sized for the most there can be."""
import ctypes as C

import pytest

import paper_2404_16517_gb300 as sss
from paper_2404_16517_gb300 import _build


def _sizes(h, n, p, prm):
    return (h.sss_workspace_bytes(n, 30 * n, p, C.byref(prm)), h.sss_batch_workspace_bytes(n, 64, C.byref(prm)),
            h.sss_suffix_workspace_bytes(n, C.byref(prm)))


KNOBS = [{}, {"cta_cap": 64}, {"direct_cap": 8192}, {"cta_cap": 2048, "direct_cap": 2048}, {"bucket_target": 256}]


# around every power of two (defaults that follow the size change there if anywhere),
# by one string and by a sixteenth
@pytest.mark.parametrize("p", [1, 4, 16, 64, 256, 1000])
@pytest.mark.parametrize("knobs", KNOBS)
def test_sizes_do_not_decrease(p, knobs):
    _build.build()
    h = sss.lib()
    prm = sss.params(**knobs)
    ns = sorted({max(1, (1 << k) + d) for k in range(0, 28) for d in (-2, -1, 0, 1, 2, (1 << k) // 16, (1 << k) // 64)})
    last = (0, 0, 0)
    for n in ns:
        cur = _sizes(h, n, p, prm)
        assert all(a <= b for a, b in zip(last, cur)), (n, last, cur)
        last = cur
