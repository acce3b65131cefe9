"""The refinement's workspace is a matter of the block length alone: one workspace serves descriptors of any phase order
and number of steps."""
import ctypes as C

import pytest

from paper_2110_13115_gb300 import _native as N


@pytest.mark.parametrize("n", [1 << 10, 1 << 13, 1 << 20])
def test_size(n):
    lib = N.load()
    sizes = {lib.rb_refine_workspace_bytes(C.byref(N.rb_refine_desc(2048.0, n, f, pn, steps, 1e-3, 0.05)))
             for f in (10.0, 30.0) for pn in (0, 2, 3) for steps in (0, 20)}
    assert len(sizes) == 1
    assert 52 * n <= sizes.pop() <= 52 * n + n // 16 + 4096
