"""Rows into device arrays: row starts at any address, and what a capacity that
is too small leaves untouched."""
import ctypes as C

import numpy as np
import pytest

from paper_1903_11749_gb300 import inputs as I
from paper_1903_11749_gb300 import ppr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [5, 4097])
@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("fits", [True, False])
def test_row_starts_at_any_address(S, shift, fits):
    """row_ptr need not lie on eight bytes (shift counts four-byte words)."""
    import torch
    g = I.random_small_graph(5000, 20000, seed=3, dangling=50)
    ctx = ppr.Context(0)
    G = ctx.load_graph(g.n, g.row_ptr, g.col, g.w)
    r = G.run(alpha=0.2, R=20, seed=2, src_end=S)
    rp, col, cnt = r.sparse_rows()
    out = torch.full((2 * (S + 1) + 4,), -7, dtype=torch.int32, device="cuda")
    dcol, dcnt = (torch.full((len(col),), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    n = C.c_int64()
    code = ppr.lib().ppr_sparse_rows(r.h, out.data_ptr() + 4 * shift, dcol.data_ptr(), dcnt.data_ptr(),
                                     len(col) if fits else len(col) - 1, C.byref(n), ppr.PPR_PTRS_DEVICE)
    assert code == (0 if fits else ppr.PPR_ERANGE) and n.value == len(col)
    words = out.cpu().numpy()
    assert np.array_equal(words[shift: shift + 2 * (S + 1)].copy().view(np.int64), rp)
    assert (words[:shift] == -7).all() and (words[shift + 2 * (S + 1):] == -7).all()
    want = (col, cnt) if fits else (np.full(len(col), -7),) * 2
    assert np.array_equal(dcol.cpu().numpy(), want[0]) and np.array_equal(dcnt.cpu().numpy().astype(want[1].dtype), want[1])
