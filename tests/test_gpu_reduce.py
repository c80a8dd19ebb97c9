"""The reduction of a source's endpoints (rows and top-k) against the oracle at
the walk counts where its kernels change (a register a lane more, a block per
source) and for top-k lengths below, at and above the number of distinct
endpoints.  Counts are integers: every comparison is exact."""
import pytest

from paper_1903_11749_gb300 import inputs as I
from test_gpu_parity import assert_same, ctx, oracle_rows, ppr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 32, 33, 64, 65, 128, 129, 255, 256, 257, 512, 513, 1024, 1025, 2047, 2049, 4096])
def test_rows_and_topk_at_every_size(ppr, ctx, oracle, R):  # noqa: F811
    # 4,000 nodes: mostly distinct endpoints; 9 nodes: a handful met very often;
    # node 8 of the small one and 200 of the large one restart at themselves
    for g in (I.random_small_graph(4000, 9000, seed=3, dangling=200), I.random_small_graph(9, 30, seed=4, dangling=1)):
        G = ctx.load_graph(g.n, g.row_ptr, g.col, g.w)
        b, e = max(0, g.n - 230), g.n
        ref = oracle_rows(oracle, g, 0.12, R, 6, s_begin=b, s_end=e, topk=1)
        for k in (1, 31, 33, 300, 4096):
            ref["topk"] = oracle.topk(*ref["rows"], k)
            assert_same(G.run(alpha=0.12, R=R, seed=6, src_begin=b, src_end=e, topk=k), ref, topk=k)
        G.free()
