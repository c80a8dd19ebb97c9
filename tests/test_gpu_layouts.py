"""Every form of the layout that the library otherwise takes by size alone (how
many edges a slot's range holds on average, rows classed by degree or not,
fetches by 64 bytes) on small graphs, against the oracle, exactly."""
import pytest

from test_gpu_alias import ref_rows
from test_gpu_parity import assert_same, oracle_rows
from test_gpu_slots import graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppr():
    from paper_1903_11749_gb300 import build as B
    B.build()
    from paper_1903_11749_gb300 import ppr as P
    return P


@pytest.fixture(scope="module")
def refs(oracle):
    """Oracle rows by style and mode, made once (the layout does not change them)."""
    made = {}

    def get(style, mode):
        if (style, mode) not in made:
            g = graph(style, seed=11)
            if mode == "alias":
                made[style, mode] = g, dict(sampler=1), ref_rows(oracle, g, 0.15, 300, 3, topk=8)
            else:
                kw = dict(segments=mode == "segments")
                made[style, mode] = g, kw, oracle_rows(oracle, g, 0.15, 300, 3, topk=8, **kw)
        return made[style, mode]

    return get


@pytest.mark.parametrize("exact", [0, 1])
@pytest.mark.parametrize("lam_bits", [0, 1, 2, 4, 9, 23])
@pytest.mark.parametrize("style", ["equal", "light_runs", "near_2_32", "one_giant"])
def test_rows_under_every_layout(ppr, refs, style, lam_bits, exact):
    ctx = ppr.Context(0)
    ctx.debug_layout(lam_bits, exact)
    wide = style == "one_giant"
    G = None
    for mode in ("prefix", "segments") if wide else ("prefix", "segments", "alias"):
        g, kw, ref = refs(style, mode)
        G = G or ctx.load_graph(g.n, g.row_ptr, g.col, g.w)
        assert G.info().wide == int(wide)
        for far in (-1,) if wide else (0, 1):
            ctx.debug_layout(lam_bits, exact, far)
            r = G.run(alpha=0.15, R=300, seed=3, topk=8, **kw)
            assert_same(r, ref, topk=8)
            r.free()
        r = G.run(alpha=0.15, R=300, seed=3, topk=8, kernel=ppr.KERNEL_PLAIN, **kw)
        assert_same(r, ref, topk=8)
        r = G.run(alpha=0.15, R=300, seed=3, topk=8, stats=True, **kw)
        assert_same(r, ref, topk=8)
    G.free()


@pytest.mark.parametrize("bad", [(-2, -1, -1), (24, -1, -1), (-1, 2, -1), (-1, -1, -2)])
def test_invalid_choices_are_refused(ppr, bad):
    ctx = ppr.Context(0)
    with pytest.raises(ppr.PPRError) as e:
        ctx.debug_layout(*bad)
    assert e.value.code == ppr.PPR_EINVAL
