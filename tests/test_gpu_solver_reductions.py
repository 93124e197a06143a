"""Reductions of the solver at the edges of their launch rules: the last block's lanes per problem (one problem to more
problems than the block has threads for) and the restriction to hats longer than one warp serves."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import dev, host, make_ctx, need_gpu, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle as O
    O.build_library()
    return O


# Both sides solve to a residual of 1e-9 in FP64; a condition number up to 1e5 leaves 1e-4 of the norm (a wrong sum
# moves the result by O(1)).
@pytest.mark.parametrize("curves", [2, 9, 36, 300])
def test_gradients_of_a_batch_match_single_curves(torch, curves):
    from paper_2006_07859_gb300 import tpe
    sizes = [24 + (7 * k) % 41 for k in range(curves)]
    c = S.batch_of_knots(sizes, 3, 41)
    kw = dict(precision=0, precond=tpe.TP_PRECOND_JACOBI, independent=1, cg_rtol=1e-9)
    ctx = make_ctx(c, **kw)
    g = host(tpe.sobolev_gradient(ctx, dev(c.gamma), tpe.tp_differential(ctx, dev(c.gamma)))[0])
    for k in sorted({0, 1, curves // 2, curves - 1}):
        gk, _ = c.curve(k)
        one = S.single(gk)
        cx = make_ctx(one, **kw)
        ref = host(tpe.sobolev_gradient(cx, dev(gk), tpe.tp_differential(cx, dev(gk)))[0])
        assert rel(g[c.vertex_offsets[k]:c.vertex_offsets[k + 1]], ref) <= 1e-4, k


# hats of 600 vertices; the tolerance is that of the FP64 cases of the balanced preconditioner (~1e-8 measured there)
def test_restriction_to_long_hats(torch, orc):
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(900, 6, 4))
    ctx = make_ctx(c, precision=0, precond=tpe.TP_PRECOND_TWOLEVEL_BALANCED, coarse_dim=3)
    r = np.random.default_rng(6).normal(size=(900, 3))
    r -= r.mean(0)
    z = host(tpe.tp_precond_apply(ctx, dev(c.gamma), dev(r)))
    B, B0 = orc.gram_dense(*c.curve(0), 0.75)
    zo = orc.twolevel_balanced_apply(B + B0, 900, 0.75, 3, r)
    assert rel(z - z.mean(0), zo - zo.mean(0)) <= 1e-6
