"""Edges of the blocking of the pair passes: 64-row sections, 128-row tiles and 256-row super-blocks of the
symmetric passes, the short source chunks of the gather passes, edges whose neighbours lie in other tiles (a
curve with its edges shuffled) and the passes a new context picks by size, all against the FP64 oracle.

Tolerances are those of the same quantities elsewhere in the suite: relative to the largest entry 1e-6 for the
mixed energy rows and apply, 1e-5 for the mixed differential, 1e-10 for FP64."""
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


def _check(torch, orc, ctx, c, prec, tol):
    from paper_2006_07859_gb300 import tpe
    g = dev(c.gamma)
    rows = torch.empty(c.n_edges, dtype=torch.float64, device="cuda")
    E = host(tpe.tp_energy(ctx, g, rows=rows))
    dE = host(tpe.tp_differential(ctx, g))
    u = np.random.default_rng(5).normal(size=(c.n_vertices, 3))
    Au = host(tpe.sobolev_apply(ctx, g, dev(u)))
    for k in range(ctx.n_problems):
        if ctx.n_problems == 1:
            gk, ek, v, e = c.gamma, c.edges, slice(None), slice(None)
        else:
            gk, ek = c.curve(k)
            v = slice(c.vertex_offsets[k], c.vertex_offsets[k + 1])
            e = slice(c.edge_offsets[k], c.edge_offsets[k + 1])
        ref = orc.energy_rows(gk, ek, np.arange(len(ek), dtype=np.int32))
        if not np.abs(ref).max() > 0:
            assert np.all(host(rows)[e] == 0) and np.all(dE[v] == 0) and np.all(Au[v] == 0)
            continue
        assert rel(host(rows)[e], ref) <= tol["energy"], (k, len(ek))
        assert abs(E[k] - ref.sum()) <= tol["energy"] * ref.sum()
        if prec != 1:   # the plain FP32 differential has its own test
            assert rel(dE[v], orc.differential(gk, ek)) <= tol["diff"], (k, len(ek))
        assert rel(Au[v], orc.gram_apply(gk, ek, 0.75, u[v])) <= tol["apply"], (k, len(ek))


MIXED = {"energy": 1e-6, "diff": 1e-5, "apply": 1e-6}
FP64 = {"energy": 1e-10, "diff": 1e-10, "apply": 1e-10}


@pytest.mark.parametrize("n", [3, 4, 5, 31, 63, 64, 65, 127, 128, 129, 192, 193, 255, 256, 257, 384, 385, 640])
@pytest.mark.parametrize("variant", [0, 1])
def test_mixed_passes_at_block_edges(torch, orc, n, variant):
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(n, 4, 40 + n))
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_energy_variant(ctx, variant)
    tpe.tp_set_diff_variant(ctx, variant)
    tpe.tp_set_apply_variant(ctx, variant)
    _check(torch, orc, ctx, c, 2, MIXED)


@pytest.mark.parametrize("n", [4, 130, 257, 900])
def test_fp64_passes_in_short_chunks(torch, orc, n):
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(n, 4, 60 + n))
    _check(torch, orc, make_ctx(c, precision=tpe.TP_FP64, precond=tpe.TP_PRECOND_JACOBI), c, 0, FP64)


@pytest.mark.parametrize("variant", [0, 1])
def test_shuffled_edges_find_their_neighbours(torch, orc, variant):
    """The two neighbours of an edge lie anywhere in the edge order; some edges are flipped too."""
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(700, 4, 3))
    rng = np.random.default_rng(8)
    e = c.edges[rng.permutation(c.n_edges)].copy()
    flip = rng.random(len(e)) < 0.3
    e[flip] = e[flip][:, ::-1]
    c = S.Curves(c.gamma, e, c.vertex_offsets, c.edge_offsets)
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_energy_variant(ctx, variant)
    tpe.tp_set_diff_variant(ctx, variant)
    tpe.tp_set_apply_variant(ctx, variant)
    _check(torch, orc, ctx, c, 2, MIXED)


@pytest.mark.parametrize("prec", [1, 2])
def test_new_context_of_many_ragged_curves(torch, orc, prec):
    """Enough work for the symmetric passes by default: 209 curves of 4 to 700 edges."""
    from paper_2006_07859_gb300 import tpe
    sizes = [4, 5, 63, 64, 65, 128, 129, 255, 256, 257, 300, 513, 700] * 16 + [700]
    c = S.batch_of_knots(sizes, 4, 77)
    ctx = make_ctx(c, precision=prec, precond=tpe.TP_PRECOND_JACOBI, independent=1)
    # plain FP32 positions: the suite's FP32 bar for the energy, and 1e-4 of the largest entry for the apply
    # (positions rounded to 6e-8 of the curve's size against edges of 1e-2 of it)
    _check(torch, orc, ctx, c, prec, MIXED if prec == 2 else {"energy": 1e-4, "diff": 1.0, "apply": 1e-4})


@pytest.mark.parametrize("m", [1, 2, 3, 5])
def test_multi_field_apply_on_the_symmetric_pass(torch, orc, m):
    """Fields two by two and an odd last one, per field against the oracle and against the single apply (1e-6 of
    the largest entry each, the mixed apply's bar)."""
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(449, 4, 12))
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_apply_variant(ctx, 1)
    U = np.random.default_rng(m).normal(size=(m, c.n_vertices, 3))
    AU = host(tpe.sobolev_apply_multi(ctx, dev(c.gamma), dev(U)))
    for f in range(m):
        assert rel(AU[f], orc.gram_apply(c.gamma, c.edges, 0.75, U[f])) <= 1e-6
        assert rel(AU[f], host(tpe.sobolev_apply(ctx, dev(c.gamma), dev(U[f])))) <= 1e-6


def test_accurate_apply_after_a_change_of_exponents(torch, orc):
    """The accurate apply's work list follows the exponents of the context (tolerance of its own tests)."""
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(300, 4, 21))
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    u = np.random.default_rng(2).normal(size=(c.n_vertices, 3))
    for alpha, beta in ((2.0, 4.5), (3.0, 6.0), (2.0, 4.5)):
        ctx.set_params(alpha=alpha, beta=beta)
        ref = orc.gram_apply(c.gamma, c.edges, orc.sigma_of(alpha, beta), u)
        assert rel(host(tpe.sobolev_apply_accurate(ctx, dev(c.gamma), dev(u))), ref) <= 1e-11
        assert rel(host(tpe.sobolev_apply(ctx, dev(c.gamma), dev(u))), ref) <= 1e-5


# Both forms add the same FP32 pair terms (about 1e-6 of the largest entry each); a lost or doubled pair of the smallest
# curves moves a row by 1e-2.
@pytest.mark.parametrize("n,k", [(2600, 1), (300, 16), (65, 300), (3950, 1)])
def test_new_context_between_the_passes(torch, n, k):
    """Either side of the work from which a new context runs each pass in symmetric form, with half tiles per item
    (152 SMs: 2,587 and 3,899 edges of one curve), against the gather form."""
    from paper_2006_07859_gb300 import tpe
    c = S.batch_of_knots([n] * k, 5, 31)
    g, u = dev(c.gamma), dev(np.random.default_rng(5).normal(size=(c.n_vertices, 3)))
    out = []
    for gather in (False, True):
        ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI, independent=1)
        if gather:
            tpe.tp_set_energy_variant(ctx, 0)
            tpe.tp_set_diff_variant(ctx, 0)
            tpe.tp_set_apply_variant(ctx, 0)
        rows = torch.empty(c.n_edges, dtype=torch.float64, device="cuda")
        tpe.tp_energy(ctx, g, rows=rows)
        out.append([host(rows), host(tpe.tp_differential(ctx, g)), host(tpe.sobolev_apply(ctx, g, u))])
    for new, old in zip(*out):
        assert rel(new, old) <= 1e-5


def test_default_passes_return_with_the_exponents(torch):
    """5,000 edges: a new context runs the symmetric passes.  Other exponents have none; back at (2, 4.5) the context
    runs them again, to the bit, and a pass that was set to the gather form stays in it."""
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(5000, 5, 17))
    g, u = dev(c.gamma), dev(np.random.default_rng(5).normal(size=(c.n_vertices, 3)))

    def passes(ctx):
        rows = torch.empty(c.n_edges, dtype=torch.float64, device="cuda")
        tpe.tp_energy(ctx, g, rows=rows)
        return [host(rows), host(tpe.tp_differential(ctx, g)), host(tpe.sobolev_apply(ctx, g, u))]

    def there_and_back(ctx):
        ctx.set_params(alpha=3.0, beta=6.0)
        passes(ctx)
        ctx.set_params(alpha=2.0, beta=4.5)

    new = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    first = passes(new)
    there_and_back(new)
    gather = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_energy_variant(gather, 0)
    tpe.tp_set_diff_variant(gather, 0)
    tpe.tp_set_apply_variant(gather, 0)
    ordered = passes(gather)
    there_and_back(gather)
    for a, b, c0, c1 in zip(first, passes(new), ordered, passes(gather)):
        assert np.array_equal(a, b) and np.array_equal(c0, c1)
        assert not np.array_equal(a, c0)


# plain FP32 positions: the bars of test_new_context_of_many_ragged_curves
@pytest.mark.parametrize("n", [3, 4, 63, 64, 65, 127, 128, 129, 192, 193, 255, 256, 257, 385])
@pytest.mark.parametrize("variant", [0, 1, 2])
def test_fp32_passes_at_block_edges(torch, orc, n, variant):
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(n, 4, 40 + n))
    ctx = make_ctx(c, precision=tpe.TP_FP32, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_energy_variant(ctx, 1)
    tpe.tp_set_apply_variant(ctx, 1)
    tpe.tp_set_energy_variant(ctx, variant)
    tpe.tp_set_apply_variant(ctx, variant)
    with pytest.raises(tpe.TpError) as err:
        tpe.tp_set_diff_variant(ctx, 1)
    assert err.value.status == tpe.TP_ERR_UNSUPPORTED
    _check(torch, orc, ctx, c, 1, {"energy": 1e-4, "diff": 1.0, "apply": 1e-4})
