"""The gather passes at sizes where a new context runs the symmetric ones: every comparison selects its pass."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import cosine, dev, host, make_ctx, need_gpu, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle as O
    O.build_library()
    return O


def _select(ctx, variant):
    from paper_2006_07859_gb300 import tpe
    tpe.tp_set_energy_variant(ctx, variant)
    tpe.tp_set_diff_variant(ctx, variant)
    tpe.tp_set_apply_variant(ctx, variant)


# bars of test_symmetric_differential_matches_gather_and_oracle
@pytest.mark.parametrize("variant", [1, 2, 3, 4])
def test_symmetric_differential_of_a_fine_curve_matches_the_gather_pass(torch, variant):
    """3,000 edges with many pairs inside the near cutoff."""
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(3000, 16, 4))
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    g = dev(c.gamma)
    tpe.tp_set_diff_variant(ctx, 0)
    gather = host(tpe.tp_differential(ctx, g))
    tpe.tp_set_diff_variant(ctx, variant)
    sym = host(tpe.tp_differential(ctx, g))
    assert not np.array_equal(sym, gather)    # two forms, not one against itself
    assert rel(sym, gather) <= 1e-5 and cosine(sym, gather) >= 1 - 1e-10


# bars of test_multi_apply_on_independent_batch and of the mixed applies
@pytest.mark.parametrize("variant", [0, 1])
def test_multi_field_apply_of_a_batch_in_both_forms(torch, orc, variant):
    """Several source chunks per target block in the four-field gather pass, ragged tails, no pair across curves."""
    from paper_2006_07859_gb300 import tpe
    b = S.batch_of_knots([1500, 2600, 2049], 6, 300)
    ctx = make_ctx(b, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI, independent=1)
    tpe.tp_set_apply_variant(ctx, variant)
    U = np.random.default_rng(5).normal(size=(5, b.n_vertices, 3))
    AU = host(tpe.sobolev_apply_multi(ctx, dev(b.gamma), dev(U)))
    for k in range(b.n_curves):
        gk, ek = b.curve(k)
        v = slice(b.vertex_offsets[k], b.vertex_offsets[k + 1])
        for f in range(U.shape[0]):
            assert rel(AU[f, v], orc.gram_apply(gk, ek, 0.75, U[f, v])) <= 1e-6, (k, f)


# bars of test_mixed_precision_at_scale
@pytest.mark.parametrize("variant", [0, 1])
def test_mixed_passes_at_65536_edges_in_both_forms(torch, orc, variant):
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(65536, 16, 100))
    rng = np.random.default_rng(101)
    rows_i = np.sort(rng.choice(c.n_edges, 64, replace=False)).astype(np.int32)
    v_i = np.sort(rng.choice(c.n_vertices, 24, replace=False)).astype(np.int32)
    u = np.random.default_rng(102).normal(size=(c.n_vertices, 3))
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    _select(ctx, variant)
    g = dev(c.gamma)
    rows = torch.empty(c.n_edges, dtype=torch.float64, device="cuda")
    tpe.tp_energy(ctx, g, rows=rows)
    dE = host(tpe.tp_differential(ctx, g))
    Au = host(tpe.sobolev_apply(ctx, g, dev(u)))
    ref = orc.differential_at(c.gamma, c.edges, v_i)
    assert rel(host(rows)[rows_i], orc.energy_rows(c.gamma, c.edges, rows_i)) <= 1e-6
    assert cosine(dE[v_i], ref) >= 0.9999 and rel(dE[v_i], ref) <= 1e-5
    assert rel(Au[v_i], orc.gram_apply_at(c.gamma, c.edges, 0.75, u, v_i)) <= 1e-6
