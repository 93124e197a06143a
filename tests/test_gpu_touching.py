"""Strands so close that |d|^-4.5 overflows FP32: the energy is infinite on the rows of both strands, not NaN, and no
other row takes harm."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import dev, host, make_ctx, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def _touching(n):
    """Two open curves of 40 and n - 40 edges whose first vertices are 1e-10 apart; the second one's edges in reverse
    order, so that the touching rows are the first and the last (which the idle lanes of a block repeat)."""
    a = S.fourier_knot(90, 3, 2)[:41]
    b = S.fourier_knot(n + 60, 3, 5)[:n - 39]
    g = np.concatenate([a - a[0], b - b[0] + 1e-10 * np.array([0.36, 0.48, 0.8])])
    e = np.concatenate([S.open_edges(41), S.open_edges(n - 39, 41)[::-1]])
    return S.Curves(g, e, [0, 41, n + 2], [0, 40, n])


@pytest.mark.parametrize("n", [64, 65, 300])
@pytest.mark.parametrize("prec,variant,exponents", [(1, 0, (2.0, 4.5)), (1, 1, (2.0, 4.5)), (2, 0, (2.0, 4.5)),
                                                    (2, 1, (2.0, 4.5)), (2, 2, (2.0, 4.5)), (2, 0, (3.0, 6.0))])
def test_energy_of_touching_strands_is_infinite(torch, n, prec, variant, exponents):
    from paper_2006_07859_gb300 import tpe
    c = _touching(n)
    ctx = make_ctx(c, precision=prec, precond=tpe.TP_PRECOND_JACOBI, alpha=exponents[0], beta=exponents[1])
    tpe.tp_set_energy_variant(ctx, variant)
    rows = torch.empty(n, dtype=torch.float64, device="cuda")
    E = host(tpe.tp_energy(ctx, dev(c.gamma), rows=rows))
    rows = host(rows)
    assert E[0] == np.inf and np.isinf(rows[[0, n - 1]]).all()
    assert np.isfinite(rows[1:n - 1]).all()
