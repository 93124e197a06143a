"""Positions that the edge records refuse."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import dev, make_ctx, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("bad", ["nan", "inf", "sum"])
def test_nonfinite_positions_are_refused(torch, prec, bad):
    """A NaN, an infinity, and coordinates whose sum overflows (finite edges at 1.2e308)."""
    from paper_2006_07859_gb300 import tpe
    g = np.array(S.regular_polygon(8))
    if bad == "sum":
        g[:, :2] = 1.2e308
        g[:, 2] = [0.0, 1.0, 2.0, 3.0, 2.75, 2.5, 1.5, 0.5]
    else:
        g[3, 1] = float(bad)
    ctx = make_ctx(S.single(g), precision=prec, precond=tpe.TP_PRECOND_JACOBI)
    with pytest.raises(tpe.TpError) as err:
        tpe.tp_energy(ctx, dev(g))
    assert err.value.status == tpe.TP_ERR_NONFINITE
