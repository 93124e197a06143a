"""The mixed differential's near band: chords that cross an axis plane."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import dev, host, make_ctx, need_gpu, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


# A regular polygon's differential is what its edge rows leave after they cancel by (n / 2 pi)^2: one FP32 rounding of a far
# pair's terms (2^-24) is 6e-3 of it at 2,048 edges.  Near chords whose coordinates change sign have inexact FP32
# differences; rounded, they alone gave 3e-2 to 1e-1.
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_chords_across_the_axis_planes(torch, variant, seed):
    from paper_2006_07859_gb300 import tpe
    n = 2048
    q, _ = np.linalg.qr(np.random.default_rng(seed).normal(size=(3, 3)))
    t = 2.0 * np.pi * (np.arange(n) + 0.37) / n
    c = S.single(np.stack([np.cos(t), np.sin(t), 0.0 * t], 1) @ q)
    g = dev(c.gamma)
    ref = host(tpe.tp_differential(make_ctx(c, precision=tpe.TP_FP64, precond=tpe.TP_PRECOND_JACOBI), g))
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_diff_variant(ctx, variant)
    assert rel(host(tpe.tp_differential(ctx, g)), ref) <= 2.0 ** -24 * (n / (2.0 * np.pi)) ** 2
