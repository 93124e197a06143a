"""The mixed differential's near band: chords that cross an axis plane, whole curves of any size, and strands far closer
than an edge."""
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


# A power of four scales every quantity of the differential exactly (its degree is -1.5), so the scaled result is the
# same to the bit as long as no exponent runs out; 1e-12 leaves room for the FP64 sums' order alone.
@pytest.mark.parametrize("variant", [0, 1, 3])
@pytest.mark.parametrize("power", [-12, -10, 10, 12])
def test_scaled_curves_have_the_scaled_differential(torch, variant, power):
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(500, 4, 23))
    out = []
    for p in (0, power):
        ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
        tpe.tp_set_diff_variant(ctx, variant)
        out.append(host(tpe.tp_differential(ctx, dev(c.gamma * 4.0 ** p))) * 8.0 ** p)
    assert np.all(np.isfinite(out[1]))
    assert rel(out[1], out[0]) <= 1e-12


# The positions of a double-float curve of size 1 are known to 2^-49, so a gap g has an error of 4 x 2^-49 / g of itself at
# most and its gradient (degree -3.5 in it) 3.5 times that; 1e-6 on top for the other pairs.
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("gap", [1e-6, 1e-8, 1e-10, 1e-11])
def test_strands_much_closer_than_an_edge(torch, orc, variant, gap):
    from paper_2006_07859_gb300 import tpe
    g = S.fourier_knot(64, 3, 2)
    g[40] = g[7] + gap * np.array([0.36, 0.48, 0.8])
    c = S.single(g)
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI, near_cutoff=16.0)
    tpe.tp_set_diff_variant(ctx, variant)
    dE = host(tpe.tp_differential(ctx, dev(c.gamma)))
    assert rel(dE, orc.differential(c.gamma, c.edges)) <= 1e-6 + 14 * 2.0 ** -49 / gap
