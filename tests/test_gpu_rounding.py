"""Rounding of the FP64 arithmetic against extended precision: forms that save instructions may not cost digits.  The
bounds lie between the errors of the two forms compared (deterministic on one GPU), well above the spread of seeds."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import dev, host, make_ctx, need_gpu

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def _error(x, ref):
    return float(np.linalg.norm((x - ref).astype(float)) / np.linalg.norm(ref.astype(float)))


def test_spectral_preconditioner_keeps_its_digits(torch):
    """z = D^-1/2 F^-1 diag(1 / lambda) F D^-1/2 r, mean over four curves of each of nine sizes (one curve's error differs from
    the next one's by 20%): 3.1e-16, as with complex products and two sums; 3.3e-16 with 2 u - (u + w b) in the butterflies."""
    from scipy import fft
    from paper_2006_07859_gb300 import tpe
    errors = []
    for n in (64, 256, 300, 777, 1024, 1500, 2048, 4096, 8192):
        for seed in range(4):
            c = S.single(S.fourier_knot(n, 8, seed))
            ctx = make_ctx(c, precision=tpe.TP_FP64, precond=tpe.TP_PRECOND_SPECTRAL)
            r = np.random.default_rng(seed).normal(size=(n, 3))
            z = host(tpe.tp_precond_apply(ctx, dev(c.gamma), dev(r)))
            lam = host(tpe.tp_spectral_symbols(ctx, 0)).astype(LD)
            d = 1 / np.sqrt(host(tpe.tp_gram_diagonal(ctx, dev(c.gamma))).astype(LD))[:, None]
            x = (d * r.astype(LD)).astype(np.clongdouble)
            errors.append(_error(z, d * fft.ifft(fft.fft(x, axis=0) / lam[:, None], axis=0).real))
    assert np.mean(errors) <= 3.2e-16, errors


def _pairs(g, u):
    """Energy rows and A u of one closed curve in extended precision (Eqs. 17-19 at (2, 4.5))."""
    g, u = g.astype(LD), u.astype(LD)
    n = len(g)
    p, q = g, np.roll(g, -1, 0)
    ell = np.sqrt(((q - p) ** 2).sum(1))
    T = (q - p) / ell[:, None]
    i = np.arange(n)
    gap = (i[:, None] - i[None]) % n
    keep = (gap > 1) & (gap < n - 1)
    e = w = w0 = 0
    for a in (p, q):
        for b in (p, q):
            d = a[:, None] - b[None]
            d2 = np.where(keep, (d ** 2).sum(2), 1)
            cI = d2 - (T[:, None] * d).sum(2) ** 2
            cJ = d2 - (T[None] * d).sum(2) ** 2
            f = np.where(keep, d2 ** LD(-1.25), 0)
            e = e + cI * f / d2
            w = w + f
            w0 = w0 + (cI + cJ) * f / d2 ** 2
    du, ub = (np.roll(u, -1, 0) - u) / ell[:, None], (np.roll(u, -1, 0) + u) / 2
    omt = ((T[:, None] - T[None]) ** 2).sum(2) / 2
    w, w0 = w * ell, w0 * ell
    h = (w.sum(1)[:, None] * du - (w * (1 - omt)) @ du) / 2
    m = ell[:, None] * (w0.sum(1)[:, None] * ub - w0 @ ub) / 8
    return ell / 4 * (e @ ell), m - h + np.roll(m + h, 1, 0)


def test_fp64_powers_keep_their_digits(torch):
    """Energy rows and A u of knots of 150 edges, mean over eight curves: 2.0e-16 and 1.7e-16 (4.3e-16 and 1.8e-16 with
    rsqrt() and sqrt(); 2.7e-16 and 2.8e-16 from one root of order 1/4)."""
    from paper_2006_07859_gb300 import tpe
    rows_err, apply_err = [], []
    for seed in range(8):
        c = S.single(S.fourier_knot(150, 8, 50 + seed))
        ctx = make_ctx(c, precision=tpe.TP_FP64, precond=tpe.TP_PRECOND_JACOBI)
        u = np.random.default_rng(seed).normal(size=(150, 3))
        rows = torch.empty(150, dtype=torch.float64, device="cuda")
        tpe.tp_energy(ctx, dev(c.gamma), rows=rows)
        Au = host(tpe.sobolev_apply(ctx, dev(c.gamma), dev(u)))
        rows_ref, Au_ref = _pairs(c.gamma, u)
        rows_err.append(_error(host(rows), rows_ref))
        apply_err.append(_error(Au, Au_ref))
    assert np.mean(rows_err) <= 2.4e-16 and np.mean(apply_err) <= 2.3e-16, (rows_err, apply_err)


@pytest.mark.parametrize("n", [150, 500])
def test_accurate_apply_keeps_its_digits(torch, n):
    """The double-float apply of a jittered trefoil, mean over eight: 9.6e-15 and 2.7e-14, as fully renormalised arithmetic
    has it (1.7e-14 and 3.3e-14 with sums that are not renormalised)."""
    from paper_2006_07859_gb300 import tpe
    errors = []
    for seed in range(8):
        c = S.single(S.trefoil(n, 0.01 * 256 / max(n, 256), seed))
        u = np.random.default_rng(seed).normal(size=(n, 3))
        ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
        errors.append(_error(host(tpe.sobolev_apply_accurate(ctx, dev(c.gamma), dev(u))), _pairs(c.gamma, u)[1]))
    assert np.mean(errors) <= (1.2e-14 if n == 150 else 2.95e-14), errors
