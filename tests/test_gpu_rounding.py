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


@pytest.mark.parametrize("n", [1500, 2048])
def test_spectral_preconditioner_keeps_its_digits(torch, n):
    """z = D^-1/2 F^-1 diag(1 / lambda) F D^-1/2 r, mean over four curves: 3.1e-16 and 3.3e-16 with butterflies u + v, u - v
    (1,500 vertices with 2 u - (u + v): 4.1e-16)."""
    from scipy import fft
    from paper_2006_07859_gb300 import tpe
    errors = []
    for seed in range(4):
        c = S.single(S.fourier_knot(n, 8, seed))
        ctx = make_ctx(c, precision=tpe.TP_FP64, precond=tpe.TP_PRECOND_SPECTRAL)
        r = np.random.default_rng(seed).normal(size=(n, 3))
        z = host(tpe.tp_precond_apply(ctx, dev(c.gamma), dev(r)))
        lam = host(tpe.tp_spectral_symbols(ctx, 0)).astype(LD)
        d = 1 / np.sqrt(host(tpe.tp_gram_diagonal(ctx, dev(c.gamma))).astype(LD))[:, None]
        x = (d * r.astype(LD)).astype(np.clongdouble)
        errors.append(_error(z, d * fft.ifft(fft.fft(x, axis=0) / lam[:, None], axis=0).real))
    assert np.mean(errors) <= 3.6e-16, errors
