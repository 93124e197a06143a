"""The buffer of partial sums that all pair passes of a context share: passes whose buffer cannot be had are refused
and leave the context as it was."""
import numpy as np
import pytest

import synth as S
from tests.gpu_util import dev, host, make_ctx, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return need_gpu()


def _knot_among_polygons(n, k, m=256):
    """One Fourier knot of n edges and k regular polygons of m edges: the knot sets the slots of a row (n / 256), all
    edges together the size of a slot."""
    t = 2.0 * np.pi * np.arange(m) / m
    ring = np.stack([np.cos(t), np.sin(t), 0.1 * np.sin(2 * t)], 1)
    gamma = np.concatenate([S.fourier_knot(n, 16, 5), np.tile(ring, (k, 1))])
    edges = np.concatenate([S.closed_edges(n)] +
                           [np.stack([np.tile(np.arange(m), k), np.tile((np.arange(m) + 1) % m, k)], 1) +
                            (n + m * np.repeat(np.arange(k), m))[:, None]]).astype(np.int32)
    off = np.concatenate([[0], n + m * np.arange(k + 1)]).astype(np.int32)
    return S.Curves(gamma, edges, off, off)


def test_refused_partial_sums_leave_the_context_sound(torch):
    """1,026 slots of 3.9M edges x 10 values: 324 GB of partial sums, more than the device has.  The selection fails and
    the passes run on in the form, with the buffer and to the bits they had before."""
    from paper_2006_07859_gb300 import tpe
    c = _knot_among_polygons(262144, 14400)
    assert 1026 * c.n_edges * 80 > torch.cuda.get_device_properties(0).total_memory
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI, independent=1)
    g = dev(c.gamma)
    rows = torch.empty(c.n_edges, dtype=torch.float64, device="cuda")
    E = host(tpe.tp_energy(ctx, g, rows=rows))
    before = host(rows)
    with pytest.raises(tpe.TpError) as err:
        tpe.tp_set_diff_variant(ctx, 1)
    assert err.value.status == tpe.TP_ERR_OOM
    rows.zero_()
    assert np.array_equal(host(tpe.tp_energy(ctx, g, rows=rows)), E)
    assert np.array_equal(host(rows), before)
    ctx.close()


def test_two_fields_without_memory_take_the_gather_pass(torch):
    """1,026 slots of 364,544 edges: the apply's partial sums take 18 GB and are asked for; those of its two-field form
    (36 GB) are more than a pass takes unasked, so two fields run the gather pass.  Tolerance of the two forms of the
    apply: 1e-6 of the largest entry."""
    from paper_2006_07859_gb300 import tpe
    c = _knot_among_polygons(262144, 400)
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI, independent=1)
    tpe.tp_set_apply_variant(ctx, 1)
    g = dev(c.gamma)
    U = dev(np.random.default_rng(3).normal(size=(2, c.n_vertices, 3)))
    one = [tpe.sobolev_apply(ctx, g, U[f]) for f in range(2)]
    AU = torch.empty_like(U)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    AU = tpe.sobolev_apply_multi(ctx, g, U, AU)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 8e9
    for f in range(2):
        assert float((AU[f] - one[f]).abs().max()) <= 1e-6 * float(one[f].abs().max())
    ctx.close()


def test_new_context_leaves_memory_to_others(torch):
    """50,000 edges: 198 slots, so the symmetric differential's partial sums take 0.79 GB, the apply's 0.48 GB and the
    energy's 0.08 GB.  A new context takes them where the device is free, and with 20 GB left only the energy's (a
    64th); its other arrays are the same.  Both give the same differential (1e-5 of the largest entry)."""
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(50000, 16, 9))
    g = dev(c.gamma)

    def create():
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
        torch.cuda.synchronize()
        return ctx, free - torch.cuda.mem_get_info()[0]

    create()[0].close()    # loads the kernels
    ctx, used = create()
    dE = host(tpe.tp_differential(ctx, g))
    ctx.close()
    free = torch.cuda.mem_get_info()[0]
    held = torch.empty(free - (20 << 30), dtype=torch.uint8, device="cuda")
    ctx, used_full = create()
    dE_full = host(tpe.tp_differential(ctx, g))
    ctx.close()
    del held
    torch.cuda.empty_cache()
    assert used - used_full > 0.4e9, (used, used_full)
    assert np.abs(dE - dE_full).max() <= 1e-5 * np.abs(dE).max()
