"""tp_energy_static sums in the order of a context's gather pass over the same graph."""
import pytest

import synth as S
from tests.gpu_util import dev, host, make_ctx, need_gpu

pytestmark = pytest.mark.gpu


# sizes on either side of one target per thread and of the short source chunks; the largest the scratch holds.  The order
# of the compensated FP32 sums moves the energy by 1e-9 at 256 edges, the order of FP64 sums by 1e-15.
@pytest.mark.parametrize("n", [4, 64, 256, 300, 1023, 1500, 3000, 5000, 8191, 20000, 65536])
def test_static_energy_is_the_gather_energy(n):
    torch = need_gpu()
    from paper_2006_07859_gb300 import tpe
    c = S.single(S.fourier_knot(n, 6, 8))
    g = dev(c.gamma)
    ctx = make_ctx(c, precision=tpe.TP_MIXED, precond=tpe.TP_PRECOND_JACOBI)
    tpe.tp_set_energy_variant(ctx, 0)
    ref = host(tpe.tp_energy(ctx, g))[0]
    E = host(tpe.tp_energy_static(g, torch.as_tensor(c.edges).cuda()))[0]
    assert abs(E - ref) <= 1e-13 * abs(ref), (E, ref)
