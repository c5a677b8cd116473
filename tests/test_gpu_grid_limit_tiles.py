"""A limit on the CTAs of a state on resident launches picks larger tiles: the state's bits stay, whatever
the limit, also when it changes between the calls of one run."""
import numpy as np
import pytest

from instances import generate_ec3, xx_pairs

from _helpers import C64, C128

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


def _run(n, prec, limits):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    ctx = Context(n, prec)
    HB.load_ec3(ctx, generate_ec3(n, 3), pairs=xx_pairs(n, 3))
    ctx.set_schedule(4.0, HB.nonlinear_schedule())
    ctx.set_integrator(400, 0.0)
    ctx.set_initial_state("uniform")
    for k in limits:
        ctx.set_grid_limit(k)
        ctx.propagate(24 // len(limits))
    out = ctx.state()
    assert abs(ctx.norm2() - 1.0) < 1e-4
    ctx.close()
    return out


# limits that make one tile of everything, fill the largest tiles once, and leave several visits
@pytest.mark.parametrize("prec,n", [(C64, 10), (C64, 12), (C64, 15), (C64, 18), (C64, 20), (C128, 9), (C128, 13), (C128, 17)])
def test_limits_keep_the_bits(prec, n):
    want = _run(n, prec, [0])
    for limits in ([1], [3], [8], [40], [100], [0, 8], [16, 0, 2, 64]):
        assert np.array_equal(_run(n, prec, limits), want)
