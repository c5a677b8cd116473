"""A context whose steps run as layout passes before and after a stay in a batch of resident launches,
which keep three derivatives, not four: the passes after it must not read the fourth."""
import numpy as np
import pytest

from instances import generate_ec3, xx_pairs

from _helpers import C64, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


@pytest.mark.parametrize("n", [16, 18])
def test_layout_passes_after_a_batch(n):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Batch, Context

    def make():
        ctx = Context(n, C64)
        # so many couplings that no order holds them all: the turn of layouts asks for layout
        # passes and then does not apply
        HB.load_ec3(ctx, generate_ec3(n, 2), pairs=xx_pairs(n, 2, 60))
        ctx.set_schedule(4.0, HB.nonlinear_schedule())
        ctx.set_integrator(400, 0.0)
        ctx.set_layout_turns(1)
        ctx.set_initial_state("uniform")
        ctx.propagate(8)
        return ctx

    ref = make()
    ref.propagate(22)
    ctx = make()
    ctx.set_layout_turns(0)
    b = Batch(C64, max_members=1, max_items=4096, steps_per_round=10)
    slot = b.add(ctx)
    b.run(1)
    b.poll()
    b.remove(slot)
    ctx.set_layout_turns(1)
    ctx.propagate(12)
    # 30 steps of rounding in another order
    assert rel_err(ctx.state(), ref.state()) < 2e-6
    b.close()
    ctx.close()
    ref.close()
