"""The qubit order that keeps multi-qubit flips inside tiles applies to states of resident size whose
evaluations run as layout passes: a clause-by-clause sequence, the turn of layouts.  Seen from
outside by its rounding: sums in another order give other bits than the identity's order, the same
state otherwise."""
import numpy as np
import pytest

from instances import generate_ec3, xx_pairs

from _helpers import C64, C128, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


def _state(n, prec, path, relabel):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    inst = generate_ec3(n, 5)
    ctx = Context(n, prec)
    ctx.set_relabel(relabel)
    if path == "cbc":
        sched, k = HB.load_xy(ctx, inst, driver="xy", clause_by_clause=True)
        start = ("dicke", k)
    else:
        HB.load_ec3(ctx, inst, pairs=xx_pairs(n, 5))
        sched, start = HB.nonlinear_schedule(), "uniform"
        ctx.set_layout_turns(1 if path == "turn" else 0)
    ctx.set_schedule(20.0, sched)
    ctx.set_integrator(0, 0.0)
    ctx.set_initial_state(start)
    ctx.propagate(12)
    out = ctx.state()
    ctx.close()
    return out


@pytest.mark.parametrize("path", ["cbc", "turn", "plain"])
@pytest.mark.parametrize("prec,n", [(C128, 16), (C128, 18), (C64, 20)])
def test_layout_passes_choose_an_order(prec, n, path):
    a, b = _state(n, prec, path, True), _state(n, prec, path, False)
    assert rel_err(a, b) < (1e-6 if prec == C64 else 1e-14)
    # resident launches (the plain step) have no use for an order
    assert np.array_equal(a, b) == (path == "plain")
