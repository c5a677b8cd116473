"""Batch members whose tables and partner buffers fill a multiprocessor's shared memory: counts of
products around the points where one buffer less fits, and every pair of qubits coupled by a hop."""
import numpy as np
import pytest

from instances import generate_ec3

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


def _ctx(n, prec, pairs, hops, steps=20):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    ctx = Context(n, prec)
    HB.load_ec3(ctx, generate_ec3(n, 2))
    m = [(1 << i) | (1 << j) for i, j in pairs]
    ctx.load_terms(2, m, [0] * len(m), [0.02] * len(m))
    if hops:
        ctx.load_terms(2, m, m, [0.02] * len(m))
    ctx.set_schedule(0.4, HB.nonlinear_schedule())
    ctx.set_integrator(steps, 0.0)
    ctx.set_initial_state("uniform")
    return ctx


def _check(specs, prec):
    from paper_1311_3938_gb300.engine import Batch

    b = Batch(prec, max_members=len(specs), max_items=4096, steps_per_round=16)
    ctxs = [_ctx(*s) for s in specs]
    slots = [b.add(c) for c in ctxs]
    b.run(2)
    assert b.poll()[1] == 0
    for k, c, s in zip(slots, ctxs, specs):
        b.remove(k)
        alone = _ctx(*s)
        alone.propagate(-1)
        # the sums of a batch and of a lone launch may be cut differently: one rounding per product
        assert rel_err(c.state(), alone.state()) < (2e-6 if prec == C64 else 1e-13)
        alone.close()
        c.close()
    b.close()


def _pairs(n, k):
    every = [(i, j) for i in range(n) for j in range(i)]
    order = np.random.default_rng(5).permutation(len(every))
    return [every[i] for i in order[:k]]


def test_members_with_every_hop():
    n = 18
    _check([(n, C64, _pairs(n, 153), True)] * 4, C64)


@pytest.mark.parametrize("prec,n,counts", [(C128, 16, range(44, 66, 3)), (C64, 17, range(112, 137, 4)),
                                           (C128, 15, range(80, 105, 4))])
def test_counts_of_couplings_across_a_buffer(prec, n, counts):
    for k in counts:
        _check([(n, prec, _pairs(n, k), False)], prec)
