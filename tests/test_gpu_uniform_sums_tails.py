"""Equal-coefficient products summed as integers (complex128 layout passes) keep FP64's bits in every
amplitude, also in those far below the largest of their tile: H psi against extended precision, part
by part; steps from a basis state, whose amplitudes fall off with the Hamming distance, against the
oracle; the same steps cut into odd pieces, replayed from graphs and in a batch."""
import numpy as np
import pytest

from instances import generate_ec3, random_state
from oracle import oracle as O

from _helpers import C128

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

T, STEPS = 2.0, 100


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


def _ctx(n, tile_bits):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    inst = generate_ec3(n, 3)
    ctx = Context(n, C128)
    if tile_bits:
        ctx.set_tile_bits(tile_bits)
    HB.load_ec3(ctx, inst)
    ctx.set_schedule(T, HB.linear_schedule())
    ctx.set_integrator(STEPS, 0.0)
    return ctx, inst


def _states(n):
    r, k = random_state(n, 3), np.arange(1 << n)
    far = np.array([bin(z ^ 77).count("1") for z in range(1 << n)])
    yield r * 10.0 ** (-1.7 * far)
    yield r + 3e9 * (k == 5)
    yield r.real + 1e-17j * r.imag  # one part far below the other
    yield r * np.where(k & 64, 1e-30, 1.0)
    yield r * np.where(k == 9, 1e200, 1.0) * 1e-40
    yield (k == 77) + 0j


@pytest.mark.parametrize("n,tile_bits", [(12, 12), (16, 12), (15, 7), (19, 0)])
def test_matvec_part_by_part(n, tile_bits):
    ctx, inst = _ctx(n, tile_bits)
    s = 0.35
    z = np.arange(1 << n)
    d = sum((sum(((z >> b) & 1) for b in c) != 1).astype(np.longdouble) for c in inst.clauses)
    d = s * d + (1.0 - s) * 0.5 * n
    for psi in _states(n):
        got = ctx.hpsi(s * T, torch.from_numpy(psi).cuda()).cpu().numpy()
        for g, v in ((got.real, psi.real), (got.imag, psi.imag)):
            v = v.astype(np.longdouble)
            flips = [v[z ^ (1 << q)] * np.longdouble(-0.5 * (1.0 - s)) for q in range(n)]
            want, size = d * v + sum(flips), np.abs(d * v) + sum(np.abs(f) for f in flips)
            # n products, the diagonal (its sum and weights) and the sums of the layouts, each rounded
            # by half an ulp of at most the sum of the terms' sizes; doubled for the integer products
            assert np.all(np.abs(g - want) <= 2 * (n + 10) * 2.0**-53 * size)
    ctx.close()


def _tails(got, ref):
    big = np.abs(ref) > 1e-280  # (a step's weighted sums lose bits to subnormals below)
    return np.max(np.abs(got - ref)[big] / np.abs(ref)[big])


# one layout; two, with tiles whose amplitudes span 40 orders of magnitude; the default tiles, from graphs
@pytest.mark.parametrize("n,tile_bits", [(12, 12), (16, 12), (19, 0)])
def test_amplitudes_far_from_a_basis_state(n, tile_bits):
    ctx, inst = _ctx(n, tile_bits)
    psi0 = np.zeros(1 << n, complex)
    psi0[77] = 1.0
    ref = O.propagate(O.ec3_hamiltonian(inst), O.linear_path(T), STEPS, psi0, max_steps=24, nthreads=16)
    ctx.set_initial_state(77)
    ctx.propagate(24)
    whole = ctx.state()
    # every amplitude is a sum of paths of one sign and phase to leading order: relative rounding of a
    # few ulps per product and step
    assert _tails(whole, ref.psi) < 24 * 4 * (n + 10) * 2.0**-53
    for pieces in ((5, 1, 17, 1), (3, 16, 2, 3)):
        ctx.set_initial_state(77)
        for m in pieces:
            ctx.propagate(m)
        assert np.array_equal(ctx.state(), whole)
    ctx.close()


def test_batch_members_on_layout_passes():
    from paper_1311_3938_gb300.engine import Batch

    n = 19
    alone, _ = _ctx(n, 0)
    alone.set_initial_state(77)
    alone.propagate(3 + 15)
    b = Batch(C128, max_members=2, max_items=4096, steps_per_round=5)
    ctxs = [_ctx(n, 0)[0] for _ in range(2)]
    for c in ctxs:
        c.set_initial_state(77)
    slots = [b.add(c) for c in ctxs]
    b.run(3)
    b.poll()
    for k, c in zip(slots, ctxs):
        b.remove(k)
        assert np.array_equal(c.state(), alone.state())
    # a member that goes on alone after an odd number of steps
    ctxs[0].propagate(7)
    alone.propagate(7)
    assert np.array_equal(ctxs[0].state(), alone.state())
    b.close()
    for c in ctxs + [alone]:
        c.close()
