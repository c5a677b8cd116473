"""The TMA-fed layout passes of complex64 (X strings and hops): every mode of the contiguous layout
(step, Runge-Kutta stages, derivative, energy, matvec) with clause bytes, other clause classes, Z
strings and identities, products that no layout holds, and calls that end anywhere (y is stored by
the last step of a call), against the oracle; and that the kernel's fallbacks agree with it."""
import numpy as np
import pytest

from instances import generate_ec3, random_state, xx_pairs
from oracle import oracle as O

from _helpers import C64, TOL_STATE, load_both, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


def _pair(n, general=False):
    """X driver, couplings, hops (also between the lowest and the highest bit), Z strings, identity,
    clauses of three classes; with `general`, one Y product (the passes that hold it fall back)."""
    inst = generate_ec3(n, 4)
    terms = [(0, 1 << q, 0, -0.5) for q in range(n)]
    terms += [(2, (1 << i) | (1 << j), 0, 0.3 * J) for (i, j, J) in xx_pairs(n, 4, 10)]
    for i, j in ((0, n - 1), (0, 6), (6, 8), (3, n - 2), (1, 2)):
        m = (1 << i) | (1 << j)
        terms += [(1, m, 0, -0.25), (1, m, m, -0.25)]
    terms += [(1, 0, 5, 0.2), (0, 0, 1 << (n - 1), -0.4), (0, 0, 0, 0.75)]
    if general:
        terms += [(0, 2, 2, 0.3)]
    clauses = [(1, c, 0, 1.0) for c in inst.clauses] + [(2, c, 0, 1.0) for c in inst.clauses[:-1]]
    clauses += [(0, inst.clauses[0], 1, 0.4)]
    return terms, clauses


def _ctx(n, T, steps, general=False, tile_bits=13):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    ctx, H = Context(n, C64), O.Hamiltonian(n)
    if tile_bits:
        ctx.set_tile_bits(tile_bits)
    load_both(ctx, H, *_pair(n, general))
    ctx.set_schedule(T, HB.nonlinear_schedule(), 1)
    ctx.set_integrator(steps, 0.0)
    return ctx, H, O.nonlinear_path(T, 1)


# one layout; two (1, 2 and 8 bits in the strided one); three; products no layout holds where the
# top bits are read from memory (22, 23)
@pytest.mark.parametrize("n,general,tile_bits", [(13, False, 13), (14, False, 13), (15, True, 13), (16, False, 13),
                                                 (21, False, 0), (22, False, 0), (23, False, 0)])
def test_solve_matvec_and_energy_against_the_oracle(n, general, tile_bits):
    steps = 80 if n < 20 else 14
    T = 0.02 * steps / n
    ctx, H, sched = _ctx(n, T, steps, general, tile_bits)
    psi0 = random_state(n, n).astype(np.complex64)
    ctx.set_initial_state(psi0)
    done = 0
    for m in (2, 1, 1, 3, 2):
        ctx.propagate(m)
        done += m
    ref = O.propagate(H, sched, steps, psi0.astype(np.complex128), max_steps=done, nthreads=16)
    assert rel_err(ctx.state(), ref.psi) < 1e-6
    st = ctx.propagate(-1)
    ref = O.propagate(H, sched, steps, psi0.astype(np.complex128), nthreads=16)
    got = ctx.state()
    assert rel_err(got, ref.psi) < TOL_STATE[C64] * 0.2
    assert abs(st["norm2"] - np.linalg.norm(got.astype(complex)) ** 2) < 1e-6
    t = 0.4 * T
    want = O.hpsi(H, sched.weights(t), psi0.astype(np.complex128), nthreads=16)
    out = ctx.hpsi(t, torch.from_numpy(psi0).cuda()).cpu().numpy()
    assert rel_err(out, want) < 1e-6
    y = got.astype(np.complex128)
    e = np.vdot(y, O.hpsi(H, sched.weights(t), y, nthreads=16)).real
    assert abs(ctx.energy_at(t) - e) < 2e-6 * max(1.0, abs(e))
    ctx.close()


def test_split_calls_and_cta_limits_keep_the_bits():
    ref = None
    for calls, limit in (((-1,), 0), ((1, 2, 1, 1, 7, 1, -1), 0), ((-1,), 3)):
        ctx, _, _ = _ctx(15, 0.1, 40)
        ctx.set_grid_limit(limit)
        ctx.set_initial_state("uniform")
        for m in calls:
            st = ctx.propagate(m)
        got = (ctx.state(), st["norm2"])
        ctx.close()
        ref = ref or got
        assert np.array_equal(got[0], ref[0]) and got[1] == ref[1]


def test_compensated_and_controlled_steps_agree_with_the_plain_ones():
    """Those keep y in memory (k_apply); the plain step does not."""
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    inst = generate_ec3(16, 3)
    H = O.ec3_hamiltonian(inst)
    ref = O.propagate(H, O.linear_path(1.0), 200, O.uniform_state(16), nthreads=16)
    for opt in ("", "ycomp", "adaptive"):
        ctx = Context(16, C64, extra_vector=True)
        ctx.set_tile_bits(13)
        HB.load_ec3(ctx, inst)
        ctx.set_schedule(1.0, HB.linear_schedule())
        ctx.set_integrator(200, 0.0, adaptive=opt == "adaptive", tol=1.0)
        ctx.set_step_growth(0)
        if opt == "ycomp":
            ctx.set_y_compensation(True)
        ctx.set_initial_state("uniform")
        st = ctx.propagate(-1)
        assert rel_err(ctx.state(), ref.psi) < 1e-6
        assert st["max_err_est"] < 1e-6
        ctx.close()


# every pair of bits as a hop (both, one or none of them held by a thread; two layouts; bits that no
# layout holds) and X strings over the thread's own bits, coefficients all different.  A sum of m <= 270
# products in FP32 errs by about sqrt(m) * 2^-24 * 0.5 < 5e-7 relative.
@pytest.mark.parametrize("n,tile_bits,strings", [(13, 13, False), (13, 13, True), (16, 13, False), (23, 0, True)])
def test_matvec_with_hops_between_all_bits(n, tile_bits, strings):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    terms = []
    for i in range(n):
        for j in range(i):
            m, c = (1 << i) | (1 << j), 0.1 + 0.01 * i - 0.013 * j
            if not (strings and j == 0 and i in (6, 7, 8)):
                terms += [(0, m, 0, c), (0, m, m, c)]
    for k in range(8):
        if strings or k not in (1, 2, 4):
            terms.append((1, (k << 6) | 1, 0, 0.3 - 0.07 * k))
    ctx, H = Context(n, C64), O.Hamiltonian(n)
    if tile_bits:
        ctx.set_tile_bits(tile_bits)
    load_both(ctx, H, terms, [(1, c, 0, 1.0) for c in generate_ec3(n, 4).clauses])
    ctx.set_schedule(1.0, HB.linear_schedule())
    sched = O.linear_path(1.0)
    psi = random_state(n, 3).astype(np.complex64)
    want = O.hpsi(H, sched.weights(0.4), psi.astype(np.complex128), nthreads=16)
    assert rel_err(ctx.hpsi(0.4, torch.from_numpy(psi).cuda()).cpu().numpy(), want) < 1e-6
    ctx.close()
