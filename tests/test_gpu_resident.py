"""Resident launches (states up to 20 qubits in complex64, 18 in complex128): one launch runs many
evaluations, tiles exchange the vector H acts on through partner copies.  Sizes at the edges of
the tile rule (one tile; the first size with several; one, two, four and eight slots per thread),
Hamiltonians with every kind of product, the options that change the launch, against the oracle
and bit for bit against the same run with fewer CTAs or one step per launch."""
import numpy as np
import pytest

from instances import generate_ec3, random_state, xx_pairs
from oracle import oracle as O

from _helpers import C64, C128, TOL_STATE, load_both, random_clauses, random_terms, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


def _random(n, prec, seed, T=0.6, steps=90):
    """X strings, Y/Z phases, hops, Z strings, identity and clauses of every group."""
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    ctx, H = Context(n, prec), O.Hamiltonian(n)
    terms = [(g, x, z, 0.3 * c) for (g, x, z, c) in random_terms(n, seed, nterms=20)]
    if n >= 2:
        m = 1 | (1 << (n - 1))  # a hop between the lowest and the highest bit
        terms += [(0, m, 0, -0.25), (0, m, m, -0.25)]
    load_both(ctx, H, terms, random_clauses(n, seed))
    ctx.set_schedule(T, HB.nonlinear_schedule())
    ctx.set_integrator(steps, 0.0)
    return ctx, H, O.nonlinear_path(T)


@pytest.mark.parametrize("prec", [C128, C64])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 7, 8, 9, 10, 11, 13, 14, 15, 17, 18, 19, 20])
def test_solve_matvec_and_energy_against_the_oracle(n, prec):
    steps = 90 if n < 15 else 12
    ctx, H, sched = _random(n, prec, 40 + n, steps=steps)
    psi0 = random_state(n, n)
    dt = np.complex128 if prec == C128 else np.complex64
    ctx.set_initial_state(psi0.astype(dt))
    st = ctx.propagate(-1)
    got = ctx.state()
    ref = O.propagate(H, sched, steps, psi0.astype(dt).astype(np.complex128), nthreads=16)
    assert st["steps_done"] == steps and st["evaluations"] == ref.evaluations
    assert rel_err(got, ref.psi) < TOL_STATE[prec]
    out = ctx.hpsi(0.3, torch.from_numpy(psi0.astype(dt)).cuda()).cpu().numpy()
    w = sched.weights(0.3)
    want = O.hpsi(H, w, psi0.astype(dt).astype(np.complex128))
    assert rel_err(out, want) < TOL_STATE[prec]
    e = ctx.energy_at(0.3)
    y = got.astype(np.complex128)
    assert abs(e - np.vdot(y, O.hpsi(H, w, y)).real) < TOL_STATE[prec] * max(1.0, abs(e)) * 10
    ctx.close()


@pytest.mark.parametrize("prec", [C128, C64])
@pytest.mark.parametrize("n", [9, 11, 13, 14, 17, 19])
def test_fewer_ctas_and_single_steps_keep_the_bits(n, prec):
    """A limit on the CTAs (several tiles per CTA, owned vectors in memory, no cluster), one step per
    launch, and calls that end anywhere give the same state and norm: cluster and memory exchange,
    owned vectors in registers and in memory."""
    ref = None
    for limit, k, calls in ((0, -1, (-1,)), (1, -1, (-1,)), (5, 0, (-1,)), (0, 0, (1, 1, 2, 1, 30, -1)),
                            (0, 8, (2, 3, 17, -1))):
        ctx, _, _ = _random(n, prec, 7, steps=75)
        ctx.set_grid_limit(limit)
        ctx.set_graph_steps(k)
        ctx.set_initial_state("uniform")
        for m in calls:
            st = ctx.propagate(m)
        got = (ctx.state(), st["norm2"], st["steps_done"])
        ctx.close()
        if ref is None:
            ref = got
        assert np.array_equal(got[0], ref[0]) and got[1:] == ref[1:]


@pytest.mark.parametrize("n", [6, 12, 18, 19, 20])
def test_options_on_resident_launches(n):
    """The compensated corrector (complex64) and step-size control, XY hops and the catalyst."""
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    inst = generate_ec3(n, 3)
    H = O.ec3_hamiltonian(inst, pairs=xx_pairs(n, 3))
    steps = 60 if n < 18 else 24
    T = 0.02 * steps / n
    ref = O.propagate(H, O.nonlinear_path(T), steps, O.uniform_state(n), nthreads=16)
    for prec, opt in ((C64, "ycomp"), (C128, "adaptive")):
        ctx = Context(n, prec, extra_vector=True)
        HB.load_ec3(ctx, inst, pairs=xx_pairs(n, 3))
        ctx.set_schedule(T, HB.nonlinear_schedule())
        if opt == "adaptive":
            ctx.set_integrator(steps, 0.0, adaptive=True, tol=1.0)
            ctx.set_step_growth(0)
        else:
            ctx.set_integrator(steps, 0.0)
            ctx.set_y_compensation(True)
        ctx.set_initial_state("uniform")
        st = ctx.propagate(-1)
        assert st["steps_done"] == steps
        assert rel_err(ctx.state(), ref.psi) < (TOL_STATE[C128] if prec == C128 else 5e-7)
        ctx.close()
    ctx = Context(n, C64)
    sched, k = HB.load_xy(ctx, inst, driver="xy", catalyst_alpha=8.0)
    ctx.set_schedule(20.0, sched)
    ctx.set_integrator(0, 0.0)
    ctx.set_initial_state(("dicke", k))
    ctx.propagate(20)
    psi = ctx.state()
    ones = np.array([bin(z).count("1") for z in range(1 << n)]) if n <= 12 else None
    if ones is not None:  # hops keep the Hamming weight exactly
        assert not np.any(psi[ones != k])
    assert abs(ctx.norm2() - 1.0) < 1e-5
    ctx.close()


@pytest.mark.parametrize("prec", [C64, C128])
def test_batch_of_resident_and_other_members(prec):
    """Members of every size class beside members on layout passes (too large, own tile bits), an odd
    number of steps per round, members that end inside a round; removed before the end, they go on
    alone."""
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Batch, Context

    def make(n, tile_bits, driver, total):
        inst = generate_ec3(n, n)
        ctx = Context(n, prec)
        if tile_bits:
            ctx.set_tile_bits(tile_bits)
        if driver == "xy":
            sched, k = HB.load_xy(ctx, inst, driver="xy", catalyst_alpha=8.0)
            start = ("dicke", k)
        else:
            HB.load_ec3(ctx, inst, pairs=xx_pairs(n, n))
            sched, start = HB.nonlinear_schedule(), "uniform"
        ctx.set_schedule(0.02 * total / n, sched, 1)
        ctx.set_integrator(total, 0.0)
        ctx.set_initial_state(start)
        return ctx

    big = 21 if prec == C64 else 19
    specs = [(6, 0, "x", 40), (9, 0, "xy", 20), (10, 0, "x", 80), (12, 0, "xy", 80), (13, 9, "x", 60), (14, 0, "x", 31),
             (17, 0, "x", 40), (18, 0, "xy", 40), (big, 0, "x", 30)]
    alone = []
    for s in specs:
        c = make(*s)
        st = c.propagate(-1)
        alone.append((c.state(), st["steps_done"]))
        c.close()
    tol = 2e-6 if prec == C64 else 1e-13
    b = Batch(prec, max_members=16, max_items=4096, steps_per_round=7)
    ctxs = [make(*s) for s in specs]
    slots = [b.add(c) for c in ctxs[:5]]
    b.run(2)
    slots += [b.add(c) for c in ctxs[5:]]  # join while others are under way
    b.run(3)
    steps, active, launches = b.poll()
    assert launches > 0 and active > 0
    assert [steps[k] for k in slots] == [min(t, 3 + 7 * (5 if i < 5 else 3)) for i, (_, _, _, t) in enumerate(specs)]
    for k, c, (want, total) in zip(slots, ctxs, alone):
        b.remove(k)
        st = c.propagate(-1)
        assert st["steps_done"] == total and abs(st["norm2"] - 1.0) < 1e-4
        assert rel_err(c.state(), want) < tol
        c.close()
    b.close()


@pytest.mark.parametrize("max_items,fits", [(15, False), (16, True)])
def test_batch_work_items_bound_resident_members_too(max_items, fits):
    """A batch counts 2^(n - tile_bits) work items per member (two of n = 16 on 2^13 tiles: 16)."""
    import paper_1311_3938_gb300 as P
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Batch, Context

    b = Batch(C64, max_members=2, max_items=max_items, steps_per_round=2)
    ctxs = []
    for _ in range(2):
        ctx = Context(16, C64)
        HB.load_ec3(ctx, generate_ec3(16, 1))
        ctx.set_schedule(10.0, HB.linear_schedule())
        ctx.set_integrator(20, 0.0)
        ctx.set_initial_state("uniform")
        b.add(ctx)
        ctxs.append(ctx)
    if fits:
        b.run(1)
        assert b.poll()[1] == 2
    else:
        with pytest.raises(P.AqcError, match="max_items"):
            b.run(1)
    b.close()
    for c in ctxs:
        c.close()
