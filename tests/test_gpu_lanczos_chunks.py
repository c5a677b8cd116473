"""Lanczos steps issued several at a time: an invariant subspace found inside a chunk ends the
iteration there (the steps after it are ignored), iteration limits that are no multiple of a chunk,
vectors of fewer elements than a block's threads, and complex64 starts with subnormal, zero and very
small entries (the exact widening of floats)."""
import numpy as np
import pytest

from instances import generate_ec3, random_state
from oracle import oracle as O

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


def _ctx(n, prec):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    inst = generate_ec3(n, 2)
    ctx = Context(n, prec)
    HB.load_ec3(ctx, inst)
    ctx.set_schedule(1.0, HB.linear_schedule())
    return ctx, O.dense_matrix(O.ec3_hamiltonian(inst), [0.6, 0.4, 0.0, 0.0])


@pytest.mark.parametrize("n,max_iter", [(4, 40), (5, 32), (7, 13), (9, 64)])
def test_eigenvalues_and_iterations(n, max_iter):
    ctx, M = _ctx(n, C128)
    start = random_state(n, 6)
    eig, _, iters = ctx.lanczos(0.4, torch.from_numpy(start).cuda(), max_iter=max_iter, n_eig=2, tol=0.0)
    V, a, b = [start / np.linalg.norm(start)], [], []  # the recurrence in numpy
    for j in range(max_iter):
        r = M @ V[j]
        al = np.vdot(V[j], r).real
        for _ in range(2):
            for v in V:
                r = r - np.vdot(v, r) * v
        a.append(al)
        b.append(np.linalg.norm(r))
        if b[-1] <= 1e-13 * max(1.0, abs(al)):
            break
        V.append(r / b[-1])
    k = len(a)
    want = np.linalg.eigvalsh(np.diag(a) + np.diag(b[: k - 1], 1) + np.diag(b[: k - 1], -1))[:2]
    assert np.max(np.abs(np.array(eig) - want)) < 1e-11 * max(1.0, abs(want[1]))
    assert iters <= max_iter and (iters == max_iter or iters <= (1 << n))
    x, theta, resid, _ = ctx.lanczos_ground(0.4, torch.from_numpy(start).cuda(), max_iter=max(max_iter, 60), tol=1e-12)
    lowest = np.linalg.eigvalsh(M)[0]
    assert abs(theta - lowest) < 1e-11 * max(1.0, abs(lowest)) and resid < 1e-10
    ctx.close()


def test_complex64_start_with_tiny_entries():
    n = 9
    ctx, M = _ctx(n, C64)
    start = random_state(n, 4).astype(np.complex64)
    start[3] = 1e-42 - 3e-41j  # subnormal
    start[7] = 0.0
    start[11] = 2e-38
    eig, _, _ = ctx.lanczos(0.4, torch.from_numpy(start).cuda(), max_iter=96, n_eig=2, tol=0.0)
    want = np.linalg.eigvalsh(M)[:2]
    assert np.max(np.abs(np.array(eig) - want)) < 1e-4
    ctx.close()
