"""Z strings and clause classes beside the cached one, in the kernels that take each once for many
amplitudes: strings on every combination of the bits that vary within a thread, random ones, many
of them; H psi per amplitude against NumPy in double precision."""
import numpy as np
import pytest

from instances import generate_ec3, random_state

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


# resident launches: one tile, clusters, one to sixteen slots per thread; tiles of layout passes
@pytest.mark.parametrize("prec,n,tile_bits", [(C64, 1, 0), (C64, 9, 0), (C64, 12, 0), (C64, 18, 0), (C64, 20, 0), (C64, 13, 13),
                                              (C64, 16, 13), (C64, 21, 0), (C128, 3, 0), (C128, 10, 0), (C128, 18, 0)])
def test_diagonal_per_amplitude(prec, n, tile_bits):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    rng = np.random.default_rng(n)
    low = [0, 6, 7, 8, 9, 10]
    masks = [sum(1 << b for i, b in enumerate(low) if (k >> i) & 1) for k in range(1, 64)]
    masks = sorted({m & ((1 << n) - 1) for m in masks} - {0}) + [int(m) for m in rng.integers(1, 1 << n, 40)]
    coef = rng.normal(size=len(masks))
    ctx = Context(n, prec)
    if tile_bits:
        ctx.set_tile_bits(tile_bits)
    ctx.load_terms(0, [1 << q for q in range(n)], [0] * n, [-0.5] * n)
    ctx.load_terms(1, [0] * len(masks), masks, coef)
    z = np.arange(1 << n)
    parity = lambda m: 1.0 - 2.0 * (np.bitwise_count(z & m) & 1)
    s = 0.4
    d = sum(s * c * parity(m) for m, c in zip(masks, coef))
    size = s * np.abs(coef).sum()
    clauses = list(generate_ec3(n, 3).clauses) if n >= 5 else []
    if clauses:
        count = lambda cl: sum((sum(((z >> b) & 1) for b in c) != 1).astype(float) for c in cl)
        for g, cl, scale in ((1, clauses, 1.0), (2, clauses[:-1], 0.7), (0, clauses[1:4], 1.3)):
            ctx.load_clauses(g, cl, scale=scale)
            w = (1.0 - s, s, s * (1.0 - s))[g] * scale
            d = d + w * count(cl)
            size += w * len(cl)
    ctx.set_schedule(1.0, HB.nonlinear_schedule())
    dt = np.complex64 if prec == C64 else np.complex128
    psi = random_state(n, 5).astype(dt)
    got = ctx.hpsi(s, torch.from_numpy(psi).cuda()).cpu().numpy()
    p = psi.astype(complex)
    want = d * p - 0.5 * (1.0 - s) * sum(p[z ^ (1 << q)] for q in range(n))
    # every term of the diagonal and every product rounds once, relative to the sizes added so far
    eps = 2.0 ** (-24 if prec == C64 else -53)
    terms = len(masks) + 3 + n + 4
    near = sum(np.abs(p[z ^ (1 << q)]) for q in range(n))
    assert np.all(np.abs(got - want) <= 2 * terms * eps * (size * np.abs(p) + 0.5 * near) + 1e-300)
    ctx.close()
