"""Equal-coefficient products summed as integers (complex128 layout passes): H psi and a step against
the oracle on states whose amplitudes span many orders of magnitude, tiles of the smallest and the
default size, the fewest and the most products a layout takes that way, and tiles holding
infinities or NaN (which keep the FP64 products)."""
import numpy as np
import pytest

from instances import generate_ec3, random_state
from oracle import oracle as O

from _helpers import C128, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


def _ctx(n, tile_bits, weights=None):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    inst = generate_ec3(n, 3)
    ctx = Context(n, C128)
    ctx.set_tile_bits(tile_bits)  # the layout passes
    HB.load_ec3(ctx, inst, x_weights=weights)
    ctx.set_schedule(2.0, HB.linear_schedule())
    ctx.set_integrator(100, 0.0)
    return ctx, O.ec3_hamiltonian(inst, x_weights=weights)


def _states(n):
    r = random_state(n, 3)
    k = np.arange(1 << n)
    yield r
    yield np.full(1 << n, 2.0 ** (-n / 2), complex)
    for v in (r * np.exp2(-(k % 61)), r + 3.0 * (k == 5), r * np.where(k & 64, 1e-30, 1.0), (k == 77 % len(k)) + 0j):
        yield v / np.linalg.norm(v)
    yield r * 1e-250  # below the scale range: FP64 products
    yield r * 1e150
    yield r * (1.0 - 2.0**-53) + 1j * 2.0**-60


# (n, tile bits): one layout of 12; 12 + 4 (the fewest); 7-bit tiles (4 per strided layout, tiles of
# two warps); 3 products left over (FP64)
@pytest.mark.parametrize("n,tile_bits", [(12, 12), (16, 12), (15, 7), (11, 8), (15, 12)])
def test_matvec_against_the_oracle(n, tile_bits):
    ctx, H = _ctx(n, tile_bits)
    sched = O.linear_path(2.0)
    w = sched.weights(0.7)
    for psi in _states(n):
        got = ctx.hpsi(0.7, torch.from_numpy(psi).cuda()).cpu().numpy()
        want = O.hpsi(H, w, psi)
        # FP64 rounding of n + 2 products and sums on either side, relative to sum |terms| <= 2 n ||psi||
        assert np.linalg.norm(got - want) <= 4 * (n + 2) * 2.0**-53 * 2 * n * np.linalg.norm(psi)
    for bad in (np.inf, np.nan, -np.inf):
        psi = random_state(n, 5)
        psi[3] = bad
        got = ctx.hpsi(0.7, torch.from_numpy(psi).cuda()).cpu().numpy()
        hit = np.zeros(1 << n, bool)
        hit[3] = True
        hit[[3 ^ (1 << q) for q in range(n)]] = True
        assert np.array_equal(~np.isfinite(got), hit)
    ctx.close()


# (also the corrector's integer sums: states beyond their scale range take the FP64 ones)
@pytest.mark.parametrize("scale", [1.0, 1e-240, 1e140])
@pytest.mark.parametrize("n,tile_bits,weights", [(16, 12, None), (13, 8, None), (14, 12, np.arange(14) % 3 + 0.5)])
def test_solve_and_energy_against_the_oracle(n, tile_bits, weights, scale):
    ctx, H = _ctx(n, tile_bits, weights)
    psi0 = random_state(n, 8) * scale
    ctx.set_initial_state(psi0)
    ctx.propagate(20)
    ref = O.propagate(H, O.linear_path(2.0), 100, psi0, max_steps=20, nthreads=8)
    got = ctx.state()
    assert rel_err(got / scale, ref.psi / scale) < 1e-14
    if scale == 1.0:
        assert abs(ctx.energy() - O.energy(H, got)) < 1e-12
    ctx.close()
