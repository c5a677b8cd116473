"""H psi into vectors that start on an 8-byte boundary: taken up to 6 qubits in complex64, refused on the
host above; psi itself needs 16 bytes."""
import pytest

from instances import generate_ec3

from _helpers import C64

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_3938_gb300 as P

    P.build()
    yield


@pytest.mark.parametrize("n", [3, 5, 6, 7, 12, 20, 21])
def test_unaligned_vectors(n):
    import paper_1311_3938_gb300 as P
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    ctx = Context(n, C64)
    if n >= 5:
        HB.load_ec3(ctx, generate_ec3(n, 3))
    else:
        ctx.load_terms(0, [1, 4, 6], [0, 4, 0], [0.5, -0.25, 1.5])
    ctx.set_schedule(1.0, HB.linear_schedule())
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.randn(1 << n, dtype=torch.complex64, device="cuda", generator=g)
    want = ctx.hpsi(0.3, psi)
    room = torch.empty((1 << n) + 1, dtype=torch.complex64, device="cuda")
    off = room[1:]
    assert off.data_ptr() % 16 == 8
    if n <= 6:
        torch.testing.assert_close(ctx.hpsi(0.3, psi, off), want, rtol=1e-5, atol=1e-6)
    else:
        with pytest.raises(P.AqcError, match="aligned"):
            ctx.hpsi(0.3, psi, off)
    off.copy_(psi)
    with pytest.raises(P.AqcError, match="aligned"):
        ctx.hpsi(0.3, off, torch.empty_like(psi))
    ctx.close()
