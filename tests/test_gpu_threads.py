"""Host threads with contexts of their own, of different shapes and sizes of shared memory, launching the same
kernels at the same time: every run ends and gives what it gives alone."""
import threading

import numpy as np
import pytest

from instances import generate_ec3, xx_pairs

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


def _run(n, prec, pairs, stream=None):
    from paper_1311_3938_gb300 import hamiltonians as HB
    from paper_1311_3938_gb300.engine import Context

    ctx = Context(n, prec, stream=stream)
    HB.load_ec3(ctx, generate_ec3(n, 2), pairs=xx_pairs(n, 2, pairs))
    ctx.set_schedule(4.0, HB.nonlinear_schedule())
    ctx.set_integrator(400, 0.0)
    ctx.set_initial_state("uniform")
    ctx.propagate(80)
    out = ctx.state()
    ctx.close()
    return out


@pytest.mark.parametrize("prec,sizes", [(C64, [10, 11, 12, 13, 14, 16, 21, 22]), (C128, [8, 9, 10, 11, 12, 14, 19, 20])])
def test_threads_with_other_shapes(prec, sizes):
    specs = [(n, prec, p) for n in sizes for p in (0, n)]
    alone = [_run(*s) for s in specs]
    errors = []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(3):
                    if not np.array_equal(_run(*specs[i], stream=stream), alone[i]):
                        errors.append((specs[i], "another state"))
        except Exception as e:  # noqa: BLE001
            errors.append((specs[i], repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(specs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
