"""Meshes of one order but other sizes stepped from two host threads at once: what one launch sets
up for a kernel must not take it from the other's."""
import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_00098_gb300 as p
    from paper_1609_00098_gb300 import build as b
    b.build()
    return p


def _run(calls):
    """Every call in a thread of its own, all at once; their exceptions."""
    errors, start = [], threading.Barrier(len(calls))

    def body(call):
        start.wait()
        try:
            call()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
    threads = [threading.Thread(target=body, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def test_summaries_of_meshes_with_other_element_groups(pkg):
    """n = 8: two and three elements per CTA, whose shared memory is above the default limit."""
    import torch
    calls = []
    for K in ((10, 5, 4), (8, 6, 10)):
        m = pkg.Mesh(system=0, K=K, n=8, flux=0, limiter=1, precision=0)
        U, S = m.state(), torch.zeros(m.E, 5, 10, dtype=torch.float64, device="cuda")
        U.fill_(1.0)
        s = torch.cuda.Stream()
        torch.cuda.synchronize()

        def loop(m=m, U=U, S=S, s=s):
            for _ in range(4000):
                pkg.abi.dg_limiter_summaries(m.h, U, S, s)
        calls.append(loop)
    errors = _run(calls)
    torch.cuda.synchronize()
    assert not errors, errors[0]
