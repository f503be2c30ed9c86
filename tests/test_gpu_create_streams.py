"""A mesh is ready when its creation returns, whatever the default stream still has to do."""
import pytest

pytestmark = pytest.mark.gpu


def test_new_mesh_on_a_side_stream_while_the_default_stream_is_busy():
    """The status word raised by a pass on a side stream is still there when the default stream
    gets to what was queued on it before (the new mesh's scratch is not zeroed from there)."""
    import torch
    import paper_1609_00098_gb300 as dg
    from paper_1609_00098_gb300 import build as b
    b.build()
    kw = dict(system=1, K=(2, 2, 2), n=3, flux=1, precision=0, gamma=4.0 / 3.0)
    U = torch.zeros(8, 5, 27, dtype=torch.float64, device="cuda")
    U[:, 0], U[:, 4] = 1.0, 1.0
    U[3, 4, 5] = -1.0  # one unphysical node
    P = torch.zeros(8, 4, 27, dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    dg.Mesh(**kw).close()  # (everything loaded)
    torch.cuda.synchronize()
    for _ in range(3):
        torch.cuda._sleep(200_000_000)  # the default stream, some 0.1 s
        m = dg.Mesh(**kw)
        busy = not torch.cuda.default_stream().query()
        with torch.cuda.stream(side):
            dg.abi.dg_primitives(m.h, U, P)
        torch.cuda.synchronize()
        assert m.sync_status() == dg.abi.DG_ERR_C2P
        m.close()
    assert busy  # else nothing was tested
