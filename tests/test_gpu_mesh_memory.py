"""How much device memory a mesh holds."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("system", [0, 1])
def test_fp64_mesh_scratch(n, system):
    """No more than two state copies, primitives, limiter summaries and a byte per element (what a
    mesh needs whose stage kernel forms every face flux itself), and one allocation granule (2 MiB)
    for each of the ten buffers."""
    import torch
    import paper_1609_00098_gb300 as dg
    from paper_1609_00098_gb300 import build as b
    b.build()
    K = int((400e6 / (1300 + 112 * n ** 3)) ** (1.0 / 3.0))  # some 400 MB
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    m = dg.Mesh(system=system, K=(K, K, K), n=n, flux=0, limiter=1, precision=0, gamma=4.0 / 3.0)
    used = free - torch.cuda.mem_get_info()[0]
    m.close()
    assert 0 < used <= K ** 3 * (8 * (14 * n ** 3 + 50) + 1) + 10 * (2 << 20)
