"""Edges of the FP64 and training kernels against the oracle: counts around a warp's
batch, element counts that leave the last CTA short, states outside the range of the
integer-ALU products (which take the FP64 instructions instead), and mini-batches of
every shape the training epoch distinguishes."""
import numpy as np
import pytest

import dg_inputs as di
import oracle
from oracle import mlp

pytestmark = pytest.mark.gpu

G = 4.0 / 3.0


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_00098_gb300 as p
    from paper_1609_00098_gb300 import build as b
    b.build()
    return p


def _gpu(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("count", [1, 31, 32, 33, 255, 4127])
def test_con2prim_counts_scales_and_bad_states(pkg, count, inplace):
    """Bits, iteration counts and statuses of the oracle, for states scaled by 2^-490
    and 2^490 (con2prim is homogeneous of degree one; its products then leave the integer
    range) and not scaled, unphysical ones among them, with and without guesses."""
    import torch
    cons = oracle.prim2con(1, G, di.c2p_samples(31, count, gamma=G))
    k = np.arange(count)
    cons = cons * np.where(k % 5 == 2, 2.0 ** -490, np.where(k % 5 == 4, 2.0 ** 490, 1.0))
    cons[4, k % 11 == 6] *= -1.0
    for guess in (None, np.where(k % 3 == 0, -1.0, cons[4] * 0.25)):
        po, ito, sto = oracle.con2prim(G, cons, guess)
        a = _gpu(cons)
        out = a if inplace else torch.empty_like(a)
        it = torch.empty(count, dtype=torch.int32, device="cuda")
        st = torch.empty(count, dtype=torch.int32, device="cuda")
        pkg.abi.dg_con2prim(count, G, a, out, None if guess is None else _gpu(guess), it, st)
        good = sto == 0
        assert np.array_equal(st.cpu().numpy(), sto) and np.array_equal(good, k % 11 != 6)
        assert np.array_equal(out.cpu().numpy()[:, good], po[:, good])
        assert np.array_equal(it.cpu().numpy()[good], ito[good])


@pytest.mark.parametrize("K", [(1, 1, 1), (5, 3, 1)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -560])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 6, 7, 8])
def test_newtonian_steps_bitwise(pkg, n, scale, K):
    """Two steps with and without the limiter (without it the stage kernel writes the
    next primitives), on a state and on the same state scaled by a power of two (the
    equations are homogeneous of degree one)."""
    import torch
    for limiter, flux in ((0, 0), (0, 1), (1, 1), (2, 0)):
        kw = dict(system=0, K=K, n=n, flux=flux, limiter=limiter, gamma=1.4, lo=(-0.5,) * 3, hi=(0.5,) * 3)
        om, gm = oracle.Mesh(oracle.MeshSpec(**kw)), pkg.Mesh(**kw)
        U = om.from_prim(di.kh_ne(om.coords(), seed=2)) * scale
        Ug = _gpu(U)
        t = torch.zeros(om.E, dtype=torch.uint8, device="cuda")
        for _ in range(2):
            h, to = om.cfl_dt(U, 0.2), np.zeros(om.E, dtype=np.uint8)
            U = om.rk3_step(U, h, to)
            gm.rk3_step(Ug, cfl=0.2, troubled=t)
            assert np.array_equal(t.cpu().numpy(), to), (limiter, flux)
        assert np.array_equal(Ug.cpu().numpy(), U), (limiter, flux)


@pytest.mark.parametrize("system", [0, 1])
@pytest.mark.parametrize("n,K", [(2, (11, 9, 9)), (3, (11, 9, 9)), (4, (11, 9, 9)), (5, (11, 9, 9)), (6, (11, 9, 7)),
                                 (7, (7, 5, 11)), (8, (7, 5, 11)), (2, (31, 5, 1)), (5, (31, 5, 1)), (8, (31, 5, 1))])
def test_summaries_of_several_elements_per_cta(pkg, n, K, system):
    """The summaries take ceil(E / 152) elements per CTA up to a largest group (6 for n <= 5, 4 for n = 6, 3
    for n = 7, 8): that group with a short last CTA (891 = 6 * 148 + 3, 693 = 4 * 173 + 1, 385 = 3 * 128
    + 1) and two elements with one left over (155), unphysical states in the last element among them,
    against the oracle."""
    import torch
    kw = dict(system=system, K=K, n=n, flux=1, limiter=1, gamma=G, lo=(0,) * 3, hi=(1,) * 3)
    om, gm = oracle.Mesh(oracle.MeshSpec(**kw)), pkg.Mesh(**kw)
    xyz = om.coords()
    U = om.from_prim(di.blast_sr(xyz, seed=3) if system else di.kh_ne(xyz - 0.5, seed=3))
    assert np.array_equal(gm.summaries(_gpu(U)).cpu().numpy(), om.summaries(U))
    V = U.copy()
    if system:
        V[[0, om.E // 2, om.E - 1], 4, n] *= -1.0  # every variable of these elements is replaced
    Ug, t = _gpu(V), torch.zeros(om.E, dtype=torch.uint8, device="cuda")
    V, to = om.limit(V)
    gm.limit(Ug, t)
    assert np.array_equal(t.cpu().numpy(), to) and np.array_equal(Ug.cpu().numpy(), V)
    if system:
        assert (to[[0, om.E // 2, om.E - 1]] == 31).all()


@pytest.mark.parametrize("system,n,limiter", [(0, 4, 0), (0, 6, 1), (1, 5, 1), (1, 4, 0)])
def test_captured_steps_bitwise(pkg, system, n, limiter):
    """FP64 steps captured into a CUDA graph (their launches' programmatic edges with them) and replayed."""
    import torch
    kw = dict(system=system, K=(5, 3, 4), n=n, flux=1, limiter=limiter, gamma=G, lo=(-0.5,) * 3, hi=(0.5,) * 3)
    om, gm = oracle.Mesh(oracle.MeshSpec(**kw)), pkg.Mesh(**kw)
    xyz = om.coords()
    U = om.from_prim(di.blast_sr(xyz + 0.5, seed=2) if system else di.kh_ne(xyz, seed=2))
    Ug, dt = _gpu(U), torch.zeros(1, dtype=torch.float64, device="cuda")
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        for _ in range(2):
            gm.rk3_step(Ug, cfl=0.2, dt_used=dt)
    for _ in range(2):
        g.replay()
        for _ in range(2):
            h = om.cfl_dt(U, 0.2)
            U = om.rk3_step(U, h)
        torch.cuda.synchronize()
        assert np.array_equal(Ug.cpu().numpy(), U) and dt.item() == h


@pytest.mark.parametrize("n", [2, 4, 6, 7, 8])
def test_relativistic_steps_bitwise(pkg, n):
    for limiter, flux in ((0, 1), (1, 0)):
        kw = dict(system=1, K=(3, 1, 5), n=n, flux=flux, limiter=limiter, gamma=G, lo=(0,) * 3, hi=(1,) * 3)
        om, gm = oracle.Mesh(oracle.MeshSpec(**kw)), pkg.Mesh(**kw)
        U = om.from_prim(di.blast_sr(om.coords(), seed=2))
        Ug = _gpu(U)
        for _ in range(2):
            h = om.cfl_dt(U, 0.2)
            U = om.rk3_step(U, h)
            gm.rk3_step(Ug, cfl=0.2)
        assert gm.sync_status() == 0 and np.array_equal(Ug.cpu().numpy(), U)


def _net(seed, count):
    prim = di.c2p_samples(seed, count, gamma=G)
    params = mlp.init_params(di.uniform(seed, 9, np.arange(mlp.N_PARAMS)))
    return oracle.prim2con(1, G, prim), prim[4], params.astype(np.float32)


@pytest.mark.parametrize("count", [1, 31, 33, 257])
def test_guess_counts(pkg, count):
    import torch
    cons, _, params = _net(41, count)
    ref = params.astype(np.float64)
    o = mlp.OFFSETS["W2"]
    ref[o:o + 4096] = torch.from_numpy(params[o:o + 4096]).to(torch.bfloat16).to(torch.float64).numpy()
    net = pkg.abi.dg_c2p_net_create(params, mlp.DEFAULT_SCALES)
    out = torch.empty(count, dtype=torch.float64, device="cuda")
    pkg.abi.dg_c2p_net_guess(net, count, G, _gpu(cons), out)
    pkg.abi.dg_c2p_net_destroy(net)
    # BF16 rounding of h1 (2^-9) times the output scale, as for the full batch
    assert np.abs(np.log10(out.cpu().numpy()) - np.log10(mlp.guess(ref, cons, G))).max() < 5e-2


@pytest.mark.parametrize("count,batch", [(3, 1), (100, 2048), (391, 130), (4096 + 77, 2048), (2048 * 2, 2048),
                                         (2 * 2049 + 5, 2049), (4096 + 300, 4096)])
def test_training_minibatches(pkg, count, batch):
    """Two epochs against Adam in FP64 on the gradients of dg_c2p_net_grad, mini-batch by
    mini-batch (the last one short): batches of up to 2048 run in one cluster, larger
    ones in launches of their own.

    Tolerance: the two sum a gradient's FP32 terms in different orders, which moves it
    by some 1e-5 of its terms' size.  Adam divides every component by its own size, so
    components smaller than that may change sign and move by 2 lr instead of 0: a share
    of 1e-4 of them (a component's size is spread over the range of its terms), hence
    sqrt(1e-4) * 2 = 2e-2 of the parameters' way in norm.
    """
    import torch
    cons, p, params = _net(43, count)
    lr, a, pg = 1e-3, _gpu(cons), _gpu(p)
    net = pkg.abi.dg_c2p_net_create(params, mlp.DEFAULT_SCALES)
    loss = torch.zeros(2, dtype=torch.float32, device="cuda")
    pkg.abi.dg_c2p_net_train(net, count, a, pg, 2, batch, lr, loss)
    got = pkg.abi.dg_c2p_net_get_params(net).astype(np.float64)
    pkg.abi.dg_c2p_net_destroy(net)

    q, m, v, step = params.astype(np.float64), 0.0, 0.0, 0
    grad = torch.empty(mlp.N_PARAMS, dtype=torch.float32, device="cuda")
    one = torch.empty(1, dtype=torch.float32, device="cuda")
    means = []
    for _ in range(2):
        total = 0.0
        for i in range(0, count, batch):
            c, t = a[:, i:i + batch].contiguous(), pg[i:i + batch].contiguous()
            net = pkg.abi.dg_c2p_net_create(q.astype(np.float32), mlp.DEFAULT_SCALES)
            pkg.abi.dg_c2p_net_grad(net, t.numel(), c, t, grad, one)
            pkg.abi.dg_c2p_net_destroy(net)
            step += 1
            q, m, v = mlp.adam_step(q, grad.cpu().numpy().astype(np.float64), m, v, step, lr=lr)
            q = q.astype(np.float32).astype(np.float64)
            total += one.item() * t.numel()
        means.append(total / count)
    way = np.linalg.norm(q - params)
    assert way > 0.0 and np.linalg.norm(got - q) <= 2e-2 * way, np.linalg.norm(got - q) / way
    # the loss moves by its gradient times the parameters' difference: a share of its change
    assert np.allclose(loss.cpu().numpy(), means, rtol=2e-2)
