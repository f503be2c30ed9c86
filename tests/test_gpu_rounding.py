"""Outputs whose rounding is part of what the kernels promise."""
import ctypes
import os

import numpy as np
import pytest

import dg_inputs as di
from oracle import mlp

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


@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("n", [3, 4, 5, 6, 7, 8])
def test_relativistic_volume_term_of_a_uniform_flow_is_zero(pkg, n, flux):
    """The fluxes enter the mixed relativistic contraction as differences to node 0's, each flux
    and the difference rounded on their own: equal fluxes differ by zero, and the right-hand side
    of a uniform flow is zero at every node that no face lifts into.  (A product fused with the
    subtraction leaves its rounding error, 1e-8 of the flux, times the sum of |D|.)"""
    import torch
    m = pkg.Mesh(system=1, K=(3, 2, 2), n=n, flux=flux, limiter=0, gamma=5.0 / 3.0, lo=(0, 0, 0), hi=(1, 1, 1),
                 precision=1)
    prim = torch.tensor([1.3, 0.31, -0.23, 0.17, 0.7], dtype=torch.float64, device="cuda")
    R = m.rhs(m.from_prim(prim[:, None].expand(5, m.E * n ** 3).contiguous())).cpu().numpy()
    inner = R.reshape(m.E, 5, n, n, n)[:, :, 1:-1, 1:-1, 1:-1]
    assert inner.size and np.abs(inner).max() == 0.0



# ---- training of the guess network, bit for bit ------------------------------------------
# The states and weights are built from seeded uniforms by operations that IEEE arithmetic rounds
# the same everywhere.  tests/golden/c2p_net_bits.txt holds gradients and trained values of some
# of the parameters as hexadecimal floats, from kernels that evaluate every layer and sum in the
# order that the comments of csrc/dg_c2p_net.cu give.
NET_PICK, NET_GRAD, NET_TRAIN = slice(3, None, 61), (100, 300), ((300, 128), (4500, 2048), (5000, 2200))


def net_states(count):
    u = [di.uniform(77, s, np.arange(count)) for s in range(1, 9)]
    D = np.ldexp(0.5 + u[1], (12.0 * u[0]).astype(int) - 8)
    tau = D * np.ldexp(0.5 + u[3], (14.0 * u[2]).astype(int) - 7)
    cons = np.stack([D, tau * (u[4] - 0.5), tau * (u[5] - 0.5), tau * (u[6] - 0.5), tau])
    return cons, tau * (0.01 + 0.25 * u[7])


def net_params():
    p = mlp.init_params(di.uniform(5, 9, np.arange(mlp.N_PARAMS)))
    for name in ("b1", "b2"):
        o = mlp.OFFSETS[name]
        p[o:o + 64] = 0.4 * (di.uniform(5, 10, np.arange(o, o + 64)) - 0.5)
    return p.astype(np.float32)


def net_grad(pkg, params, cons, p):
    import torch
    net = pkg.abi.dg_c2p_net_create(params, mlp.DEFAULT_SCALES)
    grad = torch.empty(mlp.N_PARAMS, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    pkg.abi.dg_c2p_net_grad(net, cons.shape[1], cons.contiguous(), p.contiguous(), grad, loss)
    pkg.abi.dg_c2p_net_destroy(net)
    return grad.cpu().numpy(), np.float32(loss.item())


class Adam:
    """The update in FP32, every operation rounded on its own, the bias corrections from the host's powf."""

    def __init__(self, params, lr):
        self.p, self.lr = params.copy(), np.float32(lr)
        self.m, self.v, self.step = np.zeros_like(self.p), np.zeros_like(self.p), 0
        self.powf = ctypes.CDLL("libm.so.6").powf
        self.powf.restype, self.powf.argtypes = ctypes.c_float, [ctypes.c_float, ctypes.c_float]

    def update(self, g):
        f = np.float32
        self.step += 1
        self.m = f(0.9) * self.m + f(0.1) * g
        self.v = f(0.999) * self.v + f(0.001) * g * g
        b1, b2 = (f(1.0) - f(self.powf(b, self.step)) for b in (0.9, 0.999))
        self.p = self.p - self.lr * (self.m / b1) / (np.sqrt(self.v / b2) + f(1e-8))


@pytest.mark.parametrize("count,steps", [(96, 300), (1000, 3), (2048, 3), (2049, 3)])
def test_training_steps_are_adam_on_the_gradients(pkg, count, steps):
    """Every parameter after every step, one mini-batch each, is Adam's update of the one before with
    dg_c2p_net_grad's gradient, to the bit, whichever launch takes the mini-batch (the device's powf
    gives other bias corrections for some of the first 300 steps)."""
    import torch
    cons, p = (torch.from_numpy(x).cuda() for x in net_states(count))
    adam = Adam(net_params(), 1e-3)
    net = pkg.abi.dg_c2p_net_create(adam.p, mlp.DEFAULT_SCALES)
    for step in range(steps):
        adam.update(net_grad(pkg, adam.p, cons, p)[0])
        pkg.abi.dg_c2p_net_train(net, count, cons, p, 1, count, 1e-3)
        assert np.array_equal(pkg.abi.dg_c2p_net_get_params(net), adam.p), step
    pkg.abi.dg_c2p_net_destroy(net)


@pytest.mark.parametrize("tiles", [2, 16, 32, 256])
def test_gradient_is_the_sum_of_its_tiles_in_order(pkg, tiles):
    """Gradient and loss of 128 t samples are those of every 128, added one after another in FP32 (a
    power of two in the number of samples scales every term exactly)."""
    import torch
    cons, p = (torch.from_numpy(x).cuda() for x in net_states(128 * tiles))
    g, loss = net_grad(pkg, net_params(), cons, p)
    sg, sl = np.zeros_like(g), np.float32(0.0)
    for i in range(0, 128 * tiles, 128):
        q, one = net_grad(pkg, net_params(), cons[:, i:i + 128], p[i:i + 128])
        sg, sl = sg + q, sl + one
    assert np.array_equal(g, sg / np.float32(tiles)) and loss == sl / np.float32(tiles)


def net_grad_bits(pkg, count):
    import torch
    g, loss = net_grad(pkg, net_params(), *(torch.from_numpy(x).cuda() for x in net_states(count)))
    return np.concatenate([[loss], g[NET_PICK]])


def net_train_bits(pkg, count, batch):
    import torch
    cons, p = (torch.from_numpy(x).cuda() for x in net_states(count))
    net = pkg.abi.dg_c2p_net_create(net_params(), mlp.DEFAULT_SCALES)
    loss = torch.zeros(2, dtype=torch.float32, device="cuda")
    pkg.abi.dg_c2p_net_train(net, count, cons, p, 2, batch, 2e-3, loss)
    out = pkg.abi.dg_c2p_net_get_params(net)
    pkg.abi.dg_c2p_net_destroy(net)
    return np.concatenate([loss.cpu().numpy(), out[NET_PICK]])


def golden_bits(key):
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "c2p_net_bits.txt")) as f:
        rows = [ln.split() for ln in f if ln[0] != "#"]
    return np.array([float.fromhex(x) for row in rows if row[0] == key for x in row[1:]])


@pytest.mark.parametrize("count", NET_GRAD)
def test_gradient_bits(pkg, count):
    assert np.array_equal(net_grad_bits(pkg, count), golden_bits(f"grad{count}"))


@pytest.mark.parametrize("count,batch", NET_TRAIN)
def test_training_bits(pkg, count, batch):
    assert np.array_equal(net_train_bits(pkg, count, batch), golden_bits(f"train{count}x{batch}"))


def test_epochs_of_many_mini_batches(pkg):
    """An epoch longer than one launch takes (448 mini-batches): two launches, one running loss."""
    import torch
    cons, p = (torch.from_numpy(x).cuda() for x in net_states(449 * 2 + 1))
    params, out = net_params(), []
    for whole in (True, False):
        net = pkg.abi.dg_c2p_net_create(params, mlp.DEFAULT_SCALES)
        if whole:
            loss = torch.zeros(1, dtype=torch.float32, device="cuda")
            pkg.abi.dg_c2p_net_train(net, 449 * 2 + 1, cons, p, 1, 2, 1e-3, loss)
            total = loss.item()
        else:  # the same mini-batches, one call for each
            total, one = 0.0, torch.zeros(1, dtype=torch.float32, device="cuda")
            for i in range(0, 449 * 2 + 1, 2):
                c, t = cons[:, i:i + 2].contiguous(), p[i:i + 2].contiguous()
                pkg.abi.dg_c2p_net_train(net, t.numel(), c, t, 1, 2, 1e-3, one)
                total += one.item() * t.numel() / (449 * 2 + 1)
        out.append((pkg.abi.dg_c2p_net_get_params(net), total))
        pkg.abi.dg_c2p_net_destroy(net)
    assert np.array_equal(out[0][0], out[1][0])
    # 450 terms of FP32 rounding each
    assert abs(out[0][1] - out[1][1]) <= 450 * 2.0 ** -24 * out[1][1]
