"""The sums of the weight gradients. Unit gauge field, every layer the identity on the
first four channels, no bias: all activations and their gradients are the input and the
output's gradient themselves, so that the weight gradients are plain sums of products.

On whole numbers of 560 to 591 the FP32 sums of up to 24 products (2 * 24 * 591^2 < 2^24)
are exact, those of 28 are not, and every sum of sums has more bits than the result: the
gradients equal the oracle's, rounded once to FP32."""
import numpy as np
import pytest
import torch

import oracle
from paper_1601_03184_gb300 import (MRHS_F32, MRHS_PREC_FP32, Lattice, inputs, mrhs_nn_backward, mrhs_nn_create,
                                    mrhs_nn_forward, mrhs_nn_get_grads, mrhs_nn_set_weights, mrhs_nn_zero_grads)

pytestmark = pytest.mark.gpu

DIMS, AGG, NRHS = (4, 6, 4, 4), (2, 3, 2, 2), 8


def gradients(widths, x, dout):
    """dW of all layers as [9][out][in] complex, and the flat weights"""
    lat = Lattice(DIMS, AGG, 4, MRHS_PREC_FP32)
    U = inputs.unit_gauge_field(DIMS)
    lat.set_gauge(U)
    mrhs_nn_create(lat.ctx, widths, 1)
    layers = list(zip(widths[:3], widths[1:]))
    W = []
    for i, o in layers:
        w = np.zeros((9, o, i), complex)
        w[0, range(4), range(4)] = 1
        W.append(w.ravel())
    W, b = np.concatenate(W), np.zeros(widths[1] + widths[2])
    flat = np.concatenate([np.stack((W.real, W.imag), -1).ravel(), b]).astype(np.float32)
    mrhs_nn_set_weights(lat.ctx, flat)
    if isinstance(x, np.ndarray):
        x, dout = lat.to_device(x, MRHS_F32), lat.to_device(dout, MRHS_F32)
    y = lat.field(NRHS, MRHS_F32)
    mrhs_nn_forward(lat.ctx, x, y, NRHS)
    mrhs_nn_zero_grads(lat.ctx)
    mrhs_nn_backward(lat.ctx, dout, None, NRHS)
    g = mrhs_nn_get_grads(lat.ctx)
    lat.close()
    got, off = [], 0
    for i, o in layers:
        n = 2 * 9 * i * o
        got.append((g[off:off + n:2] + 1j * g[off + 1:off + n:2].astype(complex)).reshape(9, o, i))
        off += n
    return got, U, W, b


# groups of 256 threads to a tile of channels, 64, 28 and 4 (tiles of 2, 6, 14 and 48 products
# a thread)
@pytest.mark.parametrize("widths", [(4, 4, 4, 4), (4, 8, 8, 4), (4, 11, 11, 4), (4, 32, 32, 4)])
def test_whole_numbers(widths):
    rng = np.random.default_rng(1901)
    x, dout = (rng.integers(560, 592, (2, NRHS, int(np.prod(DIMS)), 12)) for _ in range(2))
    x, dout = x[0] + 1j * x[1], dout[0] + 1j * dout[1]
    got, U, W, b = gradients(widths, x, dout)
    ref = oracle.nn_backward(DIMS, U, widths, W, b, x, dout, want_din=True)[0]
    off = 0
    for g in got:
        r = ref[off:off + g.size].reshape(g.shape)
        off += g.size
        assert np.array_equal(g.real, r.real.astype(np.float32).astype(float))
        assert np.array_equal(g.imag, r.imag.astype(np.float32).astype(float))


def test_range():
    """Sums that leave the range of FP32 (products of 2^120, more than a thousand to a
    thread): infinite where the total is, finite where the halves of the lattice cancel."""
    widths, V = (4, 32, 32, 4), int(np.prod(DIMS))
    x, dout = (torch.zeros(V, 12, 2, NRHS, device="cuda") for _ in range(2))
    x[:, :, 0], dout[:, :, 0] = 1, 2.0 ** 120
    for g in gradients(widths, x, dout)[0]:
        assert np.all(g[0, :4, :4].real == np.inf) and np.all(g[0, 4:].real == 0)
    dout[V // 2:] *= -1
    for g in gradients(widths, x, dout)[0]:
        assert np.all(g[0, :4, :4] == 0)
