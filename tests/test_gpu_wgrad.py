"""The weight gradients at the edges of their tiles, against the oracle's backward
pass at the bound of the other gradient tests.

Widths (4, 1, 32, 4): tiles of one and of 64 groups of channels (the fewest and the
most threads to a tile); (4, 11, 11, 4): the generator's; right-hand sides 1 (one per
tile column), 7 (does not divide the columns) and 11 (a second, ragged group)."""
import numpy as np
import pytest

import oracle
from paper_1601_03184_gb300 import (MRHS_F32, MRHS_PREC_FP32, Lattice, inputs, mrhs_nn_backward, mrhs_nn_create,
                                    mrhs_nn_forward, mrhs_nn_get_grads, mrhs_nn_get_weights, mrhs_nn_set_weights,
                                    mrhs_nn_zero_grads)

pytestmark = pytest.mark.gpu

DIMS, AGG = (4, 6, 4, 4), (2, 3, 2, 2)


@pytest.mark.parametrize("widths", [(4, 1, 32, 4), (4, 32, 32, 4), (4, 11, 11, 4)])
@pytest.mark.parametrize("nrhs", [1, 7, 11])
def test_weight_gradients(widths, nrhs):
    U = inputs.gauge_field(DIMS, 0.4, 5301)
    lat = Lattice(DIMS, AGG, 4, MRHS_PREC_FP32)
    lat.set_gauge(U)
    mrhs_nn_create(lat.ctx, widths, 1)
    nw, nb = oracle.nn_sizes(widths)
    rng = np.random.default_rng(5302)
    flat = np.concatenate([0.2 * rng.standard_normal(2 * nw), 0.3 * rng.standard_normal(nb)]).astype(np.float32)
    mrhs_nn_set_weights(lat.ctx, flat)
    flat = mrhs_nn_get_weights(lat.ctx, 1)
    W, b = flat[0:2 * nw:2].astype(complex) + 1j * flat[1:2 * nw:2], flat[2 * nw:].astype(float)
    x = inputs.gaussian_field((nrhs, lat.V, 12), 5303)
    dout = inputs.gaussian_field((nrhs, lat.V, 12), 5304)
    y = lat.field(nrhs, MRHS_F32)
    mrhs_nn_forward(lat.ctx, lat.to_device(x, MRHS_F32), y, nrhs)
    mrhs_nn_zero_grads(lat.ctx)
    mrhs_nn_backward(lat.ctx, lat.to_device(dout, MRHS_F32), None, nrhs)
    g = mrhs_nn_get_grads(lat.ctx)
    rW, rb, _ = oracle.nn_backward(DIMS, U, widths, W, b, x, dout, want_din=True)
    off = 0
    for i, o in zip(widths[:3], widths[1:]):  # layer by layer
        n = 9 * i * o
        got = g[2 * off:2 * (off + n):2] + 1j * g[2 * off + 1:2 * (off + n):2]
        assert np.linalg.norm(got - rW[off:off + n]) < 1e-4 * np.linalg.norm(rW[off:off + n]), (i, o)
        off += n
    lat.close()
