"""Calls recorded into a CUDA graph keep their meaning: a replay gives the result of
a direct call on the inputs and the setup of the moment, whatever the context has done
with its workspaces in between."""
import pytest
import torch

from paper_1601_03184_gb300 import MRHS_DC_ALU, MRHS_F32, MRHS_PREC_FP32, Lattice, inputs, mrhs_trim

pytestmark = pytest.mark.gpu


def rel(a, b):
    return (torch.linalg.vector_norm((a - b).double()) / torch.linalg.vector_norm(b.double())).item()


def test_recorded_smoothing_outlives_the_workspace():
    """4^4 domains, 8 vectors, two sweeps: the direct call works on copies held by the
    context, which a trim frees and a smoothing of more vectors moves. Both give the
    smoother's result to the bound of the FP32 forms (1e-5 each)."""
    dims, agg, n = (8, 8, 8, 8), (4, 4, 4, 4), 8
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lat = Lattice(dims, agg, 8, MRHS_PREC_FP32)
        lat.set_gauge(inputs.gauge_field(dims, 0.4, 1601))
        lat.build_clover(-0.1, 1.2)
        gen = torch.Generator("cuda").manual_seed(2)
        b, x0, b2 = (torch.randn(lat.V * 24 * n, device="cuda", generator=gen) for _ in range(3))
        big = torch.randn(lat.V * 24 * 32, device="cuda", generator=gen)
        x = x0.clone()
        lat.sap(b, x, n, MRHS_F32, 2, 3)  # the workspace is there before the recording
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.sap(b, x, n, MRHS_F32, 2, 3)
        for step in (lambda: None, lambda: mrhs_trim(lat.ctx),
                     lambda: lat.sap(big, torch.zeros_like(big), 32, MRHS_F32, 2, 3)):
            step()
            b.copy_(b2)
            direct = x0.clone()
            lat.sap(b, direct, n, MRHS_F32, 2, 3)
            x.copy_(x0)
            g.replay()
            s.synchronize()
            assert rel(x, direct) <= 2e-5
        lat.close()


def test_recorded_coarse_stencil_follows_the_setup():
    """20 right-hand sides: after the recording D_c is rebuilt from other test vectors
    with the CUDA-core engine, which leaves the tensor-core operand images behind; the
    replay applies the new D_c (each form to FP32 accuracy, 1e-5)."""
    dims, agg, ntv, n = (8, 8, 8, 8), (4, 4, 4, 4), 8, 20
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lat = Lattice(dims, agg, ntv, MRHS_PREC_FP32)
        lat.set_gauge(inputs.gauge_field(dims, 0.4, 1602))
        lat.build_clover(-0.1, 1.2)
        for k in range(2):
            lat.set_tv(lat.to_device(inputs.test_vectors(ntv, dims, 2602 + k), MRHS_F32), MRHS_F32)
            lat.build_P()
            lat.build_Dc()
            if k == 0:
                x = torch.randn(lat.nagg * 4 * ntv * n, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
                y, direct = torch.zeros_like(x), torch.zeros_like(x)
                lat.apply_Dc(x, y, n, MRHS_F32)
                s.synchronize()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    lat.apply_Dc(x, y, n, MRHS_F32)
                lat.set_dc_engine(MRHS_DC_ALU)
        lat.apply_Dc(x, direct, n, MRHS_F32)
        g.replay()
        lat.sync()
        assert rel(y, direct) <= 2e-5
        lat.close()


def test_direct_smoothing_beside_a_recording():
    """A smoothing on its own stream while another stream is being captured neither fails
    nor ends the recording, though it takes its workspace anew each time."""
    dims, agg, n = (8, 8, 8, 8), (4, 4, 4, 4), 8
    own, s = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(own):
        lat = Lattice(dims, agg, 8, MRHS_PREC_FP32)
        lat.set_gauge(inputs.gauge_field(dims, 0.4, 1603))
        lat.build_clover(-0.1, 1.2)
        b = torch.randn(lat.V * 24 * n, device="cuda", generator=torch.Generator("cuda").manual_seed(6))
        x, y = torch.zeros_like(b), torch.zeros_like(b)
        lat.sap(b, x, n, MRHS_F32, 2, 3)
        mrhs_trim(lat.ctx)
    z = torch.zeros(16, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        z.add_(1)
        lat.sap(b, y, n, MRHS_F32, 2, 3)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, y) and bool((z == 1).all())
    lat.close()
