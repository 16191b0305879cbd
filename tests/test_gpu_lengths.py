"""Every specialised transform length (csrc/k_fft_x_fast.cuh, csrc/k_fft_z_fast.cuh): the forward and
the inverse x- and z-transforms through the solve, against the oracle, in all three precisions (FP64
Stockham stages with fused twiddles and the paired real split, at even and odd half-lengths; the FP32
register transforms; the FP64 streams of the refined form).  Tolerances as in the parity tests.  The
grids are small in the other directions and ragged against the tiles (an odd number of lines or
planes per CTA)."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 2e-5, 2: 1e-12}
HALF = [8, 9, 12, 16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256, 288, 324,
        384, 432, 486, 512, 576, 648, 729, 768, 1024]
NZ = [16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256, 288, 324, 384, 432,
      486, 512, 576, 648, 729, 768, 864, 1024]


def _check(nx, ny, nz, precision):
    import paper_2104_08863_gb300 as P
    faces = W.tanh_faces(ny, 1.6)
    g = oracle.Grid(nx, nz, faces)
    f = oracle.divergence(g, *W.random_velocity(nx + nz, nx, ny, nz))
    want = oracle.solve(g, f)
    plan = P.Plan(nx, ny, nz, faces, precision=precision, refine_steps=2, device="cuda:0")
    got = plan.solve(torch.from_numpy(f).to("cuda:0", plan.dtype))
    torch.cuda.synchronize()
    err = np.max(np.abs(got.double().cpu().numpy() - want)) / np.max(np.abs(want))
    assert err <= TOL[precision]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("half", HALF)
def test_every_x_length(half, precision):
    _check(2 * half, 7, 9, precision)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nz", NZ)
def test_every_z_length(nz, precision):
    _check(36, 5, nz, precision)
