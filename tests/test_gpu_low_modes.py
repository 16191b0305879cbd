"""The modes solved by extra CTAs of the wall-normal launch (csrc/low_modes.cuh): the (0, 0) mode of
every plan and the FP64 low modes of the FP32 forms, at the row counts where their split over
threads can go wrong (fewer rows than threads, one more or less than a multiple of the thread
count, the counts on both sides of the launch of their own above 3072 rows), against the oracle.

On the grids below kx <= 4 and |kz| <= 4 are all the modes, so an FP32 plan with 4 low modes solves
every system in FP64: its error is the FP32 transforms' (2e-5, as in the parity tests), and a
refined plan's two corrections bring it to 1e-12."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,precision", [(ny, p) for ny in (2, 3, 31, 33, 127, 128, 129, 384) for p in (0, 1, 2)]
                         + [(3072, 1), (3076, 0), (3076, 1)])
def test_modes_solved_apart_match_oracle(ny, precision):
    import paper_2104_08863_gb300 as P
    nx, nz = 8, 9
    # the oracle solves its (0, 0) system by a dense LU whose condition number grows as ny^2 (the
    # second difference on ny rows): its own rounding is up to 2^-53 ny^2 of the result
    tol = {0: 1e-12, 1: 2e-5, 2: 1e-12}[precision] + 2.0 ** -53 * ny * ny
    faces = W.tanh_faces(ny, 1.3)
    g = oracle.Grid(nx, nz, faces)
    f = oracle.divergence(g, *W.random_velocity(7, nx, ny, nz))
    want = oracle.solve(g, f)
    plan = P.Plan(nx, ny, nz, faces, precision=precision, fp64_low_modes=4, refine_steps=2, device="cuda:0")
    got = plan.solve(torch.from_numpy(f).to("cuda:0", plan.dtype))
    torch.cuda.synchronize()
    err = np.max(np.abs(got.double().cpu().numpy() - want)) / np.max(np.abs(want))
    assert err <= tol
