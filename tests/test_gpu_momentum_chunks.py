"""Momentum stages with few tiles and more than 512 rows, whose coefficients, a row chunk of them in
shared memory beside the FP64 kernel's edge fluxes, exceed the 48 KB that a kernel has without asking:
against the oracle, at the tolerances of the time step's parity tests."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 2e-5)])
def test_one_chunk_of_many_rows(precision, tol):
    import oracle
    import paper_2104_08863_gb300 as P
    from oracle.momentum import rk2_predictor
    nx, ny, nz, s, dt = 72, 520, 324, 1.2, 1e-4
    faces = W.tanh_faces(ny, s)
    u, v, w = W.poiseuille_plus_noise(1, W.ChannelCase("t", nx, ny, nz, s))
    want = rk2_predictor(oracle.Grid(nx, nz, faces), u, v, w, dt, 1e-3, 2e-3)
    plan = P.Plan(nx, ny, nz, faces, precision=precision, device="cuda:0")
    f = [torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0", plan.dtype) for a in (u, v, w)]
    plan.predict(*f, dt, 1e-3, 2e-3)
    torch.cuda.synchronize()
    scale = max(np.max(np.abs(a)) for a in want)
    for got, ref in zip(f, want):
        assert float(np.max(np.abs(got.double().cpu().numpy() - ref))) <= tol * scale
