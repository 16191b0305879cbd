"""Batches whose spectra exceed the L2, so that the FP32 forms share a few branches of the graph
between the instances (csrc/batch.cu), and batches on the other side of that line: every instance
equals its solve by a plan of its own, which runs the same kernels on the same data (bitwise in
FP32; the refined form sums its mean with atomic additions, whose order moves the last bits: 1e-13),
also after a second capture on other buffers and in place."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

# (nx, ny, nz) and how many of each: about 170 MB of FP32 half spectra, and about 17 MB
LARGE = [((256, 128, 128), 9), ((64, 33, 48), 3), ((192, 96, 96), 3)]
SMALL = [((64, 33, 48), 4), ((128, 64, 32), 12)]


@pytest.mark.parametrize("shapes,precision", [(LARGE, 0), (LARGE, 1), (LARGE, 2), (SMALL, 1)])
def test_batch_equals_single_solves(shapes, precision):
    import paper_2104_08863_gb300 as P
    specs = [dict(nx=nx, ny=ny, nz=nz, y_faces=W.tanh_faces(ny, 1.4)) for (nx, ny, nz), n in shapes for _ in range(n)]
    specs = specs[::2] + specs[1::2]
    batch = P.BatchPlan(specs, precision=precision)
    gen = torch.Generator(device="cuda").manual_seed(3)
    rhs = [torch.randn(s["ny"], s["nz"], s["nx"], device="cuda", dtype=batch.dtype, generator=gen) for s in specs]
    want = []
    for s, f in zip(specs, rhs):
        plan = P.Plan(s["nx"], s["ny"], s["nz"], s["y_faces"], precision=precision, device="cuda:0")
        want.append(plan.solve(f.clone()))
    first = batch.solve(rhs)
    for _ in range(2):
        again = batch.solve(rhs)
    if precision != 2:
        inplace = [f.clone() for f in rhs]
        batch.solve(inplace, inplace)
    else:
        inplace = again
    torch.cuda.synchronize()
    for w, *got in zip(want, first, again, inplace):
        for g in got:
            if precision == 1:
                assert torch.equal(g, w)
            else:
                assert float((g - w).abs().max()) <= 1e-13 * float(w.abs().max())
