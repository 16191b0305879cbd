"""Row counts whose tiled block heights give more than 32 blocks and that the automatic partition of
the FP32 forms cuts into at most 32 blocks of another height instead: one per height and its
register kernel (csrc/k_tridiag.cu), against the oracle and beside the general kernel, which another
partition of the same rows takes, at the tolerances of the parity tests (2e-5 for FP32, 1e-12 after two
corrections).  Named, the automatic partition gives the automatic plan's result."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

ROWS = {5: 155, 7: 203, 9: 261, 10: 290, 11: 121, 13: 143, 14: 406, 15: 435, 17: 221, 18: 522, 19: 247, 20: 260,
        21: 231, 22: 242, 23: 253}


@pytest.mark.parametrize("precision", (1, 2))
@pytest.mark.parametrize("height", ROWS)
def test_blocks_of_any_height_match_oracle(height, precision):
    import paper_2104_08863_gb300 as P
    ny, nx, nz = ROWS[height], 24, 18
    faces = W.tanh_faces(ny, 1.5)
    g = oracle.Grid(nx, nz, faces)
    f = oracle.divergence(g, *W.random_velocity(11, nx, ny, nz))
    want = oracle.solve(g, f)
    # the oracle's dense (0, 0) system has a condition number that grows as ny^2
    tol = {1: 2e-5, 2: 1e-12}[precision] + 2.0 ** -53 * ny * ny
    plan = P.Plan(nx, ny, nz, faces, precision=precision, refine_steps=2, device="cuda:0")
    other = next(p for p in range(31, 0, -1) if ny % p == 0 and p != ny // height)
    named, given = (P.Plan(nx, ny, nz, faces, precision=precision, tridiag=P.PT_PDD_EXACT, pdd_parts=parts,
                           refine_steps=2, device="cuda:0")
                    for parts in (ny // height, other))   # given: the general kernel with the factors of a table
    rhs = torch.from_numpy(f).to("cuda:0", plan.dtype)
    if precision == 1:   # the refined form's gauge sum is not added up in a fixed order
        assert torch.equal(named.solve(rhs.clone()), plan.solve(rhs.clone()))
    for p in (plan, named, given):
        got = p.solve(rhs.clone())
        torch.cuda.synchronize()
        assert np.max(np.abs(got.double().cpu().numpy() - want)) <= tol * np.max(np.abs(want))
