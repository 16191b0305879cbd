"""The out-of-place projection and adjoint (projection_step_to, projection_step_adjoint_to) behind
ProjectionFn: bit for bit the in-place calls, on the vector widths of the stencils (nx a multiple of 4,
of 2 only), with and without the 16-byte alignment and the layout that they read in place; the inputs
are not written; aliased buffers are refused."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _plan(nx, ny, nz, precision):
    import paper_2104_08863_gb300 as P
    return P, P.Plan(nx, ny, nz, W.tanh_faces(ny, 1.4), precision=precision, device="cuda:0")


def _fields(plan, seed, how):
    gen = torch.Generator(device="cuda:0").manual_seed(seed)
    out = []
    for s in (plan.cell_shape, plan.v_shape, plan.cell_shape):
        t = torch.randn(s, generator=gen, device="cuda:0", dtype=plan.dtype)
        if how == "misaligned":     # contiguous, one value past a 16-byte boundary
            b = torch.empty(t.numel() + 1, device="cuda:0", dtype=plan.dtype)
            b[1:] = t.reshape(-1)
            t = b[1:].view(s)
        elif how == "strided":      # every second line of a larger tensor: its clone is contiguous
            b = torch.zeros((s[0], 2 * s[1], s[2]), device="cuda:0", dtype=plan.dtype)
            b[:, ::2] = t
            t = b[:, ::2]
        elif how == "negated":      # contiguous, the memory holding -t
            t = torch._neg_view(-t)
        out.append(t)
    return out


@pytest.mark.parametrize("how", ["plain", "misaligned", "strided", "negated"])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny,nz", [(8, 2, 2), (18, 5, 6), (36, 7, 9), (256, 3, 4)])
def test_projection_fn_equals_in_place_calls(nx, ny, nz, precision, how):
    P, plan = _plan(nx, ny, nz, precision)
    x = _fields(plan, 1, how)
    keep = [t.clone() for t in x]
    want = [t.clone().contiguous() for t in x]
    plan.project(*want, 0.1)
    leaves = [t.requires_grad_(True) for t in x]
    out = P.ProjectionFn.apply(*leaves, plan, 0.1)
    for a, b in zip(out, want):
        assert torch.equal(a, b)
    g = _fields(plan, 2, how)
    gw = [t.clone().contiguous() for t in g]
    plan.project_adjoint(*gw)
    grads = torch.autograd.grad(out, leaves, grad_outputs=g)
    for a, b in zip(grads, gw):
        assert torch.equal(a, b)
    for a, b in zip(x, keep):
        assert torch.equal(a.detach(), b)


def test_permuted_fields():
    """A dense permuted velocity is refused (its copy keeps the layout), a gradient of that layout is not."""
    P, plan = _plan(16, 4, 6, 0)
    turn = lambda t: t.permute(2, 0, 1).contiguous().permute(1, 2, 0)
    x, g = _fields(plan, 6, "plain"), _fields(plan, 7, "plain")
    with pytest.raises(ValueError):
        P.ProjectionFn.apply(*map(turn, x), plan, 0.1)
    leaves = [t.requires_grad_(True) for t in x]
    out = P.ProjectionFn.apply(*leaves, plan, 0.1)
    want = torch.autograd.grad(out, leaves, grad_outputs=g, retain_graph=True)
    for a, b in zip(torch.autograd.grad(out, leaves, grad_outputs=list(map(turn, g))), want):
        assert torch.equal(a, b)


def test_zero_tensor_gradient():
    P, plan = _plan(16, 4, 6, 0)
    leaves = [t.requires_grad_(True) for t in _fields(plan, 8, "plain")]
    out = P.ProjectionFn.apply(*leaves, plan, 0.1)
    zeros = [torch._efficientzerotensor(tuple(t.shape), device=t.device, dtype=t.dtype) for t in out]
    for a in torch.autograd.grad(out, leaves, grad_outputs=zeros):
        assert not a.any()


def test_refused_arguments():
    P, plan = _plan(16, 4, 6, 0)
    L, st = P._native.lib(), torch.cuda.current_stream().cuda_stream
    x, o = _fields(plan, 3, "plain"), _fields(plan, 4, "plain")
    xp, op = [t.data_ptr() for t in x], [t.data_ptr() for t in o]
    ok = lambda i, q, h=plan._h, dt=0.1: L.projection_step_to(h, *i, *q, dt, st)
    adj = lambda i, q, h=plan._h: L.projection_step_adjoint_to(h, *i, *q, st)
    assert ok(xp, op) == P._native.PS_OK and adj(xp, op) == P._native.PS_OK
    for bad in ([xp[0], op[1], op[2]], [op[0], op[1], op[0]], [xp[2], op[1], op[2]], [op[0] + 8, op[1], op[2]], [0, op[1], op[2]]):
        assert ok(xp, bad) == P._native.PS_EINVAL and adj(xp, bad) == P._native.PS_EINVAL
    assert ok(xp, op, dt=0.0) == P._native.PS_EINVAL
    _, ref = _plan(16, 4, 6, 2)
    assert ok(xp, op, h=ref._h) == P._native.PS_EUNSUPPORTED
    torch.cuda.synchronize()


def test_refined_plan_still_projects():
    P, plan = _plan(16, 4, 6, 2)
    x = _fields(plan, 5, "plain")
    want = [t.clone() for t in x]
    plan.project(*want, 0.1)
    for a, b in zip(P.ProjectionFn.apply(*x, plan, 0.1), want):
        assert torch.allclose(a, b, rtol=0, atol=1e-12)   # the gauge sum's atomics
