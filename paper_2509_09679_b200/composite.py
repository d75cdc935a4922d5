"""Gradients of the composite transform Q = Q1 (x) Q2 (paper Sec. 3.3) composed from the library's entry points.

With a token row as an n1 x n2 matrix X and Y = Q1 (X Q2^T), for an upstream gradient G = dL/dY:

    G' = Q1^T G                       gradient at X' = X Q2^T (the rows after the butterfly)
    dL/dX      = G' Q2                = bfq_composite_inverse(G): per run, dx of the butterfly for upstream G'
    dL/dtheta2 = butterfly d-theta of the n1 * tokens runs with upstream G'   (bfq_backward on the n2-point plan)
    dL/dQ1     = sum over tokens of G X'^T                                    (a small dense product)
    dL/dparams = dL/dQ1 pulled back through Q1 = (I - A)(I + A)^-1 (A skew from the parameters): with
                 M = (I + A)^-1, dQ1 = -(I + Q1) dA M, so dL/dA = -(I + Q1)^T (dL/dQ1) M^T and the parameter (i < j)
                 receives dL/dA[i][j] - dL/dA[j][i].

bfq_composite_backward computes the first four in one pass for 128 <= n2 <= 1024, bfq_cayley_backward the last; other sizes and
types are composed from the butterfly's own entry points and torch (the n1 x n1 algebra in float64).
"""
from __future__ import annotations

import torch

from .binding import Plan


def cayley_pullback(params: torch.Tensor, n1: int, dQ1: torch.Tensor) -> torch.Tensor:
    """dL/dparams from dL/dQ1 (both on the same device; float64 inside)."""
    p = params.double()
    iu = torch.triu_indices(n1, n1, 1, device=p.device)
    A = torch.zeros((n1, n1), dtype=torch.float64, device=p.device)
    A[iu[0], iu[1]] = p
    A = A - A.t()
    eye = torch.eye(n1, dtype=torch.float64, device=p.device)
    M = torch.linalg.inv(eye + A)
    Q1 = (eye - A) @ M
    dA = -(eye + Q1).t() @ dQ1.double() @ M.t()
    return (dA - dA.t())[iu[0], iu[1]].to(params.dtype)


def _one_pass(plan: Plan, n1: int) -> bool:
    """Whether bfq_composite_backward takes these sizes (its limits are in the header)."""
    return 128 <= plan.n <= 1024 and 2 <= n1 <= 64 and 12 * n1 * (plan.n + 4) + 4 * n1 * (-(-n1 // 8) * 8) <= 227 * 1024


def composite_backward(plan: Plan, q1: torch.Tensor, params: torch.Tensor | None, x: torch.Tensor, g: torch.Tensor):
    """x, g: [tokens][n1 * n2] (same dtype).  Returns (dx, dtheta2, dQ1, dparams or None)."""
    n1, n2 = q1.shape[0], plan.n
    tokens = x.shape[0]
    if _one_pass(plan, n1) and q1.dtype == torch.float32:
        g2 = g.reshape(tokens, n1 * n2).contiguous()
        g2 = g2 if g2.dtype in (torch.float32, torch.bfloat16) else g2.float()
        if g2.data_ptr() % 16:  # g may lie at any address, the kernel's rows may not
            g2 = g2.clone()
        dx, dtheta2, dQ1 = plan.composite_backward(q1.contiguous(), x.reshape(tokens, n1 * n2).contiguous(), g2)
    else:
        gp = torch.einsum("ki,rkj->rij", q1, g.reshape(tokens, n1, n2).float())      # G' = Q1^T G
        runs_x = x.reshape(tokens * n1, n2)
        runs_g = gp.reshape(tokens * n1, n2).to(x.dtype)
        dx_runs, dtheta2 = plan.backward(runs_x, runs_g)                             # dx = G' Q2 per run, d-theta summed over runs
        xp = plan.forward(runs_x, out_dtype=torch.float32).reshape(tokens, n1, n2)   # X' = X Q2^T
        dQ1 = torch.einsum("rij,rkj->ik", g.reshape(tokens, n1, n2).float(), xp)
        dx = dx_runs.reshape(tokens, n1 * n2)
    if params is None:
        return dx, dtheta2, dQ1, None
    if params.dtype == torch.float32 and q1.dtype == torch.float32 and params.device == plan.device and params.dim() == 1 and params.is_contiguous() and 2 <= n1 <= 64:
        return dx, dtheta2, dQ1, plan.cayley_backward(params, q1.contiguous(), dQ1.contiguous())
    return dx, dtheta2, dQ1, cayley_pullback(params, n1, dQ1)
