"""The probe-residual subspace of the fit: S = Rb^T W Rb, the one matrix of the eigen-solver that is not a plain Gram matrix, and the basis made
of it, read through the correction O - O^sp.

The scratch of a head holds, in float64, Xb [M][d] Rb [M][d] G [d][d] B [d][d] S [d][d] mu_x [d] mu_R [d] s_x [d] wt [M]; it is found in the attend
workspace by its weights, which follow from the exported plan."""
import numpy as np
import pytest
import torch

from paper_2608_18484_b200 import binding as B
from tests.gpu_util import to_np

pytestmark = pytest.mark.gpu

EPS = {torch.bfloat16: 2.0 ** -24, torch.float32: 2.0 ** -53}       # unit roundoff of the Gram matrices and of the eigen-solver


def _fit_scratch(plan, M, d):
    w = B.sparsepr_plan_export(plan)["probe_w"][0].astype(np.float64)
    wt = M * w / w.sum()
    assert wt.max() > 1.5 * wt.min()                                # roundings of w r differ from row to row
    ws = plan.attend_workspace.cpu().numpy().view(np.float64)
    with np.errstate(invalid="ignore"):
        at = [i for i in np.flatnonzero(np.abs(ws - wt[0]) <= 1e-14 * wt[0]) if np.allclose(ws[i:i + M], wt, rtol=1e-14, atol=0)]
    assert len(at) == 1
    o, out = at[0], {"wt": wt}
    for name, shape in (("s_x", (d,)), ("mu_R", (d,)), ("mu_x", (d,)), ("S", (d, d)), ("B", (d, d)), ("G", (d, d)), ("Rb", (M, d))):
        o -= int(np.prod(shape))
        out[name] = ws[o:o + int(np.prod(shape))].reshape(shape)
    return out


@pytest.mark.parametrize("M", [33, 96])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128), (torch.float32, 64)])
def test_residual_subspace(dtype, d, M):
    N, r, eps = 1537, 16, EPS[dtype]
    gen = torch.Generator(device="cuda").manual_seed(M + d)
    ids = torch.randint(24, (N,), device="cuda", generator=gen) % torch.randint(1, 25, (N,), device="cuda", generator=gen)   # regions of unequal size
    mu = torch.randn(2, 24, d, device="cuda", generator=gen)
    Q, K = [(mu[0][ids] + 0.5 * torch.randn(N, d, device="cuda", generator=gen))[None, None].to(dtype) for _ in range(2)]
    # values of r directions and a hundredth of that beside them: the retained eigenvalues of S lie apart from the others
    V = (mu[1][ids, :r] + 0.5 * torch.randn(N, r, device="cuda", generator=gen)) @ torch.randn(r, d, device="cuda", generator=gen)
    V = (V + 0.01 * torch.randn(N, d, device="cuda", generator=gen))[None, None].to(dtype)
    plan = B.sparsepr_plan(Q, K, V, density=0.2, block=64, n_probe=M, r_out=r, lam=1.0, softmax_scale=2.0 / d)
    O, Osp = B.sparsepr_attend(plan, Q, K, V, return_sparse=True)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    f = _fit_scratch(plan, M, d)
    S, Rb = f["S"], f["Rb"]
    assert np.array_equal(S, S.T)
    # a product rounds w r, r and every addition
    assert np.all(np.abs(S - Rb.T @ (f["wt"][:, None] * Rb)) <= (M + 3) * eps * (np.abs(Rb).T @ (f["wt"][:, None] * np.abs(Rb))))
    # O - O^sp = (x - mu_x) / s_x B Psi Psi^T + mu_R = y Psi Psi^T + mu_R.  The solver's basis is that of S + E, ||E|| <= 4 d eps ||S||, which turns
    # eigenvectors i and j into each other by E_ij / (lam_i - lam_j): only retained against dropped ones (i, j) move the projection of y.
    # The output (2^-23, 2^-9) and the map (2^-23, bf16 words 2^-16) round.  (Probe rows are exact and left out.)
    rows = np.setdiff1d(np.arange(N), B.sparsepr_plan_export(plan)["probe_idx"][0])
    lam, vec = np.linalg.eigh(S)
    Psi = vec[:, -r:]
    x = to_np(Osp[0, 0])[rows]
    y = (x - f["mu_x"]) / f["s_x"] @ f["B"]
    want = x + f["mu_R"] + y @ Psi @ Psi.T
    part = np.linalg.norm(y @ vec, axis=0)                          # of y along each eigenvector
    turn = 4 * d * eps * lam[-1] / (lam[None, -r:] - lam[:-r, None])
    basis = np.sqrt((turn ** 2 * (part[None, -r:] ** 2 + part[:-r, None] ** 2)).sum())
    store = 2.0 ** -9 if dtype == torch.bfloat16 else 2.0 ** -23
    words = 2.0 ** -16 if dtype == torch.bfloat16 else 2.0 ** -23
    bound = basis + d * words * np.linalg.norm(y) + 2 * store * np.linalg.norm(want)
    err = np.linalg.norm(to_np(O[0, 0])[rows] - want)
    assert bound < 0.05 * np.linalg.norm(y @ Psi)                    # (at most 0.03: bf16, M = 33, d = 128) a bound that says something
    assert err <= bound, (err, bound)
