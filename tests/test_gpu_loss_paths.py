"""ft_abs_mse_backward where the row kernel does not add up the loss: the partials
are summed by a launch of their own when the columns run a fixed-length kernel and
the rows do not (the band-limited interpolator, an n_slope without a schedule), and
the loss gradient goes through the workspace when the columns have no schedule.
Same bounds as between the fused call and its two parts elsewhere: FP32 rounding of
a sum of squares (2e-6) and of two transforms (1e-6, 1e-5 against FP64)."""
import numpy as np
import pytest

import oracle
from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


@pytest.mark.parametrize("H,W,S,Hp,interp,space", [
    (120, 128, 128, 128, "fourier", "regular"),     # register-resident chirp-z rows
    (100, 64, 72, 144, "fourier", "regular"),       # generic chirp-z rows
    (100, 48, 54, 128, "linear", "regular"),        # n_slope 54 has no schedule
    (48, 100, 48, 128, "cubic", "inverse"),         # nor has 48
    (50, 48, 64, 54, "linear", "regular"),          # n_intercept 54 has none: through the workspace
])
def test_loss_backward_equals_the_two_calls(torch, H, W, S, Hp, interp, space):
    from paper_1904_09409_gb300 import funnel as f
    n = 3
    rng = np.random.default_rng(H + S + Hp)
    P = torch.from_numpy(rng.standard_normal((n, Hp, S)).astype(np.float32) * 20).cuda()
    t = torch.from_numpy(rng.random((n, Hp, S)).astype(np.float32)).cuda()
    with f.Plan(H, W, S, Hp, interp, space) as plan:
        loss_a, dP = f.ft_abs_mse_grad(plan, P, t, 2.0 / S)
        gx_a = torch.empty((n, H, W), device="cuda")
        f.ft_backward(plan, dP, gx_a)
        loss_b, gx_b = f.ft_abs_mse_backward(plan, P, t, 2.0 / S)
        loss_c, gx_c = f.ft_abs_mse_backward(plan, P, t, 2.0 / S)
        torch.cuda.synchronize()
    assert torch.equal(loss_b, loss_c) and torch.equal(gx_b, gx_c)
    la, lb = loss_a.cpu().numpy().astype(np.float64), loss_b.cpu().numpy().astype(np.float64)
    for i in range(n):
        p64, t64 = P[i].cpu().numpy().astype(np.float64), t[i].cpu().numpy().astype(np.float64)
        ref = float(np.mean((np.abs(p64) * (2.0 / S) - t64) ** 2))
        assert abs(lb[i] - ref) <= 2e-6 * ref and abs(la[i] - lb[i]) <= 2e-6 * ref
        assert _gpu.rel_l2(gx_b[i].cpu().numpy(), gx_a[i].cpu().numpy().astype(np.float64)) <= 1e-6
        adj = oracle.adjoint_ref(dP[i].cpu().numpy().astype(np.float64), *((W, H) if space == "inverse" else (H, W)),
                                 interp)
        assert _gpu.rel_l2(gx_b[i].cpu().numpy(), adj.T if space == "inverse" else adj) <= 1e-5
