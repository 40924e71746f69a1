"""The fixed-length kernels of the lengths 2^a 3^b with wide radices (6 to 36):
every length as both map sides, with ragged images (odd height, so an uneven
expansion, and W < S), against the generic kernels of the same plan and, where
it is quick, the FP64 oracle.

Tolerances: a forward or adjoint map of these sizes is within 1e-6 of FP64 by
FP32 rounding alone (three FFTs of at most 6 passes, a few eps each in the
2-norm), so two implementations are within 2e-6 of each other; the oracle bound
is the suite's 1e-5.
"""
import numpy as np
import pytest

import oracle
from tests import _gpu

pytestmark = pytest.mark.gpu

WIDE = [144, 162, 216, 288, 324, 432, 486, 576, 648, 864, 972, 1152, 1296, 1458, 1728, 1944,
        2304, 2592, 2916, 3072, 3456, 3888]


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


def _all_results(f, torch, plan, x, g, target):
    """Forward map, adjoint of g, and the loss and gradient of the map g itself
    (one map for both sides: the loss's gradient jumps with the sign of a map
    cell near zero)."""
    m = torch.empty_like(g)
    gi = torch.empty_like(x)
    f.ft_forward(plan, x, m)
    f.ft_backward(plan, g, gi)
    loss, gl = f.ft_abs_mse_backward(plan, g, target, 2.0 / plan.W)
    torch.cuda.synchronize()
    assert f.ft_plan_tc_errors(plan) == 0
    return [t.cpu().numpy().astype(np.float64) for t in (m, gi, loss, gl)]


@pytest.mark.parametrize("interp", ["linear", "cubic"])
@pytest.mark.parametrize("N", WIDE)
def test_wide_length_matches_generic_kernels_and_oracle(torch, N, interp):
    from paper_1904_09409_gb300 import funnel as f
    H, W, n = N - 5, N - (6 if N % 4 else 2), 2
    rng = np.random.default_rng(N)
    imgs = rng.standard_normal((n, H, W)).astype(np.float32)
    x = torch.from_numpy(imgs).cuda()
    g = torch.from_numpy(rng.standard_normal((n, N, N)).astype(np.float32)).cuda()
    target = torch.from_numpy(rng.standard_normal((n, N, N)).astype(np.float32)).cuda()
    with f.Plan(H, W, N, N, interp) as plan:
        assert f.ft_plan_get_variant(plan) == 0
        fast = _all_results(f, torch, plan, x, g, target)
        f.ft_plan_set_variant(plan, 1)
        slow = _all_results(f, torch, plan, x, g, target)
    for a, b in zip(fast, slow):
        assert np.all(np.isfinite(a))
        assert _gpu.rel_l2(a, b) <= 2e-6
    if N <= 324:
        assert _gpu.rel_l2(fast[0][0], oracle.funnel_ref(imgs[0], N, N, interp)) <= 1e-5
        ref = oracle.adjoint_ref(g[0].cpu().numpy().astype(np.float64), H, W, interp)
        assert _gpu.rel_l2(fast[1][0], ref) <= 1e-5
