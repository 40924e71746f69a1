"""The fixed-length kernels of the lengths 2^a 3^b with wide radices (6 to 36) and of
the shortest lengths: every length as both map sides, with ragged images (odd
height, so an uneven expansion, and W < S), against the generic kernels of the
same plan and, where it is quick, the FP64 oracle.

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

SHORT = [64, 72, 96, 108]
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
@pytest.mark.parametrize("N", SHORT + WIDE)
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


FOURIER = [128, 144, 162, 192, 216, 256, 288, 324, 384, 432, 486, 512, 576, 648, 768, 864, 972, 1024, 1152, 1536, 2048]


@pytest.mark.parametrize("W", FOURIER)
def test_fourier_rows_match_generic_kernel(torch, W):
    """The register-resident chirp-z row kernels (n_slope = W) against the generic
    ones, forward and adjoint, with a number of rows that leaves the last block
    partly empty; same bound as between any two FP32 implementations above."""
    from paper_1904_09409_gb300 import funnel as f
    H, n = 96, 3
    rng = np.random.default_rng(W)
    x = torch.from_numpy(rng.standard_normal((n, H, W)).astype(np.float32)).cuda()
    g = torch.from_numpy(rng.standard_normal((n, H, W)).astype(np.float32)).cuda()
    out = []
    with f.Plan(H, W, W, H, "fourier") as plan:
        for variant in (0, 1):
            f.ft_plan_set_variant(plan, variant)
            m, gi = torch.empty_like(g), torch.empty_like(x)
            f.ft_forward(plan, x, m)
            f.ft_backward(plan, g, gi)
            torch.cuda.synchronize()
            out.append((m.cpu().numpy().astype(np.float64), gi.cpu().numpy().astype(np.float64)))
    for a, b in zip(*out):
        assert np.all(np.isfinite(a))
        assert _gpu.rel_l2(a, b) <= 2e-6
    lhs = float(np.sum(out[0][0] * g.cpu().numpy()))
    rhs = float(np.sum(out[0][1] * x.cpu().numpy()))
    scale = np.linalg.norm(out[0][0]) * np.linalg.norm(g.cpu().numpy().astype(np.float64))
    assert abs(lhs - rhs) <= 1e-5 * scale
