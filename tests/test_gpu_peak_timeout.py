"""The peak pass over the whole GPU after a step 4 whose waits ran out: the blocks
that gave up write no tile maxima, so the pass meets whatever the workspace held,
here spectra of both signs.  It stays within its bins and buffers, the error is
reported, and the next call gives the right records."""
import pytest

from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


@pytest.mark.parametrize("thr", [float("-inf"), 0.0])
def test_detect_after_a_timeout_of_step_4(torch, monkeypatch, thr):
    from paper_1904_09409_gb300 import funnel as f
    monkeypatch.setenv("FT_PEAKS", "multi")
    N, K = 256, 8
    g = torch.Generator(device="cuda").manual_seed(2)
    x = torch.randn((8, N, N), generator=g, device="cuda")
    m = torch.zeros_like(x)
    with f.Plan(N, N, N, N) as plan, f.Plan(N, N, N, N) as fresh:
        assert f.ft_detect_launches(plan, 2, K) == 5
        f.ft_forward(plan, x, m)                        # 8 images' spectra where 2 images' maxima will be
        f.ft_plan_set_wait_cycles(plan, 0)
        f.ft_detect(plan, x, m, K, thr, batch=2)
        with pytest.raises(f.FunnelError) as e:
            f.ft_plan_tc_errors(plan)
        assert e.value.status == f.FT_ERR_TIMEOUT
        f.ft_plan_set_wait_cycles(plan, f.FT_WAIT_CYCLES_DEFAULT)
        out, cnt = f.ft_detect(plan, x, m, K, thr, batch=2)
        m2 = torch.empty_like(x)
        out2, cnt2 = f.ft_detect(fresh, x, m2, K, thr, batch=2)
        torch.cuda.synchronize()
        assert f.ft_plan_tc_errors(plan) == 0
    assert torch.equal(m[:2], m2[:2]) and torch.equal(cnt, cnt2) and torch.equal(out, out2)
