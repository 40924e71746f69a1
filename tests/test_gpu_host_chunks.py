"""ft_detect_host over several chunks: the records and counts equal ft_forward and
ft_peaks on device buffers, with a shorter last chunk, with one that takes another
peak pass, with small images in large maps, whose workspace does not grow with the
batch, and without the memory for a full chunk.
"""
import numpy as np
import pytest

from tests import _gpu

pytestmark = pytest.mark.gpu

CHUNK = 24 << 20       # bytes of images per chunk


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


def _check(f, torch, plan, n, K, calls=2):
    """Records of ft_detect_host against ft_forward + ft_peaks, `calls` times."""
    g = torch.Generator(device="cuda").manual_seed(n + K)
    x = torch.randn((n, plan.H, plan.W), generator=g, device="cuda")
    with f.Plan(plan.H, plan.W, plan.S, plan.Hp) as ref:
        m = torch.empty((n, plan.Hp, plan.S), device="cuda")
        f.ft_forward(ref, x, m)
        want, want_n = f.ft_peaks(ref, m, K)
        torch.cuda.synchronize()
        want, want_n = want.cpu(), want_n.cpu()
        del m
    h = x.cpu().pin_memory()
    for _ in range(calls):
        out, cnt = f.ft_detect_host(plan, h, K)
        assert torch.equal(cnt, want_n)
        assert np.array_equal(out.numpy().view(np.uint8).reshape(-1), want.numpy().reshape(-1))
    return h


@pytest.mark.parametrize("H,W,n,K", [(1024, 1024, 14, 8),      # 6 + 6 + 2 images
                                     (512, 1024, 27, 40),      # 12 + 12 + 3
                                     (480, 640, 45, 8)])       # 20 + 20 + 5, in maps of 486 x 648
def test_several_chunks_match_device_calls(torch, monkeypatch, H, W, n, K):
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    S, Hp = (648, 486) if H == 480 else (W, H)
    per = CHUNK // (H * W * 4)
    assert n > 2 * per and n % per                       # three chunks, the last one shorter
    with f.Plan(H, W, S, Hp) as plan:
        if K == 40:                                      # the last chunk spreads its peak pass over the GPU
            assert f.ft_detect_launches(plan, per, K) == 4 and f.ft_detect_launches(plan, n % per, K) == 5
        _check(f, torch, plan, n, K)


def test_workspace_of_small_images_in_large_maps(torch):
    """64 images of 64^2 in maps of 2048^2 (16.8 MB of workspace each): beside the
    buffers of the batch (images, maps, records) the call holds the workspace of one
    chunk, the 16 images whose maps are 256 MiB, and its peak scratch (at most 0.5 MiB
    an image); the workspace of the whole batch would be 1 GiB."""
    from paper_1904_09409_gb300 import funnel as f
    n, N, K = 64, 2048, 8
    with f.Plan(64, 64, N, N) as plan:
        h = _check(f, torch, plan, n, K, calls=1)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with f.Plan(64, 64, N, N) as plan:
        free0 = torch.cuda.mem_get_info()[0]
        f.ft_detect_host(plan, h, K)
        used = free0 - torch.cuda.mem_get_info()[0]
    assert used <= n * (N * N * 4 + 64 * 64 * 4) + (320 << 20), used


def test_small_chunks_where_memory_is_short(torch):
    """A plan that cannot have the workspace of a full chunk works in chunks of 8."""
    from paper_1904_09409_gb300 import funnel as f
    n, N, K = 44, 256, 6
    with f.Plan(N, N, N, N) as plan:
        h = _check(f, torch, plan, n, K, calls=1)
        want = [t.clone() for t in f.ft_detect_host(plan, h, K)]
        x = torch.zeros((2 * n, N, N), device="cuda")
        m = torch.empty_like(x)
        f.ft_plan_inject_alloc_failures(plan, 1)
        with pytest.raises(f.FunnelError):
            f.ft_forward(plan, x, m)                     # the plan has no workspace now
        f.ft_plan_inject_alloc_failures(plan, 1)
        got = f.ft_detect_host(plan, h, K)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        f.ft_plan_inject_alloc_failures(plan, 1)
        with pytest.raises(f.FunnelError):
            f.ft_forward(plan, x, m)
        f.ft_plan_inject_alloc_failures(plan, 2)         # nor the memory for 8 images
        with pytest.raises(f.FunnelError) as e:
            f.ft_detect_host(plan, h, K)
        assert e.value.status == f.FT_ERR_OOM
        got = f.ft_detect_host(plan, h, K)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
