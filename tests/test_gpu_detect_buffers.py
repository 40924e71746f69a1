"""ft_detect where the buffers of the pass that its cost model prefers are not
there: a call captured into a graph, which can allocate nothing, takes a pass whose
buffers earlier calls left, and a call whose allocation fails the pass that needs the
least, with the same records.
"""
import pytest

from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


# (image H, W, n_slope, n_intercept, space, batch and top_k of the call before, batch
# and top_k of the captured call)
CAPTURED = [
    # 32 x 8 tiles from step 4, fewer bytes than the 16 x 16 tiles of ft_peaks: the
    # captured call prefers the per-tile keys, then a smaller batch that does
    (768, 648, 648, 768, "regular", 8, 8, 8, 200),
    (768, 648, 648, 768, "regular", 16, 8, 4, 300),
    # the same map of the inverse space
    (648, 768, 648, 768, "inverse", 8, 8, 8, 200),
    # equal tile counts; the keys' buffers first, then tile maxima
    (480, 640, 648, 486, "regular", 8, 8, 8, 100),
    (768, 648, 648, 768, "regular", 8, 200, 8, 8),
    # whole-GPU pass first, the one-block pass or the keys captured
    (1024, 1024, 1024, 1024, "regular", 4, 200, 4, 8),
    (1024, 1024, 1024, 1024, "regular", 4, 100, 4, 1000),
]


@pytest.mark.parametrize("H,W,S,Hp,space,b0,k0,b1,k1", CAPTURED)
@pytest.mark.parametrize("call", ["ft_detect", "ft_detect_batches"])
def test_captured_call_takes_buffers_of_earlier_ones(torch, monkeypatch, H, W, S, Hp, space, b0, k0, b1, k1, call):
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    g = torch.Generator(device="cuda").manual_seed(H + k1)
    x = torch.randn((b0, H, W), generator=g, device="cuda")
    m = torch.empty((b0, Hp, S), device="cuda")
    out = torch.zeros(b1 * k1 * f.PEAK_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(b1, dtype=torch.int32, device="cuda")
    xs = x[:b1].contiguous()
    with f.Plan(H, W, S, Hp, space=space) as plan, f.Plan(H, W, S, Hp, space=space) as fresh:
        f.ft_detect(plan, x, m, k0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            if call == "ft_detect":
                f.ft_detect(plan, xs, m, k1, out=out, count=cnt, batch=b1)
            else:
                f.ft_detect_batches(plan, [xs], m, k1, out=out, count=cnt)
        m.fill_(float("nan"))
        graph.replay()
        m2 = torch.empty((b1, Hp, S), device="cuda")
        out2, cnt2 = f.ft_detect(fresh, xs, m2, k1)
        torch.cuda.synchronize()
    assert torch.equal(m[:b1], m2) and torch.equal(cnt, cnt2) and torch.equal(out, out2)


@pytest.mark.parametrize("H,W,Hp,n,k0,k1", [(150, 3888, 162, 1, 14, 5),    # 4 x 64 tiles of step 4: 2501, 16 x 16: 2673
                                            (2500, 2, 2592, 9, 23, 44)])   # 32 x 8 tiles of step 4: 81, 16 x 16: 162
def test_captured_peaks_after_detect(torch, monkeypatch, H, W, Hp, n, k0, k1):
    """ft_peaks captured after ft_detect calls alone, at lengths whose tiles in step 4
    are fewer than those of ft_peaks."""
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    g = torch.Generator(device="cuda").manual_seed(Hp)
    x = torch.randn((n, H, W), generator=g, device="cuda")
    m = torch.empty((n, Hp, W), device="cuda")
    out = torch.zeros(n * k1 * f.PEAK_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    with f.Plan(H, W, W, Hp) as plan, f.Plan(H, W, W, Hp) as fresh:
        f.ft_detect(plan, x, m, k0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            f.ft_peaks(plan, m, k1, out=out, count=cnt)
        graph.replay()
        out2, cnt2 = f.ft_peaks(fresh, m, k1)
        torch.cuda.synchronize()
    assert torch.equal(cnt, cnt2) and torch.equal(out, out2)


@pytest.mark.parametrize("H,W,Hp,S", [(150, 160, 162, 162), (480, 640, 486, 648), (70, 72, 72, 72)])
@pytest.mark.parametrize("call", ["ft_detect", "ft_peaks", "ft_abs_mse_grad"])
def test_captured_call_after_loss_backward(torch, monkeypatch, H, W, Hp, S, call):
    """The calls that need little scratch find it under capture after
    ft_abs_mse_backward alone, whichever way its columns run."""
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    n, K = 3, 5
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((n, H, W), generator=g, device="cuda")
    m = torch.randn((n, Hp, S), generator=g, device="cuda")
    t = torch.rand((n, Hp, S), generator=g, device="cuda")
    out = torch.zeros(n * K * f.PEAK_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    res = []
    with f.Plan(H, W, S, Hp) as plan, f.Plan(H, W, S, Hp) as fresh:
        f.ft_abs_mse_backward(plan, m, t, 0.5)
        torch.cuda.synchronize()

        def go(p):
            if call == "ft_abs_mse_grad":
                return f.ft_abs_mse_grad(p, m, t, 0.5)
            if call == "ft_peaks":
                f.ft_peaks(p, m, K, out=out, count=cnt)
            else:
                f.ft_detect(p, x, m, K, out=out, count=cnt)
            return out, cnt

        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            a = go(plan)
        graph.replay()
        torch.cuda.synchronize()
        res = [v.clone() for v in a]
        b = go(fresh)
        torch.cuda.synchronize()
    assert all(torch.equal(u, v) for u, v in zip(res, b))


# the preferred passes: over the whole GPU, per-tile keys, tile maxima; ft_peaks with keys
@pytest.mark.parametrize("call,H,W,n,K,more", [("ft_detect", 1024, 1024, 16, 200, True), ("ft_detect", 768, 648, 8, 200, True),
                                               ("ft_detect", 1024, 1024, 16, 8, False), ("ft_peaks", 768, 648, 8, 200, True)])
def test_failed_allocation_takes_the_pass_of_least_memory(torch, monkeypatch, call, H, W, n, K, more):
    """One failed allocation of the preferred pass leaves the one from tile maxima; a
    second one is the call's error, and the plan stays usable."""
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    g = torch.Generator(device="cuda").manual_seed(K)
    x = torch.randn((n, H, W), generator=g, device="cuda")
    m = torch.empty_like(x)

    def go(p):
        return f.ft_detect(p, x, m, K) if call == "ft_detect" else f.ft_peaks(p, m, K)

    with f.Plan(H, W, W, H) as plan, f.Plan(H, W, W, H) as fresh:
        f.ft_forward(fresh, x, m)
        want = go(fresh)
        f.ft_plan_inject_alloc_failures(plan, 2 if more else 1)
        with pytest.raises(f.FunnelError) as e:
            go(plan)
        assert e.value.status == f.FT_ERR_OOM
        f.ft_plan_inject_alloc_failures(plan, 1 if more else 0)
        a = go(plan)
        b = go(plan)                                     # allocates what it prefers
        torch.cuda.synchronize()
    for u, v, w in zip(a, b, want):
        assert torch.equal(u, w) and torch.equal(v, w)


def test_scratch_of_the_pass_over_the_whole_gpu_follows_the_map(torch, monkeypatch):
    """The candidate list of a small map holds the strict local maxima it can have (a
    quarter of its cells): 256 maps of 64 x 128 take 4 MiB, not 65536 keys each (128 MiB)."""
    monkeypatch.setenv("FT_PEAKS", "multi")
    from paper_1904_09409_gb300 import funnel as f
    n, H, W, K = 256, 128, 64, 4
    x = torch.randn((n, H, W), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    m = torch.empty_like(x)
    with f.Plan(H, W, W, H) as plan:
        f.ft_detect(plan, x, m, K)                       # modules loaded, outputs in torch's pool
    torch.cuda.synchronize()
    with f.Plan(H, W, W, H) as plan:
        assert f.ft_detect_launches(plan, n, K) == 5
        free0 = torch.cuda.mem_get_info()[0]
        f.ft_detect(plan, x, m, K)
        used = free0 - torch.cuda.mem_get_info()[0]
    assert used <= (32 << 20), used                      # 8 MiB of spectra, 4 of keys, allocation granules
