"""The callers that took the fixed-length kernels of the lengths with factors of 3
along: ft_detect_batches as a pipeline (step 1 of a batch beside the peak pass of the
one before) and the plans of a mixed batch on side streams, also in a graph.  Records,
counts and maps equal those of one ft_detect call per batch or image, bit for bit."""
import numpy as np
import pytest

from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


# lengths whose step 4 reduces its tiles through shared memory, with a ragged last band
# (486, 162) and without (1152), by whole warps (192) and without tiles (96)
@pytest.mark.parametrize("H,W,S,Hp,batch,K", [(480, 640, 648, 486, 5, 8), (150, 160, 162, 162, 9, 32),
                                              (1080, 1000, 1152, 1152, 3, 8), (190, 200, 216, 192, 7, 8),
                                              (90, 100, 108, 96, 4, 8)])
@pytest.mark.parametrize("pdl", ["1", "0"])
def test_pipelined_batches(torch, monkeypatch, H, W, S, Hp, batch, K, pdl):
    monkeypatch.setenv("FT_PDL", pdl)
    monkeypatch.setenv("FT_PEAKS", "sparse")             # the pass the pipeline runs
    from paper_1904_09409_gb300 import funnel as f
    g = torch.Generator(device="cuda").manual_seed(H + K)
    xs = [torch.randn((batch, H, W), generator=g, device="cuda") for _ in range(5)]
    with f.Plan(H, W, S, Hp) as plan:
        m = torch.empty((batch, Hp, S), device="cuda")
        want = [f.ft_detect(plan, x, m, K) for x in xs]
        last = m.clone()
        m.fill_(float("nan"))
        out, cnt = f.ft_detect_batches(plan, xs, m, K)
        torch.cuda.synchronize()
    assert torch.equal(out, torch.cat([o for o, _ in want])) and torch.equal(cnt, torch.cat([c for _, c in want]))
    assert torch.equal(m, last)


@pytest.mark.parametrize("graph", [False, True])
def test_mixed_batch_with_wide_lengths(torch, monkeypatch, graph):
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    shapes = [(486, 648), (128, 192), (162, 216), (486, 648), (96, 72), (1152, 864), (256, 256)]
    K = 40
    rng = np.random.default_rng(4)
    imgs = [rng.standard_normal(s).astype(np.float32) for s in shapes]
    rec = K * f.PEAK_DTYPE.itemsize
    stream = torch.cuda.Stream()
    with f.Batch(shapes) as b, torch.cuda.stream(stream):
        x = torch.from_numpy(b.pack(imgs)).cuda()
        m = torch.zeros(b.map_total, device="cuda")
        out = torch.empty(b.n * rec, dtype=torch.uint8, device="cuda")
        cnt = torch.empty(b.n, dtype=torch.int32, device="cuda")
        for _ in range(2):
            b.run(x, m, K, out=out, count=cnt, stream=stream, graph=graph)
        stream.synchronize()
        maps = b.unpack_maps(m.cpu().numpy())
        for j, i in enumerate(b.order):
            H, W = shapes[i]
            with f.Plan(H, W, W, H) as plan:
                ref = torch.empty((1, H, W), device="cuda")
                o, c = f.ft_detect(plan, torch.from_numpy(imgs[i][None]).cuda(), ref, K)
                torch.cuda.synchronize()
            assert np.array_equal(maps[i], ref[0].cpu().numpy()), (H, W)
            assert int(c[0]) == int(cnt[j]) and torch.equal(o, out[j * rec:(j + 1) * rec]), (H, W)
