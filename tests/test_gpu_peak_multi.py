"""The peak pass over the whole GPU (FT_PEAKS=multi): records and counts equal the
list procedure on the forward's own map, byte for byte equal to the one-block
pass, for every tile shape, ragged columns, the inverse space, ties, thresholds,
K above the number of peaks, and maps whose candidates overflow the pass's list.
The input of the forward is chosen so that the map is known: the pass only sees
maps, and any image gives one.
"""
import numpy as np
import pytest

import oracle
from tests import _gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


def _detect(torch, monkeypatch, mode, H, W, S, Hp, K, thr, x, space="regular", calls=1):
    from paper_1904_09409_gb300 import funnel as f
    monkeypatch.setenv("FT_PEAKS", mode)
    with f.Plan(H, W, S, Hp, "linear", space) as plan:
        m = torch.full((x.shape[0], Hp, S), float("nan"), dtype=torch.float32, device="cuda")
        for _ in range(calls):                          # the pass's counters are zero again after every call
            out, cnt = f.ft_detect(plan, x, m, K, thr)
        torch.cuda.synchronize()
        n_launch = f.ft_detect_launches(plan, x.shape[0], K)
    return m.cpu().numpy(), out.cpu().numpy(), cnt.cpu().numpy(), f.peaks_to_numpy(out, cnt, K), n_launch


CASES = [
    (256, 256, 256, 256, 3, float("-inf")),       # 8 x 32 tiles, K below one warp
    (1024, 1024, 1024, 1024, 32, float("-inf")),  # 16 x 16 tiles
    (200, 200, 216, 256, 40, float("-inf")),      # ragged against 32-column tiles
    (100, 96, 96, 192, 17, float("-inf")),        # H' = 192
    (128, 200, 216, 4096, 100, float("-inf")),    # 32 x 8 tiles
    (64, 16, 16, 8192, 5, float("-inf")),         # 64 x 4 tiles, 4 tile columns
    (64, 4, 4, 8192, 5, float("-inf")),           # one tile column: a tile is its own neighbour
    (480, 640, 648, 486, 8, float("-inf")),       # tiles reduced through shared memory, a ragged last band
    (150, 96, 108, 162, 5, float("-inf")),        # 4 x 64 tiles, wider than half the map
    (1000, 200, 216, 1152, 20, float("-inf")),    # 16 x 16 tiles, S no multiple of 16
    (300, 60, 64, 3888, 33, float("-inf")),       # 32 x 8 tiles, 36 samples per thread
    (256, 256, 256, 256, 1024, float("-inf")),    # K above the number of tiles
    (256, 256, 256, 256, 64, 30.0),               # a threshold few peaks pass
    (256, 256, 256, 256, 64, 1e9),                # a threshold none passes
]


@pytest.mark.parametrize("H,W,S,Hp,K,thr", CASES)
def test_multi_matches_oracle_and_sparse(torch, monkeypatch, H, W, S, Hp, K, thr):
    rng = np.random.default_rng(H + W + S + K)
    x = torch.from_numpy(rng.standard_normal((3, H, W)).astype(np.float32)).cuda()
    m, raw, cnt, res, n_launch = _detect(torch, monkeypatch, "multi", H, W, S, Hp, K, thr, x, calls=3)
    assert n_launch == 5
    m1, raw1, cnt1, _, _ = _detect(torch, monkeypatch, "sparse", H, W, S, Hp, K, thr, x)
    assert np.array_equal(m, m1) and np.array_equal(cnt, cnt1) and np.array_equal(raw, raw1)
    for i in range(3):
        got = [(int(p["t"]), int(p["s"]), float(p["value"])) for p in res[i]]
        assert got == oracle.peaks_ref(np.abs(m[i]).astype(np.float64), K, thr), i


def test_multi_inverse_space_and_zero_image(torch, monkeypatch):
    x = torch.zeros((2, 192, 256), dtype=torch.float32, device="cuda")
    x[1] = torch.randn((192, 256), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    m, raw, cnt, res, n_launch = _detect(torch, monkeypatch, "multi", 192, 256, 192, 256, 12, float("-inf"), x,
                                         space="inverse")
    assert n_launch == 6
    assert [(int(p["t"]), int(p["s"])) for p in res[0]] == [(0, 0)]     # every cell ties
    got = [(int(p["t"]), int(p["s"]), float(p["value"])) for p in res[1]]
    assert got == oracle.peaks_ref(np.abs(m[1]).astype(np.float64), 12)


def test_multi_list_overflow(torch, monkeypatch):
    """A single bright pixel in every other 2 x 2 block of a large map of equal
    tile maxima leaves no strict tile maximum, so every tile is a candidate and
    the list overflows: a constant tone per column pair gives such a map."""
    H = W = 1024
    x = torch.zeros((1, H, W), dtype=torch.float32, device="cuda")
    x[0, ::2, W // 2] = 1.0                              # a comb along y: a map periodic in t
    a = _detect(torch, monkeypatch, "multi", H, W, W, H, 1024, float("-inf"), x, calls=2)
    b = _detect(torch, monkeypatch, "sparse", H, W, W, H, 1024, float("-inf"), x)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


def test_capture_without_the_pass_buffers(torch, monkeypatch):
    """The pass depends on the batch and K.  A call captured into a graph after
    calls that took another pass cannot allocate what its own pass would want: it
    takes one whose buffers are there, with the same records."""
    monkeypatch.delenv("FT_PEAKS", raising=False)
    from paper_1904_09409_gb300 import funnel as f
    n, N, K = 16, 1024, 200
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((n, N, N), generator=g, device="cuda")
    with f.Plan(N, N, N, N) as plan, f.Plan(N, N, N, N) as fresh:
        assert f.ft_detect_launches(plan, n, 8) == 4 and f.ft_detect_launches(plan, n, K) == 5
        m = torch.empty_like(x)
        out = torch.zeros(n * K * f.PEAK_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
        f.ft_detect(plan, x, m, 8)                       # one block per image: no buffers of the other pass
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            f.ft_detect(plan, x, m, K, out=out, count=cnt)
        graph.replay()
        m2 = torch.empty_like(x)
        out2, cnt2 = f.ft_detect(fresh, x, m2, K)
        torch.cuda.synchronize()
    assert torch.equal(m, m2) and torch.equal(cnt, cnt2) and torch.equal(out, out2)
