"""The peak pass over the whole GPU (FT_PEAKS=multi) where its list of candidates
overflows: more than 65536 strict local maxima at or above the bound, which needs
fewer strict tile maxima than top_k (the bound is then the threshold)."""
import numpy as np
import pytest

import oracle
from tests import _gpu

pytestmark = pytest.mark.gpu

LIST = 65536           # keys the pass keeps per image


@pytest.fixture(scope="module")
def torch():
    return _gpu.torch_cuda()


def _strict_maxima(a):
    """Cells larger than their 8 neighbours (wrapped); ties count as none."""
    ok = np.ones(a.shape, bool)
    for dt in (-1, 0, 1):
        for ds in (-1, 0, 1):
            if (dt, ds) != (0, 0):
                ok &= a > np.roll(a, (dt, ds), (0, 1))
    return int(ok.sum())


def test_list_overflow_falls_back_to_the_one_block_pass(torch, monkeypatch):
    from paper_1904_09409_gb300 import funnel as f
    N, K = 1024, 1024
    g = torch.Generator(device="cuda").manual_seed(11)
    x = torch.randn((2, N, N), generator=g, device="cuda")
    x[1] *= 0.0                                          # the other image of the call does not overflow
    x[1, 100:200, 300:420] = 1.0
    res = {}
    for mode in ("multi", "sparse"):
        monkeypatch.setenv("FT_PEAKS", mode)
        with f.Plan(N, N, N, N) as plan:
            assert f.ft_detect_launches(plan, 2, K) == (5 if mode == "multi" else 4)
            for _ in range(2):                           # the counters are zero again after an overflow
                m = torch.full((2, N, N), float("nan"), device="cuda")
                out, cnt = f.ft_detect(plan, x, m, K)
            torch.cuda.synchronize()
            res[mode] = m.cpu().numpy(), out.cpu().numpy(), cnt.cpu().numpy(), f.peaks_to_numpy(out, cnt, K)
    a = np.abs(res["multi"][0][0]).astype(np.float64)
    assert _strict_maxima(a) > LIST                      # every one is a candidate ...
    assert _strict_maxima(a.reshape(64, 16, 64, 16).max((1, 3))) < K     # ... as the bound is the threshold
    for u, v in zip(res["multi"][:3], res["sparse"][:3]):
        assert np.array_equal(u, v)
    got = [(int(p["t"]), int(p["s"]), float(p["value"])) for p in res["multi"][3][0]]
    assert got == oracle.peaks_ref(a, K)
