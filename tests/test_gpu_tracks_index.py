"""GPU parity of the track linking's ways to a detection's neighbours: few
detections of a large grid (no table of velocities, binary search), many at
one velocity (search within its part of the list), and few each (one by one),
against the oracle on drawn lists."""
import numpy as np
import pytest

import synth
from oracle import tracks as otracks

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def st():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2303_07293_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return m


@pytest.mark.parametrize("nvx,nvy,n,W,H", [
    (400, 399, 300, 64, 48), (3, 3, 2000, 60, 50), (1, 1, 900, 64, 48), (40, 37, 3000, 40, 24),
    (7, 5, 1, 32, 32), (20, 20, 257, 16, 16), (2, 90, 24 * 180, 90, 70)])
@pytest.mark.parametrize("r_xy,r_v", [(2, 1), (0, 0), (1, 3)])
def test_drawn_lists_equal_oracle(st, nvx, nvy, n, W, H, r_xy, r_v):
    rng = np.random.default_rng(nvx * 1000 + n)
    fields = [synth.field_params(W, H, 9, 4.0, -0.1, 0.05, nvx, 0.2, 0.03, nvy) for _ in range(2)]
    # half of the list about a few places, half anywhere; distinct, sorted
    f = rng.integers(0, 2, n)
    k = np.where(rng.random(n) < 0.5, rng.integers(0, nvx * nvy, n),
                 (rng.integers(0, 4, n) * 7919 + rng.integers(-1, 2, n) * nvx +
                  rng.integers(-1, 2, n)) % (nvx * nvy))
    y = np.where(rng.random(n) < 0.5, rng.integers(0, H, n), rng.integers(3, 9, n))
    x = np.where(rng.random(n) < 0.5, rng.integers(0, W, n), rng.integers(3, 12, n))
    rows = np.unique(np.stack([f, k, y, x], 1), axis=0)
    cand = np.zeros(len(rows), st.CAND_DTYPE)
    cand["field"], cand["k"], cand["y"], cand["x"] = rows.T
    cand["snr"] = np.round(rng.normal(6, 1, len(rows)), 1)   # ties
    cand["stack"] = cand["snr"] * 3
    cand["n_cov"] = 9
    d = torch.from_numpy(cand.view(np.int32).reshape(-1, 7).copy()).cuda()
    with st.Plan(fields) as p:
        fr = [torch.zeros((9, H, W), device="cuda") for _ in fields]
        p.search(fr, [np.arange(9.0)] * 2)
        got = p.link_tracks(d, r_xy=r_xy, r_v=r_v)
    ref = otracks.link_tracks(cand, [(g["vx0"], g["dvx"], g["nvx"], g["vy0"], g["dvy"], g["nvy"])
                                     for g in fields], r_xy=r_xy, r_v=r_v)
    assert len(got) == len(ref)
    for g, r in zip(got, ref):
        for key in ("x", "y", "k", "field", "n_cov", "members"):
            assert int(g[key]) == r[key], (key, g, r)
        assert g["snr"] == np.float32(r["snr"])
