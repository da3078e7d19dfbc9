"""GPU parity of the sky statistics and the normalisation (k_prep.cu): the
pivoted integer sums against the oracle's clipped FP64 statistics, and the
stored values against the FP64 formula on the returned statistics, bit for
bit, for levels, ranges and sizes at which the pivot, the range and the vector
loads change."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def st():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2303_07293_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return m


# level and scale of the frames, and what is put into them
@pytest.mark.parametrize("level,scale,extra", [
    (0.0, 1.0, None), (1e-3, 1.0, None), (250.0, 10.0, None), (-7.0, 1.0, None),
    (6.2e4, 3.0, None), (1e7, 2.0, None), (0.0, 1e-33, None), (0.0, 1e31, None),
    (5.0, 1e-4, None), (300.0, 12.0, "outliers"), (300.0, 12.0, "stars"), (0.0, 1.0, "nan"),
    (0.0, 1.0, "zeros")])
@pytest.mark.parametrize("W,H,N,lead", [(64, 32, 3, 0), (37, 53, 5, 1), (7, 3, 2, 3),
                                        (301, 257, 2, 2)])
def test_sky_statistics_and_stored_values(st, level, scale, extra, W, H, N, lead):
    rng = np.random.default_rng(W + N)
    raw = (level + scale * rng.standard_normal((N, H, W))).astype(np.float32)
    flat = raw.reshape(N, -1)
    if extra == "outliers":
        flat[:, 5], flat[:, 11], flat[:, 13] = 3e8, -1e9, np.inf
    elif extra == "stars":   # a tenth of the pixels far above the sky
        flat[rng.random(flat.shape) < 0.1] += 4000.0
    elif extra == "nan":
        flat[rng.random(flat.shape) < 0.3] = np.nan
    elif extra == "zeros":
        flat[:, ::3] = 0.0
    # frames that start `lead` values past a 16-byte boundary
    buf = torch.zeros(lead + raw.size, device="cuda")
    frames = buf[lead:].view(N, H, W)
    frames.copy_(torch.from_numpy(raw))
    f = synth.field_params(W, H, N, 0.0, 0.0, 1.0, 1, 0.0, 1.0, 1)
    with st.Plan(f, normalize=True) as p:
        cube, mu, sd = p.normalize(0, frames)
    _, omu, osd = oracle.normalize(raw)
    # the bar of the other normalisation tests (a mean near zero: of sigma)
    assert np.all(np.abs(mu - omu) <= 1e-12 * np.maximum(np.abs(omu), osd))
    assert np.all(np.abs(sd - osd) <= 1e-12 * osd)
    with np.errstate(over="ignore", invalid="ignore"):
        want = ((raw.astype(np.float64) - mu[:, None, None]) * (1.0 / sd)[:, None, None])
        want = np.where(np.isfinite(raw), want, 0.0).astype(np.float32)
    assert np.array_equal(cube.cpu().numpy(), want)
