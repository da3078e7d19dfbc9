"""GPU parity of the median over more than 64 frames (k_median_long, bisection
on integer keys) against the oracle: every number of keys a thread can hold
and the counts about them, masked samples of either parity, ties, signed
zeros, infinities, the ends of the FP32 range, ragged pixel counts, in place."""
import numpy as np
import pytest

from oracle import front

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def st():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2303_07293_gb300 as m
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return m


@pytest.mark.parametrize("kind", ["noise", "ties", "wide", "masked"])
@pytest.mark.parametrize("N", [65, 95, 96, 97, 128, 129, 160, 161, 192, 193, 224, 225, 256, 257,
                               320, 321, 384, 385, 512, 513, 640, 641, 767, 768])
def test_median_of_long_groups_bitexact(st, N, kind):
    H, W = (3, 37) if N % 2 else (1, 64)
    rng = np.random.default_rng(N)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    if kind == "ties":
        fr = np.round(fr).astype(np.float32)   # -0, +0 and a few values
    elif kind == "wide":
        fr = (fr * 10.0 ** rng.uniform(-38, 38, fr.shape)).astype(np.float32)
        fr[rng.random(fr.shape) < 0.05] = np.inf
        fr[rng.random(fr.shape) < 0.05] = -np.inf
        fr[0, 0, :8] = np.finfo(np.float32).max
        fr[1, 0, :8] = -np.finfo(np.float32).max
    elif kind == "masked":
        fr[rng.random(fr.shape) < rng.random((H, W))] = np.nan
        fr[:, 0, 0] = np.nan
        fr[1:, 0, 1] = np.nan
        fr[2:, 0, 2] = np.nan
    with np.errstate(over="ignore", invalid="ignore"):
        ref, rmed = front.median_subtract(fr)
    d = torch.from_numpy(fr).cuda()
    out, med = st.median_subtract(d, with_median=True)
    assert np.array_equal(med.cpu().numpy(), rmed, equal_nan=True)
    assert np.array_equal(out.cpu().numpy(), ref, equal_nan=True)
    st.median_subtract(d, out=d)
    assert np.array_equal(d.cpu().numpy(), ref, equal_nan=True)
