"""GPU parity of the vector forms of the frame sums and the binning against
the oracle, at the sizes and alignments at which they are chosen or not: rows
about a multiple of 8, frames about a multiple of 4 pixels, cubes that start
1 to 4 values past a 16-byte boundary."""
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


@pytest.mark.parametrize("lead", [0, 1, 2, 4])
@pytest.mark.parametrize("N,H,W", [(7, 9, 8), (3, 2, 264), (4, 11, 520), (2, 5, 1032), (5, 3, 12),
                                   (6, 1, 16), (2, 8, 1028), (1, 2, 7)])
def test_sums_and_bins_bitexact(st, N, H, W, lead):
    rng = np.random.default_rng(W + lead)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    fr.reshape(-1)[::7] = np.nan
    buf = torch.zeros(lead + fr.size, device="cuda")
    x = buf[lead:].view(N, H, W)
    x.copy_(torch.from_numpy(fr))
    n = min(N, 3)
    t = np.arange(N, dtype=np.float64)
    ref, rt = front.sum_frames(fr, t, n)
    out, tout = st.sum_frames(x, t, n)
    assert np.array_equal(out.cpu().numpy(), ref, equal_nan=True)
    assert np.array_equal(tout, rt)
    ref = front.bin2x2(fr)
    out = st.bin2x2(x)
    assert tuple(out.shape) == ref.shape
    assert np.array_equal(out.cpu().numpy(), ref, equal_nan=True)


@pytest.mark.parametrize("lead", [0, 1, 4])
@pytest.mark.parametrize("N,H,W", [(1, 1, 4), (2, 3, 44), (3, 7, 9), (5, 1, 127), (8, 2, 66),
                                   (33, 4, 33), (50, 3, 172), (63, 5, 51), (64, 2, 130),
                                   (65, 2, 66), (97, 1, 40), (200, 3, 31), (600, 1, 68)])
def test_medians_bitexact(st, N, H, W, lead):
    # masked and infinite samples, whole columns of them, zeros of both signs
    rng = np.random.default_rng(100 * N + W)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    hide = rng.random(fr.shape) < rng.random((H, W)) - 0.4
    fr[hide] = rng.choice(np.array([np.nan, np.inf, -np.inf], np.float32), int(hide.sum()))
    fr[:, 0, 0], fr[:, 0, 1] = np.nan, np.float32(-0.0)
    fr[N // 2:, H - 1, W - 1] = 0.0
    buf = torch.zeros(lead + fr.size, device="cuda")
    x = buf[lead:].view(N, H, W)
    x.copy_(torch.from_numpy(fr))
    with np.errstate(invalid="ignore"):
        ref, rmed = front.median_subtract(fr)
    out, med = st.median_subtract(x, with_median=True)
    assert np.array_equal(med.cpu().numpy(), rmed, equal_nan=True)
    assert np.array_equal(out.cpu().numpy(), ref, equal_nan=True)
