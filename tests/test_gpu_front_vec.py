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
