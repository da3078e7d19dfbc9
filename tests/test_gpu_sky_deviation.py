"""GPU parity of the sky's mean and deviation with an extended-precision
reference: they keep the accuracy of sums about the mean whatever the level
of the frame, near zero and at the ends of the FP32 range."""
import numpy as np
import pytest

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


def normalized(st, raw):
    N, H, W = raw.shape
    f = synth.field_params(W, H, N, 0.0, 0.0, 1.0, 1, 0.0, 1.0, 1)
    with st.Plan(f, normalize=True) as p:
        cube, mu, sd = p.normalize(0, torch.from_numpy(raw).cuda())
    return cube, mu, sd


def statistics(frame):
    """Clipped mean and deviation (3 sigma, at most 5 statistics) in extended
    precision."""
    x = frame.astype(np.longdouble).ravel()
    keep = np.ones(x.size, bool)
    for it in range(5):
        mu = x[keep].mean()
        sd = np.sqrt(((x[keep] - mu) ** 2).mean())
        now = np.abs(x - mu) <= 3.0 * sd
        if it == 4 or np.array_equal(now, keep):
            return mu, sd
        keep = now


@pytest.mark.parametrize("level", [0.0, 1.0, 3.0, 5.0, 9.0, 14.0, 40.0, -6.0])
def test_deviation_at_any_level(st, level):
    # a variance after two roundings and its root: 2^-53 + 2^-53 relative, and
    # the squares' parts below the sums' grid, thousands of times less
    assert np.finfo(np.longdouble).eps <= 2.0 ** -63
    rng = np.random.default_rng(int(10 * abs(level)))
    raw = (7.0 * (level + rng.standard_normal((48, 128, 96)))).astype(np.float32)
    _, mu, sd = normalized(st, raw)
    ref = [statistics(f) for f in raw]
    err = max(float(abs(np.longdouble(s) - r[1]) / r[1]) for s, r in zip(sd, ref))
    assert err <= 1.01 * 2.0 ** -52
    assert max(float(abs(np.longdouble(m) - r[0]) / r[1]) for m, r in zip(mu, ref)) <= \
        1.01 * 2.0 ** -52 * (1.0 + abs(level))


@pytest.mark.parametrize("level,scale", [(1e36, 1e31), (1e-28, 1e-32), (-3e-30, 1e-32)])
def test_deviation_far_below_the_level_at_the_ends_of_the_range(st, level, scale):
    # sums in FP64, 10^4 to 10^5 deviations from zero: the bar of the other
    # normalisation tests
    rng = np.random.default_rng(5)
    raw = (level + scale * rng.standard_normal((6, 64, 96))).astype(np.float32)
    _, mu, sd = normalized(st, raw)
    for i in range(len(raw)):
        m, s = statistics(raw[i])
        assert abs(mu[i] - m) <= 1e-12 * abs(m)
        assert abs(sd[i] - s) <= 1e-12 * s
