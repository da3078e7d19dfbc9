"""GPU parity of the normalisation at the ends of the FP32 range: where a
frame's mean or 1/sigma has no exact parts in FP32 the stored values are still
those of the FP64 formula on the returned statistics."""
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


def normalized(st, raw, **kw):
    N, H, W = raw.shape
    f = synth.field_params(W, H, N, 0.0, 0.0, 1.0, 1, 0.0, 1.0, 1)
    with st.Plan(f, normalize=True, **kw) as p:
        cube, mu, sd = p.normalize(0, torch.from_numpy(raw).cuda())
    return cube.cpu().numpy(), mu, sd


def mirrored(v):
    """v and -v, so that the frame's mean is 0."""
    v = v.astype(np.float32).astype(np.float64)
    return np.concatenate([v, -v], 1)


def frames(kind, H, W, N=4):
    rng = np.random.default_rng(len(kind))
    n = H * W
    half = rng.standard_normal((N, n // 4))
    if kind == "beyond":       # 1/sigma beyond FP32, pixels equal to the mean
        x = mirrored(1e-40 * half)
    elif kind == "between":    # a mean between two FP32 values, next to pixels of 0
        x = mirrored(1e-38 * half)
        x = np.concatenate([x, np.full((N, int(0.3 * n)), 2.0 ** -149)], 1)
    elif kind == "wide":       # pixels of ordinary size beside a tiny deviation
        x = mirrored(3e-37 * half)
        x[:, 7::97] = 10.0 ** rng.uniform(-15, -3, x[:, 7::97].shape)
    elif kind == "huge":       # half of the pixels near the mean, a deviation of 1e36
        x = np.concatenate([mirrored(1e36 * (1.0 + 0.01 * half)),
                            mirrored(1e30 * rng.uniform(-1.0, 1.0, half.shape))], 1)
    else:                      # an ordinary sky
        return (300.0 + 12.0 * rng.standard_normal((N, H, W))).astype(np.float32)
    out = np.zeros((N, n))
    out[:, :x.shape[1]] = x
    return rng.permuted(out, axis=1).astype(np.float32).reshape(N, H, W)


@pytest.mark.parametrize("kind", ["beyond", "between", "wide", "huge", "sky"])
@pytest.mark.parametrize("W", [64, 61])
def test_stored_values_are_the_fp64_formulas(st, kind, W):
    raw = frames(kind, 96, W)
    cube, mu, sd = normalized(st, raw)
    assert np.all(sd > 0.0)
    with np.errstate(over="ignore"):
        want = (raw.astype(np.float64) - mu[:, None, None]) * (1.0 / sd)[:, None, None]
        want = want.astype(np.float32)
    assert np.array_equal(cube, want)
