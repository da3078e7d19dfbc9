"""GPU parity of the run kernel (k_stack_runs.cu): it sums frames with equal
relative shifts first and keeps points down to a margin below the threshold,
so its candidate lists are compared, bit for bit, with the direct-gather
kernel's (frame order, no window) on the same frames: ragged sizes, velocity
counts about its tiles of 4, 8 and 32, few and many frames, both directions
of motion, every storage type, and the fields that it must leave to the other
kernels."""
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


def field(seed, W=96, H=45, N=19, nvx=13, nvy=11, step=0.4, tau=2.5, ref=None, v0=None):
    """step: largest shift between adjacent velocities, px; a step of 0: one
    velocity grid point repeated."""
    rng = np.random.default_rng(seed)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    t = np.sort(rng.uniform(0.0, 2.0, N))
    t_ref = float(t[N // 3 if ref is None else ref])
    dv = step / max(float(np.abs(t - t_ref).max()), 1e-9)
    vx0 = -dv * (nvx // 2) - 0.1 if v0 is None else v0
    f = synth.field_params(W, H, N, t_ref, vx0, dv, nvx, -dv * (nvy // 2) + 0.05, dv, nvy, tau=tau)
    synth.render_movers(fr, t, t_ref, [[W * 0.4, H * 0.5, 3 * dv, -2 * dv, 3.0]])
    return fr, t, f


RUNS = {"f32": 9, "f16": 7, "bf16": 7}   # plan option `tile` of the run kernel


def lists(st, fr, t, f, tiles, **kw):
    out = []
    x = torch.from_numpy(fr).cuda()
    for tile in tiles:
        with st.Plan(f, tile=tile, **kw) as p:
            out.append((p.candidates(x, t), p.stack_variant_name(0)))
    return out


def same(a, b):
    for k in a.dtype.names:
        assert np.array_equal(a[k], b[k]), k
    assert len(a) > 0


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [
    dict(), dict(W=128, H=64, N=40, nvx=16, nvy=16), dict(W=40, H=17, N=9, nvx=5, nvy=3),
    dict(W=200, H=33, N=64, nvx=33, nvy=9, step=0.1), dict(W=8, H=5, N=8, nvx=70, nvy=17, tau=1.5),
    dict(W=64, H=16, N=17, nvx=32, nvy=64), dict(W=72, H=100, N=33, nvx=65, nvy=16, step=0.5),
    dict(W=64, H=40, N=48, nvx=36, nvy=18, ref=47), dict(W=64, H=40, N=31, nvx=67, nvy=5, ref=0),
    dict(W=320, H=40, N=50, nvx=20, nvy=20, v0=30.0, tau=3.0),   # samples far outside the frame
    dict(W=64, H=40, N=16, nvx=1, nvy=1, tau=1.0), dict(W=64, H=24, N=300, nvx=18, nvy=18)])
def test_runs_equal_direct_gather(st, shape, storage):
    fr, t, f = field(5, **shape)
    kw = dict(normalize=True, cr_clip=10.0, storage=storage)
    (a, na), (b, nb), (c, nc) = lists(st, fr, t, f, (RUNS[storage], 1, 0), **kw)
    assert "runs" in na and nb == "direct-gather"
    if f["n_frames"] < 32:   # the default's rule
        assert "runs" not in nc
    same(a, b)
    same(c, b)


@pytest.mark.parametrize("storage,normalize,scale", [("f32", False, 1.0), ("f32", True, 1.0),
                                                     ("bf16", False, 1.0), ("f32", False, 3e4)])
def test_runs_margin_found_on_the_device(st, storage, normalize, scale):
    # no clip: the largest value decides; values far above the noise that the
    # threshold is for leave the field to the other kernels
    fr, t, f = field(6, nvx=24, nvy=20, N=40)
    fr[3, 10, 20] = 30.0 * scale
    if normalize:   # (stored as 0)
        fr[7, 11, 22] = np.nan
    (a, na), (b, _) = lists(st, fr, t, f, (RUNS[storage], 1), normalize=normalize,
                            storage=storage)
    assert ("runs" in na) == (scale == 1.0)
    same(a, b)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("W", [96, 93])
def test_raw_nan_pixels_reach_only_their_own_stacks(st, storage, W):
    # a NaN beside the mover's path, in an early and in a late frame: the
    # stacks that never read it keep their values
    for i in (0, 19, 39):
        fr, t, f = field(6, W=W, nvx=24, nvy=20, N=40)
        p = [f[k] for k in ("vx0", "dvx", "vy0", "dvy", "t_ref")]
        x = round(W * 0.4 + 3 * p[1] * (t[i] - p[4]))
        y = round(f["height"] * 0.5 - 2 * p[3] * (t[i] - p[4]))
        fr[i, y + 1, x] = fr[i, y - 1, x] = fr[i, y, x + 2] = np.nan
        (a, na), (b, _) = lists(st, fr, t, f, (RUNS[storage], 1), normalize=False, storage=storage)
        assert "runs" not in na
        same(a, b)


def test_runs_infinite_pixels(st):
    fr, t, f = field(7, nvx=24, nvy=20, N=33)
    fr[3, 10, 20], fr[4, 12, 21], fr[9, 30, 50] = np.inf, -np.inf, np.inf
    (a, na), (b, _) = lists(st, fr, t, f, (9, 1))
    assert "runs" not in na
    same(a, b)


@pytest.mark.parametrize("shape", [dict(step=0.95, nvx=40, N=40), dict(step=2.0, N=40), dict(N=7)])
def test_fields_beyond_the_run_kernel(st, shape):
    fr, t, f = field(8, **shape)
    (a, na), (b, _) = lists(st, fr, t, f, (9, 1), normalize=True, cr_clip=10.0)
    assert "runs" not in na
    same(a, b)


def test_runs_pending_list_that_holds_the_points_but_not_the_margin(st):
    # the margin's points do not fit: the search falls back and succeeds
    fr, t, f = field(9, N=60, nvx=24, nvy=20, W=128, H=64, tau=1.0)
    x = torch.from_numpy(fr).cuda()
    kw = dict(normalize=True, cr_clip=10.0)
    (b, _), = lists(st, fr, t, f, (2,), **kw)
    lo, hi = len(b), 1 << 20
    while lo < hi:   # the smallest capacity of the frame-order kernel
        mid = (lo + hi) // 2
        with st.Plan(f, tile=2, pending_capacity=mid, **kw) as p:
            try:
                p.search(x, t)
                hi = mid
            except st.StError:
                lo = mid + 1
    for tile in (0, 9):
        with st.Plan(f, tile=tile, pending_capacity=lo, **kw) as p:
            a = p.candidates(x, t)
        same(a, b)


def test_runs_several_fields_and_graph(st):
    made = [field(20 + k, W=64 + 32 * k, H=40 + 7 * k, N=24 + 9 * k, nvx=9 + 13 * k, nvy=7 + 3 * k)
            for k in range(4)]
    fr = [torch.from_numpy(m[0]).cuda() for m in made]
    t, f = [m[1] for m in made], [m[2] for m in made]
    got = []
    for tile, graph in ((1, False), (9, False), (9, True), (0, True)):
        with st.Plan(f, tile=tile, use_graph=graph, normalize=True) as p:
            got.append(p.candidates(fr, t))
            again = p.candidates(fr, t)
        same(got[-1], again)
    for g in got[1:]:
        same(got[0], g)
