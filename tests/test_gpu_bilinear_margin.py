"""Bilinear searches of frames whose values are far above the threshold: the
register-window kernel forms a sample in factored form, the direct gather and
the resolver as four weighted taps, so the kernel keeps points down to a
margin that bounds the difference for the field's largest value.  Lists equal
the direct gather's whatever the values; where the margin would be too wide,
or a value is infinite, the field is searched by the direct gather."""
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


def field(W, H=48, N=32, nv=13, tau=2.0, seed=4, high=0.0):
    """high: the first half of the frames lies that far above the second, so
    that partial sums are large where the whole is noise."""
    rng = np.random.default_rng(seed)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    fr[:N // 2] += np.float32(high)
    fr[N // 2:] -= np.float32(high)
    t = np.sort(rng.uniform(0.0, 2.0, N))
    f = synth.field_params(W, H, N, float(t[N // 3]), -0.2 * (nv // 2) - 0.03, 0.2, nv,
                           -0.2 * (nv // 2) + 0.05, 0.2, nv, tau=tau)
    return fr, t, f


def lists(st, fr, t, f, **kw):
    x = [torch.from_numpy(v).cuda() for v in fr] if isinstance(fr, list) else \
        torch.from_numpy(fr).cuda()
    out = []
    for tile in (1, 0):
        with st.Plan(f, mode="bilinear", tile=tile, **kw) as p:
            out.append(p.candidates(x, t))
            variants = [p.last_stack_variant(k) for k in range(len(p.fields))]
            again = p.candidates(x, t)
            assert again.tobytes() == out[-1].tobytes()
    assert len(out[0]) > 0
    assert out[0].tobytes() == out[1].tobytes()
    return variants


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("W", [96, 93])
@pytest.mark.parametrize("high,kept", [(0.0, True), (3e2, True), (5e3, True), (1e6, False)])
def test_values_far_above_the_threshold(st, W, high, kept, storage):
    fr, t, f = field(W, high=high)
    assert lists(st, fr, t, f, storage=storage) == [1 if kept else 0]


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("W", [96, 93])
def test_infinite_pixels(st, W, graph):
    fr, t, f = field(W)
    fr[3, 10, 20:22] = np.inf
    fr[9, 30, 50], fr[20, 11, 40] = -np.inf, np.inf
    assert lists(st, fr, t, f, use_graph=graph) == [0]


@pytest.mark.parametrize("W", [96, 93])
def test_masked_pixels_stay_with_the_window_kernel(st, W):
    # NaN reaches the same stacks either way
    fr, t, f = field(W)
    fr[np.random.default_rng(1).random(fr.shape) < 0.002] = np.nan
    assert lists(st, fr, t, f) == [1]


def test_half_precision_values_beyond_its_range(st):
    fr, t, f = field(96, N=8, tau=1.0)
    fr[3, 10, 20:22] = 7e4   # stored as infinities
    assert lists(st, fr, t, f, storage="f16") == [0]


@pytest.mark.parametrize("graph", [False, True])
def test_one_field_of_several(st, graph):
    # the field with an infinite pixel alone goes to the direct gather
    made = [field(96 - 4 * k, H=40 + k, seed=k, nv=9) for k in range(3)]
    made[1][0][5, 6, 7] = np.inf
    fr, t, f = [m[0] for m in made], [m[1] for m in made], [m[2] for m in made]
    assert lists(st, fr, t, f, use_graph=graph) == [1, 0, 1]


@pytest.mark.parametrize("clip", [0.0, 10.0, 1e5])
def test_normalised_frames(st, clip):
    fr, t, f = field(96, nv=16, tau=1.5)
    fr = 250.0 + 10.0 * fr
    fr[7, 11, 22] = 1e5
    assert lists(st, fr.astype(np.float32), t, f, normalize=True, cr_clip=clip) == [1]


def test_list_that_holds_the_points_but_not_the_margin(st):
    # the exact filter's points fit: the search succeeds as it does there
    fr, t, f = field(96, high=5e3)
    x = torch.from_numpy(fr).cuda()
    lo, hi = 1, 1 << 20
    while lo < hi:
        mid = (lo + hi) // 2
        with st.Plan(f, mode="bilinear", tile=1, pending_capacity=mid) as p:
            try:
                p.search(x, t)
                hi = mid
            except st.StError:
                lo = mid + 1
    with st.Plan(f, mode="bilinear", tile=1) as p:
        want = p.candidates(x, t)
    with st.Plan(f, mode="bilinear", pending_capacity=lo) as p:
        for _ in range(2):
            assert p.candidates(x, t).tobytes() == want.tobytes()


def test_autotuned_plan_keeps_its_variant_in_a_second_pass(st, tmp_path):
    # the field that the variant was tuned on goes to the direct gather; the
    # other one is not tuned for it
    import json
    made = [field(96, H=60 - 20 * k, N=32, seed=k, nv=12) for k in range(2)]
    made[0][0][5, 6, 7] = np.inf
    x, t, f = ([torch.from_numpy(m[0]).cuda() for m in made], [m[1] for m in made],
               [m[2] for m in made])
    cache = tmp_path / "tune.json"
    with st.Plan(f, mode="bilinear", tile=1) as p:
        want = p.candidates(x, t)
    with st.Plan(f, mode="bilinear", tile=-1, tune_cache=str(cache)) as p:
        for _ in range(2):
            assert p.candidates(x, t).tobytes() == want.tobytes()
            assert [p.last_stack_variant(k) for k in range(2)] == [0, 1]
    assert len(json.loads(cache.read_text())) == 1
