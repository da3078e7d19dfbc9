"""Searches whose pending list overflows: the second pass runs only where it
can differ from the first, is counted with it, and is not repeated for the
next frames of the same times."""
import time

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


def field(W=128, H=64, N=60, nv=24, tau=1.0, seed=9):
    rng = np.random.default_rng(seed)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    t = np.sort(rng.uniform(0.0, 2.0, N))
    dv = 0.4 / float(np.abs(t - t[N // 3]).max())
    f = synth.field_params(W, H, N, float(t[N // 3]), -dv * (nv // 2), dv, nv, -dv * (nv // 2), dv,
                           nv, tau=tau)
    return torch.from_numpy(fr).cuda(), t, f


def least_capacity(st, x, t, f, **kw):
    lo, hi = 1, 1 << 21
    while lo < hi:
        mid = (lo + hi) // 2
        with st.Plan(f, pending_capacity=mid, **kw) as p:
            try:
                p.search(x, t)
                hi = mid
            except st.StError:
                lo = mid + 1
    return lo


@pytest.mark.parametrize("graph", [False, True])
def test_margin_that_does_not_fit_is_found_out_once(st, graph):
    x, t, f = field()
    kw = dict(normalize=True, cr_clip=10.0)
    cap = least_capacity(st, x, t, f, tile=2, **kw)
    with st.Plan(f, tile=2, **kw) as p:
        want = p.candidates(x, t)
    with st.Plan(f, tile=9, use_graph=graph, pending_capacity=cap, **kw) as p:
        passes = []
        for _ in range(4):
            got = p.candidates(x, t)
            assert got.tobytes() == want.tobytes()
            passes.append(p.last_stack_kernel_time()[1])
        assert passes == [2, 1, 1, 1]   # both passes counted; then the one that fits
        assert p.last_graph_replayed() == graph
        # other times: the margin is tried again
        t2 = t + 1e-12
        for expect in (2, 1):
            assert p.candidates(x, t2).tobytes() == want.tobytes()
            assert p.last_stack_kernel_time()[1] == expect
    with st.Plan(f, tile=9, use_graph=graph, **kw) as p:   # room for the margin: one pass
        p.candidates(x, t)
        assert p.last_stack_kernel_time()[1] == 1 and "runs" in p.stack_variant_name(0)


@pytest.mark.parametrize("mode,tile", [("nearest", 2), ("nearest", 4), ("nearest", 1),
                                       ("bilinear", 0)])
def test_overflow_is_reported_after_one_pass(st, mode, tile):
    # a few more points than the list holds: the search takes no longer than
    # one that succeeds (half as long again for the clock's sake)
    # (interpolated noise is weaker)
    x, t, f = field(W=512, H=512, N=48, nv=64, tau=4.7 if mode == "nearest" else 3.0)
    kw = dict(mode=mode, tile=tile, normalize=True, cr_clip=10.0)
    best = {}
    for cap in (1, 1 << 22):
        with st.Plan(f, pending_capacity=cap, **kw) as p:
            took = []
            for _ in range(6):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                if cap == 1:
                    with pytest.raises(st.StError):
                        p.search(x, t)
                else:
                    p.search(x, t)
                took.append(time.perf_counter() - t0)
            best[cap] = min(took)
    assert best[1] <= 1.5 * best[1 << 22]
