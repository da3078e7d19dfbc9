"""GPU parity of fields whose rows are no multiple of 16 bytes: the plan keeps
them with padded rows for the register-window kernels.  Candidate lists equal
the direct-gather kernel's on the same frames, and the stack planes the
oracle's, at widths about the padding, for every storage, with and without
normalisation and for both samplings; what needs the caller's own rows
(refinement) still refuses them."""
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


def field(W, H, N, nv=13, tau=2.5):
    rng = np.random.default_rng(W * H + N)
    fr = rng.standard_normal((N, H, W)).astype(np.float32)
    t = np.sort(rng.uniform(0.0, 2.0, N))
    f = synth.field_params(W, H, N, float(t[N // 2]), -0.4 * (nv // 2), 0.4, nv,
                           -0.4 * (nv // 2) + 0.1, 0.4, nv, tau=tau)
    synth.render_movers(fr, t, f["t_ref"], [[W * 0.5, H * 0.5, 1.0, -0.7, 3.0]])
    return fr, t, f


@pytest.mark.parametrize("storage,normalize,mode", [
    ("f32", True, "nearest"), ("f32", False, "nearest"), ("f16", True, "nearest"),
    ("bf16", False, "nearest"), ("f32", True, "bilinear"), ("f32", False, "bilinear"),
    ("f16", True, "bilinear")])
@pytest.mark.parametrize("W,H,N", [(61, 40, 12), (63, 17, 40), (33, 64, 9), (101, 33, 33),
                                   (1025, 3, 10), (9, 9, 8)])
def test_odd_widths_equal_direct_gather(st, storage, normalize, mode, W, H, N):
    fr, t, f = field(W, H, N)
    x = torch.from_numpy(fr).cuda()
    got = []
    for tile in (0, 1):
        with st.Plan(f, storage=storage, mode=mode, normalize=normalize, tile=tile) as p:
            got.append(p.candidates(x, t))
            again = p.candidates(x, t)   # the padded rows are the same every time
            assert p.last_stack_variant(0) == (1 if tile == 0 else 0)
        for k in again.dtype.names:
            assert np.array_equal(again[k], got[-1][k])
    assert len(got[0]) > 0
    for k in got[0].dtype.names:
        assert np.array_equal(got[0][k], got[1][k]), k


def test_odd_width_planes_and_limits(st):
    fr, t, f = field(61, 23, 14)
    x = torch.from_numpy(fr).cuda()
    ks = np.arange(f["nvx"] * f["nvy"], dtype=np.int32)
    oS, oC = oracle.stack_planes(fr, t, f, ks, prec="fp32")
    with st.Plan(f) as p:
        S, C = p.dump_stack(0, x, t, ks)
        assert np.array_equal(S.cpu().numpy(), oS.astype(np.float32))
        assert np.array_equal(C.cpu().numpy(), oC)
        out, n, _ = p.search(x, t)
        with pytest.raises(st.StError):   # as without the copy
            p.refine(out[:1])
    # motion beyond the boxes: the frames themselves are searched
    g = dict(f, dvx=3.0, vx0=-18.0)
    with st.Plan(g) as p, st.Plan(g, tile=1) as q:
        a, b = p.candidates(x, t), q.candidates(x, t)
        assert p.last_stack_variant(0) == 0
    for k in a.dtype.names:
        assert np.array_equal(a[k], b[k])
