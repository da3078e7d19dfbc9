"""The padded copy of raw frames whose rows are no multiple of 16 bytes is
taken when a search uses it, leaves the caller at least as much device memory
as it takes, and is given back when the motion no longer fits the kernels that
read it."""
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


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("mode", ["nearest", "bilinear"])
def test_copy_is_held_only_while_it_is_read(st, mode):
    N, H, W, nv = 40, 1021, 1023, 13
    x = torch.randn((N, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    copy = 4 * N * H * (W + 1)
    slow = np.linspace(0.0, 2.0, N)
    fast = slow * 40.0   # adjacent velocities many pixels apart
    f = synth.field_params(W, H, N, 0.0, -0.2 * (nv // 2), 0.2, nv, -0.2 * (nv // 2), 0.2, nv,
                           tau=5.0)
    got = {}
    for tile in (1, 0):
        before = free()
        with st.Plan(f, mode=mode, tile=tile) as p:
            rest = before - free()   # what a plan of this kind holds without a copy
            assert rest < 0.9 * copy + 400e6
            got[tile] = [p.candidates(x, fast)]
            assert abs(before - free() - rest) < 0.5 * copy   # the motion does not fit
            got[tile].append(p.candidates(x, slow))
            held = before - free() - rest
            assert (held > 0.9 * copy) == (tile == 0)
            assert p.last_stack_variant(0) == (1 if tile == 0 else 0)
            got[tile].append(p.candidates(x, fast))
            assert before - free() - rest < 0.5 * copy
            assert p.last_stack_variant(0) == 0
    for a, b in zip(got[0], got[1]):
        assert a.tobytes() == b.tobytes()


def test_copy_leaves_as_much_memory_as_it_takes(st):
    # less than twice the copy is free: the direct gather reads the frames
    N, H, W, nv = 40, 1021, 1023, 13
    x = torch.randn((N, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    copy = 4 * N * H * (W + 1)
    t = np.linspace(0.0, 2.0, N)
    f = synth.field_params(W, H, N, 0.0, -0.2 * (nv // 2), 0.2, nv, -0.2 * (nv // 2), 0.2, nv,
                           tau=5.0)
    with st.Plan(f) as p:
        want = p.candidates(x, t)
        assert p.last_stack_variant(0) == 1
    with st.Plan(f, tile=1) as p:
        p.candidates(x, t)
    torch.cuda.empty_cache()
    with st.Plan(f) as p:
        hold = torch.empty(int(free() - 1.6 * copy), dtype=torch.uint8, device="cuda")
        got = p.candidates(x, t)
        assert p.last_stack_variant(0) == 0
        del hold
        torch.cuda.empty_cache()
    assert got.tobytes() == want.tobytes()
