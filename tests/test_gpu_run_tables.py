"""A plan that has no room for what only the default stack kernel reads is
still made, and its searches give the same lists by another kernel."""
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


def test_plan_without_room_for_the_run_tables(st):
    # tables that only the default kernel reads: without them another runs
    W, H, N, nvx = 64, 32, 1500, 100000
    f = synth.field_params(W, H, N, 0.0, 0.0, 1e-5, nvx, 0.0, 1.0, 1, tau=8.0)
    tables = 4 * N * nvx // 4   # a word for every 4 x-velocities and frame
    x = torch.randn((N, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    t = np.linspace(0.0, 1.0, N)
    kw = dict(pending_capacity=1 << 16)
    torch.cuda.empty_cache()
    before = free()
    with st.Plan(f, **kw) as p:
        need = before - free()
        out, n, _ = p.search(x, t, capacity=1 << 10)
        want = p.to_numpy(out, n)
    with st.Plan(f, tile=2, **kw) as p:   # (every kernel is loaded before the memory is full)
        p.search(x, t, capacity=1 << 10)
    torch.cuda.empty_cache()
    hold = torch.empty(int(free() - need + 0.5 * tables), dtype=torch.uint8, device="cuda")
    with st.Plan(f, **kw) as p:
        del hold
        torch.cuda.empty_cache()
        out, n, _ = p.search(x, t, capacity=1 << 10)
        assert "runs" not in p.stack_variant_name(0)
        assert p.to_numpy(out, n).tobytes() == want.tobytes()
