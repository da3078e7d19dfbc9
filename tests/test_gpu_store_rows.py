"""GPU parity of the store pass for frames off 16 bytes: pixels are taken in
their order whatever the rows' length, at widths about the 256 pixels between
a thread's, one-pixel rows and lengths about the 2048 pixels of a block."""
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


# (8 frames of 2 Mi pixels: blocks that take more than one round)
@pytest.mark.parametrize("N,H,W", [(3, 700, 1), (2, 333, 3), (5, 31, 33), (2, 9, 255), (2, 9, 257),
                                   (3, 5, 511), (2, 3, 1023), (2, 3, 1025), (1, 1, 1021),
                                   (8, 2051, 1021), (200, 7, 29), (2, 2, 1024), (3, 1, 2047), (2, 1, 2049)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_rows_of_any_length(st, N, H, W, storage):
    rng = np.random.default_rng(W)
    raw = (250.0 + 10.0 * rng.standard_normal((N, H, W))).astype(np.float32)
    raw.reshape(-1)[::53] = np.nan
    buf = torch.zeros(1 + raw.size, device="cuda")
    x = buf[1:].view(N, H, W)   # off 16 bytes whatever the width
    x.copy_(torch.from_numpy(raw))
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage]
    f = synth.field_params(W, H, N, 0.0, 0.0, 1.0, 1, 0.0, 1.0, 1, tau=0.0)
    with st.Plan(f, normalize=True, storage=storage, cr_clip=2.5) as p:
        cube, mu, sd = p.normalize(0, x)
    with np.errstate(invalid="ignore", divide="ignore"):
        v = ((raw.astype(np.float64) - mu[:, None, None]) * (1.0 / sd)[:, None, None])
    v = np.where(np.isfinite(raw), v, 0.0).astype(np.float32)
    v[np.abs(v) > 2.5] = 0.0
    assert torch.equal(cube.cpu(), torch.from_numpy(v).to(dt))
    if W < 8:
        return
    # padded rows of a plan's own cube, as a search fills them: its stack of
    # no motion is the frames' sum in frame order
    x.copy_(torch.from_numpy(np.where(np.isfinite(raw), raw, 0.0).astype(np.float32)))
    with st.Plan(f, storage=storage) as p:
        S, _ = p.dump_stack(0, x, np.zeros(N), [0])
    want = torch.zeros((H, W))
    for i in range(N):
        want += x[i].cpu().to(dt).float()
    assert torch.equal(S[0].cpu(), want)


def test_narrow_rows_cost_what_their_bytes_do(st):
    # 28 MB take 4 us at the HBM rate: ten times that is allowed above the
    # same number of pixels in rows of 16 bytes
    best = {}
    for H, W in ((2000, 37), (1000, 74), (925, 80)):
        x = torch.randn((64, H, W), device="cuda")
        f = synth.field_params(W, H, 64, 0.0, 0.0, 1.0, 1, 0.0, 1.0, 1, tau=1e6)
        out = torch.zeros((1, 7), dtype=torch.int32, device="cuda")
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        with st.Plan(f, storage="f16") as p:
            took = []
            for _ in range(30):
                a.record()
                p.search(x, np.arange(64.0), capacity=1, out=out)
                b.record()
                torch.cuda.synchronize()
                took.append(a.elapsed_time(b) - p.last_stack_kernel_time()[0])
        best[W] = min(took[3:])
    assert best[37] <= best[80] + 0.04 and best[74] <= best[80] + 0.04
