"""A tune cache serves only the list of variants that it was written for."""
import json

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


def test_entries_of_another_list_are_left_alone(st, tmp_path):
    W, H, N, nv = 128, 96, 40, 16
    rng = np.random.default_rng(2)
    x = torch.from_numpy(rng.standard_normal((N, H, W)).astype(np.float32)).cuda()
    t = np.linspace(0.0, 2.0, N)
    f = synth.field_params(W, H, N, 1.0, -1.6, 0.2, nv, -1.6, 0.2, nv, tau=3.0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    old = f"W{W}_H{H}_N{N}_nvx{nv}_nvy{nv}_st0_m0_sm{sms}"   # without the list's mark
    cache = tmp_path / "tune.json"
    cache.write_text(json.dumps({old: 7}) + "\n")
    with st.Plan(f, tile=-1, tune_cache=str(cache)) as p:
        first, name = p.candidates(x, t), p.stack_variant_name(0)
    tab = json.loads(cache.read_text())
    assert tab.pop(old) == 7 and len(tab) == 1
    (key, v), = tab.items()
    assert key.startswith(old)
    with st.Plan(f, tile=-1, tune_cache=str(cache)) as p:   # served
        assert p.candidates(x, t).tobytes() == first.tobytes()
        assert p.stack_variant_name(0) == name
    assert json.loads(cache.read_text()) == {old: 7, key: v}
