"""CPU check of k_sky_pass's shared variables (k_prep.cu), read from its
source: whatever all threads read after a barrier is written again only behind
another barrier, with the loop's body taken twice.  (A warp that still has to
read a flag must find the value that the barrier published: a warp that leaves
early takes its pixels out of the frame's statistics.)"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2303_07293_gb300", "csrc", "k_prep.cu")


def block(text, at):
    """The text of the brace block that opens at or after `at`, and its end."""
    at = text.index("{", at)
    depth = 0
    for k in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[at + 1:k], k + 1
    raise AssertionError("unbalanced braces")


def source():
    with open(SRC) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def events(text, body, name):
    """Reads and writes of `name` and barriers, in the order of the source;
    a loop without a condition counts twice, a device function that meets a
    barrier is one."""
    m = re.search(r"for \([^;]*;;[^)]*\)", body)
    if m:
        inner, end = block(body, m.end())
        body = body[:m.start()] + inner + inner + body[end:]
    out = []
    for t in re.finditer(r"__syncthreads\w*\(|\bsky_sums\(|\b%s\b(\s*=(?!=))?" % name, body):
        if t.group(0) == "sky_sums(":
            assert "__syncthreads()" in block(text, text.index("SkyPartial sky_sums("))[0]
            out.append("barrier")
        elif t.group(0).startswith("__sync"):
            out.append("barrier")
        else:
            out.append("write" if t.group(1) else "read")
    return out


def shared_names(body):
    decl = re.findall(r"__shared__\s+(?:bool|SkyState)\s+([^;]+);", body)
    return [n.strip() for d in decl for n in d.split(",")]


def test_flags_are_published_and_read_between_barriers():
    text = source()
    body, _ = block(text, text.index("k_sky_pass("))
    names = shared_names(body)
    assert len(names) >= 2
    body = re.sub(r"__shared__[^;]*;", "", body)
    for name in names:
        seq = events(text, body, name)
        assert "write" in seq and "read" in seq, name
        last = None
        for e in seq:
            if e == "write":
                assert last != "read", f"{name}: written while warps may still read it"
            if e == "read":
                assert last != "write", f"{name}: read without a barrier after its write"
            last = e


@pytest.mark.gpu
def test_far_outliers_give_the_same_statistics_every_time():
    # pixels far beyond the rest, once they are clipped, leave a set that is
    # summed again with a range of its own
    torch = pytest.importorskip("torch")
    import numpy as np

    import __graft_entry__
    import oracle
    import synth
    __graft_entry__.build()
    import paper_2303_07293_gb300 as st
    rng = np.random.default_rng(3)
    N, H, W = 64, 96, 128
    raw = (300.0 + 12.0 * rng.standard_normal((N, H, W))).astype(np.float32)
    raw.reshape(N, -1)[:, 77] = 10.0 ** rng.uniform(5, 9, N)
    x = torch.from_numpy(raw).cuda()
    f = synth.field_params(W, H, N, 0.0, 0.0, 1.0, 1, 0.0, 1.0, 1)
    _, omu, osd = oracle.normalize(raw)
    with st.Plan(f, normalize=True) as p:
        for _ in range(50):
            _, mu, sd = p.normalize(0, x)
            # (the bar of the other normalisation tests)
            assert np.all(np.abs(mu - omu) <= 1e-12 * np.abs(omu))
            assert np.all(np.abs(sd - osd) <= 1e-12 * osd)
