"""CPU check of the generated bilinear bodies (gen_bodies.py): a symbolic run
of every pattern's body gives each accumulator pair the upper window pair with
weight 1 - fy_j and then the lower one with weight fy_j, once each."""
import importlib.util
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_07293_gb300", "csrc")


def test_bilinear_bodies_weigh_both_rows_of_each_sample():
    spec = importlib.util.spec_from_file_location("gen", os.path.join(CSRC, "gen_bodies.py"))
    g = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(g)
    for ky, frames, row_bytes, stages, warps, dtype in g.ITEMS_BL:
        kh, esz = ky // 2, g.ELEM[dtype]
        lines, n_acc = g.item_loop_bl(ky, frames, row_bytes, stages, warps, dtype)
        assert n_acc == 4 * kh
        text = "\n".join(lines)
        head = text.split("SLOOP:\n", 1)[1].split("BTT:", 1)[0]
        for j in range(4):
            assert f"ld.shared.v2.b64 {{sF{j}, sG{j}}}, [syp+{16 * j}];" in head
        for p in range(15):
            body = text.split(f"BT{p}:\n", 1)[1].split("bra.uni SNEXT;", 1)[0]
            raw, sv, reg, got = {}, {}, {}, {}
            for ln in head.splitlines() + body.splitlines():
                m = re.fullmatch(r"ld\.shared\.(f32 sv|b16 sh|u16 su)(\d), \[sa\+(\d+)\];", ln)
                if m:
                    (sv if m.group(1) == "f32 sv" else raw)[m.group(2)] = int(m.group(3))
                    continue
                m = re.fullmatch(r"(?:cvt\.f32\.f16|mov\.b32) sv(\d), s[hu](\d);", ln)
                if m:
                    sv[m.group(1)] = raw[m.group(2)]
                    continue
                m = re.fullmatch(r"mov\.b64 (s[AB]), \{sv(\d), sv(\d)\};", ln)
                if m:
                    reg[m.group(1)] = (sv[m.group(2)], sv[m.group(3)])
                elif ln == "sub.rn.f32x2 sB, sB, sA;":
                    reg["sB"] = ("diff", reg["sB"], reg["sA"])
                elif ln == "fma.rn.f32x2 sH, sX, sB, sA;":
                    _, b, a = reg["sB"]
                    assert a == reg["sA"] and b == tuple(v + esz for v in a)
                    reg["sH"] = a
                else:
                    m = re.fullmatch(r"fma\.rn\.f32x2 %(\d+), s([FG])(\d), sH, %(\d+);", ln)
                    if m:
                        assert m.group(1) == m.group(4)
                        got.setdefault(int(m.group(1)), []).append(
                            (m.group(2), int(m.group(3)), reg["sH"]))
            for a in range(n_acc):
                j, mm = divmod(a, kh)
                r = mm + g.pat_off(p, j)
                assert got[a] == [
                    ("G", j, (r * row_bytes, (r + kh) * row_bytes)),
                    ("F", j, ((r + 1) * row_bytes, (r + 1 + kh) * row_bytes))], (ky, p, a)
