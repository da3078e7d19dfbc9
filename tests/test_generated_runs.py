"""CPU checks of the run kernel's generated PTX (gen_runs.py): a symbolic run
of every case, of every step between row offsets and of the pattern table
against their definitions, and the committed include against its generator."""
import importlib.util
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_07293_gb300", "csrc")


def _gen(name="gen_runs"):
    spec = importlib.util.spec_from_file_location(name, os.path.join(CSRC, name + ".py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def test_committed_include_is_the_generator_output():
    with open(os.path.join(CSRC, "st_runs.inc")) as fh:
        assert fh.read() == _gen().render()


def test_patterns_are_those_of_the_other_bodies_and_each_is_taken_once():
    g, b = _gen(), _gen("gen_bodies")
    assert [[g.pat_off(p, j) for j in range(4)] for p in range(15)] == \
        [[b.pat_off(p, j) for j in range(4)] for p in range(15)]
    assert sorted(g.ORDER) == list(range(15))
    with open(os.path.join(CSRC, "k_stack_runs.cu")) as fh:
        src = fh.read()
    m = re.search(r"order\[kPatterns\] = \{([0-9, ]+)\}", src)
    assert tuple(int(v) for v in m.group(1).split(",")) == g.ORDER
    # neighbours differ by one step of one y-velocity, but for two pairs
    diff = [sum(abs(g.pat_off(p, j) - g.pat_off(q, j)) for j in range(4))
            for p, q in zip(g.ORDER, g.ORDER[1:])]
    assert sorted(diff) == [1] * 12 + [2, 2]


def test_cases_add_each_velocitys_window():
    # after a case, pair q of velocity x has gained rows q and q + 4 of the
    # column that x reads, once each
    g = _gen()
    for dtype, (esz, pitch, _, _) in g.DTYPES.items():
        text = "\n".join(g.item_loop(dtype))
        head = text.split("RFRAME:\n", 1)[1].split("RT:", 1)[0]
        targets = text.split("RT: .branchtargets ", 1)[1].split(";", 1)[0].split(", ")
        for case in range(64):
            d, rows, down = case & 7, 8 + (case >> 3 & 3), case >> 5
            lab = targets[case]
            assert lab == f"RB{g.case_of(d, rows, down)}"
            body = text.split(lab + ":\n", 1)[1].split("bra.uni RNEXT;", 1)[0]
            v, w, half, got = {}, None, {}, {}
            for ln in head.splitlines() + body.splitlines():
                m = re.fullmatch(r"ld\.shared\.(f32 v|b16 h|u16 u)(\d+), \[sa\+(-?\d+)\];", ln)
                if m:
                    (v if m.group(1) == "f32 v" else half)[int(m.group(2))] = int(m.group(3))
                    continue
                m = re.fullmatch(r"(?:cvt\.f32\.f16|mov\.b32) v(\d+), [hu](\d+);", ln)
                if m:
                    v[int(m.group(1))] = half[int(m.group(2))]
                    continue
                m = re.fullmatch(r"mov\.b64 W, \{v(\d+), v(\d+)\};", ln)
                if m:
                    w = (v[int(m.group(1))], v[int(m.group(2))])
                    continue
                m = re.fullmatch(r"add\.rn\.f32x2 %(\d+), %(\d+), W;", ln)
                if m:
                    assert m.group(1) == m.group(2) and int(m.group(1)) not in got
                    got[int(m.group(1))] = w
            for x in range(4):
                col = bin(d & ((1 << x) - 1)).count("1") * (-1 if down else 1)
                for q in range(7):
                    want = (q * pitch + col * esz, (q + 4) * pitch + col * esz)
                    assert got.get(7 * x + q) == (want if q < rows - 4 else None), (case, x, q)


def test_steps_move_the_sum_from_one_offset_to_the_next():
    # accumulator m of x-velocity x gains pair m + c less pair m + n
    g = _gen()
    for c, n in ((0, 1), (1, 2), (2, 3), (1, 0), (2, 1), (3, 2)):
        acc, col = {}, {}
        first = {}
        table, w = acc, None
        for ln in g.step(c, n):
            if ln.startswith("RZ"):
                table, col = first, {}
                continue
            m = re.fullmatch(r"tcgen05\.ld.*\[sa\+(\d+)\];", ln)
            if m:
                col = {f"t{k}": ("acc", int(m.group(1)) + k) for k in range(g.TW)}
                continue
            m = re.fullmatch(r"mov\.b64 W, \{(t\d+), (t\d+)\};", ln)
            if m:
                w = [col[m.group(1)], col[m.group(2)]]
                continue
            m = re.fullmatch(r"(add|sub)\.rn\.f32x2 W, (W|%\d+), %(\d+);", ln)
            if m:
                if m.group(2) != "W":
                    w = [int(m.group(2)[1:])]
                w = w + [(m.group(1), int(m.group(3)))]
                continue
            m = re.fullmatch(r"mov\.b64 \{(t\d+), (t\d+)\}, W;", ln)
            if m:
                col[m.group(1)] = col[m.group(2)] = tuple(w)
                continue
            m = re.fullmatch(r"tcgen05\.st.*\[sa\+(\d+)\], .*", ln)
            if m:
                for k in range(g.TW):
                    table[int(m.group(1)) + k] = col[f"t{k}"]
        for k in range(32):
            x, mm = k // 8, k % 8 // 2
            plus, minus = 7 * x + mm + c, 7 * x + mm + n
            pair = k // 2 * 2
            assert acc[k] == (("acc", pair), ("acc", pair + 1), ("add", plus), ("sub", minus))
            assert first[k] == (plus, ("sub", minus))


def test_pattern_words_give_each_patterns_offsets():
    # the instructions between a frame that ends a run and the step loop, run
    # on that frame's word for every pattern of the next run
    g = _gen()
    for dtype in g.DTYPES:
        lines = g.item_loop(dtype)
        k = lines.index("@pl bra.uni RKEEP;", lines.index("RNEXT:")) + 1
        code = lines[k:lines.index("RSTEP:")]
        for pid in range(15):
            reg = {"sn": pid << g.PAT_BIT | 1 << g.END_BIT | 0x155, "pl": None}

            def val(t):
                return reg[t] if t in reg else int(t, 0) & 0xffffffff
            for ln in code:
                op, rest = ln.rstrip(";").split(" ", 1)
                d, *a = [t.strip() for t in rest.split(",")]
                v = [bool(reg[t]) if t == "pl" else val(t) for t in a]
                reg[d] = {"shr.u32": lambda: v[0] >> v[1], "and.b32": lambda: v[0] & v[1],
                          "setp.lt.u32": lambda: v[0] < v[1], "setp.eq.u32": lambda: v[0] == v[1],
                          "selp.b32": lambda: v[0] if v[2] else v[1]}[op]()
            assert [reg["st0"] >> (2 * j) & 3 for j in range(4)] == \
                [g.pat_off(pid, j) for j in range(4)], pid
            assert reg["st0"] < 256
