"""Writes st_runs.inc: the consumer loop of the run kernel (k_stack_runs.cu) as
inline PTX, one block per storage type.

A thread holds, for each of its 4 x-velocities, the sum S of the windows of the
frames so far: pair q = (window rows q, q + 4), q = 0..6, as a paired FP32
register.  A frame's word gives the window's byte offset in the ring, a case
(D: bit j set where x-velocity j + 1 reads the column next to that of
x-velocity j; R = 8..11 rows; the columns' direction), the ends of run and
stage, and, at the end of a run that another follows, that run's pattern.  The
case's body, entered by one indexed branch, loads R rows of each distinct
column once and adds its pairs to the sums of the x-velocities that read it.

Between two runs the row offset c of a y-velocity changes where their patterns
differ (the patterns are ordered so that mostly one y-velocity's does, by 1):
S moved by the old offset is added to its accumulators and S moved by the new
one subtracted, so that when S, moved by the last offset, is added at the end,
every frame has counted at its own offset.  The accumulators are in tensor
memory, columns j * 32 + x * 8 + ..: y-velocity j, x-velocity x, output rows
m, m + 4 in turn.

The block is one item up to the last addition: per stage a bounded wait on its
full barrier (all lanes; the first stage's wait is the caller's), its frames,
and the release of the slot.  Operands: %0..%27 S (zero on entry), %28 ring slot (out:
STAGES where a wait ran out), %29 its phase, %30 the current offsets, 2 bits per
y-velocity, and from bit 8 which accumulators hold anything (read-write); %31 stages of the item, negative where the warp has no
group, %32 address of the CTA's barriers (full, then empty), %33 address of the
warp's words in slot 0, %34 the lane's base address in the ring, %35 the warp's
tensor-memory address.

Run `python gen_runs.py` after a change; a CPU test runs the bodies
symbolically and checks that the committed file is this script's output.
"""
import os

HERE = os.path.dirname(os.path.abspath(__file__))
OUT = os.path.join(HERE, "st_runs.inc")
VEL, YVEL, PAIRS, ROWS = 4, 4, 7, 8
FRAMES, STAGES, GROUPS = 16, 2, 4
OFF_MASK, PAT_BIT, END_BIT, STAGE_BIT, CASE_BIT = 0x3FFFF, 18, 22, 23, 26
SLOT, PHASE, OFFS, NSTAGES, BASE, WORDS, LANE, TM = (f"%{28 + k}" for k in range(8))
TW = 16  # tensor-memory columns per access
WAIT_NS = 2000000000
# the order in which a tile's frames are taken: neighbours differ at one
# y-velocity by 1 (but for 3, 6 and 10, 13: at two)
ORDER = (7, 3, 6, 5, 1, 2, 4, 0, 8, 9, 11, 12, 10, 13, 14)
# storage: (element bytes, box row bytes, load, conversion to FP32)
DTYPES = {
    "f32": (4, 176, "ld.shared.f32 {d}, [{a}+{o}];", None),
    "f16": (2, 96, "ld.shared.b16 h{r}, [{a}+{o}];", "cvt.f32.f16 {d}, h{r};"),
    "bf16": (2, 96, "ld.shared.u16 u{r}, [{a}+{o}];", "shl.b32 u{r}, u{r}, 16;\nmov.b32 {d}, u{r};"),
}


def pat_off(pid, j):
    """Row offset of y-velocity j in pattern pid (minimum offset 0): ids 0..7
    rise by steps (bit 0, bit 1, bit 2); ids 8..14 fall by the steps of
    t = id - 7 read from the other end."""
    s = [((pid if pid < 8 else pid - 7) >> b) & 1 for b in range(3)]
    return sum(s[:j]) if pid < 8 else sum(s[j:])


def columns(d):
    """Distinct columns of case bits d: [(column, velocities that read it)]."""
    out = [(0, [0])]
    for j in range(VEL - 1):
        if (d >> j) & 1:
            out.append((out[-1][0] + 1, []))
        out[-1][1].append(j + 1)
    return out


def load_row(dtype, reg, row, col, tmp):
    esz, pitch, ld, cvt = DTYPES[dtype]
    L = [ld.format(d=reg, a="sa", o=row * pitch + col * esz, r=tmp)]
    if cvt:
        L += cvt.format(d=reg, r=tmp).split("\n")
    return L


def body(d, rows, down, dtype, pre):
    """PTX of one case; rows 0..pre-1 of column 0 are in v0.. already.  down:
    the columns step towards lower x."""
    L = []
    for col, vels in columns(d):
        for r in range(pre if col == 0 else 0, rows):
            L += load_row(dtype, f"v{r}", r, -col if down else col, r)
        for q in range(rows - 4):
            L.append(f"mov.b64 W, {{v{q}, v{q + 4}}};")
            for x in vels:
                L.append(f"add.rn.f32x2 %{x * PAIRS + q}, %{x * PAIRS + q}, W;")
    return L


def case_of(d, rows, down):
    """Case number: steps (3 bits), rows - 8 (2 bits), direction (1 bit; 0
    without steps)."""
    return d | (rows - 8) << 3 | (1 if down and d else 0) << 5


def step(c, n):
    """S from offset c to offset n in one y-velocity's accumulators (tensor
    memory at sa), two x-velocities (16 columns) at a time; pz: the item's
    first change there, which reads nothing."""
    regs = ", ".join(f"t{k}" for k in range(TW))
    L = []
    for first in (False, True):
        if first:
            L.append(f"RZ{c}{n}:")
        for h in range(0, VEL * ROWS, TW):
            if not first:
                L += [f"tcgen05.ld.sync.aligned.32x32b.x{TW}.b32 {{{regs}}}, [sa+{h}];",
                      "tcgen05.wait::ld.sync.aligned;"]
            for k in range(TW // 2):
                e = (h // 2 + k) // 4 * PAIRS + k % 4
                if first:
                    L.append(f"sub.rn.f32x2 W, %{e + c}, %{e + n};")
                else:
                    L += [f"mov.b64 W, {{t{2 * k}, t{2 * k + 1}}};",
                          f"add.rn.f32x2 W, W, %{e + c};",
                          f"sub.rn.f32x2 W, W, %{e + n};"]
                L.append(f"mov.b64 {{t{2 * k}, t{2 * k + 1}}}, W;")
            L.append(f"tcgen05.st.sync.aligned.32x32b.x{TW}.b32 [sa+{h}], {{{regs}}};")
        L += ["tcgen05.wait::st.sync.aligned;", "bra.uni RSTEP;"]
    return [f"@pz bra.uni RZ{c}{n};"] + L


def offsets(pid):
    """The 4 offsets of a pattern, 2 bits each."""
    return sum(pat_off(pid, j) << (2 * j) for j in range(YVEL)) if pid < 15 else 0


def item_loop(dtype):
    regs = ", ".join(f"t{k}" for k in range(TW))
    empty0 = 8 * STAGES
    L = ["{",
         ".reg .u32 sa, sid, sw, sn, sp, sleft, st0, st1, sj;",
         ".reg .f32 v<11>;", ".reg .b64 W;", f".reg .b32 t<{TW}>;",
         ".reg .pred pna, pz, pf, pl, pt, pall, pany;"]
    if dtype == "f16":
        L.append(".reg .b16 h<11>;")
    if dtype == "bf16":
        L.append(".reg .u32 u<11>;")
    L += [f"setp.lt.s32 pna, {NSTAGES}, 0;",
          f"abs.s32 sleft, {NSTAGES};",
          "bra.uni RRUN;",
          "RSTAGE:",
          f"mad.lo.u32 sa, {SLOT}, 8, {BASE};",
          f"mbarrier.try_wait.parity.shared::cta.b64 pt, [sa], {PHASE};",
          "vote.sync.all.pred pall, pt, 0xffffffff;",
          "@pall bra.uni RRUN;",
          "mov.u32 st0, %globaltimer_lo;",
          "RWAIT:",
          # (a warp without a group has nothing to be late for)
          "@pna nanosleep.u32 1000;",
          f"mbarrier.try_wait.parity.shared::cta.b64 pt, [sa], {PHASE}, 20000;",
          "vote.sync.all.pred pall, pt, 0xffffffff;",
          "@pall bra.uni RRUN;",
          "mov.u32 st1, %globaltimer_lo;",
          "sub.u32 st1, st1, st0;",  # modulo 2^32 ns: exact below 4.29 s
          f"setp.gt.u32 pt, st1, {WAIT_NS};",
          "vote.sync.any.pred pany, pt, 0xffffffff;",
          "@!pany bra.uni RWAIT;",
          f"mov.u32 {SLOT}, {STAGES};",
          "bra.uni REND;",
          "RRUN:",
          "@pna bra.uni RDONE;",
          f"mad.lo.u32 sp, {SLOT}, {GROUPS * FRAMES * 4}, {WORDS};",
          "ld.shared.u32 sw, [sp];",
          # a frame: its window and case, the next frame's word, whether the
          # run or the stage ends with it
          "RFRAME:",
          f"and.b32 sa, sw, {OFF_MASK};",
          f"add.u32 sa, sa, {LANE};"]
    for r in range(ROWS):   # every case uses these: loaded before the branch
        L += load_row(dtype, f"v{r}", r, 0, r)
    ncase = 64
    L += ["ld.shared.u32 sn, [sp+4];",
          f"shr.u32 sid, sw, {CASE_BIT};",
          f"and.b32 sw, sw, {(1 << END_BIT) | (1 << STAGE_BIT)};",
          "setp.eq.u32 pf, sw, 0;",
          "mov.u32 sw, sn;",
          "RT: .branchtargets " + ", ".join(
              f"RB{k & 31 if not k & 7 else k}" for k in range(ncase)) + ";",
          "brx.idx.uni sid, RT;"]
    for down in (False, True):
        for rows in range(8, 12):
            for d in range(1 if down else 0, 8):
                L.append(f"RB{case_of(d, rows, down)}:")
                L += body(d, rows, down, dtype, ROWS)
                L.append("bra.uni RNEXT;")
    # 8-bit offsets of 16 patterns in four 32-bit constants: select by the id
    words = [sum(offsets(4 * w + k) << (8 * k) for k in range(4)) for w in range(4)]
    L += ["RNEXT:",
          "add.u32 sp, sp, 4;",
          "@pf bra.uni RFRAME;",
          "ld.shared.u32 sn, [sp+-4];",   # the frame's word again
          f"and.b32 sa, sn, {1 << END_BIT};",
          "setp.eq.u32 pl, sa, 0;",
          "@pl bra.uni RKEEP;",
          # another run follows: its pattern's offsets
          f"shr.u32 sid, sn, {PAT_BIT - 3};",
          "and.b32 sid, sid, 120;",
          "setp.lt.u32 pl, sid, 64;",
          f"selp.b32 st0, {words[0]}, {words[2]}, pl;",
          f"selp.b32 st1, {words[1]}, {words[3]}, pl;",
          "and.b32 sj, sid, 32;",
          "setp.eq.u32 pl, sj, 0;",
          "selp.b32 st0, st0, st1, pl;",
          "and.b32 sid, sid, 24;",
          "shr.u32 st0, st0, sid;",
          "and.b32 st0, st0, 255;",
          # the y-velocities whose offset changes, one step of 1 at a time
          "RSTEP:",
          f"xor.b32 sid, st0, {OFFS};",
          "and.b32 sid, sid, 255;",
          "setp.eq.u32 pl, sid, 0;",
          "@pl bra.uni RKEEP;",
          "neg.s32 sj, sid;",
          "and.b32 sj, sj, sid;",
          "bfind.u32 sj, sj;",
          "and.b32 sj, sj, 6;",                    # 2 j of the lowest that differs
          f"shl.b32 sa, sj, {(VEL * ROWS // 2).bit_length() - 1};",
          f"add.u32 sa, sa, {TM};",
          f"shr.u32 sid, {OFFS}, sj;",
          "and.b32 st1, sid, 256;",                # (bit 8 + 2 j: touched before)
          "setp.eq.u32 pz, st1, 0;",
          "and.b32 sid, sid, 3;",
          "shr.u32 st1, st0, sj;",
          "and.b32 st1, st1, 3;",
          "setp.gt.u32 pl, st1, sid;",
          "mov.u32 st1, 1;",
          "shl.b32 st1, st1, sj;",
          f"@pl add.u32 {OFFS}, {OFFS}, st1;",
          f"@!pl sub.u32 {OFFS}, {OFFS}, st1;",
          "shl.b32 st1, st1, 8;",
          f"or.b32 {OFFS}, {OFFS}, st1;",
          "@!pl add.u32 sid, sid, 2;",             # up from 0, 1, 2; down from 1, 2, 3
          "RFT: .branchtargets RF0, RF1, RF2, RF3, RF4, RF5;",
          "brx.idx.uni sid, RFT;"]
    for k in range(6):
        L.append(f"RF{k}:")
        L += step(k, k + 1) if k < 3 else step(k - 2, k - 3)
    L += [
          "RKEEP:",
          f"and.b32 sn, sn, {1 << STAGE_BIT};",
          "setp.eq.u32 pl, sn, 0;",
          "@pl bra.uni RFRAME;",
          "RDONE:",
          # release the slot (every lane's reads are done), next slot
          "bar.warp.sync 0xffffffff;",
          f"mad.lo.u32 sa, {SLOT}, 8, {BASE};",
          "mov.u32 sid, %laneid;",
          "setp.eq.u32 pl, sid, 0;",
          f"@pl mbarrier.arrive.shared::cta.b64 _, [sa+{empty0}];",
          f"add.u32 {SLOT}, {SLOT}, 1;",
          f"setp.eq.u32 pl, {SLOT}, {STAGES};",
          f"@pl mov.u32 {SLOT}, 0;",
          f"@pl xor.b32 {PHASE}, {PHASE}, 1;",
          "sub.u32 sleft, sleft, 1;",
          "setp.ne.u32 pl, sleft, 0;",
          "@pl bra.uni RSTAGE;",
          "REND:", "}"]
    return L


def render():
    out = ["// Generated by gen_runs.py: the consumer loop of the run kernel.  Do not edit.",
           "#pragma once", ""]
    for dtype in DTYPES:
        out.append(f"#define ST_RUN_ITEM_{dtype.upper()} \\")
        for ln in item_loop(dtype):
            out.append(f'  "{ln}\\n\\t" \\')
        out.append("")
    ops = ", ".join(f'"+l"(s[{k}])' for k in range(VEL * PAIRS))
    out.append("#define ST_RUN_OPERANDS(s, slot, ph, off, stages, base, words, lane, tm) \\")
    out.append(f'  : {ops}, "+r"(slot), "+r"(ph), "+r"(off) \\')
    out.append('  : "r"(stages), "r"(base), "r"(words), "r"(lane), "r"(tm) : "memory"')
    out.append("")
    return "\n".join(out)


if __name__ == "__main__":
    with open(OUT, "w") as fh:
        fh.write(render())
    print(OUT)
