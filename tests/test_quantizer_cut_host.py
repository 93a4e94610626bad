"""How the quantizer's launches are cut, on the CPU: every layer gets a cut that fits in shared memory, and in none of them can a team
of warps take a ring slot's phase before last for the last one, in whatever order the copies land."""
import ctypes
import itertools
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIELDS = ("groups", "stages", "teams", "ntiles", "nchunks", "slots", "xslots", "refetch", "smem")
NONE, INT, F16, MXFP, MXINT = range(5)
SOURCE = """
#include "lq_quant_cut.h"
extern "C" int cut(int br, int M, int nst, int rn, int planes, int groups, int stages, int* out) {
  lqcut::QuantCut c{};
  if (!lqcut::plan_cut_as_asked(br, M, nst, rn, planes, 148, groups, stages, c)) return 0;
  const int v[] = {c.groups, c.stages, c.teams, c.ntiles, c.nchunks, c.slots, c.xslots, c.refetch, c.smem};
  for (int i = 0; i < 9; ++i) out[i] = v[i];
  return 1;
}
extern "C" int leaves_first(int refetch, int two_planes, double bytes) {
  lqcut::QuantCut c{};
  c.refetch = refetch;
  return lqcut::x_leaves_first(c, two_planes != 0, bytes);
}
"""


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("cut")
    (d / "cut.cpp").write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2604_18117_b200", "csrc"), "-I", os.path.join(cuda, "include"), str(d / "cut.cpp"), "-o", str(d / "cut.so")],
                   check=True)
    lib = ctypes.CDLL(str(d / "cut.so"))

    lib.leaves_first.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_double]

    def get(br, M, nst, rn, planes=1, groups=0, stages=0):
        out = (ctypes.c_int * 9)()
        return dict(zip(FIELDS, out)) if lib.cut(br, M, nst, rn, planes, groups, stages, out) else None

    get.leaves_first = lambda c, M, K, planes=1: bool(lib.leaves_first(c["refetch"], planes == 2, M * (2.0 * K + planes * -(-K // 128) * 128)))
    return get


def _layers():
    """(branch kind, rows of the first factor, digit planes) of every rank the formats take."""
    yield NONE, 16, 1
    for br, top, planes in ((INT, 128, 1), (F16, 64, 1), (MXFP, 128, 1), (MXINT, 128, 1), (MXINT, 64, 2)):
        for rn in range(16, top + 1, 16):
            yield br, rn, planes


def _mistaken(br, c, tiles=4):
    """The chunk of X or of operands (if any) whose late landing lets a team go on too early.  One chunk's copy lands last of all,
    everything else happens as soon as it can; a wait sees one bit of a barrier's phase, as mbarrier.try_wait.parity does."""
    T, n, S, XS = c["teams"], c["nchunks"], c["slots"], c["xslots"]
    walks = [(t, w) for t in range(tiles) for w in range(2 if br == INT else 1)]
    streams = [(t, w) for t, w in walks if w == 0 or c["refetch"]]                 # what the producer fetches, chunk by chunk
    seq_of = {tw: i * n for i, tw in enumerate(streams)}
    has_branch = br != NONE
    plan = [[] for _ in range(T)]                                                   # a team's steps: a chunk, or None: all teams meet
    for t, w in walks:
        last = w == (1 if br == INT else 0)
        x0 = seq_of[(t, w)] if (t, w) in seq_of else seq_of[(t, 0)]
        for k in range(n):
            plan[(t * n + k) % T].append((x0 + k, t * n + k if last and has_branch else None, last or c["refetch"]))
        if br == INT and w == 0:
            for p in plan:
                p.append(None)
    total = len(streams) * n
    for late in range(total):
        landed, released, made, retired = [0] * XS, [0] * XS, [0] * S, [0] * S     # completed phases of the slots' barriers
        is_landed, at, issued, done_mma, met = set(), [0] * T, 0, 0, 0
        open_ops, forced = {}, False
        passes = lambda count, use: (count & 1) != (use & 1)                       # noqa: E731
        while True:
            moved = False
            while issued < total and passes(released[issued % XS], issued // XS + 1):
                if issued != late or forced:
                    landed[issued % XS] += 1
                    is_landed.add(issued)
                issued, moved = issued + 1, True
            for t in range(T):
                while at[t] < len(plan[t]):
                    step = plan[t][at[t]]
                    if step is None:
                        if min(sum(s is None for s in plan[u][:at[u]]) + (at[u] < len(plan[u]) and plan[u][at[u]] is None) for u in range(T)) \
                                <= sum(s is None for s in plan[t][:at[t]]):
                            break
                        at[t], moved = at[t] + 1, True
                        continue
                    x, e, free = step
                    if not passes(landed[x % XS], x // XS):
                        break
                    if x not in is_landed:
                        return ("X", x, late)
                    if e is not None:
                        if not passes(retired[e % S], e // S + 1):
                            break
                        if retired[e % S] < e // S:
                            return ("operands", e, late)
                        open_ops[e] = True
                    if free:
                        released[x % XS] += 1
                    at[t], moved = at[t] + 1, True
            while open_ops.pop(done_mma, False):                                    # MMAs retire in order
                retired[done_mma % S] += 1
                done_mma, moved = done_mma + 1, True
            if not moved:
                if late in is_landed or issued <= late:
                    break
                landed[late % XS] += 1                                              # nothing else can move: the late copy lands
                is_landed.add(late)
                forced = True
        assert all(at[t] == len(plan[t]) for t in range(T)), (c, late)
    return None


def test_every_layer_has_a_cut_and_no_phase_is_mistaken_for_another(cut):
    seen = {}
    for (br, rn, planes), M, nst in itertools.product(_layers(), (1, 40, 256, 1000, 4096, 8192, 32768), (1, 2, 3, 5, 8, 9, 12, 18, 19, 24, 27, 36, 44, 64)):
        c = cut(br, M, nst, rn, planes)
        assert c is not None, (br, rn, planes, M, nst)
        assert c["smem"] <= 227 * 1024 and c["teams"] * c["groups"] * c["stages"] <= 15 and c["xslots"] <= 12 and c["slots"] <= 4
        seen.setdefault((br, c["teams"], c["nchunks"], c["slots"], c["xslots"], c["refetch"]), c)
    wrong = [(key, m) for key, c in seen.items() if (m := _mistaken(key[0], c)) is not None]
    assert not wrong, wrong[:5]


def test_every_value_of_the_options_gives_a_cut(cut):
    """What lq_set_option takes for "quant_warps" and "quant_ctas" never refuses a launch; a cut that a launch can have is the one asked
    for, and none mistakes a phase."""
    seen = {}
    for (br, rn, planes), M, nst in itertools.product(_layers(), (1, 300, 8192), (1, 3, 9, 44)):
        for groups, stages in itertools.product(range(10), range(5)):
            c = cut(br, M, nst, rn, planes, groups, stages)
            assert c is not None and c["smem"] <= 227 * 1024, (br, rn, planes, M, nst, groups, stages)
            g = min(groups, 8)
            if br == NONE and g * stages <= 15 and stages <= nst:
                assert (g or c["groups"], stages or c["stages"]) == (c["groups"], c["stages"])
            seen.setdefault((br, c["teams"], c["nchunks"], c["slots"], c["xslots"], c["refetch"]), c)
    wrong = [(key, m) for key, c in seen.items() if (m := _mistaken(key[0], c, tiles=2)) is not None]
    assert not wrong, wrong[:5]


def _rounds(br, c):
    """A launch in rounds (one chunk for every team) of so many warps: what the cost model compares."""
    return -(-c["ntiles"] // 148) * -(-c["nchunks"] // c["teams"]), c["groups"] * c["stages"] * c["teams"]


def test_long_chunks_leave_an_integer_branch_its_ring(cut):
    """A cut that is taken for its longer chunks alone has no ring of two large chunks, and it gives up a ring that would hold the whole
    tile (so that X is streamed twice) only for chunks that K fills, or where the factors are wide and K is long."""
    for rn, M, nst in itertools.product(range(16, 129, 16), (1, 1000, 4096, 8192, 16384, 17600, 32768), range(8, 65)):
        c = cut(INT, M, nst, rn)
        equal = [a for g, s in itertools.product(range(1, 9), range(1, 5)) if (a := cut(INT, M, nst, rn, 1, g, s))["groups"] == c["groups"]
                 and a["stages"] == s < c["stages"] and _rounds(INT, a) == _rounds(INT, c)]
        if c["stages"] <= 4 and equal:
            assert c["xslots"] >= 3 or c["groups"] <= 4, (rn, M, nst, c)
            if c["refetch"] and not all(a["refetch"] for a in equal):
                assert c["stages"] > 2 or nst % 2 == 0 or (rn > 48 and nst >= 12), (rn, M, nst, c)


# (branch kind, rows, stages of K, columns of the first factor) -> row groups and stages of the cut timed as the fastest there
TIMED = [((INT, 8192, 11, 32), (7, 1)), ((INT, 32768, 11, 32), (7, 1)), ((INT, 32768, 12, 64), (7, 2)), ((INT, 8192, 9, 96), (7, 1)), ((INT, 17600, 10, 128), (5, 1)),
         ((INT, 17600, 13, 128), (5, 1)), ((INT, 1365, 44, 32), (2, 7)), ((INT, 2048, 8, 48), (2, 4)), ((INT, 4096, 18, 48), (4, 3)), ((INT, 3000, 13, 128), (3, 4)),
         ((INT, 17600, 7, 32), (5, 1)), ((INT, 17600, 5, 32), (5, 1)), ((INT, 26000, 7, 96), (6, 1)), ((INT, 17600, 3, 128), (8, 1)),
         ((MXFP, 8192, 9, 64), (7, 1)), ((MXFP, 7000, 11, 32), (6, 1)), ((MXFP, 16384, 9, 64), (7, 2)),
         ((NONE, 22000, 9, 16), (5, 1)), ((NONE, 17600, 8, 16), (5, 1)), ((NONE, 26000, 12, 16), (5, 1))]


@pytest.mark.parametrize("size,best", TIMED)
def test_cuts_that_were_timed_as_the_fastest(cut, size, best):
    c = cut(*size)
    assert (c["groups"], c["stages"]) == best


@pytest.mark.parametrize("br,rn,planes,M,K,first", [
    (INT, 32, 1, 8192, 1152, False), (INT, 32, 1, 16384, 1152, False), (INT, 32, 1, 32768, 1152, True), (INT, 32, 1, 8192, 4608, False),
    (MXFP, 64, 1, 8192, 1152, False), (MXFP, 64, 1, 4096, 4608, False), (MXFP, 64, 1, 8192, 4608, True), (MXFP, 64, 1, 32768, 4608, False),
    (MXINT, 64, 2, 8192, 4608, False)])
def test_x_leaves_the_l2_first_only_where_it_would_not_stay(cut, br, rn, planes, M, K, first):
    """What another layer or a residual sum may read again is not marked as read for the last time where the L2 could keep it."""
    assert cut.leaves_first(cut(br, M, -(-K // 128), rn), M, K, planes) == first
