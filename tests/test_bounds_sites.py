"""The index checks of the debug build in the source: one site code per check,
and a check for every computed index by which the cell grid's kernels (the
default path) read or write."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_10000_gb300", "csrc")

# what is indexed -> (check, access), each a pattern of the source; the check
# stands before the access, within the lines of one statement or branch
GRID = {
    "cell word": (r"c < g\.n\[0\] \* g\.n\[1\] \* g\.n\[2\], a\.status", r"__ldg\(g\.words \+ c\)"),
    "cell block": (r"kOffsetMask\) \+ 1u.*?a\.status", r"return w;"),
    "chunks of a block": (r"chunks <= kMaxList / kSub, a\.status", r"b < chunks"),
    "triangle of an entry": (r"t < a\.comps\[g\.comp\]\.tri_cnt, a\.status", r"g\.tris\[3 \* t \+ k\]"),
    "node, walk of a warp": (r"i < a\.n_nodes, a\.status", r"a\.nodes\[i\]"),
    "group, walk of a warp": (r"pos \+ 4 <= a\.n_cseg, a\.status", r"group64\(a\.cseg, pos"),
    "node, walk of a block": (r"o0\.x < a\.n_nodes, a\.status", r"a\.nodes\[o0\.x\]"),
    "field cell": (r"at < a\.field\.n\[0\] \* a\.field\.n\[1\] \* a\.field\.n\[2\], a\.status", r"a\.field\.cells\) \+ at"),
    "queue of the fused kernel": (r"at < kGlQueue, a\.status", r"s_q\[wid\]\[at\] = p;"),
    "queue of the streaming kernel": (r"at < kGsQueue, a\.status", r"s_q\[wid\]\[at\] = \(int32_t\)"),
    "list of open points": (r"at \+ j < \(unsigned long long\)a\.pend_cap, a\.status", r"a\.pending\[at \+ j\] ="),
    "listed point": (r"i >= 0 && i < \(a\.n_host >= 0 \? a\.n_host : a\.counters\[CNT_N\]\), a\.status", r"a\.pts \+ 3 \* \(off \+ i\)"),
    "point on a surface": (r"p\.i < n, a\.status", r"M mask = \(M\)p\.ins"),
}


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_every_site_code_names_one_check():
    seen = {}
    for f in sorted(os.listdir(CSRC)):
        for code in re.findall(r"status, (\d+)\)", _source(f)) if f.endswith((".cu", ".cuh")) else []:
            assert code not in seen, (code, seen[code], f)
            seen[code] = f
    assert len(seen) > 20


def test_grid_kernels_check_their_indices():
    src = _source("zef_grid.cu")
    for what, (check, access) in GRID.items():
        m = re.search(r"ZEF_BOUNDS_OK\([^;]*?" + check, src, re.S)
        assert m, f"no check: {what}"
        a = re.search(access, src[m.start():], re.S)
        assert a and src[m.start():m.start() + a.start()].count("\n") <= 10, f"the check does not stand by the access: {what}"
