"""Host-side test of the team apply's index maps (csrc/team_map.h): the header is
compiled for the host and its partitions, tiles, slots and index sets are checked
over sizes and rank counts that a test on a GPU does not reach.  No GPU is needed.

What the kernel relies on:
  * a rank's row groups are disjoint and cover the operator; every rank owns a
    part of every input (a slot is written again when its owner has seen parts of
    later inputs from every rank);
  * a column of a slab has the same owner in every rect that spans the slab's
    window (the coupling a row feeds stays in its rank, its line's values too);
  * stored tiles are disjoint and fill the operator;
  * the index sets hold what the sweep's next right-hand sides read;
  * an input's slot is not used again for the next two inputs of its team.
"""
import os
import shutil
import subprocess
import tempfile

import pytest

from oracle.operator import Grid
from oracle.sweep import axis_schedule, axis_window
from paper_1502_07266_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1502_07266_gb300", "csrc")

DRIVER = r'''
#define __host__
#define __device__
#define __forceinline__ inline
#include <cstddef>
#include <cstdio>
#include <vector>
struct AxisWin { int lo, L, ia, ib; int moving, moving_hi; };
struct DRect { int line0, nl, z0, nz; };
namespace {
#include "dense_sched.h"
#include "team_map.h"
}
static void part(char t, int n, int nl, int full, int C) {
    printf("%c", t);
    for (int r = 0; r < C; ++r) {
        int lo, hi;
        tm_part(n, nl, full, r, C, &lo, &hi);
        printf(" %d %d", lo, hi);
    }
    printf("\n");
}
int main() {
    int N, B, cen, two, C;
    if (scanf("%d %d %d %d %d", &N, &B, &cen, &two, &C) != 5) return 1;
    std::vector<AxisWin> win(B);
    for (AxisWin& w : win)
        if (scanf("%d %d %d %d", &w.lo, &w.L, &w.ia, &w.ib) != 4) return 1;
    for (int team = 0; team <= two; ++team) {
        const int ns = tm_solves(B, cen, team);
        for (int i = 0; i < ns; ++i) {
            const TeamSolve t = tm_solve(i, B, cen, team);
            printf("V %d %d %d %d %d %d\n", team, i, t.Mp, t.bwd, t.role, slot_of_solve(i, ns, cen, team));
        }
    }
    for (int M = 0; M < B; ++M)
        for (int Mp = 0; Mp < B; ++Mp)
            for (int bwd = 0; bwd < 2; ++bwd) {
                if (!two && Mp == B - 1 && bwd) continue;
                const SolveGeo g = tm_geo(win[M], win[Mp], N, Mp, bwd, B, two);
                printf("G %d %d %d %d %d %d %d %d %d %d %d", M, Mp, bwd, g.nrect, g.fin, g.f0, g.f1, g.K, g.n0, g.n1, g.boundary);
                const DRect* R[3] = {&g.in, &g.out0, &g.out1};
                for (const DRect* q : R) printf(" %d %d %d %d", q->line0, q->nl, q->z0, q->nz);
                printf("\n");
                part('I', g.K, g.in.nl, g.fin, C);
                part('O', g.n0, g.out0.nl, g.f0, C);
                if (g.nrect > 1) part('P', g.n1, g.out1.nl, g.f1, C);
            }
    // stored tiles of a few shapes: every byte once
    for (int halves = 1; halves <= 2; ++halves)
        for (int K : {1, 16, 17, 63, 64, 65, 130, 417})
            for (int ng : {1, 3, 40}) {
                const int KP = tm_kp(K);
                std::vector<int> hit(tm_bytes(ng, KP, halves), 0);
                bool in = true;
                for (int c = 0; c * TKC < KP; ++c)
                    for (int h = 0; h < halves; ++h)
                        for (int gr = 0; gr < ng; ++gr) {
                            int bytes;
                            const size_t o = tm_tile(c, h, gr, ng, KP, halves, &bytes);
                            for (int q = 0; q < bytes; ++q)
                                if (o + q < hit.size()) ++hit[o + q]; else in = false;
                        }
                bool once = in;
                for (int v : hit) once = once && v == 1;
                printf("T %d %d %d %d\n", halves, K, ng, once);
            }
    // the same where some groups have lo parts: units
    for (int K : {16, 64, 65, 417})
        for (int units : {2, 45}) {
            const int KP = tm_kp(K);
            std::vector<int> hit((size_t)units * KP * 32, 0);
            bool once = true;
            for (int c = 0; c * TKC < KP; ++c)
                for (int u = 0; u < units; ++u) {
                    const int kc = KP - c * TKC < TKC ? KP - c * TKC : TKC;
                    const size_t o = tm_unit(c, u, units, KP);
                    for (int q = 0; q < 32 * kc; ++q)
                        if (o + q < hit.size()) ++hit[o + q]; else once = false;
                }
            for (int v : hit) once = once && v == 1;
            printf("T 0 %d %d %d\n", K, units, once);
        }
    return 0;
}
'''


@pytest.fixture(scope="module")
def driver():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tempfile.mkdtemp()
    src = os.path.join(d, "map.cpp")
    open(src, "w").write(DRIVER)
    exe = os.path.join(d, "map")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, src, "-o", exe], check=True)
    yield exe
    shutil.rmtree(d, ignore_errors=True)


def _ceil(a, b):
    return -(-a // b)


def _entries(rect, N):
    """Entries (line, z row) of a rect; every x belongs to it."""
    l0, nl, z0, nz = rect
    return {(line, z) for line in range(l0, l0 + nl) for z in range(z0, z0 + nz)}


CASES = [(4, 2, 1, 2, "two_front"), (9, 3, 1, 1, "two_front"), (16, 4, 2, 2, "two_front"), (15, 4, 3, 2, "two_front"),
         (31, 6, 1, 4, "one_front"), (22, 5, 2, 6, "one_front"), (10, 2, 1, 3, "one_front"), (63, 6, 1, 2, "two_front"),
         (30, 8, 2, 1, "two_front"), (13, 1, 1, 1, "one_front")]


@pytest.mark.parametrize("n,b,d,b_aux,schedule", CASES)
@pytest.mark.parametrize("share", [1, 3, 1000])
def test_maps(driver, n, b, d, b_aux, schedule, share):
    grid = Grid(n, b, W.omega_for(n))
    N, two = grid.N, schedule == "two_front"
    blocks, roles, cen = axis_schedule(N, b, d, schedule)
    B = len(blocks)
    win = []
    for M in range(B):
        lo = blocks[M][0] - axis_window(grid, blocks, M, b_aux, roles[M])[1][0]
        prof, (ia, ib) = axis_window(grid, blocks, M, b_aux, roles[M])
        hi = blocks[M][1] + (b_aux if roles[M] in ("U", "C") and blocks[M][1] < N else 0)
        win.append((lo, min(hi, N) - lo, ia, ib))

    def run(C):
        text = "%d %d %d %d %d\n" % (N, B, cen, two, C) + "".join("%d %d %d %d\n" % w for w in win)
        out = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout
        return [(line[0], list(map(int, line.split()[1:]))) for line in out.splitlines()]

    # the fewest groups (of columns, where a rect spans the window) an input or such a rect has bound the ranks
    gmin = 10 ** 9
    for t, v in run(1):
        if t == "G":
            nrect, fin, f0, f1, K, n0, n1 = v[3:10]
            rin, r0, r1 = v[11:15], v[15:19], v[19:23]
            gmin = min(gmin, _ceil(K // rin[1], 8) if fin else _ceil(K, 8))
            gmin = min([gmin] + [_ceil(m // r[1], 8) for m, r, f in ((n0, r0, f0), (n1, r1, f1)) if f])
    C = max(1, min(gmin, 152, gmin // share if share < 1000 else 1))
    recs = run(C)

    # solves of the teams: every solve of the visit once, in the sweep's order; slots
    order = [(M, 0) for M in list(range(cen)) + list(range(B - 1, cen, -1)) + [cen]]
    order += [(M, 1) for M in list(range(cen - 1, -1, -1)) + list(range(cen + 1, B))]
    for team in range(2 if two else 1):
        mine = [v for t, v in recs if t == "V" and v[0] == team]
        want = [s for s in order if (s[0] > cen) == (team == 1)]
        if team == 0:
            want = [s for s in want if s[1] == 0] + [s for s in want if s[1] == 1]
        assert [(v[2], v[3]) for v in mine] == want
        slots = [v[5] for v in mine]
        for i, s in enumerate(slots):
            assert s not in slots[i + 1:i + 3]
    # index sets and ownership
    owner = {}
    for q, (t, v) in enumerate(recs):
        if t != "G":
            continue
        M, Mp, bwd, nrect, fin, f0, f1, K, n0, n1, boundary = v[:11]
        rin, r0, r1 = v[11:15], v[15:19], v[19:23]
        L, za, zb = win[M][1], win[M][2], win[M][3]
        y0, y1 = blocks[Mp]
        top = two and Mp == B - 1
        own = {(y, z) for y in range(y0, y1) for z in range(za, zb)}
        e_in, e_out = _entries(rin, N), _entries(r0, N) | (_entries(r1, N) if nrect > 1 else set())
        cl = y0 if top else y1 - 1
        line = {(cl, z) for z in range(L)}
        assert K == N * len(e_in) and n0 + n1 == N * len(e_out)
        assert all(y0 <= y < y1 and 0 <= z < L for y, z in e_in | e_out)
        # the right-hand side: the slab's own layers forward, the neighbour's coupling on the line next to it
        if not bwd:
            assert own <= e_in
        if not (boundary and not bwd):
            first = {(y0, z) for z in range(L)} if (roles[Mp] != "U") != bool(bwd) else {(y1 - 1, z) for z in range(L)}
            assert (line if boundary else first) <= e_in
        # the result: own layers, and forward the line that feeds the next block
        assert own <= e_out
        if not bwd:
            assert line <= e_out or not boundary
        parts = {}
        k = q + 1
        while k < len(recs) and recs[k][0] in "IOP":
            parts[recs[k][0]] = list(zip(recs[k][1][::2], recs[k][1][1::2]))
            k += 1
        for name, n_, rect, full in (("I", K, rin, fin), ("O", n0, r0, f0), ("P", n1, r1, f1)):
            if name not in parts:
                continue
            p = parts[name]
            assert p[0][0] == 0 and p[-1][1] == _ceil(n_, 8)
            assert all(a[1] == c[0] and a[0] <= a[1] for a, c in zip(p, p[1:]))
            if name == "I":
                assert all(lo < hi for lo, hi in p)
            if full:
                # column e = x L + z of the slab: one owner in all its operators
                for r, (lo, hi) in enumerate(p):
                    assert lo % rect[1] == 0
                    cols = (8 * lo // rect[1], min(N * L, 8 * hi // rect[1]) if r + 1 < len(p) else N * L)
                    assert owner.setdefault((M, r), cols) == cols
    assert all(v[3] for t, v in recs if t == "T")
