// Index maps of the team apply (team.cu): which rows and inputs of a restricted
// operator a rank of a team owns, how both are numbered, and which solve a step
// of a team carries.  Plain integer code, shared by the kernels, the setup and a
// host-side test; included after dense_sched.h inside an anonymous namespace.
#pragma once

// A rect (lines x window z rows x every x) is numbered with the line fastest,
// then the z row, then x: i = (x nz + zr) nl + l, in groups of 8 entries.  A rect
// that spans every z row of the slab window is "full": its entry i belongs to
// column e = x Lz + lz (e = i / nl), and a column belongs to the same rank in
// every operator of the slab, so that the coupling a row feeds lands in the
// rank's own part of the next input.  Other rects (own layers only) are split
// evenly; what crosses ranks there is read after a barrier.
__host__ __device__ __forceinline__ int tm_ceil(int a, int b) { return (a + b - 1) / b; }

// 8-entry groups [lo, hi) of a rect with n entries on nl lines that rank r of C
// owns; every rank owns at least one when there are C or more of them.
__host__ __device__ __forceinline__ void tm_part(int n, int nl, int full, int r, int C, int* lo, int* hi) {
    const int ng = tm_ceil(n, 8);
    if (full) {
        const int cg = tm_ceil(n / nl, 8);           // groups of 8 columns
        *lo = nl * (r * cg / C);
        *hi = nl * ((r + 1) * cg / C);
        if (*lo > ng) *lo = ng;
        if (*hi > ng) *hi = ng;
    } else {
        *lo = r * ng / C;
        *hi = (r + 1) * ng / C;
    }
}

// Solves of one slab visit for a team: with one front (or the lower front, which
// also takes the centre) blocks 0 .. c-1 forward, the centre c, then c-1 .. 0
// backward; the upper front's team B-1 .. c+1 forward, then c+1 .. B-1 backward.
__host__ __device__ __forceinline__ int tm_solves(int B, int c, int upper) {
    return upper ? 2 * (B - 1 - c) : 2 * c + 1;
}
struct TeamSolve {
    int Mp, bwd, role;
};
__host__ __device__ __forceinline__ TeamSolve tm_solve(int i, int B, int c, int upper) {
    TeamSolve t;
    if (upper) {
        const int U = B - 1 - c;
        t.bwd = i >= U;
        t.Mp = t.bwd ? c + 1 + (i - U) : B - 1 - i;
        t.role = ROLE_U;
        return t;
    }
    t.bwd = i > c;
    t.Mp = i <= c ? i : 2 * c - i;
    t.role = i == c ? ROLE_C : ROLE_L;
    return t;
}

// Slots of published inputs: a ring for the solves of a visit, one each for the
// centre, the last solve and the first.  A slot's next input comes at least two
// solves later, when every rank has read the one before.
constexpr int NRING = 4, SLOT_CENTRE = NRING, SLOT_END = NRING + 1, SLOT_START = NRING + 2;
__host__ __device__ __forceinline__ int slot_of_solve(int i, int nsol, int cen, int upper) {
    if (i == 0) return SLOT_START;
    if (i == nsol - 1) return SLOT_END;
    if (upper) return (i - 1) & (NRING - 1);
    if (i == cen) return SLOT_CENTRE;
    return (i < cen ? i - 1 : i - 2) & (NRING - 1);
}
// Index sets of solve (slab window wz, line block window wy) of a team.  A
// boundary line block (0, and B-1 with two fronts) takes its own entries forward
// and feeds the one line next to its neighbour; backward it takes that line.
// Every other block maps its lines x every z row to themselves.
struct SolveGeo {
    DRect in, out0, out1;
    int nrect;
    int fin, f0, f1;      // full rects
    int K, n0, n1;        // input entries, output entries of each rect
    int boundary;
};
__host__ __device__ __forceinline__ SolveGeo tm_geo(const AxisWin& wz, const AxisWin& wy, int N, int Mp, int bwd,
                                                    int B, int two) {
    SolveGeo g;
    const int Lz = wz.L, za = wz.ia, dz = wz.ib - wz.ia;
    const int y0 = wy.lo + wy.ia, y1 = wy.lo + wy.ib, nl = y1 - y0;
    const int top = two && Mp == B - 1;
    g.boundary = Mp == 0 || top;
    g.nrect = 1;
    g.out1 = DRect{0, 0, 0, 0};
    if (g.boundary) {
        const int cl = top ? y0 : y1 - 1;             // the line next to the neighbour
        if (!bwd) {
            g.in = DRect{y0, nl, za, dz};
            const DRect line = DRect{cl, 1, 0, Lz};
            const DRect rest = DRect{top ? y0 + 1 : y0, nl - 1, za, dz};
            if (nl == 1) {
                g.out0 = line;
            } else {
                g.nrect = 2;
                g.out0 = top ? line : rest;
                g.out1 = top ? rest : line;
            }
        } else {
            g.in = DRect{cl, 1, 0, Lz};
            g.out0 = DRect{y0, nl, za, dz};
        }
    } else {
        g.in = g.out0 = DRect{y0, nl, 0, Lz};
    }
    g.fin = g.in.nz == Lz;
    g.f0 = g.out0.nz == Lz;
    g.f1 = g.nrect > 1 && g.out1.nz == Lz;
    g.K = g.in.nl * g.in.nz * N;
    g.n0 = g.out0.nl * g.out0.nz * N;
    g.n1 = g.nrect > 1 ? g.out1.nl * g.out1.nz * N : 0;
    return g;
}

// Stored tiles of one operator (FP16 forms): chunks of TKC input columns; in a
// chunk of kc columns every row group (8 complex rows) in turn: the hi parts of its
// 8 real and of its 8 imaginary parts, then their lo parts, each 8 rows x kc in
// K-major core matrices of 8 x 16 bytes.  A rank's groups are contiguous, so a chunk
// of them is one copy.
constexpr int TKC = 64;
__host__ __device__ __forceinline__ int tm_kp(int K) { return 16 * tm_ceil(K, 16); }
// byte offset of (chunk c, part h, group gr) and its size per group
__host__ __device__ __forceinline__ size_t tm_tile(int c, int h, int gr, int ng, int KP, int halves, int* bytes) {
    const int kc = KP - c * TKC < TKC ? KP - c * TKC : TKC;
    *bytes = 2 * kc * 16;
    return ((size_t)c * TKC * halves * ng + (size_t)kc * (gr * halves + h)) * 32;
}
// The same where only some groups have lo parts (nlo of them): a chunk holds units of
// (16 real rows) x kc, the hi parts of all ng groups, then the lo parts there are.
__host__ __device__ __forceinline__ size_t tm_unit(int c, int unit, int units, int KP) {
    const int kc = KP - c * TKC < TKC ? KP - c * TKC : TKC;
    return ((size_t)c * TKC * units + (size_t)kc * unit) * 32;
}
__host__ __device__ __forceinline__ size_t tm_bytes(int ng, int KP, int halves) {
    return (size_t)ng * KP * halves * 32;
}
