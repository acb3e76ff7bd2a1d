// Dense restricted-operator form of the recursive sweep.
//
// Section 6 notes that the quasi-1D solves of Algorithm 4 are the sequential
// bottleneck and can be restructured.  Every use of |T~_{M'}| in Algorithms 4
// and 6 maps the values on a few lines of the quasi-1D window to values on a
// few lines: |T~| = R_out H~^{-1} R_in^T.  This form stores that map densely
// (G, about 973 x 973 complex entries per problem at n = 127, b = 6, d = 1) and
// replaces each 2 N-step block substitution by one complex matrix product over
// all right-hand sides: the same preconditioner M up to rounding.
//
// Index sets (in the window of problem (M, M'); see DProb):
//   M' >= 1   in = out = the block's lines x every z row of the window.
//   M' = 0    forward:  in  = lines [0, b) x the slab's own layers [za, zb)
//                       out = lines [0, b-1) x [za, zb)  and  line b-1 x every z row
//             backward: in  = line b-1 x every z row
//                       out = lines [0, b) x [za, zb)
// (the first line block is only ever fed on its own layers, its backward input
// is the coupling into line b-1, and only the slab's own layers and the line
// that couples to M' = 1 are read from it).
//
// Setup: the quasi-1D problems are factored chunk by chunk (the twisted block
// LDU of factor.cu into a temporary buffer), k_dense_G solves with the unit
// columns of R_in^T and keeps the rows of R_out, and k_dense_pack stores G in
// the FP32 apply's tiles.  The tensor-core forms (FP16 hi + lo parts, or hi) pack and
// apply it in team.cu.
//
// FP32 apply: one persistent launch of clusters of 8 CTAs walks the (2B-1)^2 solves
// of Algorithm 6 over Algorithm 4 in order (dense_sched.h: with two fronts a
// step carries a lower-front and an upper-front solve on two groups of
// clusters).  A solve computes Y = G q for up to 64 right-hand sides: cluster c
// of its group takes 64-row output tiles c, c + ncl, ...; rank r of the cluster
// takes input entries [r KR, (r+1) KR).  Each CTA gathers its slice of q
// straight from the slab vector and the outer vectors (the couplings of
// Algorithms 4 and 6), multiplies it by its G tile (streamed by one thread
// through a shared-memory ring with bulk copies), the 8 partial products are
// summed through distributed shared memory, and the owner of each output row
// applies the step's update (store, subtract, restrict to the output).  Step
// s+1 starts when every CTA has arrived on a global counter for step s.  All waits are
// bounded by a clock limit; on expiry the kernel sets the error word, drains its copies
// and returns.
#include "helm_internal.h"
#include "ptx.cuh"

#include <cuda_fp16.h>
#include <string.h>

#include <algorithm>
#include <vector>

namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ void cfma(float2& acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// y - c v, the coupling step of the substitutions, with every rounding written out:
// left to the compiler it contracts to other multiply-adds in k_dense_G than in
// k_dense_G_cols, and operators that differ in their last bit differ by a whole
// FP16 step here and there once they are rounded to FP16.  FIRST says which product
// of the real part is rounded before the other is added to it.
enum { FIRST_YY = 0, FIRST_XX = 1 };
__device__ __forceinline__ float2 sub_coupled(float2 y, float2 c, float2 v, int first) {
    const float re = first == FIRST_XX ? __fmaf_rn(-c.y, v.y, __fmul_rn(c.x, v.x))
                                       : __fmaf_rn(c.x, v.x, -__fmul_rn(c.y, v.y));
    const float im = __fmaf_rn(c.y, v.x, __fmul_rn(c.x, v.y));
    return make_float2(__fsub_rn(y.x, re), __fsub_rn(y.y, im));
}

int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Bytes per K column of the main part of one stored tile (FP32 form): 64 complex
// rows.  A tile also carries xr extra complex rows (8 bytes per row and K column).
constexpr int TILE_UNIT = 512;

#include "dense_sched.h"

// ============================================================== setup ========

constexpr int GW = 64;      // input columns per setup work item
constexpr int GT = 128;     // threads of k_dense_G
constexpr int TLD = 68;     // row stride (complex) of the transposed factor block in shared memory

struct GItem { int p, j0; };

// T_i of the chunk's factors as a pointer (row-major, row stride ldk, complex FP32).
__device__ __forceinline__ const float2* fac_block(const float2* fac, const Prob& P, long long off0, int i) {
    return fac + (P.off - off0 + (long long)i * P.kstride);
}

// acc[8 rows][4 columns] = T W over the block's k columns; this thread's rows
// are 2 rg + 16 ii + e (ii < 4, e < 2), its columns 4 cg + cc.
__device__ __forceinline__ void setup_product(const float2* __restrict__ Tt, const float2* __restrict__ W, int k,
                                              int rg, int cg, float2 (&acc)[8][4]) {
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) acc[q][cc] = make_float2(0.f, 0.f);
    for (int kk = 0; kk < k; ++kk) {
        const float4* tr = reinterpret_cast<const float4*>(Tt + kk * TLD + 2 * rg);
        const float4* wr = reinterpret_cast<const float4*>(W + kk * GW + 4 * cg);
        float2 a[8], b[4];
#pragma unroll
        for (int ii = 0; ii < 4; ++ii) {
            const float4 v = tr[8 * ii];              // rows 2rg + 16 ii, +1
            a[2 * ii] = make_float2(v.x, v.y);
            a[2 * ii + 1] = make_float2(v.z, v.w);
        }
        const float4 w0 = wr[0], w1 = wr[1];
        b[0] = make_float2(w0.x, w0.y);
        b[1] = make_float2(w0.z, w0.w);
        b[2] = make_float2(w1.x, w1.y);
        b[3] = make_float2(w1.z, w1.w);
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) cfma(acc[q][cc], a[q], b[cc]);
    }
}

__device__ __forceinline__ int setup_row(int rg, int q) { return 2 * rg + 16 * (q >> 1) + (q & 1); }

// One work item = operator p, input columns [j0, j0 + GW).  X = H~^{-1} E with
// E the unit columns, by the twisted substitution of the factor layout
// (left chain T_0..T_{m-1}, right chain T_{N-1}..T_{m+1}, middle T_m):
//   left   y_i = T_i (e_i - cdn(i) y_{i-1})       from the first column's x up to m-1
//   right  y_i = T_i (e_i - cup(i) y_{i+1})       from the last column's x down to m+1
//   middle x_m = T_m (e_m - cdn(m) y_{m-1} - cup(m) y_{m+1})
//   back   x_i = y_i - cup(i) T_i x_{i+1}  (i < m),   x_i = y_i - cdn(i) T_i x_{i-1}  (i > m)
// (y is zero below the first column's x on the left and above the last
// column's x on the right).  Row a of x_i is written to G row so[a] + i.
__global__ void __launch_bounds__(GT)
k_dense_G(Geom g, Tables t, const DProb* __restrict__ dp, const GItem* __restrict__ items, int nitems,
          const float2* __restrict__ fac, long long off0, float2* __restrict__ Gt,
          const long long* __restrict__ goff, float2* __restrict__ yscr, size_t yslot) {
    extern __shared__ __align__(16) float2 gsm[];
    float2* Tt = gsm;                      // [64][TLD]: Tt[c][r] = T_i[r][c]
    float2* W = Tt + 64 * TLD;             // [64][GW]   product input
    float2* Xm = W + 64 * GW;              // [64][GW]   x_m for the second back pass
    int* sa = reinterpret_cast<int*>(Xm + 64 * GW);   // [GW] block row of column jj's unit entry
    int* sx = sa + GW;                     // [GW] x of column jj (-1: no column)
    int* so = sx + GW;                     // [64] output row of block row a at x = 0 (-1: not an output)
    const int tid = threadIdx.x;
    const int rg = tid & 7, cg = tid >> 3;
    const int N = g.N, m = (N - 1) / 2;
    float2* Y = yscr + (size_t)blockIdx.x * yslot;    // [N][64][GW] forward values

    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const GItem I = items[it];
        const DProb D = dp[I.p];
        const Prob P = t.prob[D.fp];
        const int k = P.k, Lz = P.Lz;
        float2* Gp = Gt + goff[I.p];
        __syncthreads();                   // previous item done with the shared arrays
        int xa = N, xb = -1;
        for (int jj = tid; jj < GW; jj += GT) {
            const int j = I.j0 + jj;
            int a = -1, x = -1;
            if (j < D.n_in) {
                const int per = D.in.nz * D.in.nl;
                x = j / per;
                const int r = j - x * per, l = r / D.in.nz;
                const int lz = D.in.z0 + (r - l * D.in.nz), line = D.in.line0 + l;
                a = lz + Lz * (line - P.ylo);
            }
            sa[jj] = a;
            sx[jj] = x;
        }
        for (int a = tid; a < 64; a += GT) {
            int o = -1;
            if (a < k) {
                const int lz = a % Lz, line = P.ylo + a / Lz;
                int base = 0;
                for (int q = 0; q < D.nrect; ++q) {
                    const DRect R = D.out[q];
                    if (line >= R.line0 && line < R.line0 + R.nl && lz >= R.z0 && lz < R.z0 + R.nz)
                        o = base + N * ((lz - R.z0) + R.nz * (line - R.line0));
                    base += R.nl * R.nz * N;
                }
            }
            so[a] = o;
        }
        for (int e = tid; e < 64 * TLD; e += GT) Tt[e] = make_float2(0.f, 0.f);
        __syncthreads();
        // first and last x of the item's columns (columns are in x order)
        xa = sx[0];
        {
            int last = GW - 1;
            while (last > 0 && sx[last] < 0) --last;
            xb = sx[last];
        }
        const bool do_left = xa < m, do_right = xb > m;
        const int jn = min(GW, D.n_in - I.j0);
        const int c0 = 4 * cg;

        // the step list: left forward, right forward, middle, back left, back right
        const int nlf = do_left ? m - xa : 0;
        const int nrf = do_right ? xb - m : 0;
        const int nsteps = nlf + nrf + 1 + m + (N - 1 - m);
        auto step_x = [&](int q) -> int {
            if (q < nlf) return xa + q;
            q -= nlf;
            if (q < nrf) return xb - q;
            q -= nrf;
            if (q == 0) return m;
            q -= 1;
            if (q < m) return m - 1 - q;
            return m + 1 + (q - m);
        };
        auto has_y = [&](int i) -> bool {
            return (i < m && do_left && i >= xa) || (i > m && do_right && i <= xb);
        };
        // load T of the first step (transposed)
        {
            const float2* T0 = fac_block(fac, P, off0, step_x(0));
            for (int e = tid; e < k * k; e += GT) {
                const int r = e / k, c = e - r * k;
                Tt[c * TLD + r] = T0[(size_t)r * P.ldk + c];
            }
        }
        // the first step's input: e at block step_x(0)
        {
            const int i0 = step_x(0);
            for (int e = tid; e < 64 * GW; e += GT) {
                const int a = e / GW, jj = e - a * GW;
                W[e] = make_float2((sx[jj] == i0 && sa[jj] == a) ? 1.f : 0.f, 0.f);
            }
        }
        __syncthreads();
        for (int q = 0; q < nsteps; ++q) {
            const int i = step_x(q);
            // prefetch the next step's factor block into registers
            constexpr int PF = (64 * 64 + GT - 1) / GT;
            float2 pf[PF];
            const bool more = q + 1 < nsteps;
            if (more) {
                const float2* Tn = fac_block(fac, P, off0, step_x(q + 1));
#pragma unroll
                for (int u = 0; u < PF; ++u) {
                    const int e = tid + u * GT;
                    pf[u] = make_float2(0.f, 0.f);
                    if (e < k * k) {
                        const int r = e / k, c = e - r * k;
                        pf[u] = Tn[(size_t)r * P.ldk + c];
                    }
                }
            }
            float2 acc[8][4];
            setup_product(Tt, W, k, rg, cg, acc);
            __syncthreads();                                   // Tt and W consumed
            if (more) {
#pragma unroll
                for (int u = 0; u < PF; ++u) {
                    const int e = tid + u * GT;
                    if (e < k * k) {
                        const int r = e / k, c = e - r * k;
                        Tt[c * TLD + r] = pf[u];
                    }
                }
            }
            const int inext = more ? step_x(q + 1) : -1;
            const bool fwd = q < nlf + nrf;                     // this step produced y_i
            const bool mid = q == nlf + nrf;
            // the next step's input, row by row of this thread's tile
#pragma unroll
            for (int qq = 0; qq < 8; ++qq) {
                const int a = setup_row(rg, qq);
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const int jj = c0 + cc;
                    float2 val = acc[qq][cc];                   // T_i W
                    float2* ys = Y + ((size_t)i * 64 + a) * GW + jj;
                    if (fwd) {
                        *ys = val;                               // y_i
                    } else if (!mid) {
                        // back substitution: x_i = y_i - coupling * (T_i x_prev)
                        const float2 cp = (i < m) ? t.c_up[i] : t.c_dn[i];
                        const float2 yv = has_y(i) ? *ys : make_float2(0.f, 0.f);
                        val = sub_coupled(yv, cp, val, !has_y(i) && i < m ? FIRST_XX : FIRST_YY);
                    }
                    if (!fwd) {                                  // val = x_i: output rows
                        if (mid) Xm[a * GW + jj] = val;
                        const int o = so[a];
                        if (o >= 0 && jj < jn) Gp[(size_t)(o + i) * D.n_in + I.j0 + jj] = val;
                    }
                    acc[qq][cc] = val;
                }
            }
            if (more) {
                // W for step q+1
                const bool nfwd = q + 1 < nlf + nrf, nmid = q + 1 == nlf + nrf;
#pragma unroll
                for (int qq = 0; qq < 8; ++qq) {
                    const int a = setup_row(rg, qq);
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        const int jj = c0 + cc;
                        const float2 e = make_float2((sx[jj] == inext && sa[jj] == a) ? 1.f : 0.f, 0.f);
                        float2 w;
                        if (nfwd) {
                            const bool first = (q + 1 == 0) || (q + 1 == nlf);   // a chain starts at its end block
                            if (first) {
                                w = e;
                            } else {
                                const float2 cp = (inext < m) ? t.c_dn[inext] : t.c_up[inext];
                                w = sub_coupled(e, cp, acc[qq][cc], FIRST_XX);
                            }
                        } else if (nmid) {
                            w = e;
                            if (do_left) w = sub_coupled(w, t.c_dn[m], Y[((size_t)(m - 1) * 64 + a) * GW + jj], FIRST_XX);
                            if (do_right) w = sub_coupled(w, t.c_up[m], Y[((size_t)(m + 1) * 64 + a) * GW + jj], FIRST_XX);
                        } else if (inext == m + 1) {
                            w = Xm[a * GW + jj];                 // the right back pass starts from x_m
                        } else {
                            w = acc[qq][cc];                     // x of the previous block
                        }
                        W[a * GW + jj] = w;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// The same for blocks of k <= KM: one thread per column.  With 64-row tiles a block
// of 9 leaves six of seven rows and most of the scratch traffic to padding.  Here a
// column's product input stays in its thread's shared slot and its k results in
// registers, the factor block is read by broadcast (KM / 2 16-byte loads for 4 KM
// fused multiply-adds), the columns share nothing else, and one barrier a step hands
// over the next factor block.  The sums run in k_dense_G's order and round as there:
// the same bits.
// Setup at n = 95, two fronts, b_aux = 2 (blocks of 9 to 25): 479 -> 173 ms.  What bounds it
// then is the steps' chain of dependent shared-memory products; the operator entries' way
// to memory and back (19.8 GB, 2.9 ms each) is 3 % of it.
template <int KM>
__global__ void __launch_bounds__(GW)
k_dense_G_cols(Geom g, Tables t, const DProb* __restrict__ dp, const GItem* __restrict__ items, int nitems,
               const float2* __restrict__ fac, long long off0, float2* __restrict__ Gt,
               const long long* __restrict__ goff, float2* __restrict__ yscr, size_t yslot) {
    __shared__ __align__(16) float2 Tt[2][KM * KM];   // [c][r]: two steps' factor blocks, transposed
    __shared__ float2 W[KM][GW];                       // product input
    __shared__ int so[KM], s_x[2];
    const int jj = threadIdx.x;
    const int N = g.N, m = (N - 1) / 2;
    float2* Y = yscr + (size_t)blockIdx.x * yslot + jj;    // [N][KM][GW] forward values; x_m at block m

    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const GItem I = items[it];
        const DProb D = dp[I.p];
        const Prob P = t.prob[D.fp];
        const int k = P.k, Lz = P.Lz;
        float2* Gp = Gt + goff[I.p];
        const int jn = min(GW, D.n_in - I.j0);
        int sa = -1, sx = -1;              // block row and x of the column's unit entry (-1: no column)
        if (jj < jn) {
            const int j = I.j0 + jj, per = D.in.nz * D.in.nl;
            sx = j / per;
            const int r = j - sx * per, l = r / D.in.nz;
            sa = D.in.z0 + (r - l * D.in.nz) + Lz * (D.in.line0 + l - P.ylo);
        }
        __syncthreads();                   // previous item done with the shared arrays
        if (jj == 0) s_x[0] = sx;
        if (jj == jn - 1) s_x[1] = sx;
        for (int a = jj; a < k; a += GW) {
            const int lz = a % Lz, line = P.ylo + a / Lz;
            int o = -1, base = 0;
            for (int q = 0; q < D.nrect; ++q) {
                const DRect R = D.out[q];
                if (line >= R.line0 && line < R.line0 + R.nl && lz >= R.z0 && lz < R.z0 + R.nz)
                    o = base + N * ((lz - R.z0) + R.nz * (line - R.line0));
                base += R.nl * R.nz * N;
            }
            so[a] = o;
        }
        __syncthreads();
        const int xa = s_x[0], xb = s_x[1];
        const bool do_left = xa < m, do_right = xb > m;
        const int nlf = do_left ? m - xa : 0, nrf = do_right ? xb - m : 0;
        const int nsteps = nlf + nrf + N;
        auto step_x = [&](int q) -> int {
            if (q < nlf) return xa + q;
            q -= nlf;
            if (q < nrf) return xb - q;
            q -= nrf;
            if (q == 0) return m;
            return q <= m ? m - q : q;
        };
        int i = step_x(0);
        {
            const float2* T0 = fac_block(fac, P, off0, i);
            for (int e = jj; e < k * k; e += GW) {
                const int r = e / k, c = e - r * k;
                Tt[0][c * KM + r] = T0[(size_t)r * P.ldk + c];
            }
        }
        for (int a = 0; a < k; ++a) W[a][jj] = make_float2(sx == i && sa == a ? 1.f : 0.f, 0.f);
        __syncthreads();
        for (int q = 0; q < nsteps; ++q) {
            const bool more = q + 1 < nsteps;
            const int inext = more ? step_x(q + 1) : -1;
            constexpr int PF = (KM * KM + GW - 1) / GW;
            float2 pf[PF];
            if (more) {
                const float2* Tn = fac_block(fac, P, off0, inext);
#pragma unroll
                for (int u = 0; u < PF; ++u) {
                    const int e = jj + u * GW;
                    pf[u] = make_float2(0.f, 0.f);
                    if (e < k * k) pf[u] = Tn[(size_t)(e / k) * P.ldk + e % k];
                }
            }
            float2 acc[KM];
#pragma unroll
            for (int a = 0; a < KM; ++a) acc[a] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int kk = 0; kk < k; ++kk) {
                const float4* tr = reinterpret_cast<const float4*>(&Tt[q & 1][kk * KM]);
                const float2 w = W[kk][jj];
#pragma unroll
                for (int a = 0; a < KM; a += 2) {
                    const float4 v = tr[a / 2];
                    cfma(acc[a], make_float2(v.x, v.y), w);
                    cfma(acc[a + 1], make_float2(v.z, v.w), w);
                }
            }
            if (more) {
#pragma unroll
                for (int u = 0; u < PF; ++u) {
                    const int e = jj + u * GW;
                    if (e < k * k) Tt[(q + 1) & 1][(e % k) * KM + e / k] = pf[u];
                }
            }
            const bool fwd = q < nlf + nrf, mid = q == nlf + nrf;
            const bool nfwd = q + 1 < nlf + nrf, nmid = q + 1 == nlf + nrf;
            const bool has_y = i < m ? do_left && i >= xa : do_right && i <= xb;
            const float2 cb = i < m ? t.c_up[i] : t.c_dn[i];                  // back substitution
            const float2 cf = !more ? make_float2(0.f, 0.f) : (inext < m ? t.c_dn[inext] : t.c_up[inext]);
            float2* Yi = Y + (size_t)i * KM * GW;
#pragma unroll
            for (int a = 0; a < KM; ++a) {
                if (a >= k) break;
                float2 val = acc[a];
                if (fwd) {
                    Yi[a * GW] = val;                                          // y_i
                } else {
                    if (mid) {
                        Yi[a * GW] = val;                                      // x_m
                    } else {
                        // x_i = y_i - coupling * (T_i x_prev)
                        const float2 yv = has_y ? Yi[a * GW] : make_float2(0.f, 0.f);
                        val = sub_coupled(yv, cb, val, !has_y && i < m ? FIRST_XX : FIRST_YY);
                    }
                    const int o = so[a];
                    if (o >= 0 && jj < jn) Gp[(size_t)(o + i) * D.n_in + I.j0 + jj] = val;
                }
                if (more) {
                    const float2 e = make_float2(sx == inext && sa == a ? 1.f : 0.f, 0.f);
                    float2 w;
                    if (nfwd) {
                        w = q + 1 == nlf ? e : sub_coupled(e, cf, val, FIRST_XX);         // a chain starts at its end block
                    } else if (nmid) {
                        w = e;
                        if (do_left) w = sub_coupled(w, t.c_dn[m], Y[((size_t)(m - 1) * KM + a) * GW], FIRST_XX);
                        if (do_right) w = sub_coupled(w, t.c_up[m], Y[((size_t)(m + 1) * KM + a) * GW], FIRST_XX);
                    } else if (inext == m + 1) {
                        w = Y[((size_t)m * KM + a) * GW];                      // the right back pass starts from x_m
                    } else {
                        w = val;
                    }
                    W[a][jj] = w;
                }
            }
            i = inext;
            __syncthreads();
        }
    }
}

// Pack one output tile (operator p, 64 complex rows) into the apply's format.
struct PItem { int p, mt; };

__global__ void __launch_bounds__(256)
k_dense_pack(const DProb* __restrict__ dp, const PItem* __restrict__ items, const float2* __restrict__ Gt,
             const long long* __restrict__ goff, unsigned char* __restrict__ G) {
    __shared__ float2 stage[64][33];
    const PItem I = items[blockIdx.x];
    const DProb D = dp[I.p];
    const float2* src = Gt + goff[I.p];
    const int tid = threadIdx.x;
    const int n_in = D.n_in;
    const int row0 = I.mt * (64 + D.xr);             // first output row of the tile
    const int unit_x = TILE_UNIT + 8 * D.xr;
    for (int r = 0; r < HELM_DENSE_CS; ++r) {
        for (int c = 0; c < D.nkc; ++c) {
            const int kw = min(128, D.KR - 128 * c);
            const int jb = r * D.KR + 128 * c;
            unsigned char* tile = G + D.off + ((long long)(I.mt * HELM_DENSE_CS + r) * D.KR + 128 * c) * unit_x;
            // [kw][64] complex: element (kj, row) at kj * 64 + row
            float2* T = reinterpret_cast<float2*>(tile);
            for (int k0 = 0; k0 < kw; k0 += 32) {
                __syncthreads();
                for (int e = tid; e < 64 * 32; e += 256) {
                    const int row = e >> 5, kj = e & 31;
                    const int o = row0 + row, j = jb + k0 + kj;
                    stage[row][kj] = (row < 64 && o < D.n_out && j < n_in && k0 + kj < kw)
                                         ? src[(size_t)o * n_in + j] : make_float2(0.f, 0.f);
                }
                __syncthreads();
                for (int e = tid; e < 64 * 32; e += 256) {
                    const int kj = e >> 6, row = e & 63;
                    if (k0 + kj < kw) T[(size_t)(k0 + kj) * 64 + row] = stage[row][kj];
                }
            }
            // extra rows: [xr][kw] after the main part
            float2* X = reinterpret_cast<float2*>(tile + (size_t)TILE_UNIT * kw);
            for (int e = tid; e < D.xr * kw; e += 256) {
                const int x = e / kw, kj = e - x * kw;
                const int o = row0 + 64 + x, j = jb + kj;
                X[e] = (o < D.n_out && j < n_in) ? src[(size_t)o * n_in + j] : make_float2(0.f, 0.f);
            }
        }
    }
}

// Read one stored operator back as complex FP32 [n_out][n_in] (for tests).
__global__ void k_dense_unpack(DProb D, const unsigned char* __restrict__ G, float2* __restrict__ out) {
    const long long total = (long long)D.n_out * D.n_in;
    const int unit_x = TILE_UNIT + 8 * D.xr, rows = 64 + D.xr;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(e / D.n_in), j = (int)(e - (long long)o * D.n_in);
        const int mt = o / rows, row = o - mt * rows;
        const int r = j / D.KR, jr = j - r * D.KR, c = jr >> 7, kj = jr & 127;
        const int kw = min(128, D.KR - 128 * c);
        const unsigned char* tile = G + D.off + ((long long)(mt * HELM_DENSE_CS + r) * D.KR + 128 * c) * unit_x;
        out[e] = row >= 64 ? reinterpret_cast<const float2*>(tile + (size_t)TILE_UNIT * kw)[(size_t)(row - 64) * kw + kj]
                           : reinterpret_cast<const float2*>(tile)[(size_t)kj * 64 + row];
    }
}

// ============================================================== apply ========

constexpr int DT = 256;                 // compute threads (8 warps)
constexpr int PT = 32;                  // the thread that issues the ring's copies (warp 1, lane 0)
constexpr int DSTAGES = 2;              // operator tiles in flight
constexpr int TILE_BYTES = 128 * 528;  // one ring stage: 128 K columns x (512 + 2 extra rows x 8) bytes
constexpr int BBUF_BYTES = 128 * 64 * 8;     // the input slice [128][64], then the partial sums [64][64]
constexpr int PF_AHEAD = 4;             // tiles prefetched into L2 ahead of the ring
constexpr long long DEFAULT_WAIT = 4000000000ll;   // about 2 s at 2 GHz
// shared memory before the per-slab tables: ring, input slice / partials, gather
// plan, extra-row partials, update operands, barriers, flags and the tile walk
constexpr int DENSE_SMEM_FIXED = DSTAGES * TILE_BYTES + BBUF_BYTES + 128 * 4 + 2 * 64 * 8 + 3 * 256 * 8 +
                                 (DSTAGES + 2) * 8 + 16 + 2 * 48;
constexpr int DENSE_MAX_B = 172;        // blocks per axis the dense forms take (n = 165 with b = 6, d = 1)

// Work space of one apply launch (R8 right-hand sides, right-hand side fastest):
//   V   [N lines][Wmax z rows][N x][R8]   forward values of the current slab
//   Q   [N lines][Wmax z rows][N x][R8]   inputs of the next solves: the line
//                                         couplings of Algorithm 4, written by
//                                         the solve that produces them
//   Gv  [N lines][DZ layers][N x][R8]     the slab's right-hand side on its own layers
//   Zv  [N lines][DZ layers][N x][R8]     the slab's restricted result
struct DenseArgs {
    Geom g;
    const AxisWin* win;
    const DProb* dp;
    const unsigned char* G;
    const float2* c_dn;
    const float2* c_up;
    const float2* rin;
    float2* zout;
    float2* V;
    float2* Q;
    float2* Gv;
    float2* Zv;
    unsigned* ctr;
    int* err;
    int nrhs, R8, nclus, nsteps, DZ;
    long long wait_cycles;
    int unmet;
};

__device__ __forceinline__ int vbase(const DenseArgs& A, int line, int lz, int x) {
    return ((line * A.g.Wmax + lz) * A.g.N + x) * A.R8;
}
__device__ __forceinline__ int zbase(const DenseArgs& A, int line, int zr, int x) {
    return ((line * A.DZ + zr) * A.g.N + x) * A.R8;
}

__device__ __forceinline__ void named_sync_compute() { asm volatile("bar.sync 1, %0;" ::"n"(DT) : "memory"); }

// Bounded wait on an mbarrier phase; gives up after `limit` cycles or when
// *stop is set (stop may be null).
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t ph, long long limit, bool cluster_scope,
                                         volatile int* stop) {
    const long long t0 = clock64();
    for (;;) {
        if (cluster_scope ? ptx::mbar_try_cluster(bar, ph) : ptx::mbar_try(bar, ph)) return true;
        if (clock64() - t0 > limit) return false;
        if (stop && *stop) return false;
    }
}

// The walk over this CTA's operator tiles in consumption order, with the
// fields of the current step's operator cached (one thread of the CTA runs it
// and keeps it in shared memory between calls).  Operator records of the slab
// visit whose table is in shared memory (tab_jo) are read from there, others
// from global memory.
template <int TWO>
struct TileIter {
    int s, mt, c, done;
    int n_mt, nkc, KR, xr;
    int m0, mstride;            // this cluster's first tile of step s and its tile stride
    long long off;
    __device__ void load(const DenseArgs& A, int cid, const DProb* tab, int tab_jo) {
        const StepInfo t = step_info(s, A.g.B, A.g.cen, TWO, cid, A.nclus);
        m0 = t.mcid;
        mstride = t.mncl;
        if (t.phase) {
            n_mt = 0;
            return;
        }
        if (t.jo == tab_jo) {
            const DProb& D = tab[op_slot(t.o.Mp, t.o.id, A.g.B)];
            n_mt = D.n_mt;
            nkc = D.nkc;
            KR = D.KR;
            xr = D.xr;
            off = D.off;
        } else {
            const DProb* D = &A.dp[t.o.p];
            n_mt = __ldg(&D->n_mt);
            nkc = __ldg(&D->nkc);
            KR = __ldg(&D->KR);
            xr = __ldg(&D->xr);
            off = __ldg(&D->off);
        }
    }
    __device__ void fix(const DenseArgs& A, int cid, const DProb* tab, int tab_jo) {
        while (s < A.nsteps) {
            load(A, cid, tab, tab_jo);
            mt = m0;
            c = 0;
            if (mt < n_mt) return;
            ++s;
        }
        done = 1;
    }
    __device__ void start(const DenseArgs& A, int cid) {
        s = 0;
        done = 0;
        fix(A, cid, nullptr, -1);
    }
    __device__ void next(const DenseArgs& A, int cid, const DProb* tab, int tab_jo) {
        if (++c < nkc) return;
        c = 0;
        mt += mstride;
        if (mt < n_mt) return;
        ++s;
        fix(A, cid, tab, tab_jo);
    }
    __device__ const unsigned char* ptr(const DenseArgs& A, int rank, uint32_t* bytes) const {
        const int kw = min(128, KR - 128 * c);
        const int ux = TILE_UNIT + 8 * xr;
        *bytes = (uint32_t)(kw * ux);
        return A.G + off + ((long long)(mt * HELM_DENSE_CS + rank) * KR + 128 * c) * ux;
    }
};

// Gather plan of one K-chunk: the single source of each input entry's value,
// encoded as 2 * offset (into Q) or 2 * offset + 1 (into Gv), or -1 for zero.
// Forward solves read the line couplings earlier solves wrote into Q on the
// lines next to the neighbours they come from (the first line for the lower
// front, the last for the upper, both for the centre), and the slab
// right-hand side Gv on its own layers elsewhere; backward solves read the
// coupling on the line next to the block their pass comes from.
__device__ __forceinline__ void gather_plan(const DenseArgs& A, const DProb& D, const OpInfo& o, const AxisWin& wz,
                                            int yb0, int yb1, int k0, int kw, int* s_src, int tid) {
    for (int jj = tid; jj < 128; jj += DT) {
        const int j = k0 + jj;
        int src = -1;
        if (jj < kw && j < D.n_in) {
            const int per = D.in.nz * D.in.nl;
            const int x = j / per;
            const int r = j - x * per, l = r / D.in.nz;
            const int lz = D.in.z0 + (r - l * D.in.nz), line = D.in.line0 + l;
            if (o.id == 0) {
                const bool from_below = o.ry != ROLE_U && o.Mp > 0 && line == yb0;
                const bool from_above = o.ry != ROLE_L && o.Mp < A.g.B - 1 && line == yb1 - 1;
                if (from_below || from_above) src = 2 * vbase(A, line, lz, x);
                else if (lz >= wz.ia && lz < wz.ib) src = 2 * zbase(A, line, lz - wz.ia, x) + 1;
            } else if (o.ry == ROLE_L ? line == yb1 - 1 : line == yb0) {
                src = 2 * vbase(A, line, lz, x);
            }
        }
        s_src[jj] = src;
    }
}

__device__ __forceinline__ float2 gather_val(const DenseArgs& A, const int* s_src, int jj, int rhs) {
    const int src = s_src[jj];
    if (src < 0) return make_float2(0.f, 0.f);     // no load for an absent entry
    const float2* base = (src & 1) ? A.Gv : A.Q;
    return __ldcg(base + (src >> 1) + rhs);
}

// TWO: the sweep schedule (0 one front, 1 two fronts) as a compile-time constant:
// the one-front kernel carries none of the two-front step mapping.
template <int TWO>
__global__ void __launch_bounds__(DT, 1) k_dense(const __grid_constant__ DenseArgs A) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int B = A.g.B;
    unsigned char* ring = smem;
    unsigned char* Bbuf = smem + DSTAGES * TILE_BYTES;
    int* s_src = reinterpret_cast<int*>(Bbuf + BBUF_BYTES);          // [128] gather plan
    float2* s_xp = reinterpret_cast<float2*>(s_src + 128);           // [2][64] extra rows' partial sums
    float2* s_pre = s_xp + 2 * 64;                                   // [3][DT] update operands (cp.async)
    uint64_t* full = reinterpret_cast<uint64_t*>(s_pre + 3 * DT);
    uint64_t* ready = full + DSTAGES;      // every rank's partial sums are in place (8 arrivals)
    uint64_t* done = ready + 1;            // every rank has read the partial sums (8 arrivals)
    volatile int* s_stop = reinterpret_cast<volatile int*>(done + 1);
    volatile int* s_issued = s_stop + 1;   // tiles issued into the ring
    volatile int* s_pend = s_issued + 1;   // released stages whose refill waits for the next step
    TileIter<TWO>* s_itr = reinterpret_cast<TileIter<TWO>*>(const_cast<int*>(s_stop) + 4);   // [2] fill, prefetch (8-byte aligned)
    static_assert(sizeof(TileIter<TWO>) <= 48, "the tile walk's shared slot");
    DProb* s_dp = reinterpret_cast<DProb*>(smem + DENSE_SMEM_FIXED);  // [B+1] operators of the current slab
    AxisWin* s_win = reinterpret_cast<AxisWin*>(s_dp + (B + 2));      // [B] windows

    const int tid = threadIdx.x;
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int cid = blockIdx.x / HELM_DENSE_CS;
    const int R8 = A.R8, N = A.g.N;
    const long long limit = A.wait_cycles > 0 ? A.wait_cycles : DEFAULT_WAIT;

    if (tid == 0) {
        for (int q = 0; q < DSTAGES; ++q) {
            ptx::mbar_init(&full[q], 1);
        }
        ptx::mbar_init(ready, HELM_DENSE_CS);
        ptx::mbar_init(done, HELM_DENSE_CS);
        *s_stop = 0;
        *s_issued = 0;
        *s_pend = 0;
        ptx::fence_mbar_init();
    }
    for (int q = tid; q < B; q += DT) s_win[q] = A.win[q];
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");

    int consumed = 0;                      // ring tiles seen landed by thread 0
    int tab_jo = -1;                       // the slab visit whose operator table is in s_dp
    // Thread PT keeps the ring full: tile t goes into stage t mod DSTAGES once the
    // stage's previous tile is released, and one more tile is prefetched into L2
    // PF_AHEAD tiles ahead.  A release whose next tile belongs to a later step is
    // only counted (s_pend); its refill runs at the top of the next step, while
    // thread 0 polls the step counter, instead of on this step's critical path.
    auto refill = [&]() {
        TileIter<TWO> f = s_itr[0], pf = s_itr[1];
        const int stage = *s_issued % DSTAGES;
        if (!f.done) {
            uint32_t bytes;
            const unsigned char* src = f.ptr(A, (int)rank, &bytes);
            ptx::mbar_expect_tx(&full[stage], bytes);
            ptx::bulk_g2s(ring + (size_t)stage * TILE_BYTES, src, bytes, &full[stage]);
            *s_issued = *s_issued + 1;
            f.next(A, cid, s_dp, tab_jo);
        }
        if (!pf.done) {
            uint32_t pb;
            const unsigned char* ps = pf.ptr(A, (int)rank, &pb);
            ptx::prefetch_l2(ps, pb);
            pf.next(A, cid, s_dp, tab_jo);
        }
        s_itr[0] = f;
        s_itr[1] = pf;
    };
    if (tid == PT) {
        TileIter<TWO> f, pf;
        f.start(A, cid);
        pf.start(A, cid);
        for (int q = 0; q < PF_AHEAD && !pf.done; ++q) pf.next(A, cid, nullptr, -1);
        s_itr[0] = f;
        s_itr[1] = pf;
        for (int q = 0; q < DSTAGES; ++q) refill();
    }
    {
        // ---------------- compute warps ----------------
        int stg = 0;
        uint32_t sph = 0, rph = 0, dph = 0;
        const size_t NN = (size_t)N * N;
        for (int s = 0; s < A.nsteps; ++s) {
            const StepInfo si = step_info(s, B, A.g.cen, TWO, cid, A.nclus);
            const int mcid = si.mcid, mncl = si.mncl;   // this cluster among the clusters of its solve
            // ---- the operator of an op step (phase steps: unused placeholders) ----
            const OpInfo o = si.o;
            const DProb& D = s_dp[op_slot(o.Mp, o.id, B)];
            const AxisWin wz = s_win[o.M], wy = s_win[o.Mp];
            const int yb0 = wy.lo + wy.ia, yb1 = wy.lo + wy.ib;
            const int n_mt = D.n_mt, nkc = D.nkc, KR = D.KR, xr = D.xr, rows = 64 + xr;
            const int cen = A.g.cen;
            // Couplings of Algorithm 4 this solve's result feeds (constants of the
            // operator), by the line block's role: a forward solve of the lower front
            // feeds the next block's first line (-c_dn), of the upper front the block
            // below's last line (-c_up); the centre's forward value is final and feeds
            // the backward passes of both neighbours (c_up below, c_dn above, the
            // second target); a backward solve feeds the next block of its pass
            // (c_up below for the lower front, c_dn above for the upper).
            float2 cf = make_float2(0.f, 0.f), cf2 = make_float2(0.f, 0.f);
            if (!si.phase) {
                const float2 dn = A.c_dn[yb1 < N ? yb1 : N - 1], up = A.c_up[yb0 > 0 ? yb0 - 1 : 0];
                if (o.id == 0 && o.ry == ROLE_L) cf = make_float2(-dn.x, -dn.y);
                else if (o.id == 0 && o.ry == ROLE_U) cf = make_float2(-up.x, -up.y);
                else if (o.id == 0) { cf = up; cf2 = dn; }
                else cf = (o.ry == ROLE_L) ? up : dn;
            }
            // the upper front's last forward solve adds its coupling to the centre's
            // line that the lower front already coupled into, when the centre block
            // is a single line (its first line is its last)
            const bool cen_one = s_win[cen].ib - s_win[cen].ia == 1;
            // Plan of one output row (tile-relative index orow): offsets of its forward
            // value (V), restricted result (Zv), coupling target (Q) and the target's
            // update source (>= 0: a slab term in Gv; <= -2: Q itself at -2 - value),
            // -1 where absent; z2 is the centre's second coupling target.
            int z2m = -1, z2x = -1;
            auto row_plan = [&](int orow, int* z2) {
                int4 pl = make_int4(-1, -1, -1, -1);
                *z2 = -1;
                if (orow < D.n_out) {
                    int q = orow;
                    const int s0 = D.out[0].nl * D.out[0].nz * N;
                    const bool r1 = D.nrect > 1 && q >= s0;
                    if (r1) q -= s0;
                    const int l0 = r1 ? D.out[1].line0 : D.out[0].line0;
                    const int z0 = r1 ? D.out[1].z0 : D.out[0].z0;
                    const int nz = r1 ? D.out[1].nz : D.out[0].nz;
                    const int x = q % N, t = q / N;
                    const int lz = z0 + t % nz, line = l0 + t / nz;
                    const bool zint = lz >= wz.ia && lz < wz.ib;
                    pl.x = vbase(A, line, lz, x);
                    if (zint) pl.y = zbase(A, line, lz - wz.ia, x);
                    if (o.id == 0 && o.ry == ROLE_L) {
                        if (line == yb1 - 1) {                      // into the next block's first line
                            pl.z = vbase(A, yb1, lz, x);
                            if (zint) pl.w = zbase(A, yb1, lz - wz.ia, x);
                        }
                    } else if (o.id == 0 && o.ry == ROLE_U) {
                        if (line == yb0) {                          // into the block below's last line
                            pl.z = vbase(A, yb0 - 1, lz, x);
                            if (o.Mp == cen + 1 && cen_one) pl.w = -2 - pl.z;
                            else if (zint) pl.w = zbase(A, yb0 - 1, lz - wz.ia, x);
                        }
                    } else if (o.id == 0) {                         // the centre: final, feeds both backward passes
                        if (o.Mp > 0 && line == yb0) pl.z = vbase(A, yb0 - 1, lz, x);
                        if (o.Mp < B - 1 && line == yb1 - 1) *z2 = vbase(A, yb1, lz, x);
                    } else if (o.ry == ROLE_L) {
                        if (o.Mp > 0 && line == yb0) pl.z = vbase(A, yb0 - 1, lz, x);   // the block below's last line
                    } else {
                        if (o.Mp < B - 1 && line == yb1 - 1) pl.z = vbase(A, yb1, lz, x);   // the block above's first line
                    }
                }
                return pl;
            };
            // Thread tid < 4 R8 owns output row mi of this rank's 8 and the right-hand
            // sides mrhs, mrhs + 1; thread tid < R8 also owns right-hand side tid of the
            // extra row this rank sums (tile row 64 + xown), if the tile has it.
            const int mi = tid / (R8 / 2), mrhs = 2 * (tid - mi * (R8 / 2));
            const int xown = HELM_DENSE_CS - 1 - (int)rank;
            int4 plm = make_int4(-1, -1, -1, -1), plx = make_int4(-1, -1, -1, -1);
            // This thread's plans for output tile mt (static data).
            auto tile_plans = [&](int mt) {
                if (tid < 4 * R8) plm = row_plan(rows * mt + 8 * (int)rank + mi, &z2m);
                if (xown < xr && tid < R8) plx = row_plan(rows * mt + 64 + xown, &z2x);
            };
            // The update operands of those rows, fetched asynchronously: forward values
            // of the block (a backward solve; written by its forward solve, two or more
            // steps back), the slab terms of the coupling (a forward solve; written by
            // the visit's boundary phase) or the coupled centre line (written by the
            // lower front's last forward solve, two or more steps back).
            auto pre_src = [&](const int4& pl) -> const float2* {
                if (o.id == 1) return pl.x >= 0 ? A.V + pl.x : nullptr;
                if (pl.w >= 0) return A.Gv + pl.w;
                if (pl.w <= -2) return A.Q + (-2 - pl.w);
                return nullptr;
            };
            auto fetch_pre = [&]() {
                if (tid < 4 * R8) {
                    const float2* src = pre_src(plm);
                    if (src) ptx::cp_async16(&s_pre[2 * tid], src + mrhs);
                }
                if (xown < xr && tid < R8) {
                    const float2* src = pre_src(plx);
                    if (src) ptx::cp_async8(&s_pre[2 * DT + tid], src + tid);
                }
                ptx::cp_async_commit();
            };
            // ---- prologue: the first tile's plans and the chunk-0 gather plan are made
            //      while thread 0 waits for step s-1.  The update operands are fetched here
            //      too unless step s-1 is the boundary phase that writes them (then after the
            //      wait). ----
            const bool pro = !si.phase && mcid < n_mt;
            // (two fronts: the upper front's last forward solve reads the centre line the
            // lower front wrote one step before)
            const bool pre_early = si.k >= 2 && !(TWO && o.id == 0 && o.ry == ROLE_U && o.Mp == cen + 1 && cen_one);
            if (pro) {
                tile_plans(mcid);
                if (pre_early) fetch_pre();
                gather_plan(A, D, o, wz, yb0, yb1, (int)rank * KR, min(128, KR), s_src, tid);
            }
            if (tid == PT && *s_pend > 0 && !*s_stop) {
                for (int q = *s_pend; q > 0; --q) refill();
                *s_pend = 0;
            }
            // ---- every CTA has finished step s-1 ----
            if (s > 0 || A.unmet) {
                if (tid == 0) {
                    const unsigned target =
                        A.unmet ? 0xFFFFFFF0u : (unsigned)(HELM_DENSE_CS * A.nclus) * (unsigned)s;
                    const long long t0 = clock64();
                    while (ptx::ld_acquire_gpu(A.ctr) < target) {
                        if (clock64() - t0 > limit) {
                            atomicOr(A.err, 2);
                            *s_stop = 1;
                            break;
                        }
                    }
                }
                named_sync_compute();
                if (*s_stop) break;
            }
            if (si.phase) {
                // ---- boundary of slab visits jo-1 and jo (Algorithm 6) ----
                // The previous visit's result goes to z (a backward visit subtracts its
                // correction); then the new visit's right-hand side on its own layers:
                // forward, f minus the couplings of the neighbours already swept (the
                // block below for the lower front and the centre, the block above for
                // the upper front and the centre); backward, the coupling of the
                // neighbour its pass comes from (above for the lower front, below for
                // the upper).  Neighbour values are read back from z: each thread owns
                // whole (x, y, right-hand side) columns, so it reads what it wrote.
                PassPos vp{0, 0, 0}, vc{0, 0, 0};
                if (si.jo > 0) vp = pass_pos(si.jo - 1, B, A.g.cen);
                const bool cur = si.jo < 2 * B - 1;
                if (cur) {
                    vc = pass_pos(si.jo, B, A.g.cen);
                    // the operators of the new slab (slots of op_slot)
                    for (int q = tid; q <= B + 1; q += DT) s_dp[q] = A.dp[op_index(vc.M, q, B)];
                    tab_jo = si.jo;
                }
                const AxisWin wp = s_win[vp.M], wc = s_win[vc.M];
                const int dzp = wp.ib - wp.ia, dzc = wc.ib - wc.ia;
                const int mc = wc.lo + wc.ia, ec = wc.lo + wc.ib;       // the new slab's own layers [mc, ec)
                const bool cpl_lo = cur && (vc.bwd ? vc.role == ROLE_U : (vc.role != ROLE_U && vc.M > 0));
                const bool cpl_hi = cur && (vc.bwd ? vc.role == ROLE_L : (vc.role != ROLE_L && vc.M < B - 1));
                const float sgn = vc.bwd ? 1.f : -1.f;
                // a neighbour layer the previous visit just wrote is taken from registers
                const int pv0 = wp.lo + wp.ia, pv1 = wp.lo + wp.ib;
                const bool reg_lo = si.jo > 0 && mc - 1 >= pv0 && mc - 1 < pv1;
                const bool reg_hi = si.jo > 0 && ec >= pv0 && ec < pv1;
                const long long total = (long long)NN * R8;
                const long long stride = (long long)gridDim.x * DT;
                constexpr int PP = 4;                           // points per thread and pass
                for (long long p0 = (long long)blockIdx.x * DT + tid; p0 < total; p0 += PP * stride) {
                    int xs[PP], ls[PP], rs[PP];
                    bool ok[PP];
                    float2 nb_lo[PP], nb_hi[PP];
#pragma unroll
                    for (int q = 0; q < PP; ++q) {
                        nb_lo[q] = nb_hi[q] = make_float2(0.f, 0.f);
                        const long long p = min(p0 + q * stride, total - 1);
                        ok[q] = p0 + q * stride < total;
                        xs[q] = (int)(p % N);
                        const long long t = p / N;
                        ls[q] = (int)(t % N);
                        rs[q] = (int)(t / N);
                    }
                    if (si.jo > 0) {
                        for (int zr = 0; zr < dzp; ++zr) {
                            const int layer = wp.lo + wp.ia + zr;
                            float2 v[PP], old[PP];
#pragma unroll
                            for (int q = 0; q < PP; ++q) {
                                const int rr = min(rs[q], A.nrhs - 1);
                                v[q] = __ldcg(A.Zv + zbase(A, ls[q], zr, xs[q]) + rs[q]);
                                old[q] = (vp.bwd && rs[q] < A.nrhs)
                                             ? A.zout[((size_t)rr * N + layer) * NN + (size_t)ls[q] * N + xs[q]]
                                             : make_float2(0.f, 0.f);
                            }
#pragma unroll
                            for (int q = 0; q < PP; ++q) {
                                const float2 nz = vp.bwd ? csub(old[q], v[q]) : v[q];
                                if (ok[q] && rs[q] < A.nrhs)
                                    A.zout[((size_t)rs[q] * N + layer) * NN + (size_t)ls[q] * N + xs[q]] = nz;
                                if (layer == mc - 1) nb_lo[q] = nz;
                                if (layer == ec) nb_hi[q] = nz;
                            }
                        }
                    }
                    if (cur) {
                        // neighbour values (z, after the write above) times the couplings
                        float2 add_lo[PP], add_hi[PP];
#pragma unroll
                        for (int q = 0; q < PP; ++q) {
                            const int rr = min(rs[q], A.nrhs - 1);
                            const size_t col = (size_t)ls[q] * N + xs[q];
                            add_lo[q] = make_float2(0.f, 0.f);
                            add_hi[q] = make_float2(0.f, 0.f);
                            if (cpl_lo && rs[q] < A.nrhs) {
                                const float2 u = reg_lo ? nb_lo[q] : A.zout[((size_t)rr * N + mc - 1) * NN + col];
                                const float2 c = cmul(A.c_dn[mc], u);
                                add_lo[q] = make_float2(sgn * c.x, sgn * c.y);
                            }
                            if (cpl_hi && rs[q] < A.nrhs) {
                                const float2 u = reg_hi ? nb_hi[q] : A.zout[((size_t)rr * N + ec) * NN + col];
                                const float2 c = cmul(A.c_up[ec - 1], u);
                                add_hi[q] = make_float2(sgn * c.x, sgn * c.y);
                            }
                        }
                        for (int zr = 0; zr < dzc; ++zr) {
                            const int layer = mc + zr;
                            float2 rv[PP];
#pragma unroll
                            for (int q = 0; q < PP; ++q) {
                                const int rr = min(rs[q], A.nrhs - 1);
                                rv[q] = vc.bwd ? make_float2(0.f, 0.f)
                                               : A.rin[((size_t)rr * N + layer) * NN + (size_t)ls[q] * N + xs[q]];
                            }
#pragma unroll
                            for (int q = 0; q < PP; ++q) {
                                float2 gv = make_float2(0.f, 0.f);
                                if (rs[q] < A.nrhs) {
                                    gv = rv[q];
                                    if (zr == 0) gv = cadd(gv, add_lo[q]);
                                    if (zr == dzc - 1) gv = cadd(gv, add_hi[q]);
                                }
                                if (ok[q]) A.Gv[zbase(A, ls[q], zr, xs[q]) + rs[q]] = gv;
                            }
                        }
                    }
                }
                named_sync_compute();
                if (tid == 0) ptx::red_release_gpu_add(A.ctr, 1u);
                continue;
            }
            // this CTA's tiles of the step after tile (mt, c)
            auto tiles_left = [&](int mt_, int c_) {
                const int total = ((n_mt - mcid + mncl - 1) / mncl) * nkc;
                return total - (((mt_ - mcid) / mncl) * nkc + c_) - 1;
            };
            for (int mt = mcid; mt < n_mt; mt += mncl) {
                const bool first = (mt == mcid);
                if (!first || !pro) {
                    // a later tile of this step: plans inline
                    named_sync_compute();
                    tile_plans(mt);
                    fetch_pre();
                } else if (!pre_early) {
                    fetch_pre();
                }
                for (int q = tid; q < 2 * 64; q += DT) s_xp[q] = make_float2(0.f, 0.f);
                float2 acc[4][4];                               // SIMT form: rows 4 rg.., RHS 4 cg..
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);
                for (int c = 0; c < nkc; ++c) {
                    const int kw = min(128, KR - 128 * c);
                    const int k0 = (int)rank * KR + 128 * c;
                    const bool planned = first && pro && c == 0;   // the prologue made this chunk's plan
                    {
                        // ---- SIMT: q slice as complex FP32 [kw][64], then the tile product ----
                        if (!planned) {
                            named_sync_compute();
                            gather_plan(A, D, o, wz, yb0, yb1, k0, kw, s_src, tid);
                            named_sync_compute();
                        }
                        float2* Bq = reinterpret_cast<float2*>(Bbuf);
                        const int rhs = tid & 63, kq = tid >> 6, rc = min(rhs, R8 - 1);
                        for (int t0 = 0; t0 < 32; t0 += 8) {               // slots kq + 4 t, t < 32
                            float2 vals[8];
#pragma unroll
                            for (int t = 0; t < 8; ++t) vals[t] = gather_val(A, s_src, kq + 4 * (t0 + t), rc);
#pragma unroll
                            for (int t = 0; t < 8; ++t) {
                                const int kj = kq + 4 * (t0 + t);
                                if (kj < kw) Bq[kj * 64 + rhs] = (rhs < R8) ? vals[t] : make_float2(0.f, 0.f);
                            }
                        }
                        if (!wait_bar(&full[stg], sph, limit, false, s_stop)) {
                            atomicOr(A.err, 2);
                            *s_stop = 1;
                        } else if (tid == 0) {
                            ++consumed;
                        }
                        named_sync_compute();
                        if (*s_stop) break;
                        const float2* At = reinterpret_cast<const float2*>(ring + (size_t)stg * TILE_BYTES);
                        const int rg = tid >> 4, cg = tid & 15;
                        if (4 * cg < R8) {
                            for (int kk = 0; kk < kw; ++kk) {
                                const float4* ar = reinterpret_cast<const float4*>(At + kk * 64 + 4 * rg);
                                const float4* br = reinterpret_cast<const float4*>(Bq + kk * 64 + 4 * cg);
                                const float4 a0 = ar[0], a1 = ar[1], b0 = br[0], b1 = br[1];
                                const float2 av[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w),
                                                      make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
                                const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                                                      make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
                                for (int a = 0; a < 4; ++a)
#pragma unroll
                                    for (int b = 0; b < 4; ++b) cfma(acc[a][b], av[a], bv[b]);
                            }
                        }
                        if (xr > 0) {
                            const float2* X = reinterpret_cast<const float2*>(ring + (size_t)stg * TILE_BYTES +
                                                                              (size_t)TILE_UNIT * kw);
                            const int rr = tid & 63, kq2 = tid >> 6;
                            for (int ex = 0; ex < xr; ++ex) {
                                float2 acc2 = make_float2(0.f, 0.f);
                                for (int kj = kq2; kj < kw; kj += 4) cfma(acc2, X[ex * kw + kj], Bq[kj * 64 + rr]);
                                atomicAdd(&s_xp[ex * 64 + rr].x, acc2.x);
                                atomicAdd(&s_xp[ex * 64 + rr].y, acc2.y);
                            }
                        }
                        named_sync_compute();
                        if (tid == PT) {
                            if (tiles_left(mt, c) >= DSTAGES) refill();
                            else *s_pend = *s_pend + 1;
                        }
                        if (++stg == DSTAGES) { stg = 0; sph ^= 1u; }
                    }
                }
                if (*s_stop) break;
                // the update operands fetched asynchronously with the plans
                ptx::cp_async_wait_all();
                // ---- this rank's partial sums into Bbuf ----
                {
                    float2* Pp = reinterpret_cast<float2*>(Bbuf);
                    const int rg = tid >> 4, cg = tid & 15;
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) Pp[(4 * rg + a) * 64 + 4 * cg + b] = acc[a][b];
                }
                named_sync_compute();
                if (tid < HELM_DENSE_CS) ptx::mbar_arrive_remote(ptx::mapa(ready, (uint32_t)tid));
                if (!wait_bar(ready, rph, limit, true, nullptr)) {
                    atomicOr(A.err, 2);
                    *s_stop = 1;
                }
                rph ^= 1u;
                // ---- sum the 8 partials of this rank's 8 output rows; apply the update ----
                // Thread tid < 4 R8: row i = tid / (R8/2), right-hand sides rhs, rhs + 1; the
                // eight remote loads are issued before the first is used.
                const float2 coef = cf;
                const bool main_ok = tid < 4 * R8;
                float4 rv[HELM_DENSE_CS];
                if (main_ok) {
                    const int row = 8 * (int)rank + mi;
                    const float* src = reinterpret_cast<const float*>(Bbuf) + 2 * (row * 64 + mrhs);
#pragma unroll
                    for (int q = 0; q < HELM_DENSE_CS; ++q) rv[q] = ptx::ld_dsmem_f32x4(ptx::mapa(src, (uint32_t)q));
                }
                float2 rx[HELM_DENSE_CS];
                const bool xown_ok = xown < xr && tid < R8;
                if (xown_ok) {
#pragma unroll
                    for (int q = 0; q < HELM_DENSE_CS; ++q)
                        rx[q] = ptx::ld_dsmem_f32x2(ptx::mapa(s_xp + xown * 64 + tid, (uint32_t)q));
                }
                if (main_ok) {
                    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < HELM_DENSE_CS; ++q) {
                        y.x += rv[q].x;
                        y.y += rv[q].y;
                        y.z += rv[q].z;
                        y.w += rv[q].w;
                    }
                    const float2 Y0 = make_float2(y.x, y.y), Y1 = make_float2(y.z, y.w);
                    const int4 pl = plm;
                    if (pl.x >= 0) {
                        const float4 pre = *reinterpret_cast<const float4*>(&s_pre[2 * tid]);
                        const float2 p0 = make_float2(pre.x, pre.y), p1 = make_float2(pre.z, pre.w);
                        if (o.id == 0) {
                            *reinterpret_cast<float4*>(A.V + pl.x + mrhs) = y;   // forward values of the line block
                            if (o.ry == ROLE_C && pl.y >= 0)                       // the centre has no backward step
                                *reinterpret_cast<float4*>(A.Zv + pl.y + mrhs) = y;
                            if (pl.z >= 0) {
                                const bool has = pl.w != -1;
                                const float2 g0 = has ? p0 : make_float2(0.f, 0.f);
                                const float2 g1 = has ? p1 : make_float2(0.f, 0.f);
                                const float2 q0 = cadd(g0, cmul(coef, Y0)), q1 = cadd(g1, cmul(coef, Y1));
                                *reinterpret_cast<float4*>(A.Q + pl.z + mrhs) = make_float4(q0.x, q0.y, q1.x, q1.y);
                            }
                            if (z2m >= 0) {
                                const float2 q0 = cmul(cf2, Y0), q1 = cmul(cf2, Y1);
                                *reinterpret_cast<float4*>(A.Q + z2m + mrhs) = make_float4(q0.x, q0.y, q1.x, q1.y);
                            }
                        } else {
                            const float2 v0 = csub(p0, Y0), v1 = csub(p1, Y1);   // backward correction
                            if (pl.y >= 0) *reinterpret_cast<float4*>(A.Zv + pl.y + mrhs) = make_float4(v0.x, v0.y, v1.x, v1.y);
                            if (pl.z >= 0) {
                                const float2 q0 = cmul(coef, v0), q1 = cmul(coef, v1);
                                *reinterpret_cast<float4*>(A.Q + pl.z + mrhs) = make_float4(q0.x, q0.y, q1.x, q1.y);
                            }
                        }
                    }
                }
                if (xown_ok) {
                    float2 Y = make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < HELM_DENSE_CS; ++q) Y = cadd(Y, rx[q]);
                    const int4 pl = plx;
                    const int rhs = tid;
                    if (pl.x >= 0) {
                        const float2 pre = s_pre[2 * DT + tid];
                        if (o.id == 0) {
                            A.V[pl.x + rhs] = Y;
                            if (o.ry == ROLE_C && pl.y >= 0) A.Zv[pl.y + rhs] = Y;
                            if (pl.z >= 0) A.Q[pl.z + rhs] = cadd(pl.w != -1 ? pre : make_float2(0.f, 0.f), cmul(coef, Y));
                            if (z2x >= 0) A.Q[z2x + rhs] = cmul(cf2, Y);
                        } else {
                            const float2 v = csub(pre, Y);
                            if (pl.y >= 0) A.Zv[pl.y + rhs] = v;
                            if (pl.z >= 0) A.Q[pl.z + rhs] = cmul(coef, v);
                        }
                    }
                }
                if (mt + mncl < n_mt) {
                    // another tile of this solve reuses Bbuf: wait until every rank has read it
                    named_sync_compute();
                    if (tid < HELM_DENSE_CS) ptx::mbar_arrive_remote(ptx::mapa(done, (uint32_t)tid));
                    if (!wait_bar(done, dph, limit, true, nullptr)) {
                        atomicOr(A.err, 2);
                        *s_stop = 1;
                    }
                    dph ^= 1u;
                }
                named_sync_compute();
                if (*s_stop) break;
            }
            if (*s_stop) break;
            // ---- this CTA's share of step s is written ----
            if (tid == 0) ptx::red_release_gpu_add(A.ctr, 1u);
        }
    }
    named_sync_compute();
    // ---- teardown: let issued copies land, leave with the cluster ----
    if (tid == 0) {
        const int issued = *s_issued;
        int q = consumed % DSTAGES;
        uint32_t ph = (uint32_t)((consumed / DSTAGES) & 1);
        for (int u = consumed; u < issued; ++u) {
            wait_bar(&full[q], ph, limit, false, nullptr);
            if (++q == DSTAGES) { q = 0; ph ^= 1u; }
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

size_t dense_smem_bytes(int B) {
    return (size_t)DENSE_SMEM_FIXED + (size_t)(B + 2) * sizeof(DProb) + (size_t)B * sizeof(AxisWin);
}

const void* dense_kernel_for(int sched) {
    return sched == HELM_TWO_FRONT ? (const void*)k_dense<1> : (const void*)k_dense<0>;
}

}  // namespace

// ================================================================ host =======

// The operator table: sizes, index sets and storage offsets.
static void build_dense_table(helm_ctx* h, const std::vector<AxisWin>& win, int nclus, std::vector<DProb>& out,
                              size_t* gbytes) {
    const int B = h->g.B, N = h->g.N, b = h->g.b;
    const bool two = h->g.sched == HELM_TWO_FRONT;
    out.assign((size_t)dense_nops(B), DProb());
    size_t off = 0;
    for (int p = 0; p < dense_nops(B); ++p) {
        DProb D;
        memset(&D, 0, sizeof(D));
        // slab M, slot q (op_index inverted)
        const int M = p < B * B ? p / B : (p < B * B + B ? p - B * B : p - B * B - B);
        const int q = p < B * B ? p % B : (p < B * B + B ? B : B + 1);
        const int Mp = q < B ? q : (q == B ? 0 : B - 1);
        const AxisWin& wz = win[M];
        const AxisWin& wy = win[Mp];
        const int Lz = wz.L, za = wz.ia, zb = wz.ib;
        D.fp = M * B + Mp;
        if (q == B + 1 && !two) {
            out[p] = D;                                   // no backward map of the last block (one front)
            continue;
        }
        if (q == 0) {
            // the low boundary slab's forward map: its own entries in, the line
            // next to block 1 whole and the others' interest rows out
            D.in = DRect{0, b, za, zb - za};
            D.nrect = 0;
            if (b > 1) D.out[D.nrect++] = DRect{0, b - 1, za, zb - za};
            D.out[D.nrect++] = DRect{b - 1, 1, 0, Lz};
        } else if (q == B) {
            // its backward map: the coupling line in, the interest rows out
            D.in = DRect{b - 1, 1, 0, Lz};
            D.out[0] = DRect{0, b, za, zb - za};
            D.nrect = 1;
        } else if (two && q == B - 1) {
            // the high boundary slab's forward map (mirror of q = 0)
            D.in = DRect{N - b, b, za, zb - za};
            D.nrect = 0;
            D.out[D.nrect++] = DRect{N - b, 1, 0, Lz};
            if (b > 1) D.out[D.nrect++] = DRect{N - b + 1, b - 1, za, zb - za};
        } else if (q == B + 1) {
            D.in = DRect{N - b, 1, 0, Lz};
            D.out[0] = DRect{N - b, b, za, zb - za};
            D.nrect = 1;
        } else {
            D.in = DRect{wy.lo + wy.ia, wy.ib - wy.ia, 0, Lz};
            D.out[0] = D.in;
            D.nrect = 1;
        }
        D.n_in = D.in.nl * D.in.nz * N;
        D.n_out = 0;
        for (int r = 0; r < D.nrect; ++r) D.n_out += D.out[r].nl * D.out[r].nz * N;
        // tiles of 64 + xr rows: up to 2 extra rows let the operator fit the resident clusters in one round
        const int per_cluster = ceil_div(D.n_out, nclus);
        D.xr = (per_cluster > 64 && per_cluster <= 66) ? per_cluster - 64 : 0;
        D.n_mt = ceil_div(D.n_out, 64 + D.xr);
        D.KR = 16 * ceil_div(ceil_div(D.n_in, HELM_DENSE_CS), 16);
        D.nkc = ceil_div(D.KR, 128);
        D.off = (long long)off;
        off += (size_t)D.n_mt * HELM_DENSE_CS * D.KR * (TILE_UNIT + 8 * D.xr);
        out[p] = D;
    }
    *gbytes = off;
}

// Kernels of the operator columns by block size: one thread per column up to k = 32,
// where its k results fit in registers (166 of them at 32); 64-row tiles beyond, which they
// fill by more than half.  Setup at n = 95 with blocks of 9 to 25: 173 ms against 479 ms
// with 64-row tiles throughout.
typedef void (*GCols)(Geom, Tables, const DProb*, const GItem*, int, const float2*, long long, float2*, const long long*,
                      float2*, size_t);
struct GClass { int km; GCols fn; };
const GClass G_COLS[] = {{10, k_dense_G_cols<10>}, {16, k_dense_G_cols<16>}, {26, k_dense_G_cols<26>}, {32, k_dense_G_cols<32>}};
constexpr int GCLASSES = sizeof(G_COLS) / sizeof(G_COLS[0]) + 1;
int g_class(int k) {
    int q = 0;
    while (q < GCLASSES - 1 && k > G_COLS[q].km) ++q;
    return q;
}

// Factors and restricted operators of slabs Ma..Mb, for the line blocks
// Pa..Pb (and the first block's backward operator when Pa = 0): the build of
// helm_setup (all of them) and of helm_update_velocity (those a box touches).
static int dense_build(helm_ctx* h, const Prob* prob, int Ma, int Mb, int Pa, int Pb, cudaStream_t st) {
    const int B = h->g.B, N = h->g.N;
    const int P = dense_nops(B);
    const DProb* dp = h->dprob_h;
    cudaError_t e;
#define DTRY(x) do { e = (x); if (e != cudaSuccess) { helm_set_cuda_error(e); return e == cudaErrorMemoryAllocation ? HELM_ENOMEM : HELM_ECUDA; } } while (0)
    // ---- chunks of slabs: factors, then the operators of the chunk's problems ----
    // the first-block backward operator of slab M (index B*B+M) uses problem (M, 0)
    const size_t budget = (size_t)6 << 30;            // bytes of temporary factors + G per chunk
    int dev = 0;
    cudaGetDevice(&dev);
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int gblocks = 2 * std::max(nsm, 1);
    const size_t yslot = (size_t)N * 64 * GW;           // complex entries per setup CTA
    float2* yscr = nullptr;
    DTRY(cudaMalloc(&yscr, (size_t)gblocks * yslot * sizeof(float2)));
    const size_t gsm = (size_t)(64 * TLD + 2 * 64 * GW) * sizeof(float2) + (2 * GW + 64) * sizeof(int);
    e = ensure_dyn_smem((const void*)k_dense_G, gsm);
    if (e != cudaSuccess) { cudaFree(yscr); helm_set_cuda_error(e); return HELM_ECUDA; }
    float2* fac = nullptr;
    float2* Gt = nullptr;
    size_t fac_cap = 0, gt_cap = 0;
    GItem* d_items = nullptr;
    PItem* d_pitems = nullptr;
    void* d_tpack = nullptr;
    size_t tpack_cap = 0;
    long long* d_goff = nullptr;
    size_t items_cap = 0, pitems_cap = 0;
    int rc = HELM_OK;
    DTRY(cudaMalloc(&d_goff, sizeof(long long) * P));
    std::vector<long long> goff(P, 0);
    int M0 = Ma;
    while (M0 <= Mb && rc == HELM_OK) {
        // grow the chunk while it fits the budget
        int M1 = M0;
        size_t fbytes = 0, gtb = 0;
        for (;;) {
            const int M = M1;
            const long long f0 = prob[(size_t)M0 * B].off;
            const long long f1 = prob[(size_t)M * B + B - 1].off + (long long)N * prob[(size_t)M * B + B - 1].kstride;
            size_t fb = (size_t)(f1 - f0) * sizeof(float2);
            size_t gb = gtb;
            for (int Mp = 0; Mp < B; ++Mp) gb += (size_t)dp[(size_t)M * B + Mp].n_out * dp[(size_t)M * B + Mp].n_in;
            gb += (size_t)dp[(size_t)B * B + M].n_out * dp[(size_t)B * B + M].n_in;
            gb += (size_t)dp[(size_t)B * B + B + M].n_out * dp[(size_t)B * B + B + M].n_in;
            if (M1 > M0 && fb + gb * sizeof(float2) > budget) break;
            fbytes = fb;
            gtb = gb;
            ++M1;
            if (M1 > Mb) break;
        }
        const long long off0 = prob[(size_t)M0 * B].off;
        if (fbytes > fac_cap) {
            if (fac) cudaFree(fac);
            fac = nullptr;
            DTRY(cudaMalloc(&fac, fbytes));
            fac_cap = fbytes;
        }
        if (gtb * sizeof(float2) > gt_cap) {
            if (Gt) cudaFree(Gt);
            Gt = nullptr;
            DTRY(cudaMalloc(&Gt, gtb * sizeof(float2)));
            gt_cap = gtb * sizeof(float2);
        }
        DTRY(launch_factor_range(h, M0 * B, (M1 - M0) * B, fac, off0, HELM_FP32, st));
        // work items and temporary operator offsets of the chunk
        std::vector<GItem> items, by_class[GCLASSES];
        std::vector<PItem> pitems;
        std::vector<int> ops;
        long long go = 0;
        for (int M = M0; M < M1; ++M) {
            for (int q = 0; q <= B + 1; ++q) {
                // an operator the build leaves as it is (slot B: block 0's backward map, B + 1: block B-1's)
                if (q < B ? (q < Pa || q > Pb) : (q == B ? Pa != 0 : Pb != B - 1)) continue;
                const int p = op_index(M, q, B);
                if (dp[p].n_out == 0) continue;
                goff[p] = go;
                go += (long long)dp[p].n_out * dp[p].n_in;
                for (int j0 = 0; j0 < dp[p].n_in; j0 += GW) by_class[g_class(prob[dp[p].fp].k)].push_back(GItem{p, j0});
                if (h->opts.precision == HELM_FP32)
                    for (int mt = 0; mt < dp[p].n_mt; ++mt) pitems.push_back(PItem{p, mt});
                else
                    ops.push_back(p);
            }
        }
        for (const std::vector<GItem>& v : by_class) items.insert(items.end(), v.begin(), v.end());
        if (items.size() > items_cap) {
            if (d_items) cudaFree(d_items);
            d_items = nullptr;
            DTRY(cudaMalloc(&d_items, items.size() * sizeof(GItem)));
            items_cap = items.size();
        }
        if (!pitems.empty() && pitems.size() > pitems_cap) {
            if (d_pitems) cudaFree(d_pitems);
            d_pitems = nullptr;
            DTRY(cudaMalloc(&d_pitems, pitems.size() * sizeof(PItem)));
            pitems_cap = pitems.size();
        }
        DTRY(cudaMemcpyAsync(d_items, items.data(), items.size() * sizeof(GItem), cudaMemcpyHostToDevice, st));
        if (!pitems.empty())
            DTRY(cudaMemcpyAsync(d_pitems, pitems.data(), pitems.size() * sizeof(PItem), cudaMemcpyHostToDevice, st));
        DTRY(cudaMemcpyAsync(d_goff, goff.data(), sizeof(long long) * P, cudaMemcpyHostToDevice, st));
        size_t first = 0;
        for (int q = 0; q < GCLASSES; ++q) {
            const size_t n = by_class[q].size();
            if (n == 0) continue;
            const GItem* it = d_items + first;
            first += n;
            if (q == GCLASSES - 1) {
                k_dense_G<<<(int)std::min<size_t>(n, (size_t)gblocks), GT, gsm, st>>>(
                    h->g, h->t, h->dprob, it, (int)n, fac, off0, Gt, d_goff, yscr, yslot);
            } else {
                // as many blocks as fit on the chip and the forward values' scratch holds
                int occ = 1;
                DTRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, G_COLS[q].fn, GW, 0));
                const size_t slot = (size_t)N * G_COLS[q].km * GW;
                const size_t blk = std::min(std::min(n, (size_t)nsm * std::max(occ, 1)), gblocks * yslot / slot);
                G_COLS[q].fn<<<(int)blk, GW, 0, st>>>(h->g, h->t, h->dprob, it, (int)n, fac, off0, Gt, d_goff, yscr, slot);
            }
            h->launches++;
            DTRY(cudaGetLastError());
        }
        if (h->opts.precision == HELM_FP32) {
            k_dense_pack<<<(int)pitems.size(), 256, 0, st>>>(h->dprob, d_pitems, Gt, d_goff, h->dG);
            h->launches++;
            DTRY(cudaGetLastError());
        } else {
            DTRY(team_pack(h, ops.data(), (int)ops.size(), Gt, d_goff, &d_tpack, &tpack_cap, st));
        }
        // the host arrays above must outlive their copies
        DTRY(cudaStreamSynchronize(st));
        M0 = M1;
    }
    cudaFree(yscr);
    cudaFree(fac);
    cudaFree(Gt);
    cudaFree(d_items);
    cudaFree(d_pitems);
    cudaFree(d_tpack);
    cudaFree(d_goff);
#undef DTRY
    return rc;
}

int dense_setup(helm_ctx* h, const void* win_host, const void* prob_host, cudaStream_t st) {
    const std::vector<AxisWin>& win = *static_cast<const std::vector<AxisWin>*>(win_host);
    const std::vector<Prob>& prob = *static_cast<const std::vector<Prob>*>(prob_host);
    const int B = h->g.B;
    const int P = dense_nops(B);
    cudaError_t e;
    // ---- the FP32 form's apply launch: clusters of 8 CTAs, as many as can be resident (<= 16) ----
    h->dsmem = dense_smem_bytes(B);
    if (B > DENSE_MAX_B) return HELM_ENOTSUP;
    const bool fp32 = h->opts.precision == HELM_FP32;
    const void* kfn = dense_kernel_for(h->g.sched);
    e = ensure_dyn_smem(kfn, h->dsmem);
    if (e != cudaSuccess) { helm_set_cuda_error(e); return HELM_ECUDA; }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = HELM_DENSE_CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(HELM_DENSE_CS * 16, 1, 1);
    cfg.blockDim = dim3(DT, 1, 1);
    cfg.dynamicSmemBytes = h->dsmem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int ncl = 0;
    e = cudaOccupancyMaxActiveClusters(&ncl, kfn, &cfg);
    if (e != cudaSuccess) { helm_set_cuda_error(e); return HELM_ECUDA; }
    if (ncl < 1) return HELM_ENOTSUP;
    // the tensor-core forms take the tiles of this launch for the rows they keep in more than 16 bits
    int nclus = std::min(ncl, 16);
    if (h->opts.dense_clusters > 0) nclus = std::min(nclus, h->opts.dense_clusters);
    if (fp32) {
        h->dclus = nclus;
    } else {
        const int rc = team_configure(h);
        if (rc != HELM_OK) return rc;
    }
    std::vector<DProb> dp;
    std::vector<int> lo;
    size_t gbytes = 0, nscale = 0;
    build_dense_table(h, win, nclus, dp, &gbytes);
    if (!fp32) {
        h->tprob_h = new TProb[P];
        team_table(h, dp.data(), h->tprob_h, &gbytes, &nscale, &lo);
    }
    h->dprob_h = new DProb[P];
    memcpy(h->dprob_h, dp.data(), sizeof(DProb) * P);
#define DTRY(x) do { e = (x); if (e != cudaSuccess) { helm_set_cuda_error(e); return e == cudaErrorMemoryAllocation ? HELM_ENOMEM : HELM_ECUDA; } } while (0)
    DTRY(cudaMalloc(&h->dprob, sizeof(DProb) * P));
    DTRY(cudaMemcpyAsync(h->dprob, dp.data(), sizeof(DProb) * P, cudaMemcpyHostToDevice, st));
    if (!fp32) {
        DTRY(cudaMalloc(&h->tprob, sizeof(TProb) * P));
        DTRY(cudaMemcpyAsync(h->tprob, h->tprob_h, sizeof(TProb) * P, cudaMemcpyHostToDevice, st));
    }
    DTRY(cudaMalloc(&h->dG, gbytes));
    h->dG_bytes = gbytes;
    if (!lo.empty()) {
        DTRY(cudaMalloc(&h->dlo, lo.size() * sizeof(int)));
        DTRY(cudaMemcpyAsync(h->dlo, lo.data(), lo.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    }
    if (nscale) {
        DTRY(cudaMalloc(&h->dscale, nscale * sizeof(float)));
        h->dscale_elems = nscale;
    }
#undef DTRY
    const int rc = dense_build(h, prob.data(), 0, B - 1, 0, B - 1, st);
    if (rc != HELM_OK || !fp32) return rc;
    int most = 0;
    for (int p = 0; p < P; ++p) most = std::max(most, dp[p].n_mt);
    // two fronts run two solves side by side: at least two clusters, up to twice the tiles
    const bool two = h->g.sched == HELM_TWO_FRONT;
    h->dclus = std::min(h->dclus, std::max(two ? 2 * most : most, two ? 2 : 1));
    if (two && h->dclus < 2) return HELM_ENOTSUP;
    return HELM_OK;
}

// Right-hand sides of one apply launch padded to a power of two >= 8 (the gather maps
// 256 threads onto the columns).
static int dense_r8(int nr) {
    int r = 8;
    while (r < nr) r <<= 1;
    return r;
}

// Layers of a slab's own block: b for the boundary slabs, at most d otherwise (2d for the two-front centre).
static int dense_dz(const helm_ctx* h) {
    return std::max(h->g.b, h->g.sched == HELM_TWO_FRONT ? 2 * h->g.d : h->g.d);   // two fronts: the centre <= 2d
}

// Work space of the FP32 form; also the bound that helm_apply_precond_noalloc puts on every dense form.
size_t dense_noalloc_elems(const helm_ctx* h, int nrhs) {
    // V, Q, Gv and Zv for one launch group (<= 64 right-hand sides), then the step counter (16 bytes)
    const size_t r8 = (size_t)dense_r8(std::min(nrhs, 64));
    const size_t NN = (size_t)h->g.N * h->g.N;
    return 2 * NN * h->g.Wmax * r8 + 2 * NN * dense_dz(h) * r8 + 2;
}

size_t dense_work_elems(const helm_ctx* h, int nrhs, size_t limit) {
    return h->opts.precision == HELM_FP32 ? dense_noalloc_elems(h, nrhs) : team_work_elems(h, nrhs, limit);
}

cudaError_t launch_dense_apply(helm_ctx* h, const float2* r, float2* z, int nrhs, float2* work, size_t elems,
                               cudaStream_t st) {
    if (h->opts.precision != HELM_FP32) return launch_team_apply(h, r, z, nrhs, work, elems, st);
    const size_t n3 = (size_t)h->g.N * h->g.N * h->g.N;
    const void* kfn = dense_kernel_for(h->g.sched);
    const size_t r8max = (size_t)dense_r8(std::min(nrhs, 64));
    const size_t NN = (size_t)h->g.N * h->g.N;
    float2* V = work;
    float2* Qb = V + NN * h->g.Wmax * r8max;
    float2* Gv = Qb + NN * h->g.Wmax * r8max;
    float2* Zv = Gv + NN * dense_dz(h) * r8max;
    unsigned* ctr = reinterpret_cast<unsigned*>(Zv + NN * dense_dz(h) * r8max);
    const int B = h->g.B;
    for (int r0 = 0; r0 < nrhs; r0 += 64) {
        const int nr = std::min(64, nrhs - r0);
        DenseArgs A;
        memset(&A, 0, sizeof(A));
        A.g = h->g;
        A.win = h->t.win;
        A.dp = h->dprob;
        A.G = h->dG;
        A.c_dn = h->t.c_dn;
        A.c_up = h->t.c_up;
        A.rin = r + (size_t)r0 * n3;
        A.zout = z + (size_t)r0 * n3;
        A.V = V;
        A.Q = Qb;
        A.Gv = Gv;
        A.Zv = Zv;
        A.ctr = ctr;
        A.err = h->dev_err;
        A.nrhs = nr;
        A.R8 = dense_r8(nr);
        A.nclus = h->dclus;
        A.nsteps = (2 * B - 1) * (inner_steps(B, h->g.cen, h->g.sched == HELM_TWO_FRONT) + 1) + 1;
        A.DZ = dense_dz(h);
        A.wait_cycles = h->opts.wait_cycles;
        A.unmet = h->opts.debug_unmet_wait;
        cudaError_t e = cudaMemsetAsync(ctr, 0, sizeof(unsigned), st);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = HELM_DENSE_CS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(HELM_DENSE_CS * h->dclus, 1, 1);
        cfg.blockDim = dim3(DT, 1, 1);
        cfg.dynamicSmemBytes = h->dsmem;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        void* args[] = {&A};
        e = cudaLaunchKernelExC(&cfg, kfn, args);
        if (e != cudaSuccess) return e;
        h->launches++;
    }
    return cudaSuccess;
}

int dense_rebuild(helm_ctx* h, int Ma, int Mb, int Pa, int Pb, cudaStream_t st) {
    if (!h->dense || !h->prob_h || !h->dprob_h) return HELM_EINVAL;
    return dense_build(h, h->prob_h, Ma, Mb, Pa, Pb, st);
}

void dense_free(helm_ctx* h) {
    void* ptrs[] = {h->dprob, h->tprob, h->dG, h->dscale, h->dlo, h->dV};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete[] h->dprob_h;
    delete[] h->tprob_h;
    h->tprob = nullptr;
    h->tprob_h = nullptr;
    h->dprob = nullptr;
    h->dprob_h = nullptr;
    h->dG = nullptr;
    h->dscale = nullptr;
    h->dlo = nullptr;
    h->dV = nullptr;
}

extern "C" int helm_dense_operator(helm_handle h, int M, int Mp, int dir, int* n_out, int* n_in, int* rects,
                                   void* G, void* stream) {
    if (!h || h->nsub || !h->dense) return HELM_ENOTSUP;
    const int B = h->g.B;
    if (M < 0 || M >= B || Mp < 0 || Mp >= B || dir < 0 || dir > 1) return HELM_EINVAL;
    if (dir == 1 && Mp != 0 && !(h->g.sched == HELM_TWO_FRONT && Mp == B - 1)) return HELM_EINVAL;
    const int p = op_index(M, op_slot(Mp, dir, B), B);
    const DProb& D = h->dprob_h[p];
    if (n_out) *n_out = D.n_out;
    if (n_in) *n_in = D.n_in;
    if (rects) {
        // [nrect, in(4), out0(4), out1(4)]
        rects[0] = D.nrect;
        const DRect rs[3] = {D.in, D.out[0], D.nrect > 1 ? D.out[1] : DRect{0, 0, 0, 0}};
        for (int q = 0; q < 3; ++q) {
            rects[1 + 4 * q] = rs[q].line0;
            rects[2 + 4 * q] = rs[q].nl;
            rects[3 + 4 * q] = rs[q].z0;
            rects[4 + 4 * q] = rs[q].nz;
        }
    }
    if (!G) return HELM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    if (h->opts.precision == HELM_FP32) {
        k_dense_unpack<<<512, 256, 0, st>>>(D, h->dG, (float2*)G);
        h->launches++;
        e = cudaGetLastError();
    } else {
        e = team_unpack(h, p, (float2*)G, st);
    }
    if (e != cudaSuccess) {
        helm_set_cuda_error(e);
        return HELM_ECUDA;
    }
    return HELM_OK;
}
