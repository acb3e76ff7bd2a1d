// Tensor-core apply of the dense restricted-operator form (HELM_SPLIT_FP16 and
// HELM_FP16; the operators and what they map are described in dense.cu).
//
// Right-hand sides are independent, and in Algorithm 4 everything but a solve's
// input vector is local to one (x, z) column of the slab: the couplings and the
// updates join values of the same column on neighbouring lines.  So a group of
// RG <= 16 right-hand sides is swept by a team of C CTAs of its own (with two
// fronts by two teams, one per front), each rank owning a share of the columns
// for the whole slab visit.  A solve then needs one exchange: every rank gathers
// the whole input vector (K entries x RG), multiplies it by its own rows of G on
// the tensor core, and applies the update to its own columns.  No partial sums
// cross CTAs, and groups never wait for one another.
//
// What bounds it: the latency of one solve, i.e. epilogue -> publish -> gather ->
// product, 33 thousand times in a row at n = 127.  Measured on GB300 (cycles at 2.07
// GHz): bulk copies from L2 land 550 cycles after their issue and stream at about
// 60 B/clk on every SM at once; distributed shared memory moves 20 B/clk, so an
// all-gather of 27 kB takes 1.9 k cycles there, and of 55 kB 3.1 k; publishing
// through L2 takes about 1.2 k plus the bulk copy, whatever the group's size.  Hence
// the exchange goes through L2.  One apply, split FP16, two fronts: n = 127 with 64
// right-hand sides 314 ms (K split over clusters of 8, partial sums through
// distributed shared memory and one step counter for all CTAs: 16.7 k cycles a
// solve) -> 191 ms; n = 63 with one 57.8 -> 41.5 ms; one front, n = 50 with 33,
// FP16 operators 104 -> 62 ms.
//
// Exchange.  q is published as FP16 hi + lo parts in the layout of the tensor
// core's B operand (N-major core matrices), so a gather is a plain bulk copy into
// shared memory, and the product starts when its first half has landed.  The
// power-of-two scale of a right-hand side has to be known before the parts are
// formed: it comes from the largest entry of the solve before and of the slab
// right-hand side on the next line (a table made in the boundary phase), with
// room for a growth by 2^7; entries down to 2^-10 of that maximum keep both parts in
// full, smaller ones an absolute error of 2^-33 of it.  So an input that shrinks by 2^k
// against what its scale comes from loses k bits more.  A rank whose entries do
// not fit (they grew more) scales them by their own maximum and says so in the
// header of the 8 entries; a gather that finds unequal scales brings them to the
// smallest in shared memory before the product (in FP16: the same absolute error).
//
// Headers carry the solve's number and are released at GPU scope after the parts; the
// gathering warp reads them until they are all there, fences (acquire, and a proxy
// fence, for bulk copies are another proxy), and only then copies the parts.  A slot is written again NRING ring solves later: whoever does that
// has read headers of the solves between, which their ranks stored after they had
// multiplied, hence gathered, the slot's input.
//
// Per CTA: eight warps apply the updates, one warp issues the products, one
// streams the operator through a ring, one polls headers and gathers.  The loops
// that run every solve are kept small and straight (the instruction cache holds 32
// kB; code beyond it runs at a third of the rate and branchy code worse): solves of
// one line in one tile run in run_lines, of 2 or 4 lines or of several tiles in
// run_blocks, every other one in run_general.
// All waits are bounded; on expiry the error word is set, copies and products in
// flight are drained, TMEM is freed and the kernel returns.
#include "helm_internal.h"
#include "ptx.cuh"

#include <cuda_fp16.h>
#include <string.h>

#include <algorithm>
#include <vector>

namespace {

#include "dense_sched.h"
#include "team_map.h"

typedef unsigned long long u64;

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float4 cmul2(float2 c, float4 v) {
    return make_float4(c.x * v.x - c.y * v.y, c.x * v.y + c.y * v.x, c.x * v.z - c.y * v.w, c.x * v.w + c.y * v.z);
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 sub4(float4 a, float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}

// Exponent of the power-of-two scale that puts a largest magnitude f 2^ex
// (f in [0.5, 1)) into [2^14, 2^15), clamped to normal FP32 scales.
__host__ __device__ __forceinline__ int scale_exp(int ex) {
    const int e = 15 - ex;
    return e < -120 ? -120 : (e > 120 ? 120 : e);
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }
// v 2^t for |t| <= 250, in two exact steps of like size: no intermediate leaves
// the FP32 range unless the result does.
__device__ __forceinline__ float scale2(float v, int t) {
    const int h = t >> 1;
    return v * pow2f(h) * pow2f(t - h);
}

// ------------------------------------------------------------ stored operators

struct PackItem { int p, gr; };

// One row group (8 complex rows) of operator p, from its complex FP32 rows in Gt
// (dense.cu's entry order) into the chunks of team_map.h, with one power-of-two
// scale per real row.  In the FP16 form an operator with xr > 0 keeps hi parts alone
// but for the last xr of every 64 + xr rows, whose groups have lo parts (lo: which).
__global__ void __launch_bounds__(128)
k_team_pack(const TProb* __restrict__ tp, const PackItem* __restrict__ items, const float2* __restrict__ Gt,
            const long long* __restrict__ goff, unsigned char* __restrict__ G, float* __restrict__ scale, const int* __restrict__ lo,
            int N) {
    __shared__ int s_row[8];
    __shared__ float s_sc[16];
    const PackItem I = items[blockIdx.x];
    const TProb D = tp[I.p];
    const float2* src = Gt + goff[I.p];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ng = D.ng0 + D.ng1, n_in = D.n_in, KP = D.KP, halves = D.halves;
    if (tid < 8) {
        const int q = I.gr >= D.ng0;
        const DRect R = D.out[q];
        const int i = 8 * (I.gr - (q ? D.ng0 : 0)) + tid, n = R.nl * R.nz * N;
        int o = -1;
        if (i < n) {
            const int l = i % R.nl, t = i / R.nl, zr = t % R.nz, x = t / R.nz;
            o = (q ? D.out[0].nl * D.out[0].nz * N : 0) + x + N * (zr + R.nz * l);
        }
        s_row[tid] = o;
    }
    __syncthreads();
    for (int rr = warp; rr < 16; rr += 4) {
        const int part = rr >> 3, o = s_row[rr & 7];
        float mx = 0.f;
        if (o >= 0)
            for (int j = lane; j < n_in; j += 32) {
                const float2 v = src[(size_t)o * n_in + j];
                mx = fmaxf(mx, fabsf(part ? v.y : v.x));
            }
        for (int s = 16; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
        if (lane == 0) {
            float sc = 1.f;
            if (mx > 0.f) {
                int ex;
                frexpf(mx, &ex);
                sc = ldexpf(1.f, scale_exp(ex));
            }
            s_sc[rr] = sc;
            scale[D.soff + (long long)I.gr * 16 + rr] = sc;
        }
    }
    __syncthreads();
    unsigned char* dst = G + D.off;
    const int nli = D.in.nl, nzi = D.in.nz;
    for (int e = tid; e < 8 * (KP / 8); e += 128) {
        const int row = e & 7, k8 = e >> 3, c = (8 * k8) / TKC;
        const int kc = min(TKC, KP - c * TKC), kk = 8 * k8 - c * TKC;
        const int o = s_row[row];
        const bool hi_only = D.xr > 0 && o % (64 + D.xr) < 64;
        __align__(16) __half hi[2][8], lw[2][8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = 8 * k8 + u;
            float2 z = make_float2(0.f, 0.f);
            if (o >= 0 && k < n_in) {
                const int l = k % nli, t = k / nli, zr = t % nzi, x = t / nzi;
                z = src[(size_t)o * n_in + zr + nzi * (l + nli * x)];
            }
            const float v[2] = {z.x * s_sc[row], z.y * s_sc[8 + row]};
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                hi[p][u] = __float2half_rn(v[p]);
                lw[p][u] = __float2half_rn(hi_only ? 0.f : v[p] - __half2float(hi[p][u]));
            }
        }
        int bytes;
        const int idx = D.nlo ? lo[D.lob + I.gr] : 0;
        const size_t bh = D.nlo ? tm_unit(c, I.gr, ng + D.nlo, KP) : tm_tile(c, 0, I.gr, ng, KP, halves, &bytes);
        const size_t pos = (size_t)(kk >> 3) * 128 + row * 16;
#pragma unroll
        for (int p = 0; p < 2; ++p)
            *reinterpret_cast<uint4*>(dst + bh + (size_t)p * kc * 16 + pos) = *reinterpret_cast<const uint4*>(hi[p]);
        if (halves == 2 && idx >= 0) {
            const size_t bl = D.nlo ? tm_unit(c, ng + idx, ng + D.nlo, KP) : tm_tile(c, 1, I.gr, ng, KP, halves, &bytes);
#pragma unroll
            for (int p = 0; p < 2; ++p)
                *reinterpret_cast<uint4*>(dst + bl + (size_t)p * kc * 16 + pos) =
                    *reinterpret_cast<const uint4*>(lw[p]);
        }
    }
}

// Reads one stored operator back as complex FP32 [n_out][n_in] in dense.cu's
// entry order (for tests).
__global__ void k_team_unpack(TProb D, const unsigned char* __restrict__ G, const float* __restrict__ scale,
                              const int* __restrict__ lo, int N, float2* __restrict__ out) {
    const int ng = D.ng0 + D.ng1;
    const int n0 = D.out[0].nl * D.out[0].nz * N;
    const long long total = (long long)D.n_out * D.n_in;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(e / D.n_in), j = (int)(e - (long long)o * D.n_in);
        const int q = o >= n0;
        const DRect R = D.out[q];
        int t = o - (q ? n0 : 0);
        const int x = t % N;
        t /= N;
        const int i = (x * R.nz + t % R.nz) * R.nl + t / R.nz;
        const int gr = (q ? D.ng0 : 0) + (i >> 3), row = i & 7;
        const int per = D.in.nz * D.in.nl, xi = j / per, r = j - xi * per;
        const int k = (xi * D.in.nz + r % D.in.nz) * D.in.nl + r / D.in.nz;
        const int c = k / TKC, kc = min(TKC, D.KP - c * TKC), kk = k - c * TKC;
        int bytes;
        const int idx = D.nlo ? lo[D.lob + gr] : 0;
        const size_t bh = D.nlo ? tm_unit(c, gr, ng + D.nlo, D.KP) : tm_tile(c, 0, gr, ng, D.KP, D.halves, &bytes);
        const size_t bl = D.nlo ? tm_unit(c, ng + max(idx, 0), ng + D.nlo, D.KP) : tm_tile(c, 1, gr, ng, D.KP, D.halves, &bytes);
        float part[2];
        for (int p = 0; p < 2; ++p) {
            const size_t pos = (size_t)p * kc * 16 + (size_t)(kk >> 3) * 128 + row * 16 + (kk & 7) * 2;
            float v = __half2float(*reinterpret_cast<const __half*>(G + D.off + bh + pos));
            if (D.halves == 2 && idx >= 0) v += __half2float(*reinterpret_cast<const __half*>(G + D.off + bl + pos));
            part[p] = v / scale[D.soff + (long long)gr * 16 + p * 8 + row];
        }
        out[e] = make_float2(part[0], part[1]);
    }
}

// ---------------------------------------------------------------------- apply

constexpr int CW = 8;                       // update warps
constexpr int MMA_WARP = 8, RING_WARP = 9, GATHER_WARP = 10;
constexpr int TT = 32 * 11;                 // threads of a CTA
constexpr int MAXST = 16;                   // most ring stages
constexpr int NBC = 2;                      // parts a gather is split into
// Accumulators of a tile in TMEM: its 512 columns over products of 64 rows by 4 RG columns
// (more than 8 would only stretch the read-out).
__host__ __device__ constexpr int acc_slots(int RG, int MT) { return RG == 16 && MT == 128 ? 4 : 8; }
constexpr long long TEAM_WAIT = 4000000000ll;   // about 2 s at 2 GHz

struct TeamArgs {
    Geom g;
    const AxisWin* win;
    const TProb* tp;
    const unsigned char* G;
    const float* scale;
    const int* lo;          // FP16 form: a chunk's unit of zeros, then the numbers of the groups' lo parts (-1: none)
    const float2* c_dn;
    const float2* c_up;
    const float2* rin;
    float2* zout;
    float2* V;              // [group][line][column e][RG]  forward values of the current slab
    float2* Gv;             // [group][line][x dz + zr][RG] the slab's right-hand side on its own layers
    float2* Zv;             // the same layout: the slab's restricted result
    float2* Qf;             // [group][4][e][RG] couplings kept in FP32: lower and upper front into the centre, per team
    unsigned char* X;       // [group][team] published inputs: SLOT_START slots of slot_bytes, one of start_bytes
    u64* hdr;               // [group][team] their headers: SLOT_START of hdr_words, one of start_words
    unsigned* gmax;         // [group][2][line][RG] largest |Gv| of a line (float bits), by visit parity
    unsigned* ctr;          // [group] barrier counters, 128 bytes apart
    int* err;
    size_t slot_bytes, start_bytes;
    int hdr_words, start_words;
    int nrhs, T, C;
    int DZ, Emax, KB;       // KB: input entries a gather pass holds (multiple of TKC)
    int stages, stage_bytes;
    int off_b, off_misc;    // shared memory: the B operand, the rest (the ring starts at 0)
    long long wait_cycles;
    int unmet;
};

// Bounded wait of a warp on an mbarrier phase; gives up at the cycle limit or when
// the CTA has been aborted.  Every lane polls and votes, and the first try stands
// before the loop: 80 cycles on a completed phase and 109 from the arrival to the
// return, against 247 and 268 with one polling lane in a branch of its own.  And the
// compiler sees the caller's control flow as uniform: the products issue at 33
// cycles each, with a divergent wait (or a warp index it cannot prove uniform)
// before them at 100 to 600.
__device__ __forceinline__ bool wait_phase(uint64_t* bar, uint32_t ph, long long limit, volatile int* abort_) {
    if (__all_sync(0xffffffffu, ptx::mbar_try(bar, ph))) return true;
    const long long t0 = clock64();
    for (;;) {
        if (__all_sync(0xffffffffu, ptx::mbar_try(bar, ph))) return true;
        if (__any_sync(0xffffffffu, clock64() - t0 > limit || *abort_)) return false;
    }
}

// K = 16 steps of a part of a gather of n16 steps: whole operator chunks, so that a
// chunk never waits for two parts.
__device__ __forceinline__ int gather_part(int n16) {
    constexpr int U = TKC / 16;
    return (n16 + NBC * U - 1) / (NBC * U) * U;
}

// An accumulator's rows of a thread, for one pair of right-hand sides: of the row in
// lane t/4 its real parts, 8 lanes on its imaginary parts, times q's re hi, im hi, re
// lo, im lo (8 columns each); with split operators the products of their lo parts with
// q's hi parts 16 lanes further on.
struct AccRows {
    float h[4][4], l[2][4];
};
__device__ __forceinline__ void load_rows(uint32_t ta, bool split, AccRows& v) {
    ptx::tmem_ld16x32(ta, v.h);
    if (split) ptx::tmem_ld16x16(ta + (16u << 16), v.l);
}
// Adds them to R and I after the wait.  The accumulators cover successive runs of the
// input (Shape) and are added here in rounded FP32: the tensor core's own additions do
// not round to nearest, and the error of an apply grows with their chain.
__device__ __forceinline__ void add_rows(AccRows& v, bool split, float (&R)[4], float (&I)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) ptx::reg_tie4(v.h[q]);
    if (split) {
#pragma unroll
        for (int q = 0; q < 2; ++q) ptx::reg_tie4(v.l[q]);
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            ptx::add2(v.h[2] + q, v.l[0] + q);
            ptx::add2(v.h[3] + q, v.l[1] + q);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
        ptx::add2(v.h[0] + q, v.h[2] + q);
        ptx::add2(v.h[1] + q, v.h[3] + q);
        ptx::add2(R + q, v.h[0] + q);
        ptx::add2(I + q, v.h[1] + q);
    }
}

// Y = G q from the sums.  er, ei: exponents of the row's scales; c0, c1: of the columns'.
__device__ __forceinline__ float4 scale_rows(const float (&R)[4], const float (&I)[4], int er, int ei, int c0, int c1) {
    const int a0 = -(er + c0), a1 = -(er + c1), b0 = -(ei + c0), b1 = -(ei + c1);
    const int lo = min(min(a0, a1), min(b0, b1)), hi = max(max(a0, a1), max(b0, b1));
    if (__any_sync(0xffffffffu, lo < -126 || hi > 127))          // far from one: in two steps
        return make_float4(scale2(R[0], a0) - scale2(I[2], b0), scale2(I[0], a0) + scale2(R[2], b0),
                           scale2(R[1], a1) - scale2(I[3], b1), scale2(I[1], a1) + scale2(R[3], b1));
    const float fa0 = pow2f(a0), fa1 = pow2f(a1), fb0 = pow2f(b0), fb1 = pow2f(b1);
    return make_float4(R[0] * fa0 - I[2] * fb0, I[0] * fa0 + R[2] * fb0, R[1] * fa1 - I[3] * fb1, I[1] * fa1 + R[3] * fb1);
}

// 2^d (d <= 0) as FP16 bits; 0 below the subnormal range.
__device__ __forceinline__ unsigned half_pow2(int d) {
    return d >= -14 ? (unsigned)(15 + d) << 10 : (d >= -24 ? 1u << (24 + d) : 0u);
}

// The products of one operator chunk (kc <= TKC input entries): one per 16 entries
// and 4 row groups, all of one shape (only then do products into the same
// accumulator keep their order).  With split operators a group's hi and lo rows
// stand in the same product (128 rows: re hi, im hi, re lo, im lo of each group), which
// takes 38 cycles where a 64-row product for hi and one for lo take 65; without, 64
// rows.  One elected lane of the converged warp issues them; a full chunk is
// straight-line code: a condition around each, even a uniform one, made a product
// take 70 to 85 cycles to issue instead of 33.  rsh: an accumulator takes 1 << rsh
// products, or (2) whole chunks; add: the chunk goes on with its accumulator.
template <int RG, int NSUB>
__device__ __forceinline__ void chunk_products(uint32_t d, uint64_t ad, uint32_t sub, uint64_t bd, uint32_t idesc, uint32_t add,
                                               int rsh, int kc) {
    constexpr int BSTEP = 2 * 64 * RG / 16, ASTEP = 256 / 16, SUBC = acc_slots(RG, 64 * NSUB) * 4 * RG;
    const uint32_t mask = (1u << rsh) - 1u;
    if (kc == TKC) {
#pragma unroll
        for (int ks = 0; ks < TKC / 16; ++ks)
#pragma unroll
            for (int u = 0; u < NSUB; ++u)
                ptx::umma_f16_warp(d + ((uint32_t)ks >> rsh) * (4 * RG) + u * SUBC, ad + ks * ASTEP + u * sub, bd + ks * BSTEP, idesc,
                                   ks == 0 ? add : ks & mask);
        return;
    }
#pragma unroll 1
    for (int ks = 0; 16 * ks < kc; ++ks) {
#pragma unroll
        for (int u = 0; u < NSUB; ++u)
            ptx::umma_f16_warp(d + ((uint32_t)ks >> rsh) * (4 * RG) + u * SUBC, ad + ks * ASTEP + u * sub, bd + ks * BSTEP, idesc,
                               ks == 0 ? add : ks & mask);
    }
}

// What the roles of a CTA need to know of a solve's shape.  A visit has four kinds
// of solves (the first, those of the ring, the centre, the last); each role keeps
// the four records of its current visit in shared memory, made once per visit, so
// that the step loops carry no index divisions (inlined in every role they made
// the code larger than the instruction caches: 258 kB and 5 to 8 cycles per
// instruction).
//
// An accumulator takes a run of products, rounded down to 1, 2 or a multiple of 4 so that
// runs and chunks end together: a quarter of the input's, 2 up to 14 products, and at most
// 8 or an eighth.  With FP16 operators 2 up to 16 products and 4 up to 32: what they lose in
// the chain is the only difference from eight partial sums, and adds up over the solves (n
// = 111, two fronts, b_aux 1, 16 products: runs of 4 moved results by 1.3e-5, locally 3.3e-4;
// runs of 2 by 1.5e-6).  The products signal a few accumulators at a time, a unit: those of a
// chunk, or two, or one where there are at most four.  Before the teams every input went
// into eight partial sums; error of a split FP16 apply against 64 bits then, with an
// accumulator for every chunk or more, and now: n = 33, two fronts, b_aux 1 (6 products)
// 6.4e-6, 8.0e-6, 4.6e-6; n = 31, one front, b_aux 4 (14) 4.3e-6, 4.5e-6, 3.9e-6; n = 50, one
// front, b_aux 3 (16) 8.9e-6, 8.5e-6, 8.5e-6; the same with d = 2 (39) 8.1e-6, 6.7e-6, 6.4e-6.
// Reading an accumulator costs a warp 150 cycles or more: runs of an eighth for all give n
// = 50 6.0e-6 in 64.8 ms instead of 60.2 and n = 63 with one right-hand side 43.2 ms instead of
// 40.6; at 27 products runs of 8 gave n = 127 9.4e-6 in 188.5 ms, those of 4 5.4e-6 in 190.6.
enum { KIND_START = 0, KIND_RING = 1, KIND_CENTRE = 2, KIND_END = 3 };
struct Shape {
    int K, KP;                    // input entries, padded to a multiple of 16
    int rsh, cpa, nu, w, wl;      // chunk_products' rsh, chunks of an accumulator, units of a tile, accumulators of each and of the last
    int a0, c0, a1, c1;           // this rank's row groups [a, a + c) of the two out rects
    int ng0, ng, nt, kg0;         // row groups of rect 0 and of the operator, tiles, first own input group
    int kg1, nl, nz, z0;          // end of the own input groups; the in rect's lines, z rows and first row
    int halves, nlo, lob;         // 2: the operator has lo parts; nlo > 0: of that many groups (table at lob)
};
__device__ __forceinline__ int kind_of(int i, int nsol, int cen, int upper) {
    return i == 0 ? KIND_START : (i == nsol - 1 ? KIND_END : (!upper && i == cen ? KIND_CENTRE : KIND_RING));
}

__device__ __noinline__ void make_shapes(Shape* out, const AxisWin* win, const TProb* tp, int N, int B, int cen, int two, int upper,
                                         int M, int rank, int C, int GT, int lane) {
    __syncwarp();
    if (lane < 4) {
        const int nsol = tm_solves(B, cen, upper);
        // a solve of this kind (kinds a visit does not have get the first solve's record)
        int i = lane == KIND_START ? 0 : (lane == KIND_END ? nsol - 1 : (lane == KIND_CENTRE ? cen : (!upper && cen == 1 ? 2 : 1)));
        if (kind_of(i, nsol, cen, upper) != lane) i = 0;
        const TeamSolve t = tm_solve(i, B, cen, upper);
        const SolveGeo g = tm_geo(win[M], win[t.Mp], N, t.Mp, t.bwd, B, two);
        Shape s;
        s.K = g.K;
        s.KP = tm_kp(g.K);
        int hi;
        tm_part(g.n0, g.out0.nl, g.f0, rank, C, &s.a0, &hi);
        s.c0 = hi - s.a0;
        s.a1 = s.c1 = 0;
        if (g.nrect > 1) {
            tm_part(g.n1, g.out1.nl, g.f1, rank, C, &s.a1, &hi);
            s.c1 = hi - s.a1;
        }
        s.ng0 = tm_ceil(g.n0, 8);
        s.ng = s.ng0 + tm_ceil(g.n1, 8);
        s.nt = tm_ceil(s.c0 + s.c1, GT);
        const int n16 = s.KP / 16, nch = tm_ceil(s.KP, TKC), q = tm_ceil(n16, 4);
        const TProb& D = tp[op_index(M, op_slot(t.Mp, t.bwd, B), B)];
        const bool fp16 = D.halves == 1 || D.nlo > 0;
        const int run = n16 <= (fp16 ? 16 : 14) ? min(q, 2)
                                                : (fp16 && n16 <= 32 ? 4 : min(q, max(8, tm_ceil(n16, 8))));
        s.rsh = run >= 4 ? 2 : (run > 1 ? 1 : 0);
        s.cpa = max(1, run / 4);
        const int na = run >= 4 ? tm_ceil(nch, s.cpa) : tm_ceil(n16, 1 << s.rsh);
        s.w = run == 1 ? 4 : (run >= 4 && na <= 4 ? 1 : 2);
        s.nu = s.nt > 0 ? tm_ceil(na, s.w) : 1;
        s.wl = na - (tm_ceil(na, s.w) - 1) * s.w;
        tm_part(g.K, g.in.nl, g.fin, rank, C, &s.kg0, &s.kg1);
        s.nl = g.in.nl;
        s.nz = g.in.nz;
        s.z0 = g.in.z0;
        s.halves = D.halves;
        s.nlo = D.nlo;
        s.lob = D.lob;
        out[lane] = s;
    }
    __syncwarp();
}

// Shared memory of a CTA after the ring and the B operand; the tables behind it
// are reached through its pointers.
struct Sm {
    uint64_t full[MAXST];        // operator chunk landed
    uint64_t empty[MAXST];       // operator chunk consumed
    uint64_t bfull[NBC];         // part of the gather landed
    uint64_t bgo;                // a gather pass may be multiplied
    uint64_t eready;             // its scale exponents are in shared memory
    uint64_t mdone;              // its products are complete
    uint64_t sacc[8];            // a unit's products are complete, by its place in TMEM
    uint64_t afree[8];           // its accumulators have been read (CW arrivals), where another unit of the tile follows
    uint64_t sdone;              // a tile's products are complete (stands for its last unit)
    uint64_t tfree;              // its accumulators have been read (CW arrivals)
    uint64_t cbar;               // barrier of the update warps (CW arrivals)
    uint64_t xbar;               // teardown
    uint32_t tslot;
    volatile int abort;
    int ecol[16];                // scale exponents of the gathered input
    int epred[16];               // scale exponents of the next input
    Shape shape[12];             // [3 users][4 kinds]: ring, gather and products, update warps
    long long limit;
    int N, B, cen, two, U, C, grp, team, rank, nsol;
    int VL, GL;                  // line strides of V and of Gv, Zv (float2)
    float2 *V, *Gv, *Zv, *Qf;    // this group's fields
    unsigned* gm;
    unsigned* ctr;
    unsigned char* X;            // this team's published inputs and headers
    u64* H;
    size_t Xteam, Hteam;         // and the strides to the next team's
    unsigned char* Bbuf;
    float2 *cdn, *cup;           // [N] couplings of the operator
    long long *soff, *off;       // [B + 2] scale offsets of the visit's operators; tile offsets of the ring's
    AxisWin* win;                // [B]
};

// An update warp's place in the barriers' phases.
struct Upd {
    uint32_t sph, cph, xph;      // sph: a parity bit per place of a unit, bit 8 for sdone
    unsigned arrivals, tag;      // tag: number of the solve, from 1
};

// The warp that publishes group gi of the rank, right-hand sides
// 8 pcb ..: the one whose accumulator rows they are in a one-tile solve, so that an
// entry's words stay with one warp.
template <int RG, int MT>
__device__ __forceinline__ int warp_of(int gi, int pcb) {
    if (RG == 16) return (gi & 3) + 4 * pcb;
    return MT == 64 ? gi & 3 : gi & 7;
}
// Where a lane's part of a row lies in its group of 8 entries, for right-hand sides
// 8 pcb ..: part lane mod 4 (re hi, im hi, re lo, im lo) of row lane / 4.  A block of
// right-hand sides has its four parts side by side, 32 accumulator columns for one load.
__device__ __forceinline__ int part_offset(int pcb, int lane) { return (pcb * 4 + (lane & 3)) * 128 + (lane >> 2) * 16; }
__device__ __forceinline__ void fail(const TeamArgs& A, Sm& S) {
    if (!S.abort) atomicOr(A.err, 2);
    S.abort = 1;
}

// Stores one row's value for two right-hand sides: FP16 hi and lo parts, scaled by
// 2^e0 and 2^e1.  The four lanes of a row trade their words so that each stores one
// part of the row for 8 right-hand sides (16 bytes, at p).  Returns the value half of
// the lane's header word (lanes 0..3: those of the 8 entries).
__device__ __forceinline__ unsigned store_parts(unsigned char* p, float4 v, int e0, int e1) {
    const int lane = threadIdx.x & 31;
    unsigned m = max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))) >> 23 |
                 max(__float_as_uint(fabsf(v.z)), __float_as_uint(fabsf(v.w))) >> 23 << 16;
#pragma unroll
    for (int s = 4; s < 32; s <<= 1) m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, s));
    const int f0 = (int)(m & 0xffffu), f1 = (int)(m >> 16);
    if (f0 - 126 + e0 > 15) e0 = scale_exp(f0 - 126);          // grew out of the predicted range
    if (f1 - 126 + e1 > 15) e1 = scale_exp(f1 - 126);
    const float s0 = pow2f(e0), s1 = pow2f(e1);
    const float re0 = v.x * s0, im0 = v.y * s0, re1 = v.z * s1, im1 = v.w * s1;
    const __half2 hr = __floats2half2_rn(re0, re1), hm = __floats2half2_rn(im0, im1);
    const float2 fr = __half22float2(hr), fm = __half22float2(hm);
    const __half2 lr = __floats2half2_rn(re0 - fr.x, re1 - fr.y), lm = __floats2half2_rn(im0 - fm.x, im1 - fm.y);
    const unsigned w0 = *reinterpret_cast<const unsigned*>(&hr), w1 = *reinterpret_cast<const unsigned*>(&hm);
    const unsigned w2 = *reinterpret_cast<const unsigned*>(&lr), w3 = *reinterpret_cast<const unsigned*>(&lm);
    const bool c0 = lane & 1, c1 = lane & 2;
    const unsigned r0 = __shfl_xor_sync(0xffffffffu, c0 ? w0 : w1, 1), r1 = __shfl_xor_sync(0xffffffffu, c0 ? w2 : w3, 1);
    const unsigned px = c0 ? r0 : w0, py = c0 ? w1 : r0, qx = c0 ? r1 : w2, qy = c0 ? w3 : r1;
    const unsigned rx = __shfl_xor_sync(0xffffffffu, c1 ? px : qx, 2), ry = __shfl_xor_sync(0xffffffffu, c1 ? py : qy, 2);
    __stcg(reinterpret_cast<uint4*>(p), make_uint4(c1 ? rx : px, c1 ? ry : py, c1 ? qx : rx, c1 ? qy : ry));
    return (unsigned)(f0 | (e0 + 128) << 8 | f1 << 16 | (e1 + 128) << 24);
}
// The header words of a warp's parts, after a __syncwarp that orders the other lanes'
// parts before: released, or relaxed behind the warp's own release fence.  One apply,
// two fronts, n = 127 with 64 right-hand sides: 182 ms with releasing stores, 190 ms
// with a release fence, 207 ms with acquire-release fences here and at the gather.
__device__ __forceinline__ void release_header(u64* hd, unsigned w, unsigned tag) {
    const int lane = threadIdx.x & 31;
    if (lane < 4) ptx::st_release_gpu_u64(hd + lane, (u64)tag << 32 | w);
}
__device__ __forceinline__ void store_header(u64* hd, unsigned w, unsigned tag) {
    const int lane = threadIdx.x & 31;
    if (lane < 4) ptx::st_relaxed_gpu_u64(hd + lane, (u64)tag << 32 | w);
}

// A warp's rows of a tile: the sum of its accumulators, read as their units complete
// while the next ones are multiplied.  fv: whether the warp has rows (the second group's
// sums are of no use where it does not exist).
template <int RG, int MT, int NRS>
__device__ __forceinline__ bool read_tile(Sm& T, Upd& u, const Shape& S, uint32_t tlane, bool split, bool fv,
                                          float (&R)[NRS][4], float (&I)[NRS][4]) {
    constexpr int SLOTS = acc_slots(RG, MT), SUBC = SLOTS * 4 * RG;
    const int nu = S.nu, w = S.w, NU = SLOTS >> (w >> 1);
    int s = 0;
#pragma unroll 1
    for (int a = 0; a < nu; ++a) {
        const bool last = a == nu - 1;
        const int b = last ? 8 : s;
        if (!wait_phase(last ? &T.sdone : &T.sacc[s], u.sph >> b & 1u, T.limit, &T.abort)) return false;
        u.sph ^= 1u << b;
        ptx::tc_fence_after();
        const int n = last ? S.wl : w;
        __syncwarp();                                // the TMEM loads are warp-collective
        if (fv)
#pragma unroll 1
            for (int v = 0; v < n; ++v)
#pragma unroll
                for (int j = 0; j < NRS; ++j) {
                    AccRows t;
                    load_rows(tlane + (s * w + v) * 4 * RG + j * SUBC, split, t);
                    ptx::tmem_wait_ld();
                    add_rows(t, split, R[j], I[j]);
                }
        if (a + NU < nu) {
            ptx::tc_fence_before();
            __syncwarp();
            if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(&T.afree[s]);
        }
        if (++s == NU) s = 0;
    }
    return true;
}

// Boundary of slab visits jo-1 and jo (Algorithm 6).
// The previous visit's result goes to z (a backward visit subtracts its correction);
// then the new visit's right-hand side on its own layers: forward, f minus the couplings
// of the neighbours already swept; backward, the coupling of the neighbour its pass
// comes from.  Each thread owns whole (line, x, right-hand side) columns, so it reads
// what it wrote.
template <int RG>
__device__ __noinline__ void boundary_phase(const TeamArgs& A, Sm* T, int jo) {
    const int N = T->N, B = T->B, cen = T->cen, grp = T->grp, GL = T->GL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool cur = jo < 2 * B - 1;
    const PassPos vp = jo > 0 ? pass_pos(jo - 1, B, cen) : PassPos{0, 0, 0};
    const PassPos vc = cur ? pass_pos(jo, B, cen) : PassPos{0, 0, 0};
    const AxisWin* win = T->win;
    const float2 *cdn = T->cdn, *cup = T->cup;
    float2* Gp = T->Gv;
    const float2* Zp = T->Zv;
    unsigned* gm = T->gm;
    const AxisWin wp = win[vp.M], wc = win[vc.M];
    const int dz = wc.ib - wc.ia;
    const int dzp = wp.ib - wp.ia;
    const int mc = wc.lo + wc.ia, ec = wc.lo + wc.ib;
    const bool cpl_lo = cur && (vc.bwd ? vc.role == ROLE_U : (vc.role != ROLE_U && vc.M > 0));
    const bool cpl_hi = cur && (vc.bwd ? vc.role == ROLE_L : (vc.role != ROLE_L && vc.M < B - 1));
    const float sgn = vc.bwd ? 1.f : -1.f;
    const int pv0 = wp.lo + wp.ia, pv1 = wp.lo + wp.ib;
    const bool reg_lo = jo > 0 && mc - 1 >= pv0 && mc - 1 < pv1;
    const bool reg_hi = jo > 0 && ec >= pv0 && ec < pv1;
    const size_t NN = (size_t)N * N;
    const int wid = (T->team * T->C + T->rank) * CW + warp, nw = A.T * T->C * CW;
    const int nxb = (N + 7) >> 3, ntask = N * nxb * (RG / 4);
    // a warp task: 8 x of one line, 4 right-hand sides (whole 32-byte sectors on both sides)
    constexpr int PP = 4;
#pragma unroll 1
    for (int t0 = wid; t0 < ntask; t0 += PP * nw) {
        int gi_[PP], zx[PP], ls[PP], rr[PP];
        size_t zi[PP];
        bool in[PP], live[PP];
        float2 nlo[PP], nhi[PP];
        unsigned gmx[PP];
#pragma unroll
        for (int u = 0; u < PP; ++u) {
            const int t = min(t0 + u * nw, ntask - 1);
            const int rq = t % (RG / 4), r2 = t / (RG / 4);
            ls[u] = r2 / nxb;
            const int x = (r2 - ls[u] * nxb) * 8 + (lane & 7);
            rr[u] = rq * 4 + (lane >> 3);
            in[u] = t0 + u * nw < ntask && x < N;
            live[u] = in[u] && grp * RG + rr[u] < A.nrhs;
            zi[u] = (size_t)(grp * RG + rr[u]) * N * NN + (size_t)ls[u] * N + x;
            gi_[u] = ls[u] * GL + x * dz * RG + rr[u];
            zx[u] = ls[u] * GL + x * dzp * RG + rr[u];
            nlo[u] = nhi[u] = make_float2(0.f, 0.f);
            gmx[u] = 0u;
        }
        if (jo > 0)
#pragma unroll 1
            for (int zr = 0; zr < dzp; ++zr) {
                const int layer = pv0 + zr;
                float2 v[PP], old[PP];
#pragma unroll
                for (int u = 0; u < PP; ++u) {
                    v[u] = old[u] = make_float2(0.f, 0.f);
                    if (live[u]) {
                        v[u] = __ldcg(Zp + zx[u] + zr * RG);
                        if (vp.bwd) old[u] = A.zout[zi[u] + (size_t)layer * NN];
                    }
                }
#pragma unroll
                for (int u = 0; u < PP; ++u) {
                    const float2 nz = vp.bwd ? make_float2(old[u].x - v[u].x, old[u].y - v[u].y) : v[u];
                    if (live[u]) A.zout[zi[u] + (size_t)layer * NN] = nz;
                    if (layer == mc - 1) nlo[u] = nz;
                    if (layer == ec) nhi[u] = nz;
                }
            }
        if (!cur) continue;
#pragma unroll
        for (int u = 0; u < PP; ++u) {
            float2 wl = make_float2(0.f, 0.f), wh = wl;
            if (cpl_lo && live[u]) wl = reg_lo ? nlo[u] : A.zout[zi[u] + (size_t)(mc - 1) * NN];
            if (cpl_hi && live[u]) wh = reg_hi ? nhi[u] : A.zout[zi[u] + (size_t)ec * NN];
            nlo[u] = cmul(cdn[mc], wl);
            nhi[u] = cmul(cup[ec - 1], wh);
        }
#pragma unroll 1
        for (int zr = 0; zr < dz; ++zr) {
            float2 rv[PP];
#pragma unroll
            for (int u = 0; u < PP; ++u)
                rv[u] = (!vc.bwd && live[u]) ? A.rin[zi[u] + (size_t)(mc + zr) * NN] : make_float2(0.f, 0.f);
            const float sl = zr == 0 ? sgn : 0.f, sh = zr == dz - 1 ? sgn : 0.f;
#pragma unroll
            for (int u = 0; u < PP; ++u) {
                float2 gv = rv[u];
                if (zr == 0) gv = make_float2(gv.x + sl * nlo[u].x, gv.y + sl * nlo[u].y);
                if (zr == dz - 1) gv = make_float2(gv.x + sh * nhi[u].x, gv.y + sh * nhi[u].y);
                if (in[u]) Gp[gi_[u] + zr * RG] = gv;
                gmx[u] = max(gmx[u], max(__float_as_uint(fabsf(gv.x)), __float_as_uint(fabsf(gv.y))));
            }
        }
#pragma unroll
        for (int u = 0; u < PP; ++u) {
            unsigned m = in[u] ? gmx[u] : 0u;
            for (int s = 1; s < 8; s <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, s));
            if ((lane & 7) == 0 && m > 0u) atomicMax(gm + ((jo & 1) * N + ls[u]) * RG + rr[u], m);
        }
    }
    // the next visit's table starts at zero (nobody reads it in this visit)
    for (int q = (T->team * T->C + T->rank) * 32 * CW + tid; q < N * RG; q += A.T * T->C * 32 * CW)
        gm[((jo + 1) & 1) * N * RG + q] = 0u;
}

// Updates of a tile of any shape: couplings go through FP32 buffers.
template <int RG, int MT>
__device__ __noinline__ bool general_rows(const TeamArgs& A, Sm* T, Upd* pu, int M, int i, int tl, long long soff,
              uint32_t tmem, int ec0, int ec1) {
    constexpr int GT = MT / 16, NRS = RG == 16 && MT == 128 ? 2 : 1, SUBC = acc_slots(RG, MT) * 4 * RG;
    const int N = T->N, B = T->B, cen = T->cen, two = T->two, U = T->U, team = T->team, VL = T->VL, GL = T->GL;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q4 = warp & 3, hh = warp >> 2, ii = lane >> 2, c = lane & 3;
    const int cb = RG == 16 ? hh : 0, rhs0 = 8 * cb + 2 * c;
    const int gi0 = RG == 8 && MT == 128 ? warp : q4;
    const bool idle = RG == 8 && MT == 64 && hh == 1;
    const uint32_t tlane = tmem + ((uint32_t)(32 * q4) << 16) + 32 * cb + (gi0 >> 2) * SUBC;
    const int nsol = tm_solves(B, cen, team);
    const TeamSolve t = tm_solve(i, B, cen, team);
    const AxisWin wz = T->win[M], wy = T->win[t.Mp];
    const int Lz = wz.L, za = wz.ia, dz = wz.ib - wz.ia, y0 = wy.lo + wy.ia, y1 = wy.lo + wy.ib;
    const int kind = kind_of(i, nsol, cen, team);
    const Shape& S = T->shape[8 + kind];
    const bool more = i + 1 < nsol, centre = kind == KIND_CENTRE;
    const bool into_centre = two && !t.bwd && (team ? i == U - 1 : i == cen - 1);
    float2 *V = T->V + rhs0, *Zv = T->Zv + rhs0, *Qf = T->Qf + rhs0;
    const float2 dn = T->cdn[y1 < N ? y1 : N - 1], up = T->cup[y0 > 0 ? y0 - 1 : 0];
    const float fs = t.bwd || centre ? 1.f : -1.f;
    float2 cf = (t.bwd ? t.role == ROLE_L : t.role != ROLE_L) ? up : dn;
    cf = make_float2(fs * cf.x, fs * cf.y);
    const SolveGeo g = tm_geo(wz, wy, N, t.Mp, t.bwd, B, two);
    const int lc = (t.bwd ? t.role == ROLE_L : t.role != ROLE_L) ? y0 : y1 - 1;   // the line that feeds the next
    float2* qb = Qf + (into_centre ? team : (centre && two ? 0 : 2 + team)) * VL;
    const int p0 = tl * GT + gi0, np = S.c0 + S.c1;
    float R[NRS][4] = {}, I[NRS][4] = {};
    Upd u = *pu;
    const bool ok = read_tile<RG, MT, NRS>(*T, u, S, tlane, S.halves == 2, !idle && p0 < np, R, I);
    *pu = u;
    if (!ok) return false;
    ptx::tc_fence_before();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&T->tfree);
#pragma unroll
    for (int j = 0; j < NRS; ++j) {
        const int pos = p0 + 4 * j;
        if (!idle && pos < np) {                           // the same in the whole warp
            const int rect = pos >= S.c0, gid = rect ? S.a1 + pos - S.c0 : S.a0 + pos;
            const int r = 8 * gid + ii;
            const int nl = rect ? g.out1.nl : g.out0.nl, nz = rect ? g.out1.nz : g.out0.nz;
            const float* sc = A.scale + soff + (long long)((rect ? S.ng0 : 0) + gid) * 16 + ii;
            float4 X = scale_rows(R[j], I[j], (__float_as_int(__ldg(sc)) >> 23) - 127, (__float_as_int(__ldg(sc + 8)) >> 23) - 127,
                                  ec0, ec1);
            if (r < (rect ? g.n1 : g.n0)) {
                const int l = r % nl, tt = r / nl, x = tt / nz;
                const int lz = (rect ? g.out1.z0 : g.out0.z0) + tt - x * nz;
                const int line = (rect ? g.out1.line0 : g.out0.line0) + l, eo = (x * Lz + lz) * RG;
                float4* pv = reinterpret_cast<float4*>(V + line * VL + eo);
                if (t.bwd) X = sub4(__ldcg(pv), X);        // a backward solve is a correction
                else if (!centre) *pv = X;
                if ((t.bwd || centre) && lz >= za && lz < za + dz)
                    *reinterpret_cast<float4*>(Zv + line * GL + (x * dz + lz - za) * RG) = X;
                if (more && line == lc) *reinterpret_cast<float4*>(qb + eo) = cmul2(cf, X);
                if (centre && two && line == y1 - 1)
                    *reinterpret_cast<float4*>(Qf + VL + eo) = cmul2(dn, X);
            }
            __syncwarp();
        }
    }
    return true;
}

// Publishes the rank's entries of an input of the given kind for team T->team + up,
// from FP32 values: the slab's right-hand side (useg) plus the couplings in buffer
// b1 on line l1 and b2 on line l2 of the rect (-1: none), whose first line is l0.
template <int RG, int MT>
__device__ __noinline__ void publish_input(const TeamArgs& A, Sm* T, int jo, int M, int kind, int slot, int up,
                                           unsigned tag, bool useg, int l0, int q1, int l1, int q2, int l2) {
    constexpr int NB = RG / 8, KGB = 64 * RG;
    const int N = T->N, VL = T->VL, GL = T->GL;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ii = lane >> 2, c = lane & 3;
    const AxisWin wz = T->win[M];
    const int Lz = wz.L, za = wz.ia, dz = wz.ib - wz.ia;
    const Shape S = T->shape[8 + kind];
    const float2 *b1 = T->Qf + max(q1, 0) * VL, *b2 = T->Qf + max(q2, 0) * VL;
    unsigned char* xs = T->X + up * T->Xteam + slot * A.slot_bytes;
    u64* hd = T->H + up * T->Hteam + (size_t)slot * A.hdr_words;
    constexpr int PB = 4;                    // groups of 8 entries a warp stores under one fence
    unsigned hw[PB];
    u64* hp[PB];
    int held = 0;
#pragma unroll 1
    for (int t = 0; t < (S.kg1 - S.kg0) * NB; ++t) {
        const int gi = t / NB, pcb = t % NB, kg = S.kg0 + gi;
        if (warp_of<RG, MT>(gi, pcb) != warp) continue;
        const int r0 = 8 * pcb + 2 * c;
        int e0 = T->epred[r0], e1 = T->epred[r0 + 1];
        if (kind == KIND_START) {
            unsigned m0 = 0u, m1 = 0u;
            for (int q = 0; q < S.nl; ++q) {
                const unsigned* pm = T->gm + ((jo & 1) * N + l0 + q) * RG + r0;
                m0 = max(m0, __ldcg(pm));
                m1 = max(m1, __ldcg(pm + 1));
            }
            e0 = min(120, max(-120, 134 - (int)(m0 >> 23)));
            e1 = min(120, max(-120, 134 - (int)(m1 >> 23)));
        }
        const int k = 8 * kg + ii;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < S.K) {
            const int l = k % S.nl, tt = k / S.nl, x = tt / S.nz, lz = S.z0 + tt - x * S.nz;
            const int eo = (x * Lz + lz) * RG + r0;
            if (useg && lz >= za && lz < za + dz)
                v = __ldcg(reinterpret_cast<const float4*>(T->Gv + (l0 + l) * GL + (x * dz + lz - za) * RG + r0));
            if (l == l1) v = add4(v, __ldcg(reinterpret_cast<const float4*>(b1 + eo)));
            if (l == l2) v = add4(v, __ldcg(reinterpret_cast<const float4*>(b2 + eo)));
        }
        const unsigned w = store_parts(xs + (size_t)kg * KGB + part_offset(pcb, lane), v, e0, e1);
#pragma unroll
        for (int q = 0; q < PB; ++q)
            if (q == held) {
                hw[q] = w;
                hp[q] = hd + (kg * NB + pcb) * 4;
            }
        if (++held == PB) {
            __syncwarp();
            ptx::fence_release_gpu();
#pragma unroll
            for (int q = 0; q < PB; ++q) store_header(hp[q], hw[q], tag);
            held = 0;
        }
    }
    if (held > 0) {
        __syncwarp();
        ptx::fence_release_gpu();
#pragma unroll
        for (int q = 0; q < PB; ++q)
            if (q < held) store_header(hp[q], hw[q], tag);
    }
}

// Barrier of the update warps.
__device__ __forceinline__ bool cta_sync(Sm& T, Upd& u, long long limit) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(&T.cbar);
    const bool r = wait_phase(&T.cbar, u.cph, limit, &T.abort);
    u.cph ^= 1u;
    return r;
}

// Barrier of the group's teams (update warps).
__device__ __noinline__ bool group_sync(const TeamArgs& A, Sm* Tp, Upd* up) {
    Sm& T = *Tp;
    Upd u = *up;
    const long long limit = T.limit;
    const int lane = threadIdx.x & 31;
    bool ok = cta_sync(T, u, limit);
    u.arrivals += (unsigned)(A.T * A.C);
    if (ok && threadIdx.x < 32) {
        int good = 1;
        if (lane == 0) {
            ptx::red_release_gpu_add(T.ctr, 1u);
            const unsigned target = A.unmet ? 0xFFFFFFF0u : u.arrivals;
            const long long t0 = clock64();
            while (ptx::ld_acquire_gpu(T.ctr) < target)
                if (clock64() - t0 > limit || T.abort) {
                    good = 0;
                    break;
                }
        }
        if (!__shfl_sync(0xffffffffu, good, 0)) {
            fail(A, T);
            ok = false;
        }
    }
    ok = cta_sync(T, u, limit) && ok;
    *up = u;
    return ok;
}

// Slots a visit uses, the kind of input in each, and the groups of 8 entries (0 or
// 1) that pad such an input to a multiple of 16.
__device__ __forceinline__ unsigned used_slots(int nsol, int cen, int upper) {
    unsigned m = 0u;
    for (int i = 0; i < min(nsol, cen + NRING + 3); ++i) m |= 1u << slot_of_solve(i, nsol, cen, upper);
    return m | 1u << slot_of_solve(nsol - 1, nsol, cen, upper);
}
__device__ __forceinline__ int kind_of_slot(int sl) {
    return sl < NRING ? KIND_RING : (sl == SLOT_CENTRE ? KIND_CENTRE : (sl == SLOT_END ? KIND_END : KIND_START));
}
__device__ __forceinline__ int tail_groups(const Shape& S) { return S.KP / 8 - ((S.K + 7) >> 3); }   // 0 or 1

// A visit's beginning: the result of the visit before and the new right-hand side pass
// through z, the records are made, the entries that pad an input are set to zero, and
// (after the group's barrier) the first input is published.
template <int RG, int MT>
__device__ __noinline__ bool begin_visit(const TeamArgs& A, Sm* Tp, Upd* up, int jo) {
    Sm& T = *Tp;
    const int B = T.B, cen = T.cen, team = T.team, nsol = T.nsol;
    const int tid = threadIdx.x;
    Shape* shapes = T.shape + 8;
    boundary_phase<RG>(A, Tp, jo);
    if (jo == 2 * B - 1) return true;
    const int M = pass_pos(jo, B, cen).M;
    for (int q = tid; q < B + 2; q += 32 * CW) T.soff[q] = A.tp[op_index(M, q, B)].soff;
    Upd u = *up;
    bool ok = cta_sync(T, u, T.limit);                 // everybody is done with the records of the visit before
    *up = u;
    if (tid < 32) {
        make_shapes(shapes, T.win, A.tp, T.N, B, cen, T.two, team, M, T.rank, T.C, MT / 16, tid & 31);
        // the entries that pad an input are the last rank's, zero for the whole visit
        const unsigned slots = T.rank == T.C - 1 ? used_slots(nsol, cen, team) : 0u;
#pragma unroll 1
        for (int sl = 0; sl <= SLOT_START; ++sl) {
            const Shape& S = shapes[kind_of_slot(sl)];
            if ((slots >> sl & 1u) && tail_groups(S))
                for (int q = tid; q < 4 * RG; q += 32)
                    __stcg(reinterpret_cast<uint4*>(T.X + sl * A.slot_bytes + (size_t)S.kg1 * 64 * RG) + q,
                           make_uint4(0u, 0u, 0u, 0u));
        }
    }
    ok = ok && group_sync(A, Tp, up);
    if (!ok) return false;
    const AxisWin& w0 = T.win[tm_solve(0, B, cen, team).Mp];
    publish_input<RG, MT>(A, Tp, jo, M, KIND_START, SLOT_START, 0, up->tag + 1u, true, w0.lo + w0.ia, -1, -1, -1, -1);
    return true;
}

// Consecutive solves of a pass that map one line to itself in one tile, each
// feeding the next line: solves [i, end) of visit jo.  The loop of the apply; kept
// small (with the other roles' loops it has to stay in the instruction cache:
// about 100 misses a solve cost more than everything else together).
template <int RG, int MT>
__device__ __noinline__ bool run_lines(const TeamArgs& A, Sm* Tp, Upd* up, int jo, int i, int end) {
    Sm& T = *Tp;
    constexpr int NB = RG / 8, KGB = 64 * RG;
    constexpr int NRS = RG == 16 && MT == 128 ? 2 : 1;    // row sets of a thread in a tile
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q4 = warp & 3, hh = warp >> 2;
    const int ii = lane >> 2, c = lane & 3;               // row of a group, pair of right-hand sides
    const int cb = RG == 16 ? hh : 0;
    const int rhs0 = 8 * cb + 2 * c;                      // this thread's right-hand sides rhs0, rhs0 + 1
    const int gi0 = RG == 8 && MT == 128 ? warp : q4;     // its first row group of a tile (the second: 4 on)
    const bool idle = RG == 8 && MT == 64 && hh == 1;     // no accumulator columns for this warp
    constexpr int SUBC = acc_slots(RG, MT) * 4 * RG;
    const uint32_t tlane = T.tslot + ((uint32_t)(32 * q4) << 16) + 32 * cb + (gi0 >> 2) * SUBC;
    const int B = T.B, cen = T.cen, team = T.team, nsol = T.nsol;
    const AxisWin wz = T.win[pass_pos(jo, B, cen).M];
    const int Lz = wz.L, za = wz.ia, dz = wz.ib - wz.ia, E = T.N * Lz;
    const Shape& S = T.shape[8 + KIND_RING];
    const bool split = S.halves == 2;
    int cg0, cg1;                                         // this rank's groups of 8 columns
    tm_part(E, 1, 1, T.rank, T.C, &cg0, &cg1);
    cg0 += gi0;                                           // this warp's (first) group
    const bool fv = !idle && cg0 < cg1, fv1 = NRS == 2 && cg0 + 4 < cg1;   // it exists (rows beyond E are zero)
    int fe[NRS], fz[NRS];                                 // column and own-layer offsets (-1: none) per row set
#pragma unroll
    for (int j = 0; j < NRS; ++j) {
        const int e = 8 * (cg0 + 4 * j) + ii, x = e / Lz, lz = e - x * Lz;
        fe[j] = (j ? fv1 : fv) && e < E ? e * RG + rhs0 : -1;
        fz[j] = fe[j] >= 0 && lz >= za && lz < za + dz ? (x * dz + lz - za) * RG + rhs0 : -1;
    }
    // the pass: line by line up or down; the coupling of the line's neighbour that the result feeds
    const TeamSolve t0 = tm_solve(i, B, cen, team);
    const bool bwd = t0.bwd;
    const int dy = (bwd != (t0.role == ROLE_U)) ? -1 : 1; // lower front: up, then down; upper front: down, then up
    int y = T.win[t0.Mp].lo + T.win[t0.Mp].ia;
    const float2* pc = (dy > 0 ? T.cdn : T.cup) + y + dy;
    const float fs = bwd ? 1.f : -1.f;
    const long long* po = T.soff + t0.Mp;
    float2* line = T.V + y * T.VL;         // forward values of the line
    const float2* gl = T.Gv + (y + dy) * T.GL;            // the right-hand side on the next line
    float2* zl = T.Zv + y * T.GL;
    const int VL = T.VL * dy, GL = T.GL * dy;
    unsigned char* X = T.X + (size_t)cg0 * KGB + part_offset(cb, lane);    // this thread's parts in slot 0
    u64* H = T.H + (cg0 * NB + cb) * 4;
    const float* scale = A.scale + cg0 * 16 + ii;
    int ri = slot_of_solve(i, nsol, cen, team);           // ring slot of solve i
    Upd u = *up;
    bool ok = true;
#pragma unroll 1
    for (; i < end; ++i) {
        ++u.tag;
        // operands of this thread's rows, in flight during the product
        const float* sc = scale + *po;
        float4 pre[NRS];
        int er[NRS], ei[NRS];
#pragma unroll
        for (int j = 0; j < NRS; ++j) {
            pre[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            er[j] = ei[j] = 0;
            if (fe[j] >= 0) {
                er[j] = __float_as_int(ptx::ld_nc_f32_here(sc + 64 * j));
                ei[j] = __float_as_int(ptx::ld_nc_f32_here(sc + 64 * j + 8));
            }
            const int o = bwd ? fe[j] : fz[j];
            if (o >= 0) pre[j] = ptx::ld_cg_f32x4_here((bwd ? line : gl) + o);
        }
        const float2 k = make_float2(fs * pc->x, fs * pc->y);
        ok = wait_phase(&T.eready, u.xph, T.limit, &T.abort);
        u.xph ^= 1u;
        if (!ok) break;
        const int2 ec = *reinterpret_cast<const int2*>(&T.ecol[rhs0]), ep = *reinterpret_cast<const int2*>(&T.epred[rhs0]);
        float R[NRS][4] = {}, I[NRS][4] = {};
        if (!(ok = read_tile<RG, MT, NRS>(T, u, S, tlane, split, fv, R, I))) break;
        float4 W[NRS];
#pragma unroll
        for (int j = 0; j < NRS; ++j)
            if (j ? fv1 : fv) W[j] = scale_rows(R[j], I[j], (er[j] >> 23) - 127, (ei[j] >> 23) - 127, ec.x, ec.y);
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&T.tfree);
        unsigned hw[NRS];
        const int rn = i + 1 == nsol - 1 ? SLOT_END : (!team && i + 1 == cen ? SLOT_CENTRE : (ri + 1) & (NRING - 1));
#pragma unroll
        for (int j = 0; j < NRS; ++j)
            if (j ? fv1 : fv) {
                if (bwd) W[j] = sub4(pre[j], W[j]);           // a backward solve is a correction
                if (fe[j] < 0) W[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                float4 q = cmul2(k, W[j]);
                if (!bwd) q = add4(q, pre[j]);
                hw[j] = store_parts(X + rn * A.slot_bytes + 4 * j * KGB, q, ep.x, ep.y);
            }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NRS; ++j)
            if (j ? fv1 : fv) release_header(H + rn * A.hdr_words + 4 * j * NB * 4, hw[j], u.tag + 1u);
#pragma unroll
        for (int j = 0; j < NRS; ++j) {
            const int o = bwd ? fz[j] : fe[j];
            if (o >= 0) *reinterpret_cast<float4*>((bwd ? zl : line) + o) = W[j];
        }
        ri = rn & (NRING - 1);
        pc += dy;
        po += dy;
        line += VL;
        gl += GL;
        zl += GL;
    }
    *up = u;
    return ok;
}

// The same for blocks of nl lines, 8 a multiple of nl, and for several tiles a rank.
// A column's nl lines are neighbouring rows of one group, so the coupling gets from the
// line that feeds the next block to the one that takes it by a shuffle, and a warp
// publishes the groups whose rows it holds, each tile while the next is multiplied.
// Against run_general (couplings through L2, a barrier of the CTA, index divisions
// after the product) one apply: two lines, n = 50, one
// front with 24 right-hand sides 31.0 -> 21.4 ms (the K split over clusters 25.3), n = 30, two
// fronts with 9 6.7 -> 4.5 (5.4), n = 17 with two 1.90 -> 1.44 (1.71)
template <int RG, int MT>
__device__ __noinline__ bool run_blocks(const TeamArgs& A, Sm* Tp, Upd* up, int jo, int i, int end) {
    Sm& T = *Tp;
    constexpr int GT = MT / 16, NB = RG / 8, KGB = 64 * RG;
    constexpr int NRS = RG == 16 && MT == 128 ? 2 : 1, SUBC = acc_slots(RG, MT) * 4 * RG;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q4 = warp & 3, hh = warp >> 2, ii = lane >> 2, c = lane & 3;
    const int cb = RG == 16 ? hh : 0, rhs0 = 8 * cb + 2 * c;
    const int gi0 = RG == 8 && MT == 128 ? warp : q4;
    const bool idle = RG == 8 && MT == 64 && hh == 1;
    const uint32_t tlane = T.tslot + ((uint32_t)(32 * q4) << 16) + 32 * cb + (gi0 >> 2) * SUBC;
    const int B = T.B, cen = T.cen, team = T.team, nsol = T.nsol, VL = T.VL, GL = T.GL;
    const Shape& S = T.shape[8 + KIND_RING];
    const bool split = S.halves == 2;
    const int nl = S.nl, nt = S.nt, K = S.K, a0 = S.a0, c0 = S.c0;
    const AxisWin wz = T.win[pass_pos(jo, B, cen).M];
    const int Lz = wz.L, za = wz.ia, dz = wz.ib - wz.ia;
    const TeamSolve t0 = tm_solve(i, B, cen, team);
    const bool bwd = t0.bwd;
    const int dy = (bwd != (t0.role == ROLE_U)) ? -1 : 1;
    const int lsrc = dy > 0 ? nl - 1 : 0, ldst = nl - 1 - lsrc;   // the line that feeds the next block, the one that takes it
    const float fs = bwd ? 1.f : -1.f;
    int y = T.win[t0.Mp].lo + T.win[t0.Mp].ia;            // the block's first line
    const long long* po = T.soff + t0.Mp;
    int ri = slot_of_solve(i, nsol, cen, team);
    const int sh = __ffs(nl) - 1;                         // nl is a power of two
    const int l = ii & (nl - 1), src = lane + 4 * (l == ldst ? lsrc - ldst : 0);
    Upd u = *up;
    bool ok = true;
#pragma unroll 1
    for (; i < end && ok; ++i, y += dy * nl, po += dy) {
        ++u.tag;
        const float2 kc = dy > 0 ? T.cdn[y + nl] : T.cup[y - 1];
        const float2 k = make_float2(fs * kc.x, fs * kc.y);
        const float* sc = A.scale + *po + ii;
        float2* line = T.V + (y + l) * VL;
        const float2* gl = T.Gv + (y + dy * nl + l) * GL;
        float2* zl = T.Zv + (y + l) * GL;
        const int rn = i + 1 == nsol - 1 ? SLOT_END : (!team && i + 1 == cen ? SLOT_CENTRE : (ri + 1) & (NRING - 1));
        unsigned char* X = T.X + rn * A.slot_bytes + part_offset(cb, lane);
        u64* H = T.H + rn * A.hdr_words + cb * 4;
        int2 ec = make_int2(0, 0), ep = ec;
#pragma unroll 1
        for (int tl = 0; (tl < nt || tl == 0) && ok; ++tl) {
            const int p0 = tl * GT + gi0;
            const bool fv = !idle && p0 < c0, fv1 = NRS == 2 && p0 + 4 < c0;
            // operands of this thread's rows, in flight during the product
            int fe[NRS], fz[NRS], er[NRS], ei[NRS];
            float4 pre[NRS];
#pragma unroll
            for (int j = 0; j < NRS; ++j) {
                const int gid = a0 + p0 + 4 * j, r = 8 * gid + ii;
                const int e = r >> sh, x = e / Lz, lz = e - x * Lz;
                fe[j] = (j ? fv1 : fv) && r < K ? e * RG + rhs0 : -1;
                fz[j] = fe[j] >= 0 && lz >= za && lz < za + dz ? (x * dz + lz - za) * RG + rhs0 : -1;
                pre[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                er[j] = ei[j] = 0;
                if (fe[j] >= 0) {
                    er[j] = __float_as_int(ptx::ld_nc_f32_here(sc + 16 * gid));
                    ei[j] = __float_as_int(ptx::ld_nc_f32_here(sc + 16 * gid + 8));
                }
                const int o = bwd ? fe[j] : fz[j];
                if (o >= 0) pre[j] = ptx::ld_cg_f32x4_here((bwd ? line : gl) + o);
            }
            if (tl == 0) {
                if (!(ok = wait_phase(&T.eready, u.xph, T.limit, &T.abort))) break;
                u.xph ^= 1u;
                ec = *reinterpret_cast<const int2*>(&T.ecol[rhs0]);
                ep = *reinterpret_cast<const int2*>(&T.epred[rhs0]);
            }
            float R[NRS][4] = {}, I[NRS][4] = {};
            if (!(ok = read_tile<RG, MT, NRS>(T, u, S, tlane, split, fv, R, I))) break;
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&T.tfree);
            float4 W[NRS];
#pragma unroll
            for (int j = 0; j < NRS; ++j)
                if (j ? fv1 : fv) W[j] = scale_rows(R[j], I[j], (er[j] >> 23) - 127, (ei[j] >> 23) - 127, ec.x, ec.y);
            unsigned hw[NRS];
#pragma unroll
            for (int j = 0; j < NRS; ++j)
                if (j ? fv1 : fv) {
                    if (bwd) W[j] = sub4(pre[j], W[j]);
                    if (fe[j] < 0) W[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    float4 q = cmul2(k, W[j]);
                    q = make_float4(__shfl_sync(0xffffffffu, q.x, src), __shfl_sync(0xffffffffu, q.y, src),
                                    __shfl_sync(0xffffffffu, q.z, src), __shfl_sync(0xffffffffu, q.w, src));
                    if (l != ldst) q = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (!bwd) q = add4(q, pre[j]);
                    hw[j] = store_parts(X + (size_t)(a0 + p0 + 4 * j) * KGB, q, ep.x, ep.y);
                }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < NRS; ++j)
                if (j ? fv1 : fv) release_header(H + (a0 + p0 + 4 * j) * NB * 4, hw[j], u.tag + 1u);
#pragma unroll
            for (int j = 0; j < NRS; ++j) {
                const int o = bwd ? fz[j] : fe[j];
                if (o >= 0) *reinterpret_cast<float4*>((bwd ? zl : line) + o) = W[j];
            }
        }
        ri = rn & (NRING - 1);
    }
    *up = u;
    return ok;
}

// First solve after the run of run_lines or run_blocks that starts with solve i (i itself: none).
__device__ __forceinline__ int run_end(Sm& T, int jo, int i) {
    const int B = T.B, cen = T.cen, team = T.team, nsol = T.nsol;
    const Shape& S = T.shape[8 + KIND_RING];
    if (kind_of(i, nsol, cen, team) != KIND_RING || 8 % S.nl != 0) return i;
    // backward up to the last solve, which takes one line; forward up to the front's last solve (two
    // fronts: it feeds the centre) or the centre, which has to have as many lines
    if (tm_solve(i, B, cen, team).bwd) return S.nl == 1 ? nsol - 1 : nsol - 2;
    if (T.two) return (team ? T.U : cen) - 1;
    return T.shape[8 + KIND_CENTRE].nl == S.nl ? cen : cen - 1;
}

// A solve of any shape.
template <int RG, int MT>
__device__ __noinline__ bool run_general(const TeamArgs& A, Sm* Tp, Upd* up, int jo, int i) {
    Sm& T = *Tp;
    const int lane = threadIdx.x & 31, c = lane & 3, rhs0 = 8 * (RG == 16 ? (int)(threadIdx.x >> 7) : 0) + 2 * c;
    const int B = T.B, cen = T.cen, team = T.team, nsol = T.nsol, U = T.U;
    const bool two = T.two;
    const long long limit = T.limit;
    Shape* shapes = T.shape + 8;
    const int M = pass_pos(jo, B, cen).M;
    const TeamSolve t = tm_solve(i, B, cen, team);
    const int kind = kind_of(i, nsol, cen, team);
    const Shape& S = shapes[kind];
    const bool more = i + 1 < nsol, centre = kind == KIND_CENTRE;
    const bool into_centre = two && !t.bwd && (team ? i == U - 1 : i == cen - 1);
    Upd u = *up;
    ++u.tag;
    bool ok = true;
    ok = wait_phase(&T.eready, u.xph, limit, &T.abort);
    u.xph ^= 1u;
    *up = u;
    const int ec0 = T.ecol[rhs0], ec1 = T.ecol[rhs0 + 1];
#pragma unroll 1
    for (int tl = 0; (tl < S.nt || tl == 0) && ok; ++tl)
        ok = general_rows<RG, MT>(A, Tp, up, M, i, tl, T.soff[op_slot(t.Mp, t.bwd, B)], T.tslot, ec0, ec1);
    u = *up;
    if (ok && more && !into_centre) {
        ok = cta_sync(T, u, limit);
        if (ok) {
            const TeamSolve tn = tm_solve(i + 1, B, cen, team);
            const int nkind = kind_of(i + 1, nsol, cen, team);
            const AxisWin& wn = T.win[tn.Mp];
            const int l0 = nkind == KIND_END ? (team ? T.N - A.g.b : A.g.b - 1) : wn.lo + wn.ia;
            // the coupled line of the next input
            const int l1 = (tn.bwd ? tn.role == ROLE_L : tn.role == ROLE_U) ? shapes[nkind].nl - 1 : 0;
            // the centre also feeds the upper front's first backward solve: first, for the predicted scales may
            // change once this rank's own input is out
            if (centre && two)
                publish_input<RG, MT>(A, Tp, jo, M, KIND_RING, slot_of_solve(U, 2 * U, cen, 1), 1,
                                      (unsigned)(jo * 2 * U + U) + 1u, false, T.win[cen + 1].lo + T.win[cen + 1].ia, 1, 0, -1, -1);
            publish_input<RG, MT>(A, Tp, jo, M, nkind, slot_of_solve(i + 1, nsol, cen, team), 0, u.tag + 1u, !tn.bwd, l0,
                                  centre && two ? 0 : 2 + team, l1, -1, -1);
        }
    }
    *up = u;
    return ok;
}

template <int RG, int MT>
__global__ void __launch_bounds__(TT, 1) k_team(const __grid_constant__ TeamArgs A) {
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int NB = RG / 8;               // blocks of 8 right-hand sides
    constexpr int KGB = 64 * RG;             // bytes of 8 published entries
    constexpr int GT = MT / 16;              // row groups of a tile
    constexpr int ACOLS = 4 * RG;            // columns of an accumulator: G times q's re hi, im hi, re lo, im lo
    constexpr int NSUB = MT / 64;            // products of 4 row groups per tile and 16 input entries
    constexpr int SLOTS = acc_slots(RG, MT); // accumulators of each
    const int B = A.g.B, N = A.g.N, cen = A.g.cen;
    const int two = A.T == 2;
    unsigned char* ring = smem;
    unsigned char* Bbuf = smem + A.off_b;
    Sm& S_ = *reinterpret_cast<Sm*>(smem + A.off_misc);
    float2* s_cdn = reinterpret_cast<float2*>(&S_ + 1);          // [N]
    float2* s_cup = s_cdn + N;                                   // [N]
    long long* s_soff = reinterpret_cast<long long*>(s_cup + N); // [B + 2]
    long long* s_off = s_soff + B + 2;                           // [B + 2]
    AxisWin* s_win = reinterpret_cast<AxisWin*>(s_off + B + 2);  // [B]
    uint64_t *full = S_.full, *empty = S_.empty, *bfull = S_.bfull;
    uint64_t *bgo = &S_.bgo, *eready = &S_.eready, *mdone = &S_.mdone, *sdone = &S_.sdone, *tfree = &S_.tfree;
    volatile int* s_abort = &S_.abort;
    Shape* s_shape = S_.shape;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int grp = blockIdx.x / (A.T * A.C), team = (blockIdx.x / A.C) % A.T, rank = blockIdx.x % A.C;
    const int C = A.C;
    const long long limit = A.wait_cycles > 0 ? A.wait_cycles : TEAM_WAIT;
    const int nsol = tm_solves(B, cen, team);
    const int nvis = 2 * B - 1;

    const size_t tg = (size_t)grp * A.T + team;
    if (tid == 0) {
        for (int q = 0; q < MAXST; ++q) {
            ptx::mbar_init(&full[q], 1);
            ptx::mbar_init(&empty[q], 1);
        }
        for (int q = 0; q < NBC; ++q) ptx::mbar_init(&bfull[q], 1);
        ptx::mbar_init(bgo, 1);
        ptx::mbar_init(eready, 1);
        ptx::mbar_init(mdone, 1);
        ptx::mbar_init(sdone, 1);
        for (int q = 0; q < 8; ++q) {
            ptx::mbar_init(&S_.sacc[q], 1);
            ptx::mbar_init(&S_.afree[q], CW);
        }
        ptx::mbar_init(tfree, CW);
        ptx::mbar_init(&S_.cbar, CW);
        ptx::mbar_init(&S_.xbar, 1);
        S_.abort = 0;
        S_.limit = limit;
        S_.N = N; S_.B = B; S_.cen = cen; S_.two = two; S_.U = B - 1 - cen; S_.C = C;
        S_.grp = grp; S_.team = team; S_.rank = rank; S_.nsol = nsol;
        S_.VL = A.Emax * RG;
        S_.GL = N * A.DZ * RG;
        S_.V = A.V + (size_t)grp * N * S_.VL;
        S_.Gv = A.Gv + (size_t)grp * N * S_.GL;
        S_.Zv = A.Zv + (size_t)grp * N * S_.GL;
        S_.Qf = A.Qf + (size_t)grp * 4 * S_.VL;
        S_.gm = A.gmax + (size_t)grp * 2 * N * RG;
        S_.ctr = A.ctr + 32 * grp;
        S_.Xteam = SLOT_START * A.slot_bytes + A.start_bytes;
        S_.Hteam = (size_t)(SLOT_START * A.hdr_words + A.start_words);
        S_.X = A.X + tg * S_.Xteam;
        S_.H = A.hdr + tg * S_.Hteam;
        S_.Bbuf = Bbuf;
        S_.cdn = s_cdn; S_.cup = s_cup; S_.soff = s_soff; S_.off = s_off; S_.win = s_win;
        ptx::fence_mbar_init();
    }
    for (int q = tid; q < N; q += TT) {
        s_cdn[q] = A.c_dn[q];
        s_cup[q] = A.c_up[q];
    }
    for (int q = tid; q < B; q += TT) s_win[q] = A.win[q];
    if (warp == 0) {
        ptx::tmem_alloc(&S_.tslot, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, S_.tslot, 0);

    if (warp == RING_WARP) {
        // ------------------------------------------- operator stream -> ring
        Shape* shapes = s_shape;
        int stage = 0, issued = 0;
        uint32_t zeros = 0;                  // stages where this lane's part is zero
        uint32_t eph = 1;                    // the first round finds every stage free
        bool ok = true;
        for (int jo = 0; jo < nvis && ok; ++jo) {
            const int M = pass_pos(jo, B, cen).M;
            make_shapes(shapes, s_win, A.tp, N, B, cen, two, team, M, rank, C, GT, lane);
            for (int q = lane; q < B + 2; q += 32) s_off[q] = A.tp[op_index(M, q, B)].off;
            __syncwarp();
#pragma unroll 1
            for (int i = 0; i < nsol && ok; ++i) {
                const TeamSolve t = tm_solve(i, B, cen, team);
                const Shape& S = shapes[kind_of(i, nsol, cen, team)];
                const int c0 = S.c0, cs = c0 + S.c1, nt = S.nt, KP = S.KP, ng = S.ng;
                const unsigned char* base = A.G + s_off[op_slot(t.Mp, t.bwd, B)];
#pragma unroll 1
                for (int tl = 0; tl < nt && ok; ++tl) {
                    // the tile's groups: at most two runs of stored groups (lane & 1: this lane's)
                    const int g0 = tl * GT, g1 = min(cs, g0 + GT);
                    const int m0 = max(0, min(g1, c0) - g0);
                    const int run = lane & 1;
                    const int cnt = run ? g1 - g0 - m0 : m0;
                    const int gr = run ? S.ng0 + S.a1 + max(0, g0 - c0) : S.a0 + g0;
                    // lo parts of some groups only: every group's parts for themselves (lane & 1: lo), zeros where there
                    // are none (not again into a stage whose place holds them: copying them each time made an
                    // apply of such operators 20 % longer)
                    const int mg = lane >> 1, nlo = S.nlo;
                    int unit = 0;
                    bool some = false;
                    if (nlo && mg < g1 - g0) {
                        const int q = mg < m0 ? S.a0 + g0 + mg : S.ng0 + S.a1 + max(0, g0 - c0) + mg - m0;
                        unit = run ? __ldg(A.lo + S.lob + q) : q;
                        some = unit >= 0;
                        if (run) unit += ng;
                    }
#pragma unroll 1
                    for (int kc0 = 0; kc0 < KP; kc0 += TKC) {
                        ok = wait_phase(&empty[stage], eph, limit, s_abort);
                        if (!ok) break;
                        const int kc = min(TKC, KP - kc0), per = 32 * kc * S.halves;      // bytes of a group
                        if (nlo) {
                            const bool mine = mg < g1 - g0, none = mine && run && !some && kc == TKC;
                            const bool go = mine && !(none && (zeros >> stage & 1u));
                            const unsigned n = __popc(__ballot_sync(0xffffffffu, go));
                            if (lane == 0) ptx::mbar_expect_tx(&full[stage], n * 32u * (uint32_t)kc);
                            __syncwarp();
                            if (go)
                                ptx::bulk_g2s(ring + stage * A.stage_bytes + mg * per + run * 32 * kc,
                                              some ? base + tm_unit(kc0 / TKC, unit, ng + nlo, KP)
                                                   : reinterpret_cast<const unsigned char*>(A.lo),
                                              (uint32_t)(32 * kc), &full[stage]);
                            zeros = none ? zeros | 1u << stage : zeros & ~(1u << stage);
                        } else {
                            if (lane == 0) ptx::mbar_expect_tx(&full[stage], (uint32_t)((g1 - g0) * per));
                            __syncwarp();
                            if (lane < 2 && cnt > 0)
                                ptx::bulk_g2s(ring + stage * A.stage_bytes + (run ? m0 : 0) * per,
                                              base + ((size_t)kc0 * ng + (size_t)kc * gr) * S.halves * 32,
                                              (uint32_t)(cnt * per), &full[stage]);
                            zeros &= ~(1u << stage);
                        }
                        ++issued;
                        if (++stage == A.stages) { stage = 0; eph ^= 1u; }
                    }
                }
            }
        }
        if (!ok) fail(A, S_);
        // copies in flight land before the CTA leaves: the last one of every stage
        for (int q = 0; q < A.stages && q < issued; ++q) {
            const int n = issued - 1 - q;                        // issue number, its stage and phase
            const int s = n % A.stages;
            const uint32_t ph = (uint32_t)((n / A.stages) & 1);
            const long long t0 = clock64();
            while (!__all_sync(0xffffffffu, ptx::mbar_try(&full[s], ph)) && clock64() - t0 < limit) {
            }
        }
    } else if (warp == MMA_WARP) {
        // ------------------------------------------------------ products
        // the whole warp runs the loop: uniform operands, one elected lane issues; nothing is called
        // (after a call the compiler takes nothing for uniform), the gather warp makes the records
        const Shape* shapes = s_shape + 4;
        const uint64_t bdesc0 = ptx::umma_desc(ptx::smem_u32(Bbuf), KGB, 128u);
        const uint32_t a_s = ptx::smem_u32(ring);
        int stage = 0, seen = 0;                                  // seen: chunks ahead known to have landed
        uint32_t fph = 0, gph = 0, tph = 1, bph = 0, aph = 0;     // bph, aph: a parity bit per part and per place of a unit
        bool ok = true;
        for (int jo = 0; jo < nvis && ok; ++jo) {
#pragma unroll 1
            for (int i = 0; i < nsol && ok; ++i) {
                // the solve before has been read out of TMEM; operator chunks that have landed by then need no
                // wait between the products
                if (!(ok = wait_phase(tfree, tph, limit, s_abort))) break;
                tph ^= 1u;
#pragma unroll 1
                for (; seen < A.stages; ++seen) {
                    const int st = stage + seen, wrap = st >= A.stages;
                    if (!__all_sync(0xffffffffu, ptx::mbar_try(&full[wrap ? st - A.stages : st], fph ^ (uint32_t)wrap))) break;
                }
                if (!(ok = wait_phase(bgo, gph, limit, s_abort))) break;    // of the solve's first gather
                const Shape& S = shapes[kind_of(i, nsol, cen, team)];
                const int KP = __shfl_sync(0xffffffffu, S.KP, 0), nt = __shfl_sync(0xffffffffu, S.nt, 0);
                const int nu = __shfl_sync(0xffffffffu, S.nu, 0), cpa = __shfl_sync(0xffffffffu, S.cpa, 0);
                const int w = __shfl_sync(0xffffffffu, S.w, 0), NU = SLOTS >> (w >> 1);
                const int rsh = __shfl_sync(0xffffffffu, S.rsh, 0), per = rsh == 2 ? 1 : w;   // per: accumulators of a chunk or run
                const int hv = __shfl_sync(0xffffffffu, S.halves, 0);
                const uint32_t idesc = ptx::umma_idesc_f16_bn(64 * hv, 4 * RG);
                const bool passes = KP > A.KB;                    // every tile gathers the input anew, in passes
#pragma unroll 1
                for (int tl = 0; (tl < nt || tl == 0) && ok; ++tl) {
                    if (tl > 0) {                                 // the tile before has been read out too
                        if (!(ok = wait_phase(tfree, tph, limit, s_abort))) break;
                        tph ^= 1u;
                    }
                    int un = 0, us = 0, va = 0, ca = 0;           // unit, its place, accumulators done, chunks of the next
#pragma unroll 1
                    for (int k0 = 0; k0 < KP && ok; k0 += A.KB) {
                        const int ke = min(KP, k0 + A.KB), part = 16 * gather_part((ke - k0) >> 4);
                        const bool gathered = tl == 0 || passes;  // a gather of its own: wait for its parts
                        if (gathered) {
                            if (tl + k0 > 0 && !(ok = wait_phase(bgo, gph, limit, s_abort))) break;
                            gph ^= 1u;
                        }
                        uint64_t bd = bdesc0;
#pragma unroll 1
                        for (int kc0 = k0, pj = 0; kc0 < ke; ++pj) {
                            if (gathered) {
                                if (!(ok = wait_phase(&bfull[pj], bph >> pj & 1u, limit, s_abort))) break;
                                bph ^= 1u << pj;
                            }
                            const int kpe = min(ke, kc0 + part);
                            if (nt == 0) kc0 = kpe;               // a rank without rows only sees them
                            ptx::tc_fence_after();
#pragma unroll 1
                            for (; kc0 < kpe; kc0 += TKC) {
                                const int kc = min(TKC, KP - kc0);
                                if (--seen < 0) {
                                    seen = 0;
                                    if (!(ok = wait_phase(&full[stage], fph, limit, s_abort))) break;
                                    ptx::tc_fence_after();
                                }
                                if (un >= NU && va + ca == 0) {   // the unit there before has been read
                                    if (!(ok = wait_phase(&S_.afree[us], aph >> us & 1u, limit, s_abort))) break;
                                    aph ^= 1u << us;
                                    ptx::tc_fence_after();
                                }
                                const uint32_t d = tmem + (uint32_t)((us * w + va) * ACOLS);
                                const uint32_t ahi = a_s + (uint32_t)(stage * A.stage_bytes), sbo = (uint32_t)(kc * 16);
                                const uint64_t ad = ptx::umma_desc(ahi, 128u, sbo);
                                chunk_products<RG, NSUB>(d, ad, 8 * hv * sbo / 16, bd, idesc, ca > 0, rsh, kc);
                                bd += TKC / 16 * 2 * KGB / 16;
                                ptx::umma_commit_warp(&empty[stage]);
                                if (++stage == A.stages) { stage = 0; fph ^= 1u; }
                                if (++ca == cpa) {
                                    ca = 0;
                                    if ((va += per) == w) {
                                        va = 0;
                                        if (++un < nu) ptx::umma_commit_warp(&S_.sacc[us]);
                                        if (++us == NU) us = 0;
                                    }
                                }
                            }
                            if (!ok) break;
                        }
                        if (ok && (passes || tl + 1 >= nt)) ptx::umma_commit_warp(mdone);
                    }
                    if (ok) ptx::umma_commit_warp(sdone);
                }
            }
        }
        if (!ok) fail(A, S_);
        // products in flight end before TMEM is freed
        ptx::umma_commit_warp(&S_.xbar);
        const long long t0 = clock64();
        while (!__all_sync(0xffffffffu, ptx::mbar_try(&S_.xbar, 0)) && clock64() - t0 < limit) {
        }
    } else if (warp == GATHER_WARP) {
        // ------------------------------------- headers, scales and gathers
        Shape* shapes = s_shape + 4;
        uint32_t mph = 0, lph = 0;           // lph: a bit per part, the phase its next copy completes
        bool ok = true, fresh = true;
        unsigned tag = 0, tiles = 0;         // tiles: of the solves before
        int ri = 0;
        // lane's header words: right-hand sides 8 cb + 4 cp .. + 3 of every group of 8 entries
        const int cp = lane & 1, cb = RG == 16 ? (lane >> 1) & 1 : 0;
        const unsigned* gm = A.gmax + (size_t)grp * 2 * N * RG + 8 * cb + 4 * cp;
        for (int jo = 0; jo < nvis && ok; ++jo) {
            // the records are the products' too: the visit before has been multiplied
            if (!fresh) {
                if (!(ok = wait_phase(mdone, mph, limit, s_abort))) break;
                mph ^= 1u;
                fresh = true;
            }
            make_shapes(shapes, s_win, A.tp, N, B, cen, two, team, pass_pos(jo, B, cen).M, rank, C, GT, lane);
            ri = 0;
#pragma unroll 1
            for (int i = 0; i < nsol && ok; ++i) {
                const int kind = kind_of(i, nsol, cen, team);
                const Shape& S = shapes[kind];
                const int K = S.K, KP = S.KP, nt = S.nt, ng8 = (K + 7) >> 3;
                ++tag;
                const int slot = kind == KIND_RING ? ri++ & (NRING - 1)
                                                   : (kind == KIND_START ? SLOT_START : (kind == KIND_END ? SLOT_END : SLOT_CENTRE));
                const unsigned char* xs = S_.X + slot * A.slot_bytes;
                const u64* hw0 = S_.H + slot * A.hdr_words;
                const u64* hd = hw0 + 2 * lane;
                // the lines the slab's right-hand side enters the next input on
                int gl0 = 0, gln = 0;
                if (i + 1 < nsol) {
                    const TeamSolve tn = tm_solve(i + 1, B, cen, team);
                    if (!tn.bwd) {
                        const AxisWin& wn = s_win[tn.Mp];
                        gl0 = wn.lo + wn.ia;
                        gln = wn.ib - wn.ia;
                    }
                }
                // the input before has been multiplied
                if (!fresh) {
                    if (!(ok = wait_phase(mdone, mph, limit, s_abort))) break;
                    mph ^= 1u;
                }
                // lane's part of the first gather: everything that does not need the headers before the poll
                int kb = min(KP, A.KB), n16 = kb >> 4, part = gather_part(n16), my = lane * part;
                uint32_t by = lane < NBC && my < n16 ? (uint32_t)(min(part, n16 - my) * 2 * KGB) : 0u;
                unsigned char* dst = Bbuf + my * 2 * KGB;
                const unsigned char* src = xs + (size_t)my * 2 * KGB;
                if (by) ptx::mbar_expect_tx(&bfull[lane], by);
                // poll the headers: max and used exponents of this lane's 4 right-hand sides
                const int nv = ng8 * NB * 2;
                unsigned mx0 = 0, mx1 = 0, mn0 = 0xffffffffu, mn1 = 0xffffffffu;
                const long long t0 = clock64();
#pragma unroll 1
                for (int v0 = 0; v0 < nv && ok; v0 += 32 * 8) {
                    ulonglong2 w[8];
                    unsigned pend = 0;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (v0 + lane + 32 * u < nv) pend |= 1u << u;
                    while (__any_sync(0xffffffffu, pend != 0)) {
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (pend >> u & 1) w[u] = ptx::ld_relaxed_gpu_v2u64(hd + 2 * (v0 + 32 * u));
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if ((pend >> u & 1) && (unsigned)(w[u].x >> 32) == tag && (unsigned)(w[u].y >> 32) == tag) {
                                pend &= ~(1u << u);
                                mx0 = __vmaxu4(mx0, (unsigned)w[u].x);
                                mx1 = __vmaxu4(mx1, (unsigned)w[u].y);
                                mn0 = __vminu4(mn0, (unsigned)w[u].x);
                                mn1 = __vminu4(mn1, (unsigned)w[u].y);
                            }
                        if (__any_sync(0xffffffffu, pend != 0 && (clock64() - t0 > limit || *s_abort))) {
                            ok = false;
                            break;
                        }
                    }
                }
                if (!ok) break;
                // every lane has read headers released after their parts: its fence, then the warp's barrier, order
                // the parts before the copies of lanes 0 and 1
                ptx::fence_acquire_gpu();
                __syncwarp();
                ptx::fence_proxy_async_global();
                if (by) ptx::bulk_g2s(dst, src, by, &bfull[lane]);
                // each right-hand side has one scale in all headers: lane's columns are those of lane mod 2 NB
                const unsigned x0 = __shfl_sync(0xffffffffu, mx0, lane & (2 * NB - 1));
                const unsigned x1 = __shfl_sync(0xffffffffu, mx1, lane & (2 * NB - 1));
                const bool none = lane >= nv;                         // fewer header words than lanes
                const bool even = __all_sync(0xffffffffu, none || (((mx0 ^ mn0) | (mx1 ^ mn1) | (mx0 ^ x0) | (mx1 ^ x1)) &
                                                                    0xff00ff00u) == 0u);
                // one gather for all tiles, or every tile's passes
#pragma unroll 1
                for (int tl = 0; (tl == 0 || (tl < nt && KP > A.KB)) && ok; ++tl)
#pragma unroll 1
                    for (int k0 = 0; k0 < KP && ok; k0 += A.KB) {
                        // the pass before has been multiplied
                        const bool first = tl == 0 && k0 == 0;
                        if (!first) {
                            if (!(ok = wait_phase(mdone, mph, limit, s_abort))) break;
                            mph ^= 1u;
                            kb = min(KP, k0 + A.KB) - k0, n16 = kb >> 4, part = gather_part(n16), my = lane * part;
                            by = lane < NBC && my < n16 ? (uint32_t)(min(part, n16 - my) * 2 * KGB) : 0u;
                            if (by) {
                                ptx::mbar_expect_tx(&bfull[lane], by);
                                ptx::bulk_g2s(Bbuf + my * 2 * KGB, xs + (size_t)(k0 / 8 + my * 2) * KGB, by, &bfull[lane]);
                            }
                        }
                        fresh = false;
                        for (int q = 0; q < NBC; ++q)
                            if (q * part < n16) lph ^= 1u << q;
                        __syncwarp();
                        if (even && lane == 0) ptx::mbar_arrive(bgo);
                        __syncwarp();
                        if (first) {
                            for (int s = 2 * NB; s < 32; s <<= 1) {
                                mx0 = __vmaxu4(mx0, __shfl_xor_sync(0xffffffffu, mx0, s));
                                mx1 = __vmaxu4(mx1, __shfl_xor_sync(0xffffffffu, mx1, s));
                                mn0 = __vminu4(mn0, __shfl_xor_sync(0xffffffffu, mn0, s));
                                mn1 = __vminu4(mn1, __shfl_xor_sync(0xffffffffu, mn1, s));
                            }
                            // scale exponents: of this input (the smallest used one), of the next; every update
                            // warp has read those of the solve before
                            if (tiles > 0 && !(ok = wait_phase(tfree, (tiles - 1) & 1u, limit, s_abort))) break;
                            tiles += max(nt, 1);
                            if (lane < 2 * NB) {
                                float gn[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                                for (int q = 0; q < gln; ++q) {
                                    const float4 m4 = __ldcg(reinterpret_cast<const float4*>(
                                        gm + ((jo & 1) * N + gl0 + q) * RG));
                                    gn[0] = fmaxf(gn[0], m4.x);
                                    gn[1] = fmaxf(gn[1], m4.y);
                                    gn[2] = fmaxf(gn[2], m4.z);
                                    gn[3] = fmaxf(gn[3], m4.w);
                                }
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const unsigned mx = (q < 2 ? mx0 : mx1) >> (16 * (q & 1));
                                    const unsigned mn = (q < 2 ? mn0 : mn1) >> (16 * (q & 1));
                                    const int f = max((int)(mx & 0xffu), (int)(__float_as_uint(gn[q]) >> 23));
                                    S_.ecol[8 * cb + 4 * cp + q] = (int)((mn >> 8) & 0xffu) - 128;
                                    S_.epred[8 * cb + 4 * cp + q] = min(120, max(-120, 134 - f));
                                }
                            }
                            __syncwarp();
                            if (lane == 0) ptx::mbar_arrive(eready);
                        }
                        if (!even) {
                            // unequal scales: bring every group of 8 entries to the smallest exponent
                            for (int q = 0; q < NBC && ok; ++q)
                                if (q * part < n16) ok = wait_phase(&bfull[q], ~(lph >> q) & 1u, limit, s_abort);
                            if (!ok) break;
#pragma unroll 1
                            for (int v = lane; v < n16 * 2 * 4 * NB * 8; v += 32) {
                                const int kg = v / (4 * NB * 8), b8 = (v >> 5) % NB;
                                if (k0 / 8 + kg >= ng8) continue;
                                const u64* hw = hw0 + ((size_t)(k0 / 8 + kg) * NB + b8) * 4;
                                __half* p = reinterpret_cast<__half*>(Bbuf) + v * 8;
#pragma unroll 1
                                for (int u = 0; u < 8; ++u) {
                                    const unsigned w = (unsigned)__ldcg(hw + (u >> 1)) >> (16 * (u & 1));
                                    const int dd = S_.ecol[8 * b8 + u] - ((int)((w >> 8) & 0xffu) - 128);
                                    if (dd < 0) {
                                        const int d1 = max(dd, -14);
                                        const __half m1 = __ushort_as_half((unsigned short)half_pow2(d1));
                                        const __half m2 = __ushort_as_half((unsigned short)half_pow2(dd - d1));
                                        p[u] = __hmul(__hmul(p[u], m1), m2);
                                    }
                                }
                            }
                            ptx::fence_proxy_async_smem();
                            __syncwarp();
                            if (lane == 0) ptx::mbar_arrive(bgo);
                        }
                    }
            }
        }
        if (!ok) fail(A, S_);
        // gathers in flight land before the CTA leaves
        for (int q = 0; q < NBC; ++q) {
            const long long t0 = clock64();
            while (!fresh && !__all_sync(0xffffffffu, ptx::mbar_try(&bfull[q], ~(lph >> q) & 1u)) && clock64() - t0 < limit) {
            }
        }
    } else {
        // ------------------------------------------------------ update warps
        Upd u = {0, 0, 0, 0, 0};
        bool ok = true;
#pragma unroll 1
        for (int jo = 0; jo <= nvis && ok; ++jo) {
            if (jo > 0 || A.unmet) ok = group_sync(A, &S_, &u);
            ok = ok && begin_visit<RG, MT>(A, &S_, &u, jo);
            const int last = jo < nvis ? nsol : 0;
#pragma unroll 1
            for (int i = 0; i < last && ok;) {
                const int n = run_end(S_, jo, i);
                if (n > i) {
                    const Shape& R = S_.shape[8 + KIND_RING];
                    ok = R.nl == 1 && R.nt == 1 ? run_lines<RG, MT>(A, &S_, &u, jo, i, n) : run_blocks<RG, MT>(A, &S_, &u, jo, i, n);
                    i = n;
                } else {
                    ok = run_general<RG, MT>(A, &S_, &u, jo, i);
                    ++i;
                }
                // the centre joins the fronts after each team's last forward solve (one front: after the
                // centre; forward values of the boundary block may be read by other ranks in its backward
                // solve, after this barrier)
                if (ok && i - 1 == (two ? (team ? B - 2 - cen : cen - 1) : cen)) {
                    ok = group_sync(A, &S_, &u);
                    if (ok && two && team == 0) {
                        const AxisWin& wc = s_win[cen];
                        publish_input<RG, MT>(A, &S_, jo, pass_pos(jo, B, cen).M, KIND_CENTRE, SLOT_CENTRE, 0, u.tag + 1u, true,
                                              wc.lo + wc.ia, 0, 0, 1, S_.shape[8 + KIND_CENTRE].nl - 1);
                    }
                }
            }
        }
        if (!ok) fail(A, S_);
    }
    __syncwarp();
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(S_.tslot, 512);
}

// ----------------------------------------------------------------------- host

// The launch shape for nr right-hand sides.
struct TeamPlan {
    int RG, G, T, C, MT, per_launch;
    int KPmax, hdr_words, start_words, Emax, DZ, KB, stages, stage_bytes, off_b, off_misc;
    size_t smem, slot_bytes, start_bytes;
    // work space, in float2 units: FP32 fields, then what every launch starts at zero
    size_t oGv, oZv, oQf, oX, oH, oM, oC, total;
};

constexpr size_t SMEM_MAX = (size_t)227 * 1024;

size_t misc_bytes(int N, int B) {
    return sizeof(Sm) + (size_t)2 * N * sizeof(float2) + (size_t)2 * (B + 2) * 8 + (size_t)B * sizeof(AxisWin);
}

// The plan with G groups at a time.
bool plan_groups(const helm_ctx* h, int nr, int G, TeamPlan* P) {
    const int N = h->g.N, B = h->g.B, cen = h->g.cen;
    const bool two = h->g.sched == HELM_TWO_FRONT;
    const AxisWin* win = static_cast<const AxisWin*>(h->win_h);
    const int halves = h->team_halves;
    P->T = two ? 2 : 1;
    // one block of 8 right-hand sides, or groups of 16: the operator is streamed once per group
    P->RG = nr <= 8 ? 8 : 16;
    P->G = G;
    P->per_launch = P->G * P->RG;
    // the input sizes of every solve (each rank owns a part of each); blocks with windows of the same
    // shape give the same
    int kmax = 0, kstart = 0, gmin = 1 << 30;     // the first solve of a visit has a slot of its own
    std::vector<int> kinds = {0, B - 1};
    for (int q = 1; q < B - 1; ++q) {
        bool seen = false;
        for (size_t u = 2; u < kinds.size() && !seen; ++u)
            seen = win[kinds[u]].L == win[q].L && win[kinds[u]].ib - win[kinds[u]].ia == win[q].ib - win[q].ia;
        if (!seen) kinds.push_back(q);
    }
    for (int M : kinds)
        for (int Mp : kinds)
            for (int bwd = 0; bwd < 2; ++bwd) {
                const SolveGeo g = tm_geo(win[M], win[Mp], N, Mp, bwd, B, two);
                (g.boundary && !bwd ? kstart : kmax) = std::max(g.boundary && !bwd ? kstart : kmax, g.K);
                gmin = std::min(gmin, g.fin ? tm_ceil(g.K / g.in.nl, 8) : tm_ceil(g.K, 8));
                if (g.f0) gmin = std::min(gmin, tm_ceil(g.n0 / g.out0.nl, 8));
                if (g.f1) gmin = std::min(gmin, tm_ceil(g.n1 / g.out1.nl, 8));
            }
    // the usual solve: half way up the lower front
    const int Mt = std::max(1, cen / 2);
    const SolveGeo gt = tm_geo(win[Mt], win[Mt], N, Mt, 0, B, two);
    const int cg = tm_ceil(gt.K / gt.in.nl, 8);
    int C = std::max(1, std::min(h->dclus / (P->G * P->T), gmin));
    // groups of columns of a rank; its row groups at least team_min_groups with one line (below that
    // more ranks only add headers and polls), a group of columns with two (the longer rows stream
    // slower: n = 50, one front, d = 2 with 24 right-hand sides 23.8 -> 22.1 ms), then as few ranks as
    // keep that number
    const int want = std::max(tm_ceil(cg, C), std::max(1, h->team_min_groups / gt.in.nl));
    C = std::min(C, tm_ceil(cg, want));
    P->C = C;
    P->MT = gt.in.nl * tm_ceil(cg, C) <= 4 ? 64 : 128;
    P->KPmax = tm_kp(kmax);
    P->hdr_words = tm_ceil(kmax, 8) * (P->RG / 8) * 4;
    P->slot_bytes = (size_t)P->KPmax * 8 * P->RG;
    P->start_words = tm_ceil(kstart, 8) * (P->RG / 8) * 4;
    P->start_bytes = (size_t)tm_kp(kstart) * 8 * P->RG;
    P->Emax = N * h->g.Wmax;
    P->DZ = 0;
    for (int M = 0; M < B; ++M) P->DZ = std::max(P->DZ, win[M].ib - win[M].ia);
    // shared memory: the gathered input of the usual solve (larger ones in passes), the ring
    P->stage_bytes = P->MT / 16 * 2 * TKC * 16 * halves;
    const size_t misc = misc_bytes(N, B);
    const int cap = (int)((SMEM_MAX - misc - 4 * (size_t)P->stage_bytes - 256) / (size_t)(8 * P->RG)) / TKC * TKC;
    P->KB = std::min(TKC * tm_ceil(gt.K, TKC), cap);
    if (P->KB < TKC) return false;
    const size_t bb = (size_t)P->KB * 8 * P->RG;
    P->stages = (int)std::min<size_t>((SMEM_MAX - misc - bb - 256) / P->stage_bytes, MAXST);
    if (P->stages < 2) return false;
    P->off_b = P->stages * P->stage_bytes;
    P->off_misc = P->off_b + (int)bb;
    P->smem = (size_t)P->off_misc + misc;
    // ---- work space ----
    const size_t gN = (size_t)P->G * N, RG = P->RG, nt = (size_t)P->G * P->T;
    size_t o = 0;
    auto take = [&](size_t n) { const size_t r = o; o += (n + 15) & ~(size_t)15; return r; };
    take(gN * P->Emax * RG);                                     // V
    P->oGv = take(gN * N * P->DZ * RG);
    P->oZv = take(gN * N * P->DZ * RG);
    P->oQf = take((size_t)P->G * 4 * P->Emax * RG);
    P->oX = take(nt * (SLOT_START * P->slot_bytes + P->start_bytes) / 8);
    P->oH = take(nt * (size_t)(SLOT_START * P->hdr_words + P->start_words));
    P->oM = take(gN * RG);                                       // two tables of 4-byte words
    P->oC = take((size_t)P->G * 16);
    P->total = o;
    return true;
}

// The plan of an apply of nrhs right-hand sides in at most `limit` float2 of work
// space: as many groups of at most 64 right-hand sides in one launch as fit.
bool team_plan(const helm_ctx* h, int nrhs, TeamPlan* P, size_t limit) {
    const int nr = std::min(nrhs, 64), T = h->g.sched == HELM_TWO_FRONT ? 2 : 1;
    const int most = std::min(tm_ceil(nr, nr <= 8 ? 8 : 16), std::max(1, h->dclus / T));
    for (int G = most; G >= 1; --G)
        if (plan_groups(h, nr, G, P) && P->total <= limit) return true;
    return false;
}

const void* team_kernel(int RG, int MT) {
    if (RG == 8) return MT == 64 ? (const void*)k_team<8, 64> : (const void*)k_team<8, 128>;
    return MT == 64 ? (const void*)k_team<16, 64> : (const void*)k_team<16, 128>;
}

}  // namespace

// Operator table of the tensor-core forms; fills the byte and scale counts.  lo, where an
// operator has lo parts of some groups only: a unit of zeros, which stands for the others'
// parts, then of each such shape, per row group, the number of its lo parts or -1.
void team_table(helm_ctx* h, const DProb* dp, TProb* tp, size_t* gbytes, size_t* nscale, std::vector<int>* lo) {
    const int N = h->g.N, P = dense_nops(h->g.B);
    const bool fp16 = h->opts.precision == HELM_FP16;
    h->team_halves = fp16 ? 1 : 2;
    size_t off = 0, soff = 0;
    for (int p = 0; p < P; ++p) {
        TProb t;
        memset(&t, 0, sizeof(t));
        const DProb& D = dp[p];
        t.off = (long long)off;
        t.soff = (long long)soff;
        if (D.n_out > 0) {
            t.n_out = D.n_out;
            t.n_in = D.n_in;
            t.in = D.in;
            t.out[0] = D.out[0];
            t.out[1] = D.nrect > 1 ? D.out[1] : DRect{0, 1, 0, 1};
            t.ng0 = tm_ceil(D.out[0].nl * D.out[0].nz * N, 8);
            t.ng1 = D.nrect > 1 ? tm_ceil(D.out[1].nl * D.out[1].nz * N, 8) : 0;
            t.KP = tm_kp(D.n_in);
            t.xr = fp16 ? D.xr : 0;
            t.halves = fp16 && D.xr == 0 ? 1 : 2;
            if (t.xr > 0) {
                // a shape seen before has its table already
                int q = 0;
                while (q < p && !(tp[q].nlo > 0 && tp[q].xr == t.xr && tp[q].n_out == t.n_out && tp[q].ng0 == t.ng0 &&
                                  tp[q].out[0].nl == t.out[0].nl && tp[q].out[0].nz == t.out[0].nz &&
                                  tp[q].out[1].nl == t.out[1].nl && tp[q].out[1].nz == t.out[1].nz))
                    ++q;
                if (q < p) {
                    t.nlo = tp[q].nlo;
                    t.lob = tp[q].lob;
                } else {
                    if (lo->empty()) lo->assign(TKC * 32 / sizeof(int), 0);
                    t.lob = (int)lo->size();
                    for (int g = 0; g < t.ng0 + t.ng1; ++g) {
                        const int r = g >= t.ng0, n0 = t.out[0].nl * t.out[0].nz * N;
                        const DRect& R = t.out[r];
                        bool some = false;
                        for (int u = 0; u < 8; ++u) {
                            const int i = 8 * (g - (r ? t.ng0 : 0)) + u, l = i % R.nl, tt = i / R.nl, zr = tt % R.nz, x = tt / R.nz;
                            const int o = (r ? n0 : 0) + x + N * (zr + R.nz * l);
                            some = some || (x < N && o % (64 + t.xr) >= 64);
                        }
                        lo->push_back(some ? t.nlo++ : -1);
                    }
                }
            }
            h->team_halves = std::max(h->team_halves, t.halves);
            off += t.nlo > 0 ? (size_t)(t.ng0 + t.ng1 + t.nlo) * t.KP * 32 : tm_bytes(t.ng0 + t.ng1, t.KP, t.halves);
            soff += (size_t)(t.ng0 + t.ng1) * 16;
        }
        tp[p] = t;
    }
    *gbytes = off;
    *nscale = soff;
}

// Packs the listed operators (their complex FP32 rows in Gt at goff).
cudaError_t team_pack(helm_ctx* h, const int* ops, int nops, const float2* Gt, const long long* d_goff,
                      void** d_items, size_t* cap, cudaStream_t st) {
    std::vector<PackItem> items;
    for (int q = 0; q < nops; ++q)
        for (int g = 0; g < h->tprob_h[ops[q]].ng0 + h->tprob_h[ops[q]].ng1; ++g) items.push_back(PackItem{ops[q], g});
    if (items.empty()) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (items.size() * sizeof(PackItem) > *cap) {
        if (*d_items) cudaFree(*d_items);
        *d_items = nullptr;
        *cap = 0;
        e = cudaMalloc(d_items, items.size() * sizeof(PackItem));
        if (e != cudaSuccess) return e;
        *cap = items.size() * sizeof(PackItem);
    }
    const PackItem* di = static_cast<const PackItem*>(*d_items);
    e = cudaMemcpyAsync(*d_items, items.data(), items.size() * sizeof(PackItem), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    k_team_pack<<<(unsigned)items.size(), 128, 0, st>>>(h->tprob, di, Gt, d_goff, h->dG, h->dscale, h->dlo, h->g.N);
    h->launches++;
    e = cudaGetLastError();
    // the item list above must outlive its copy
    const cudaError_t e2 = cudaStreamSynchronize(st);
    return e != cudaSuccess ? e : e2;
}

cudaError_t team_unpack(helm_ctx* h, int p, float2* G, cudaStream_t st) {
    k_team_unpack<<<512, 256, 0, st>>>(h->tprob_h[p], h->dG, h->dscale, h->dlo, h->g.N, G);
    h->launches++;
    return cudaGetLastError();
}

// CTAs an apply launch may use: every one is resident (one per SM), at most 8
// per opts.dense_clusters.
int team_configure(helm_ctx* h) {
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const void* kfns[4] = {team_kernel(8, 64), team_kernel(8, 128), team_kernel(16, 64), team_kernel(16, 128)};
    for (const void* k : kfns) {
        if (e == cudaSuccess) e = ensure_dyn_smem(k, SMEM_MAX);
        int q = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k, TT, SMEM_MAX);
        if (q < 1 && e == cudaSuccess) return HELM_ENOTSUP;
    }
    if (e != cudaSuccess) {
        helm_set_cuda_error(e);
        return HELM_ECUDA;
    }
    h->dclus = nsm;
    if (h->opts.dense_clusters > 0) h->dclus = std::min(h->dclus, HELM_DENSE_CS * h->opts.dense_clusters);
    h->team_min_groups = 3;
    h->team_halves = 2;                  // until the operators are known
    if (h->dclus < (h->g.sched == HELM_TWO_FRONT ? 2 : 1)) return HELM_ENOTSUP;
    TeamPlan P;
    return team_plan(h, 1, &P, (size_t)-1) && team_plan(h, 64, &P, (size_t)-1) ? HELM_OK : HELM_ENOTSUP;
}

size_t team_work_elems(const helm_ctx* h, int nrhs, size_t limit) {
    TeamPlan P;
    return team_plan(h, nrhs, &P, limit) ? P.total : (size_t)-1;
}

cudaError_t launch_team_apply(helm_ctx* h, const float2* r, float2* z, int nrhs, float2* work, size_t elems,
                              cudaStream_t st) {
    const size_t n3 = (size_t)h->g.N * h->g.N * h->g.N;
    TeamPlan P0;
    if (!team_plan(h, nrhs, &P0, elems)) return cudaErrorInvalidValue;
    for (int r0 = 0; r0 < nrhs; r0 += P0.per_launch) {
        const int nr = std::min(P0.per_launch, nrhs - r0);
        TeamPlan P;                                   // the last launch may need fewer groups
        if (!team_plan(h, nr, &P, elems)) return cudaErrorInvalidValue;
        TeamArgs A;
        memset(&A, 0, sizeof(A));
        A.g = h->g;
        A.win = h->t.win;
        A.tp = h->tprob;
        A.G = h->dG;
        A.scale = h->dscale;
        A.lo = h->dlo;
        A.c_dn = h->t.c_dn;
        A.c_up = h->t.c_up;
        A.rin = r + (size_t)r0 * n3;
        A.zout = z + (size_t)r0 * n3;
        A.V = work;
        A.Gv = work + P.oGv;
        A.Zv = work + P.oZv;
        A.Qf = work + P.oQf;
        A.X = reinterpret_cast<unsigned char*>(work + P.oX);
        A.hdr = reinterpret_cast<u64*>(work + P.oH);
        A.gmax = reinterpret_cast<unsigned*>(work + P.oM);
        A.ctr = reinterpret_cast<unsigned*>(work + P.oC);
        A.err = h->dev_err;
        A.slot_bytes = P.slot_bytes;
        A.hdr_words = P.hdr_words;
        A.start_bytes = P.start_bytes;
        A.start_words = P.start_words;
        A.nrhs = nr;
        A.T = P.T;
        A.C = P.C;
        A.DZ = P.DZ;
        A.Emax = P.Emax;
        A.KB = P.KB;
        A.stages = P.stages;
        A.stage_bytes = P.stage_bytes;
        A.off_b = P.off_b;
        A.off_misc = P.off_misc;
        A.wait_cycles = h->opts.wait_cycles;
        A.unmet = h->opts.debug_unmet_wait;
        // no header of this launch, empty tables and counters
        cudaError_t e = cudaMemsetAsync(work + P.oH, 0, (P.total - P.oH) * sizeof(float2), st);
        if (e != cudaSuccess) return e;
        // the CTAs wait on one another: a cooperative launch starts them together or not at all
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.gridDim = dim3((unsigned)(P.G * P.T * P.C), 1, 1);
        cfg.blockDim = dim3(TT, 1, 1);
        cfg.dynamicSmemBytes = P.smem;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const void* kfn = team_kernel(P.RG, P.MT);
        e = ensure_dyn_smem(kfn, SMEM_MAX);
        if (e != cudaSuccess) return e;
        void* args[] = {&A};
        e = cudaLaunchKernelExC(&cfg, kfn, args);
        if (e != cudaSuccess) return e;
        h->launches++;
    }
    return cudaSuccess;
}
