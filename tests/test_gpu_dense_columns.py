"""The two kernels of the dense setup's operator columns give the same bits.

Blocks up to 32 are solved one thread per column, larger ones in 64-row tiles.  Both
follow one substitution, and an operator entry must not depend on which one made it:
rounded to FP16, entries that differ in their last bit differ by a whole step of 2^-11.
The kernels are compiled here as the library compiles them and run on the same
random factor blocks and complex couplings, at block sizes on both sides of each
limit between the column kernel's instances.
"""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

HARNESS = r'''
#include "dense.cu"
#include <stdio.h>
#include <stdlib.h>

static float rnd() { return (float)rand() / (float)RAND_MAX - 0.5f; }

int main() {
    const int shapes[][2] = {{3, 3}, {2, 5}, {11, 1}, {4, 4}, {1, 17}, {5, 5}, {2, 13}, {9, 3}, {4, 8}};   // Ly, Lz
    int bad = 0;
    for (const auto& sh : shapes)
        for (int N = 6; N <= 21; N += 5) {
            const int Ly = sh[0], Lz = sh[1], k = Ly * Lz, ldk = 8 * ((k + 7) / 8) + 2, q = g_class(k);
            Geom g;
            memset(&g, 0, sizeof(g));
            g.N = N;
            Prob P;
            memset(&P, 0, sizeof(P));
            P.k = k; P.Ly = Ly; P.Lz = Lz; P.ylo = 4; P.ldk = ldk; P.kstride = k * ldk;
            DProb D;
            memset(&D, 0, sizeof(D));
            // all but the last line in; the first line's upper rows and the other lines out
            D.in = DRect{4, Ly > 1 ? Ly - 1 : 1, 0, Lz};
            D.nrect = Ly > 1 ? 2 : 1;
            D.out[0] = DRect{4, 1, Lz / 2, Lz - Lz / 2};
            D.out[1] = DRect{5, Ly - 1, 0, Lz};
            D.n_in = D.in.nl * D.in.nz * N;
            for (int r = 0; r < D.nrect; ++r) D.n_out += D.out[r].nl * D.out[r].nz * N;
            std::vector<GItem> items;
            for (int j0 = 0; j0 < D.n_in; j0 += GW) items.push_back(GItem{0, j0});
            std::vector<float2> fac((size_t)N * k * ldk), cdn(N), cup(N);
            for (auto& v : fac) v = make_float2(rnd(), rnd());
            // complex in the outer third on each side, real between, as in a PML
            for (int x = 0; x < N; ++x) {
                const bool pml = x < N / 3 || x >= N - N / 3;
                cdn[x] = make_float2(1.f + rnd(), pml ? rnd() : 0.f);
                cup[x] = make_float2(1.f + rnd(), pml ? rnd() : 0.f);
            }
            const long long goff0 = 0;
            const size_t ng = (size_t)D.n_out * D.n_in, yslot = (size_t)N * 64 * GW;
            Tables t;
            memset(&t, 0, sizeof(t));
            void *d_dn, *d_up, *d_prob, *d_dp, *d_items, *d_fac, *d_goff, *d_y, *d_g[2];
            const size_t nb = items.size();
            cudaMalloc(&d_dn, N * 8); cudaMalloc(&d_up, N * 8); cudaMalloc(&d_prob, sizeof(P)); cudaMalloc(&d_dp, sizeof(D));
            cudaMalloc(&d_items, nb * sizeof(GItem)); cudaMalloc(&d_fac, fac.size() * 8); cudaMalloc(&d_goff, 8);
            cudaMalloc(&d_y, nb * yslot * 8); cudaMalloc(&d_g[0], ng * 8); cudaMalloc(&d_g[1], ng * 8);
            cudaMemcpy(d_dn, cdn.data(), N * 8, cudaMemcpyHostToDevice);
            cudaMemcpy(d_up, cup.data(), N * 8, cudaMemcpyHostToDevice);
            cudaMemcpy(d_prob, &P, sizeof(P), cudaMemcpyHostToDevice);
            cudaMemcpy(d_dp, &D, sizeof(D), cudaMemcpyHostToDevice);
            cudaMemcpy(d_items, items.data(), nb * sizeof(GItem), cudaMemcpyHostToDevice);
            cudaMemcpy(d_fac, fac.data(), fac.size() * 8, cudaMemcpyHostToDevice);
            cudaMemcpy(d_goff, &goff0, 8, cudaMemcpyHostToDevice);
            for (void* p : d_g) cudaMemset(p, 0xff, ng * 8);
            t.c_dn = (float2*)d_dn; t.c_up = (float2*)d_up; t.prob = (Prob*)d_prob;
            const size_t gsm = (size_t)(64 * TLD + 2 * 64 * GW) * sizeof(float2) + (2 * GW + 64) * sizeof(int);
            cudaFuncSetAttribute(k_dense_G, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm);
            k_dense_G<<<(int)nb, GT, gsm>>>(g, t, (DProb*)d_dp, (GItem*)d_items, (int)nb, (float2*)d_fac, 0, (float2*)d_g[0],
                                            (long long*)d_goff, (float2*)d_y, yslot);
            G_COLS[q].fn<<<(int)nb, GW>>>(g, t, (DProb*)d_dp, (GItem*)d_items, (int)nb, (float2*)d_fac, 0, (float2*)d_g[1],
                                          (long long*)d_goff, (float2*)d_y, yslot);
            std::vector<unsigned long long> a(ng), b(ng);
            cudaMemcpy(a.data(), d_g[0], ng * 8, cudaMemcpyDeviceToHost);
            cudaMemcpy(b.data(), d_g[1], ng * 8, cudaMemcpyDeviceToHost);
            if (cudaGetLastError() != cudaSuccess) return 2;
            size_t diff = 0, unset = 0;
            for (size_t e = 0; e < ng; ++e) diff += a[e] != b[e], unset += a[e] == ~0ull;
            if (diff || unset) {
                printf("k %d (at most %d), N %d: %zu of %zu entries differ, %zu not written\n", k, G_COLS[q].km, N, diff, ng, unset);
                bad = 1;
            }
            void* ptrs[] = {d_dn, d_up, d_prob, d_dp, d_items, d_fac, d_goff, d_y, d_g[0], d_g[1]};
            for (void* p : ptrs) cudaFree(p);
        }
    return bad;
}
'''


def test_both_column_kernels_give_the_same_bits(tmp_path):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1502_07266_gb300 import build as B
    src, exe = tmp_path / "columns.cu", str(tmp_path / "columns")
    src.write_text(HARNESS)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    r = subprocess.run([nvcc, *B.ARCH, *B.FLAGS, "-I", B.CSRC, str(src), "-o", exe, "-L", B.LIBDIR, "-lhelm",
                        "-Xlinker", "-rpath", "-Xlinker", B.LIBDIR], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300, env=dict(os.environ))
    assert r.returncode == 0, r.stdout + r.stderr
