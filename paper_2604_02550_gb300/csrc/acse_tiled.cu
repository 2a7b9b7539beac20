// Shared-memory, register-tiled O(r^5) kernels of a contraction pass: Z of the split path, and the B kernels
// of both arithmetic paths (T = double for the FP64 path, T = float for the split-precision path).
//
//   Z^{kp}_{js} = sum_q W^{kp}_{qs} 1D^j_q  ->  for each (k, p): Z_kp = 1D . W_kp   (r x r x r)
//   w^k_s = sum_pq W^{kp}_{qs} 1D^p_q = sum_p Z^{kp}_{ps}: the diagonal j = p of Z, so the Z kernel
//       also writes its rows j = p and a small kernel sums them over p
//   B spin types (one block per pair (i, j)): X1 = X_ij . 1D and X2 = w . M_ij^T as r x r x r
//       products plus gathered terms; the block then forms directly
//         H_b^{ij}_{kl} = 4 Y_b^{ij}_{kl} - 12 (P^{ij}_{kl} - P'^{ij}_{lk}),
//       (P, P') = (B_aaaa, B_aaaa), (B_abab, B_abba), (B_bbbb, B_bbbb) for b = aa, ab, bb, so that the
//       residual / update is G_b = H_b - s H_b^T (a plain pair transpose, acse_elem.cu).
// Thread micro-tiles are 4 x 4 outputs over r padded to a multiple of 4; operands sit in shared
// memory laid out so that each thread reads 4-vectors.
#include <cuda_bf16.h>
#include <type_traits>

#include "acse_internal.h"
#include "dfloat.cuh"

#define ZP_MAX_THREADS 288

__device__ __forceinline__ float tl_tf32(float x) {
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
    return __uint_as_float(u);
}

__host__ __device__ __forceinline__ int pad4(int r) { return (r + 3) & ~3; }

// --------------------------------------------------------------------------- outputs of Z
struct ZOut {
    void* Zd;      // (2 r^2) rows
    void* Zf[2];   // r^2 rows
    int mode;      // 1 = BF16x3 (A pattern [hi|hi|lo]), 2 = TF32, 3 = TF32x3 ([hi|hi|lo])
    int ldd, ldf;  // row length in elements
    int Kp1, Kp2;  // K segment length
    void* diag;    // [4][r][r][r]: rows j = p of Zd(a,a), Zd(b,b), Zf1, Zf2
    int ntypes;    // spin types computed (6, or 3 with the spin-flip specialisation) ...
    int tmap[6];   // ... and which: block type index -> t
};

__device__ __forceinline__ void z_store(const ZOut& o, int which, size_t row, int col, float v) {
    void* base = which < 0 ? o.Zd : o.Zf[which];
    const size_t ld = which < 0 ? (size_t)o.ldd : (size_t)o.ldf;
    const int Kp = which < 0 ? o.Kp2 : o.Kp1;
    if (o.mode == 1) {
        __nv_bfloat16* p = (__nv_bfloat16*)base + row * ld;
        const float x = v;
        const __nv_bfloat16 hi = __float2bfloat16_rn(x);
        const __nv_bfloat16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
        p[col] = hi;
        p[Kp + col] = hi;
        p[2 * Kp + col] = lo;
    } else if (o.mode == 3) {
        float* p = (float*)base + row * ld;
        const float hi = tl_tf32(v);
        const float lo = tl_tf32(v - hi);
        p[col] = hi;
        p[Kp + col] = hi;
        p[2 * Kp + col] = lo;
    } else {
        ((float*)base + row * ld)[col] = tl_tf32(v);
    }
}

// Four consecutive columns col..col+3 of one output row (requires row * ld + col % 4 == 0); MODE is
// the ZOut mode.
template <int MODE>
__device__ __forceinline__ void z_store4(const ZOut& o, int which, size_t row, int col, const float (&v)[4]) {
    void* base = which < 0 ? o.Zd : o.Zf[which];
    const size_t ld = which < 0 ? (size_t)o.ldd : (size_t)o.ldf;
    const int Kp = which < 0 ? o.Kp2 : o.Kp1;
    if (MODE == 1) {
        __nv_bfloat16 hi[4], lo[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            hi[u] = __float2bfloat16_rn(v[u]);
            lo[u] = __float2bfloat16_rn(v[u] - __bfloat162float(hi[u]));
        }
        uint2 H, L;
        memcpy(&H, hi, 8);
        memcpy(&L, lo, 8);
        __nv_bfloat16* q = (__nv_bfloat16*)base + row * ld + col;
        *reinterpret_cast<uint2*>(q) = H;
        *reinterpret_cast<uint2*>(q + Kp) = H;
        *reinterpret_cast<uint2*>(q + 2 * Kp) = L;
    } else if (MODE == 3) {
        float hi[4], lo[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            hi[u] = tl_tf32(v[u]);
            lo[u] = tl_tf32(v[u] - hi[u]);
        }
        float* q = (float*)base + row * ld + col;
        *reinterpret_cast<float4*>(q) = make_float4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<float4*>(q + Kp) = make_float4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<float4*>(q + 2 * Kp) = make_float4(lo[0], lo[1], lo[2], lo[3]);
    } else {
        float* q = (float*)base + row * ld + col;
        *reinterpret_cast<float4*>(q) =
            make_float4(tl_tf32(v[0]), tl_tf32(v[1]), tl_tf32(v[2]), tl_tf32(v[3]));
    }
}

// Asynchronous global -> shared copies (cp.async, completion tracked per thread by commit groups).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// The r x r slice W_kp[q][s] of spin type t (t = 0..5, see k_Z_pipe) and whether it is stored [s][q].
__device__ __forceinline__ const float* z_slice(int t, int k, int p, int r, const float* Waa, const float* Wab,
                                                const float* Wbb, bool& transposed) {
    const size_t r3 = (size_t)r * r * r, R2 = (size_t)r * r;
    switch (t) {
        case 0: transposed = false; return Waa + k * r3 + p * R2;
        case 1: transposed = false; return Wab + k * r3 + p * R2;
        case 2: transposed = true; return Wab + p * r3 + k * R2;
        case 3: transposed = false; return Wbb + k * r3 + p * R2;
        case 4: transposed = true; return Wab + k * r3 + p * R2;
        default: transposed = false; return Wab + p * r3 + k * R2;
    }
}

// Z_kp = 1D . W_kp for spin type t and all p of a chunk, one block per (t, k, p-chunk):
//   t=0 Zd(a,a): W_kp[q][s] = Waa[k][p][q][s], ga      t=1 Zd(a,b): Wab[k][p][q][s], ga
//   t=2 Zd(b,a): W_kp[q][s] = Wab[p][k][s][q], gb      t=3 Zd(b,b): Wbb[k][p][q][s], gb
//   t=4 Zf1:     W_kp[q][s] = Wab[k][p][s][q], gb      t=5 Zf2:     Wab[p][k][q][s], ga
// (the spin-flip sectors drop a sign -1 that their M operand drops too).  The W slices of the next ipb
// values of p are copied into shared memory (cp.async) while the current ipb slices are multiplied;
// each thread owns one 4 x 4 output tile of one slice (ipb * (rp/4)^2 threads).  W is its FP32 copy, so that
// no FP64 conversion runs here (split path; the FP64-accurate paths transform after the product, acse_ph.cu).
template <int MODE, int RP = 0>   // RP > 0: compile-time padded size (product loop fully unrolled)
__global__ void __launch_bounds__(ZP_MAX_THREADS, 3) k_Z_pipe(int r, int ipb, int pchunk, const float* __restrict__ Waa,
                                                              const float* __restrict__ Wab,
                                                              const float* __restrict__ Wbb,
                                                              const double* __restrict__ gam,
                                                              const __grid_constant__ ZOut o) {
    constexpr int WV = 4;                                // elements of a 16-byte copy
    extern __shared__ __align__(16) unsigned char tl_smem[];
    const int rp = RP ? RP : pad4(r), ldw = rp + 4, R2 = r * r, R2e = (R2 + WV - 1) / WV * WV;
    const int nt = rp / 4, nt2 = nt * nt;
    float* stage = (float*)tl_smem;                            // [ipb][R2e] raw W slices
    float* gT = (float*)(stage + (size_t)ipb * R2e);             // [q][j] = 1D[j][q], row pitch ldw
    float* Ws = gT + (size_t)rp * ldw;                       // [ipb][q][s], row pitch ldw
    const int nchunk = (r + pchunk - 1) / pchunk;
    const int tb = blockIdx.x / (r * nchunk);
    const int t = o.tmap[tb];
    const int rem = blockIdx.x - tb * r * nchunk;
    const int k = rem / nchunk;
    const int pb = (rem - k * nchunk) * pchunk;
    const int pe = min(r, pb + pchunk);
    const double* g = gam + ((t == 2 || t == 3 || t == 4) ? R2 : 0);
    // (int)((e + 1/2) / r) = e / r for e < r^2: the fraction stays at least 1/(2r) from an integer
    const float invr = 1.f / (float)r;
    const bool vec_ld = R2 % WV == 0 && ((reinterpret_cast<uintptr_t>(Waa) | reinterpret_cast<uintptr_t>(Wab) |
                                          reinterpret_cast<uintptr_t>(Wbb)) & 15) == 0;
    for (int e = threadIdx.x; e < (1 + ipb) * rp * ldw; e += blockDim.x) gT[e] = 0.f;
    __syncthreads();
    for (int e = threadIdx.x; e < R2; e += blockDim.x) {
        const int u = e / r, v = e - u * r;
        gT[v * ldw + u] = (float)g[e];                // g[j][q] -> gT[q][j]
    }
    auto issue = [&](int p0) {
        const int n = min(ipb, pe - p0);
        for (int it = 0; it < n; ++it) {
            bool tr;
            const float* src = z_slice(t, k, p0 + it, r, Waa, Wab, Wbb, tr);
            float* dst = stage + (size_t)it * R2e;
            if (vec_ld)
                for (int e = threadIdx.x; e < R2 / WV; e += blockDim.x) cp_async16(dst + WV * e, src + WV * e);
            else
                for (int e = threadIdx.x; e < R2; e += blockDim.x) cp_async4(dst + e, src + e);
        }
        cp_async_commit();
    };
    issue(pb);
    int which, sK, sP;
    if (t < 4) { which = -1; sK = t >> 1; sP = t & 1; }
    else { which = t - 4; sK = 0; sP = 0; }
    const int dslot = t == 0 ? 0 : t == 3 ? 1 : t == 4 ? 2 : t == 5 ? 3 : -1;
    const int it_me = threadIdx.x / nt2, tile = threadIdx.x - it_me * nt2;
    const int j0 = (tile / nt) * 4, s0 = (tile % nt) * 4;
    const size_t ld = which < 0 ? (size_t)o.ldd : (size_t)o.ldf;
    for (int p0 = pb; p0 < pe; p0 += ipb) {
        const int n = min(ipb, pe - p0);
        cp_async_wait_all();
        __syncthreads();                                 // slices landed; previous products done with Ws
        for (int it = 0; it < n; ++it) {
            bool tr;
            z_slice(t, k, p0 + it, r, Waa, Wab, Wbb, tr);
            const float* st = stage + (size_t)it * R2e;
            float* W = Ws + (size_t)it * rp * ldw;
            for (int e = threadIdx.x; e < R2; e += blockDim.x) {
                const int u = (int)(((float)e + 0.5f) * invr), v = e - u * r;   // e / r, see invr
                const float x = st[e];
                if (tr) W[v * ldw + u] = x;                // src[s][q] -> W[q][s]
                else W[u * ldw + v] = x;
            }
        }
        __syncthreads();                                 // Ws ready, stage free
        if (p0 + ipb < pe) issue(p0 + ipb);              // the next slices load during the products
        if (it_me >= n) continue;
        const int p = p0 + it_me;
        float acc[4][4];
        const float* W = Ws + (size_t)it_me * rp * ldw;
        // with RP the loop runs over the zero-padded rows too (q < RP), at a constant trip count
        // packed FP32x2 FMA, pairs along s (the same FMA sequence per element as scalar code)
        float2 c2[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) c2[u][0] = c2[u][1] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int q = 0; q < (RP ? RP : r); ++q) {
            float a[4], b[4];
            ld4(gT + q * ldw + j0, a);
            ld4(W + q * ldw + s0, b);
            const float2 b0 = make_float2(b[0], b[1]), b1 = make_float2(b[2], b[3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 x = make_float2(a[u], a[u]);
                c2[u][0] = __ffma2_rn(x, b0, c2[u][0]);
                c2[u][1] = __ffma2_rn(x, b1, c2[u][1]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            acc[u][0] = c2[u][0].x; acc[u][1] = c2[u][0].y; acc[u][2] = c2[u][1].x; acc[u][3] = c2[u][1].y;
        }
        const int col0 = sP * R2 + p * r + s0;
        const bool vec_st = s0 + 3 < r && ((size_t)col0 & 3) == 0 && (ld & 3) == 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u;
            if (j >= r) continue;
            const size_t row = (size_t)sK * R2 + (size_t)k * r + j;
            if (vec_st) z_store4<MODE>(o, which, row, col0, acc[u]);
            else
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (s0 + v < r) z_store(o, which, row, col0 + v, acc[u][v]);
            if (dslot >= 0 && j == p)
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (s0 + v < r) {
                        const size_t di = ((size_t)dslot * R2 + (size_t)k * r + p) * r + s0 + v;
                        ((float*)o.diag)[di] = acc[u][v];
                    }
        }
    }
    cp_async_wait_all();
}

// w_a[k][s] = sum_p (Zd(a,a)[(k,p)][(p,s)] - Zf1[(k,p)][(p,s)]),  w_b likewise with Zd(b,b), Zf2
// (= sum_pq Waa[k][p][q][s] ga[p][q] - sum_pq Wab[k][p][s][q] gb[p][q], and the b analogue).
// One block per (spin, k): warp w sums p = w, w + 8, ...; lanes over s; the 8 partials are added
// in a fixed order.
template <typename T>
__global__ void __launch_bounds__(256) k_w_from_diag(int r, const T* __restrict__ diag, T* __restrict__ wout,
                                                     int flip) {
    __shared__ T part[8][ACSE_MAX_R];
    const int R2 = r * r;
    const int sp = blockIdx.x / r, k = blockIdx.x % r;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // flip: w_b = w_a (spin-flip specialisation; slots 1 and 3 are not formed)
    const T* d0 = diag + (size_t)(sp == 0 || flip ? 0 : 1) * R2 * r;
    const T* d1 = diag + (size_t)(sp == 0 || flip ? 2 : 3) * R2 * r;
    for (int s = lane; s < r; s += 32) {
        T acc = 0;
        for (int p = w; p < r; p += 8) acc += d0[((size_t)k * r + p) * r + s] - d1[((size_t)k * r + p) * r + s];
        part[w][s] = acc;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < r; s += blockDim.x) {
        T acc = 0;
#pragma unroll
        for (int g = 0; g < 8; ++g) acc += part[g][s];
        wout[(size_t)sp * R2 + (size_t)k * r + s] = acc;
    }
}

// ------------------------------------------------------------------------- B -> H
struct BTiledArgs {
    int r;
    const float* X[3];      // pair GEMM outputs X^{ij}_{kp}, row stride r^2
    const float* Y[3];      // pair GEMM outputs Y^{ij}_{kl}
    const float* X5d;       // (2r^2) x (2r^2), rows (sK,k,j), columns (sI,i,l)
    const float* X5f1;      // r^2 x r^2
    const float* X5f2;
    const float* M[3];
    const float* gam;
    const float* w;
    const float* Q;
    float* H[3];
    const float* ny[4];     // NY three-body term per spin type (acse_ny.cu), added to B; null for V
    int flip;           // spin-flip specialisation: no bb items; the b-led particle-hole blocks and the
                        // second flip sector are read as their alpha-led flips
    const float* bx[8];   // precomputed products (k_B_pipe<.., true>): per type t, x1 rows at bx[2t] and x2^T rows at
                          // bx[2t + 1], r^2 per item (the type's item number, see acse_btc.cu)
};

// Arguments of k_B_pre (FP64 and Ozaki paths): Y, the particle-hole product, 1D, Q, the NY term or null, and the
// precomputed products, per type t x1 rows at bx[2t] and x2^T rows at bx[2t + 1] of every pair ij.
struct BPreArgs {
    int r;
    const double* Y[3];
    const double* X5d;
    const double* X5f1;
    const double* X5f2;
    const double* gam;
    const double* Q;
    double* H[3];
    const double* ny[4];
    const double* bx[8];
    const int* pmap;    // pair number -> i r + j (i < j)
};

// FP64 and Ozaki paths.  Spin types t = 0 (aaaa), 1 (bbbb), 2 (abab), 3 (abba); the products x1[k][l] and x2^T[l][k]
// of every type come precomputed (a.bx: launch_Bx), so that a block only gathers and combines.  With U = x2^T read
// in its own order, U[a][b] = x2[b][a], and R = x1 - x4 + 2 x5 + x7 - 2 x8 (the gathered terms of acse_elem.cu),
//     9 (B_t[k][l] - B_t[l][k]) = V[k][l] - V[l][k],  V = R + 2 U,                         t = 0, 1
//     9 (B_2[k][l] - B_3[l][k]) = N[k][l] - N'[l][k],  N = R_2 + 2 U_3,  N' = R_3 - 2 U_2  (x1 of type 3 negated),
// so every operand is read in rows of l and one r x r array crosses through shared memory:
//     H_aa = 4 Y_aa - (4/3)(V - V^T), H_bb likewise, H_ab = 4 Y_ab - (4/3)(N - N'^T).
// Blocks: the pairs i < j of aa and of bb (row (j, i) of H is minus row (i, j), rows (i, i) are zero), every pair of
// ab.  The FP64 pipe (two operations a clock and SM) bounds it at about 19 r^4 operations, HBM at 17 r^4 doubles:
// r = 48: 217 us, against 628 us for the kernel that combined all r^2 pairs of each type entry by entry.
__global__ void __launch_bounds__(256) k_B_pre(const __grid_constant__ BPreArgs a) {
    extern __shared__ __align__(16) double bp_sm[];   // N [r][ld], N' [r][ld] (ab)
    const int r = a.r, R2 = r * r, ld = r | 1, P = r * (r - 1) / 2;
    const size_t R22 = 2 * (size_t)R2;
    const double *ga = a.gam, *gb = a.gam + R2, *Qa = a.Q, *Qb = a.Q + R2;
    if ((int)blockIdx.x < 2 * P) {
        const int sec = (int)blockIdx.x / P, ij = a.pmap[(int)blockIdx.x - sec * P], i = ij / r, j = ij - i * r;
        const double* g = sec ? gb : ga;
        const double* Q = sec ? Qb : Qa;
        const double* X5 = a.X5d + (sec ? R2 * R22 + R2 : 0);
        const double* x1 = a.bx[2 * sec] + (size_t)ij * R2;
        const double* U = a.bx[2 * sec + 1] + (size_t)ij * R2;
        const double* ny = a.ny[sec] ? a.ny[sec] + (size_t)ij * R2 : nullptr;
        for (int e = threadIdx.x; e < R2; e += blockDim.x) {
            const int k = e / r, l = e - k * r;
            const double x5 = X5[((size_t)k * r + j) * R22 + (size_t)i * r + l], x8 = X5[((size_t)k * r + i) * R22 + (size_t)j * r + l];
            double v = fma(2.0, (x5 - x8) + U[e], x1[e]);
            v = fma(-Q[k * r + i], g[j * r + l], v);
            v = fma(Q[k * r + j], g[i * r + l], v);
            if (ny) v = fma(9.0, ny[e], v);
            bp_sm[k * ld + l] = v;
        }
        __syncthreads();
        const double* Y = a.Y[2 * sec] + (size_t)ij * R2;
        double* H = a.H[2 * sec] + (size_t)ij * R2;
        double* Hm = a.H[2 * sec] + ((size_t)j * r + i) * R2;
        for (int e = threadIdx.x; e < R2; e += blockDim.x) {
            const int k = e / r, l = e - k * r;
            const double h = fma(-4.0 / 3.0, bp_sm[k * ld + l] - bp_sm[l * ld + k], 4.0 * Y[e]);
            H[e] = h;
            Hm[e] = -h;
        }
    } else {
        const int ij = (int)blockIdx.x - 2 * P, i = ij / r, j = ij - i * r;
        double* Nt = bp_sm + r * ld;
        const double *x12 = a.bx[4] + (size_t)ij * R2, *U2 = a.bx[5] + (size_t)ij * R2;
        const double *x13 = a.bx[6] + (size_t)ij * R2, *U3 = a.bx[7] + (size_t)ij * R2;
        const double* ny2 = a.ny[2] ? a.ny[2] + (size_t)ij * R2 : nullptr;
        const double* ny3 = a.ny[3] ? a.ny[3] + (size_t)ij * R2 : nullptr;
        for (int e = threadIdx.x; e < R2; e += blockDim.x) {
            const int k = e / r, l = e - k * r;
            // type 2: x5 = X5f1, x8 = X5d(a,b), x4 = Qa 1Db;  type 3: x5 = X5d(b,a), x8 = X5f2, x7 = Qb 1Da
            const double x52 = a.X5f1[((size_t)k * r + j) * R2 + (size_t)i * r + l];
            const double x82 = a.X5d[((size_t)k * r + i) * R22 + R2 + (size_t)j * r + l];
            const double x53 = a.X5d[(R2 + (size_t)k * r + j) * R22 + (size_t)i * r + l];
            const double x83 = a.X5f2[((size_t)k * r + i) * R2 + (size_t)j * r + l];
            double n = fma(2.0, (x52 - x82) + U3[e], x12[e]);
            n = fma(-Qa[k * r + i], gb[j * r + l], n);
            double m = fma(2.0, (x53 - x83) - U2[e], -x13[e]);
            m = fma(Qb[k * r + j], ga[i * r + l], m);
            if (ny2) {
                n = fma(9.0, ny2[e], n);
                m = fma(9.0, ny3[e], m);
            }
            bp_sm[k * ld + l] = n;
            Nt[k * ld + l] = m;
        }
        __syncthreads();
        const double* Y = a.Y[1] + (size_t)ij * R2;
        double* H = a.H[1] + (size_t)ij * R2;
        for (int e = threadIdx.x; e < R2; e += blockDim.x) {
            const int k = e / r, l = e - k * r;
            H[e] = fma(-4.0 / 3.0, bp_sm[k * ld + l] - Nt[l * ld + k], 4.0 * Y[e]);
            if (i == j) a.H[0][(size_t)ij * R2 + e] = a.H[2][(size_t)ij * R2 + e] = 0.0;
        }
    }
}

// ------------------------------------------------------------- B -> H, split-precision path
// Persistent variant for FP32: each block walks pairs (i, j) with a stride of the grid and, per pair,
// three rounds (aa: type 0, bb: type 1, ab: types 2 and 3).  A round's X and M rows are copied into
// shared memory (cp.async) while the previous round is computed.  1D (as [p][l]) and w (as w^T[p][k])
// of both spins are loaded once per block.  Within a type, the warps of group 1 (threads [0, S),
// S = nt^2 rounded up to a warp) own 4 x 4 tiles of x1 and the warps of group 2 (threads
// [S, S + nt^2)) own tiles of x2, so no warp runs both products; each product uses the tile
// ownership that makes all of its shared loads 16-byte vectors without bank conflicts:
//   RR (A as [k][q], B as [q][l]): rows k = kb + nt a, columns l = 4 lb + b, four q per step
//   CR (A as [q][k], B as [q][l]): k = 4 kb + a, l = 4 lb + b, one q per step
//   CC (A as [q][k], B as [l][q]): k = 4 kb + a, l = lb + nt b, four q per step
// x2 threads also gather x5, x8 (loads issued before their product) and store
// (-2 sgn2 x2 + 2 x5 - 2 x8) / 9 into Bs; x1 threads form x7 - x4 before their product and, after a
// barrier, add (sgn1 x1 - x4 + x7) / 9.
// Each thread's share of the Y row of the round is loaded into registers at the start of the round
// and used when H is formed at its end.
#define BP_MAX_THREADS 512   // r = 64: S = 256, 256 + 256 threads

// RP > 0: the padded size is a compile-time constant (loops fully unrolled, addresses folded); the
// padding rows and columns of the shared tiles are zero, so the loops may run to RP.
template <int KIND, int RP>
__device__ __forceinline__ void bp_product(float (&acc)[4][4], const float* A, const float* B, int ld_, int r_, int rp_,
                                           int nt_, int kb, int lb) {
    const int rp = RP ? RP : rp_, ld = RP ? RP + 4 : ld_, nt = RP ? RP / 4 : nt_, r = RP ? RP : r_;
    // paired accumulators for the packed FP32x2 FMA (two independent round-to-nearest FMAs, the same
    // sequence per element as scalar FMAs): c[a][h] = (acc[a][2h], acc[a][2h+1]) for RR and CR,
    // c[a][h] = (acc[2h][a], acc[2h+1][a]) for CC
    float2 c[4][2];
#pragma unroll
    for (int a = 0; a < 4; ++a) c[a][0] = c[a][1] = make_float2(0.f, 0.f);
    if (KIND == 0) {   // RR
        for (int q = 0; q < rp; q += 4) {
            float av[4][4], bv[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a) ld4(A + (kb + nt * a) * ld + q, av[a]);
#pragma unroll
            for (int u = 0; u < 4; ++u) ld4(B + (q + u) * ld + 4 * lb, bv[u]);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 x = make_float2(av[a][u], av[a][u]);
                    c[a][0] = __ffma2_rn(x, make_float2(bv[u][0], bv[u][1]), c[a][0]);
                    c[a][1] = __ffma2_rn(x, make_float2(bv[u][2], bv[u][3]), c[a][1]);
                }
        }
    } else if (KIND == 1) {   // CR
#pragma unroll 4
        for (int q = 0; q < r; ++q) {
            float av[4], bv[4];
            ld4(A + q * ld + 4 * kb, av);
            ld4(B + q * ld + 4 * lb, bv);
            const float2 b0 = make_float2(bv[0], bv[1]), b1 = make_float2(bv[2], bv[3]);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float2 x = make_float2(av[a], av[a]);
                c[a][0] = __ffma2_rn(x, b0, c[a][0]);
                c[a][1] = __ffma2_rn(x, b1, c[a][1]);
            }
        }
    } else {   // CC
        for (int q = 0; q < rp; q += 4) {
            float av[4][4], bv[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) ld4(A + (q + u) * ld + 4 * kb, av[u]);
#pragma unroll
            for (int b = 0; b < 4; ++b) ld4(B + (lb + nt * b) * ld + q, bv[b]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 a0 = make_float2(av[u][0], av[u][1]), a1 = make_float2(av[u][2], av[u][3]);
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const float2 y = make_float2(bv[b][u], bv[b][u]);
                    c[b][0] = __ffma2_rn(a0, y, c[b][0]);
                    c[b][1] = __ffma2_rn(a1, y, c[b][1]);
                }
            }
        }
    }
    if (KIND == 2) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            acc[0][b] = c[b][0].x; acc[1][b] = c[b][0].y; acc[2][b] = c[b][1].x; acc[3][b] = c[b][1].y;
        }
    } else {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            acc[a][0] = c[a][0].x; acc[a][1] = c[a][0].y; acc[a][2] = c[a][1].x; acc[a][3] = c[a][1].y;
        }
    }
}

// Output coordinates of element (a, b) of a thread's tile for ownership KIND.
__device__ __forceinline__ int bp_k(int kind, int kb, int nt, int a) { return kind == 0 ? kb + nt * a : 4 * kb + a; }
__device__ __forceinline__ int bp_l(int kind, int lb, int nt, int b) { return kind == 2 ? lb + nt * b : 4 * lb + b; }

// PRE: the products x1 and x2 come precomputed (the tensor-core kernel of acse_btc.cu, r a multiple of
// 16): no operand staging, each thread reads its 4 x 4 tile of x1 and of x2^T with 16-byte loads; the
// shared memory holds only the B rows.
template <int MAXT, int MINB, int RP, bool PRE = false>
__global__ void __launch_bounds__(MAXT, MINB) k_B_pipe(const __grid_constant__ BTiledArgs a) {
    extern __shared__ __align__(16) unsigned char tl_smem[];
    const int r = a.r, rp = RP ? RP : pad4(r), ld = rp + 4, R2 = r * r, bpitch = r + 1;
    const int nt = rp / 4, nt2 = nt * nt, S = (nt2 + 31) & ~31;
    const size_t tile = PRE ? 0 : (size_t)rp * ld;
    float* gA = (float*)tl_smem;          // 1D_a [p][l]
    float* gB = gA + tile;                // 1D_b
    float* wAT = gB + tile;               // w_a^T [p][k]
    float* wBT = wAT + tile;              // w_b^T
    float* buf = wBT + tile;              // [2][X, M] operand tiles, element (u, v) of a row at u * ld + v
    float* Bs = buf + 4 * tile;           // [2][r][r + 1]
    const size_t R22 = 2 * (size_t)R2;
    if (!PRE) {
        for (int e = threadIdx.x; e < 8 * (int)tile; e += blockDim.x) gA[e] = 0.f;
        __syncthreads();
        for (int e = threadIdx.x; e < R2; e += blockDim.x) {
            const int u = e / r, v = e - u * r;
            gA[u * ld + v] = a.gam[e];
            gB[u * ld + v] = a.gam[R2 + e];
            wAT[v * ld + u] = a.w[e];          // w[k][p] -> w^T[p][k]
            wBT[v * ld + u] = a.w[R2 + e];
        }
    }
    const bool vec = (r & 3) == 0;
    const bool yvec = (r & 1) == 0;
    // row index of a flat index e < r^2 as (int)((e + 1/2) / r): the fraction stays at least 1/(2r)
    // away from an integer, far above the float rounding of the product for r <= 64
    const float invr = 1.f / (float)r;
    // Work items: [0, P) the aa pairs i < j, [P, 2P) the bb pairs i < j, [2P, 2P + r^2) every ab
    // pair (P = r(r-1)/2).  B and H of a same-spin sector are antisymmetric in (i, j), so the item
    // (i, j) also writes row (j, i) = -row (i, j); the rows (i, i) are zero.
    const int P = r * (r - 1) / 2, NB = a.flip ? 0 : P, NI = P + NB + R2;   // NB: bb items
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < 2 * (size_t)r * R2;
         e += (size_t)gridDim.x * blockDim.x) {
        const int sec = e < (size_t)r * R2 ? 0 : 2;
        const size_t f = e - (sec ? (size_t)r * R2 : 0);
        const int d = (int)(f / R2);
        a.H[sec][(size_t)(d * r + d) * R2 + (f - (size_t)d * R2)] = 0.f;
    }
    auto item = [&](int L, int& round, int& i, int& j) {
        if (L < P + NB) {
            round = L < P ? 0 : 1;
            const int q = L - round * P;
            int ii = 0;
            while (q >= ii * r - ii * (ii + 1) / 2 + (r - ii - 1)) ++ii;
            i = ii;
            j = q - (ii * r - ii * (ii + 1) / 2) + ii + 1;
        } else {
            round = 2;
            i = (L - P - NB) / r;
            j = (L - P - NB) - i * r;
        }
    };
    const int nsteps = (int)blockIdx.x < NI ? (NI - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    // operands of step s (item blockIdx.x + s gridDim.x): X and M rows of its sector
    // (round 0 -> aa (0), round 1 -> bb (2), round 2 -> ab (1))
    auto issue = [&](int step, int slot) {
        if (PRE) return;
        int round, ii, jj;
        item((int)blockIdx.x + step * (int)gridDim.x, round, ii, jj);
        const size_t ij = (size_t)ii * r + jj;
        const int sec = round == 0 ? 0 : round == 1 ? 2 : 1;
        const float* src[2] = {a.X[sec] + ij * R2, a.M[sec] + ij * R2};
        for (int h = 0; h < 2; ++h) {
            float* dst = buf + (size_t)(2 * slot + h) * tile;
            if (vec) {
                const int c4 = r / 4;
                const float inv_c4 = 4.f / (float)r;
                for (int e = threadIdx.x; e < r * c4; e += blockDim.x) {
                    const int u = (int)(((float)e + 0.5f) * inv_c4), v = (e - u * c4) * 4;
                    cp_async16(dst + u * ld + v, src[h] + u * r + v);
                }
            } else {
                for (int e = threadIdx.x; e < R2; e += blockDim.x) {
                    const int u = e / r, v = e - u * r;
                    const unsigned d = (unsigned)__cvta_generic_to_shared(dst + u * ld + v);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src[h] + e) : "memory");
                }
            }
        }
        cp_async_commit();
    };
    if (nsteps > 0) issue(0, 0);
    const int grp = threadIdx.x < S ? 0 : (threadIdx.x < S + nt2 ? 1 : 2);   // x1, x2, idle
    const int idx = grp == 0 ? threadIdx.x : threadIdx.x - S;
    const bool active = grp == 0 ? idx < nt2 : grp == 1;
    const int kb = idx / nt, lb = idx - (idx / nt) * nt;
    constexpr int YPT = 2;                         // float4 groups of the Y row held per thread
    for (int step = 0; step < nsteps; ++step) {
        int round, i, j;
        item((int)blockIdx.x + step * (int)gridDim.x, round, i, j);
        const int ij = i * r + j;
        const int cur = step & 1;
        const int b = round == 0 ? 0 : round == 1 ? 2 : 1;
        cp_async_wait_all();
        __syncthreads();                                    // operands landed; Bs and the other buffer free
        if (step + 1 < nsteps) issue(step + 1, cur ^ 1);
        // this thread's part of the Y row (used when H is formed at the end of the round)
        const float* Yrow = a.Y[b] + (size_t)ij * R2;
        float4 yv[YPT];
        if (yvec) {
#pragma unroll
            for (int u = 0; u < YPT; ++u) {
                const int g = threadIdx.x + u * blockDim.x;
                yv[u] = g < R2 / 4 ? reinterpret_cast<const float4*>(Yrow)[g] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        const float* Xs = buf + (size_t)(2 * cur) * tile;
        const float* Ms = Xs + tile;
        const int ntypes = round < 2 ? 1 : 2;
        for (int tt = 0; tt < ntypes; ++tt) {
            const int t = round < 2 ? round : 2 + tt;
            float* Bt = Bs + (size_t)tt * r * bpitch;
            float x1[4][4];
            // the particle-hole sources: x5 at row (k, j), column (i, l); x8 at row (k, i), column (j, l)
            const float* X5b;
            const float* X8b;
            size_t ld5, ld8;
            if (t == 0) { X5b = X8b = a.X5d; ld5 = ld8 = R22; }
            else if (t == 1) { X5b = X8b = a.X5d + R2 * R22 + R2; ld5 = ld8 = R22; }
            else if (t == 2) { X5b = a.X5f1; ld5 = R2; X8b = a.X5d + R2; ld8 = R22; }
            else if (!a.flip) { X5b = a.X5d + R2 * R22; ld5 = R22; X8b = a.X5f2; ld8 = R2; }
            else { X5b = a.X5d + R2; ld5 = R22; X8b = a.X5f1; ld8 = R2; }   // flips of X5d(b,a), X5f2
            float part1[4][4];   // x1 group: (s1 x1 + x7 - x4 - 2 x8) / 9, added after the barrier
            // this item's number among the type's items (rows of the precomputed products)
            const int it = round == 0 ? (int)blockIdx.x + step * (int)gridDim.x
                         : round == 1 ? (int)blockIdx.x + step * (int)gridDim.x - P : ij;
            if (grp == 1) {
                // x2 = sum_p w[k][p] M(l, p) (types 0, 1, 3: M row holds M[l][p]; type 2: M[p][l]) and the
                // gathered x5 (loaded before the product)
                // PRE: no product, so every type takes the 4 x 4 ownership k = 4 kb + u, l = 4 lb + v, under
                // which x2^T (four consecutive k) and x5 (four consecutive l) are 16-byte loads (r % 4 == 0)
                const int kind = (PRE || t == 2) ? 1 : 2;
                float g5[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = bp_k(kind, kb, nt, u);
                    const int kc = k < r ? k : r - 1;
                    const float* x5r = X5b + ((size_t)kc * r + j) * ld5 + (size_t)i * r;
                    if (PRE) {
                        const float4 q = *reinterpret_cast<const float4*>(x5r + 4 * lb);
                        g5[u][0] = q.x; g5[u][1] = q.y; g5[u][2] = q.z; g5[u][3] = q.w;
                    } else {
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int l = bp_l(kind, lb, nt, v);
                            g5[u][v] = x5r[l < r ? l : r - 1];
                        }
                    }
                }
                float acc[4][4];
                if (PRE) {   // x2[k][l] = x2^T row l, column k: four consecutive k per load
                    const float* x2t = a.bx[2 * t + 1] + (size_t)it * R2;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int l = bp_l(kind, lb, nt, v);
                        const float4 q = *reinterpret_cast<const float4*>(x2t + (size_t)l * r + 4 * kb);
                        acc[0][v] = q.x; acc[1][v] = q.y; acc[2][v] = q.z; acc[3][v] = q.w;
                    }
                } else {
                    const float* wT = (t == 0 || t == 2) ? wAT : wBT;
                    if (kind == 1) bp_product<1, RP>(acc, wT, Ms, ld, r, rp, nt, kb, lb);
                    else bp_product<2, RP>(acc, wT, Ms, ld, r, rp, nt, kb, lb);
                }
                const float c2 = t == 2 ? 2.f : -2.f;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = bp_k(kind, kb, nt, u);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int l = bp_l(kind, lb, nt, v);
                        if (k < r && l < r)
                            Bt[k * bpitch + l] = (c2 * acc[u][v] + 2.f * g5[u][v]) * (1.f / 9.f) +
                                                 (a.ny[t] ? a.ny[t][(size_t)ij * R2 + (size_t)k * r + l] : 0.f);
                    }
                }
            } else if (grp == 0 && active) {
                const int kind1 = t == 3 ? 1 : 0;
                // x7 - x4 - 2 x8, x7 - x4 = Q7[k][j] g7[i][l] - Q4[k][i] g4[j][l] (zero where a type has no
                // such term), loaded before the product
                const float* ga = a.gam;
                const float* gb = a.gam + R2;
                const float* Q4 = t == 0 ? a.Q : t == 1 ? a.Q + R2 : t == 2 ? a.Q : nullptr;
                const float* g4 = t == 0 ? ga : t == 1 ? gb : t == 2 ? gb : nullptr;
                const float* Q7 = t == 0 ? a.Q : t == 1 ? a.Q + R2 : t == 3 ? a.Q + R2 : nullptr;
                const float* g7 = t == 0 ? ga : t == 1 ? gb : t == 3 ? ga : nullptr;
                if (PRE) {   // r % 4 == 0: the 1D rows and the x8 row as 16-byte loads
                    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 g7v = g7 ? *reinterpret_cast<const float4*>(g7 + i * r + 4 * lb) : z4;
                    const float4 g4v = g4 ? *reinterpret_cast<const float4*>(g4 + j * r + 4 * lb) : z4;
                    const float g7a[4] = {g7v.x, g7v.y, g7v.z, g7v.w}, g4a[4] = {g4v.x, g4v.y, g4v.z, g4v.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int k = bp_k(kind1, kb, nt, u);
                        const float q4 = Q4 ? Q4[k * r + i] : 0.f;
                        const float q7 = Q7 ? Q7[k * r + j] : 0.f;
                        const float4 x8 = *reinterpret_cast<const float4*>(X8b + ((size_t)k * r + i) * ld8 + (size_t)j * r + 4 * lb);
                        const float x8a[4] = {x8.x, x8.y, x8.z, x8.w};
#pragma unroll
                        for (int v = 0; v < 4; ++v) part1[u][v] = (q7 * g7a[v] - q4 * g4a[v]) - 2.f * x8a[v];
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int k = bp_k(kind1, kb, nt, u);
                        const int kc = k < r ? k : r - 1;
                        const float q4 = Q4 ? Q4[kc * r + i] : 0.f;
                        const float q7 = Q7 ? Q7[kc * r + j] : 0.f;
                        const float* x8r = X8b + ((size_t)kc * r + i) * ld8 + (size_t)j * r;
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int l = 4 * lb + v;
                            const int lc = l < r ? l : r - 1;
                            const float x47 = (Q7 ? q7 * g7[i * r + lc] : 0.f) - (Q4 ? q4 * g4[j * r + lc] : 0.f);
                            part1[u][v] = x47 - 2.f * x8r[lc];
                        }
                    }
                }
                if (PRE) {   // x1 row k, four consecutive l per load
                    const float* x1r = a.bx[2 * t] + (size_t)it * R2;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int k = bp_k(kind1, kb, nt, u);
                        const float4 q = *reinterpret_cast<const float4*>(x1r + (size_t)k * r + 4 * lb);
                        x1[u][0] = q.x; x1[u][1] = q.y; x1[u][2] = q.z; x1[u][3] = q.w;
                    }
                } else {
                    const float* g1 = (t == 0 || t == 3) ? gA : gB;
                    if (t == 3) bp_product<1, RP>(x1, Xs, g1, ld, r, rp, nt, kb, lb);
                    else bp_product<0, RP>(x1, Xs, g1, ld, r, rp, nt, kb, lb);
                }
                const float s1 = t == 3 ? -1.f : 1.f;
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) part1[u][v] = (s1 * x1[u][v] + part1[u][v]) * (1.f / 9.f);
            }
            __syncthreads();                                // x2, x5 and ny in Bt
            if (grp == 0 && active) {
                const int kind1 = t == 3 ? 1 : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = bp_k(kind1, kb, nt, u);
                    if (k >= r) continue;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int l = 4 * lb + v;
                        if (l < r) Bt[k * bpitch + l] += part1[u][v];
                    }
                }
            }
        }
        __syncthreads();                                    // B types of this round complete
        const float* Pb = Bs;
        const float* Px = round < 2 ? Bs : Bs + (size_t)r * bpitch;
        float* Hrow = a.H[b] + (size_t)ij * R2;
        float* Hmir = round < 2 ? a.H[b] + (size_t)(j * r + i) * R2 : nullptr;   // row (j, i) = -row (i, j)
        if (yvec) {
#pragma unroll
            for (int u = 0; u < YPT; ++u) {
                const int g = threadIdx.x + u * blockDim.x;
                if (g < R2 / 4) {
                    const float yy[4] = {yv[u].x, yv[u].y, yv[u].z, yv[u].w};
                    float hh[4];
                    int k = (int)(((float)(4 * g) + 0.5f) * invr), l = 4 * g - k * r;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        hh[c] = 4.f * yy[c] - 12.f * (Pb[k * bpitch + l] - Px[l * bpitch + k]);
                        if (++l == r) { l = 0; ++k; }
                    }
                    reinterpret_cast<float4*>(Hrow)[g] = make_float4(hh[0], hh[1], hh[2], hh[3]);
                    if (Hmir) reinterpret_cast<float4*>(Hmir)[g] = make_float4(-hh[0], -hh[1], -hh[2], -hh[3]);
                }
            }
            for (int g = threadIdx.x + YPT * blockDim.x; g < R2 / 4; g += blockDim.x) {   // rows beyond the prefetch
                const float4 y4 = reinterpret_cast<const float4*>(Yrow)[g];
                const float yy[4] = {y4.x, y4.y, y4.z, y4.w};
                float hh[4];
                int k = (int)(((float)(4 * g) + 0.5f) * invr), l = 4 * g - k * r;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    hh[c] = 4.f * yy[c] - 12.f * (Pb[k * bpitch + l] - Px[l * bpitch + k]);
                    if (++l == r) { l = 0; ++k; }
                }
                reinterpret_cast<float4*>(Hrow)[g] = make_float4(hh[0], hh[1], hh[2], hh[3]);
                if (Hmir) reinterpret_cast<float4*>(Hmir)[g] = make_float4(-hh[0], -hh[1], -hh[2], -hh[3]);
            }
        } else {
            for (int e = threadIdx.x; e < R2; e += blockDim.x) {
                const int k = e / r, l = e - k * r;
                const float hv = 4.f * Yrow[e] - 12.f * (Pb[k * bpitch + l] - Px[l * bpitch + k]);
                Hrow[e] = hv;
                if (Hmir) Hmir[e] = -hv;
            }
        }
    }
    cp_async_wait_all();
}

static size_t bp_smem(int r) {
    const size_t rp = pad4(r), tile = rp * (rp + 4);
    return (8 * tile + 2 * (size_t)r * (r + 1)) * sizeof(float);
}

// ------------------------------------------------------------------------------- launch
// Launch shape of k_Z_pipe: ipb slices per round (ipb * (rp/4)^2 <= ZP_MAX_THREADS threads, at most 4) and
// the p-chunk per block, chosen to balance the waves over the SMs (a block's first slices are not
// overlapped, hence the +1 round per block).
struct ZPlan {
    int ipb, threads, pchunk, blocks;
    size_t smem;
};
static ZPlan z_plan_compute(int r, const void* kern) {
    ZPlan z;
    const int rp = pad4(r), nt = rp / 4, nt2 = nt * nt;
    z.ipb = ZP_MAX_THREADS / nt2;
    if (z.ipb > 4) z.ipb = 4;
    if (z.ipb < 1) z.ipb = 1;
    z.threads = (z.ipb * nt2 + 31) / 32 * 32;
    const int R2e = (r * r + 3) / 4 * 4;
    z.smem = ((size_t)z.ipb * R2e + (size_t)(1 + z.ipb) * rp * (rp + 4)) * sizeof(float);
    int per_sm = 1, nsm = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, z.threads, z.smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const long slots = (long)nsm * per_sm;
    double best = 1e30;
    z.pchunk = r;
    for (int pc = z.ipb; pc <= r; pc += z.ipb) {
        const long blocks = 6L * r * ((r + pc - 1) / pc);
        const double cost = (double)((blocks + slots - 1) / slots) * ((pc + z.ipb - 1) / z.ipb + 1);
        if (cost < best - 1e-9) { best = cost; z.pchunk = pc; }
    }
    z.blocks = 6 * r * ((r + z.pchunk - 1) / z.pchunk);
    return z;
}

// cached per host thread, output mode and r (the occupancy query is not free)
static ZPlan z_plan(int r, int mode, const void* kern) {
    static thread_local int cached_r[4] = {-1, -1, -1, -1};
    static thread_local ZPlan cached[4];
    if (cached_r[mode] != r) {
        cached[mode] = z_plan_compute(r, kern);
        cached_r[mode] = r;
    }
    return cached[mode];
}

// Z of the split path from the FP32 copy of W.
int launch_Z_tiled(acse_ctx* c, const float* const W32[3]) {
    const int r = c->r;
    ZOut o;
    Work& w = c->w;
    const int R2 = r * r;
    const bool sf = acse_singlet(c);
    // spin-flip specialisation: Zd(b,b), Zd(b,a), Zf2 are the flips of Zd(a,a), Zd(a,b), Zf1 and only
    // the alpha-led rows of the diagonal particle-hole GEMM are formed
    o.ntypes = sf ? 3 : 6;
    const int tm_sf[6] = {0, 1, 4, 0, 0, 0};
    for (int k = 0; k < 6; ++k) o.tmap[k] = sf ? tm_sf[k] : k;
    o.Zd = w.tc_Zd; o.Zf[0] = w.tc_Zf[0]; o.Zf[1] = w.tc_Zf[1];
    o.mode = c->opt.prec == ACSE_BF16X3 ? 1 : (c->opt.prec == ACSE_TF32X3 ? 3 : 2);
    o.ldd = c->nsplit * w.Kp2; o.ldf = c->nsplit * w.Kp1; o.Kp1 = w.Kp1; o.Kp2 = w.Kp2; o.diag = w.zdiag32;
    // BF16x3 with r a multiple of 16: the products on the tensor cores (acse_ztc.cu)
    const int zs = launch_Z_tc(c, W32, o.ntypes, o.tmap);
    if (zs == ACSE_OK) {
        k_w_from_diag<float><<<2 * r, 256, 0, c->stream>>>(r, w.zdiag32, w.w32, sf ? 1 : 0);
        ACSE_LAUNCHED(c);
        return ACSE_OK;
    }
    if (zs != ACSE_ERR_UNSUPPORTED) return zs;
    const bool r48 = o.mode == 1 && pad4(r) == 48;
    const void* kern = r48 ? (const void*)k_Z_pipe<1, 48>
                           : o.mode == 1 ? (const void*)k_Z_pipe<1> : o.mode == 3 ? (const void*)k_Z_pipe<3>
                                                                                  : (const void*)k_Z_pipe<2>;
    const ZPlan zp = z_plan(r, o.mode, kern);
    if (r48)
        k_Z_pipe<1, 48><<<zp.blocks / 6 * o.ntypes, zp.threads, zp.smem, c->stream>>>(r, zp.ipb, zp.pchunk, W32[0], W32[1], W32[2], w.gam, o);
    else if (o.mode == 1)
        k_Z_pipe<1><<<zp.blocks / 6 * o.ntypes, zp.threads, zp.smem, c->stream>>>(r, zp.ipb, zp.pchunk, W32[0], W32[1], W32[2], w.gam, o);
    else if (o.mode == 3)
        k_Z_pipe<3><<<zp.blocks / 6 * o.ntypes, zp.threads, zp.smem, c->stream>>>(r, zp.ipb, zp.pchunk, W32[0], W32[1], W32[2], w.gam, o);
    else
        k_Z_pipe<2><<<zp.blocks / 6 * o.ntypes, zp.threads, zp.smem, c->stream>>>(r, zp.ipb, zp.pchunk, W32[0], W32[1], W32[2], w.gam, o);
    ACSE_LAUNCHED(c);
    k_w_from_diag<float><<<2 * r, 256, 0, c->stream>>>(r, w.zdiag32, w.w32, sf ? 1 : 0);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// w of the FP64 and Ozaki paths from the terms of k_ph_w_diag.
int launch_w_sum(acse_ctx* c) {
    k_w_from_diag<double><<<2 * c->r, 256, 0, c->stream>>>(c->r, c->w.zdiag, c->w.w, 0);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

static size_t b_smem(int r) { return 2 * (size_t)r * (r | 1) * sizeof(double); }
static const size_t k_smem_cap = 227 * 1024;

int launch_B_tiled(acse_ctx* c) {
    const int r = c->r;
    const int R2 = r * r;
    Work& w = c->w;
    if (c->opt.prec == ACSE_FP64) {
        BPreArgs a;
        a.r = r;
        for (int s = 0; s < 3; ++s) { a.Y[s] = w.Y[s]; a.H[s] = w.H[s]; }
        a.X5d = w.X5d; a.X5f1 = w.X5f1; a.X5f2 = w.X5f2;
        for (int t = 0; t < 4; ++t) a.ny[t] = (const double*)ny_terms(c, t);
        a.gam = w.gam; a.Q = w.Q;
        a.pmap = w.pmap;
        ACSE_TRY(launch_Bx(c));
        for (int k = 0; k < 8; ++k) a.bx[k] = w.bx64[k];
        k_B_pre<<<r * (r - 1) + R2, 256, b_smem(r), c->stream>>>(a);
    } else {
        BTiledArgs a;
        a.r = r;
        for (int s = 0; s < 3; ++s) {
            a.X[s] = w.tc_pairC[s];
            a.Y[s] = w.tc_pairC[s] + (size_t)R2 * R2;   // rows r^2.. of [X; Y]
        }
        for (int s = 0; s < 3; ++s) {
            a.M[s] = w.M32[s];
            a.H[s] = w.H32[s];
        }
        a.flip = acse_singlet(c) ? 1 : 0;
        a.X5d = w.tc_X5d; a.X5f1 = w.tc_X5f[0]; a.X5f2 = w.tc_X5f[1];
        for (int t = 0; t < 4; ++t) a.ny[t] = (const float*)ny_terms(c, t);
        a.gam = w.gam32; a.w = w.w32; a.Q = w.Q32;
        for (int k = 0; k < 8; ++k) a.bx[k] = w.bx[k];
        // BF16x3, r a multiple of 16: the products on the tensor cores first, then the B kernel without them
        const int bs = launch_Bx_tc(c);
        if (bs == ACSE_OK) {
            static thread_local int pre_r = -1, pre_flip = -1, pre_grid = 0;
            const int nt = pad4(r) / 4, nt2 = nt * nt;
            const int threads = (((nt2 + 31) & ~31) + nt2 + 31) / 32 * 32;
            const size_t smem = 2 * (size_t)r * (r + 1) * sizeof(float);
            const bool r48 = r == 48;
            const void* kern = r48 ? (const void*)k_B_pipe<320, 2, 48, true> : threads <= 320
                                   ? (const void*)k_B_pipe<320, 2, 0, true> : (const void*)k_B_pipe<BP_MAX_THREADS, 1, 0, true>;
            if (pre_r != r || pre_flip != a.flip) {
                int per_sm = 1, nsm = 152, dev = 0;
                if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
                if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess ||
                    per_sm < 1) {
                    cudaGetLastError();
                    per_sm = 1;
                }
                const int items = (a.flip ? 1 : 2) * (r * (r - 1) / 2) + R2;
                pre_grid = nsm * per_sm < items ? nsm * per_sm : items;
                pre_r = r;
                pre_flip = a.flip;
            }
            if (r48) k_B_pipe<320, 2, 48, true><<<pre_grid, threads, smem, c->stream>>>(a);
            else if (threads <= 320) k_B_pipe<320, 2, 0, true><<<pre_grid, threads, smem, c->stream>>>(a);
            else k_B_pipe<BP_MAX_THREADS, 1, 0, true><<<pre_grid, threads, smem, c->stream>>>(a);
            ACSE_LAUNCHED(c);
            return ACSE_OK;
        }
        if (bs != ACSE_ERR_UNSUPPORTED) return bs;
        static thread_local int cached_r = -1, cached_flip = -1, cached_grid = 0;
        const int nt2 = (pad4(r) / 4) * (pad4(r) / 4);
        const int threads = (((nt2 + 31) & ~31) + nt2 + 31) / 32 * 32;
        const bool small = threads <= 320;
        const bool r48 = pad4(r) == 48;
        const void* kern = r48 ? (const void*)k_B_pipe<320, 2, 48>
                               : small ? (const void*)k_B_pipe<320, 2, 0> : (const void*)k_B_pipe<BP_MAX_THREADS, 1, 0>;
        if (cached_r != r || cached_flip != a.flip) {
            int per_sm = 1, nsm = 152, dev = 0;
            if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, bp_smem(r)) != cudaSuccess ||
                per_sm < 1) {
                cudaGetLastError();
                per_sm = 1;
            }
            const int items = (a.flip ? 1 : 2) * (r * (r - 1) / 2) + R2;   // same-spin pairs i < j, mixed pairs
            cached_grid = nsm * per_sm < items ? nsm * per_sm : items;
            cached_r = r;
            cached_flip = a.flip;
        }
        if (r48) k_B_pipe<320, 2, 48><<<cached_grid, threads, bp_smem(r), c->stream>>>(a);
        else if (small) k_B_pipe<320, 2, 0><<<cached_grid, threads, bp_smem(r), c->stream>>>(a);
        else k_B_pipe<BP_MAX_THREADS, 1, 0><<<cached_grid, threads, bp_smem(r), c->stream>>>(a);
    }
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

int tiled_set_attrs() {
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_B_pre, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b_smem(ACSE_MAX_R)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_B_pipe<320, 2, 48>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bp_smem(48)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_B_pipe<320, 2, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bp_smem(48)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_B_pipe<BP_MAX_THREADS, 1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bp_smem(ACSE_MAX_R)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_Z_pipe<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k_smem_cap));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_Z_pipe<1, 48>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k_smem_cap));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_Z_pipe<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k_smem_cap));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_Z_pipe<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k_smem_cap));
    return ACSE_OK;
}
