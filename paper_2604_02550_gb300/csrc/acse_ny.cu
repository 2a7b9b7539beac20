// Nakatsuji-Yasuda (NY) 3-cumulant contribution to a contraction pass (Eq. NY and its appendix).
//
// With the NY reconstruction the three-body sum of every pass gains
//     T^{ij}_{kl} = sum_{pqr} W^{kp}_{rq} 3Delta^{ijp}_{rql},
//     3Delta^{ijp}_{rql} = 1/6 sum_a sigma_a A(2Delta^{ia}_{rq} 2Delta^{jp}_{al})  (36 signed terms),
// sigma_a = +1 for HF-occupied spin orbitals (aufbau by orbital index), -1 otherwise.  Using the
// pair antisymmetry of W and 2Delta the 36 terms collapse (nine-term form of the appendix, then
// terms 7-9 equal 4-6) to
//     T = 4/6 [ S1^{ij}_{kl} - S1^{ji}_{kl} - S3 - 2 S4^{ij}_{kl} + 2 S4^{ji}_{kl} + 2 S6 ],
//     X^{ia}_{kp} = sum_{rq} 2Delta^{ia}_{rq} W^{kp}_{rq}          (GEMM, rows (i,a), K (r,q))
//     Y4^{kq}_{ja} = sum_{pr} W^{kp}_{rq} 2Delta^{jp}_{ar}         (GEMM, rows (k,q), K (p,r))
//     Y6^{kr}_{al} = sum_{pq} W^{kp}_{rq} 2Delta^{pa}_{lq}         (GEMM, rows (k,r), K (p,q))
//     S1[k][i][j][l] = sum_{ap} X^{ia}_{kp} sigma_a 2Delta^{jp}_{al} (GEMM, rows (k,i), K (a,p))
//     S4[k][j][i][l] = sum_{aq} Y4^{kq}_{ja} sigma_a 2Delta^{ia}_{lq} (GEMM, rows (k,j), K (a,q))
//     S6[j][i][k][l] = sum_{ar} 2Delta^{ji}_{ar} sigma_a Y6^{kr}_{al} (GEMM, rows (j,i), K (a,r))
//     S3^{ij}_{kl} = sum_a Q[a][k] sigma_a 2Delta^{ji}_{al},  Q[a][k] = sum_p X^{pa}_{kp}.
// Layout: spin-orbital index pairs are numbered spin-major, pair (x, y) -> (2 s_x + s_y) r^2 + x' r + y'
// (x = s_x r + x'), so every spin block of an n^2 x n^2 matrix (n = 2r) is a contiguous r^2 x r^2
// block.  Pack kernels write each GEMM operand in its row layout (index permutation, sigma scaling
// and, in the split precisions, the hi/lo split, K arranged per spin block); spin conservation of
// the operands leaves about 10 of the 64 (row, column, K) spin-block triples of a GEMM nonzero, and
// the K blocks of each nonzero output block are ordered to be contiguous, so each output block is
// one r^2 x r^2 problem of one grouped launch (FP64 DFMA or tcgen05).  A final kernel forms T for
// the four spin types of the B kernel, which adds it to B.
#include <math.h>
#include <type_traits>

#include "acse_internal.h"
#include "acse_split.cuh"
#include "dfloat.cuh"

struct NyWork {
    int n;                 // spin orbitals
    size_t n2, n4;
    int Kb;                // padded r^2: K elements of one spin block per split term
    void* delta[3];        // 2Delta blocks aa, ab, bb (double; float on the split path)
    double* sig;           // [n] sigma_a
    void* opA[3];          // operand rows of the three GEMMs of a stage
    void* opB[3];
    void* out[6];          // X, Y4, Y6, S1, S4, S6 (n^4 each; double or float)
    void* Q;               // [n][n]
    void* tny[4];          // T for the B spin types (r^4 each; double or float)
    TcTable st[2];         // split precisions: the two GEMM stages
    int Kbw;               // elements of one K spin block of an operand row (ns * padded r^2)
    int korder[6][4];      // per GEMM: spin pair (2 s + s') of K block position q
    int nprob[6];
    int prob[6][16][4];    // per GEMM: (row block, column block, first K block, K blocks)
};

// Element T^{x1 x2}_{x3 x4} (spin-orbital indices, alpha first) of a pair-antisymmetric tensor stored
// as its aa, ab, bb blocks (the other nonzero blocks follow by antisymmetry within each pair).
template <typename T>
__device__ __forceinline__ T so_get(const T* aa, const T* ab, const T* bb, int r, int x1, int x2, int x3, int x4) {
    const int s1 = x1 >= r, s2 = x2 >= r, s3 = x3 >= r, s4 = x4 >= r;
    const int a = x1 - s1 * r, b = x2 - s2 * r, c = x3 - s3 * r, d = x4 - s4 * r;
    const size_t R = r;
    auto at = [&](const T* t, int i, int j, int k, int l) { return t[((i * R + j) * R + k) * R + l]; };
    if (s1 + s2 != s3 + s4) return (T)0;
    if (s1 == s2) return s1 ? at(bb, a, b, c, d) : at(aa, a, b, c, d);
    if (s1 == 0 && s3 == 0) return at(ab, a, b, c, d);     // (a b | a b)
    if (s1 == 1 && s3 == 1) return at(ab, b, a, d, c);     // (b a | b a)
    if (s1 == 0) return -at(ab, a, b, d, c);               // (a b | b a)
    return -at(ab, b, a, c, d);                            // (b a | a b)
}

// 2Delta = 2D - 1D^1D per block: aa/bb: D - 1/2 (g_ik g_jl - g_jk g_il), ab: D - 1/2 ga_ik gb_jl.
template <typename T>   // formed in FP64, rounded once to T
__global__ void k_ny_delta(int r, const double* __restrict__ gam, const double* __restrict__ Daa,
                           const double* __restrict__ Dab, const double* __restrict__ Dbb, T* daa, T* dab, T* dbb) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    const double* ga = gam;
    const double* gb = gam + R2;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
        const int l = (int)(e % r), k = (int)((e / r) % r), j = (int)((e / R2) % r), i = (int)(e / (R2 * r));
        daa[e] = (T)(Daa[e] - 0.5 * (ga[i * r + k] * ga[j * r + l] - ga[j * r + k] * ga[i * r + l]));
        dbb[e] = (T)(Dbb[e] - 0.5 * (gb[i * r + k] * gb[j * r + l] - gb[j * r + k] * gb[i * r + l]));
        dab[e] = (T)(Dab[e] - 0.5 * ga[i * r + k] * gb[j * r + l]);
    }
}

// sigma_a: +1 for the first n_alpha alpha and the first n_beta beta orbitals, -1 otherwise.
__global__ void k_ny_sigma(int r, int na, int nb, double* sig) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= 2 * r) return;
    sig[x] = (x < r ? x < na : x - r < nb) ? 1.0 : -1.0;
}

// Spin-major number of the spin-orbital pair (x, y).
__device__ __forceinline__ size_t ny_pidx(int r, int x, int y) {
    const int sx = x >= r, sy = y >= r;
    return (size_t)(2 * sx + sy) * r * r + (size_t)(x - sx * r) * r + (y - sy * r);
}

// Element (x1 x2 | x3 x4) of a dense intermediate stored as [pair(x1,x2)][pair(x3,x4)].
template <typename T>
__device__ __forceinline__ T ny_dense(const T* t, int r, int x1, int x2, int x3, int x4) {
    return t[ny_pidx(r, x1, x2) * (size_t)(4 * r * r) + ny_pidx(r, x3, x4)];
}

// Packing of the six operands of a stage, one launch.  A piece is one spin block of one operand: rows (u0, u1) of row
// block rb, K positions t = u2 r + u3 of K block position q, value sign sigma[u2] src[base + sum_m u_m st_m].  The
// source is contiguous in u3, u2 or u1 (mode 0, 1, 2); a block takes nslab r x r slabs of u3 against u2 (modes 0, 1; fixed
// u0, u1: r^2 consecutive K positions of one row) or u1 (mode 2; fixed u0, u2) through shared memory, so that reads and
// writes are both coalesced and about 16 loads a thread are in flight.  (A thread per output element read the permuted
// source at stride r or r^2 in FP64 with four integer divisions an element: 34 us a launch at r = 32, 24 launches a
// step; one slab a block 146 us a stage, 97 now for 36 pieces: 230 MB written and 150 read.)
// Values are those of the FP64 source rounded once (2Delta and W are read as their FP32 copies on the split path).
struct NyPiece {
    const void* src;
    size_t base;
    int st[4];
    void* dst;
    int rb, q, mode, sp2;   // sp2: spin of u2
    int pat, use_sigma;
    float sign;
};
#define NY_MAXPC 96   // six operands of at most 16 spin blocks
struct NyPackList {
    NyPiece p[NY_MAXPC];
    const double* sig;
    size_t ld;              // row length of dst in elements
    int Kb, Kbw;            // K elements of a spin block per split term, and in all
};

template <int PREC>
__global__ void __launch_bounds__(256) k_ny_pack(int r, int nslab, const __grid_constant__ NyPackList a) {
    using T = typename std::conditional<PREC == ACSE_FP64, double, float>::type;
    extern __shared__ __align__(16) unsigned char ny_smem[];
    T* tile = (T*)ny_smem;   // [nslab][r][r + 1]
    const int R2 = r * r, ld = r + 1, nblk = (R2 + nslab - 1) / nslab;
    const float invr = 1.f / (float)r, invR2 = 1.f / (float)R2;   // e / r as (int)((e + 1/2) / r), exact for e < 2^16
    const int ip = blockIdx.x / nblk;
    const NyPiece& pc = a.p[ip];
    const int fb = (blockIdx.x - ip * nblk) * nslab, nf = min(nslab, R2 - fb);   // slabs (u0, u1), or (u0, u2) in mode 2
    const int mode = pc.mode;
    const bool m2 = mode == 2;
    const int sf0 = pc.st[0], sf1 = pc.st[m2 ? 2 : 1], slow = mode == 0 ? pc.st[2] : pc.st[3];
    const T* src = (const T*)pc.src + pc.base;
    // sigma in T once a block: a conversion from FP64 runs at 1/64 of the FP32 rate
    __shared__ T sig[ACSE_MAX_R];
    if (threadIdx.x < r) sig[threadIdx.x] = (T)a.sig[pc.sp2 * r + threadIdx.x];
#pragma unroll 4
    for (int e = threadIdx.x; e < nf * R2; e += 256) {
        const int w = (int)(((float)e + 0.5f) * invR2), g = e - w * R2;
        const int s = (int)(((float)g + 0.5f) * invr), c = g - s * r;
        const int f = fb + w, f0 = (int)(((float)f + 0.5f) * invr), f1 = f - f0 * r;
        const T v = src[(size_t)f0 * sf0 + (size_t)f1 * sf1 + (size_t)s * slow + c];
        tile[w * r * ld + (mode == 0 ? s * ld + c : c * ld + s)] = v;   // [u2 or u1][u3]
    }
    __syncthreads();
    const T sign = (T)pc.sign;
    const int use_sigma = pc.use_sigma, pat = pc.pat;
    const size_t rows0 = (size_t)pc.rb * R2;
    if constexpr (PREC == ACSE_FP64) {
        for (int e = threadIdx.x; e < nf * R2; e += 256) {
            const int w = e / R2, g = e - w * R2, d = g / r, u3 = g - d * r;
            const int f0 = (fb + w) / r, f1 = fb + w - f0 * r;
            T v = sign * tile[w * r * ld + d * ld + u3];
            if (use_sigma) v = sig[m2 ? f1 : d] * v;
            const size_t row = rows0 + (size_t)f0 * r + (m2 ? d : f1);
            ((double*)pc.dst)[row * a.ld + (size_t)pc.q * R2 + (m2 ? f1 * r + u3 : g)] = v;
        }
    } else {
        // groups of four K positions where they start on a multiple of four (a K block does)
        const size_t off = (size_t)pc.q * a.Kbw;
        void* base = PREC == ACSE_BF16X3 ? (void*)((__nv_bfloat16*)pc.dst + off) : (void*)((float*)pc.dst + off);
        const int n4 = !m2 || (r & 3) == 0 ? R2 / 4 : 0;
        const float invn4 = n4 ? 1.f / (float)n4 : 0.f;
        for (int h = threadIdx.x; h < nf * n4; h += 256) {
            const int w = (int)(((float)h + 0.5f) * invn4), g = h - w * n4;
            const int f = fb + w, f0 = (int)(((float)f + 0.5f) * invr), f1 = f - f0 * r;
            const int d = (int)(((float)(4 * g) + 0.5f) * invr);
            const T* tw = tile + w * r * ld;
            int u2 = d, u3 = 4 * g - d * r;
            const int k = m2 ? f1 * r + u3 : 4 * g;
            float x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                x[c] = sign * tw[u2 * ld + u3];
                if (use_sigma) x[c] = sig[m2 ? f1 : u2] * x[c];
                if (++u3 == r) { u3 = 0; ++u2; }   // mode 2: r % 4 == 0, the group stays in its row
            }
            const size_t row = rows0 + (size_t)f0 * r + (m2 ? d : f1);
            if (pat) put4<PREC, 1>(base, row, a.ld, a.Kb, k, x);
            else put4<PREC, 0>(base, row, a.ld, a.Kb, k, x);
        }
        const int nrest = R2 - 4 * n4;
        for (int h = threadIdx.x; h < nf * nrest; h += 256) {
            const int w = h / nrest, g = 4 * n4 + h - w * nrest, d = g / r, u3 = g - d * r;
            const int f0 = (fb + w) / r, f1 = fb + w - f0 * r;
            float v = sign * tile[w * r * ld + d * ld + u3];
            if (use_sigma) v = sig[m2 ? f1 : d] * v;
            const size_t row = rows0 + (size_t)f0 * r + (m2 ? d : f1);
            const int k = m2 ? f1 * r + u3 : g;
            if (pat) put<PREC, 1>(base, row, a.ld, a.Kb, k, v);
            else put<PREC, 0>(base, row, a.ld, a.Kb, k, v);
        }
    }
}

// Q[a][k] = sum_p X^{pa}_{kp}: one warp per (a, k).
template <typename T>
__global__ void __launch_bounds__(256) k_ny_Q(int r, const T* __restrict__ X, T* __restrict__ Q) {
    const int n = 2 * r;
    const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= n * n) return;
    const int a = t / n, k = t - (t / n) * n;
    T s = 0;
    for (int p = lane; p < n; p += 32) s += ny_dense(X, r, p, a, k, p);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) Q[t] = s;
}

// T for the spin type tt of block (i', j') (types of the B kernel: 0 aaaa, 1 bbbb, 2 (ia jb | ka lb),
// 3 (ia jb | kb la)).  S3 from factors staged in shared memory, qs[a][k'] = sigma_a Q[a][k], dv[a][l'] =
// 2Delta^{ji}_{al} (rows padded to rp = r rounded up to 4): a thread owns 2 x 4 outputs (k', l'), two vector loads for eight
// FMAs of the a loop (one output a thread took two loads a FMA: 109 us a launch at r = 32, 73 now).
template <typename T>
__global__ void __launch_bounds__(256) k_ny_assemble(int r, const T* __restrict__ S1, const T* __restrict__ S4,
                                                     const T* __restrict__ S6, const T* __restrict__ Q,
                                                     const T* __restrict__ daa, const T* __restrict__ dab,
                                                     const T* __restrict__ dbb, const double* __restrict__ sig,
                                                     T* t0, T* t1, T* t2, T* t3) {
    extern __shared__ __align__(16) unsigned char ny_smem[];
    const int n = 2 * r, R2 = r * r, rp = (r + 3) & ~3;
    T* qs = (T*)ny_smem;            // [n][rp]
    T* dv = qs + (size_t)n * rp;    // [n][rp]
    const int tt = blockIdx.x / R2, ij = blockIdx.x % R2;
    const int ip = ij / r, jp = ij % r;
    const int si = tt == 1, sj = tt == 0 ? 0 : 1, sk = tt == 1 || tt == 3, sl = tt == 1 || tt == 2;
    const int i = si * r + ip, j = sj * r + jp;
    __shared__ T sg[2 * ACSE_MAX_R];   // +-1: exact in T
    if (threadIdx.x < n) sg[threadIdx.x] = (T)sig[threadIdx.x];
    __syncthreads();
    for (int e = threadIdx.x; e < n * rp; e += blockDim.x) {
        const int aa_ = e / rp, c = e - aa_ * rp;
        qs[e] = c < r ? sg[aa_] * Q[(size_t)aa_ * n + sk * r + c] : (T)0;
        dv[e] = c < r ? so_get<T>(daa, dab, dbb, r, j, i, aa_, sl * r + c) : (T)0;
    }
    __syncthreads();
    T* out = (tt == 0 ? t0 : tt == 1 ? t1 : tt == 2 ? t2 : t3) + (size_t)ij * R2;
    const int nl = rp / 4, nk = rp / 2;
    for (int g = threadIdx.x; g < nk * nl; g += blockDim.x) {
        const int k0 = 2 * (g / nl), l0 = 4 * (g % nl);
        T s3[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) s3[u][v] = (T)0;
#pragma unroll 4
        for (int a_ = 0; a_ < n; ++a_) {
            T q[2], d[4];
            q[0] = qs[a_ * rp + k0];
            q[1] = qs[a_ * rp + k0 + 1];
            ld4(dv + a_ * rp + l0, d);
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) s3[u][v] += q[u] * d[v];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int kp = k0 + u;
            if (kp >= r) continue;
            const int k = sk * r + kp, l = sl * r + l0;
            const T *p1a = &S1[ny_pidx(r, k, i) * (size_t)(4 * R2) + ny_pidx(r, j, l)],
                    *p1b = &S1[ny_pidx(r, k, j) * (size_t)(4 * R2) + ny_pidx(r, i, l)];
            const T *p4a = &S4[ny_pidx(r, k, j) * (size_t)(4 * R2) + ny_pidx(r, i, l)],
                    *p4b = &S4[ny_pidx(r, k, i) * (size_t)(4 * R2) + ny_pidx(r, j, l)];
            const T* p6 = &S6[ny_pidx(r, j, i) * (size_t)(4 * R2) + ny_pidx(r, k, l)];
            T s1a[4], s1b[4], s4a[4], s4b[4], s6[4];
            if ((r & 3) == 0) {   // rows of l start on 16-byte boundaries
                ld4(p1a, s1a); ld4(p1b, s1b); ld4(p4a, s4a); ld4(p4b, s4b); ld4(p6, s6);
            } else {
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int o = l0 + v < r ? v : 0;
                    s1a[v] = p1a[o]; s1b[v] = p1b[o]; s4a[v] = p4a[o]; s4b[v] = p4b[o]; s6[v] = p6[o];
                }
            }
#pragma unroll
            for (int v = 0; v < 4; ++v)
                if (l0 + v < r)
                    out[kp * r + l0 + v] = (T)(4.0 / 6.0) * (s1a[v] - s1b[v] - s3[u][v] - (T)2 * s4a[v] + (T)2 * s4b[v] + (T)2 * s6[v]);
        }
    }
}

// ------------------------------------------------------------------------------ host side
static int ny_malloc(void** p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return ACSE_ERR_NOMEM;
    }
    return ACSE_OK;
}

void ny_free(acse_ctx* c) {
    NyWork* y = (NyWork*)c->ny;
    if (!y) return;
    void* ptrs[] = {y->delta[0], y->delta[1], y->delta[2], y->sig, y->opA[0], y->opA[1], y->opA[2], y->opB[0],
                    y->opB[1], y->opB[2], y->out[0], y->out[1], y->out[2], y->out[3], y->out[4], y->out[5], y->Q,
                    y->tny[0], y->tny[1], y->tny[2], y->tny[3]};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    for (int s = 0; s < 2; ++s)
        if (y->st[s].host) tc_table_free(&y->st[s]);
    free(y);
    c->ny = nullptr;
}

// Operands of the six GEMMs (stage 1: X, Y4, Y6; stage 2: S1, S4, S6).  src: 0 = 2Delta blocks,
// 1 = W blocks, 2 + o = dense intermediate o; cons: 0 when the source conserves s1 + s2 = s3 + s4
// (2Delta, W, X), 1 when it conserves s1 + s4 = s2 + s3 (Y4, Y6).
struct NyOp {
    int src, P[4], sigma, cons;
};
static const NyOp k_ny_ops[6][2] = {
    {{0, {0, 1, 2, 3}, 0, 0}, {1, {0, 1, 2, 3}, 0, 0}},   // X  = 2Delta(i,a|r,q) . W(k,p|r,q)
    {{1, {0, 2, 3, 1}, 0, 0}, {0, {0, 2, 1, 3}, 0, 0}},   // Y4 = W(k,q|p,r) . 2Delta(j,a|p,r)
    {{1, {0, 2, 1, 3}, 0, 0}, {0, {2, 0, 1, 3}, 0, 0}},   // Y6 = W(k,r|p,q) . 2Delta(a,l|p,q)
    {{2, {1, 2, 0, 3}, 1, 0}, {0, {0, 3, 2, 1}, 0, 0}},   // S1 = sigma X(k,i|a,p) . 2Delta(j,l|a,p)
    {{3, {0, 3, 1, 2}, 1, 1}, {0, {0, 2, 1, 3}, 0, 0}},   // S4 = sigma Y4(k,j|a,q) . 2Delta(i,l|a,q)
    {{0, {0, 1, 2, 3}, 1, 0}, {4, {0, 3, 2, 1}, 0, 1}},   // S6 = sigma 2Delta(j,i|a,r) . Y6(k,l|a,r)
};

static bool ny_allowed(const NyOp& op, int rb, int kb) {
    const int su[4] = {rb >> 1, rb & 1, kb >> 1, kb & 1};
    const int v0 = su[op.P[0]], v1 = su[op.P[1]], v2 = su[op.P[2]], v3 = su[op.P[3]];
    return op.cons == 0 ? v0 + v1 == v2 + v3 : v0 + v3 == v1 + v2;
}

// Spin-block problems of GEMM g: for each output block (rb, cb) the K blocks allowed by both
// operands, with a K order that makes every such set contiguous.
static int ny_plan_gemm(NyWork* y, int g) {
    int mask[4][4];
    for (int rb = 0; rb < 4; ++rb)
        for (int cb = 0; cb < 4; ++cb) {
            mask[rb][cb] = 0;
            for (int kb = 0; kb < 4; ++kb)
                if (ny_allowed(k_ny_ops[g][0], rb, kb) && ny_allowed(k_ny_ops[g][1], cb, kb)) mask[rb][cb] |= 1 << kb;
        }
    int order[4] = {0, 1, 2, 3};
    for (int trial = 0; trial < 24; ++trial) {
        // trial-th permutation (Lehmer code)
        int pool[4] = {0, 1, 2, 3}, np_ = 4, code = trial;
        for (int q = 0; q < 4; ++q) {
            const int f = q == 0 ? 6 : q == 1 ? 2 : 1;
            const int pick = q < 3 ? code / f : 0;
            if (q < 3) code %= f;
            order[q] = pool[pick];
            for (int m = pick; m < np_ - 1; ++m) pool[m] = pool[m + 1];
            --np_;
        }
        int pos[4];
        for (int q = 0; q < 4; ++q) pos[order[q]] = q;
        bool ok = true;
        int np = 0;
        for (int rb = 0; rb < 4 && ok; ++rb)
            for (int cb = 0; cb < 4 && ok; ++cb) {
                const int m = mask[rb][cb];
                if (!m) continue;
                int lo = 4, hi = -1, cnt = 0;
                for (int kb = 0; kb < 4; ++kb)
                    if (m >> kb & 1) {
                        lo = pos[kb] < lo ? pos[kb] : lo;
                        hi = pos[kb] > hi ? pos[kb] : hi;
                        ++cnt;
                    }
                if (hi - lo + 1 != cnt) ok = false;
                else {
                    y->prob[g][np][0] = rb;
                    y->prob[g][np][1] = cb;
                    y->prob[g][np][2] = lo;
                    y->prob[g][np][3] = cnt;
                    ++np;
                }
            }
        if (ok) {
            for (int q = 0; q < 4; ++q) y->korder[g][q] = order[q];
            y->nprob[g] = np;
            return ACSE_OK;
        }
    }
    return ACSE_ERR_UNSUPPORTED;
}

int ny_alloc(acse_ctx* c) {
    NyWork* y = (NyWork*)calloc(1, sizeof(NyWork));
    if (!y) return ACSE_ERR_NOMEM;
    c->ny = y;
    const int r = c->r, n = 2 * r, R2 = r * r;
    y->n = n;
    y->n2 = (size_t)n * n;
    y->n4 = y->n2 * y->n2;
    const size_t r4 = (size_t)R2 * R2;
    const bool f64 = c->opt.prec == ACSE_FP64;
    const size_t es = f64 ? 8 : 4;                                  // GEMM output / T element
    for (int g = 0; g < 6; ++g) ACSE_TRY(ny_plan_gemm(y, g));
    for (int b = 0; b < 3; ++b) ACSE_TRY(ny_malloc(&y->delta[b], r4 * es));
    ACSE_TRY(ny_malloc((void**)&y->sig, n * sizeof(double)));
    size_t op_bytes;
    if (f64) {
        y->Kb = R2;
        y->Kbw = R2;
        op_bytes = y->n4 * sizeof(double);
    } else {
        const int ops = c->opt.prec == ACSE_BF16X3 ? 2 : 4;         // operand element bytes
        const int kb = 128 / ops;
        y->Kb = (R2 + kb - 1) / kb * kb;
        y->Kbw = c->nsplit * y->Kb;
        op_bytes = y->n2 * (size_t)4 * y->Kbw * ops;
    }
    for (int s = 0; s < 3; ++s) {
        ACSE_TRY(ny_malloc(&y->opA[s], op_bytes));
        ACSE_TRY(ny_malloc(&y->opB[s], op_bytes));
        if (!f64) {   // K padding is never written afterwards
            ACSE_CUDA_TRY(cudaMemset(y->opA[s], 0, op_bytes));
            ACSE_CUDA_TRY(cudaMemset(y->opB[s], 0, op_bytes));
        }
    }
    for (int o = 0; o < 6; ++o) {   // blocks that no problem writes stay zero
        ACSE_TRY(ny_malloc(&y->out[o], y->n4 * es));
        ACSE_CUDA_TRY(cudaMemset(y->out[o], 0, y->n4 * es));
    }
    ACSE_TRY(ny_malloc(&y->Q, y->n2 * es));
    for (int t = 0; t < 4; ++t) ACSE_TRY(ny_malloc(&y->tny[t], r4 * es));
    k_ny_sigma<<<(n + 127) / 128, 128, 0, c->stream>>>(r, c->opt.n_alpha, c->opt.n_beta, y->sig);
    ACSE_LAUNCHED(c);
    if (!f64) {
        const int kind = (c->opt.prec == ACSE_TF32 || c->opt.prec == ACSE_TF32X3) ? 1 : 0;
        const int ops = kind == 0 ? 2 : 4;
        const size_t ld = (size_t)4 * y->Kbw;
        for (int s = 0; s < 2; ++s) {
            ACSE_TRY(tc_table_init_mode(&y->st[s], kind, tc_default_bn(r), tc_use_pairs(c)));
            for (int g = 3 * s; g < 3 * s + 3; ++g)
                for (int k = 0; k < y->nprob[g]; ++k) {
                    const int rb = y->prob[g][k][0], cb = y->prob[g][k][1], q0 = y->prob[g][k][2], cnt = y->prob[g][k][3];
                    const char* A = (const char*)y->opA[g % 3] + ((size_t)rb * R2 * ld + (size_t)q0 * y->Kbw) * ops;
                    const char* B = (const char*)y->opB[g % 3] + ((size_t)cb * R2 * ld + (size_t)q0 * y->Kbw) * ops;
                    float* C = (float*)y->out[g] + (size_t)rb * R2 * y->n2 + (size_t)cb * R2;
                    ACSE_TRY(tc_table_add_ld(&y->st[s], A, ld, B, ld, C, R2, R2, cnt * y->Kbw, (int)y->n2, 1.0f));
                }
            tc_table_set_err(&y->st[s], c->w.tc_err);
            ACSE_TRY(tc_table_upload(&y->st[s]));
        }
    }
    return ACSE_OK;
}

// The pieces of operand `side` of GEMM g (the spin blocks that some problem reads), appended to list k.  S[0], S[1]:
// the 2Delta and W blocks (aa, ab, bb) in the element type of the path.
static int ny_pieces(NyWork* y, int r, int g, int side, const void* const S[2][3], void* dst, NyPackList* k, int n) {
    const NyOp& op = k_ny_ops[g][side];
    const int R2 = r * r;
    int need[4] = {0, 0, 0, 0};
    for (int p = 0; p < y->nprob[g]; ++p)
        for (int q = y->prob[g][p][2]; q < y->prob[g][p][2] + y->prob[g][p][3]; ++q)
            need[y->prob[g][p][side]] |= 1 << y->korder[g][q];
    for (int rb = 0; rb < 4; ++rb)
        for (int q = 0; q < 4; ++q) {
            const int kb = y->korder[g][q];
            if (!(need[rb] >> kb & 1)) continue;
            NyPiece& pc = k->p[n++];
            const int su[4] = {rb >> 1, rb & 1, kb >> 1, kb & 1};
            int sx[4], xst[4];   // spins and strides of the source's four indices
            for (int m = 0; m < 4; ++m) sx[m] = su[op.P[m]];
            pc.sign = 1.0f;
            pc.base = 0;
            if (op.src < 2) {   // pair-antisymmetric tensor by its aa, ab, bb blocks (as so_get)
                int pos[4] = {0, 1, 2, 3};
                int blk = sx[0] == sx[1] ? 2 * sx[0] : 1;
                if (blk == 1) {
                    if (sx[0] == 1) { pos[0] = 1; pos[1] = 0; }
                    // lower indices: alpha first
                    if (sx[2] == 1) { pos[2] = 3; pos[3] = 2; }
                    if (sx[0] != sx[2]) pc.sign = -1.0f;
                }
                const int stride[4] = {R2 * r, R2, r, 1};
                for (int m = 0; m < 4; ++m) xst[m] = stride[pos[m]];
                pc.src = S[op.src][blk];
            } else {
                const int n2 = (int)y->n2;
                const int stride[4] = {r * n2, n2, r, 1};
                for (int m = 0; m < 4; ++m) xst[m] = stride[m];
                pc.src = y->out[op.src - 2];
                pc.base = (size_t)(2 * sx[0] + sx[1]) * R2 * n2 + (size_t)(2 * sx[2] + sx[3]) * R2;
            }
            for (int m = 0; m < 4; ++m) pc.st[op.P[m]] = xst[m];
            if (pc.st[3] == 1) pc.mode = 0;
            else if (pc.st[2] == 1) pc.mode = 1;
            else if (pc.st[1] == 1) pc.mode = 2;
            else return -1;   // contiguous in u0: no operand is
            pc.dst = dst;
            pc.rb = rb;
            pc.q = q;
            pc.sp2 = su[2];
            pc.pat = side;
            pc.use_sigma = op.sigma;
        }
    return n;
}

static int ny_pack_stage(acse_ctx* c, NyWork* y, int s, const void* const S[2][3]) {
    const int r = c->r;
    NyPackList k;
    int n = 0;
    for (int g = 3 * s; g < 3 * s + 3; ++g)
        for (int side = 0; side < 2; ++side) {
            n = ny_pieces(y, r, g, side, S, side ? y->opB[g % 3] : y->opA[g % 3], &k, n);
            if (n < 0) return ACSE_ERR_UNSUPPORTED;
        }
    k.sig = y->sig;
    k.ld = (size_t)4 * y->Kbw;
    k.Kb = y->Kb;
    k.Kbw = y->Kbw;
    const size_t es = c->opt.prec == ACSE_FP64 ? sizeof(double) : sizeof(float);
    // about 4096 elements a block (16 a thread), within the 48 KB of shared memory that need no opt-in
    int nslab = 4096 / (r * r);
    nslab = nslab < 1 ? 1 : nslab > 16 ? 16 : nslab;
    while (nslab > 1 && nslab * (size_t)r * (r + 1) * es > 40 * 1024) --nslab;
    const size_t sm = nslab * (size_t)r * (r + 1) * es;
    const int blocks = n * ((r * r + nslab - 1) / nslab);
    switch (c->opt.prec) {
        case ACSE_FP64: k_ny_pack<ACSE_FP64><<<blocks, 256, sm, c->stream>>>(r, nslab, k); break;
        case ACSE_BF16X3: k_ny_pack<ACSE_BF16X3><<<blocks, 256, sm, c->stream>>>(r, nslab, k); break;
        case ACSE_TF32X3: k_ny_pack<ACSE_TF32X3><<<blocks, 256, sm, c->stream>>>(r, nslab, k); break;
        default: k_ny_pack<ACSE_TF32><<<blocks, 256, sm, c->stream>>>(r, nslab, k); break;
    }
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// The NY term T for the pass in flight (D = c->cur_D, W = c->cur_W, 1D in c->w.gam), left in the
// four spin-type buffers the B kernel adds to B.
int ny_pass(acse_ctx* c) {
    NyWork* y = (NyWork*)c->ny;
    if (!y) return ACSE_ERR_UNSUPPORTED;
    const int r = c->r, R2 = r * r;
    const bool f64 = c->opt.prec == ACSE_FP64;
    if (c->cur_prep) {   // 2Delta is that of D: the update pass finds the residual pass's
        if (f64)
            k_ny_delta<double><<<152 * 8, 256, 0, c->stream>>>(r, c->w.gam, c->cur_D[0], c->cur_D[1], c->cur_D[2],
                                                               (double*)y->delta[0], (double*)y->delta[1], (double*)y->delta[2]);
        else
            k_ny_delta<float><<<152 * 8, 256, 0, c->stream>>>(r, c->w.gam, c->cur_D[0], c->cur_D[1], c->cur_D[2],
                                                              (float*)y->delta[0], (float*)y->delta[1], (float*)y->delta[2]);
        ACSE_LAUNCHED(c);
    }
    const void* S[2][3];
    for (int b = 0; b < 3; ++b) {
        S[0][b] = y->delta[b];
        S[1][b] = f64 ? (const void*)c->cur_W[b] : (const void*)c->cur_W32[b];
    }
    const size_t ld = (size_t)4 * y->Kbw;
    for (int s = 0; s < 2; ++s) {
        ACSE_TRY(ny_pack_stage(c, y, s, S));
        if (f64) {
            GemmF64 gl[48];
            int ng = 0;
            for (int g = 3 * s; g < 3 * s + 3; ++g)
                for (int k = 0; k < y->nprob[g]; ++k) {
                    const int rb = y->prob[g][k][0], cb = y->prob[g][k][1], q0 = y->prob[g][k][2], cnt = y->prob[g][k][3];
                    const double* A = (const double*)y->opA[g % 3] + (size_t)rb * R2 * ld + (size_t)q0 * R2;
                    const double* B = (const double*)y->opB[g % 3] + (size_t)cb * R2 * ld + (size_t)q0 * R2;
                    double* C = (double*)y->out[g] + (size_t)rb * R2 * y->n2 + (size_t)cb * R2;
                    gl[ng++] = GemmF64{A, B, C, R2, R2, cnt * R2, (int)ld, (int)ld, (int)y->n2, 1.0, nullptr, nullptr, nullptr};
                }
            ACSE_TRY(gemm_f64_grouped(c, gl, ng, c->stream));
        } else {
            ACSE_TRY(tc_table_launch(&y->st[s], c->stream));
            c->launches++;
        }
    }
    const int n = y->n;
    const size_t smem = 2 * (size_t)n * ((r + 3) & ~3) * (f64 ? sizeof(double) : sizeof(float));
    if (f64) {
        k_ny_Q<double><<<(n * n + 7) / 8, 256, 0, c->stream>>>(r, (const double*)y->out[0], (double*)y->Q);
        ACSE_LAUNCHED(c);
        k_ny_assemble<double><<<4 * R2, 256, smem, c->stream>>>(
            r, (const double*)y->out[3], (const double*)y->out[4], (const double*)y->out[5], (const double*)y->Q,
            (const double*)y->delta[0], (const double*)y->delta[1], (const double*)y->delta[2], y->sig, (double*)y->tny[0], (double*)y->tny[1], (double*)y->tny[2], (double*)y->tny[3]);
    } else {
        k_ny_Q<float><<<(n * n + 7) / 8, 256, 0, c->stream>>>(r, (const float*)y->out[0], (float*)y->Q);
        ACSE_LAUNCHED(c);
        k_ny_assemble<float><<<4 * R2, 256, smem, c->stream>>>(
            r, (const float*)y->out[3], (const float*)y->out[4], (const float*)y->out[5], (const float*)y->Q,
            (const float*)y->delta[0], (const float*)y->delta[1], (const float*)y->delta[2], y->sig, (float*)y->tny[0], (float*)y->tny[1], (float*)y->tny[2], (float*)y->tny[3]);
    }
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// T buffers of the four B spin types (null without NY).
const void* ny_terms(acse_ctx* c, int t) {
    NyWork* y = (NyWork*)c->ny;
    return y ? y->tny[t] : nullptr;
}

int ny_set_attrs() {
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_ny_assemble<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       2 * 2 * ACSE_MAX_R * ACSE_MAX_R * (int)sizeof(double)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_ny_assemble<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       2 * 2 * ACSE_MAX_R * ACSE_MAX_R * (int)sizeof(float)));
    return ACSE_OK;
}
