// Adjoint of the ACSE trajectory (new; the paper has no adjoint): gradients of
//     f = wE E(D_n) + wN ||A(D_n)||^2,   D_{k+1} = D_k + eps U(D_k),   U(D) = 1/2 G(mask(A(D)); D),
//     A(D) = G(K/2; D)
// with respect to h, V (through K, Eq. 2) and D_0, FP64 path.
//
// Two vector-Jacobian products of a contraction pass G(W; D) are needed:
//  * with respect to W: the commutator bilinear form beta(X, Y) = sum_spin-orbital X . G(Y) is
//    antisymmetric, beta(X, Y) = -beta(Y, X), with the Valdemoro 3-RDM as with the exact one
//    (checked by the oracle tests).  For block cotangents Gb this gives
//        dL/dW_aa = -G(Gh)_aa,  dL/dW_bb = -G(Gh)_bb,  dL/dW_ab = -4 G(Gh)_ab,
//    Gh = (P Gb_aa, Gb_ab / 4, P Gb_bb) (P: antisymmetriser within the index pairs), evaluated as
//    one forward pass: G of a pair-Hermitian W is anti-Hermitian and of an anti-Hermitian W Hermitian, so only
//    the part of Gh with the symmetry of G's output meets it, and the pass on that part gives the gradient
//    within the symmetry class of W;
//  * with respect to D: a reverse pass through the factorisation of acse_elem.cu / acse_tiled.cu
//    (G = H - s H^T, H = 4Y - 12(P - P'_{k<->l}), the B spin types, the pair and particle-hole GEMMs,
//    V5, w, Q, M = 3D - 2(1D^1D), 1D = 2/(N-1) tr D), written out below term by term.  Cotangents are kept up to
//    parts orthogonal to the symmetries of the tensors they belong to (those parts meet nothing and leave
//    with the final projection), which puts the reversed O(r^6) products on the symmetrised pairs of the
//    forward pass (acse_ph.cu).
#include <math.h>
#include <string.h>

#include "acse_internal.h"
#include "dfloat.cuh"

#define AD_TPB 256

int acse_contract(acse_ctx* c, const double* const D[3], const double* const W[3], int sW, double scale, int mask,
                  double* const out[3], double* norm2_dst, int prep_D);

static inline int ad_grid(size_t n) {
    size_t g = (n + AD_TPB - 1) / AD_TPB;
    if (g > 152 * 16) g = 152 * 16;
    return (int)(g < 1 ? 1 : g);
}

__device__ __forceinline__ double ad_warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ double ad_block_sum(double v) {
    __shared__ double sh[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = ad_warp_sum(v);
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
    if (wid == 0) v = ad_warp_sum(v);
    __syncthreads();
    return v;
}

#define FOR_N(e, n) for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (n); e += (size_t)gridDim.x * blockDim.x)

// ------------------------------------------------------------------------ small helpers
// out_b[ij][kl] = a in_b[ij][kl] + b in_b[kl][ij] for the three blocks (pair transpose).
__global__ void k_pair_combine(int r, const double* __restrict__ i0, const double* __restrict__ i1,
                               const double* __restrict__ i2, double a, double b, double* o0, double* o1, double* o2) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(e, 3 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4, ij = g / R2, kl = g % R2;
        const double* in = blk == 0 ? i0 : blk == 1 ? i1 : i2;
        double* out = blk == 0 ? o0 : blk == 1 ? o1 : o2;
        out[g] = a * in[g] + b * in[kl * R2 + ij];
    }
}

// Block cotangent -> its part of symmetry sG (pair-Hermitian or anti-Hermitian), spin-orbital normalised: aa, bb
// antisymmetrised within pairs, ab / 4, then (x + sG x^T) / 2.
__global__ void k_adj_project(int r, const double* __restrict__ g0, const double* __restrict__ g1,
                              const double* __restrict__ g2, double sG, double* o0, double* o1, double* o2) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(e, 3 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4;
        const int i = (int)(g / (R2 * r)), j = (int)((g / R2) % r), k = (int)((g / r) % r), l = (int)(g % r);
        const size_t ij = (size_t)i * r + j, kl = (size_t)k * r + l;
        if (blk == 1) {
            o1[g] = 0.125 * (g1[g] + sG * g1[kl * R2 + ij]);
        } else {
            const double* x = blk == 0 ? g0 : g2;
            const size_t ji = (size_t)j * r + i, lk = (size_t)l * r + k;
            const double v = x[ij * R2 + kl] - x[ji * R2 + kl] - x[ij * R2 + lk] + x[ji * R2 + lk];
            const double t = x[kl * R2 + ij] - x[kl * R2 + ji] - x[lk * R2 + ij] + x[lk * R2 + ji];
            (blk == 0 ? o0 : o2)[g] = 0.125 * (v + sG * t);
        }
    }
}

// out_b = mul_b x_b.
__global__ void k_scale3(size_t n4, const double* __restrict__ x0, const double* __restrict__ x1,
                         const double* __restrict__ x2, double m0, double m1, double m2, double* o0, double* o1,
                         double* o2) {
    FOR_N(e, 3 * n4) {
        const int b = (int)(e / n4);
        const size_t g = e % n4;
        if (b == 0) o0[g] = m0 * x0[g];
        else if (b == 1) o1[g] = m1 * x1[g];
        else o2[g] = m2 * x2[g];
    }
}

// acc_b += mul_b * x_b with mul = (m0, m1, m2) per block.
__global__ void k_axpy3(size_t n4, const double* __restrict__ x0, const double* __restrict__ x1,
                        const double* __restrict__ x2, double m0, double m1, double m2, double* a0, double* a1,
                        double* a2) {
    FOR_N(e, 3 * n4) {
        const int b = (int)(e / n4);
        const size_t g = e % n4;
        if (b == 0) a0[g] += m0 * x0[g];
        else if (b == 1) a1[g] += m1 * x1[g];
        else a2[g] += m2 * x2[g];
    }
}

// out = in with the all-active entries zeroed (or a copy when mask is off).
__global__ void k_mask_copy(int r, const double* __restrict__ i0, const double* __restrict__ i1,
                            const double* __restrict__ i2, int mask, int lo, int hi, double* o0, double* o1, double* o2) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(e, 3 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4;
        const int i = (int)(g / (R2 * r)), j = (int)((g / R2) % r), k = (int)((g / r) % r), l = (int)(g % r);
        const double* in = blk == 0 ? i0 : blk == 1 ? i1 : i2;
        double v = in[g];
        if (mask && i >= lo && i < hi && j >= lo && j < hi && k >= lo && k < hi && l >= lo && l < hi) v = 0.0;
        (blk == 0 ? o0 : blk == 1 ? o1 : o2)[g] = v;
    }
}

// ------------------------------------------------------------------ reverse of the assembly
// From Hb (cotangent of H): tau = Bbar / 9 with
//   B0bar = -12 Hb_aa + 12 Hb_aa(k<->l), B1bar likewise, B2bar = -12 Hb_ab, B3bar = 12 Hb_ab(k<->l).
__global__ void k_adj_tau(int r, const double* __restrict__ Haa, const double* __restrict__ Hab,
                          const double* __restrict__ Hbb, double* t0, double* t1, double* t2, double* t3) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    const double c = 12.0 / 9.0;
    FOR_N(g, n4) {
        const size_t ij = g / R2;
        const int k = (int)((g / r) % r), l = (int)(g % r);
        const size_t lk = ij * R2 + (size_t)l * r + k;
        t0[g] = c * (Haa[lk] - Haa[g]);
        t1[g] = c * (Hbb[lk] - Hbb[g]);
        t2[g] = -c * Hab[g];
        t3[g] = c * Hab[lk];
    }
}

// The r x r x r products of every pair ij behind Xbar (x1) and the x2 part of Mbar, as eight classes
//     out_c[ij][a][b] = sum_x T(a, x) G[b][x]
//   c   T(a,x)      G[b][x]     gives
//   0   t0[a][x]    ga[b][x]    Xb_aa[k=a][p=b]           1   t0[x][a]   wa[x][b]   -Mb_aa[l=a][p=b] / 2
//   2   t1[a][x]    gb[b][x]    Xb_bb                      3   t1[x][a]   wb[x][b]   -Mb_bb / 2
//   4   t2[a][x]    gb[b][x]    Xb_ab[(a,b)]               5   t2[x][a]   wa[x][b]    Mb_ab[u=b][v=a] / 2
//   6   t3[a][x]    ga[b][x]   -Xb_ab[(b,a)]               7   t3[x][a]   wb[x][b]   -Mb_ab[u=a][v=b] / 2
// (launch_pair_rows).
// Small-matrix reductions over a large sum (tall and skinny, r x r outputs): C_j[u][v] = sum_n sum_x
// A_j(n; x, u) B_j(n; x, v) for the 14 jobs below, n over r^2 blocks of r x r.  Block (job, chunk of n): both
// operand blocks in shared memory, nt^2 threads (nt = ceil(r / 4)) own a 4 x 4 tile of C each, and where those do
// not fill the block, groups of them take every G-th x; the groups meet in shared memory and the block
// writes one partial C, summed in a fixed order by k_adj_small.  (One block per output element, as before, read
// every operand r times from L2: 2.4 ms for the 14 jobs at r = 32.)  FP64 in every context: in double-float pairs (48
// bits, the range of FP32) the gradients of an Ozaki context lost bits, and more of them the smaller the cotangent.
//   job 0-3   gbar from x1:  Xaa[ij][x][u] t0[ij][x][v],  Xbb t1,  Xab[ij][x][u] t2[ij][x][v],  Xab[ij][u][x] t3[ij][x][v]
//   job 4-7   wbar from x2:  t0[ij][u][x] Maa[ij][x][v],  t1 Mbb,  t2[ij][u][x] Mab[ij][v][x],  t3[ij][u][x] Mab[ij][x][v]
//   job 8-13  gbar from X5 = 1D V5: X5b_t[(k,u)][(i,x)] V5_t[(k,v)][(i,x)], n = (k, i), sectors t = 0-3 and the flips
#define AD_JOBS 14
struct AdjRed {
    const double* A[AD_JOBS];
    const double* B[AD_JOBS];
    int asx[AD_JOBS], asu[AD_JOBS], bsx[AD_JOBS], bsv[AD_JOBS];   // element strides of x and u / v
    size_t sn_hi[AD_JOBS];                                        // n = (n / r, n % r): offsets of both parts
    size_t sn_lo[AD_JOBS];
    double* part;   // [job][nb][r^2]
    int r, nb, groups;
};

__global__ void __launch_bounds__(256) k_adj_reduce(const __grid_constant__ AdjRed a) {
    extern __shared__ __align__(16) unsigned char ad_raw[];
    const int r = a.r, rp = (r + 3) & ~3, R2 = r * r, nt = rp / 4, nt2 = nt * nt;
    const int job = (int)blockIdx.x / a.nb, chunk = (int)blockIdx.x - job * a.nb;
    double* As = (double*)ad_raw;     // [x][u]
    double* Bs = As + (size_t)r * rp; // [x][v]
    const int g = threadIdx.x / nt2, tile = threadIdx.x - g * nt2;
    const bool active = g < a.groups;
    const int u0 = (tile / nt) * 4, v0 = (tile % nt) * 4;
    double acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.0;
    for (int e = threadIdx.x; e < r * rp; e += blockDim.x) As[e] = Bs[e] = 0.0;
    const int per = (R2 + a.nb - 1) / a.nb, n1 = min(R2, (chunk + 1) * per);
    for (int n = chunk * per; n < n1; ++n) {
        const size_t off = (size_t)(n / r) * a.sn_hi[job] + (size_t)(n % r) * a.sn_lo[job];
        const double* A = a.A[job] + off;
        const double* B = a.B[job] + off;
        __syncthreads();
        for (int e = threadIdx.x; e < R2; e += blockDim.x) {   // consecutive threads along the unit stride
            const int hi = e / r, lo = e - hi * r;
            const int ax = a.asx[job] == 1 ? lo : hi, au = a.asx[job] == 1 ? hi : lo;
            As[ax * rp + au] = A[(size_t)ax * a.asx[job] + (size_t)au * a.asu[job]];
            const int bx = a.bsx[job] == 1 ? lo : hi, bv = a.bsx[job] == 1 ? hi : lo;
            Bs[bx * rp + bv] = B[(size_t)bx * a.bsx[job] + (size_t)bv * a.bsv[job]];
        }
        __syncthreads();
        if (active)
            for (int x = g; x < r; x += a.groups) {
                double p[4], q[4];
                ld4(As + x * rp + u0, p);
                ld4(Bs + x * rp + v0, q);
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[u][v] = fma(p[u], q[v], acc[u][v]);
            }
    }
    __syncthreads();
    double* sh = (double*)ad_raw;   // [r][rp], the groups in turn
    for (int h = 0; h < a.groups; ++h) {
        if (active && g == h)
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (u0 + u < r) {
                        double* d = sh + (size_t)(u0 + u) * rp + v0 + v;
                        *d = (h ? *d : 0.0) + acc[u][v];
                    }
        __syncthreads();
    }
    double* out = a.part + (size_t)blockIdx.x * R2;
    for (int e = threadIdx.x; e < R2; e += blockDim.x) out[e] = sh[(e / r) * rp + e % r];
}

struct AdjB {
    int r;
    const double* tau[4];
    const double* gam;
    const double* Q;
    const double* part;   // k_adj_reduce
    int nb;
    double* X5bd;
    double* X5bf[2];
    double* wb;
    double* Qb;
    double* gb;
};

// X5bar, in the forward (row-major) layouts:
//   X5bd(a,a)[(k,j)][(i,l)] = 2 t0[ijkl] - 2 t0[jikl]     X5bd(b,b) likewise with t1
//   X5bd(a,b)[(k,j)][(i,l)] = -2 t2[jikl]                  X5bd(b,a)[(k,j)][(i,l)] = 2 t3[ijkl]
//   X5bf1[(k,j)][(i,l)] = 2 t2[ijkl]                        X5bf2[(k,j)][(i,l)] = -2 t3[jikl]
__global__ void k_adj_X5(const __grid_constant__ AdjB a) {
    const int r = a.r;
    const size_t R2 = (size_t)r * r, n4 = R2 * R2, R22 = 2 * R2;
    FOR_N(e, 6 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4, row = g / R2, col = g % R2;
        const int k = (int)(row / r), j = (int)(row % r), i = (int)(col / r), l = (int)(col % r);
        const size_t ijkl = (((size_t)i * r + j) * r + k) * r + l, jikl = (((size_t)j * r + i) * r + k) * r + l;
        double v;
        switch (blk) {
            case 0: v = 2.0 * (a.tau[0][ijkl] - a.tau[0][jikl]); break;
            case 1: v = -2.0 * a.tau[2][jikl]; break;
            case 2: v = 2.0 * a.tau[3][ijkl]; break;
            case 3: v = 2.0 * (a.tau[1][ijkl] - a.tau[1][jikl]); break;
            case 4: v = 2.0 * a.tau[2][ijkl]; break;
            default: v = -2.0 * a.tau[3][jikl]; break;
        }
        if (blk < 4) {
            const int sK = blk >> 1, sI = blk & 1;
            a.X5bd[(sK * R2 + row) * R22 + sI * R2 + col] = v;
        } else {
            a.X5bf[blk - 4][g] = v;
        }
    }
}

// wbar, Qbar and the first part of gbar (block per output): the partial sums of k_adj_reduce and the O(r^4) terms
//   wb_a = -2 job4 + 2 job6,  wb_b = -2 job5 - 2 job7
//   Qb_a[k][i] = -sum_{jl} t0[ijkl] ga[jl] + sum_{i'l} t0[i' i k l] ga[i'l] - sum_{jl} t2[ijkl] gb[jl]
//   Qb_b[k][i] = -sum t1[ijkl] gb[jl] + sum t1[i' i k l] gb[i'l] + sum t3[i' i k l] ga[i'l]
//   gb_a[p][l] = job0 - job3 + (job8 + job9 + job13)[p][l]
//               - sum_{ik} t0[i p k l] Qa[k][i] + sum_{jk} t0[p j k l] Qa[k][j] + sum_{jk} t3[p j k l] Qb[k][j]
//   gb_b[p][l] = job1 + job2 + (job10 + job11 + job12)[p][l]
//               - sum t1[i p k l] Qb[k][i] + sum t1[p j k l] Qb[k][j] - sum t2[i p k l] Qa[k][i]
__global__ void __launch_bounds__(128) k_adj_small(const __grid_constant__ AdjB a) {
    const int r = a.r;
    const size_t R2 = (size_t)r * r;
    const int which = blockIdx.x / (2 * (int)R2);     // 0: w, 1: Q, 2: gamma
    const int t = blockIdx.x % (2 * (int)R2);
    const int sp = t / (int)R2, k = (t / r) % r, q = t % r;
    const double* ga = a.gam;
    const double* gb = a.gam + R2;
    auto job = [&](int j, double m) {
        double v = 0.0;
        for (int b = threadIdx.x; b < a.nb; b += blockDim.x) v += a.part[((size_t)j * a.nb + b) * R2 + (size_t)k * r + q];
        return m * v;
    };
    double acc = 0.0;
    if (which == 0) {
        acc = sp == 0 ? job(4, -2.0) + job(6, 2.0) : job(5, -2.0) + job(7, -2.0);
    } else if (which == 1) {
        const int i = q;
        for (size_t e = threadIdx.x; e < R2; e += blockDim.x) {
            const int jj = (int)(e / r), l = (int)(e % r);
            const size_t ijkl = (((size_t)i * r + jj) * r + k) * r + l;      // j = jj
            const size_t jikl = (((size_t)jj * r + i) * r + k) * r + l;      // i' = jj
            if (sp == 0)
                acc += -a.tau[0][ijkl] * ga[jj * r + l] + a.tau[0][jikl] * ga[jj * r + l] - a.tau[2][ijkl] * gb[jj * r + l];
            else
                acc += -a.tau[1][ijkl] * gb[jj * r + l] + a.tau[1][jikl] * gb[jj * r + l] + a.tau[3][jikl] * ga[jj * r + l];
        }
    } else {
        const double* Qa = a.Q;
        const double* Qb = a.Q + R2;
        const int pp = k, l = q;
        acc = sp == 0 ? job(0, 1.0) + job(3, -1.0) + job(8, 1.0) + job(9, 1.0) + job(13, 1.0)
                      : job(1, 1.0) + job(2, 1.0) + job(10, 1.0) + job(11, 1.0) + job(12, 1.0);
        for (size_t e = threadIdx.x; e < R2; e += blockDim.x) {   // (x, k): x = i or j
            const int x = (int)(e / r), kk = (int)(e % r);
            const size_t xpkl = (((size_t)x * r + pp) * r + kk) * r + l;   // t[x p k l]
            const size_t pxkl = (((size_t)pp * r + x) * r + kk) * r + l;   // t[p x k l]
            if (sp == 0)
                acc += -a.tau[0][xpkl] * Qa[kk * r + x] + a.tau[0][pxkl] * Qa[kk * r + x] + a.tau[3][pxkl] * Qb[kk * r + x];
            else
                acc += -a.tau[1][xpkl] * Qb[kk * r + x] + a.tau[1][pxkl] * Qb[kk * r + x] - a.tau[2][xpkl] * Qa[kk * r + x];
        }
    }
    acc = ad_block_sum(acc);
    if (threadIdx.x == 0) (which == 0 ? a.wb : which == 1 ? a.Qb : a.gb)[t] = acc;
}

// wbar -> gbar through w (k_ph_w_diag):
//   gb_a[p][q] += sum_{ks} wb_a[k][s] Waa[k][p][q][s] - wb_b[k][s] Wab[p][k][q][s]
//   gb_b[p][q] += sum_{ks} wb_b[k][s] Wbb[k][p][q][s] - wb_a[k][s] Wab[k][p][s][q]
__global__ void __launch_bounds__(128) k_adj_w_gamma(int r, const double* __restrict__ Waa, const double* __restrict__ Wab,
                                                     const double* __restrict__ Wbb, const double* __restrict__ wb,
                                                     double* gb) {
    const size_t R2 = (size_t)r * r, r3 = R2 * r;
    const int t = blockIdx.x, sp = t / (int)R2, p = (t / r) % r, q = t % r;
    double acc = 0.0;
    for (size_t e = threadIdx.x; e < R2; e += blockDim.x) {
        const int k = (int)(e / r), s = (int)(e % r);
        if (sp == 0)
            acc += wb[e] * Waa[k * r3 + p * R2 + (size_t)q * r + s] - wb[R2 + e] * Wab[p * r3 + k * R2 + (size_t)q * r + s];
        else
            acc += wb[R2 + e] * Wbb[k * r3 + p * R2 + (size_t)q * r + s] - wb[e] * Wab[k * r3 + p * R2 + (size_t)s * r + q];
    }
    acc = ad_block_sum(acc);
    if (threadIdx.x == 0) gb[t] += acc;
}

// ------------------------------------------------- operands of the reversed O(r^6) products
// With V5 = W_ph M_ph (acse_ph.cu) and V its cotangent, the cotangent of M_ph within its symmetry class is
// M+ (symmetric in (i,l) and (p,t)) plus M- (antisymmetric in both):
//   M+[{il}][{pt}] = sum_{kq} v1[{il}][{kq}] W+[{kq}][{pt}],   M-[{il}][{pt}] = sum_{kq} v2[{il}][{kq}] W-[{kq}][{pt}]
//   v1[{il}][{k<q}] = (V(kq;il) + V(kq;li) + s V(qk;il) + s V(qk;li)) / 2,  v1[{il}][{kk}] = (V(kk;il) + V(kk;li)) / 2
//   v2[{il}][{k<q}] = (V(kq;il) - V(kq;li) - s V(qk;il) + s V(qk;li)) / 2,  v2[{il}][{kk}] = (V(kk;il) - V(kk;li)) / 2
// (v1 has the columns kk for s = +1 only, v2 for s = -1 only, as W+ and W- have those rows).  For s = +1 the
// stored W+ and W- are symmetric matrices; for s = -1 the transpose of one is the other; so both products
// read the forward operands K-major.  The flips: V5f2 = s V5f1 exchanged, so
//   vf[(i,l)][(q,k)] = s V5f1bar[(k,q)][(i,l)] + V5f2bar[(q,k)][(l,i)],  Mf1bar[(i,l)][(t,p)] = sum vf Wf1[(t,p)][(q,k)].
// Block (K, I, {k<=q}): the two rows of V go through shared memory; the outputs are written transposed (scattered
// 8-byte stores whose sectors neighbouring blocks complete in L2).
struct AdjV {
    const double* V;
    const double* f1;
    const double* f2;
    double* v1;
    double* v2;
    double* vf;
    int r, s;
};

__global__ void __launch_bounds__(256) k_adj_pack_V(const __grid_constant__ AdjV a) {
    extern __shared__ double ad_sm[];   // 2 r^2
    const int r = a.r, S = r * (r + 1) / 2, P = r * (r - 1) / 2;
    const size_t R2 = (size_t)r * r;
    const double s = (double)a.s;
    if ((int)blockIdx.x < 4 * S) {
        const int KI = (int)blockIdx.x / S, u = (int)blockIdx.x - KI * S, K = KI >> 1, I = KI & 1;
        int k, q;
        ps_unpair(r, u, k, q);
        const double* s1 = a.V + ((size_t)K * R2 + (size_t)k * r + q) * 2 * R2 + I * R2;
        const double* s2 = a.V + ((size_t)K * R2 + (size_t)q * r + k) * 2 * R2 + I * R2;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            ad_sm[e] = s1[e];
            ad_sm[R2 + e] = k < q ? s * s2[e] : 0.0;
        }
        __syncthreads();
        const int cS = K * S + u, cA = k < q ? K * P + pk_pair(r, k, q) : -1;
        const int c1 = a.s > 0 ? cS : cA, c2 = a.s > 0 ? cA : cS;
        const size_t ld1 = 2 * (size_t)(a.s > 0 ? S : P), ld2 = 2 * (size_t)(a.s > 0 ? P : S);
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int i = e / r, l = e - i * r;
            if (l < i) continue;
            const int t = l * r + i;
            if (c1 >= 0)
                a.v1[((size_t)I * S + ps_pair(r, i, l)) * ld1 + c1] =
                    0.5 * ((ad_sm[e] + ad_sm[t]) + (ad_sm[R2 + e] + ad_sm[R2 + t]));
            if (c2 >= 0 && i < l)
                a.v2[((size_t)I * P + pk_pair(r, i, l)) * ld2 + c2] =
                    0.5 * ((ad_sm[e] - ad_sm[t]) - (ad_sm[R2 + e] - ad_sm[R2 + t]));
        }
    } else {
        const int kq = (int)blockIdx.x - 4 * S, k = kq / r, q = kq - k * r;
        const double* x1 = a.f1 + (size_t)kq * R2;
        const double* x2 = a.f2 + ((size_t)q * r + k) * R2;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) ad_sm[e] = x2[e];
        __syncthreads();
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int i = e / r, l = e - i * r;
            a.vf[(size_t)e * R2 + (size_t)q * r + k] = s * x1[e] + ad_sm[l * r + i];
        }
    }
}

// Xbar and Ybar = 4 Hb as operands of Mbar += f Xbar W and Dbar += f Ybar W, W^{kp}_{rq} = s W^{rq}_{kp} read
// K-major: same-spin sectors on pairs i < j, k < p (both antisymmetrised, the sum over kp halved), all times s.
//   Xb_aa[ij][kp] = class 0 + (j = p) Qb_a[k][i]      Xb_bb[ij][kp] = class 2 + (j = p) Qb_b[k][i]
//   Xb_ab[ij][ab] = class 4 - class 6 transposed + (j = b) Qb_a[a][i] + (i = a) Qb_b[b][j]
struct AdjX {
    const double* H[3];
    const double* x0;   // classes 0, 2, 4, 6
    const double* x2;
    const double* x4;
    const double* x6;
    const double* Qb;
    double* X[3];
    double* Y[3];
    int r, s;
};

__global__ void __launch_bounds__(256) k_adj_pack_X(const __grid_constant__ AdjX a) {
    const int r = a.r, P = r * (r - 1) / 2;
    const size_t R2 = (size_t)r * r;
    const double s = (double)a.s;
    if ((int)blockIdx.x < 2 * P) {
        const int sec = (int)blockIdx.x / P, u = (int)blockIdx.x - sec * P;
        int i = 0;
        while (pk_pair(r, i, r - 1) < u) ++i;
        const int j = u - pk_pair(r, i, i + 1) + i + 1;
        const double* x = sec ? a.x2 : a.x0;
        const double* H = a.H[2 * sec];
        const double* Q = a.Qb + sec * R2;
        const double* xij = x + ((size_t)i * r + j) * R2;
        const double* xji = x + ((size_t)j * r + i) * R2;
        const double* hij = H + ((size_t)i * r + j) * R2;
        const double* hji = H + ((size_t)j * r + i) * R2;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int k = e / r, p = e - k * r;
            if (p <= k) continue;
            const int t = p * r + k, o = pk_pair(r, k, p);
            double v = (xij[e] - xij[t]) - (xji[e] - xji[t]);
            if (j == p) v += Q[k * r + i];
            if (j == k) v -= Q[p * r + i];
            if (i == p) v -= Q[k * r + j];
            if (i == k) v += Q[p * r + j];
            a.X[2 * sec][(size_t)u * P + o] = 0.5 * s * v;
            a.Y[2 * sec][(size_t)u * P + o] = 2.0 * s * ((hij[e] - hij[t]) - (hji[e] - hji[t]));
        }
    } else {
        const int ij = (int)blockIdx.x - 2 * P, i = ij / r, j = ij - i * r;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int p = e / r, q = e - p * r;
            const size_t g = (size_t)ij * R2 + e;
            double v = a.x4[g] - a.x6[(size_t)ij * R2 + (size_t)q * r + p];
            if (j == q) v += a.Qb[p * r + i];
            if (i == p) v += a.Qb[R2 + q * r + j];
            a.X[1][g] = s * v;
            a.Y[1][g] = 4.0 * s * a.H[1][g];
        }
    }
}

// Mbar blocks: the x2 part (classes 1, 3, 5, 7), the pair products and the particle-hole ones,
//   Mb_aa[i][p][l][t] = M_ph[(a,i,l)][(a,p,t)], Mb_ab[i][p][l][t] = M_ph[(a,i,l)][(b,p,t)] + M_ph[(b,p,t)][(a,i,l)],
//   Mb_ab[i][p][t][l] += Mf1bar[(i,l)][(t,p)],  M_ph = M+ +- M- by the order of i, l and of p, t.
struct AdjM {
    const double* c1;   // classes
    const double* c3;
    const double* c5;
    const double* c7;
    const double* pair[3];   // aa, bb packed (P x P), ab full
    const double* mp;        // 2S x 2S
    const double* mm;        // 2P x 2P
    const double* mf;
    double* M[3];
    int r;
};

__device__ __forceinline__ double adj_ph(const AdjM& a, int I, int i, int l, int Q, int p, int t) {
    const int r = a.r, S = r * (r + 1) / 2, P = r * (r - 1) / 2;
    const int il = i <= l ? ps_pair(r, i, l) : ps_pair(r, l, i), pt = p <= t ? ps_pair(r, p, t) : ps_pair(r, t, p);
    double v = a.mp[(size_t)(I * S + il) * 2 * S + Q * S + pt];
    if (i != l && p != t) {
        const int jl = i < l ? pk_pair(r, i, l) : pk_pair(r, l, i), qt = p < t ? pk_pair(r, p, t) : pk_pair(r, t, p);
        const double m = a.mm[(size_t)(I * P + jl) * 2 * P + Q * P + qt];
        v += ((i < l) == (p < t)) ? m : -m;
    }
    return v;
}

__global__ void __launch_bounds__(AD_TPB) k_adj_M(const __grid_constant__ AdjM a) {
    const int r = a.r, P = r * (r - 1) / 2;
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(e, 3 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4, ij = g / R2;
        const int a0 = (int)(g / (R2 * r)), a1 = (int)((g / R2) % r), a2 = (int)((g / r) % r), a3 = (int)(g % r);
        if (blk != 1) {
            double v = -2.0 * (blk == 0 ? a.c1 : a.c3)[g];
            if (a0 != a1 && a2 != a3) {
                const double x = a.pair[blk][(size_t)(a0 < a1 ? pk_pair(r, a0, a1) : pk_pair(r, a1, a0)) * P +
                                             (a2 < a3 ? pk_pair(r, a2, a3) : pk_pair(r, a3, a2))];
                v += ((a0 < a1) == (a2 < a3)) ? x : -x;
            }
            a.M[blk][g] = v + adj_ph(a, blk / 2, a0, a2, blk / 2, a1, a3);
        } else {
            double v = 2.0 * (a.c5[ij * R2 + (size_t)a3 * r + a2] - a.c7[g]) + a.pair[1][g];
            v += adj_ph(a, 0, a0, a2, 1, a1, a3) + adj_ph(a, 1, a1, a3, 0, a0, a2);
            a.M[1][g] = v + a.mf[((size_t)a0 * r + a3) * R2 + (size_t)a2 * r + a1];
        }
    }
}

// Mbar -> gbar through M = 3D - 2(1D^1D) (block per (sp, a, b)):
//   gb_a[a][b] += -sum_{jl} Mb_aa[a j b l] ga[jl] - sum_{ik} Mb_aa[i a k b] ga[ik] + sum_{il} Mb_aa[i a b l] ga[il]
//                + sum_{jk} Mb_aa[a j k b] ga[jk] - sum_{jl} Mb_ab[a j b l] gb[jl]
//   gb_b[a][b] += (the same with Mb_bb, gb) - sum_{ik} Mb_ab[i a k b] ga[ik]
__global__ void k_adj_M_gamma(int r, const double* __restrict__ Maa, const double* __restrict__ Mab,
                              const double* __restrict__ Mbb, const double* __restrict__ gam, double* gb) {
    const size_t R2 = (size_t)r * r;
    const int t = blockIdx.x;
    const int sp = t / (int)R2, a = (t / r) % r, b = t % r;
    const double* g = gam + (sp == 0 ? 0 : R2);
    const double* go = gam + (sp == 0 ? R2 : 0);
    const double* Ms = sp == 0 ? Maa : Mbb;
    double acc = 0.0;
    for (size_t e = threadIdx.x; e < R2; e += blockDim.x) {
        const int x = (int)(e / r), y = (int)(e % r);
        acc += -Ms[(((size_t)a * r + x) * r + b) * r + y] * g[x * r + y]     // (j,l) = (x,y)
               - Ms[(((size_t)x * r + a) * r + y) * r + b] * g[x * r + y]    // (i,k) = (x,y)
               + Ms[(((size_t)x * r + a) * r + b) * r + y] * g[x * r + y]    // (i,l) = (x,y)
               + Ms[(((size_t)a * r + x) * r + y) * r + b] * g[x * r + y];   // (j,k) = (x,y)
        if (sp == 0) acc -= Mab[(((size_t)a * r + x) * r + b) * r + y] * go[x * r + y];
        else acc -= Mab[(((size_t)x * r + a) * r + y) * r + b] * go[x * r + y];
    }
    acc = ad_block_sum(acc);
    if (threadIdx.x == 0) gb[t] += acc;
}

// D accumulation: Db += 3 Mb + (Ybar W), and the 1D adjoint: Db_aa[p][q][r'][q] += c gb_a[p][r'],
// Db_ab[p][q][r'][q] += c gb_a[p][r'], Db_bb[p][q][r'][q] += c gb_b[p][r'], Db_ab[q][p][q][r'] += c gb_b[p][r'].
__global__ void k_adj_to_D(int r, double cN, const double* __restrict__ Maa, const double* __restrict__ Mab,
                           const double* __restrict__ Mbb, const double* __restrict__ Yaa, const double* __restrict__ Yab,
                           const double* __restrict__ Ybb, const double* __restrict__ gb, double* Daa, double* Dab,
                           double* Dbb) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    const int P = r * (r - 1) / 2;
    FOR_N(e, 3 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4;
        const int a0 = (int)(g / (R2 * r)), a1 = (int)((g / R2) % r), a2 = (int)((g / r) % r), a3 = (int)(g % r);
        if (blk != 1) {
            double v = 3.0 * (blk == 0 ? Maa : Mbb)[g];
            if (a0 != a1 && a2 != a3) {
                const double y = (blk == 0 ? Yaa : Ybb)[(size_t)(a0 < a1 ? pk_pair(r, a0, a1) : pk_pair(r, a1, a0)) * P +
                                                        (a2 < a3 ? pk_pair(r, a2, a3) : pk_pair(r, a3, a2))];
                v += ((a0 < a1) == (a2 < a3)) ? y : -y;
            }
            if (a1 == a3) v += cN * gb[(blk == 0 ? 0 : R2) + a0 * r + a2];
            (blk == 0 ? Daa : Dbb)[g] += v;
        } else {
            double v = 3.0 * Mab[g] + Yab[g];
            if (a1 == a3) v += cN * gb[a0 * r + a2];          // gamma_a part
            if (a0 == a2) v += cN * gb[R2 + a1 * r + a3];     // gamma_b part: Dab[q][p][q][r']
            Dab[g] += v;
        }
    }
}

// ----------------------------------------------------------------------- K -> (h, V)
// Kb: cotangent of the FULL K blocks.  Vb[abcd] = 1/2 (Kaa+Kbb+Kab)[a c b d] - 1/2 (Kaa+Kbb)[a c d b];
// hb[a][b] = (sum_j (Kaa+Kbb+Kab)[a j b j] + sum_i (Kaa+Kbb+Kab)[i a i b]
//             - sum_j (Kaa+Kbb)[a j j b] - sum_i (Kaa+Kbb)[i a b i]) / (2(N-1)).
// Then symmetrised: h over p<->q, V over the 8-fold permutational symmetry.
__global__ void k_adj_K_to_V(int r, const double* __restrict__ Kaa, const double* __restrict__ Kab,
                             const double* __restrict__ Kbb, double* Vraw) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(g, n4) {
        const int a = (int)(g / (R2 * r)), b = (int)((g / R2) % r), c = (int)((g / r) % r), d = (int)(g % r);
        const size_t acbd = (((size_t)a * r + c) * r + b) * r + d, acdb = (((size_t)a * r + c) * r + d) * r + b;
        Vraw[g] = 0.5 * (Kaa[acbd] + Kbb[acbd] + Kab[acbd]) - 0.5 * (Kaa[acdb] + Kbb[acdb]);
    }
}

__global__ void k_sym_V(int r, const double* __restrict__ Vr, double* dV) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(g, n4) {
        const int p = (int)(g / (R2 * r)), q = (int)((g / R2) % r), s1 = (int)((g / r) % r), s2 = (int)(g % r);
#define VI(a, b, c, d) Vr[(((size_t)(a) * r + (b)) * r + (c)) * r + (d)]
        dV[g] = 0.125 * (VI(p, q, s1, s2) + VI(q, p, s1, s2) + VI(p, q, s2, s1) + VI(q, p, s2, s1) + VI(s1, s2, p, q) +
                         VI(s2, s1, p, q) + VI(s1, s2, q, p) + VI(s2, s1, q, p));
#undef VI
    }
}

__global__ void k_adj_K_to_h(int r, double inv2N1, const double* __restrict__ Kaa, const double* __restrict__ Kab,
                             const double* __restrict__ Kbb, double* hraw) {
    const int t = blockIdx.x;
    const int a = t / r, b = t % r;
    double acc = 0.0;
    for (int x = threadIdx.x; x < r; x += blockDim.x) {
        const size_t axbx = (((size_t)a * r + x) * r + b) * r + x, xaxb = (((size_t)x * r + a) * r + x) * r + b;
        const size_t axxb = (((size_t)a * r + x) * r + x) * r + b, xabx = (((size_t)x * r + a) * r + b) * r + x;
        acc += Kaa[axbx] + Kbb[axbx] + Kab[axbx] + Kaa[xaxb] + Kbb[xaxb] + Kab[xaxb] - Kaa[axxb] - Kbb[axxb] -
               Kaa[xabx] - Kbb[xabx];
    }
    acc = ad_block_sum(acc);
    if (threadIdx.x == 0) hraw[t] = acc * inv2N1;
}

__global__ void k_sym_h(int r, const double* __restrict__ hr, double* dh) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= r * r) return;
    const int a = e / r, b = e % r;
    dh[e] = 0.5 * (hr[a * r + b] + hr[b * r + a]);
}

// dD projection onto 2-RDM symmetries: aa, bb antisymmetric within pairs and pair-Hermitian;
// ab pair-Hermitian.
__global__ void k_project_D(int r, const double* __restrict__ i0, const double* __restrict__ i1,
                            const double* __restrict__ i2, double* o0, double* o1, double* o2) {
    const size_t R2 = (size_t)r * r, n4 = R2 * R2;
    FOR_N(e, 3 * n4) {
        const int blk = (int)(e / n4);
        const size_t g = e % n4;
        const int i = (int)(g / (R2 * r)), j = (int)((g / R2) % r), k = (int)((g / r) % r), l = (int)(g % r);
        const size_t ij = (size_t)i * r + j, ji = (size_t)j * r + i, kl = (size_t)k * r + l, lk = (size_t)l * r + k;
        if (blk == 1) {
            o1[g] = 0.5 * (i1[ij * R2 + kl] + i1[kl * R2 + ij]);
        } else {
            const double* x = blk == 0 ? i0 : i2;
            const double A = 0.25 * (x[ij * R2 + kl] - x[ji * R2 + kl] - x[ij * R2 + lk] + x[ji * R2 + lk]);
            const double At = 0.25 * (x[kl * R2 + ij] - x[lk * R2 + ij] - x[kl * R2 + ji] + x[lk * R2 + ji]);
            (blk == 0 ? o0 : o2)[g] = 0.5 * (A + At);
        }
    }
}

// ------------------------------------------------------------------------------ workspace
// Every buffer is one entry of buf[] (freed together); the names point into them.
#define AD_MAXBUF 64
struct AdjWork {
    double* buf[AD_MAXBUF];
    int nbuf;
    double* Hb[3];
    double* tau[4];
    double* cls[8];    // the eight classes of products (the scratch of the B products, free between passes)
    double* X5b[3];    // X5bar: spin blocks, flips; then overwritten by the products mp, mm, mxab; mf; yab
    double* Vb[3];     // V5bar
    double* v1;
    double* v2;
    double* vf;
    double* Xp[3];
    double* Yp[3];
    double* mp;
    double* mm;
    double* mf;
    double* mx[3];
    double* my[3];
    double* Mb[3];
    double* wb;
    double* Qb;
    double* gb;
    double* part;
    int nb, groups, threads;   // launch shape of k_adj_reduce
    double* Gp[3];     // projected cotangent
    double* Wb[3];     // dL/dW
    double* Db[3];     // running dL/dD_k
    double* Dn[3];     // next dL/dD
    double* Kb[3];     // dL/dK (full K)
    double* Dk[3];     // D_k (recomputed)
    double* Araw[3];
    double* Am[3];
    double* Ab[3];
    double* sX[3];     // intermediates of the residual pass, kept over the update's
    double* sV[3];
    double* swQ;
    double* hraw;
    double* Vraw;
};

static int adj_alloc(acse_ctx* c) {
    if (c->adj) return ACSE_OK;
    AdjWork* a = (AdjWork*)calloc(1, sizeof(AdjWork));
    if (!a) return ACSE_ERR_NOMEM;
    const size_t r = c->r, R2 = r * r, n4 = R2 * R2, S2 = r * (r + 1), P2 = r * (r - 1), PP = P2 * P2 / 4;
    int st = ACSE_OK;
    auto get = [&](double*& p, size_t n) {
        if (st != ACSE_OK) return;
        if (cudaMalloc((void**)&p, (n ? n : 1) * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            st = ACSE_ERR_NOMEM;
            return;
        }
        a->buf[a->nbuf++] = p;
    };
    for (int s = 0; s < 3; ++s) {
        double** four[] = {&a->Hb[s], &a->Mb[s], &a->Gp[s], &a->Wb[s], &a->Db[s], &a->Dn[s], &a->Kb[s], &a->Dk[s],
                           &a->Araw[s], &a->Am[s], &a->Ab[s], &a->sX[s]};
        for (double** p : four) get(*p, n4);
        get(a->X5b[s], s ? n4 : 4 * n4);
        get(a->Vb[s], s ? n4 : 4 * n4);
        get(a->sV[s], s ? n4 : 4 * n4);
    }
    // one block each: tau, the pair operands and products, the small arrays
    double *tau = nullptr, *pairs = nullptr, *small = nullptr;
    get(tau, 4 * n4);
    get(pairs, 8 * PP + 2 * n4);
    get(a->v1, S2 * S2);
    get(a->v2, P2 * S2);
    get(a->vf, n4);
    get(a->Vraw, n4);
    const int nt = (int)(r + 3) / 4, nt2 = nt * nt;
    a->groups = 256 / nt2 < (int)r ? 256 / nt2 : (int)r;
    a->threads = (a->groups * nt2 + 31) / 32 * 32;
    a->nb = R2 < 44 ? (int)R2 : 44;   // 14 jobs x 44 chunks: four blocks an SM
    get(a->part, (size_t)AD_JOBS * a->nb * R2);
    get(small, 11 * R2);
    if (st != ACSE_OK) {
        for (int i = 0; i < a->nbuf; ++i) cudaFree(a->buf[i]);
        free(a);
        return st;
    }
    for (int t = 0; t < 4; ++t) a->tau[t] = tau + t * n4;
    for (int k = 0; k < 8; ++k) a->cls[k] = c->w.bx64[k];
    a->Xp[0] = pairs; a->Xp[2] = pairs + PP; a->Yp[0] = pairs + 2 * PP; a->Yp[2] = pairs + 3 * PP;
    a->mx[0] = pairs + 4 * PP; a->mx[2] = pairs + 5 * PP; a->my[0] = pairs + 6 * PP; a->my[2] = pairs + 7 * PP;
    a->Xp[1] = pairs + 8 * PP; a->Yp[1] = a->Xp[1] + n4;
    a->mp = a->X5b[0];                 // S2^2 + P2^2 + r^4 = 3 r^4 + 2 r^2 <= 4 r^4
    a->mm = a->mp + S2 * S2;
    a->mx[1] = a->mm + P2 * P2;
    a->mf = a->X5b[1];
    a->my[1] = a->X5b[2];
    a->wb = small; a->Qb = small + 2 * R2; a->gb = small + 4 * R2; a->swQ = small + 6 * R2; a->hraw = small + 10 * R2;
    c->adj = a;
    return ACSE_OK;
}

void adj_free(acse_ctx* c) {
    AdjWork* a = (AdjWork*)c->adj;
    if (!a) return;
    for (int i = 0; i < a->nbuf; ++i) cudaFree(a->buf[i]);
    free(a);
    c->adj = nullptr;
}

#define AL(c) ACSE_LAUNCHED(c)

// -------------------------------------------------------------------------- VJP w.r.t. D
// Requires the forward intermediates of G(W; D) (X, V5, w, Q) and the packed W of the pass (launch_ph_pack_W).
// Adds dL/dD to Dacc for L = <Gb, scale (H - s H^T)>.
static int vjp_D(acse_ctx* c, const double* const W[3], int sW, double scale, const double* const Gb[3],
                 double* const Dacc[3]) {
    AdjWork* a = (AdjWork*)c->adj;
    Work& w = c->w;
    const int r = c->r, R2 = r * r, S2 = r * (r + 1), P2 = r * (r - 1), P = P2 / 2, rp = (r + 3) & ~3;
    const size_t n4 = (size_t)R2 * R2, sm2 = 2 * (size_t)r * rp * sizeof(double);
    // assembly: Hb = scale (Gb - s Gb^T)
    k_pair_combine<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, Gb[0], Gb[1], Gb[2], scale, -scale * sW, a->Hb[0],
                                                            a->Hb[1], a->Hb[2]);
    AL(c);
    k_adj_tau<<<ad_grid(n4), AD_TPB, 0, c->stream>>>(r, a->Hb[0], a->Hb[1], a->Hb[2], a->tau[0], a->tau[1], a->tau[2],
                                                     a->tau[3]);
    AL(c);
    AdjB ab;
    ab.r = r;
    for (int t = 0; t < 4; ++t) ab.tau[t] = a->tau[t];
    ab.gam = w.gam; ab.Q = w.Q;
    ab.part = a->part; ab.nb = a->nb;
    ab.X5bd = a->X5b[0]; ab.X5bf[0] = a->X5b[1]; ab.X5bf[1] = a->X5b[2];
    ab.wb = a->wb; ab.Qb = a->Qb; ab.gb = a->gb;
    // products of every pair with 1D and w
    {
        const double *ga = w.gam, *gb = w.gam + R2, *wa = w.w, *wb = w.w + R2;
        const double* G[8] = {ga, wa, gb, wb, gb, wa, ga, wb};
        const double* T[8];
        for (int k = 0; k < 8; ++k) T[k] = a->tau[k / 2];
        ACSE_TRY(launch_pair_rows(c, T, 0xAAu, G, 0xAAu, 0u, a->cls));   // odd classes: T and G transposed
    }
    k_adj_X5<<<ad_grid(6 * n4), AD_TPB, 0, c->stream>>>(ab);
    AL(c);
    {
        AdjRed d;
        d.r = r; d.nb = a->nb; d.groups = a->groups; d.part = a->part;
        auto set = [&](int j, const double* A, bool at, const double* B, bool bt, int lda, int ldb, size_t hi, size_t lo) {
            d.A[j] = A; d.B[j] = B;
            d.asx[j] = at ? 1 : lda; d.asu[j] = at ? lda : 1;   // at: A stored [u][x]
            d.bsx[j] = bt ? 1 : ldb; d.bsv[j] = bt ? ldb : 1;
            d.sn_hi[j] = hi; d.sn_lo[j] = lo;
        };
        const size_t hi = (size_t)R2 * r, lo = R2;   // n = ij
        set(0, w.X[0], false, a->tau[0], false, r, r, hi, lo);
        set(1, w.X[2], false, a->tau[1], false, r, r, hi, lo);
        set(2, w.X[1], false, a->tau[2], false, r, r, hi, lo);
        set(3, w.X[1], true, a->tau[3], false, r, r, hi, lo);
        set(4, a->tau[0], true, w.M[0], false, r, r, hi, lo);
        set(5, a->tau[1], true, w.M[2], false, r, r, hi, lo);
        set(6, a->tau[2], true, w.M[1], true, r, r, hi, lo);
        set(7, a->tau[3], true, w.M[1], false, r, r, hi, lo);
        for (int t = 0; t < 6; ++t) {   // n = (k, i)
            const int ld = t < 4 ? 2 * R2 : R2;
            const size_t o = t < 4 ? (size_t)(t >> 1) * R2 * ld + (size_t)(t & 1) * R2 : 0;
            const double* A = t < 4 ? a->X5b[0] + o : a->X5b[t - 3];
            const double* B = t < 4 ? w.V5d + o : t == 4 ? w.V5f1 : w.V5f2;
            set(8 + t, A, true, B, true, ld, ld, (size_t)r * ld, r);
        }
        k_adj_reduce<<<AD_JOBS * a->nb, a->threads, sm2, c->stream>>>(d);
        AL(c);
    }
    k_adj_small<<<6 * R2, 128, 0, c->stream>>>(ab);
    AL(c);
    k_adj_w_gamma<<<2 * R2, 128, 0, c->stream>>>(r, W[0], W[1], W[2], a->wb, a->gb);
    AL(c);
    // V5bar = 1D^T X5bar, and the operands of the reversed products
    ACSE_TRY(launch_ph_xform(c, a->X5b, a->Vb, 1));
    AdjV av;
    av.V = a->Vb[0]; av.f1 = a->Vb[1]; av.f2 = a->Vb[2]; av.v1 = a->v1; av.v2 = a->v2; av.vf = a->vf; av.r = r; av.s = sW;
    k_adj_pack_V<<<2 * S2 + R2, 256, 2 * (size_t)R2 * sizeof(double), c->stream>>>(av);
    AL(c);
    AdjX ax;
    for (int s = 0; s < 3; ++s) { ax.H[s] = a->Hb[s]; ax.X[s] = a->Xp[s]; ax.Y[s] = a->Yp[s]; }
    ax.x0 = a->cls[0]; ax.x2 = a->cls[2]; ax.x4 = a->cls[4]; ax.x6 = a->cls[6]; ax.Qb = a->Qb; ax.r = r; ax.s = sW;
    k_adj_pack_X<<<2 * P + R2, 256, 0, c->stream>>>(ax);
    AL(c);
    // M+ and M- (for s = -1 the transposes of W+ and W- are W- and W+), the flip, and X W, Y W per sector
    GemmF64 g[9];
    int n = 0;
    const int n1 = sW > 0 ? S2 : P2, n2 = sW > 0 ? P2 : S2;
    g[n++] = GemmF64{a->v1, sW > 0 ? w.Wp : w.Wm, a->mp, S2, S2, n1, n1, n1, S2, 1.0, nullptr, nullptr, nullptr};
    g[n++] = GemmF64{a->vf, w.Wf1, a->mf, R2, R2, R2, R2, R2, R2, 1.0, nullptr, nullptr, nullptr};
    g[n++] = GemmF64{a->Xp[1], W[1], a->mx[1], R2, R2, R2, R2, R2, R2, 2.0, nullptr, nullptr, nullptr};
    g[n++] = GemmF64{a->Yp[1], W[1], a->my[1], R2, R2, R2, R2, R2, R2, 2.0, nullptr, nullptr, nullptr};
    g[n++] = GemmF64{a->v2, sW > 0 ? w.Wm : w.Wp, a->mm, P2, P2, n2, n2, n2, P2, 1.0, nullptr, nullptr, nullptr};
    for (int s = 0; s < 3; s += 2) {
        g[n++] = GemmF64{a->Xp[s], W[s], a->mx[s], P, P, P, P, R2, P, 1.0, nullptr, w.pmap, nullptr};
        g[n++] = GemmF64{a->Yp[s], W[s], a->my[s], P, P, P, P, R2, P, 1.0, nullptr, w.pmap, nullptr};
    }
    ACSE_TRY(c->oz ? oz_gemm_list(c, g, n, sW > 0 ? 0 : 1) : gemm_f64_grouped(c, g, n, c->stream));
    AdjM am;
    am.c1 = a->cls[1]; am.c3 = a->cls[3]; am.c5 = a->cls[5]; am.c7 = a->cls[7];
    for (int s = 0; s < 3; ++s) { am.pair[s] = a->mx[s]; am.M[s] = a->Mb[s]; }
    am.mp = a->mp; am.mm = a->mm; am.mf = a->mf; am.r = r;
    k_adj_M<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(am);
    AL(c);
    k_adj_M_gamma<<<2 * R2, AD_TPB, 0, c->stream>>>(r, a->Mb[0], a->Mb[1], a->Mb[2], w.gam, a->gb);
    AL(c);
    k_adj_to_D<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, 2.0 / (c->N - 1), a->Mb[0], a->Mb[1], a->Mb[2], a->my[0],
                                                         a->my[1], a->my[2], a->gb, Dacc[0], Dacc[1], Dacc[2]);
    AL(c);
    return ACSE_OK;
}

// -------------------------------------------------------------------------- VJP w.r.t. W
// Wb = dL/dW within the symmetry class of W for L = <Gb, G(W; D)> (scale 1), by beta(X, Y) = -beta(Y, X): G of the
// part of the cotangent that has the symmetry sG of G's output (-s of W), with block factors -1, -4, -1; the 1D
// and M of D must be current (prep_D done).  Overwrites the pass intermediates.
static int vjp_W(acse_ctx* c, const double* const D[3], const double* const Gb[3], int sG, double* const Wb[3]) {
    AdjWork* a = (AdjWork*)c->adj;
    const int r = c->r;
    const size_t n4 = (size_t)r * r * r * r;
    k_adj_project<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, Gb[0], Gb[1], Gb[2], (double)sG, a->Gp[0], a->Gp[1],
                                                             a->Gp[2]);
    AL(c);
    const double* Wp[3] = {a->Gp[0], a->Gp[1], a->Gp[2]};
    double* out[3] = {a->Ab[0], a->Ab[1], a->Ab[2]};
    ACSE_TRY(acse_contract(c, D, Wp, sG, 1.0, 0, out, nullptr, 0));
    k_scale3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Ab[0], a->Ab[1], a->Ab[2], -1.0, -4.0, -1.0, Wb[0],
                                                       Wb[1], Wb[2]);
    AL(c);
    return ACSE_OK;
}

// Intermediates of the residual pass (X, V5, w, Q), kept while the update pass overwrites them and put back for
// the residual's own reversal: copies in place of running that pass a second time.
static int adj_save(acse_ctx* c, bool back) {
    AdjWork* a = (AdjWork*)c->adj;
    Work& w = c->w;
    const size_t R2 = (size_t)c->r * c->r, b4 = R2 * R2 * sizeof(double);
    double* V[3] = {w.V5d, w.V5f1, w.V5f2};
    auto copy = [&](double* here, double* kept, size_t bytes) {
        return cudaMemcpyAsync(back ? here : kept, back ? kept : here, bytes, cudaMemcpyDeviceToDevice, c->stream);
    };
    for (int s = 0; s < 3; ++s) {
        ACSE_CUDA_TRY(copy(w.X[s], a->sX[s], b4));
        ACSE_CUDA_TRY(copy(V[s], a->sV[s], s ? b4 : 4 * b4));
    }
    ACSE_CUDA_TRY(copy(w.w, a->swQ, 2 * R2 * sizeof(double)));
    ACSE_CUDA_TRY(copy(w.Q, a->swQ + 2 * R2, 2 * R2 * sizeof(double)));
    return ACSE_OK;
}

// ---------------------------------------------------------------------------- trajectory
static int adj_set_attrs() {
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_adj_pack_V, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       2 * ACSE_MAX_R * ACSE_MAX_R * (int)sizeof(double)));
    const int sm2 = 2 * ACSE_MAX_R * ACSE_MAX_R * (int)sizeof(double);
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_adj_reduce, cudaFuncAttributeMaxDynamicSharedMemorySize, sm2));
    return ACSE_OK;
}

extern "C" int acse_residual_backward_impl(acse_ctx* c, const double* const* D_ckpt, int n_steps, double eps,
                                            double wE, double wN, double* dh, double* dV, double* dDaa,
                                            double* dDab, double* dDbb) {
    if (c->opt.prec != ACSE_FP64) return ACSE_ERR_UNSUPPORTED;
    if (!D_ckpt || n_steps < 0 || !D_ckpt[0] || !D_ckpt[1] || !D_ckpt[2]) return ACSE_ERR_ARG;
    ACSE_TRY(adj_set_attrs());
    ACSE_TRY(adj_alloc(c));
    struct InAdjoint {   // for every return below
        acse_ctx* c;
        explicit InAdjoint(acse_ctx* x) : c(x) { c->in_adjoint = 1; }
        ~InAdjoint() { c->in_adjoint = 0; }
    } in_adjoint(c);
    AdjWork* a = (AdjWork*)c->adj;
    Work& w = c->w;
    const int r = c->r;
    const size_t n4 = (size_t)r * r * r * r, b4 = n4 * sizeof(double);
    const double* Kh[3] = {w.Kh[0], w.Kh[1], w.Kh[2]};
    const int mask = c->opt.mask_active;
    // D_k for k = 0..n: checkpoint if given, else recomputed from D_{k-1} (stored in a->Dk per use)
    auto load_D = [&](int k) -> int {
        // recompute forward from the latest available checkpoint at or below k
        int k0 = k;
        while (k0 > 0 && !(D_ckpt[3 * k0] && D_ckpt[3 * k0 + 1] && D_ckpt[3 * k0 + 2])) --k0;
        for (int b = 0; b < 3; ++b)
            ACSE_CUDA_TRY(cudaMemcpyAsync(a->Dk[b], D_ckpt[3 * k0 + b], b4, cudaMemcpyDefault, c->stream));
        const double* Dc[3] = {a->Dk[0], a->Dk[1], a->Dk[2]};
        for (int kk = k0; kk < k; ++kk) {
            double* Ar[3] = {a->Araw[0], a->Araw[1], a->Araw[2]};
            ACSE_TRY(acse_contract(c, Dc, Kh, +1, 1.0, 0, Ar, nullptr, 1));
            k_mask_copy<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, a->Araw[0], a->Araw[1], a->Araw[2], mask,
                                                                  c->opt.act_lo, c->opt.act_hi, a->Am[0], a->Am[1],
                                                                  a->Am[2]);
            AL(c);
            const double* Amc[3] = {a->Am[0], a->Am[1], a->Am[2]};
            double* Uo[3] = {a->Ab[0], a->Ab[1], a->Ab[2]};
            ACSE_TRY(acse_contract(c, Dc, Amc, -1, 0.5, 0, Uo, nullptr, 0));
            k_axpy3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Ab[0], a->Ab[1], a->Ab[2], eps, eps, eps,
                                                              a->Dk[0], a->Dk[1], a->Dk[2]);
            AL(c);
        }
        return ACSE_OK;
    };
    const double* Dc[3] = {a->Dk[0], a->Dk[1], a->Dk[2]};
    for (int b = 0; b < 3; ++b) {
        ACSE_CUDA_TRY(cudaMemsetAsync(a->Db[b], 0, b4, c->stream));
        ACSE_CUDA_TRY(cudaMemsetAsync(a->Kb[b], 0, b4, c->stream));
    }
    // ---- terminal: E = sum_b m_b K_b D_b (m = 1, 4, 1), K = 2 Kh
    ACSE_TRY(load_D(n_steps));
    if (wE != 0.0) {
        k_axpy3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, w.Kh[0], w.Kh[1], w.Kh[2], 2.0 * wE, 8.0 * wE,
                                                          2.0 * wE, a->Db[0], a->Db[1], a->Db[2]);
        AL(c);
        k_axpy3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Dk[0], a->Dk[1], a->Dk[2], wE, 4.0 * wE, wE,
                                                          a->Kb[0], a->Kb[1], a->Kb[2]);
        AL(c);
    }
    if (wN != 0.0) {
        // ||A||^2 = sum_b m_b ||A_b||^2 (before the mask): Ab = 2 wN m_b A_b
        double* Ar[3] = {a->Araw[0], a->Araw[1], a->Araw[2]};
        ACSE_TRY(acse_contract(c, Dc, Kh, +1, 1.0, 0, Ar, nullptr, 1));
        k_scale3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Araw[0], a->Araw[1], a->Araw[2], 2.0 * wN,
                                                           8.0 * wN, 2.0 * wN, a->Am[0], a->Am[1], a->Am[2]);
        AL(c);
        const double* Gb[3] = {a->Am[0], a->Am[1], a->Am[2]};
        ACSE_TRY(vjp_D(c, Kh, +1, 1.0, Gb, a->Db));
        ACSE_TRY(vjp_W(c, Dc, Gb, -1, a->Wb));
        k_axpy3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Wb[0], a->Wb[1], a->Wb[2], 0.5, 0.5, 0.5,
                                                          a->Kb[0], a->Kb[1], a->Kb[2]);
        AL(c);
    }
    // ---- reverse sweep over the steps
    for (int k = n_steps - 1; k >= 0; --k) {
        ACSE_TRY(load_D(k));
        // Dn = Db (identity part of D_{k+1} = D_k + eps U)
        for (int b = 0; b < 3; ++b)
            ACSE_CUDA_TRY(cudaMemcpyAsync(a->Dn[b], a->Db[b], b4, cudaMemcpyDeviceToDevice, c->stream));
        // forward at D_k: A_raw, Am = mask(A_raw), then the update pass (populates its intermediates)
        double* Ar[3] = {a->Araw[0], a->Araw[1], a->Araw[2]};
        ACSE_TRY(acse_contract(c, Dc, Kh, +1, 1.0, 0, Ar, nullptr, 1));
        ACSE_TRY(adj_save(c, false));
        k_mask_copy<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, a->Araw[0], a->Araw[1], a->Araw[2], mask,
                                                              c->opt.act_lo, c->opt.act_hi, a->Am[0], a->Am[1],
                                                              a->Am[2]);
        AL(c);
        const double* Amc[3] = {a->Am[0], a->Am[1], a->Am[2]};
        double* Uo[3] = {a->Ab[0], a->Ab[1], a->Ab[2]};
        ACSE_TRY(acse_contract(c, Dc, Amc, -1, 0.5, 0, Uo, nullptr, 0));
        // U = 1/2 G(Am; D_k); cotangent of U is eps Db
        const double* Ub[3] = {a->Db[0], a->Db[1], a->Db[2]};
        ACSE_TRY(vjp_D(c, Amc, -1, 0.5 * eps, Ub, a->Dn));
        // dL/dAm = 1/2 eps VJP_W(Db); the mask zeroes the same entries of dL/dA
        ACSE_TRY(vjp_W(c, Dc, Ub, +1, a->Wb));
        k_mask_copy<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, a->Wb[0], a->Wb[1], a->Wb[2], mask, c->opt.act_lo,
                                                              c->opt.act_hi, a->Ab[0], a->Ab[1], a->Ab[2]);
        AL(c);
        // Abar = 1/2 eps (masked Wb); through A = G(Kh; D_k): Dn += VJP_D, Kb += 1/2 VJP_W
        k_scale3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Ab[0], a->Ab[1], a->Ab[2], 0.5 * eps, 0.5 * eps,
                                                           0.5 * eps, a->Am[0], a->Am[1], a->Am[2]);
        AL(c);
        ACSE_TRY(adj_save(c, true));
        ACSE_TRY(launch_ph_pack_W(c, Kh, +1));
        const double* Abar[3] = {a->Am[0], a->Am[1], a->Am[2]};
        ACSE_TRY(vjp_D(c, Kh, +1, 1.0, Abar, a->Dn));
        ACSE_TRY(vjp_W(c, Dc, Abar, -1, a->Wb));
        k_axpy3<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(n4, a->Wb[0], a->Wb[1], a->Wb[2], 0.5, 0.5, 0.5,
                                                          a->Kb[0], a->Kb[1], a->Kb[2]);
        AL(c);
        for (int b = 0; b < 3; ++b)
            ACSE_CUDA_TRY(cudaMemcpyAsync(a->Db[b], a->Dn[b], b4, cudaMemcpyDeviceToDevice, c->stream));
    }
    // ---- outputs
    double* dD[3] = {dDaa, dDab, dDbb};
    if (dDaa || dDab || dDbb) {
        k_project_D<<<ad_grid(3 * n4), AD_TPB, 0, c->stream>>>(r, a->Db[0], a->Db[1], a->Db[2], a->Dn[0], a->Dn[1],
                                                              a->Dn[2]);
        AL(c);
        for (int b = 0; b < 3; ++b)
            if (dD[b]) ACSE_CUDA_TRY(cudaMemcpyAsync(dD[b], a->Dn[b], b4, cudaMemcpyDefault, c->stream));
    }
    if (dV) {
        k_adj_K_to_V<<<ad_grid(n4), AD_TPB, 0, c->stream>>>(r, a->Kb[0], a->Kb[1], a->Kb[2], a->Vraw);
        AL(c);
        k_sym_V<<<ad_grid(n4), AD_TPB, 0, c->stream>>>(r, a->Vraw, a->Dn[0]);
        AL(c);
        ACSE_CUDA_TRY(cudaMemcpyAsync(dV, a->Dn[0], b4, cudaMemcpyDefault, c->stream));
    }
    if (dh) {
        k_adj_K_to_h<<<r * r, 64, 0, c->stream>>>(r, 1.0 / (2.0 * (c->N - 1)), a->Kb[0], a->Kb[1], a->Kb[2], a->hraw);
        AL(c);
        k_sym_h<<<(r * r + 127) / 128, 128, 0, c->stream>>>(r, a->hraw, a->Dn[1]);
        AL(c);
        ACSE_CUDA_TRY(cudaMemcpyAsync(dh, a->Dn[1], (size_t)r * r * sizeof(double), cudaMemcpyDefault, c->stream));
    }
    ACSE_CUDA_TRY(cudaStreamSynchronize(c->stream));
    return ACSE_OK;
}
