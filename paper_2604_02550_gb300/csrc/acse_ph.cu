// The particle-hole products of a contraction pass on symmetrised index pairs (FP64 and Ozaki paths).
//
// With V5[(k,q)][(i,l)] = sum_{p,t} W^{kp}_{qt} M^{ip}_{lt} (spin-conserving sector: (k,q) of one spin, (p,t) of
// either, (i,l) of one spin), the operand of B is X5[(k,j)][(i,l)] = sum_q 1D^j_q V5[(k,q)][(i,l)] -- the
// transformation by 1D commutes with the sum over (p,t), so it may follow the O(r^6) product instead of
// preceding it, and then the product has a symmetry that halves both its output and its sum:
//     M^{ip}_{lt} = M^{lt}_{ip} (Hermitian) and = M^{pi}_{tl}  =>  M[(i,l)][(p,t)] = M[(l,i)][(t,p)],
//     W[(k,q)][(p,t)] = s W[(q,k)][(t,p)]  for a pair-Hermitian (s = +1) or anti-Hermitian (s = -1) W.
// Split over the exchange of (p,t): W+- = (W[.][(p,t)] +- W[.][(t,p)]) / 2, M+- likewise.  M+ is symmetric in
// (i,l) and M- antisymmetric; W+ is symmetric in (k,q) and W- antisymmetric for s = +1, the other way round
// for s = -1.  The cross terms vanish, so
//     V5 = V1 + V2,   V1 = 2 sum_{p<t} W+ M+ + sum_{p=t} W M,   V2 = 2 sum_{p<t} W- M-,
// two products on pairs a <= b (S = r(r+1)/2 per spin) and a < b (P = r(r-1)/2): 4 r^6 flop in place of the
// 16 r^6 of the full (2r^2)^3 product.  The spin-flip sectors are each other's image,
// V5f2[(k,q)][(i,l)] = s V5f1[(q,k)][(l,i)], so one of them is multiplied: 2 r^6 in place of 4 r^6.
//
// W always has that symmetry, a 2-RDM D does, but the caller's D (sampled, truncated, one-sided) need not. M+ then
// also has a part that is antisymmetric in (i,l), M- one that is symmetric, and the second flip is a product of its
// own: V1, V2 get those columns too (2P and 2S of them) by three more products, 6 r^6, which every context holds and
// runs where k_ph_pack_asym finds max |D - D^T| > 2^-47 max |D| in the D being prepared (`asym`, on the device: no
// read-back, and a captured step decides anew on every replay).  That bound is 32 units in the last place of the
// largest entry: a D that is Hermitian but for the rounding of an orbital transformation (1.2 2^-50 measured at r = 48)
// stays below it, and what is dropped of its asymmetry is below the rounding of its own entries.
//
// Kernels here: the packing of both operands and the expansion of V1, V2, V5f1 into the full V5 (the FP64 pipe two
// thirds busy at r = 32, DRAM a tenth; at r = 48 93 us a pack and 116 us for the expansion's 380 MB), the
// diagonal sums behind w, and the transformation by 1D on the CUDA cores (an Ozaki context runs it on the tensor
// cores where acse_zoz.cu applies).
#include <type_traits>

#include "acse_internal.h"
#include "dfloat.cuh"

// ------------------------------------------------------------------------------- packing
// plus[(K,{kq})][(P',{p<=t})] = f (x + x') (x at p = t), minus[(K,{kq})][(P',{p<t})] = f (x - x'), with
// x = T^{kp}_{qt}, x' = T^{kt}_{qp}, spins K of (k,q) and P' of (p,t); the rows of `plus` run over k <= q and
// those of `minus` over k < q (plusS = 1), or the other way round (plusS = 0).  flip[(k,q)][(p,t)] =
// T_ab[k][p][t][q].  W takes f = 1/2; M takes f = 1, the 2 of the halved sum over (p,t) included.
// Block (K, P', {k<=q}): the r x r slab of (p,t) goes through shared memory, both rows leave coalesced (the
// b,a slab is read at stride r: its sectors are shared by the blocks of neighbouring q).  Block (k,p) of the
// flips: an r x r transposition in shared memory.
struct PhPack {
    const double* src[3];
    double* plus;
    double* minus;
    double* flip;
    int r, plusS;
    double f;
};

__global__ void __launch_bounds__(256) k_ph_pack(const __grid_constant__ PhPack a) {
    extern __shared__ double ph_sm[];   // [r][r + 1]
    const int r = a.r, ld = r + 1, S = r * (r + 1) / 2, P = r * (r - 1) / 2;
    const size_t R2 = (size_t)r * r, r3 = R2 * r;
    if ((int)blockIdx.x < 4 * S) {
        const int kp = (int)blockIdx.x / S, u = (int)blockIdx.x - kp * S, K = kp >> 1, Q = kp & 1;
        int k, q;
        ps_unpair(r, u, k, q);
        const double* src = a.src[K == Q ? 2 * K : 1];
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int p = e / r, t = e - p * r;
            ph_sm[p * ld + t] = (K == 1 && Q == 0) ? src[p * r3 + k * R2 + (size_t)t * r + q]
                                                   : src[k * r3 + p * R2 + (size_t)q * r + t];
        }
        __syncthreads();
        const int rowS = K * S + u, rowA = k < q ? K * P + pk_pair(r, k, q) : -1;
        const int rp = a.plusS ? rowS : rowA, rm = a.plusS ? rowA : rowS;
        double* op = a.plus + (size_t)max(rp, 0) * 2 * S + (size_t)Q * S;
        double* om = a.minus + (size_t)max(rm, 0) * 2 * P + (size_t)Q * P;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int p = e / r, t = e - p * r;
            if (t < p) continue;
            const double x = ph_sm[p * ld + t], y = ph_sm[t * ld + p];
            if (rp >= 0) op[ps_pair(r, p, t)] = p < t ? a.f * (x + y) : x;
            if (rm >= 0 && p < t) om[pk_pair(r, p, t)] = a.f * (x - y);
        }
    } else {
        const int kp = (int)blockIdx.x - 4 * S, k = kp / r, p = kp - k * r;
        const double* src = a.src[1] + k * r3 + p * R2;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) ph_sm[(e / r) * ld + e % r] = src[e];   // [t][q]
        __syncthreads();
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int q = e / r, t = e - q * r;
            a.flip[((size_t)k * r + q) * R2 + (size_t)p * r + t] = ph_sm[t * ld + q];
        }
    }
}

static int launch_ph_pack(acse_ctx* c, const double* const T[3], double* plus, double* minus, double* flip, int plusS,
                          double f) {
    const int r = c->r;
    PhPack a;
    for (int s = 0; s < 3; ++s) a.src[s] = T[s];
    a.plus = plus;
    a.minus = minus;
    a.flip = flip;
    a.r = r;
    a.plusS = plusS;
    a.f = f;
    const int blocks = 4 * (r * (r + 1) / 2) + r * r;
    k_ph_pack<<<blocks, 256, (size_t)r * (r + 1) * sizeof(double), c->stream>>>(a);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// Is D pair-Hermitian (the maxima of k_build_M), for the kernels behind this one in `asym`; and where it is not (otherwise
// the blocks leave at once, 1.6 us): M+ and M- with x and x' averaged over
// the exchange of k and q, half their differences in 2P more rows of M+ (k < q) and 2S more of M- (k <= q), and
// flip2[(k,q)][(p,t)] = M_ab[t][q][k][p], the second flip with both its pairs exchanged (for a Hermitian M the first).
// Read straight from global memory: the rare case.
struct PhPackAsym {
    const double* src[3];
    double* plus;
    double* minus;
    double* flip2;
    const unsigned long long* dmax;
    int* asym;
    int r;
};

__global__ void __launch_bounds__(256) k_ph_pack_asym(const __grid_constant__ PhPackAsym a) {
    const double mx = __longlong_as_double((long long)a.dmax[0]), ma = __longlong_as_double((long long)a.dmax[1]);
    const bool sym = ma <= mx * 0x1p-47;   // NaN: not
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.asym = sym ? 0 : 1;
    if (sym) return;
    const int r = a.r, S = r * (r + 1) / 2, P = r * (r - 1) / 2;
    const size_t R2 = (size_t)r * r, r3 = R2 * r;
    for (int w = blockIdx.x; w < 4 * S + (int)R2; w += gridDim.x) {
        const int kp = w < 4 * S ? w / S : 0, u = w - kp * S, K = kp >> 1, Q = kp & 1;
        int k, q;
        if (w < 4 * S) {
            ps_unpair(r, u, k, q);
        } else {
            k = (w - 4 * S) / r;
            q = w - 4 * S - k * r;
        }
        const double* src = a.src[w < 4 * S && K == Q ? 2 * K : 1];
        // T^{kp}_{qt} of the spins K of (k,q) and Q of (p,t)
        auto at = [&](int k, int q, int p, int t) {
            return K == 1 && Q == 0 ? src[p * r3 + k * R2 + (size_t)t * r + q] : src[k * r3 + p * R2 + (size_t)q * r + t];
        };
        const int rowS = K * S + u, rowA = k < q ? K * P + pk_pair(r, k, q) : -1;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int p = e / r, t = e - p * r;
            if (w >= 4 * S) {
                a.flip2[((size_t)k * r + q) * R2 + e] = src[t * r3 + q * R2 + (size_t)k * r + p];
                continue;
            }
            if (t < p) continue;
            const double x1 = at(k, q, p, t), x2 = at(q, k, p, t), y1 = at(k, q, t, p), y2 = at(q, k, t, p);
            const double x = 0.5 * (x1 + x2), y = 0.5 * (y1 + y2), dx = 0.5 * (x1 - x2), dy = 0.5 * (y1 - y2);
            const size_t cs = (size_t)Q * S + ps_pair(r, p, t), ca = (size_t)Q * P + (p < t ? pk_pair(r, p, t) : 0);
            a.plus[(size_t)rowS * 2 * S + cs] = p < t ? x + y : x;
            if (p < t) a.minus[((size_t)2 * P + rowS) * 2 * P + ca] = x - y;
            if (rowA < 0) continue;
            a.plus[((size_t)2 * S + rowA) * 2 * S + cs] = p < t ? dx + dy : dx;
            if (p < t) a.minus[(size_t)rowA * 2 * P + ca] = dx - dy;
        }
    }
}

int launch_ph_pack_M(acse_ctx* c) {
    Work& w = c->w;
    ACSE_TRY(launch_ph_pack(c, w.M, w.Mp, w.Mm, w.Mf1, 1, 1.0));
    PhPackAsym a;
    for (int s = 0; s < 3; ++s) a.src[s] = w.M[s];
    a.plus = w.Mp;
    a.minus = w.Mm;
    a.flip2 = w.Mf2;
    a.dmax = w.dmax;
    a.asym = w.asym;
    a.r = c->r;
    k_ph_pack_asym<<<152 * 2, 256, 0, c->stream>>>(a);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

int launch_ph_pack_W(acse_ctx* c, const double* const W[3], int sW) {
    Work& w = c->w;
    return launch_ph_pack(c, W, w.Wp, w.Wm, w.Wf1, sW > 0, 0.5);
}

// ------------------------------------------------------------------------------ expansion
// V5 (rows (K,k,q), columns (I,i,l)) = V1 + V2 from the products on pairs, by the symmetries above: row (k,q),
// k < q, is V1 + sg(i,l) V2 (sg = 1 for i < l, -1 for i > l, 0 for i = l), and row (q,k) s times V1 - sg V2
// ... (s = +1: V1 is even and V2 odd in the exchange of k and q, s = -1: the other way round).  The diagonal
// rows k = q have the even part alone.  V5f2[(k,q)][(i,l)] = s V5f1[(q,k)][(l,i)].
// Rows of V1: the 2S pairs i <= l, and with asym the 2P pairs i < l of its part antisymmetric in (i,l); of V2: the 2P
// pairs i < l, and with asym the 2S pairs i <= l of its symmetric part.
struct PhUnpack {
    const double* V1;
    const double* V2;
    const double* f1;
    const double* g2;   // with asym: the product behind the second flip, in the place of f1
    const int* asym;
    double* V;
    double* f2;
    int r, s;
};

__global__ void __launch_bounds__(256) k_ph_unpack(const __grid_constant__ PhUnpack a) {
    extern __shared__ double ph_sm[];   // 2S + 2P = 2 r^2 doubles
    const int r = a.r, S = r * (r + 1) / 2, P = r * (r - 1) / 2;
    const size_t R2 = (size_t)r * r;
    const bool gen = *a.asym;
    if ((int)blockIdx.x < 2 * S) {
        const int K = (int)blockIdx.x / S, u = (int)blockIdx.x - K * S;
        int k, q;
        ps_unpair(r, u, k, q);
        const int rowS = K * S + u, rowA = k < q ? K * P + pk_pair(r, k, q) : -1;
        const int r1 = a.s > 0 ? rowS : rowA, r2 = a.s > 0 ? rowA : rowS;
        double* v1 = ph_sm;
        double* v2 = ph_sm + 2 * S;
        const double* p1 = a.V1 + (size_t)max(r1, 0) * 2 * R2;
        const double* p2 = a.V2 + (size_t)max(r2, 0) * 2 * R2;
        for (int e = threadIdx.x; e < 2 * S; e += blockDim.x) v1[e] = r1 >= 0 ? p1[e] : 0.0;
        for (int e = threadIdx.x; e < 2 * P; e += blockDim.x) v2[e] = r2 >= 0 ? p2[e] : 0.0;
        __syncthreads();
        double* o1 = a.V + ((size_t)K * R2 + (size_t)k * r + q) * 2 * R2;
        double* o2 = a.V + ((size_t)K * R2 + (size_t)q * r + k) * 2 * R2;
        for (int e = threadIdx.x; e < 2 * (int)R2; e += blockDim.x) {
            const int I = e >= (int)R2, c = e - I * (int)R2, i = c / r, l = c - i * r;
            const int us = I * S + (i <= l ? ps_pair(r, i, l) : ps_pair(r, l, i));
            double x = v1[us], y = 0.0;
            if (i < l) y = v2[I * P + pk_pair(r, i, l)];
            else if (i > l) y = -v2[I * P + pk_pair(r, l, i)];
            if (gen) {
                if (r1 >= 0 && i != l) x += i < l ? p1[2 * S + I * P + pk_pair(r, i, l)] : -p1[2 * S + I * P + pk_pair(r, l, i)];
                if (r2 >= 0) y += p2[2 * P + us];
            }
            o1[e] = x + y;
            if (k < q) o2[e] = a.s > 0 ? x - y : y - x;
        }
    } else {
        const int kq = (int)blockIdx.x - 2 * S, k = kq / r, q = kq - k * r;
        const double* src = (gen ? a.g2 : a.f1) + ((size_t)q * r + k) * R2;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) ph_sm[e] = src[e];
        __syncthreads();
        const double s = (double)a.s;
        for (int e = threadIdx.x; e < (int)R2; e += blockDim.x) {
            const int i = e / r, l = e - i * r;
            a.f2[(size_t)kq * R2 + e] = s * ph_sm[l * r + i];
        }
    }
}

static int launch_ph_unpack(acse_ctx* c, int sW) {
    const int r = c->r;
    Work& w = c->w;
    PhUnpack a;
    a.V1 = w.V1;
    a.V2 = ph_V2(c, sW);
    a.f1 = w.V5f1;
    a.g2 = w.Vf2;
    a.asym = w.asym;
    a.V = w.V5d;
    a.f2 = w.V5f2;
    a.r = r;
    a.s = sW;
    k_ph_unpack<<<r * (r + 1) + r * r, 256, 2 * (size_t)r * r * sizeof(double), c->stream>>>(a);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// ------------------------------------------------------------------------ same-spin pairs
// Same-spin pair GEMMs on packed pairs (as on the split path): in the aa and bb sectors the rows (ij),
// the columns (kp) and the contraction (rs) of [M; D] W^T are antisymmetric pairs, so those GEMMs run
// on pairs i < j only (P = r(r-1)/2; alpha 2 for the halved (rs) sum) and k_pair_unpack rebuilds the
// full X and Y rows by antisymmetry (pairs numbered by pk_pair).
//
// X_s, Y_s (s = aa, bb; r^2 x r^2 FP64) from the packed [X; Y] (2P x P): one block per output row, the
// packed source row staged in shared memory, the full row written two columns at a time.  The pass reads the
// rows i < j only (pmap set: P rows); the adjoint sums over every row (pmap null: r^2 rows).
__global__ void __launch_bounds__(256) k_pair_unpack(int r, const int* __restrict__ pmap, const double* __restrict__ Cp0,
                                                     const double* __restrict__ Cp2, double* X0, double* Y0, double* X2,
                                                     double* Y2) {
    __shared__ double srow[ACSE_MAX_R * (ACSE_MAX_R - 1) / 2];
    const int R2 = r * r, P = r * (r - 1) / 2, rows = pmap ? P : R2;
    const int sec = blockIdx.x / (2 * rows);
    const int row = blockIdx.x - sec * 2 * rows;
    const int part = row / rows, u = row - part * rows, ij = pmap ? pmap[u] : u, i = ij / r, j = ij - i * r;
    double* dst = (sec == 0 ? (part ? Y0 : X0) : (part ? Y2 : X2)) + (size_t)ij * R2;
    if (i == j) {   // block-uniform
        for (int c = threadIdx.x; c < R2; c += blockDim.x) dst[c] = 0.0;
        return;
    }
    const double si = i < j ? 1.0 : -1.0;
    const double* src = (sec == 0 ? Cp0 : Cp2) + (size_t)(part * P + (i < j ? pk_pair(r, i, j) : pk_pair(r, j, i))) * P;
    for (int e = threadIdx.x; e < P; e += blockDim.x) srow[e] = si * src[e];
    __syncthreads();
    auto val = [&](int k, int q) { return k == q ? 0.0 : (k < q ? srow[pk_pair(r, k, q)] : -srow[pk_pair(r, q, k)]); };
    if ((R2 & 1) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
        for (int g = threadIdx.x; g < R2 / 2; g += blockDim.x) {
            int k = (2 * g) / r, q = 2 * g - k * r;
            const double v0 = val(k, q);
            if (++q == r) { q = 0; ++k; }
            reinterpret_cast<double2*>(dst)[g] = make_double2(v0, val(k, q));
        }
    } else {
        for (int c = threadIdx.x; c < R2; c += blockDim.x) dst[c] = val(c / r, c - (c / r) * r);
    }
}

int launch_pair_unpack(acse_ctx* c) {
    Work& w = c->w;
    const int r = c->r;
    const int* pmap = c->in_adjoint ? nullptr : w.pmap;
    k_pair_unpack<<<2 * 2 * (pmap ? r * (r - 1) / 2 : r * r), 256, 0, c->stream>>>(r, pmap, w.Cp[0], w.Cp[1], w.X[0],
                                                                                  w.Y[0], w.X[2], w.Y[2]);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// -------------------------------------------------------- products of the pairs (CUDA cores)
// Eight classes of r x r x r products per pair ij, out_c[ij][a][b] = sum_x T_c(a, x) G_c[b][x] (bit c of tt, gt: T, G
// read transposed; bit c of tri: the pairs i < j only).  FP64 contexts, and Ozaki contexts where the digit kernel
// does not apply (C: double, or the double-float pair where acse_use_dfl).  Block: one class, nij pairs, both operands in shared
// memory as [x][.]; the MT x MT tiles of all pairs are dealt out to full warps -- a DFMA holds the FP64 pipe 16
// cycles however many lanes are active, and at r = 24 one 4 x 4 tile a thread left 28 of 64 lanes idle -- with
// nij chosen on the host so that the last round of tiles is nearly full.  r = 24, FP64: 123 us for the six pair-types'
// worth of products a pass runs (1.05 TFLOP/s), where the B kernel that formed them itself took 279 us.
struct PairRows {
    const double* T[8];
    const double* G[8];
    double* out[8];
    const int* pmap;
    unsigned tt, gt, tri;
    int start[9];   // first block of each class
    int r, nij;
};

template <typename C, int MT>
__global__ void __launch_bounds__(256) k_pair_rows(const __grid_constant__ PairRows a) {
    extern __shared__ __align__(16) unsigned char ph_raw[];
    const int r = a.r, rp = (r + MT - 1) / MT * MT, R2 = r * r, nt = rp / MT, nt2 = nt * nt, op = r * rp;
    int c = 0;
    while (c < 7 && a.start[c + 1] <= (int)blockIdx.x) ++c;
    const bool tri = (a.tri >> c) & 1, tt = (a.tt >> c) & 1, gt = (a.gt >> c) & 1;
    const int u0 = ((int)blockIdx.x - a.start[c]) * a.nij, n = min(a.nij, (tri ? r * (r - 1) / 2 : R2) - u0);
    C* Gs = (C*)ph_raw;   // [x][b]
    C* Ts = Gs + op;      // [pair][x][a]
    if (rp != r) {
        for (int e = threadIdx.x; e < (1 + n) * op; e += blockDim.x) Gs[e] = tconv<C>(0.0);
        __syncthreads();
    }
    for (int e = threadIdx.x; e < R2; e += blockDim.x) {
        const int u = e / r, v = e - u * r;
        Gs[gt ? u * rp + v : v * rp + u] = tconv<C>(a.G[c][e]);   // [b = u][x = v], or [x = u][b = v]
    }
    for (int f = threadIdx.x; f < n * R2; f += blockDim.x) {
        const int it = f / R2, e = f - it * R2, u = e / r, v = e - u * r;
        const int ij = tri ? a.pmap[u0 + it] : u0 + it;
        Ts[it * op + (tt ? u * rp + v : v * rp + u)] = tconv<C>(a.T[c][(size_t)ij * R2 + e]);
    }
    __syncthreads();
    for (int g = threadIdx.x; g < n * nt2; g += blockDim.x) {
        const int it = g / nt2, tile = g - it * nt2, a0 = (tile / nt) * MT, b0 = (tile % nt) * MT;
        const C* T = Ts + it * op + a0;
        const C* G = Gs + b0;
        C acc[MT][MT];
#pragma unroll
        for (int u = 0; u < MT; ++u)
#pragma unroll
            for (int v = 0; v < MT; ++v) acc[u][v] = tconv<C>(0.0);
#pragma unroll 4
        for (int x = 0; x < r; ++x) {
            C p[MT], q[MT];
#pragma unroll
            for (int u = 0; u < MT; ++u) {
                p[u] = T[x * rp + u];
                q[u] = G[x * rp + u];
            }
#pragma unroll
            for (int u = 0; u < MT; ++u)
#pragma unroll
                for (int v = 0; v < MT; ++v) tmac(acc[u][v], p[u], q[v]);
        }
        const int ij = tri ? a.pmap[u0 + it] : u0 + it;
        double* out = a.out[c] + (size_t)ij * R2;
#pragma unroll
        for (int u = 0; u < MT; ++u)
#pragma unroll
            for (int v = 0; v < MT; ++v)
                if (a0 + u < r && b0 + v < r) out[(a0 + u) * r + b0 + v] = (double)acc[u][v];
    }
}

#define PR_SMEM (96 * 1024)   // two blocks an SM

// nij: fewest idle lanes over the rounds of 256 tiles, within PR_SMEM; the smallest such count.
static int pair_rows_nij(int r, int mt) {
    const int rp = (r + mt - 1) / mt * mt, nt2 = (rp / mt) * (rp / mt);
    int best = 1;
    double bu = 0.0;
    for (int n = 1; n <= 32 && (size_t)(1 + n) * r * rp * sizeof(double) <= PR_SMEM; ++n) {
        const double u = (double)n * nt2 / ((n * nt2 + 255) / 256 * 256);
        if (u > bu + 0.01) {
            bu = u;
            best = n;
        }
    }
    return best;
}

int launch_pair_rows(acse_ctx* c, const double* const T[8], unsigned tt, const double* const G[8], unsigned gt, unsigned tri,
                     double* const out[8]) {
    const int st = launch_rows_oz(c, T, tt, G, gt, tri, out);
    if (st != ACSE_ERR_UNSUPPORTED) return st;
    const bool df = acse_use_dfl(c);
    const int r = c->r, mt = df ? 4 : 2, rp = (r + mt - 1) / mt * mt;
    PairRows a;
    for (int k = 0; k < 8; ++k) {
        a.T[k] = T[k];
        a.G[k] = G[k];
        a.out[k] = out[k];
    }
    a.pmap = c->w.pmap;
    a.tt = tt;
    a.gt = gt;
    a.tri = tri;
    a.r = r;
    a.nij = pair_rows_nij(r, mt);
    a.start[0] = 0;
    for (int k = 0; k < 8; ++k) {
        const int items = (tri >> k) & 1 ? r * (r - 1) / 2 : r * r;
        a.start[k + 1] = a.start[k] + (items + a.nij - 1) / a.nij;
    }
    const size_t sm = (size_t)(1 + a.nij) * r * rp * sizeof(double);
    if (df) k_pair_rows<dfl, 4><<<a.start[8], 256, sm, c->stream>>>(a);
    else k_pair_rows<double, 2><<<a.start[8], 256, sm, c->stream>>>(a);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// The two products of every B spin type into w.bx64 (same-spin types on the pairs i < j):
//     class 2 t:      x1[k][l] = sum_q X_ij[k][q] 1D[q][l]       (type 3: X_ij transposed)
//     class 2 t + 1:  x2^T[l][k] = sum_p M_ij[l][p] w[k][p]      (type 2: M_ij transposed)
int launch_Bx(acse_ctx* c) {
    Work& w = c->w;
    const int R2 = c->r * c->r;
    const double *ga = w.gam, *gb = w.gam + R2, *wa = w.w, *wb = w.w + R2;
    const double* T[8] = {w.X[0], w.M[0], w.X[2], w.M[2], w.X[1], w.M[1], w.X[1], w.M[1]};
    const double* G[8] = {ga, wa, gb, wb, gb, wa, ga, wb};
    return launch_pair_rows(c, T, 1u << 6 | 1u << 5, G, 0x55u, 0x0Fu, w.bx64);
}

// ------------------------------------------------------------------------------------- w
// diag[slot][k][p][s], whose sum over p gives w (k_w_from_diag):
//   slot 0: sum_q Waa[k][p][q][s] ga[p][q]    slot 1: sum_q Wbb[k][p][q][s] gb[p][q]
//   slot 2: sum_q Wab[k][p][s][q] gb[p][q]    slot 3: sum_q Wab[p][k][q][s] ga[p][q]
__global__ void __launch_bounds__(64) k_ph_w_diag(int r, const double* __restrict__ Waa, const double* __restrict__ Wab,
                                                  const double* __restrict__ Wbb, const double* __restrict__ gam,
                                                  double* __restrict__ diag) {
    const int slot = (int)blockIdx.x / (r * r), kp = (int)blockIdx.x - slot * r * r, k = kp / r, p = kp - k * r;
    const int s = threadIdx.x;
    if (s >= r) return;
    const size_t R2 = (size_t)r * r, r3 = R2 * r;
    const double* g = gam + ((slot == 1 || slot == 2) ? R2 : 0) + (size_t)p * r;
    const double* w = slot == 0 ? Waa + k * r3 + p * R2 : slot == 1 ? Wbb + k * r3 + p * R2
                      : slot == 2 ? Wab + k * r3 + p * R2 + (size_t)s * r : Wab + p * r3 + k * R2;
    double acc = 0.0;
    if (slot == 2)
        for (int q = 0; q < r; ++q) acc = fma(g[q], w[q], acc);
    else
        for (int q = 0; q < r; ++q) acc = fma(g[q], w[(size_t)q * r + s], acc);
    diag[(size_t)blockIdx.x * r + s] = acc;
}

int launch_ph_w_diag(acse_ctx* c, const double* const W[3]) {
    const int r = c->r;
    k_ph_w_diag<<<4 * r * r, 64, 0, c->stream>>>(r, W[0], W[1], W[2], c->w.gam, c->w.zdiag);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// ------------------------------------------------------- transformation by 1D (CUDA cores)
// out[(K,k,j)][(I,i,l)] = sum_q g_K[j][q] in[(K,k,q)][(I,i,l)] (trans: g_K[q][j]) for the six sectors t:
// 0-3 the spin blocks (K, I) of the 2r^2 x 2r^2 array, 4 and 5 the two flips (1D of beta, of alpha).
// Block (t, k, 64 columns): the columns' r rows and 1D sit in shared memory, each thread owns a 4 x 4 tile.
// C: double (bound by the DFMA pipe, 6 r^5), or the double-float pair where acse_use_dfl.
#define PHT_COLS 64

struct PhXform {
    const double* in[3];   // spin blocks, flip 1, flip 2
    double* out[3];
    const double* gam;
    int r, trans;
};

template <typename C>
__global__ void __launch_bounds__(256) k_ph_xform(const __grid_constant__ PhXform a) {
    extern __shared__ __align__(16) unsigned char ph_raw[];
    const int r = a.r, rp = (r + 3) & ~3, R2 = r * r, nch = (R2 + PHT_COLS - 1) / PHT_COLS;
    C* g = (C*)ph_raw;                      // [q][j], pitch rp
    C* v = g + (size_t)r * rp;              // [q][64]
    const int t = (int)blockIdx.x / (r * nch), rem = (int)blockIdx.x - t * r * nch, k = rem / nch;
    const int c0 = (rem - k * nch) * PHT_COLS;
    const int f = t < 4 ? 0 : t - 3, K = t < 4 ? t >> 1 : t == 4 ? 1 : 0;
    const size_t ld = t < 4 ? 2 * (size_t)R2 : (size_t)R2;
    const size_t base = (t < 4 ? (size_t)K * R2 * ld + (size_t)(t & 1) * R2 : 0) + (size_t)k * r * ld + c0;
    const double* in = a.in[f] + base;
    const double* gam = a.gam + (size_t)K * R2;
    for (int e = threadIdx.x; e < r * rp; e += blockDim.x) {
        const int q = e / rp, j = e - q * rp;
        g[e] = tconv<C>(j < r ? (a.trans ? gam[q * r + j] : gam[j * r + q]) : 0.0);
    }
    for (int e = threadIdx.x; e < r * PHT_COLS; e += blockDim.x) {
        const int q = e / PHT_COLS, c = e - q * PHT_COLS;
        v[e] = tconv<C>(c0 + c < R2 ? in[(size_t)q * ld + c] : 0.0);
    }
    __syncthreads();
    const int j0 = (threadIdx.x / (PHT_COLS / 4)) * 4, cc = (threadIdx.x % (PHT_COLS / 4)) * 4;
    if (j0 >= r) return;
    C acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[u][x] = tconv<C>(0.0);
#pragma unroll 2
    for (int q = 0; q < r; ++q) {
        C ga[4], vb[4];
        ld4(g + (size_t)q * rp + j0, ga);
        ld4(v + (size_t)q * PHT_COLS + cc, vb);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int x = 0; x < 4; ++x) tmac(acc[u][x], ga[u], vb[x]);
    }
    double* out = a.out[f] + base;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (j0 + u < r)
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (c0 + cc + x < R2) out[(size_t)(j0 + u) * ld + cc + x] = (double)acc[u][x];
}

static size_t ph_xform_smem(int r) { return (size_t)r * (((r + 3) & ~3) + PHT_COLS) * sizeof(double); }

int launch_ph_xform(acse_ctx* c, const double* const in[3], double* const out[3], int trans) {
    if (c->oz) {
        const int s = launch_xform_oz(c, in, out, trans);
        if (s != ACSE_ERR_UNSUPPORTED) return s;
    }
    const int r = c->r, nch = (r * r + PHT_COLS - 1) / PHT_COLS;
    PhXform a;
    for (int f = 0; f < 3; ++f) {
        a.in[f] = in[f];
        a.out[f] = out[f];
    }
    a.gam = c->w.gam;
    a.r = r;
    a.trans = trans;
    const int threads = (((r + 3) / 4) * (PHT_COLS / 4) + 31) / 32 * 32;
    if (acse_use_dfl(c)) k_ph_xform<dfl><<<6 * r * nch, threads, ph_xform_smem(r), c->stream>>>(a);
    else k_ph_xform<double><<<6 * r * nch, threads, ph_xform_smem(r), c->stream>>>(a);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

// X5 of the pass from its products V1, V2 and V5f1.
int launch_ph_finish(acse_ctx* c, int sW) {
    Work& w = c->w;
    ACSE_TRY(launch_ph_unpack(c, sW));
    const double* in[3] = {w.V5d, w.V5f1, w.V5f2};
    double* out[3] = {w.X5d, w.X5f1, w.X5f2};
    return launch_ph_xform(c, in, out, 0);
}

int ph_set_attrs() {
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_pair_rows<double, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, PR_SMEM));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_pair_rows<dfl, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, PR_SMEM));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_ph_unpack, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       2 * ACSE_MAX_R * ACSE_MAX_R * (int)sizeof(double)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_ph_xform<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ph_xform_smem(ACSE_MAX_R)));
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_ph_xform<dfl>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ph_xform_smem(ACSE_MAX_R)));
    return ACSE_OK;
}
