// The O(r^5) products of an FP64-accurate (Ozaki) context on the tensor cores: products of many r-element rows
// with an r x r matrix,
//     out[m][n] = sum_q A[m][q] G[n][q],
// by the error-free splitting of the Ozaki scheme (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59, 2012).
// Two uses: the transformation of the particle-hole product by 1D, X5[(k,j)][c] = sum_q 1D^j_q V5[(k,q)][c]
// (acse_ph.cu: rows m = columns c of one sector and k), and the products of every pair (i, j) with 1D and w
// (the x1 and x2 of the B kernel, and the adjoint's: rows (ij, k) of r^4 arrays, eight classes).
//
// Every row of A and of G gets a power-of-two scale 2^e (|x| 2^-e < 1/2 over the row) and each element the
// fixed-point value X = round(x 2^(8D + 1 - e)), |X| < 2^8D, cut into D base-256 digits (most significant first): the
// leading one within -256 .. 256, the others balanced, -128 .. 127 (exact in bf16).  D = ceil(6 S / 8) digits hold at
// least the 6 S bits of oz_slices = S below the row's leading one.  The products of one level L = s + t <= D + 2 are
// accumulated in FP32 in their own TMEM accumulator: a level holds at most D <= 6 products of K <= 64 terms of
// magnitude <= 2^14, twice that in the two with one leading digit and 2^16 in that of two, so it stays within 2^23
// and every level sum is an exact integer.  The epilogue adds the levels in int64 (sum_L v_L 2^(8 (D + 1 - L)), below
// 2^63, the last level rounded to that unit) and rounds once to FP64, scaled by 2^(e_m + e_n - 8 (D + 1) - 2).  What is
// left is the fixed-point rounding, 2^-(8D + 1) of the row scales: with one bit less (the leading digit balanced like
// the others) that was the larger part of the error at ragged r, U of a step at r = 20 1.39e-14 rms against 64 bits,
// where double-float products gave 1.2e-14 and this gives 9.3e-15.  With the levels up to D + 1 only, the dropped level
// D + 2 (D - 1 products a term) was the larger error (r = 30 residual 7.5e-14 against 3.4e-14 of double-float products).
// Against eight base-64 digits: 26 digit products in place of 36, seven levels in place of eight, and a digit is a byte
// of X + 128 (1 + 256 + ...): a permute and half a packed FADD.
//
// One block per SM, warp-specialised (the phases of a tile of 128 rows one after another behind block barriers
// took 20 us a tile): eight producer warps load the rows of the next tile and write its digits into one of two
// shared-memory buffers, one thread issues the MMAs (M = 128, N up to 256), eight epilogue warps read
// the levels, hand TMEM back and finish the integers while the next tile's MMAs run.  The operands sit in the
// unswizzled K-major layout (8 x 16-byte core matrices; chunk kc of eight K elements at kc * rows * 16 bytes), which
// stores only the RP used elements of a row -- with 128-byte rows two buffers of six digits would not fit -- and
// takes a thread's 16-byte chunks without bank conflicts.  K is permuted so that two adjacent threads share a
// row's loads in 32-byte sectors: element q = 16 (kc >> 1) + 4 (j >> 1) + 2 (kc & 1) + (j & 1) is element j of chunk kc.
// r = 48: 283 us for the eight classes, 290 us for the transformation (a block's phases one after another, six-bit
// digits: 906 and 679 us); r = 30: 56 and 55 us (in double-float 400 us of the B kernel and 104 us).  Bound by the ALU pipe (the
// digits and the int64 normalisation, about half busy) and the chain TMEM read - MMA - TMEM read; HBM at 2 TB/s.
// Every wait is bounded, and on expiry the kernel raises the device flag and stops.
//
// Used for S <= 8 and r >= 16; more slices take the double-float kernels of acse_ph.cu, smaller r the FP64 ones, which
// leave the rounding of the GEMMs alone in the error (U at r = 12: 7.2e-15 rms, digits of eight bits 1.28e-14,
// double-float 7.7e-15; a residual at r = 15 takes 12 us longer).
#include <cuda_bf16.h>

#include "acse_internal.h"
#include "oz_arith.cuh"
#include "tc_ptx.cuh"

#define RZ_PW 8                              // producer warps
#define RZ_EW 8                              // epilogue warps
#define RZ_THREADS (32 * (1 + RZ_PW + RZ_EW))
#define RZ_DMAX 6                            // digits
#define RZ_SMAX 8                            // slices: ceil(6 S / 8) <= RZ_DMAX
#define RZ_ESLOT 4                           // slots of the row scales (see the producer)
#define RZ_WAIT_NS 4000000000ull

struct RowsArgs {
    const double* A[8];     // MODE 0: class c, rows ij of r^2, the operand of row (ij, a), element q at [a][q] ...
                            // MODE 1: the spin blocks (2r^2 x 2r^2), flip 1, flip 2 (r^2 x r^2)
    const double* G[8];     // MODE 0: r x r operand of class c, G[n][q] ...; MODE 1: 1D of alpha, of beta
    double* out[8];
    unsigned tt, gt;        // ... or transposed (bit c): A at [q][a], G[q][n]
    int sel[8];             // MODE 0: classes with the same G (and transposition) share a number
    unsigned tri;           // MODE 0, bit c: the pairs i < j only (numbered through pmap)
    const int* pmap;
    int r, D;
    int start[9];           // MODE 0: first tile of each class
    int tpg;                // MODE 1: tiles per group (sector, k)
    int ntiles;
    int* err;
};

// Row scale from the upper word of the largest magnitude (non-negative doubles order like their bits): e with
// |x| 2^-e < 1/2, 0 where every upper word is zero, RZ_BAD for a row holding Inf or NaN.
#define RZ_BAD 0x7FFF
static __device__ __forceinline__ int rz_row_exp(unsigned int mh) {
    if (mh >= 0x7FF00000u) return RZ_BAD;
    if (mh == 0) return 0;
    return min(1000, max(-960, (int)(mh >> 20) - 1023 + 2));   // 2^(8D + 1 - e) is a normal double
}

// 2^(8D + 1 - e) of a row; 0 for a bad one (whose digits are then whatever they are: its results are set to NaN).
static __device__ __forceinline__ double rz_scale(int e, int D) {
    return e == RZ_BAD ? 0.0 : oz_pow2(8 * D + 1 - e);
}

// The D digits of the eight elements x (scale e) as bf16, one 16-byte chunk per digit tile: digit tile s - 1
// (base + (s - 1) stride) holds digit s, most significant first.  Fixed point X = round(x 2^(8D + 1 - e)) plus the bias
// 128 in every byte below the leading one: byte i of the sum minus 128 is the balanced digit of weight 256^i and
// the rest is the leading digit.  One FP64 FMA with 1.5 2^52 + bias leaves that sum in the low bits of its
// result: the FP64 pipe is otherwise idle here (42.5 M of them at r = 48 take it 73 us) while the ALU pipe bounds
// the kernel, and shifting the significand took it 20 operations an element (r = 48: transformation 399 -> 288 us).
static __device__ __forceinline__ void rz_digits8(const double (&x)[8], double scale, int D, uint8_t* dst, uint32_t stride) {
    unsigned int lo[8], hi[8];
    const double magic = __longlong_as_double(0x4338000000000000ll + (0x8080808080ll & ((1ll << (8 * (D - 1))) - 1)));
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const double y = fma(x[u], scale, magic);
        lo[u] = (unsigned int)__double2loint(y);
        hi[u] = (unsigned int)__double2hiint(y) - 0x43380000u;
    }
#pragma unroll
    for (int i = 0; i < RZ_DMAX; ++i) {   // byte i: digit s = D - i
        if (i >= D) break;
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            const unsigned int p = i < 4 ? lo[u] : hi[u], q = i < 4 ? lo[u + 1] : hi[u + 1];
            float2 f;
            if (i < D - 1) {
                f.x = __uint_as_float(__byte_perm(p, 0x4B000000u, 0x7540u | (unsigned)(i & 3)));
                f.y = __uint_as_float(__byte_perm(q, 0x4B000000u, 0x7540u | (unsigned)(i & 3)));
                f = __fadd2_rn(f, make_float2(-8388736.0f, -8388736.0f));
            } else {   // the leading digit, signed (|d| <= 256): bits 8 i .. of the sum
                const int tp = i < 4 ? (int)__funnelshift_r(lo[u], hi[u], 8 * i) : (int)hi[u] >> (8 * (i & 3));
                const int tq = i < 4 ? (int)__funnelshift_r(lo[u + 1], hi[u + 1], 8 * i) : (int)hi[u + 1] >> (8 * (i & 3));
                f = __fadd2_rn(make_float2(__int_as_float(0x4B400000 + tp), __int_as_float(0x4B400000 + tq)),
                               make_float2(-12582912.0f, -12582912.0f));
            }
            w[u / 2] = __byte_perm(__float_as_uint(f.x), __float_as_uint(f.y), 0x7632);   // exact in bf16
        }
        *reinterpret_cast<uint4*>(dst + (size_t)(D - 1 - i) * stride) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// acc 2^ex rounded to the nearest double (halves up): the significand is |acc| normalised to bit 63 and cut to 53
// bits with its rounding bit added; results outside the normal range take the general route.
static __device__ __forceinline__ double rz_scaled(long long acc, int ex) {
    const unsigned long long sg = (unsigned long long)(acc >> 63);
    const unsigned long long u = ((unsigned long long)acc ^ sg) - sg;
    const unsigned int uh = (unsigned int)(u >> 32);
    const int n = uh ? __clz(uh) : 32 + __clz((unsigned int)u);
    const int E = ex + 63 - n + 1022;   // exponent field less one: the significand's leading bit adds it
    const unsigned long long b = ((u << ((n - 1) & 63)) + 512) >> 10;   // |acc| < 2^63: n >= 1, no carry out
    if (acc == 0) return 0.0;
    if (E < 1 || E > 2044) return oz_ll_scaled(acc, ex);
    return __longlong_as_double((long long)((b + ((unsigned long long)(unsigned)E << 52)) | (sg << 63)));
}

// Descriptor of an unswizzled K-major operand: core matrices of 8 rows x 16 bytes, the next 8 rows 128 bytes on,
// the next 16 bytes of K `kstride` bytes on.
static __device__ __forceinline__ uint64_t rz_desc(const void* p, uint32_t kstride) {
    return (uint64_t)((smem_u32(p) & 0x3FFFFu) >> 4) | ((uint64_t)(kstride >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
           ((uint64_t)1 << 46);
}

static __device__ __forceinline__ void rz_tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}

// bounded_wait by lane 0 for the whole warp; on expiry the abort flag goes up (the result is warp-uniform).
static __device__ __forceinline__ bool rz_warp_wait(uint64_t* bar, uint32_t parity, int lane, int* err,
                                                    volatile int* abort_flag) {
    int go = 0;
    if (lane == 0) {
        go = bounded_wait(bar, parity, RZ_WAIT_NS, abort_flag) && !*abort_flag;
        if (!go) raise_abort(err, abort_flag);
    }
    go = __shfl_sync(0xffffffffu, go, 0);
    __syncwarp();
    return go != 0;
}

// Where tile `tile` reads and writes: rows m < nrow of the tile's group from row m0; element (m, q) of A at
// src[(m - m0) sm + q sq] (MODE 0: the row's own offset), G by number `sel`.
template <int MODE>
struct RzTile {
    const double* A;
    double* out;
    const double* G;
    int m0, nrow, sel, gt, tr, tri;
    size_t ld;
    __device__ __forceinline__ RzTile(const RowsArgs& a, int tile) {
        const int r = a.r, R2 = r * r;
        if (MODE == 0) {
            int g = 0;
            while (g < 7 && a.start[g + 1] <= tile) ++g;
            m0 = (tile - a.start[g]) * TC_BM;
            tri = (a.tri >> g) & 1;
            A = a.A[g];
            out = a.out[g];
            G = a.G[g];
            sel = a.sel[g];
            gt = (a.gt >> g) & 1;
            tr = (a.tt >> g) & 1;
            nrow = r * (tri ? r * (r - 1) / 2 : R2);
            ld = r;
        } else {   // g = (sector t, k): spin blocks (K, I) 0-3, the flips 4 (1D of beta) and 5 (of alpha)
            const int g = tile / a.tpg;
            m0 = (tile - g * a.tpg) * TC_BM;
            tri = 0;
            const int t = g / r, k = g - t * r, f = t < 4 ? 0 : t - 3;
            sel = t < 4 ? t >> 1 : t == 4 ? 1 : 0;
            ld = t < 4 ? 2 * (size_t)R2 : (size_t)R2;
            const size_t base = (t < 4 ? (size_t)sel * R2 * ld + (size_t)(t & 1) * R2 : 0) + (size_t)k * r * ld;
            A = a.A[f] + base;
            out = a.out[f] + base;
            G = a.G[sel];
            gt = a.gt & 1;
            tr = 1;
            nrow = R2;
        }
    }
};

// Row m = (pair number, a) of a class on the pairs i < j as the row (ij, a) of the full array.
static __device__ __forceinline__ int rz_pair_row(const RowsArgs& a, int m) {
    const int u = m / a.r;
    return a.pmap[u] * a.r + (m - u * a.r);
}

template <int RP, int MODE>
__global__ void __launch_bounds__(RZ_THREADS, 1) k_rows_oz(const __grid_constant__ RowsArgs a) {
    static_assert(RP % 16 == 0 && RP <= 64, "N = K = r padded to a multiple of 16");
    constexpr int NB = RP == 64 ? 1 : 2;              // buffers of A digits
    constexpr int NCH = RP / 8, NC = RP / 16;         // chunks of a row, chunks of a thread
    constexpr int A_SL = NCH * TC_BM * 16, B_SL = NCH * RP * 16;   // bytes of one digit
    constexpr int TCOLS = RP >= 48 ? 512 : RP == 32 ? 256 : 128;   // TMEM: RZ_DMAX + 1 accumulators of RP columns
    constexpr int CW = RP / 2;                        // columns of an epilogue thread
    extern __shared__ uint8_t rz_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)rz_raw + 127) & ~(uintptr_t)127);
    uint8_t* sA = smem;
    uint8_t* sB = sA + NB * RZ_DMAX * A_SL;
    int* eA = reinterpret_cast<int*>(sB + RZ_DMAX * B_SL);   // [RZ_ESLOT][128]
    int* eB = eA + RZ_ESLOT * TC_BM;                         // [RZ_ESLOT][64]
    uint64_t* full = reinterpret_cast<uint64_t*>(eB + RZ_ESLOT * 64);   // [NB]
    uint64_t* empty = full + 2;                                          // [NB]
    uint64_t* accf = empty + 2;
    uint64_t* acce = accf + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = a.r, D = a.D;
    const int per = (a.ntiles + (int)gridDim.x - 1) / (int)gridDim.x;
    const int t_beg = (int)blockIdx.x * per, t_end = min(a.ntiles, t_beg + per);
    if (threadIdx.x == 0) {
        for (int b = 0; b < NB; ++b) {
            mbar_init(&full[b], RZ_PW);
            mbar_init(&empty[b], 1);
        }
        mbar_init(accf, 1);
        mbar_init(acce, RZ_EW);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc(tmem_slot, TCOLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            const uint32_t idesc0 = make_idesc<0, 0>();   // without N
            int it = 0;
            for (int tile = t_beg; tile < t_end; ++tile, ++it) {
                const int b = it % NB;
                if (!bounded_wait(&full[b], (it / NB) & 1, RZ_WAIT_NS, abort_flag) ||
                    (it >= 1 && !bounded_wait(acce, (it - 1) & 1, RZ_WAIT_NS, abort_flag))) {
                    raise_abort(a.err, abort_flag);
                    break;
                }
                tc_fence_after();
                const uint8_t* A = sA + (size_t)b * RZ_DMAX * A_SL;
                // The digit tiles of G lie one after another along N, and those of one A digit s go to consecutive
                // levels, so that t = t0 .. are one MMA of N = nb RP columns from column (s + t0 - 2) RP (at most 256).
                // Level D + 2 starts with s = 2, t = D, the others with s = 1.  (One MMA per pair of digits, N = RP,
                // took about 200 cycles each whatever N: 9 and 3 % more for the pair products and the transformation at r = 48.)
                const uint64_t da0 = rz_desc(A, TC_BM * 16), db0 = rz_desc(sB, RZ_DMAX * RP * 16);
                for (int s = 1; s <= D; ++s) {
                    const int t1 = min(D, D + 2 - s);
                    for (int t = 1; t <= t1;) {
                        const int nb = min(256 / RP, (s == 2 && t < D ? min(t1, D - 1) : t1) - t + 1);
                        const uint32_t acc = tmem + (uint32_t)((s + t - 2) * RP);
                        const uint32_t id = idesc0 | ((uint32_t)(nb * RP >> 3) << 17);
                        const bool fresh = s == 1 || (s == 2 && t == D);
#pragma unroll
                        for (int kk = 0; kk < NC; ++kk)   // 16 K elements: two chunks
                            umma<0>(acc, da0 + (uint64_t)((s - 1) * (A_SL / 16) + kk * 2 * TC_BM),
                                    db0 + (uint64_t)((t - 1) * RP + kk * 2 * RZ_DMAX * RP), id, kk > 0 || !fresh);
                        t += nb;
                    }
                }
                umma_commit(&empty[b]);
                umma_commit(accf);
            }
            // no MMA is in flight past this point
            if (it > 0 && !bounded_wait(accf, (it - 1) & 1, RZ_WAIT_NS, nullptr)) raise_abort(a.err, abort_flag);
        }
    } else if (warp <= RZ_PW) {
        const int tid = threadIdx.x - 32, ml = tid >> 1, h = tid & 1;   // two threads per row
        int it = 0, cur = -1, slot = 0;
        double x[NC][8];
        // the row's elements of this thread (zero past r), and the scale of the whole row
        auto load = [&](const double* src, bool ok, size_t sq, bool vec) {
            unsigned int mh = 0;
            if (!ok) {
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int j = 0; j < 8; ++j) x[c][j] = 0.0;
            } else if (vec) {
                const double2* s4 = reinterpret_cast<const double2*>(src) + h;
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        const double2 v = 16 * c + 2 * j + 2 * h < r ? s4[8 * c + j] : make_double2(0.0, 0.0);
                        x[c][j] = v.x;
                        x[c][j + 1] = v.y;
                    }
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int q = 16 * c + 4 * (j >> 1) + 2 * h + (j & 1);
                        x[c][j] = q < r ? src[(size_t)q * sq] : 0.0;
                    }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int j = 0; j < 8; ++j) mh = max(mh, (unsigned int)__double2hiint(x[c][j]) & 0x7FFFFFFFu);
            mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, 1));
            return rz_row_exp(mh);
        };
        for (int tile = t_beg; tile < t_end; ++tile, ++it) {
            const RzTile<MODE> T(a, tile);
            const int b = it % NB;
            if (T.sel != cur) {   // G: its digit tiles are free once the MMAs of the last tile are done
                if (it > 0 && !rz_warp_wait(&empty[(it - 1) % NB], ((it - 1) / NB) & 1, lane, a.err, abort_flag)) break;
                cur = T.sel;
                slot = (slot + 1) & (RZ_ESLOT - 1);   // (a slot's last reader is at least three tiles back)
                const bool ok = ml < r;
                const int e = load(T.G + (size_t)(ok ? ml : 0) * (T.gt ? 1 : r), ok, T.gt ? r : 1,
                                   !T.gt && (r & 1) == 0 && (reinterpret_cast<uintptr_t>(T.G) & 15) == 0);
                if (ml < RP) {
                    if (h == 0) eB[slot * 64 + ml] = e;
#pragma unroll
                    for (int c = 0; c < NC; ++c) rz_digits8(x[c], rz_scale(e, D), D, sB + ((2 * c + h) * RZ_DMAX * RP + ml) * 16, RP * 16);
                }
            }
            const int m = T.m0 + ml;
            const bool ok = m < T.nrow;
            const double* src = T.A;
            size_t sq = 1;
            bool vec = false;
            if (MODE == 0) {
                const int row = T.tri && ok ? rz_pair_row(a, m) : m;
                if (T.tr) {
                    const int ij = row / r;
                    src += (size_t)ij * r * r + (row - ij * r);
                    sq = r;
                } else {
                    src += (size_t)row * r;
                    vec = (r & 1) == 0 && (reinterpret_cast<uintptr_t>(T.A) & 15) == 0;
                }
            } else {
                src += m;
                sq = T.ld;
            }
            const int e = load(src, ok, sq, vec);
            if (it >= NB && !rz_warp_wait(&empty[b], ((it / NB) & 1) ^ 1, lane, a.err, abort_flag)) break;
            // scales: the MMAs of tile it - NB are done, so the epilogue of tile it - NB - 1 has handed TMEM back
            // and that of tile it - 4 is over: its slot is free
            if (h == 0) eA[(it & (RZ_ESLOT - 1)) * TC_BM + ml] = e;
            uint8_t* A = sA + (size_t)b * RZ_DMAX * A_SL;
#pragma unroll
            for (int c = 0; c < NC; ++c) rz_digits8(x[c], rz_scale(e, D), D, A + (2 * c + h) * TC_BM * 16 + ml * 16, A_SL);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor cores
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[b]);
        }
    } else {
        const int q4 = warp & 3, half = (warp - 1 - RZ_PW) >> 2;   // TMEM lane quarter, column half
        const int ml = q4 * 32 + lane;
        int it = 0, cur = -1, slot = 0;
        for (int tile = t_beg; tile < t_end; ++tile, ++it) {
            const RzTile<MODE> T(a, tile);
            if (T.sel != cur) {
                cur = T.sel;
                slot = (slot + 1) & (RZ_ESLOT - 1);
            }
            if (!rz_warp_wait(accf, it & 1, lane, a.err, abort_flag)) break;
            tc_fence_after();
            long long acc[CW];
            const uint32_t t0 = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(half * CW);
#pragma unroll
            for (int g = 0; g < CW; g += 4) {
                uint32_t v[RZ_DMAX + 1][4];
                // the levels L = D - 4 + j, j = 0 .. 6 (those below 2 are zero)
#pragma unroll
                for (int j = 0; j <= RZ_DMAX; ++j) {
                    const int L = D - 4 + j;
                    if (L >= 2) rz_tmem_ld4(t0 + (uint32_t)((L - 2) * RP + g), v[j]);
                    else v[j][0] = v[j][1] = v[j][2] = v[j][3] = 0u;
                }
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    unsigned int w[RZ_DMAX + 1][2];   // level sums as integers (modulo 2^32)
#pragma unroll
                    for (int j = 0; j <= RZ_DMAX; ++j) {
                        // level j holds at most j + 1 products (the last D - 1 <= 5), in units of RP 2^14: one of 4, or two
                        // of 2 and the rest of 1 (the last: of 1 only); within the 2^22 of the FADD conversion for n RP <= 256
                        const float2 f = make_float2(__uint_as_float(v[j][c]), __uint_as_float(v[j][c + 1]));
                        if ((j == RZ_DMAX ? RZ_DMAX - 1 : j == 0 ? 4 : j + 3) * RP <= 256) {
                            const float2 m = __fadd2_rn(f, make_float2(12582912.0f, 12582912.0f));
                            w[j][0] = __float_as_uint(m.x) - 0x4B400000u;
                            w[j][1] = __float_as_uint(m.y) - 0x4B400000u;
                        } else {
                            w[j][0] = (unsigned int)__float2int_rn(f.x);
                            w[j][1] = (unsigned int)__float2int_rn(f.y);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int p1 = (int)(w[0][u] * 256u + w[1][u]), p2 = (int)(w[2][u] * 256u + w[3][u]);
                        const int p3 = (int)(w[4][u] * 256u + w[5][u]) + (((int)w[6][u] + 128) >> 8);
                        acc[g + c + u] = ((long long)p1 * 65536 + p2) * 65536 + p3;
                    }
                }
            }
            const int em = eA[(it & (RZ_ESLOT - 1)) * TC_BM + ml];
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce);   // TMEM is free for the next tile
            const int m = T.m0 + ml;
            if (m >= T.nrow) continue;
            const int* eb = eB + slot * 64 + half * CW;
            double* o = T.out + (MODE == 0 ? (size_t)(T.tri ? rz_pair_row(a, m) : m) * r + half * CW : (size_t)(half * CW) * T.ld + m);
            const bool v2 = MODE == 0 && (r & 1) == 0 && (reinterpret_cast<uintptr_t>(T.out) & 15) == 0;
#pragma unroll
            for (int n = 0; n < CW; n += 2) {
                if (half * CW + n >= r) break;
                double z[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int en = eb[n + u];
                    z[u] = (em == RZ_BAD || en == RZ_BAD) ? __longlong_as_double(0x7ff8000000000000ll)
                                                          : rz_scaled(acc[n + u], em + en - 8 * (D + 1) - 2);
                }
                if (v2) {
                    *reinterpret_cast<double2*>(o + n) = make_double2(z[0], z[1]);
                } else {
                    const size_t s = MODE == 0 ? 1 : T.ld;
                    o[n * s] = z[0];
                    if (half * CW + n + 1 < r) o[(n + 1) * s] = z[1];
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, TCOLS);
    }
}

template <int RP, int MODE>
static int rows_launch(const RowsArgs& a, cudaStream_t st) {
    constexpr int NB = RP == 64 ? 1 : 2;
    constexpr int smem = 128 + RZ_DMAX * (RP / 8) * 16 * (NB * TC_BM + RP) + RZ_ESLOT * 4 * (TC_BM + 64) + 64;
    int dev = 0, nsm = 152;
    ACSE_CUDA_TRY(cudaFuncSetAttribute(k_rows_oz<RP, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    ACSE_CUDA_TRY(cudaGetDevice(&dev));
    ACSE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    k_rows_oz<RP, MODE><<<a.ntiles < nsm ? a.ntiles : nsm, RZ_THREADS, smem, st>>>(a);
    ACSE_CUDA_TRY(cudaGetLastError());
    return ACSE_OK;
}

template <int MODE>
static int rows_dispatch(acse_ctx* c, RowsArgs& a) {
    const int r = c->r;
    a.r = r;
    a.D = (6 * c->opt.oz_slices + 7) / 8;
    a.err = c->w.tc_err;
    int s;
    switch ((r + 15) / 16) {
        case 1: s = rows_launch<16, MODE>(a, c->stream); break;
        case 2: s = rows_launch<32, MODE>(a, c->stream); break;
        case 3: s = rows_launch<48, MODE>(a, c->stream); break;
        default: s = rows_launch<64, MODE>(a, c->stream); break;
    }
    if (s == ACSE_OK) c->launches++;
    return s;
}

static bool rows_oz_applies(const acse_ctx* c) { return c->oz && c->opt.oz_slices <= RZ_SMAX && c->r >= ACSE_OZ_RMIN; }

// The transformation by 1D (trans: by its transpose) of the three arrays; ACSE_ERR_UNSUPPORTED where the kernel
// does not apply.
int launch_xform_oz(acse_ctx* c, const double* const in[3], double* const out[3], int trans) {
    if (!rows_oz_applies(c)) return ACSE_ERR_UNSUPPORTED;
    const int r = c->r;
    RowsArgs a = {};
    for (int f = 0; f < 3; ++f) {
        a.A[f] = in[f];
        a.out[f] = out[f];
    }
    a.G[0] = c->w.gam;
    a.G[1] = c->w.gam + (size_t)r * r;
    a.gt = trans ? 1u : 0u;
    a.tpg = (r * r + TC_BM - 1) / TC_BM;
    a.ntiles = 6 * r * a.tpg;
    return rows_dispatch<1>(c, a);
}

// The eight classes of tall products of launch_pair_rows; ACSE_ERR_UNSUPPORTED where the kernel does not apply.
int launch_rows_oz(acse_ctx* c, const double* const T[8], unsigned tt, const double* const G[8], unsigned gt, unsigned tri,
                   double* const out[8]) {
    if (!rows_oz_applies(c)) return ACSE_ERR_UNSUPPORTED;
    const int r = c->r;
    RowsArgs a = {};
    for (int k = 0; k < 8; ++k) {
        a.A[k] = T[k];
        a.G[k] = G[k];
        a.out[k] = out[k];
        a.sel[k] = k;
        for (int m = 0; m < k; ++m)
            if (G[m] == G[k] && ((gt >> m) & 1) == ((gt >> k) & 1)) {
                a.sel[k] = m;
                break;
            }
        const int items = (tri >> k) & 1 ? r * (r - 1) / 2 : r * r;
        a.start[k + 1] = a.start[k] + (items * r + TC_BM - 1) / TC_BM;
    }
    a.tt = tt;
    a.gt = gt;
    a.tri = tri;
    a.pmap = c->w.pmap;
    a.ntiles = a.start[8];
    return rows_dispatch<0>(c, a);
}
