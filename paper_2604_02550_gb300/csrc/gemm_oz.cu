// FP64-accurate GEMMs of the contraction pass on the BF16 tensor cores by the modular form of the Ozaki
// scheme (K. Ozaki, Y. Uchino, T. Imamura, "Ozaki Scheme II: a GEMM-oriented emulation of floating-point
// matrix multiplication using an integer modular technique", 2025).
//
// C = alpha A B^T with A (M x K) and B (N x K) FP64, both K-major.  Every operand row is scaled by a power
// of two and rounded to an integer row: with |a| 2^-e < 1/2 over the row, X = round(a 2^(nb - e)), so that
// |X| <= 2^(nb-1) and a = 2^(e - nb) X up to half a unit of the last kept bit (nb - 1 = min(6S, 53) bits
// below the row's leading bit for oz_slices = S).  The integer product X_A X_B^T then has entries of at
// most K 2^(2 nb - 2) in magnitude.  It is computed modulo T pairwise coprime moduli p_t <= 127 (the
// first T of a fixed list, T the least with 4 K 2^(2 nb - 2) <= P = prod p_t):
//   * the residue kernel writes near-balanced residues X mod p_t (|.| <= 64, exact in bf16), the B rows
//     premultiplied by y_t = (P / p_t)^-1 mod p_t, each modulus to its K segment of the row;
//   * the tensor cores multiply the residue matrices of each modulus in FP32; a chunk of at most 64 * 64
//     K elements keeps every partial sum an integer of magnitude at most 64 * 64 * 64^2 = 2^24, so the
//     accumulation is exact, and the epilogue stores a residue w (|w| <= 65) of the chunk sum (one byte);
//   * the reconstruction kernel takes x / P = sum_t w_t / p_t modulo 1 (Chinese remainder theorem: w_t is the residue
//     of x (P / p_t)^-1) in fixed point, the wrap-around modulo 2^96 being the reduction modulo 1; |x| <= P / 4, so the
//     signed fraction is x / P itself, and x = P (x / P) is rounded once to FP64 and scaled by alpha 2^(ea + eb - 2 nb).
// The result is the FP64 product up to the rounding of the operands to nb - 1 bits below each row's
// leading bit, the 2^-77 P of the fraction's constants (2^-10 of the operand rounding or less) and one final
// rounding: no product level is dropped.  Against the six-bit slice form of
// the scheme (36 slice products at S = 8) this takes 17 residue products at S = 8 and r = 48.
//
// Kernels: the persistent tcgen05 GEMM of gemm_tc.cu with the accumulation unit changed from a tile
// to a (tile, modulus, K chunk) group: the MMA thread runs the groups of a tile one after another into the
// two TMEM buffers, and the epilogue warps store each group's residue (a byte) to a staging array.  A
// second kernel rebuilds every element from its residues and writes the FP64 result once.  Every wait
// is bounded as in gemm_tc.cu.
#include <cuda.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "acse_internal.h"
#include "oz_arith.cuh"
#include "tc_ptx.cuh"

#define OZ_NMOD 19           // moduli of the fixed list
#define OZ_CHUNK_KB 64       // 64-element K blocks of one exactly accumulated chunk: 64 * 64 * 64^2 = 2^24
#define OZ_MAXCH 2           // chunks of one residue product (K <= 2 * 64 * 64 = 8192)
#define OZ_MAXP 12           // GEMMs of one launch
#define OZ_MAXJ 16           // operands of one slicing launch
#define OZ_THREADS 192
#define OZ_BN 256
#define OZ_STAGES 4
#define OZ2_STAGES 6         // ring depth of the CTA-pair form (32 KB a stage per CTA)
#define OZ_DRAIN_NS 2000000000ull
#define OZ_WAIT_NS 4000000000ull
#define OZ_FL 11                       // bytes of the reconstruction's constants 2^88 / p_t
#define OZ_NQ (OZ_NMOD * OZ_MAXCH + 3) / 4   // (modulus, chunk) groups in fours

// Pairwise coprime moduli, largest first: 127, 5^3, 3 * 41, 11^2, 7 * 17 and the primes 113 .. 59.
static const int oz_moduli[OZ_NMOD] = {127, 125, 123, 121, 119, 113, 109, 107, 103, 101, 97, 89, 83, 79, 73, 71, 67, 61, 59};

// The constants of a set of T moduli (host-computed, exact).
struct OzMods {
    int T;
    float p[OZ_NMOD];         // p_t
    float pinv[OZ_NMOD];      // 1 / p_t, rounded
    float cA[OZ_NMOD][4];     // 2^(14 l) mod p_t, l = 0..3 (limb weights of an A row)
    float cB[OZ_NMOD][4];     // 2^(14 l) y_t mod p_t, y_t = (P / p_t)^-1 mod p_t (limb weights of a B row)
    unsigned long long Pm;    // P = Pm 2^Pe, Pm with bit 63 set (truncated where P has more than 64 bits)
    int Pe;
};

struct OzProb {
    double* C;
    unsigned char* stage;   // [ngroups][M][ns]: the residue w + 128 of each (modulus, chunk) group
    int ns;                 // row pitch of stage: N rounded up to 32, so that a thread's 32 residues always leave
                            // as two aligned 16-byte stores (byte stores for odd N held the GEMM of r = 30 at
                            // 1.32 ms, 8 times its work)
    const double* sa;   // 2^ea per row of A
    const double* sb;   // 2^eb per row of B
    int ealpha;         // alpha = 2^ealpha
    int M, N, ldc;
    int kbs;            // 64-element K blocks per modulus segment
    int nch, cb;        // K chunks per modulus and 64-element blocks per chunk (the last may be shorter)
    int nb;             // operand rows rounded to X = round(a 2^(nb - e))
    int ngroups;        // T nch, modulus-major
    int tiles_n, tile_start;
    const int* gate;    // null, or the problem is skipped where *gate is zero
};

struct __align__(128) OzBatch {
    CUtensorMap tmA[OZ_MAXP];
    CUtensorMap tmB[OZ_MAXP];
    OzProb p[OZ_MAXP];
    OzMods mods;
    int nprob;
    int total_tiles;
    int* err;
    unsigned long long wait_ns;
    int inject_stall;
    const int* order;     // tiles of CTA c: order[cta_start[c] .. cta_start[c+1]) (longest first)
    const int* cta_start;
};

// A gated problem whose gate is down: every role of the kernel passes over its tiles.
__device__ __forceinline__ bool oz_skip(const OzProb& P) { return P.gate && !*P.gate; }

__device__ __forceinline__ int oz_find_problem(const OzBatch& b, int t) {
    int lo = 0, hi = b.nprob - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b.p[mid].tile_start <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Near-balanced residue of an integer-valued float |v| <= 2^24 modulo p <= 127: q = round(v pinv) (the
// fused multiply-add rounds v pinv + 1.5 * 2^23 once, to an integer), r = v - q p exactly.  pinv = 1/p
// rounded moves v / p by at most |v / p| 2^-24 <= 0.017 of a unit, so |r| <= p (1/2 + 0.017): at most 64
// for |v| < 2^23 and at most 65 for |v| <= 2^24.  No correction into the balanced range is needed: the
// residue products and the reconstruction are bounded with these limits.
__device__ __forceinline__ float oz_bal_mod(float v, float p, float pinv) {
    const float q = fmaf(v, pinv, 12582912.0f) - 12582912.0f;
    return fmaf(-q, p, v);
}

// ------------------------------------------------------------------------------ slicing
struct OzSliceJob {
    const double* src;
    size_t lds;             // source row stride (elements)
    const int* rowmap;      // source row of each output row (null: the same row)
    const int* colmap;      // source column of each K index (null: the same column)
    __nv_bfloat16* dst;     // first output row of the job
    size_t ldd;             // T * Kp
    double* scale;          // 2^e per output row (NaN for a row with a non-finite entry)
    int rows, K, Kp, nb, mul_y, row0;
};

struct OzSliceBatch {
    OzSliceJob j[OZ_MAXJ];
    int njobs;
    int T;
    float p[OZ_NMOD], pinv[OZ_NMOD];
    float cA[OZ_NMOD][4], cB[OZ_NMOD][4];
};

// 2^e of a row whose largest magnitude has the pattern mx (non-negative doubles order like their bit patterns; an
// all-ones exponent is Inf or NaN).
__device__ __forceinline__ double oz_row_scale(unsigned long long mx) {
    const bool bad = mx >= 0x7FF0000000000000ull;
    const int e = (bad || mx == 0) ? 0 : min(1000, max(-1000, (int)(mx >> 52) - 1023 + 2));
    return bad ? __longlong_as_double(0x7ff8000000000000ll) : oz_pow2(e);
}

// Row scales: one warp per operand row takes the largest magnitude over the row (through the maps), which
// fixes e (|a| 2^-e < 1/2); scale = 2^e, NaN for a row with a non-finite entry.
__global__ void __launch_bounds__(256) k_oz_rowscale(const __grid_constant__ OzSliceBatch b, int rows) {
    const int grow = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (grow >= rows) return;
    int ji = 0;
    while (ji + 1 < b.njobs && b.j[ji + 1].row0 <= grow) ++ji;
    const OzSliceJob& J = b.j[ji];
    const int row = grow - J.row0;
    const int srow = J.rowmap ? J.rowmap[row] : row;
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(J.src + (size_t)srow * J.lds);
    const int* cm = J.colmap;
    unsigned long long mx = 0;
    for (int k = lane; k < J.K; k += 32) mx = max(mx, src[cm ? cm[k] : k] & 0x7FFFFFFFFFFFFFFFull);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) J.scale[row] = oz_row_scale(mx);
}

// Residues: block (x, y) covers elements 1024 x .. 1024 x + 1023 of operand row y (rows of all jobs in
// order), four consecutive elements a thread (8-byte stores of their four bf16 residues per modulus).  The integer X = round(a 2^(nb - e)) (|X| <= 2^53) is cut into
// four base-2^14 limbs of |X|, each made an exact float through the bits of 2^23 + limb (no 64-bit
// conversion: those run on the slow FP64 unit) and given the sign of X; modulus by modulus, the residue
// is sum_l limb_l c_l (c_l = 2^(14 l) mod p_t, times y_t for a B operand; an integer below 2^23 in
// magnitude, exact in FP32) reduced by oz_bal_mod (|residue| <= 64, exact in bf16: the upper half of its
// float).  Modulus t goes to K segment t of the row.
__device__ __forceinline__ void oz_limbs(unsigned long long bits, int nb, int e, bool bad, float* L) {
    const long long X = bad ? 0 : oz_fixedb(bits, nb, e);
    const unsigned long long uX = X < 0 ? 0ull - (unsigned long long)X : (unsigned long long)X;
    const float sg = X < 0 ? -1.0f : 1.0f;
    const unsigned int lo = (unsigned int)uX, hi = (unsigned int)(uX >> 32);
    const unsigned int l0 = lo & 0x3FFF, l1 = (lo >> 14) & 0x3FFF, l2 = (lo >> 28) | ((hi & 0x3FF) << 4), l3 = hi >> 10;
    L[0] = sg * (__uint_as_float(0x4B000000u | l0) - 8388608.0f);
    L[1] = sg * (__uint_as_float(0x4B000000u | l1) - 8388608.0f);
    L[2] = sg * (__uint_as_float(0x4B000000u | l2) - 8388608.0f);
    L[3] = sg * (__uint_as_float(0x4B000000u | l3) - 8388608.0f);
}

__device__ __forceinline__ void oz_residue4(const OzSliceBatch& b, const OzSliceJob& J, int row, int qi) {
    const int K = J.K, k = 4 * qi;
    const int srow = J.rowmap ? J.rowmap[row] : row;
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(J.src + (size_t)srow * J.lds);
    const int* cm = J.colmap;
    unsigned long long v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = k + i < K ? src[cm ? cm[k + i] : k + i] : 0ull;
    const int es = (int)((__double_as_longlong(J.scale[row]) >> 52) & 0x7FF);   // 2^e, or NaN
    const bool bad = es == 0x7FF;
    float L[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) oz_limbs(v[i], J.nb, es - 1023, bad, L[i]);
    __nv_bfloat16* dst = J.dst + (size_t)row * J.ldd + k;
    const int nk = min(4, K - k);
    const float(*c)[4] = J.mul_y ? b.cB : b.cA;
    const int T = b.T;
#pragma unroll 2
    for (int t = 0; t < T; ++t, dst += J.Kp) {
        const float p = b.p[t], pinv = b.pinv[t];
        const float c0 = c[t][0], c1 = c[t][1], c2 = c[t][2], c3 = c[t][3];
        unsigned int h[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)   // |r| <= 64: the bf16 of r is the upper half of its float (exact)
            h[i] = __float_as_uint(oz_bal_mod(fmaf(L[i][3], c3, fmaf(L[i][2], c2, fmaf(L[i][1], c1, L[i][0] * c0))), p, pinv));
        if (nk == 4) {
            *reinterpret_cast<uint2*>(dst) = make_uint2(__byte_perm(h[0], h[1], 0x7632), __byte_perm(h[2], h[3], 0x7632));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < nk) reinterpret_cast<unsigned short*>(dst)[i] = (unsigned short)(h[i] >> 16);
        }
    }
}

__global__ void __launch_bounds__(256) k_oz_residue(const __grid_constant__ OzSliceBatch b) {
    const int grow = (int)blockIdx.y;
    int ji = 0;
    while (ji + 1 < b.njobs && b.j[ji + 1].row0 <= grow) ++ji;
    const int qi = (int)blockIdx.x * 256 + (int)threadIdx.x;
    if (qi < (b.j[ji].K + 3) >> 2) oz_residue4(b, b.j[ji], grow - b.j[ji].row0, qi);
}

// Scales and residues of gated operands, a block per row in turn: one launch that leaves at once (1.5 us) where *gate
// is zero.  (As rows of the launches above, 7000 of them at r = 48 took 20 us to be passed over.)
__global__ void __launch_bounds__(256) k_oz_slice_gated(const __grid_constant__ OzSliceBatch b, int rows, const int* gate) {
    if (!*gate) return;
    __shared__ unsigned long long sh[8];
    for (int grow = (int)blockIdx.x; grow < rows; grow += (int)gridDim.x) {
        int ji = 0;
        while (ji + 1 < b.njobs && b.j[ji + 1].row0 <= grow) ++ji;
        const OzSliceJob& J = b.j[ji];   // (no maps)
        const int row = grow - J.row0;
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(J.src + (size_t)row * J.lds);
        unsigned long long mx = 0;
        for (int k = threadIdx.x; k < J.K; k += 256) mx = max(mx, src[k] & 0x7FFFFFFFFFFFFFFFull);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 0; w < 8; ++w) mx = max(mx, sh[w]);
            J.scale[row] = oz_row_scale(mx);
        }
        __syncthreads();
        for (int qi = threadIdx.x; qi < (J.K + 3) >> 2; qi += 256) oz_residue4(b, J, row, qi);
    }
}

// ------------------------------------------------------------------------------- GEMM
// PAIR: the CTA-pair form of gemm_tc.cu (launched in clusters of two CTAs; pair MMA of M = 256 on
// 256 x BN tiles, each CTA loading its 128 rows of A and BN / 2 rows of B; the even CTA issues the MMAs
// and commits to the barriers of both; both CTAs' loads complete on the even CTA's full[s]; both
// CTAs' epilogue warps arrive on the even CTA's acce[ab]).
template <int BN, int STAGES, bool PAIR>
__global__ void __launch_bounds__(OZ_THREADS, 1) k_gemm_oz(const OzBatch* __restrict__ bp) {
    const OzBatch& b = *bp;
    constexpr int A_BYTES = TC_BM * 128;
    constexpr int B_BYTES = (PAIR ? BN / 2 : BN) * 128;
    constexpr int BM = PAIR ? 2 * TC_BM : TC_BM;   // rows of an output tile
    constexpr int KELEM = 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = smem + STAGES * A_BYTES;
    uint64_t* full = (uint64_t*)(sB + STAGES * B_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* accf = empty + STAGES;   // [2]
    uint64_t* acce = accf + 2;         // [2]
    uint64_t* never = acce + 2;
    uint64_t* drainb = never + 1;
    uint32_t* tmem_slot = (uint32_t*)(drainb + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
    const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;   // CTA, or CTA pair
    const int q0 = b.cta_start[unit], q1 = b.cta_start[unit + 1];        // this unit's tiles
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&accf[a], 1);
            mbar_init(&acce[a], PAIR ? 8 : 4);
        }
        mbar_init(never, 1);
        mbar_init(drainb, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        if constexpr (PAIR) tmem_alloc_pair(tmem_slot, 2 * BN);
        else tmem_alloc(tmem_slot, 2 * BN);
    }
    tc_fence_before();
    if constexpr (PAIR) cluster_sync_all();
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            const uint32_t full0 = PAIR ? mapa_rank(smem_u32(full), 0) : 0u;   // the even CTA's full[0]
            int it = 0;
            bool stop = false;
            for (int qi = q0; qi < q1 && !stop; ++qi) {
                const int t = b.order[qi];
                const int pi = oz_find_problem(b, t);
                const OzProb& P = b.p[pi];
                if (oz_skip(P)) continue;
                const int local = t - P.tile_start;
                const int m0 = (local / P.tiles_n) * BM + (int)rank * TC_BM;
                const int n0 = (local % P.tiles_n) * BN + (int)rank * (BN / 2);
                for (int gi = 0; gi < P.ngroups && !stop; ++gi) {
                    // group gi = (modulus t, chunk c): the same K range of A and B
                    const int tm = gi / P.nch, c = gi - tm * P.nch;
                    const int ka = tm * P.kbs + c * P.cb, n = min(P.cb, P.kbs - c * P.cb);
                    for (int kb = 0; kb < n; ++kb, ++it) {
                        const int s = it % STAGES;
                        if (it >= STAGES && !bounded_wait(&empty[s], ((it / STAGES) & 1) ^ 1, b.wait_ns, abort_flag)) {
                            raise_abort(b.err, abort_flag);
                            stop = true;
                            break;
                        }
                        if constexpr (PAIR) {
                            if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * (A_BYTES + B_BYTES));
                            tma_load_2d_pair(sA + s * A_BYTES, &b.tmA[pi], (ka + kb) * KELEM, m0, full0 + 8u * s);
                            tma_load_2d_pair(sB + s * B_BYTES, &b.tmB[pi], (ka + kb) * KELEM, n0, full0 + 8u * s);
                        } else {
                            mbar_arrive_expect_tx(&full[s], A_BYTES + B_BYTES);
                            tma_load_2d(sA + s * A_BYTES, &b.tmA[pi], (ka + kb) * KELEM, m0, &full[s]);
                            tma_load_2d(sB + s * B_BYTES, &b.tmB[pi], (ka + kb) * KELEM, n0, &full[s]);
                        }
                    }
                }
            }
            // every issued copy must have landed before the CTA may exit (with pairs: the even CTA's
            // full[s] counts both CTAs' bytes; the odd CTA also waits for the MMAs that read its last
            // stages, briefly after an abort)
            for (int k = it > STAGES ? it - STAGES : 0; k < it; ++k) {
                const unsigned long long lim = *abort_flag ? b.wait_ns : OZ_DRAIN_NS;
                const bool ok = rank == 0 ? bounded_wait(&full[k % STAGES], (k / STAGES) & 1, lim, nullptr)
                                          : bounded_wait(&empty[k % STAGES], (k / STAGES) & 1, lim, nullptr);
                if (!ok) {
                    raise_abort(b.err, abort_flag);
                    if (rank != 0) break;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = PAIR ? make_idesc_pair<0, BN>() : make_idesc<0, BN>();
            if (b.inject_stall && !bounded_wait(never, 0, b.wait_ns, abort_flag)) raise_abort(b.err, abort_flag);
            int it = 0, lt = 0;
            for (int qi = q0; qi < q1 && !*abort_flag; ++qi) {
                const OzProb& P = b.p[oz_find_problem(b, b.order[qi])];
                if (oz_skip(P)) continue;
                for (int gi = 0; gi < P.ngroups && !*abort_flag; ++gi, ++lt) {
                    const int c = gi % P.nch;
                    const int n = min(P.cb, P.kbs - c * P.cb);
                    const int ab = lt & 1, use = lt >> 1;
                    if (use >= 1) {
                        const bool ok = PAIR ? bounded_wait_cluster(&acce[ab], (use - 1) & 1, b.wait_ns + OZ_DRAIN_NS, abort_flag)
                                             : bounded_wait(&acce[ab], (use - 1) & 1, b.wait_ns + OZ_DRAIN_NS, abort_flag);
                        if (!ok) {
                            raise_abort(b.err, abort_flag);
                            break;
                        }
                    }
                    tc_fence_after();
                    const uint32_t acc = tmem + (uint32_t)(ab * BN);
                    for (int kb = 0; kb < n; ++kb, ++it) {
                        const int s = it % STAGES;
                        if (!bounded_wait(&full[s], (it / STAGES) & 1, b.wait_ns, abort_flag)) {
                            raise_abort(b.err, abort_flag);
                            break;
                        }
                        tc_fence_after();
                        const uint64_t da = smem_desc(sA + s * A_BYTES);
                        const uint64_t db = smem_desc(sB + s * B_BYTES);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            if constexpr (PAIR) umma_pair<0>(acc, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0);
                            else umma<0>(acc, da + 2 * kk, db + 2 * kk, idesc, (kb | kk) != 0);
                        }
                        if constexpr (PAIR) umma_commit_pair(&empty[s]);
                        else umma_commit(&empty[s]);
                    }
                    // the epilogue of this group may start when its MMAs are done
                    if constexpr (PAIR) umma_commit_pair(&accf[ab]);
                    else umma_commit(&accf[ab]);
                }
            }
            if constexpr (PAIR) umma_commit_pair(drainb);
            else umma_commit(drainb);
        }
        // no MMA is in flight past this point (bounded; with pairs in both CTAs)
        if (lane == 0 && (PAIR || rank == 0) && !bounded_wait(drainb, 0, b.wait_ns + 2 * OZ_DRAIN_NS, nullptr))
            raise_abort(b.err, abort_flag);
    } else {
        const int q = warp & 3;   // TMEM lane quadrant this warp may access
        const uint32_t acce0 = PAIR ? mapa_rank(smem_u32(acce), 0) : 0u;
        int lt = 0;
        bool run = true;
        for (int qi = q0; qi < q1 && run; ++qi) {
            const int t = b.order[qi];
            const OzProb& P = b.p[oz_find_problem(b, t)];
            if (oz_skip(P)) continue;
            const int local = t - P.tile_start;
            const int m0 = (local / P.tiles_n) * BM + (int)rank * TC_BM, n0 = (local % P.tiles_n) * BN;
            const int row = m0 + q * 32 + lane;
            const bool rok = row < P.M;
            for (int gi = 0; gi < P.ngroups; ++gi, ++lt) {
                const int ab = lt & 1, use = lt >> 1;
                int go = 0;
                if (lane == 0) {
                    const bool ok = bounded_wait(&accf[ab], use & 1, b.wait_ns + OZ_DRAIN_NS, abort_flag);
                    if (!ok) raise_abort(b.err, abort_flag);
                    go = ok && !*abort_flag;
                }
                go = __shfl_sync(0xffffffffu, go, 0);
                if (!go) {
                    run = false;
                    break;
                }
                tc_fence_after();
                const int tm = gi / P.nch;
                const float pm = b.mods.p[tm], pinv = b.mods.pinv[tm];
                // the chunk sum is an integer of magnitude at most 2^24 (exact in FP32); its residue w modulo
                // p_t (|w| <= 65) goes out as the byte w + 128 (the low byte of the float w + 128 + 1.5 * 2^23)
                unsigned char* srow = P.stage + ((size_t)gi * P.M + (rok ? row : 0)) * P.ns;
#pragma unroll 1
                for (int c = 0; c < BN / 32; ++c) {
                    uint32_t v[32];
                    __syncwarp();
                    tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * BN + c * 32), v);   // warp-collective
                    const int col0 = n0 + c * 32;
                    if (!rok || col0 >= P.N) continue;
                    uint32_t wd[8];
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        uint32_t x[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            x[i] = __float_as_uint(oz_bal_mod(__uint_as_float(v[j + i]), pm, pinv) + 12583040.0f);
                        wd[j / 4] = __byte_perm(__byte_perm(x[0], x[1], 0x0040), __byte_perm(x[2], x[3], 0x0040), 0x5410);
                    }
                    *reinterpret_cast<uint4*>(srow + col0) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                    *reinterpret_cast<uint4*>(srow + col0 + 16) = make_uint4(wd[4], wd[5], wd[6], wd[7]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {   // this warp's quarter of the buffer is free
                    if constexpr (PAIR) mbar_arrive_cluster(acce0 + 8u * ab);
                    else mbar_arrive(&acce[ab]);
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    if constexpr (PAIR) cluster_sync_all();   // neither CTA exits while the other may still signal it
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem, 2 * BN);
        else tmem_dealloc(tmem, 2 * BN);
    }
}

// --------------------------------------------------------------------------- reconstruction
// x / P = sum over the (modulus, chunk) groups of w / p_t modulo 1, in units of 2^-88: F = sum_g w_g C_t modulo 2^88
// with C_t = round(2^88 / p_t), eleven bytes.  The four residue bytes b = w + 128 of four groups meet each byte of
// their constants in one dp4a (the 128 sum C_t comes off at the start): 5 x 11 of them for 17 moduli, where the sums
// of s = sum w_t P / p_t in float limbs took 17 x 12 FMAs, an estimate of s / P and a subtraction of its multiple
// (r = 48: 31.6 M elements a pass, 733 -> 244 us, 3.2 TB/s; issue-bound, dp4a at half rate).  The
// constants are off by at most 1/2, so F by sum |w| / 2 <= 38 x 65 / 2 < 2^11 units: 2^-77 of P, against an operand
// rounding of at least 2^-67 of P (the longest list, 53 bits).  An F of that size is a zero (exact cancellations stay
// zero).  Wrap-around modulo 2^96 (F shifted by a byte) is the reduction modulo 1, and |x| <= P / 4 leaves the sign in
// the top bit.
struct OzCrtParams {
    unsigned c1[5][OZ_FL], c2[OZ_NQ][OZ_FL];   // one or two K chunks: byte l of the constants of groups 4u .. 4u + 3
    int i1[OZ_FL], i2[OZ_FL];                  // -128 sum_g (byte l of C)
    unsigned long long Pm;
    int Pe, T;
};

// The FP64 value of x 2^ex from the eleven byte sums a_l (weight 2^(8 l) of F): carries into three 32-bit words of
// 2^8 F, magnitude, its leading 64 bits times P, rounded to 53 bits.
__device__ __forceinline__ double oz_frac_value(const int (&a)[OZ_FL], unsigned long long Pm, int ex) {
    // bytes in pairs, pairs in 64-bit words of weight 2^32 (every sum below 2^21 in magnitude)
    const long long t0 = (long long)(a[0] * 256) + (long long)(a[1] + a[2] * 256) * 65536;
    const long long t1 = (long long)(a[3] + a[4] * 256) + (long long)(a[5] + a[6] * 256) * 65536;
    const long long t2 = (long long)(a[7] + a[8] * 256) + (long long)(a[9] + a[10] * 256) * 65536;
    const long long u1 = t1 + (t0 >> 32), u2 = t2 + (u1 >> 32);
    const unsigned int sg = (unsigned int)((int)u2 >> 31);   // 0, or all ones for a negative x
    unsigned int w0 = (unsigned int)t0 ^ sg, w1 = (unsigned int)u1 ^ sg, w2 = (unsigned int)u2 ^ sg;
    if (w2 == 0) {   // |x| < 2^-32 P
        if (w1 == 0 && w0 < (1u << 19)) return 0.0;
        w2 = w1;
        w1 = w0;
        w0 = 0;
        ex -= 32;
        if (w2 == 0) {
            w2 = w1;
            w1 = 0;
            ex -= 32;
        }
    }
    const int n = __clz(w2);
    const unsigned long long top = ((unsigned long long)__funnelshift_l(w1, w2, n) << 32) | __funnelshift_l(w0, w1, n);
    unsigned long long m = __umul64hi(top, Pm);   // in [2^62, 2^64)
    int e = ex - n;                                // x = m 2^e
    const int s = (int)(m >> 63) ^ 1;
    m <<= s;
    e -= s;
    const int E = e + 63 + 1022;   // exponent field less one: the significand's leading bit adds it
    if (E < 1 || E > 2044) return oz_ll_scaled(sg ? -(long long)(m >> 1) : (long long)(m >> 1), e + 1);
    return __longlong_as_double((long long)(((m >> 11) + ((m >> 10) & 1ull) + ((unsigned long long)(unsigned)E << 52)) |
                                            ((unsigned long long)(sg & 0x80000000u) << 32)));
}

// Four consecutive elements of one row per thread: a 32-bit load of residue bytes per group, all issued first; the
// words of four groups are transposed into one word per element by eight byte permutes.
template <int NCH>
__device__ __forceinline__ void oz_crt_rows(const OzProb& P, const OzCrtParams& cp) {
    constexpr int NQ = NCH == 1 ? 5 : OZ_NQ;
    const unsigned(*ct)[OZ_FL] = NCH == 1 ? cp.c1 : cp.c2;
    const int* ci = NCH == 1 ? cp.i1 : cp.i2;
    const int G = cp.T * NCH, N = P.N;
    const unsigned nq = (unsigned)(N + 3) / 4, nunit = (unsigned)P.M * nq;
    const size_t MN = (size_t)P.M * P.ns;   // bytes of a group
    const bool v2 = (P.ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(P.C) & 15) == 0;
    for (unsigned u = blockIdx.x * blockDim.x + threadIdx.x; u < nunit; u += gridDim.x * blockDim.x) {
        const int i = (int)(u / nq), j0 = 4 * (int)(u - (unsigned)i * nq);
        const unsigned char* __restrict__ sp = P.stage + (size_t)i * P.ns + j0;
        unsigned int x[NQ][4];
#pragma unroll
        for (int g = 0; g < 4 * NQ; ++g) {
            x[g / 4][g & 3] = 0u;   // past the last group: the constants are zero
            if (g < G) x[g / 4][g & 3] = __ldg(reinterpret_cast<const unsigned int*>(sp + g * MN));
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const unsigned a = __byte_perm(x[q][0], x[q][1], 0x5140), b = __byte_perm(x[q][2], x[q][3], 0x5140);
            const unsigned c = __byte_perm(x[q][0], x[q][1], 0x7362), d = __byte_perm(x[q][2], x[q][3], 0x7362);
            x[q][0] = __byte_perm(a, b, 0x5410);
            x[q][1] = __byte_perm(a, b, 0x7632);
            x[q][2] = __byte_perm(c, d, 0x5410);
            x[q][3] = __byte_perm(c, d, 0x7632);
        }
        const int ea = (int)((__double_as_longlong(P.sa[i]) >> 52) & 0x7FF);   // row scales are powers of two
        double* crow = P.C + (size_t)i * P.ldc + j0;
#pragma unroll 1
        for (int h = 0; h < 4 && j0 + h < N; h += 2) {   // two elements a round (fully unrolled the kernel spills)
            unsigned acc[2][OZ_FL];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int l = 0; l < OZ_FL; ++l) acc[k][l] = (unsigned)ci[l];
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                if (NCH > 1 && 4 * q >= G) break;
#pragma unroll
                for (int l = 0; l < OZ_FL; ++l) {
                    acc[0][l] = __dp4a(x[q][0], ct[q][l], acc[0][l]);
                    acc[1][l] = __dp4a(x[q][1], ct[q][l], acc[1][l]);
                }
                x[q][0] = x[q][2];   // the next round's
                x[q][1] = x[q][3];
            }
            double v[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                int a[OZ_FL];
#pragma unroll
                for (int l = 0; l < OZ_FL; ++l) a[l] = (int)acc[k][l];
                const int eb = (int)((__double_as_longlong(P.sb[min(j0 + h + k, N - 1)]) >> 52) & 0x7FF);
                v[k] = (ea == 0x7FF || eb == 0x7FF) ? __longlong_as_double(0x7ff8000000000000ll)
                                                    : oz_frac_value(a, cp.Pm, ea + eb - 2046 + P.ealpha - 2 * P.nb + cp.Pe);
            }
            if (v2 && j0 + h + 1 < N) {
                *reinterpret_cast<double2*>(crow + h) = make_double2(v[0], v[1]);
            } else {
                crow[h] = v[0];
                if (j0 + h + 1 < N) crow[h + 1] = v[1];
            }
        }
    }
}

// C = alpha 2^(e_i + e_j - 2 nb) x for every element, x rebuilt from the staged residues.  The residues of
// an element are read once, coalesced, and C is written once.
// TWO: some problem has two K chunks (r = 64), whose twice as many residue words take the registers of two resident
// blocks; without, three.
template <bool TWO>
__global__ void __launch_bounds__(256, TWO ? 2 : 3) k_oz_crt(const OzBatch* __restrict__ bp,
                                                             const __grid_constant__ OzCrtParams cp) {
    const OzProb& P = bp->p[blockIdx.y];
    if (oz_skip(P)) return;
    if (!TWO || P.nch == 1) oz_crt_rows<1>(P, cp);
    else oz_crt_rows<2>(P, cp);
}

// The reconstruction launch of a plan.
static int oz_launch_crt(const OzBatch* host, const OzBatch* dev, int nsm, cudaStream_t st) {
    OzCrtParams cp;
    memset(&cp, 0, sizeof(cp));
    const OzMods& m = host->mods;
    cp.T = m.T;
    cp.Pm = m.Pm;
    cp.Pe = m.Pe;
    for (int t = 0; t < m.T; ++t) {
        const unsigned __int128 one = (unsigned __int128)1 << 88;
        const int p = oz_moduli[t];
        unsigned __int128 C = (one + p / 2) / p;
        for (int l = 0; l < OZ_FL; ++l, C >>= 8) {
            const unsigned byte = (unsigned)(C & 255);
            cp.c1[t / 4][l] |= byte << (8 * (t & 3));
            cp.i1[l] -= 128 * (int)byte;
            for (int c = 0; c < 2; ++c) {
                const int g = 2 * t + c;
                cp.c2[g / 4][l] |= byte << (8 * (g & 3));
                cp.i2[l] -= 128 * (int)byte;
            }
        }
    }
    bool two = false;
    for (int p = 0; p < host->nprob; ++p) two = two || host->p[p].nch > 1;
    if (two) k_oz_crt<true><<<dim3(2 * nsm, host->nprob), 256, 0, st>>>(dev, cp);
    else k_oz_crt<false><<<dim3(3 * nsm, host->nprob), 256, 0, st>>>(dev, cp);
    ACSE_CUDA_TRY(cudaGetLastError());
    return ACSE_OK;
}

// --------------------------------------------------------------------------- host plan
// Operands of the GEMMs of a pass (the products of acse_gemm_list_f64; S2 = r(r+1), P2 = r(r-1), P = P2 / 2):
//   A: W+ and W- (rows S2 and P2 for s = +1, P2 and S2 for s = -1), Wf1, M_ab, D_ab (r^2 x r^2),
//      [M_aa; D_aa], [M_bb; D_bb] packed (2P x P);
//   B: M+ (S2 x S2), M- (P2 x P2), Mf1, W_ab (r^2 x r^2), W_aa, W_bb packed (P x P).
// The problem table of s = +1 is the plan itself; that of s = -1 (`alt`) has the same operands with the
// other row counts and borrows every buffer.  The last three products are those of a D that is not pair-Hermitian: the
// first three A with B operands of their own (the 2P odd rows of M+, the 2S even ones of M-, the second flip of M),
// gated by Work::asym, their tiles behind all others in every list.
struct OzOp {
    __nv_bfloat16* sl;
    double* scale;
    int rows, K, Kp;
    int nb;             // rows rounded to X = round(a 2^(nb - e)), |X| <= 2^(nb-1)
};

struct OzPlan {
    OzBatch* host;
    OzBatch* dev;
    int S, bn;
    int bits;           // bits kept below a row's leading bit: min(6S, 53)
    unsigned __int128 P;   // product of the plan's moduli
    int pair;           // 1: CTA-pair kernel (256 x 256 tiles on clusters of two CTAs)
    int bm;             // rows of a tile: 128, or 256 with pairs
    int nclusters;      // co-resident CTA pairs (the persistent grid of the pair kernel)
    size_t smem;
    int nsm;
    int tiles;
    OzOp A[OZ_MAXP], B[OZ_MAXP];
    int* sched;         // tile lists of the persistent kernel (OzBatch::order, cta_start)
    int* err;
    struct OzPlan* alt;       // the pass's table for s = -1
    int borrowed;             // operands and staging belong to another plan
    struct OzPlan* lists[2];  // GEMM lists of the adjoint (oz_gemm_list): a plan per list slot
    int shareB[OZ_MAXP];      // lists: problem i reads the B operand of problem shareB[i] - 1 (0: its own)
};

static size_t oz_smem(int bn) { return (size_t)OZ_STAGES * (TC_BM + bn) * 128 + 1024 + 256; }
static size_t oz_smem_pair() { return (size_t)OZ2_STAGES * (TC_BM + OZ_BN / 2) * 128 + 1024 + 256; }

// Launch of the GEMM kernel of plan pl (pl->tiles > 0): one CTA per SM, or one cluster of two per pair.
static int oz_launch_gemm(const OzPlan* pl, cudaStream_t st) {
    if (pl->pair) {
        const int g = pl->tiles < pl->nclusters ? pl->tiles : pl->nclusters;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * g, 1, 1);
        cfg.blockDim = dim3(OZ_THREADS, 1, 1);
        cfg.dynamicSmemBytes = pl->smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        ACSE_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_gemm_oz<OZ_BN, OZ2_STAGES, true>, (const OzBatch*)pl->dev));
        return ACSE_OK;
    }
    const int g = pl->tiles < pl->nsm ? pl->tiles : pl->nsm;
    if (pl->bn == 256) k_gemm_oz<256, OZ_STAGES, false><<<g, OZ_THREADS, pl->smem, st>>>(pl->dev);
    else k_gemm_oz<128, OZ_STAGES, false><<<g, OZ_THREADS, pl->smem, st>>>(pl->dev);
    ACSE_CUDA_TRY(cudaGetLastError());
    return ACSE_OK;
}

// The moduli of a plan: the least T whose product P covers 4 Kmax 2^(2 bits) (every product of the plan
// then lies within P / 4 of zero), at most the whole list, and the exact constants of the set.
static int oz_mods_init(OzPlan* pl, int S, long long Kmax) {
    const int bt = 6 * S < 53 ? 6 * S : 53;
    if (Kmax < 1) Kmax = 1;
    if (Kmax > (1ll << 18)) return ACSE_ERR_SHAPE;
    pl->bits = bt;
    const unsigned __int128 need = (unsigned __int128)Kmax << (2 * bt + 2);   // below 2^126
    unsigned __int128 P = 1;
    int T = 0;
    while (T < OZ_NMOD && P < need) P *= (unsigned __int128)oz_moduli[T++];
    pl->P = P;
    OzMods& m = pl->host->mods;
    memset(&m, 0, sizeof(m));
    m.T = T;
    for (int t = 0; t < T; ++t) {
        const int pt = oz_moduli[t];
        const unsigned __int128 Q = P / (unsigned __int128)pt;
        const int qm = (int)(Q % (unsigned __int128)pt);
        int y = 1;
        while (y < pt && (qm * y) % pt != 1) ++y;   // pairwise coprime: the inverse exists
        m.p[t] = (float)pt;
        m.pinv[t] = 1.0f / (float)pt;
        for (int l = 0; l < 4; ++l) {
            const long long cl = (1ll << (14 * l)) % pt;
            m.cA[t][l] = (float)cl;
            m.cB[t][l] = (float)((cl * y) % pt);
        }
    }
    int bits = 0;
    while (bits < 127 && (P >> bits) > 1) ++bits;   // leading bit of P
    m.Pe = bits - 63;
    m.Pm = (unsigned long long)(m.Pe >= 0 ? P >> m.Pe : P << -m.Pe);
    return ACSE_OK;
}

// nb of an operand of contraction length K: the largest b <= bits with 4 K 2^(2b) <= P, plus one.
static int oz_op_nb(const OzPlan* pl, int K) {
    int b = pl->bits;
    while (b > 0 && ((unsigned __int128)K << (2 * b + 2)) > pl->P) --b;
    return b + 1;
}

static int oz_op_alloc(OzPlan* pl, OzOp& o, int rows, int K) {
    o.rows = rows;
    o.K = K;
    o.Kp = (K + 63) / 64 * 64;
    o.nb = oz_op_nb(pl, K);
    if (o.nb < 2) return ACSE_ERR_SHAPE;
    const size_t bytes = (size_t)rows * pl->host->mods.T * o.Kp * sizeof(__nv_bfloat16);
    if (cudaMalloc((void**)&o.sl, bytes) != cudaSuccess || cudaMalloc((void**)&o.scale, rows * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        return ACSE_ERR_NOMEM;
    }
    ACSE_CUDA_TRY(cudaMemset(o.sl, 0, bytes));   // the K padding of every segment stays zero
    return ACSE_OK;
}

// One problem C = alpha A B^T; its residue staging is `stage` (borrowed) or allocated here for stage_rows >= M
// rows.
static int oz_add(OzPlan* pl, const OzOp& a, const OzOp& b, double* C, int ldc, double alpha, int stage_rows,
                  unsigned char* stage) {
    OzBatch& B = *pl->host;
    if (B.nprob >= OZ_MAXP || a.K != b.K || a.Kp != b.Kp || a.nb != b.nb) return ACSE_ERR_SHAPE;
    const int n = B.nprob;
    const size_t ld = (size_t)B.mods.T * a.Kp;
    ACSE_TRY(tc_encode_map_bf16(&B.tmA[n], a.sl, a.rows, (int)ld, TC_BM, ld));
    ACSE_TRY(tc_encode_map_bf16(&B.tmB[n], b.sl, b.rows, (int)ld, pl->pair ? pl->bn / 2 : pl->bn, ld));
    OzProb& p = B.p[n];
    p.C = C;
    p.sa = a.scale;
    p.sb = b.scale;
    int ex = 0;
    if (frexp(alpha, &ex) != 0.5) return ACSE_ERR_ARG;   // alpha must be a power of two
    p.ealpha = ex - 1;
    p.M = a.rows;
    p.N = b.rows;
    p.ldc = ldc;
    p.ns = (p.N + 31) / 32 * 32;
    p.kbs = a.Kp / 64;
    p.nb = a.nb;
    // chunks of at most OZ_CHUNK_KB blocks: every partial sum of residue products stays below 2^24
    p.nch = (p.kbs + OZ_CHUNK_KB - 1) / OZ_CHUNK_KB;
    if (p.nch > OZ_MAXCH) return ACSE_ERR_SHAPE;
    p.cb = (p.kbs + p.nch - 1) / p.nch;
    p.ngroups = B.mods.T * p.nch;
    p.stage = stage;
    if (!stage && cudaMalloc((void**)&p.stage, (size_t)p.ngroups * stage_rows * p.ns) != cudaSuccess) {
        cudaGetLastError();
        p.stage = nullptr;
        return ACSE_ERR_NOMEM;
    }
    p.tiles_n = (p.N + pl->bn - 1) / pl->bn;
    p.tile_start = B.total_tiles;
    B.total_tiles += ((p.M + pl->bm - 1) / pl->bm) * p.tiles_n;
    B.nprob = n + 1;
    return ACSE_OK;
}

static int oz_plan_finish(OzPlan* pl);

// Kernel attributes, SM count, the moduli for the plan's longest contraction Kmax and the zeroed problem
// table of a plan.
static int oz_plan_init(OzPlan* pl, int S, int bn, int pair, long long Kmax) {
    pl->S = S;
    pl->bn = bn;
    pl->pair = pair && bn == OZ_BN;
    pl->bm = pl->pair ? 2 * TC_BM : TC_BM;
    pl->smem = pl->pair ? oz_smem_pair() : oz_smem(pl->bn);
    if (pl->pair)
        ACSE_CUDA_TRY(cudaFuncSetAttribute(k_gemm_oz<OZ_BN, OZ2_STAGES, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)pl->smem));
    else if (pl->bn == 256)
        ACSE_CUDA_TRY(cudaFuncSetAttribute(k_gemm_oz<256, OZ_STAGES, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)pl->smem));
    else
        ACSE_CUDA_TRY(cudaFuncSetAttribute(k_gemm_oz<128, OZ_STAGES, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)pl->smem));
    pl->nsm = 152;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&pl->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        pl->nsm = 152;
    }
    if (pl->pair) {   // co-resident clusters of two (the persistent grid)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * (pl->nsm / 2), 1, 1);
        cfg.blockDim = dim3(OZ_THREADS, 1, 1);
        cfg.dynamicSmemBytes = pl->smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, (void*)k_gemm_oz<OZ_BN, OZ2_STAGES, true>, &cfg) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = pl->nsm / 2;
        }
        pl->nclusters = n < pl->nsm / 2 ? n : pl->nsm / 2;
    }
    pl->host = (OzBatch*)calloc(1, sizeof(OzBatch));
    if (!pl->host) return ACSE_ERR_NOMEM;
    pl->host->wait_ns = OZ_WAIT_NS;
    return oz_mods_init(pl, S, Kmax);
}

// The plan figures of one GEMM, on the host only (acse_ozaki_plan_info in include/acse.h).
extern "C" int acse_ozaki_plan_info(int oz_slices, int kmax, int k, int* moduli_count, int* bits, int* chunks,
                                    int* moduli) {
    if (oz_slices < 4 || oz_slices > 10 || kmax < 1 || kmax > 8192 || k < 1 || k > kmax) return ACSE_ERR_ARG;
    OzPlan pl;
    memset(&pl, 0, sizeof(pl));
    pl.host = (OzBatch*)calloc(1, sizeof(OzBatch));
    if (!pl.host) return ACSE_ERR_NOMEM;
    const int st = oz_mods_init(&pl, oz_slices, kmax);
    if (st == ACSE_OK) {
        const int T = pl.host->mods.T, kbs = (k + 63) / 64;
        if (moduli_count) *moduli_count = T;
        if (bits) *bits = oz_op_nb(&pl, k) - 1;
        if (chunks) *chunks = (kbs + OZ_CHUNK_KB - 1) / OZ_CHUNK_KB;
        if (moduli)
            for (int t = 0; t < T; ++t) moduli[t] = oz_moduli[t];
    }
    free(pl.host);
    return st;
}

// The ten products of a pass in the order of acse_gemm_list_f64 (the same-spin X and Y as one problem).
static int oz_pass_table(acse_ctx* c, OzPlan* pl, const OzPlan* root, int sW) {
    Work& w = c->w;
    const int r = c->r, R2 = r * r, S2 = r * (r + 1), P2 = r * (r - 1), P = P2 / 2;
    const bool own = pl == root;
    auto add = [&](int i, const OzOp& A, const OzOp& B, double* C, int ldc, double alpha, int stage_rows) {
        return oz_add(pl, A, B, C, ldc, alpha, stage_rows, own ? nullptr : root->host->p[i].stage);
    };
    ACSE_TRY(add(0, pl->A[0], pl->B[0], w.V1, 2 * R2, 1.0, S2));
    ACSE_TRY(add(1, pl->A[2], pl->B[2], w.V5f1, R2, 1.0, R2));
    ACSE_TRY(add(2, pl->A[3], pl->B[3], w.X[1], R2, 2.0, R2));
    ACSE_TRY(add(3, pl->A[4], pl->B[3], w.Y[1], R2, 2.0, R2));
    ACSE_TRY(add(4, pl->A[1], pl->B[1], ph_V2(c, sW), 2 * R2, 1.0, S2));
    ACSE_TRY(add(5, pl->A[5], pl->B[4], w.Cp[0], P, 2.0, 2 * P));
    ACSE_TRY(add(6, pl->A[6], pl->B[5], w.Cp[1], P, 2.0, 2 * P));
    ACSE_TRY(add(7, pl->A[0], pl->B[6], w.V1 + S2, 2 * R2, 1.0, S2));
    ACSE_TRY(add(8, pl->A[1], pl->B[7], ph_V2(c, sW) + P2, 2 * R2, 1.0, S2));
    ACSE_TRY(add(9, pl->A[2], pl->B[8], w.Vf2, R2, 1.0, R2));
    for (int i = 7; i < 10; ++i) pl->host->p[i].gate = w.asym;
    return oz_plan_finish(pl);
}

int oz_plan_create(acse_ctx* c) {
    OzPlan* pl = (OzPlan*)calloc(1, sizeof(OzPlan));
    if (!pl) return ACSE_ERR_NOMEM;
    c->oz_plan = pl;
    const int r = c->r, R2 = r * r, S2 = r * (r + 1), P2 = r * (r - 1), P = P2 / 2;
    const int bn = R2 >= 256 ? OZ_BN : 128, pair = c->opt.gemm_tile != 1;
    ACSE_TRY(oz_plan_init(pl, c->opt.oz_slices, bn, pair, S2));
    ACSE_TRY(oz_op_alloc(pl, pl->A[0], S2, S2));
    ACSE_TRY(oz_op_alloc(pl, pl->A[1], S2, P2));
    for (int i = 2; i < 5; ++i) ACSE_TRY(oz_op_alloc(pl, pl->A[i], R2, R2));
    for (int i = 5; i < 7; ++i) ACSE_TRY(oz_op_alloc(pl, pl->A[i], 2 * P, P));
    ACSE_TRY(oz_op_alloc(pl, pl->B[0], S2, S2));
    ACSE_TRY(oz_op_alloc(pl, pl->B[1], P2, P2));
    for (int i = 2; i < 4; ++i) ACSE_TRY(oz_op_alloc(pl, pl->B[i], R2, R2));
    for (int i = 4; i < 6; ++i) ACSE_TRY(oz_op_alloc(pl, pl->B[i], P, P));
    ACSE_TRY(oz_op_alloc(pl, pl->B[6], P2, S2));
    ACSE_TRY(oz_op_alloc(pl, pl->B[7], S2, P2));
    ACSE_TRY(oz_op_alloc(pl, pl->B[8], R2, R2));
    if (cudaMalloc((void**)&pl->err, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return ACSE_ERR_NOMEM;
    }
    ACSE_CUDA_TRY(cudaMemset(pl->err, 0, sizeof(int)));
    if (!c->w.tc_err) c->w.tc_err = pl->err;   // read by acse_sync_status
    pl->host->err = pl->err;
    pl->A[1].rows = P2;   // s = +1: W+ over S2 rows, W- over P2
    ACSE_TRY(oz_pass_table(c, pl, pl, +1));
    OzPlan* alt = (OzPlan*)calloc(1, sizeof(OzPlan));
    if (!alt) return ACSE_ERR_NOMEM;
    pl->alt = alt;
    alt->borrowed = 1;
    ACSE_TRY(oz_plan_init(alt, c->opt.oz_slices, bn, pair, S2));
    alt->host->err = pl->err;
    memcpy(alt->A, pl->A, sizeof(pl->A));
    memcpy(alt->B, pl->B, sizeof(pl->B));
    alt->A[0].rows = P2;   // s = -1: the other way round
    alt->A[1].rows = S2;
    return oz_pass_table(c, alt, pl, -1);
}

// Longest-processing-time tile lists of the persistent kernel (tile cost: its K blocks over all groups)
// and the device copy of the problem table.
static int oz_plan_finish(OzPlan* pl) {
    OzBatch& B = *pl->host;
    pl->tiles = B.total_tiles;
    if (pl->tiles > 0) {
        const int units = pl->pair ? pl->nclusters : pl->nsm;   // CTAs, or CTA pairs, of the persistent grid
        const int T = pl->tiles, G = T < units ? T : units;
        std::vector<long long> cost(T), load(G, 0);
        int Tn = 0;   // tiles that are not gated (those of the first problems)
        for (int p = 0; p < B.nprob; ++p) {
            const int n = ((B.p[p].M + pl->bm - 1) / pl->bm) * B.p[p].tiles_n;
            for (int k = 0; k < n; ++k) cost[B.p[p].tile_start + k] = (long long)B.mods.T * B.p[p].kbs + 4 * B.p[p].ngroups;
            if (!B.p[p].gate) Tn += n;
        }
        // the lists of the ungated tiles, then the gated ones onto the least loaded (at a cost of nothing they piled up
        // on the shortest lists: r = 64, a D that is not pair-Hermitian 62 ms in place of 20.8)
        std::vector<int> first(Tn), start(G + 1), extra(T - Tn), hs(T + G + 1);
        tc_lpt_schedule(cost.data(), Tn, G, first.data(), start.data());
        std::vector<std::vector<int>> lists(G);
        for (int c = 0; c < G; ++c)
            for (int k = start[c]; k < start[c + 1]; ++k) {
                lists[c].push_back(first[k]);
                load[c] += cost[first[k]];
            }
        for (int k = 0; k < T - Tn; ++k) extra[k] = Tn + k;
        std::stable_sort(extra.begin(), extra.end(), [&](int a, int b) { return cost[a] > cost[b]; });
        for (int t : extra) {
            const int c = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            lists[c].push_back(t);
            load[c] += cost[t];
        }
        int q = 0;
        for (int c = 0; c < G; ++c) {
            hs[T + c] = q;
            for (int t : lists[c]) hs[q++] = t;
        }
        hs[T + G] = q;
        const bool ok = cudaMalloc((void**)&pl->sched, (size_t)(T + G + 1) * sizeof(int)) == cudaSuccess &&
                        cudaMemcpy(pl->sched, hs.data(), (size_t)(T + G + 1) * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            return ACSE_ERR_NOMEM;
        }
        B.order = pl->sched;
        B.cta_start = pl->sched + T;
    }
    if (cudaMalloc((void**)&pl->dev, sizeof(OzBatch)) != cudaSuccess) {
        cudaGetLastError();
        return ACSE_ERR_NOMEM;
    }
    ACSE_CUDA_TRY(cudaMemcpy(pl->dev, pl->host, sizeof(OzBatch), cudaMemcpyHostToDevice));
    return ACSE_OK;
}

static void oz_plan_free(OzPlan* pl) {
    if (!pl) return;
    oz_plan_free(pl->alt);
    for (int s = 0; s < 2; ++s) oz_plan_free(pl->lists[s]);
    for (int i = 0; i < OZ_MAXP && !pl->borrowed; ++i) {
        if (pl->A[i].sl) cudaFree(pl->A[i].sl);
        if (pl->A[i].scale) cudaFree(pl->A[i].scale);
        if (pl->shareB[i]) continue;   // an earlier problem's operand
        if (pl->B[i].sl) cudaFree(pl->B[i].sl);
        if (pl->B[i].scale) cudaFree(pl->B[i].scale);
    }
    if (pl->sched) cudaFree(pl->sched);
    if (pl->err) cudaFree(pl->err);
    if (pl->host && !pl->borrowed)
        for (int i = 0; i < pl->host->nprob; ++i)
            if (pl->host->p[i].stage) cudaFree(pl->host->p[i].stage);
    if (pl->dev) cudaFree(pl->dev);
    free(pl->host);
    free(pl);
}

void oz_plan_destroy(acse_ctx* c) {
    OzPlan* pl = (OzPlan*)c->oz_plan;
    if (!pl) return;
    if (pl->err && c->w.tc_err == pl->err) c->w.tc_err = nullptr;
    oz_plan_free(pl);
    c->oz_plan = nullptr;
}

// The moduli constants of a slicing launch.
static void oz_slice_batch_init(OzSliceBatch& b, const OzMods& m) {
    memset(&b, 0, sizeof(b));
    b.T = m.T;
    for (int t = 0; t < m.T; ++t) {
        b.p[t] = m.p[t];
        b.pinv[t] = m.pinv[t];
        for (int l = 0; l < 4; ++l) {
            b.cA[t][l] = m.cA[t][l];
            b.cB[t][l] = m.cB[t][l];
        }
    }
}

// One slicing job: `rows` rows of operand o starting at output row `orow`, read from src (row stride
// lds) through the optional row / column maps; mul_y for a B operand (residues times y_t).
static void oz_job(OzSliceBatch& b, int& rows, const OzOp& o, int orow, int nrows, const double* src, size_t lds,
                   const int* rowmap, const int* colmap, int mul_y) {
    OzSliceJob& j = b.j[b.njobs++];
    j.src = src;
    j.lds = lds;
    j.rowmap = rowmap;
    j.colmap = colmap;
    j.ldd = (size_t)b.T * o.Kp;
    j.dst = o.sl + (size_t)orow * j.ldd;
    j.scale = o.scale + orow;
    j.rows = nrows;
    j.K = o.K;
    j.Kp = o.Kp;
    j.nb = o.nb;
    j.mul_y = mul_y;
    j.row0 = rows;
    rows += nrows;
}

// Launch the slicing of every job of `all`: the row scales (a warp per row), then the residues (a
// block row per operand row, 1024 elements a block).
static int oz_slice_launch(acse_ctx* c, const OzSliceBatch& all, int rows) {
    if (all.njobs == 0 || rows == 0) return ACSE_OK;
    if (rows > 65535) return ACSE_ERR_SHAPE;
    k_oz_rowscale<<<(rows + 7) / 8, 256, 0, c->stream>>>(all, rows);
    ACSE_LAUNCHED(c);
    int maxq = 1;
    for (int i = 0; i < all.njobs; ++i) maxq = (all.j[i].K + 3) / 4 > maxq ? (all.j[i].K + 3) / 4 : maxq;
    k_oz_residue<<<dim3((maxq + 255) / 256, rows), 256, 0, c->stream>>>(all);
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}

int oz_slice_operands(acse_ctx* c, int prep_D, int sW) {
    OzPlan* root = (OzPlan*)c->oz_plan;
    if (!root) return ACSE_ERR_UNSUPPORTED;
    const OzPlan* pl = sW > 0 ? root : root->alt;
    const int r = c->r, P = r * (r - 1) / 2, R2 = r * r, S2 = r * (r + 1), P2 = 2 * P;
    Work& w = c->w;
    OzSliceBatch b;
    oz_slice_batch_init(b, pl->host->mods);
    int rows = 0;
    const int* pm = w.pmap;
    // A residues as they are, B residues times y_t
    if (prep_D) {
        oz_job(b, rows, pl->A[5], 0, P, w.M[0], R2, pm, pm, 0);
        oz_job(b, rows, pl->A[5], P, P, c->cur_D[0], R2, pm, pm, 0);
        oz_job(b, rows, pl->A[3], 0, R2, w.M[1], R2, nullptr, nullptr, 0);
        oz_job(b, rows, pl->A[4], 0, R2, c->cur_D[1], R2, nullptr, nullptr, 0);
        oz_job(b, rows, pl->A[6], 0, P, w.M[2], R2, pm, pm, 0);
        oz_job(b, rows, pl->A[6], P, P, c->cur_D[2], R2, pm, pm, 0);
        oz_job(b, rows, pl->B[0], 0, S2, w.Mp, S2, nullptr, nullptr, 1);
        oz_job(b, rows, pl->B[1], 0, P2, w.Mm, P2, nullptr, nullptr, 1);
        oz_job(b, rows, pl->B[2], 0, R2, w.Mf1, R2, nullptr, nullptr, 1);
        OzSliceBatch gb;
        oz_slice_batch_init(gb, pl->host->mods);
        int grows = 0;
        oz_job(gb, grows, pl->B[6], 0, P2, w.Mp + (size_t)S2 * S2, S2, nullptr, nullptr, 1);
        oz_job(gb, grows, pl->B[7], 0, S2, w.Mm + (size_t)P2 * P2, P2, nullptr, nullptr, 1);
        oz_job(gb, grows, pl->B[8], 0, R2, w.Mf2, R2, nullptr, nullptr, 1);
        k_oz_slice_gated<<<4 * root->nsm, 256, 0, c->stream>>>(gb, grows, w.asym);
        ACSE_LAUNCHED(c);
    }
    oz_job(b, rows, pl->B[3], 0, R2, c->cur_W[1], R2, nullptr, nullptr, 1);
    oz_job(b, rows, pl->B[4], 0, P, c->cur_W[0], R2, pm, pm, 1);
    oz_job(b, rows, pl->B[5], 0, P, c->cur_W[2], R2, pm, pm, 1);
    oz_job(b, rows, pl->A[0], 0, pl->A[0].rows, w.Wp, S2, nullptr, nullptr, 0);
    oz_job(b, rows, pl->A[1], 0, pl->A[1].rows, w.Wm, P2, nullptr, nullptr, 0);
    oz_job(b, rows, pl->A[2], 0, R2, w.Wf1, R2, nullptr, nullptr, 0);
    return oz_slice_launch(c, b, rows);
}

int oz_gemm_launch(acse_ctx* c, int sW) {
    OzPlan* root = (OzPlan*)c->oz_plan;
    if (!root) return ACSE_ERR_UNSUPPORTED;
    const OzPlan* pl = sW > 0 ? root : root->alt;
    if (pl->tiles == 0) return ACSE_OK;
    ACSE_TRY(prof_begin(c));
    ACSE_TRY(oz_launch_gemm(pl, c->stream));
    ACSE_LAUNCHED(c);
    ACSE_TRY(oz_launch_crt(pl->host, pl->dev, pl->nsm, c->stream));
    ACSE_LAUNCHED(c);
    return prof_end(c);
}

int oz_set_wait_ns(acse_ctx* c, unsigned long long ns, int inject_stall) {
    OzPlan* pl = (OzPlan*)c->oz_plan;
    if (!pl) return ACSE_ERR_UNSUPPORTED;
    ACSE_CUDA_TRY(cudaStreamSynchronize(c->stream));
    for (OzPlan* q : {pl, pl->alt}) {
        q->host->wait_ns = ns ? ns : OZ_WAIT_NS;
        q->host->inject_stall = inject_stall;
        ACSE_CUDA_TRY(cudaMemcpy(q->dev, q->host, sizeof(OzBatch), cudaMemcpyHostToDevice));
    }
    return ACSE_OK;
}

// ------------------------------------------------------------------ GEMM lists of the adjoint
// The reverse sweep's FP64 GEMMs (acse_adjoint.cu) of an Ozaki context run through the same kernels: any
// list of up to OZ_MAXP GEMMs C = alpha A B^T, alpha a power of two, both operands K-major, B possibly through
// a pair map; problems with the same B share its residues.  One plan per list slot, built on the first call
// (its slices and residue staging stay until the context is destroyed); a later call whose shapes differ
// from the slot's plan is refused (ACSE_ERR_SHAPE).
static int oz_list_create(OzPlan* root, const GemmF64* g, int n, OzPlan** out) {
    OzPlan* pl = (OzPlan*)calloc(1, sizeof(OzPlan));
    if (!pl) return ACSE_ERR_NOMEM;
    *out = pl;
    int maxN = 0;
    for (int i = 0; i < n; ++i) maxN = g[i].N > maxN ? g[i].N : maxN;
    long long maxK = 1;
    for (int i = 0; i < n; ++i) maxK = g[i].K > maxK ? g[i].K : maxK;
    ACSE_TRY(oz_plan_init(pl, root->S, maxN >= 256 ? OZ_BN : 128, root->pair, maxK));
    pl->host->err = root->err;
    for (int i = 0; i < n; ++i) {
        for (int k = 0; k < i && !pl->shareB[i]; ++k)
            if (!pl->shareB[k] && g[k].B == g[i].B && g[k].N == g[i].N && g[k].K == g[i].K && g[k].mapB == g[i].mapB)
                pl->shareB[i] = k + 1;
        ACSE_TRY(oz_op_alloc(pl, pl->A[i], g[i].M, g[i].K));
        if (!pl->shareB[i]) ACSE_TRY(oz_op_alloc(pl, pl->B[i], g[i].N, g[i].K));
        else pl->B[i] = pl->B[pl->shareB[i] - 1];
        ACSE_TRY(oz_add(pl, pl->A[i], pl->B[i], g[i].C, g[i].ldc, g[i].alpha, g[i].M, nullptr));
    }
    return oz_plan_finish(pl);
}

int oz_gemm_list(acse_ctx* c, const GemmF64* g, int n, int slot) {
    OzPlan* root = (OzPlan*)c->oz_plan;
    if (!root || slot < 0 || slot > 1 || n < 1 || n > OZ_MAXP) return ACSE_ERR_UNSUPPORTED;
    for (int i = 0; i < n; ++i) {
        int ex = 0;
        if (frexp(g[i].alpha, &ex) != 0.5 || g[i].mapA) return ACSE_ERR_ARG;
    }
    if (!root->lists[slot]) {
        const int s = oz_list_create(root, g, n, &root->lists[slot]);
        if (s != ACSE_OK) {
            oz_plan_free(root->lists[slot]);
            root->lists[slot] = nullptr;
            return s;
        }
    }
    OzPlan* pl = root->lists[slot];
    OzBatch& B = *pl->host;
    if (B.nprob != n) return ACSE_ERR_SHAPE;
    for (int i = 0; i < n; ++i) {
        if (B.p[i].M != g[i].M || B.p[i].N != g[i].N || pl->A[i].K != g[i].K) return ACSE_ERR_SHAPE;
        const int k = pl->shareB[i] - 1;
        if (k >= 0 && (g[k].B != g[i].B || g[k].ldb != g[i].ldb || g[k].mapB != g[i].mapB)) return ACSE_ERR_SHAPE;
    }
    // residues of every operand (B times y_t), at most OZ_MAXJ jobs a launch
    OzSliceBatch sb;
    oz_slice_batch_init(sb, B.mods);
    int rows = 0;
    for (int i = 0; i < n; ++i) {
        for (int side = 0; side < 2; ++side) {
            if (side && pl->shareB[i]) continue;
            const OzOp& o = side ? pl->B[i] : pl->A[i];
            const int* map = side ? g[i].mapB : nullptr;
            oz_job(sb, rows, o, 0, o.rows, side ? g[i].B : g[i].A, (size_t)(side ? g[i].ldb : g[i].lda), map, map, side);
            if (sb.njobs == OZ_MAXJ) {
                ACSE_TRY(oz_slice_launch(c, sb, rows));
                oz_slice_batch_init(sb, B.mods);
                rows = 0;
            }
        }
    }
    ACSE_TRY(oz_slice_launch(c, sb, rows));
    // this call's outputs and scales
    for (int i = 0; i < n; ++i) {
        OzProb& p = B.p[i];
        int ex = 0;
        frexp(g[i].alpha, &ex);
        p.C = g[i].C;
        p.ldc = g[i].ldc;
        p.ealpha = ex - 1;
    }
    B.wait_ns = root->host->wait_ns;
    B.inject_stall = root->host->inject_stall;
    ACSE_CUDA_TRY(cudaMemcpyAsync(pl->dev, pl->host, sizeof(OzBatch), cudaMemcpyHostToDevice, c->stream));
    if (pl->tiles == 0) return ACSE_OK;
    ACSE_TRY(oz_launch_gemm(pl, c->stream));
    ACSE_LAUNCHED(c);
    ACSE_TRY(oz_launch_crt(&B, pl->dev, pl->nsm, c->stream));
    ACSE_LAUNCHED(c);
    return ACSE_OK;
}
