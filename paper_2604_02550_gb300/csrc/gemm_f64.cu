// FP64 grouped "NT" GEMM on the DFMA pipe:  C = alpha * A . B^T, A and B K-major.
//
// One launch runs every tile of up to GEMM_F64_MAXP problems (the sector GEMMs of one contraction pass).
// GB300 issues two DFMA per clock and SM, so the kernel is bound by that pipe at any tile size: a warp's
// DFMA takes 16 cycles of it, and one shared-memory operand load per DFMA still leaves the load units
// mostly idle.  What the tile size decides is the balance: a 64 x 64 tile of K = 392 holds its SM for
// 0.4 ms, and the 165 such tiles of a pass at r = 14 took two of them (0.54 ms against 0.19 ms of DFMA
// work).  So the tiles are small: 32 x 32 (2 x 2 outputs a thread) where every SM gets at least
// GF_TILES_PER_SM of them, else 16 x 16 (one output a thread).
#include "acse_internal.h"

#define GEMM_F64_MAXP 54
#define GF_TPB 256
// 32 x 32 tiles from this many per SM on: the last wave then idles at most a sixteenth of the launch, while
// at r = 20 (6.5 a SM) 16 x 16 tiles finish earlier.
#define GF_TILES_PER_SM 16

struct GemmF64Batch {
    GemmF64 p[GEMM_F64_MAXP];
    int prefix[GEMM_F64_MAXP + 1];
    int tiles_n[GEMM_F64_MAXP];
    int nprob;
};

template <int BT>   // tile BT x BT, K blocks of 512 / BT: two elements of each operand a thread
__global__ void __launch_bounds__(GF_TPB) k_gemm_f64(const __grid_constant__ GemmF64Batch b) {
    constexpr int BK = 512 / BT, RT = BT / 16;   // RT x RT outputs a thread
    const int t = blockIdx.x;
    int pi = 0;
    while (pi + 1 < b.nprob && b.prefix[pi + 1] <= t) ++pi;
    const GemmF64& P = b.p[pi];
    if (P.gate && !*P.gate) return;
    const int local = t - b.prefix[pi];
    const int m0 = (local / b.tiles_n[pi]) * BT;
    const int n0 = (local % b.tiles_n[pi]) * BT;

    __shared__ double As[BK][BT + 1];
    __shared__ double Bs[BK][BT + 1];

    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double acc[RT][RT];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < RT; ++j) acc[i][j] = 0.0;

    const int M = P.M, N = P.N, K = P.K;
    const int* __restrict__ mapA = P.mapA;
    const int* __restrict__ mapB = P.mapB;
    // this thread's two elements of an operand block: rows row and row + BT / 2, K offset kq
    const int row = tid / BK, kq = tid % BK;
    const double* asrc[2];
    const double* bsrc[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int m = m0 + row + u * (BT / 2), n = n0 + row + u * (BT / 2);
        asrc[u] = m < M ? P.A + (size_t)(mapA ? mapA[m] : m) * P.lda : nullptr;
        bsrc[u] = n < N ? P.B + (size_t)(mapB ? mapB[n] : n) * P.ldb : nullptr;
    }
    double av[2], bv[2];
    auto load = [&](int k0) {
        const int k = k0 + kq;
        const bool kok = k < K;
        const int ka = mapA && kok ? mapA[k] : k, kb = mapB && kok ? mapB[k] : k;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            av[u] = asrc[u] && kok ? asrc[u][ka] : 0.0;
            bv[u] = bsrc[u] && kok ? bsrc[u][kb] : 0.0;
        }
    };
    load(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            As[kq][row + u * (BT / 2)] = av[u];
            Bs[kq][row + u * (BT / 2)] = bv[u];
        }
        __syncthreads();
        if (k0 + BK < K) load(k0 + BK);   // in flight during the products
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[RT], c[RT];
#pragma unroll
            for (int i = 0; i < RT; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < RT; ++j) c[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < RT; ++j) acc[i][j] = fma(a[i], c[j], acc[i][j]);
        }
        __syncthreads();
    }
    const double alpha = P.alpha;
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const int m = m0 + ty + 16 * i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < RT; ++j) {
            const int n = n0 + tx + 16 * j;
            if (n >= N) continue;
            P.C[(size_t)m * P.ldc + n] = alpha * acc[i][j];
        }
    }
}

int gemm_f64_grouped(acse_ctx* c, const GemmF64* probs, int nprob, cudaStream_t s) {
    int done = 0;
    while (done < nprob) {
        GemmF64Batch b;
        int np = nprob - done;
        if (np > GEMM_F64_MAXP) np = GEMM_F64_MAXP;
        long t32 = 0;
        for (int i = 0; i < np; ++i)   // (gated products are rare)
            if (!probs[done + i].gate) t32 += (long)((probs[done + i].M + 31) / 32) * ((probs[done + i].N + 31) / 32);
        const int bt = t32 >= (long)GF_TILES_PER_SM * 152 ? 32 : 16;
        int tiles = 0;
        int used = 0;
        for (int i = 0; i < np; ++i) {
            const GemmF64& q = probs[done + i];
            if (q.M <= 0 || q.N <= 0) continue;
            b.p[used] = q;
            b.prefix[used] = tiles;
            b.tiles_n[used] = (q.N + bt - 1) / bt;
            tiles += ((q.M + bt - 1) / bt) * b.tiles_n[used];
            ++used;
        }
        b.prefix[used] = tiles;
        b.nprob = used;
        if (tiles > 0) {
            ACSE_TRY(prof_begin(c));
            if (bt == 32) k_gemm_f64<32><<<tiles, GF_TPB, 0, s>>>(b);
            else k_gemm_f64<16><<<tiles, GF_TPB, 0, s>>>(b);
            ACSE_LAUNCHED(c);
            ACSE_TRY(prof_end(c));
        }
        done += np;
    }
    return ACSE_OK;
}
