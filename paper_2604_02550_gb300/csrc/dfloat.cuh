// Element types of the FP64-accurate O(r^5) kernels on the CUDA cores: double, and the double-float pair
// the Ozaki path uses where its products do not run on the tensor cores.
#pragma once

// 4 consecutive elements of a shared array (16-byte aligned: offsets are multiples of 4 elements).
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    const double2 y = *reinterpret_cast<const double2*>(p + 2);
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}

// Double-float: an FP64 value carried as the unevaluated sum h + l of two floats (about 48 significant
// bits).  The Ozaki path runs its O(r^5) products in it: FP32 arithmetic is many times faster than
// FP64 on this GPU.  The all-zero bit pattern is 0.
struct __align__(8) dfl {
    float h, l;
    __device__ __forceinline__ operator double() const { return (double)h + (double)l; }
};
// h = x rounded to the nearest float (ties to even), l = x - h rounded to the nearest float.  With integer
// operations from the bit pattern where x is a normal double whose h and l are normal floats (the FP64
// conversions run on the slow FP64 pipe); the same values through FP64 otherwise.
__device__ __forceinline__ dfl to_dfl(double x) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(bits >> 32), lo = (unsigned)bits;
    const int e = (int)((hi >> 20) & 0x7FFu);
    if (e >= 949 && e <= 1149) {   // 2^(e - 1075) and h are normal floats
        const unsigned sign = hi & 0x80000000u;
        const unsigned m23 = ((hi & 0xFFFFFu) << 3) | (lo >> 29);    // the 23 fraction bits kept
        const unsigned rem = lo & 0x1FFFFFFFu;                        // the 29 dropped ones
        const unsigned up = (rem > 0x10000000u || (rem == 0x10000000u && (m23 & 1u))) ? 1u : 0u;
        const float h = __uint_as_float(sign | (((unsigned)(e - 1023 + 127) << 23) + m23 + up));
        const int rr = up ? (int)rem - 0x20000000 : (int)rem;        // x - h in units of 2^(e - 1075)
        const float scale = __uint_as_float((unsigned)(e - 1075 + 127) << 23);
        const float l = __fmul_rn(__int2float_rn(sign ? -rr : rr), scale);
        return dfl{h, l};
    }
    const float h = (float)x;
    return dfl{h, (float)(x - (double)h)};   // x - h is exact in FP64
}
// acc += a b: the rounding error of the product by FMA (the l.l term is dropped), that of the sum by
// Knuth's TwoSum; both go to acc.l.
__device__ __forceinline__ void df_mac(dfl& acc, const dfl& a, const dfl& b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
    const float s = acc.h + p;
    const float bb = s - acc.h;
    const float t = (acc.h - (s - bb)) + (p - bb);
    acc.h = s;
    acc.l += t + e;
}
__device__ __forceinline__ void ld4(const dfl* p, dfl (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    const float4 y = *reinterpret_cast<const float4*>(p + 2);
    v[0] = dfl{x.x, x.y}; v[1] = dfl{x.z, x.w}; v[2] = dfl{y.x, y.y}; v[3] = dfl{y.z, y.w};
}
// conversions and multiply-add for the element types of the tiled kernels
template <typename T> __device__ __forceinline__ T tconv(double x) { return (T)x; }
template <> __device__ __forceinline__ dfl tconv<dfl>(double x) { return to_dfl(x); }
template <typename T> __device__ __forceinline__ void tmac(T& acc, const T& a, const T& b) { acc += a * b; }
template <> __device__ __forceinline__ void tmac<dfl>(dfl& acc, const dfl& a, const dfl& b) { df_mac(acc, a, b); }

