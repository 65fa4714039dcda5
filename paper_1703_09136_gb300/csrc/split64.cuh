// Numbers as signed base-512 digits in f16 (see split64.cu): exponents,
// fixed-point words with biased digit fields, digit pairs, and the FP32
// mma.sync that sums digit products without rounding.
#pragma once
#include <utility>

#include "common.cuh"

constexpr int S6_NONE = -(1 << 24);      // exponent of an all-zero level (or below)
constexpr int S6_NAN = 1 << 20;          // exponent of a level with an infinity or a NaN

// D digits: 9 D - 1 bits; the bias 256 sum_{i = 0 .. D - 2} 512^i makes the low D - 1
// fields of a word digit + 256
template <int D>
__host__ __device__ constexpr long long s6_bias() {
    long long b = 0;
    for (int i = 0; i < D - 1; ++i) b = (b << 9) + 256;
    return b;
}

// largest E with |v 2^shift| < 2^E (S6_NONE for zero)
__device__ __forceinline__ int s6_exponent(double v, int shift) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 2047);
    if (e == 2047) return S6_NAN;
    if (e == 0) {                                         // m 2^-1074
        const long long m = b & 0xfffffffffffffll;
        return m ? -1010 - __clzll(m) + shift : S6_NONE;
    }
    return e - 1022 + shift;
}
__device__ __forceinline__ int s6_exponent(float v, int shift) {
    const int b = __float_as_int(v), e = (b >> 23) & 255;
    if (e == 255) return S6_NAN;
    if (e == 0) return (b & 0x7fffff) ? -125 + shift : S6_NONE;
    return e - 126 + shift;
}

// v 2^shift 2^(BITS - E) rounded to an integer, |v 2^shift| < 2^E (BITS <= 62; floats: BITS >= 24)
template <int BITS>
__device__ __forceinline__ long long s6_fixed(double v, int shift, int E) {
    const long long b = __double_as_longlong(v);
    int e = (int)((b >> 52) & 2047);
    unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
    if (e) m |= 1ull << 52; else e = 1;
    const int s = E - shift - e + 1075 - BITS;            // right shift
    if (s > 0) m = s > 54 ? 0ull : (m + (1ull << (s - 1))) >> s;
    else m <<= min(-s, BITS - 2);                         // subnormals, and more bits than a double has
    return b < 0 ? -(long long)m : (long long)m;
}
template <int BITS>
__device__ __forceinline__ long long s6_fixed(float v, int shift, int E) {
    const int b = __float_as_int(v);
    int e = (b >> 23) & 255;
    unsigned m = (unsigned)b & 0x7fffffu;
    if (e) m |= 1u << 23; else e = 1;
    const int s = E - shift - e + 150 - BITS;             // right shift, at least 24 - BITS
    if (s > 0) m = s > 25 ? 0u : (m + (1u << (s - 1))) >> s;
    else m <<= min(-s, BITS - 24);
    return b < 0 ? -(long long)m : (long long)m;
}

// field of digit i (0 = most significant) of a biased word, digit + 256 in [0, 512]
template <int D>
__device__ __forceinline__ unsigned s6_field(long long xb, int i) {
    return i == 0 ? (unsigned)((int)(xb >> (9 * (D - 1))) + 256) : (unsigned)(xb >> (9 * (D - 1 - i))) & 511u;
}

// two digits as f16 (1024 + field as bits 0x6400 | field, minus 1280)
__device__ __forceinline__ unsigned s6_half2(unsigned f0, unsigned f1) {
    unsigned h = 0x64006400u + (f0 | (f1 << 16)), r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x65006500u));
    return r;
}

// 2^e as a double (0 below the subnormals, infinite above the range)
__device__ __forceinline__ double pow2d(int e) {
    const long long b = e > 1023 ? 0x7ff0000000000000ll : e >= -1022 ? (long long)(e + 1023) << 52
                        : e >= -1074 ? 1ll << (e + 1074) : 0ll;
    return __longlong_as_double(b);
}

// x 2^e for any e (a product with one power of two loses digits where that power alone is subnormal or infinite)
__device__ __forceinline__ double scale2d(double x, int e) {
    const int f = max(-1000, min(1000, e));
    x *= pow2d(f);
    return e == f ? x : x * pow2d(e - f);
}

// an integer below 2^51 in magnitude as a double: one FP64 addition
__device__ __forceinline__ double int51d(long long x) {
    return __longlong_as_double(0x4338000000000000ll + x) - 6755399441055744.0;   // 1.5 2^52
}

__device__ __forceinline__ void s6_mma(float (&c)[4], const uint4& a, const uint2& b) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// 16-byte asynchronous copy to shared memory (zeros where !ok), its commit, and
// the wait until at most N committed groups are in flight
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Programmatic dependent launch: a kernel lets the next one of its stream start (it
// only prepares) and waits for the kernels before it before it reads their results.
__device__ __forceinline__ void pdl_start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch of a kernel that calls pdl_wait() before its first read of earlier results;
// pdl = false: an ordinary launch of it.
template <class... P, class... A>
inline cudaError_t pdl_launch_if(bool pdl, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 unsigned cluster, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <class... P, class... A>
inline cudaError_t pdl_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, unsigned cluster,
                              A&&... args) {
    return pdl_launch_if(true, kernel, grid, block, smem, st, cluster, std::forward<A>(args)...);
}
