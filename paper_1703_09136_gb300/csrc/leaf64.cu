// FP64 leaf passes: P2M from plan-time bases, and one kernel for everything a
// target sums (near field, L2P, an adaptive tree's M2P, directly summed reaction,
// result in the caller's order), launched twice where both fields are wanted: near
// field and reaction beside the tree pass, the rest after it.  Every non-empty leaf has
// a record (Leaf64Rec) with its ranges, so both trees run the same kernels.
//
// Bases.  B_m(x) = J_m(k rho) e^{-i m theta} of every point about its leaf's centre,
// m = 0 .. p + 1, is computed once per plan: J_{-m} = (-1)^m J_m makes the
// negative orders conjugates, so one product with B_m serves both m and -m (half
// the FP64 work and half the bytes of a full basis); order p + 1 serves the
// position gradient.
//
// Near field.  The plan stores (i/4) H0 of every U-list pair (near64_vals, fmm64.cu) as
// 55-bit fixed-point numbers with one exponent, each as seven base-256 digits: byte
// pairs (re, re, im, im) of two digits per 32-bit word, so that one AND or byte
// permute gives a digit of both parts as two f16 (the leading digit is signed; the
// others are the bytes themselves, read as f16 subnormals u 2^-24).  A leaf's
// strengths are cut into seven signed digits, which fill seven of the eight
// columns of an mma.sync m16n8k16: 7 MMAs per real product (2 x 7 for complex)
// give all 49 digit products of 16 targets x 8 sources, exact in FP32 over 32
// k-steps (255 x 128 x 512 < 2^24).
//
// What bounds it: FP64 instructions (64 clocks each on a sub-partition's pipe) and
// the latency of the block words.  Measured (one GB300, two layers, 262,144 points,
// one right-hand side): P2M 745 -> 51 us, near field + L2P + scatter 1370 -> 285 us
// (the blocks are 0.6 GB, 90 us of HBM; digits cut from 53-bit words with shifts
// instead of byte permutes took 333 us, FP64 partial sums per lane 453 us, loads
// without the ring 308 us); 1600 points: P2M 67 -> 11 us, the rest 360 -> 45 us.
#include <algorithm>
#include <cmath>
#include <vector>

#include "bessel.cuh"
#include "plan.cuh"
#include "split64.cuh"

namespace {

constexpr double BASIS64_MAX_BYTES = 8e9;

// B[i][m] = J_m(k rho) e^{-i m theta}, m = 0 .. nb - 1 (one CTA per leaf, a thread per point)
__global__ void basis64_kernel(const int32_t* __restrict__ lb, const double2* __restrict__ xs, double x0, double y0,
                               double h, double k, int nb, cd* __restrict__ basis) {
    extern __shared__ double jt[];
    const int64_t b = blockIdx.x;
    const double cx = x0 + (morton_x((uint32_t)b) + 0.5) * h, cy = y0 + (morton_y((uint32_t)b) + 0.5) * h;
    double* J = jt + (size_t)threadIdx.x * nb;
    for (int32_t i = lb[b] + threadIdx.x; i < lb[b + 1]; i += blockDim.x) {
        const double dx = xs[i].x - cx, dy = xs[i].y - cy;
        bessel_j_seq(k * hypot(dx, dy), nb - 1, J);
        const cd e1 = cexpi(-atan2(dy, dx));
        cd e = cmk(1.0, 0.0);
        cd* B = basis + (int64_t)i * nb;
        for (int m = 0; m < nb; ++m) {
            B[m] = cscale(e, J[m]);
            e = cmul(e, e1);
        }
    }
}

// P2M, a thread per (leaf, right-hand side, m >= 0): with q = (a, b), B = (u, v) the four
// real sums of a u, b v, a v, b u give alpha_m = sum q B_m and
// alpha_{-m} = (-1)^m sum q conj(B_m).  Also the level's exponent (split64.cu).
// PS = 4 lanes split a leaf's points where there are too few items for the GPU.
template <int PS>
__global__ void __launch_bounds__(128) p2m64_kernel(const Leaf64Rec* __restrict__ recs, const cd* __restrict__ basis,
                                                    const cd* __restrict__ qs, int64_t n, int64_t nleaf, int pitch,
                                                    int nrhs) {
    pdl_start_next();
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, it = id / PS;
    const int r = blockIdx.y, part = (int)(id % PS), m = (int)(it % pitch);
    const bool in = it < nleaf * pitch;                    // whole groups of PS lanes
    const Leaf64Rec& L = recs[in ? it / pitch : 0];
    const bool live = in && L.mult && m <= L.p;
    const int nb = L.nb;
    const cd* q = qs + (int64_t)r * n + L.tlo;
    const cd* B = basis + L.boff + m;
    double s1 = 0.0, s2 = 0.0, s3 = 0.0, s4 = 0.0;
    const int tn = live ? L.tn : 0;
    pdl_wait();
#pragma unroll 4
    for (int j = part; j < tn; j += PS) {
        const cd a = __ldcg(q + j), u = __ldg(B + (int64_t)j * nb);
        s1 = fma(a.x, u.x, s1);
        s2 = fma(a.y, u.y, s2);
        s3 = fma(a.x, u.y, s3);
        s4 = fma(a.y, u.x, s4);
    }
    __syncwarp();
#pragma unroll
    for (int o = 1; o < PS; o <<= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        s3 += __shfl_xor_sync(0xffffffffu, s3, o);
        s4 += __shfl_xor_sync(0xffffffffu, s4, o);
    }
    int e = S6_NONE;
    if (live) {
        cd* out = L.mult + (L.lidx * nrhs + r) * (2 * L.p + 1) + L.p;
        const cd ap = cmk(s1 - s2, s3 + s4), am = cmk(s1 + s2, s4 - s3);
        if (part == 0) {
            out[m] = ap;
            if (m > 0) out[-m] = (m & 1) ? cneg(am) : am;
        }
        if (L.E) {
            const int sh = -L.sx[m];
            e = max(max(s6_exponent(ap.x, sh), s6_exponent(ap.y, sh)), max(s6_exponent(am.x, sh), s6_exponent(am.y, sh)));
        }
    }
    // one level (uniform trees): one atomic per warp, else one per lane that has a value
    int* E = live ? L.E : nullptr;
    const unsigned same = __match_any_sync(0xffffffffu, (unsigned long long)E);
    if (same == 0xffffffffu) {
        e = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0 && E && e > S6_NONE) atomicMax(E + r, e);
    } else if (E && e > S6_NONE) atomicMax(E + r, e);
}

// Empty leaves of a uniform tree: zero multipoles (their parents' M2M reads them).
__global__ void zero_empty_kernel(const int32_t* __restrict__ lb, int64_t nleaf, int64_t per, cd* __restrict__ mult) {
    pdl_start_next();
    pdl_wait();
    for (int64_t b = blockIdx.x; b < nleaf; b += gridDim.x)
        if (lb[b + 1] == lb[b])
            for (int64_t i = threadIdx.x; i < per; i += blockDim.x) mult[b * per + i] = cmk(0.0, 0.0);
}

// Sorted indices of every leaf's near-field sources (uniform trees: the 3 x 3 neighbourhood
// in dy, dx order), as the block layout counts them.
__global__ void leaf_sources_kernel(const int32_t* __restrict__ lb, int L, const Leaf64Rec* __restrict__ recs,
                                    int32_t* __restrict__ src) {
    const Leaf64Rec& R = recs[blockIdx.x];
    const int m = 1 << L, ix = (int)morton_x((uint32_t)R.lidx), iy = (int)morton_y((uint32_t)R.lidx);
    int64_t o = R.soff;
    for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) {
            const int sx = ix + dx, sy = iy + dy;
            if (sx < 0 || sy < 0 || sx >= m || sy >= m) continue;
            const uint32_t s = morton((uint32_t)sx, (uint32_t)sy);
            for (int32_t j = lb[s] + threadIdx.x; j < lb[s + 1]; j += blockDim.x) src[o + (j - lb[s])] = j;
            o += lb[s + 1] - lb[s];
        }
}

struct Leaf64Args {
    const Leaf64Rec* recs;
    int nrhs, p;                     // largest order of a leaf
    int64_t n;
    const cd* qs;
    // near field: digit blocks (null: not here), their exponent, source indices
    const uint4* G;
    const int* EG;
    const int32_t* src;
    bool l2p, m2p, direct;
    const cd* basis;
    const Leaf64W* w;                // M2P
    const cd* m2pb;
    const Leaf64D* d;                // directly summed reaction
    const cd* dvals;
    const cd* ys;                    // sums made by other kernels (null: none)
    const int64_t* perm;             // null: sorted order
    bool conj_out;
    cd* y;
};

constexpr int LD = 7;                // base-256 digits
constexpr int LF_RING = 4;            // k-steps of near-field words in flight per warp (2 KB each)
constexpr int LF_TERMS = 32;         // k-steps per exact FP32 accumulation
constexpr long long LF_BIAS = 0x808080808080ll;   // 128 sum_{i = 0 .. 5} 256^i

// |v| < 2^E as a fixed-point number: 54 bits of the strengths (their leading digit has to hold the carry of the six
// signed ones below it), 55 of the blocks.  Error of a leaf's sum against extended precision, k h = 0.25 .. 25, 36 to 270
// sources: 0.7 .. 2.8e-16, FP64 multiply-adds 2.8 .. 8.1e-16 (53 bits of both: up to 1.1e-15).
constexpr int LF_QBITS = 54, LF_GBITS = 55;

// digit i of two numbers (with LF_BIAS) as f16: 1024 + field as bits 0x6400 | field, minus 1152
__device__ __forceinline__ unsigned lf_digit(long long xb, long long yb, int i) {
    const unsigned f0 = (unsigned)(int)((xb >> (8 * (LD - 1 - i))) + (i == 0 ? 128 : 0)) & 255u;
    const unsigned f1 = (unsigned)(int)((yb >> (8 * (LD - 1 - i))) + (i == 0 ? 128 : 0)) & 255u;
    unsigned h = 0x64006400u | f0 | (f1 << 16), r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x64806480u));
    return r;
}

// values v = 0 .. 3 of the four lanes of a quad -> their sums, value t in lane t
template <class T>
__device__ __forceinline__ T quad_scatter(const T (&v)[4], int t) {
    const bool hi2 = t & 2, hi1 = t & 1;
    const T k0 = hi2 ? v[2] : v[0], k1 = hi2 ? v[3] : v[1], s0 = hi2 ? v[0] : v[2], s1 = hi2 ? v[1] : v[3];
    const T a0 = k0 + __shfl_xor_sync(0xffffffffu, s0, 2), a1 = k1 + __shfl_xor_sync(0xffffffffu, s1, 2);
    return (hi1 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, hi1 ? a0 : a1, 1);
}

// One CTA of W warps per (leaf, right-hand side); a warp per 16 targets, and where a
// leaf has fewer tiles than warps these split its sources (and orders).  In the
// MMA layout lane (g, t) = (lane / 4, lane % 4) holds targets g and g + 8 of the
// tile; its part of the L2P and reaction sums is orders / sources = t mod 4.
// The digit sums stay integers until lane t converts value t of its quad (real and
// imaginary part of both targets): FP64 instructions are what this kernel has to
// save.  W = 1 keeps every warp busy and free of barriers where the launch fills
// the GPU, W = 4 shortens the chain of a launch with few leaves.
template <int W>
__global__ void __maxnreg__(128) leaf64_kernel(const __grid_constant__ Leaf64Args A) {
    extern __shared__ __align__(16) double lf_smem[];
    pdl_start_next();
    constexpr int CHUNK = 128 * W, QPT = 4;                             // sources staged at once; per thread
    const Leaf64Rec L = A.recs[blockIdx.x];
    const int32_t tlo = L.tlo, tn = L.tn;
    const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
    unsigned* sq = reinterpret_cast<unsigned*>(lf_smem);               // [CHUNK][LD] digit pairs
    double* red = lf_smem + CHUNK * LD / 2;                             // [W][3][32] (W > 1)
    uint4* ring = reinterpret_cast<uint4*>(red + (W > 1 ? W * 96 : 0));  // [W][LF_RING][4][32]
    double* coef = reinterpret_cast<double*>(ring + W * LF_RING * 128);  // [p + 1][4]
    ring += wid * (LF_RING * 128) + lane;
    const uint32_t ring_a = (uint32_t)__cvta_generic_to_shared(ring);
    __shared__ int s_e[W];
    auto sync = [&] { if (W > 1) __syncthreads(); else __syncwarp(); };
    const cd* q = A.qs + (int64_t)r * A.n;
    const int p = L.p, nb = L.nb, nc = 2 * p + 1;
    const bool l2p = A.l2p && L.loc;
    pdl_wait();
    if (l2p) {
        // y = (i/4) sum_m beta_m conj-basis: with c = beta_m, d = (-1)^m beta_{-m} and B = (u, v)
        // re y = sum u w0 + v w1, im y = sum u w2 + v w3
        const cd* beta = L.loc + (L.lidx * A.nrhs + r) * nc + p;
        for (int m = tid; m <= p; m += W * 32) {
            const cd c = __ldcg(beta + m);
            cd d = m > 0 ? __ldcg(beta - m) : cmk(0.0, 0.0);
            if (m & 1) d = cneg(d);
            coef[4 * m] = -0.25 * (c.y + d.y);
            coef[4 * m + 1] = 0.25 * (c.x - d.x);
            coef[4 * m + 2] = 0.25 * (c.x + d.x);
            coef[4 * m + 3] = 0.25 * (c.y - d.y);
        }
    }
    sync();
    const int ns = A.G ? L.ns : 0;
    const int32_t* src = A.src + L.soff;
    auto strength = [&](int j) { return j < ns ? __ldg(q + __ldg(src + j)) : cmk(0.0, 0.0); };
    // the first chunk's strengths stay in registers between their exponent and their digits
    cd qv[QPT];
    int Eq = S6_NONE;
    if (A.G) {
#pragma unroll
        for (int u = 0; u < QPT; ++u) qv[u] = strength(tid + u * W * 32);
#pragma unroll
        for (int u = 0; u < QPT; ++u) Eq = max(Eq, max(s6_exponent(qv[u].x, 0), s6_exponent(qv[u].y, 0)));
        for (int j = CHUNK + tid; j < ns; j += W * 32) {
            const cd v = strength(j);
            Eq = max(Eq, max(s6_exponent(v.x, 0), s6_exponent(v.y, 0)));
        }
        Eq = __reduce_max_sync(0xffffffffu, Eq);
        if (W > 1) {
            if (lane == 0) s_e[wid] = Eq;
            __syncthreads();
            for (int w = 0; w < W; ++w) Eq = max(Eq, s_e[w]);
        }
    }
    const bool bad = Eq >= S6_NAN / 2;
    const int EV = max(Eq, S6_NONE) + (A.G ? max(*A.EG, S6_NONE) : 0) + 40 - LF_QBITS - LF_GBITS;
    const uint4* Gb = A.G ? A.G + L.goff : nullptr;

    const int ntile = (tn + 15) / 16;
    int staged = -1;                                                     // first source of the staged chunk
    for (int t0 = 0; t0 < ntile;) {
        const int tp = min(W, ntile - t0), ks = W / tp;                  // tiles at once, warps per tile
        const int tile = t0 + wid % tp, part = wid / tp;
        const bool live = part < ks;
        const int i0 = 16 * tile + g, i1 = i0 + 8;
        const bool v0 = live && i0 < tn, v1 = live && i1 < tn;
        long long hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};            // (re, im) of target i0, of i1
        for (int c0 = 0; c0 < ns; c0 += CHUNK) {
            if (staged != c0) {
                if (staged >= 0) {
                    sync();                                              // the old chunk is read
#pragma unroll
                    for (int u = 0; u < QPT; ++u) qv[u] = strength(c0 + tid + u * W * 32);
                }
#pragma unroll
                for (int u = 0; u < QPT; ++u) {
                    const long long xr = s6_fixed<LF_QBITS>(qv[u].x, 0, Eq) + LF_BIAS, xi = s6_fixed<LF_QBITS>(qv[u].y, 0, Eq) + LF_BIAS;
#pragma unroll
                    for (int d = 0; d < LD; ++d) sq[(tid + u * W * 32) * LD + d] = lf_digit(xr, xi, d);
                }
                staged = c0;
                sync();
            }
            if (!live) continue;
            const int nk = (min(CHUNK, ns - c0) + 7) / 8;
            // this lane's words of k-step kk into slot (kk / ks) % LF_RING: (i0, j0), (i1, j0), (i0, j1),
            // (i1, j1); zeros meet zero strengths or unused rows
            auto load_G = [&](int kk) {
                if (kk < nk) {
                    const int j0 = c0 + 8 * kk + t, j1 = j0 + 4;
                    const uint4* Gj = Gb + (int64_t)j0 * tn;
                    const uint32_t dst = ring_a + (kk / ks) % LF_RING * 2048;
                    const bool a0 = v0 && j0 < ns, a1 = v1 && j0 < ns, b0 = v0 && j1 < ns, b1 = v1 && j1 < ns;
                    cp_async16(dst, a0 ? Gj + i0 : Gb, a0);
                    cp_async16(dst + 512, a1 ? Gj + i1 : Gb, a1);
                    cp_async16(dst + 1024, b0 ? Gj + 4 * (int64_t)tn + i0 : Gb, b0);
                    cp_async16(dst + 1536, b1 ? Gj + 4 * (int64_t)tn + i1 : Gb, b1);
                }
                cp_commit();
            };
#pragma unroll
            for (int u = 0; u < LF_RING - 1; ++u) load_G(part + u * ks);
            for (int kb = part; kb < nk; kb += LF_TERMS * ks) {
                float ar[LD][4], ai[LD][4];
#pragma unroll
                for (int d = 0; d < LD; ++d)
#pragma unroll
                    for (int v = 0; v < 4; ++v) ar[d][v] = ai[d][v] = 0.0f;
                const int ke = min(nk, kb + LF_TERMS * ks);
                for (int kk = kb; kk < ke; kk += ks) {
                    cp_wait<LF_RING - 2>();
                    uint4 w[4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) w[v] = ring[((kk / ks) % LF_RING * 4 + v) * 32];
                    load_G(kk + (LF_RING - 1) * ks);
                    // columns g = strength digits: (qr, -qi) for the real part, (qi, qr) for the imaginary
                    const unsigned d0 = g < LD ? sq[(8 * kk + t) * LD + g] : 0u;
                    const unsigned d1 = g < LD ? sq[(8 * kk + t + 4) * LD + g] : 0u;
                    const uint2 br = make_uint2(d0 ^ 0x80000000u, d1 ^ 0x80000000u);
                    const uint2 bi = make_uint2(__byte_perm(d0, 0, 0x1032), __byte_perm(d1, 0, 0x1032));
#pragma unroll
                    for (int d = 0; d < LD; ++d) {
                        unsigned a[4];
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const unsigned x = d < 2 ? w[v].x : d < 4 ? w[v].y : d < 6 ? w[v].z : w[v].w;
                            if (d == 0) {
                                const unsigned h = (x & 0x00ff00ffu) | 0x64006400u;
                                asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(a[v]) : "r"(h), "r"(0x64806480u));
                            } else a[v] = (d & 1) ? __byte_perm(x, 0, 0x4341) : x & 0x00ff00ffu;
                        }
                        const uint4 av = make_uint4(a[0], a[1], a[2], a[3]);
                        s6_mma(ar[d], av, br);
                        s6_mma(ai[d], av, bi);
                    }
                }
                // columns 2t, 2t + 1 of the accumulators: order k = digit + column - 2t
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int row = v >> 1;                              // 0: target i0, 1: i1
                    float (&acc)[LD][4] = (v & 1) ? ai : ar;
                    int s[LD + 1];
#pragma unroll
                    for (int k = 0; k <= LD; ++k) {
                        s[k] = 0;
                        if (k < LD) s[k] = __float2int_rn(acc[k][2 * row] * (k > 0 ? 16777216.0f : 1.0f));
                        if (k > 0) s[k] += __float2int_rn(acc[k - 1][2 * row + 1] * (k > 1 ? 16777216.0f : 1.0f));
                    }
                    hi[v] += ((long long)s[0] << 24) + ((long long)s[1] << 16) + ((long long)s[2] << 8) + s[3];
                    lo[v] += ((long long)s[4] << 24) + ((long long)s[5] << 16) + ((long long)s[6] << 8) + s[7];
                }
            }
        }
        double val[4] = {0.0, 0.0, 0.0, 0.0};
        if (live) {
            if (l2p) {
                const cd* B0 = A.basis + L.boff + (int64_t)(v0 ? i0 : 0) * nb;
                const cd* B1 = A.basis + L.boff + (int64_t)(v1 ? i1 : 0) * nb;
#pragma unroll 4
                for (int m = t + 4 * part; m <= p; m += 4 * ks) {
                    const double w0 = coef[4 * m], w1 = coef[4 * m + 1], w2 = coef[4 * m + 2], w3 = coef[4 * m + 3];
                    const cd u0 = v0 ? __ldg(B0 + m) : cmk(0.0, 0.0), u1 = v1 ? __ldg(B1 + m) : cmk(0.0, 0.0);
                    val[0] = fma(u0.x, w0, fma(u0.y, w1, val[0]));
                    val[1] = fma(u0.x, w2, fma(u0.y, w3, val[1]));
                    val[2] = fma(u1.x, w0, fma(u1.y, w1, val[2]));
                    val[3] = fma(u1.x, w2, fma(u1.y, w3, val[3]));
                }
            }
            if (A.m2p && L.wend > L.wbeg) {                              // (i/4) sum_m a_m H_m e^{i m theta}
                cd a0 = cmk(0.0, 0.0), a1 = cmk(0.0, 0.0);
                for (int32_t e = L.wbeg; e < L.wend; ++e) {
                    const Leaf64W D = A.w[e];
                    const int nw = 2 * D.p + 1;
                    const cd* am = D.mult + (D.lidx * A.nrhs + r) * nw;
                    const cd* M = A.m2pb + D.boff;
#pragma unroll 2
                    for (int m = t + 4 * part; m < nw; m += 4 * ks) {
                        const cd a = __ldcg(am + m);
                        if (v0) cfma(a0, a, __ldg(M + (int64_t)i0 * nw + m));
                        if (v1) cfma(a1, a, __ldg(M + (int64_t)i1 * nw + m));
                    }
                }
                val[0] -= 0.25 * a0.y; val[1] += 0.25 * a0.x; val[2] -= 0.25 * a1.y; val[3] += 0.25 * a1.x;
            }
            if (A.direct)
                for (int32_t e = L.dbeg; e < L.dend; ++e) {
                    const Leaf64D E = A.d[e];
                    const cd* D = A.dvals + E.blk;
#pragma unroll 2
                    for (int j = t + 4 * part; j < E.sn; j += 4 * ks) {
                        const cd v = __ldg(q + E.slo + j);
                        cd a0 = cmk(val[0], val[1]), a1 = cmk(val[2], val[3]);
                        if (v0) cfma(a0, __ldg(D + (int64_t)i0 * E.sn + j), v);
                        if (v1) cfma(a1, __ldg(D + (int64_t)i1 * E.sn + j), v);
                        val[0] = a0.x; val[1] = a0.y; val[2] = a1.x; val[3] = a1.y;
                    }
                }
        }
        // quad sums: A 2^32 + B, lane t's digits 2^(-16 t) below (what falls under the unit
        // of B is 2^-70 of the largest product)
        long long pa[4], pb[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            pa[v] = hi[v] >> (16 * t);
            pb[v] = t == 0 ? lo[v] : ((hi[v] << (64 - 16 * t)) >> 32 & 0xffffffffll) + (lo[v] >> (16 * t));
        }
        long long a = ns > 0 ? quad_scatter(pa, t) : 0, bsum = ns > 0 ? quad_scatter(pb, t) : 0;
        double x = quad_scatter(val, t);
        if (W > 1 && ks > 1) {                                           // parts of a tile, added in order by part 0
            double* mine = red + (size_t)wid * 96 + lane;
            __syncthreads();
            if (live && part > 0) {
                mine[0] = __longlong_as_double(a);
                mine[32] = __longlong_as_double(bsum);
                mine[64] = x;
            }
            __syncthreads();
            if (part == 0)
                for (int o = 1; o < ks; ++o) {
                    const double* other = mine + (size_t)o * tp * 96;
                    a += __double_as_longlong(other[0]);
                    bsum += __double_as_longlong(other[32]);
                    x += other[64];
                }
        }
        if (live && part == 0 && (t < 2 ? v0 : v1)) {
            const int64_t i = tlo + (t < 2 ? i0 : i1);
            if (ns > 0) x += scale2d(fma((double)a, 4294967296.0, (double)bsum), EV);
            if (bad) x = __longlong_as_double(0x7ff8000000000000ll);
            if (A.ys) x += __ldcg(reinterpret_cast<const double*>(A.ys + (int64_t)r * A.n + i) + (t & 1));
            reinterpret_cast<double*>(A.y + (int64_t)r * A.n + (A.perm ? A.perm[i] : i))[t & 1] = (A.conj_out && (t & 1)) ? -x : x;
        }
        t0 += tp;
    }
}

// (i/4) H0 doubles -> largest exponent below `top`; then, in place, digit words.  The other entries are counted,
// listed (near64_list_kernel) and leave zeros.
__device__ __forceinline__ int near64_exponent(cd v) { return max(s6_exponent(v.x, 0), s6_exponent(v.y, 0)); }

__global__ void near64_exponent_kernel(const cd* __restrict__ G, int64_t n, int top, int* __restrict__ E,
                                       unsigned long long* __restrict__ above) {
    int e = S6_NONE;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = near64_exponent(G[i]);
        if (x < top) e = max(e, x);
        else atomicAdd(above, 1ull);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0 && e > S6_NONE) atomicMax(E, e);
}

__global__ void near64_list_kernel(const cd* __restrict__ G, int64_t n, int top, unsigned long long* __restrict__ next,
                                   NearLarge* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const cd v = G[i];
        if (near64_exponent(v) < top) continue;
        NearLarge& o = out[atomicAdd(next, 1ull)];
        o.pair = i;
        o.val = v;
    }
}

__global__ void near64_fix_kernel(cd* G, int64_t n, int top, const int* __restrict__ E) {
    const int e = *E;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        cd v = G[i];
        if (near64_exponent(v) >= top) v = cmk(0.0, 0.0);
        const long long x = s6_fixed<LF_GBITS>(v.x, 0, e) + (128ll << 48), y = s6_fixed<LF_GBITS>(v.y, 0, e) + (128ll << 48);
        unsigned w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {                      // digits 2k, 2k + 1 = bytes 6 - 2k, 5 - 2k
            const unsigned x0 = (unsigned)(x >> (8 * (6 - 2 * k))) & 255u, y0 = (unsigned)(y >> (8 * (6 - 2 * k))) & 255u;
            const unsigned x1 = k < 3 ? (unsigned)(x >> (8 * (5 - 2 * k))) & 255u : 0u;
            const unsigned y1 = k < 3 ? (unsigned)(y >> (8 * (5 - 2 * k))) & 255u : 0u;
            w[k] = x0 | (x1 << 8) | (y0 << 16) | (y1 << 24);
        }
        reinterpret_cast<uint4*>(G)[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// The listed entries onto the sums that leaf64_kernel wrote: a warp per (target that has some, right-hand side).
__global__ void __launch_bounds__(128) near64_large_kernel(const int32_t* __restrict__ tgt, const int64_t* __restrict__ beg,
                                                              const int32_t* __restrict__ src, const cd* __restrict__ val,
                                                              int64_t ntgt, const cd* __restrict__ qs, int64_t n, int nrhs,
                                                              const int64_t* __restrict__ perm, bool conj_out,
                                                              cd* __restrict__ y) {
    const int lane = threadIdx.x & 31;
    const int64_t total = ntgt * nrhs;
    for (int64_t id = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5); id < total; id += (int64_t)gridDim.x * 4) {
        const int64_t t = id % ntgt, r = id / ntgt;
        cd a = cmk(0.0, 0.0);
        for (int64_t e = beg[t] + lane; e < beg[t + 1]; e += 32) cfma(a, val[e], qs[r * n + src[e]]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
            a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
        }
        if (lane == 0) {
            cd* o = y + r * n + (perm ? perm[tgt[t]] : tgt[t]);
            *o = cadd(*o, conj_out ? cconj(a) : a);
        }
    }
}

// ---------------------------------------------------------------------------
// Position gradients: out[t] = Re sum_r (conj(g_t) grad u_t + q_t grad w_t), u and w the fields of q
// and conj(g).  Both fields go through the same blocks, so a pair needs the one complex number
//   S = sum_r conj(g_t) q_s + q_t conj(g_s)
// and the real parts of Gx S and Gy S: 8 nrhs + 4 FP64 FMAs instead of 16 nrhs.  The far part is the
// L2P with the locals of the derivative, from the same bases (order p + 1 included):
//   d/dx sum_q b_q E_q = (k/2) sum_m (b_{m+1} - b_{m-1}) E_m,   d/dy: (i k/2) sum_m (b_{m+1} + b_{m-1}) E_m.
// Bound by FP64 FMAs (3.4 M near-field pairs of 40,000 points, one right-hand side: 12 each, 80 us);
// the pairs run beside both tree passes.  Measured there: near field 2 x 208 us (a lane per target of
// ten-point leaves) -> 104 us, locals' gradient 2 x 266 us (Bessel sequences evaluated on each
// call) -> 2 x 27 us; the whole gradient 1578 -> 768 us (804 with order 6
// of the digit products).
// ---------------------------------------------------------------------------
constexpr int GN_TB = 128;

// Near field and direct reaction.  A CTA per leaf: thread (part, i) takes the target i and every
// parts-th source, so that consecutive lanes read consecutive block entries; parts added in order.
template <bool ONE>
__global__ void __launch_bounds__(GN_TB) grad_near_kernel(const Leaf64Rec* __restrict__ recs, const int32_t* __restrict__ src,
                                                          const cd* __restrict__ Gx, const cd* __restrict__ Gy,
                                                          const Leaf64D* __restrict__ ds, const cd* __restrict__ Dx,
                                                          const cd* __restrict__ Dy, const cd* __restrict__ q,
                                                          const cd* __restrict__ gc, int64_t n, int nrhs,
                                                          double2* __restrict__ out) {
    __shared__ double2 near_s[GN_TB], direct_s[GN_TB];
    const Leaf64Rec& L = recs[blockIdx.x];
    const int tid = threadIdx.x, ns = L.ns;
    auto pair_strength = [&](int64_t t, int64_t s, cd qt, cd gt) {
        cd S = cmk(0.0, 0.0);
        if (ONE) {
            cfma(S, gt, __ldg(q + s));
            cfma(S, qt, __ldg(gc + s));
        } else
            for (int r = 0; r < nrhs; ++r) {
                cfma(S, __ldg(gc + r * n + t), __ldg(q + r * n + s));
                cfma(S, __ldg(q + r * n + t), __ldg(gc + r * n + s));
            }
        return S;
    };
    auto add = [](double2& a, cd x, cd y, cd S) {
        a.x = fma(x.x, S.x, fma(-x.y, S.y, a.x));
        a.y = fma(y.x, S.x, fma(-y.y, S.y, a.y));
    };
    for (int i0 = 0; i0 < L.tn; i0 += GN_TB) {
        const int tn = min(GN_TB, L.tn - i0), parts = GN_TB / tn;
        double2 a = make_double2(0.0, 0.0), b = a;
        if (tid < parts * tn) {
            {
                const int i = i0 + tid % tn;
                const int64_t t = L.tlo + i;
                const cd qt = __ldg(q + t), gt = __ldg(gc + t);
                const int32_t* sj = src + L.soff;
                const int64_t o = L.goff + i;
#pragma unroll 4
                for (int j = tid / tn; j < ns; j += parts) {
                    const int64_t e = o + (int64_t)j * L.tn;
                    add(a, __ldg(Gx + e), __ldg(Gy + e), pair_strength(t, __ldg(sj + j), qt, gt));
                }
            }
            const int i = i0 + tid / parts;                // entries of a direct block: consecutive sources
            const int64_t t = L.tlo + i;
            for (int32_t e = L.dbeg; e < L.dend; ++e) {
                const Leaf64D E = ds[e];
                const int64_t o = E.blk + (int64_t)i * E.sn;
                const cd qt = __ldg(q + t), gt = __ldg(gc + t);
                for (int j = tid % parts; j < E.sn; j += parts)
                    add(b, __ldg(Dx + o + j), __ldg(Dy + o + j), pair_strength(t, E.slo + j, qt, gt));
            }
        }
        __syncthreads();                                   // the last chunk's sums are read
        near_s[tid] = a;
        direct_s[tid] = b;
        __syncthreads();
        if (tid < tn) {
            double2 v = make_double2(0.0, 0.0);
            for (int k = 0; k < parts; ++k) {
                const double2 x = near_s[k * tn + tid], y = direct_s[tid * parts + k];
                v.x += x.x + y.x;
                v.y += x.y + y.y;
            }
            out[L.tlo + i0 + tid] = v;
        }
    }
}

// Far field of one of the two fields: Re sum_r v_t grad(local field)_t, four lanes a target.
// Without gxy the sums go to acc; with it, acc, the near field's sums and these go to the caller's order.
__global__ void __launch_bounds__(64) grad_far_kernel(const Leaf64Rec* __restrict__ recs, const cd* __restrict__ basis,
                                                      const cd* __restrict__ v, int64_t n, int nrhs, double k,
                                                      double2* __restrict__ acc, const double2* __restrict__ near_sum,
                                                      const int64_t* __restrict__ perm, double* __restrict__ gxy) {
    extern __shared__ __align__(16) double gf_coef[];      // [p + 2][8]
    const Leaf64Rec& L = recs[blockIdx.x];
    const int p = L.p, nb = L.nb, nc = 2 * p + 1, t = threadIdx.x & 3;
    const double f = 0.125 * k;
    for (int i0 = 0; i0 < L.tn; i0 += 16) {
        const int i = i0 + (threadIdx.x >> 2);
        const bool live = i < L.tn;
        const cd* B = basis + L.boff + (int64_t)(live ? i : 0) * nb;
        double ax = 0.0, ay = 0.0;
        for (int r = 0; r < nrhs; ++r) {
            if (i0 == 0 || nrhs > 1) {
                const cd* beta = L.loc + (L.lidx * nrhs + r) * nc + p;
                auto at = [&](int m) { return m >= -p && m <= p ? __ldg(beta + m) : cmk(0.0, 0.0); };
                __syncthreads();                           // the last coefficients are read
                for (int m = threadIdx.x; m <= p + 1; m += 64) {
                    const double sg = m == 0 ? 0.0 : (m & 1) ? -1.0 : 1.0;
                    const cd up = at(m + 1), lo = at(m - 1), nup = at(1 - m), nlo = at(-1 - m);
                    const cd cx = csub(up, lo), dx = cscale(csub(nup, nlo), sg);
                    const cd cy = cmuli(cadd(up, lo)), dy = cscale(cmuli(cadd(nup, nlo)), sg);
                    double* w = gf_coef + 8 * m;
                    w[0] = -f * (cx.y + dx.y); w[1] = f * (cx.x - dx.x); w[2] = f * (cx.x + dx.x); w[3] = f * (cx.y - dx.y);
                    w[4] = -f * (cy.y + dy.y); w[5] = f * (cy.x - dy.x); w[6] = f * (cy.x + dy.x); w[7] = f * (cy.y - dy.y);
                }
                __syncthreads();
            }
            cd x = cmk(0.0, 0.0), y = x;
            if (live) {
#pragma unroll 2
                for (int m = t; m < nb; m += 4) {
                    const cd u = __ldg(B + m);
                    const double* w = gf_coef + 8 * m;
                    x.x = fma(u.x, w[0], fma(u.y, w[1], x.x));
                    x.y = fma(u.x, w[2], fma(u.y, w[3], x.y));
                    y.x = fma(u.x, w[4], fma(u.y, w[5], y.x));
                    y.y = fma(u.x, w[6], fma(u.y, w[7], y.y));
                }
                const cd vt = __ldg(v + (int64_t)r * n + L.tlo + i);
                ax = fma(vt.x, x.x, fma(-vt.y, x.y, ax));
                ay = fma(vt.x, y.x, fma(-vt.y, y.y, ay));
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, o);
            ay += __shfl_xor_sync(0xffffffffu, ay, o);
        }
        if (live && t == 0) {
            const int64_t j = L.tlo + i;
            if (gxy) {
                const double2 a = acc[j], b = near_sum[j];
                const int64_t c = perm[j];
                gxy[2 * c] = ax + a.x + b.x;
                gxy[2 * c + 1] = ay + a.y + b.y;
            } else acc[j] = make_double2(ax, ay);
        }
    }
}

}  // namespace

// Position gradient: near field and direct reaction of both fields.
hfmm_status launch_grad_near(hfmm_plan_s* P, int nrhs, const cd* gc, double2* out, cudaStream_t st) {
    auto kernel = nrhs == 1 ? grad_near_kernel<true> : grad_near_kernel<false>;
    kernel<<<(unsigned)P->leaf64_n, GN_TB, 0, st>>>(P->leaf64, P->leaf64_src, P->near64g_x, P->near64g_y, P->leaf64_d,
                                                    P->d_gvals, P->d_gvals ? P->d_gvals + P->nd_vals : nullptr,
                                                    P->q_sorted, gc, P->n, nrhs, out);
    ++P->launches;
    HFMM_CUDA_TRY(cudaGetLastError());
    return HFMM_OK;
}

// Position gradient: the locals' part of one field, v the other field's factor at the targets.
hfmm_status launch_grad_far(hfmm_plan_s* P, int nrhs, const cd* v, double2* acc, const double2* near_sum, double* gxy,
                            cudaStream_t st) {
    grad_far_kernel<<<(unsigned)P->leaf64_n, 64, 8 * sizeof(double) * (P->leaf64_p + 2), st>>>(
        P->leaf64, P->basis64, v, P->n, nrhs, P->k, acc, near_sum, P->perm, gxy);
    ++P->launches;
    HFMM_CUDA_TRY(cudaGetLastError());
    return HFMM_OK;
}

// Digit form of `pairs` near-field values in place (E: their exponent, and two words behind it a counter).  Entries
// of 4 and more, i.e. of points within some 1e-11 wavelengths, go into *large: an infinite one (coincident points)
// has no digits, and a large one would cost every other entry of the plan some of its.  Where more than
// NEAR64_LARGE_MAX are that large, only the infinite ones do; where those are too many as well,
// *fixed = false and the values stay.
hfmm_status near64_to_fixed(cd* vals, int64_t pairs, int* E, std::vector<NearLarge>* large, bool* fixed, cudaStream_t st) {
    large->clear();
    unsigned long long* count = (unsigned long long*)(E + 2);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((pairs + 255) / 256, 16 * 152));
    unsigned long long found = 0;
    int top = 3;
    for (;; top = S6_NAN) {
        HFMM_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(*count), st));
        HFMM_CUDA_TRY(cudaMemsetAsync(E, 0x80, sizeof(int), st));
        near64_exponent_kernel<<<grid, 256, 0, st>>>(vals, pairs, top, E, count);
        HFMM_CUDA_TRY(cudaGetLastError());
        HFMM_CUDA_TRY(cudaMemcpyAsync(&found, count, sizeof(found), cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        if (found <= NEAR64_LARGE_MAX || top == S6_NAN) break;
    }
    *fixed = found <= NEAR64_LARGE_MAX;
    if (!*fixed) return HFMM_OK;
    if (found > 0) {
        NearLarge* list = nullptr;
        HFMM_CUDA_TRY(cudaMallocAsync((void**)&list, sizeof(NearLarge) * found, st));
        HFMM_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(*count), st));
        near64_list_kernel<<<grid, 256, 0, st>>>(vals, pairs, top, count, list);
        HFMM_CUDA_TRY(cudaGetLastError());
        large->resize(found);
        HFMM_CUDA_TRY(cudaMemcpyAsync(large->data(), list, sizeof(NearLarge) * found, cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        HFMM_CUDA_TRY(cudaFreeAsync(list, st));
        std::sort(large->begin(), large->end(), [](const NearLarge& a, const NearLarge& b) { return a.pair < b.pair; });
    }
    near64_fix_kernel<<<grid, 256, 0, st>>>(vals, pairs, top, E);
    HFMM_CUDA_TRY(cudaGetLastError());
    return HFMM_OK;
}

// The listed entries by target, from the leaf records (in the order of their blocks) and near-field source indices.
hfmm_status near64_upload_large(hfmm_plan_s* P, const std::vector<Leaf64Rec>& recs, cudaStream_t st) {
    const auto& list = P->near64_large;
    if (list.empty()) return HFMM_OK;
    int64_t nsrc = 0;
    for (const Leaf64Rec& R : recs) nsrc = std::max(nsrc, R.soff + R.ns);
    std::vector<int32_t> src(nsrc);
    HFMM_CUDA_TRY(cudaMemcpyAsync(src.data(), P->leaf64_src, sizeof(int32_t) * nsrc, cudaMemcpyDeviceToHost, st));
    HFMM_CUDA_TRY(cudaStreamSynchronize(st));
    struct Item { int32_t t, s; cd v; };
    std::vector<Item> items;
    size_t r = 0;
    for (const NearLarge& e : list) {
        while (e.pair >= recs[r].goff + (int64_t)recs[r].tn * recs[r].ns) ++r;
        const int64_t o = e.pair - recs[r].goff;           // source-major within the block
        items.push_back({recs[r].tlo + (int32_t)(o % recs[r].tn), src[recs[r].soff + o / recs[r].tn], e.val});
    }
    std::stable_sort(items.begin(), items.end(), [](const Item& a, const Item& b) { return a.t < b.t; });
    std::vector<int32_t> tgt, isrc;
    std::vector<int64_t> beg;
    std::vector<cd> val;
    for (const Item& it : items) {
        if (tgt.empty() || tgt.back() != it.t) {
            tgt.push_back(it.t);
            beg.push_back((int64_t)val.size());
        }
        isrc.push_back(it.s);
        val.push_back(it.v);
    }
    beg.push_back((int64_t)val.size());
    P->near64_large_n = (int64_t)tgt.size();
    HFMM_TRY(plan_alloc(P, (void**)&P->near64_large_tgt, sizeof(int32_t) * tgt.size()));
    HFMM_TRY(plan_alloc(P, (void**)&P->near64_large_beg, sizeof(int64_t) * beg.size()));
    HFMM_TRY(plan_alloc(P, (void**)&P->near64_large_src, sizeof(int32_t) * isrc.size()));
    HFMM_TRY(plan_alloc(P, (void**)&P->near64_large_val, sizeof(cd) * val.size()));
    HFMM_CUDA_TRY(cudaMemcpyAsync(P->near64_large_tgt, tgt.data(), sizeof(int32_t) * tgt.size(), cudaMemcpyHostToDevice, st));
    HFMM_CUDA_TRY(cudaMemcpyAsync(P->near64_large_beg, beg.data(), sizeof(int64_t) * beg.size(), cudaMemcpyHostToDevice, st));
    HFMM_CUDA_TRY(cudaMemcpyAsync(P->near64_large_src, isrc.data(), sizeof(int32_t) * isrc.size(), cudaMemcpyHostToDevice, st));
    HFMM_CUDA_TRY(cudaMemcpyAsync(P->near64_large_val, val.data(), sizeof(cd) * val.size(), cudaMemcpyHostToDevice, st));
    HFMM_CUDA_TRY(cudaStreamSynchronize(st));
    P->near64_large.clear();
    P->near64_large.shrink_to_fit();
    return HFMM_OK;
}

// Leaf records, near-field source indices and half bases of a uniform FP64 plan
// (a mixed plan's first gradient).  Without bases (byte budget) the P2M and
// L2P run on the kernels that evaluate them.
hfmm_status build_leaf64(hfmm_plan_s* P, cudaStream_t st) {
    if (P->leaf64 || P->ad) return HFMM_OK;
    const int L = P->L;
    const LevelInfo& lv = P->lev[L];
    const int nb = lv.p + 2;
    const double bytes = sizeof(cd) * (double)P->n * nb;
    const bool has_basis = bytes <= BASIS64_MAX_BYTES && nb * (int)sizeof(double) <= 40000 && optional_fits(bytes);
    const auto& lb = P->h_leaf_begin;
    std::vector<Leaf64Rec> recs;
    std::vector<Leaf64D> ds;
    std::vector<int32_t> dbeg, dsrc;
    std::vector<int64_t> dblk;
    if (P->nd > 0) {
        dbeg.resize((size_t)lv.nbox + 1);
        dsrc.resize(P->nd);
        dblk.resize(P->nd);
        HFMM_CUDA_TRY(cudaMemcpyAsync(dbeg.data(), P->d_begin, sizeof(int32_t) * dbeg.size(), cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dsrc.data(), P->d_src, sizeof(int32_t) * P->nd, cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dblk.data(), P->d_blk, sizeof(int64_t) * P->nd, cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
    }
    int64_t soff = 0, goff = 0;
    for (int64_t b = 0; b < lv.nbox; ++b) {
        const int32_t tn = lb[b + 1] - lb[b];
        if (tn == 0) continue;
        const int64_t ns = u_list_points(P, b);
        Leaf64Rec R{};
        R.tlo = lb[b]; R.tn = tn; R.ns = (int32_t)ns; R.p = lv.p; R.nb = nb;
        R.soff = soff; R.goff = goff; R.boff = (int64_t)lb[b] * nb; R.lidx = b;
        R.mult = lv.mult; R.loc = lv.loc; R.sx = lv.s6[0].sx;
        R.E = P->s6_ready[0] ? split_exp(P, 0, L, false) : nullptr;
        R.dbeg = (int32_t)ds.size();
        if (P->nd > 0)
            for (int32_t e = dbeg[b]; e < dbeg[b + 1]; ++e)
                ds.push_back({lb[dsrc[e]], lb[dsrc[e] + 1] - lb[dsrc[e]], dblk[e]});
        R.dend = (int32_t)ds.size();
        soff += ns;
        goff += (int64_t)tn * ns;
        P->leaf_max = std::max(P->leaf_max, (int)tn);
        recs.push_back(R);
    }
    P->leaf_empty = (int64_t)recs.size() < lv.nbox;
    P->leaf64_n = (int64_t)recs.size();
    P->leaf64_p = lv.p;
    HFMM_TRY(plan_alloc(P, (void**)&P->leaf64, sizeof(Leaf64Rec) * recs.size()));
    HFMM_TRY(plan_alloc(P, (void**)&P->leaf64_d, sizeof(Leaf64D) * ds.size()));
    HFMM_TRY(plan_alloc(P, (void**)&P->leaf64_src, sizeof(int32_t) * soff));
    HFMM_CUDA_TRY(cudaMemcpyAsync(P->leaf64, recs.data(), sizeof(Leaf64Rec) * recs.size(), cudaMemcpyHostToDevice, st));
    if (!ds.empty())
        HFMM_CUDA_TRY(cudaMemcpyAsync(P->leaf64_d, ds.data(), sizeof(Leaf64D) * ds.size(), cudaMemcpyHostToDevice, st));
    leaf_sources_kernel<<<(unsigned)recs.size(), 64, 0, st>>>(P->leaf_begin, L, P->leaf64, P->leaf64_src);
    HFMM_CUDA_TRY(cudaGetLastError());
    if (has_basis)
        HFMM_TRY(plan_optional(P, [&] { return plan_alloc(P, (void**)&P->basis64, (size_t)bytes); },
                               [&] { P->basis64 = nullptr; }));
    if (P->basis64) {
        P->buffer_bytes += bytes;
        const int thr = std::max(1, std::min(64, 5000 / nb));
        basis64_kernel<<<(unsigned)lv.nbox, thr, (size_t)thr * nb * sizeof(double), st>>>(
            P->leaf_begin, P->xy_sorted, P->x0, P->y0, lv.h, P->k, nb, P->basis64);
        HFMM_CUDA_TRY(cudaGetLastError());
    }
    HFMM_CUDA_TRY(cudaStreamSynchronize(st));             // recs and ds are locals
    return near64_upload_large(P, recs, st);
}

// The plan's memory of its leaf records and bases is gone.
void leaf64_forget(hfmm_plan_s* P) {
    P->leaf64 = nullptr;
    P->leaf64_w = nullptr;
    P->leaf64_d = nullptr;
    P->leaf64_src = nullptr;
    P->basis64 = P->m2p64 = nullptr;
    P->leaf64_n = 0;
    P->leaf64_p = P->leaf_max = 0;
}

// P2M of the sorted strengths into the leaf multipoles (and their exponents).
hfmm_status launch_p2m64(hfmm_plan_s* P, int nrhs, cudaStream_t st) {
    const int pitch = P->leaf64_p + 1;
    const int64_t items = P->leaf64_n * pitch;
    const int ps = items < 32 * 1024 ? 4 : 1;        // not by nrhs: it would change the sums' order
    auto kernel = ps == 4 ? p2m64_kernel<4> : p2m64_kernel<1>;
    if (P->leaf_empty) {
        const LevelInfo& lv = P->lev[P->L];
        HFMM_CUDA_TRY(pdl_launch(zero_empty_kernel, dim3((unsigned)std::min<int64_t>(lv.nbox, 16 * 152)), dim3(64), 0, st, 0,
                                 P->leaf_begin, lv.nbox, (int64_t)nrhs * lv.ncoef, lv.mult));
        ++P->launches;
    }
    HFMM_CUDA_TRY(pdl_launch(kernel, dim3((unsigned)((items * ps + 127) / 128), (unsigned)nrhs), dim3(128), 0, st, 0,
                             P->leaf64, P->basis64, P->q_sorted, P->n, P->leaf64_n, pitch, nrhs));
    ++P->launches;
    return HFMM_OK;
}

// Near field and direct reaction into y_sorted on the near stream, beside the far field (whose
// stream this returns in *fs): they need the strengths alone, and a tree pass leaves SMs idle
// at its coarse levels (before order 6 joined the digit products: 1600 points 138 -> 114 us an apply, two
// layers, 262,144 points 1528 -> 1461, an adaptive tree of 20,011 points 582 -> 559; with it 116, 1578 and 570).
hfmm_status fork_near64(hfmm_plan_s* P, int nrhs, bool direct, cudaStream_t st, cudaStream_t* fs) {
    HFMM_TRY(fork_near_far(P, st));
    StageTimer tn{P, P->near_st};
    tn.begin(HFMM_STAGE_P2P);
    HFMM_TRY(launch_leaf64(P, nrhs, true, false, false, direct, nullptr, false, P->y_sorted, P->near_st, true));
    tn.end(HFMM_STAGE_P2P);
    HFMM_CUDA_TRY(cudaEventRecord(P->ev_near_done, P->near_st));
    *fs = P->far_st;
    return HFMM_OK;
}

// The last pass: the locals' (and W lists') part on fs plus the near stream's sums; joins back into st.
hfmm_status join_near64(hfmm_plan_s* P, int nrhs, bool m2p, bool conj_out, cd* y, cudaStream_t fs, cudaStream_t st) {
    StageTimer tf{P, fs};
    HFMM_CUDA_TRY(cudaStreamWaitEvent(fs, P->ev_near_done, 0));
    tf.begin(HFMM_STAGE_L2P);
    HFMM_TRY(launch_leaf64(P, nrhs, false, true, m2p, false, P->y_sorted, conj_out, y, fs, false));
    tf.end(HFMM_STAGE_L2P);
    HFMM_CUDA_TRY(cudaEventRecord(P->ev_far_done, fs));
    HFMM_CUDA_TRY(cudaStreamWaitEvent(st, P->ev_far_done, 0));
    return HFMM_OK;
}

// Everything at the targets, into the caller's order (sorted: the plan's, into y): near = the stored
// blocks, l2p = the leaves' locals, m2p = the W lists, direct = the reaction blocks, ys = other sums.
hfmm_status launch_leaf64(hfmm_plan_s* P, int nrhs, bool near, bool l2p, bool m2p, bool direct, const cd* ys,
                          bool conj_out, cd* y, cudaStream_t st, bool sorted) {
    Leaf64Args A{};
    A.recs = P->leaf64;
    A.nrhs = nrhs;
    A.p = P->leaf64_p;
    A.n = P->n;
    A.qs = P->q_sorted;
    if (near) A.G = (const uint4*)P->near64_vals;
    A.EG = P->near64_E;
    A.src = P->leaf64_src;
    A.l2p = l2p;
    A.m2p = m2p;
    A.direct = direct;
    A.basis = P->basis64;
    A.w = P->leaf64_w;
    A.m2pb = P->m2p64;
    A.d = P->leaf64_d;
    A.dvals = P->d_vals;
    A.ys = ys;
    A.perm = sorted ? nullptr : P->perm;
    A.conj_out = conj_out;
    A.y = y;
    // one warp per leaf from 16 of them per SM on (leaves of at most four tiles), else four
    const bool one = P->leaf64_n >= 16 * 152 && P->leaf_max <= 64;
    const int W = one ? 1 : 4;
    const size_t sm = sizeof(double) * (128 * W * LD / 2 + (one ? 0 : W * 96) + W * LF_RING * 256 +
                                        (l2p ? 4 * (size_t)(A.p + 1) : 0));
    auto kernel = one ? leaf64_kernel<1> : leaf64_kernel<4>;
    HFMM_CUDA_TRY(smem_limit(kernel, sm));
    HFMM_CUDA_TRY(pdl_launch(kernel, dim3((unsigned)P->leaf64_n, (unsigned)nrhs), dim3(W * 32), sm, st, 0, A));
    ++P->launches;
    if (near && P->near64_large_n > 0) {
        const unsigned grid = (unsigned)std::min<int64_t>((P->near64_large_n * nrhs + 3) / 4, 16 * 152);
        near64_large_kernel<<<grid, 128, 0, st>>>(P->near64_large_tgt, P->near64_large_beg, P->near64_large_src, P->near64_large_val,
                                                     P->near64_large_n, P->q_sorted, P->n, nrhs, A.perm, conj_out, y);
        HFMM_CUDA_TRY(cudaGetLastError());
        ++P->launches;
    }
    return HFMM_OK;
}
