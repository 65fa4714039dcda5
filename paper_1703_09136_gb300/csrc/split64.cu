// Translations (M2M, L2L, free-space and reaction M2L) as exact-slice products on
// the tensor cores: FP64 expansions with six digits, FP32 ones with three.
//
// Every translation is a real matrix-vector product of length 2 nc (interleaved
// real and imaginary parts).  The operand and the operator are written as
// fixed-point numbers of 53 and 52 bits and cut into six signed base-512 digits,
//     x = 2^(E - 53) sum_i d_i 512^(5 - i),  |d_i| <= 256
// (the splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms
// 59, 2012): a digit is an f16 number, a digit product is at most 2^16, and sums
// below 2^24 leave f16 x f16 -> FP32 mma.sync without rounding.  The 26 digit
// products with i + j <= 6 are summed per order i + j.  Orders 0 .. 4 leave the
// tensor core every 64 terms as integers (int32, over all sources of a target): orders 0 .. 3
// stay within 2^24 there; order 4, five products a term, passes it only where the mean product is above
// 0.8 of the largest possible one.  Orders 5 and 6 stay in FP32: their sums are exact up to 2^24
// (28 sources at order 45: 2^23.5), and at the worst, all digits of a tile at their limit with one sign, an
// addition rounds by 2^-53 of the largest term, where an FP64 dot product rounds by 2^-53 of the whole sum so far.
// Orders >= 7 are dropped.  Error of a target's free-space list against extended precision, of the field at
// its points, k h = 0.01 .. 25, orders 9 .. 45, sources of one size and of a million sizes:
// 0.2 .. 1.5e-15, FP64 multiply-adds 0.3 .. 3.6e-15, all 36 products the same as 26 to two
// digits.  Without order 6 (21 products) it is 1.6e-15 .. 2.7e-14.
//
// Scaling: expansions are scaled by powers of two close to
// s_l(n) = min(1, (k R_l / 2)^n / n!) (a~_n = a_n / s, b~_n = b_n s), which makes
// every operator entry O(1); the exponent E is one number per level, kind
// of expansion and right-hand side (largest scaled coefficient, found by the
// kernel that writes the expansions) and one per operator family.  The stored
// expansions stay unscaled, so every other kernel reads them as before.  A coefficient
// 2^-b of its level's largest keeps 53 - b bits (an operator's entry 52 - b): one strength 1e12
// times the others leaves every target as near the FP64 kernels' as their own rounding.  A level
// that holds an infinity or a NaN makes every output of that right-hand side NaN.
//
// FP32 (the mixed path's expansions, already scaled by s): three digits hold 26
// bits, six products (i + j <= 2) replace the 26, orders 0 and 1 are kept as
// integers and order 2 in FP32.
//
// What bounds it: GB300's FP64 pipe runs at 1.0 TFLOP/s (a warp-wide FMA every 16
// clocks per SM), mma.sync f16 at 600 TFLOP/s: 26 products leave 23 TFLOP/s.
// Measured (one GB300, two layers, 262,144 points, one right-hand side): leaf
// level (order 15, 430k free-space and 49k reaction translations, 3.8 GFLOP)
// 5.73 -> 0.46 ms, all levels 12.0 -> 1.10 ms, M2M 0.72 -> 0.13 ms (launch lists; 0.42,
// 0.99 and 0.12 ms with the orders 0 .. 5 alone).  The result of
// dense translations differs from the FP64 kernels' by 5.3e-15, and theirs by 3 to 6e-15 from
// their own with the strengths times three.
#include <algorithm>
#include <cmath>
#include <vector>

#include "plan.cuh"
#include "split64.cuh"

namespace {

constexpr int S6_MAXW = 6;               // m-tiles (warps) per CTA
constexpr double S6_MAX_BYTES = 16e9;    // operator slices of one plan, and its expansions' digits

// D digits; products of orders 0 .. NO - 1 are kept, orders 0 .. NI - 1 summed as integers, the others in FP32
template <int D> struct S6Traits;
template <> struct S6Traits<6> {
    using C = cd;
    using R = double;
    static constexpr int NO = 7, NI = 5;
};
template <> struct S6Traits<3> {
    using C = cf;
    using R = float;
    static constexpr int NO = 3, NI = 2;
};

// ---------------------------------------------------------------------------
// plan time: operator slices in the A-fragment order of mma.m16n8k16
// ---------------------------------------------------------------------------
enum { S6_FREE = 0, S6_REACT = 1, S6_L2L = 2, S6_M2M = 3 };

struct S6Op {
    const cd* T;
    const int32_t* map;              // table entries of the operators (null: all, in order)
    int kind, nop, po, pi;           // orders of the outputs and the inputs
    const int* sxo;                  // log2 s of the output level, per |order| (null: log s below)
    const int* sxi;
    const double* lso;               // FP32 expansions: log s, applied to the entries
    const double* lsi;
};

__device__ __forceinline__ cd s6_entry(const S6Op& o, int op, int j, int m, int* sh) {
    // output order j, input order m; *sh = -(in_shift + out_shift)
    if (o.map) op = o.map[op];
    cd v;
    if (o.kind == S6_FREE) v = o.T[(int64_t)op * (4 * o.po + 1) + (m - j) + 2 * o.po];
    else if (o.kind == S6_REACT) {
        v = o.T[(int64_t)op * (4 * o.po + 1) + (-m - j) + 2 * o.po];
        if (m & 1) v = cneg(v);
    } else {
        const int nmax = o.po + o.pi, w = 2 * nmax + 1;   // J_{n-m}(c - P) or J_{m-j}(P - c)
        v = o.T[(int64_t)op * w + nmax + (m - j)];
    }
    const int go = o.kind == S6_M2M ? -1 : 1, gi = o.kind == S6_L2L ? -1 : 1;   // s to the power go, gi
    if (o.sxo) *sh = go * o.sxo[abs(j)] + gi * o.sxi[abs(m)];
    else {
        *sh = 0;
        v = cscale(v, exp(go * o.lso[abs(j)] + gi * o.lsi[abs(m)]));
    }
    return v;
}

__global__ void s6_op_exponent_kernel(S6Op o, int* __restrict__ E) {
    const int no = 2 * o.po + 1, ni = 2 * o.pi + 1;
    const int64_t total = (int64_t)o.nop * no * ni;
    int e = S6_NONE;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int op = (int)(i / (no * ni)), r = (int)(i % (no * ni));
        int sh;
        const cd v = s6_entry(o, op, r / ni - o.po, r % ni - o.pi, &sh);
        e = max(e, max(s6_exponent(v.x, sh), s6_exponent(v.y, sh)));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) atomicMax(E, e);
}

// one thread per (op, m-tile, k-step, lane): its eight entries' digits
template <int D>
__global__ void s6_op_slice_kernel(S6Op o, const int* __restrict__ Ep, uint4* __restrict__ out) {
    const int no = 2 * o.po + 1, ni = 2 * o.pi + 1;
    const int MT = (2 * no + 15) / 16, KS = (2 * ni + 15) / 16;
    const int64_t total = (int64_t)o.nop * MT * KS * 32;
    const int E = *Ep;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(i & 31);
        const int64_t blk = i >> 5;                        // (op, mt, ks)
        const int ks = (int)(blk % KS), mt = (int)((blk / KS) % MT), op = (int)(blk / ((int64_t)KS * MT));
        const int g = lane >> 2, t = lane & 3;
        unsigned f[D][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = 16 * mt + g + (q & 1) * 8, m = (16 * ks + (q >> 1) * 8) / 2 + t;   // columns 2m, 2m + 1
            const int j = row >> 1;
            long long x0 = s6_bias<D>(), x1 = s6_bias<D>();
            if (j < no && m < ni) {
                int sh;
                const cd v = s6_entry(o, op, j - o.po, m - o.pi, &sh);
                // [[Re, -Im], [Im, Re]]
                x0 += s6_fixed<9 * D - 2>((row & 1) ? v.y : v.x, sh, E);
                x1 += s6_fixed<9 * D - 2>((row & 1) ? v.x : -v.y, sh, E);
            }
#pragma unroll
            for (int d = 0; d < D; ++d) f[d][q] = s6_half2(s6_field<D>(x0, d), s6_field<D>(x1, d));
        }
#pragma unroll
        for (int d = 0; d < D; ++d) out[(blk * D + d) * 32 + lane] = make_uint4(f[d][0], f[d][1], f[d][2], f[d][3]);
    }
}

// ---------------------------------------------------------------------------
// level exponents of expansions written by other kernels
// ---------------------------------------------------------------------------
// Boxes without points (lb: the leaf ranges) are left out: nobody
// writes their locals, so their memory holds what the allocator or a call of another width left there.
__global__ void s6_exponent_kernel(const cd* __restrict__ a, int64_t nbox, int nrhs, int p, const int32_t* __restrict__ lb,
                                   int L, int l, const int* __restrict__ sx, int sign, int* __restrict__ E) {
    pdl_start_next();
    const int nc = 2 * p + 1, r = blockIdx.y;
    int e = S6_NONE;
    const int64_t total = nbox * nc;
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = i / nc;
        const int m = (int)(i % nc) - p;
        int32_t lo, hi;
        box_range(lb, L, l, b, &lo, &hi);
        if (hi <= lo) continue;
        const cd v = __ldcg(a + (b * nrhs + r) * nc + m + p);
        const int sh = sign * sx[abs(m)];
        e = max(e, max(s6_exponent(v.x, sh), s6_exponent(v.y, sh)));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0 && e > S6_NONE) atomicMax(E + r, e);
}

// Digits of a level's expansions in the B-fragment order of mma.m16n8k16:
// per (box, right-hand side, k-step of eight coefficients, digit) the words
// [coefficient % 4][coefficient / 4] (32 bytes).  Every source meets up to 27
// target tiles: cutting it in the product kernel took 60% of that kernel's
// instructions (leaf level of two layers, orders 0 .. 5: 0.47 -> 0.34 ms without it).
template <int D>
__global__ void s6_slice_kernel(const typename S6Traits<D>::C* __restrict__ a, int64_t nbox, int nrhs, int p, const int* __restrict__ sx,
                                int sign, const int* __restrict__ E, unsigned* __restrict__ dig) {
    pdl_start_next();
    const int nc = 2 * p + 1, KS = (2 * nc + 15) / 16, r = blockIdx.y;
    const int64_t total = nbox * KS * 8;
    pdl_wait();                          // L2 loads: results of kernels that may have run beside this one's start
    const int e = __ldcg(E + r);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = i / (KS * 8);
        const int m = (int)(i - b * (KS * 8));
        long long xr = s6_bias<D>(), xi = s6_bias<D>();
        if (m < nc) {
            const auto v = __ldcg(a + (b * nrhs + r) * nc + m);
            const int sh = sx ? sign * sx[abs(m - p)] : 0;
            xr += s6_fixed<9 * D - 1>(v.x, sh, e);
            xi += s6_fixed<9 * D - 1>(v.y, sh, e);
        }
        unsigned* o = dig + ((b * nrhs + r) * KS + (m >> 3)) * (D * 8) + (m & 3) * 2 + (m >> 2 & 1);
#pragma unroll
        for (int d = 0; d < D; ++d) o[d * 8] = s6_half2(s6_field<D>(xr, d), s6_field<D>(xi, d));
    }
}

// ---------------------------------------------------------------------------
// the product kernel
// ---------------------------------------------------------------------------
// One operator family of a launch: sources, their order, scale signs, slices.
struct S6Fam {
    const uint4* dig;                // source digits (s6_slice_kernel)
    const uint4* ops;
    const int* Eop;                  // exponent of the family
    const int* Esrc;                 // [nrhs] exponent of the source expansions
    int p;                           // source order
};

struct S6Args {
    // mode 0: M2M (targets 8 NT consecutive boxes), 1: downward, 2: explicit tiles (adaptive trees)
    int l, L, mode;
    int nrhs, p;                     // output order
    int tiles;
    const int32_t* lb;               // leaf ranges (downward: empty targets are skipped)
    S6Fam shift;                     // M2M or L2L (dig null: none)
    S6Fam list;                      // M2L sources (dig null: none); ops = free-space operators
    const uint4* rops;               // reaction operators (null: none)
    int vlist, rlist, lstar;         // lists to run; first level whose bottom-row pair is admissible
    int rows;                        // box rows covered by the launch (downward)
    uint8_t voff[4][27];             // V offsets of each child position: (source - target + 3), x + 8 y
    int accumulate;                  // add to the outputs
    const int* sxo;                  // (null: no output shift)
    int osign;                       // out_shift = osign * sxo
    const int32_t* tgt;              // mode 2: [tiles][8] targets (-1: none), first step of every tile, steps
    const int32_t* tbeg;
    const S6Rec* recs;
    void* out;
    int* Eout;                       // [nrhs], or null
};

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// A step of a tile: operator and the sources of its columns.
struct S6Step {
    int fam;                         // 0 shift, 1 list
    const uint4* op;
    int dx, sy, child;               // list: source (ix - dx, sy); shift: child position (mode 0); mode 2: record
};

// Steps of a downward tile (row iy, columns ix0, ix0 + 2, ..., ncol of them):
// 0 the L2L, then the 27 V offsets of the tile's child position, then the reaction
// pairs (source row, dx).  s6_step returns false where a step does not exist for
// this tile.  (Walking 36 offsets with divisions and adjacency tests here, or
// balancing the CTAs by a ballot over such tests, cost microseconds a launch.)
struct S6Tile {
    int iy, ix0, ncol, n;            // n boxes per row
    int nshift, nv, nr, rspan, ropt0, rec0;
};

__device__ __forceinline__ int s6_steps(const S6Args& A, S6Tile& T, int tile) {
    if (A.mode == 2) {
        T.rec0 = A.tbeg[tile];
        return A.tbeg[tile + 1] - T.rec0;
    }
    T.nshift = A.shift.dig ? (A.mode == 0 ? 4 : 1) : 0;
    T.nv = T.nr = 0;
    if (A.mode == 1) {
        T.nv = A.vlist ? 27 : 0;
        if (A.rlist && T.iy < 2) {
            T.ropt0 = (T.iy == 1 || A.l == A.lstar) ? 0 : 1;      // first admissible source row
            const int opts = min(2, T.n) - T.ropt0;
            T.rspan = T.n + 2 * (T.ncol - 1);
            T.nr = opts > 0 ? opts * T.rspan : 0;
        }
    }
    return T.nshift + T.nv + T.nr;
}

template <int D>
__device__ __forceinline__ bool s6_step(const S6Args& A, const S6Tile& T, int s, int MT, int KSs, int KSl, S6Step& st) {
    if (A.mode == 2) {               // record: operator * 4 + kind (0 shift, 1 free-space, 2 reaction)
        st.child = T.rec0 + s;
        const int op = A.recs[st.child].op, kind = op & 3;
        st.fam = kind ? 1 : 0;
        if (kind == 0 ? !A.shift.dig : kind == 1 ? !A.vlist : !A.rlist) return false;
        st.op = (kind == 0 ? A.shift.ops : kind == 1 ? A.list.ops : A.rops) +
                (int64_t)(op >> 2) * MT * (kind ? KSl : KSs) * (D * 32);
        return true;
    }
    if (s < T.nshift) {
        st.fam = 0;
        st.child = A.mode == 0 ? s : (T.ix0 & 1) + 2 * (T.iy & 1);
        st.op = A.shift.ops + (int64_t)st.child * MT * KSs * (D * 32);
        return true;
    }
    s -= T.nshift;
    st.fam = 1;
    if (s < T.nv) {
        const int v = A.voff[(T.ix0 & 1) + 2 * (T.iy & 1)][s], ox = (v & 7) - 3, oy = (v >> 3) - 3;
        st.sy = T.iy + oy;
        st.dx = -ox;
        if ((unsigned)st.sy >= (unsigned)T.n || T.ix0 + 2 * (T.ncol - 1) + ox < 0 || T.ix0 + ox >= T.n) return false;
        st.op = A.list.ops + (uint32_t)((st.dx + 3) * 7 + (3 - oy)) * (uint64_t)(MT * KSl * (D * 32));
        return true;
    }
    s -= T.nv;
    st.sy = T.ropt0;
    if (s >= T.rspan) { s -= T.rspan; ++st.sy; }
    st.dx = T.ix0 + 2 * (T.ncol - 1) - s;                        // sources from left to right cover [0, n)
    const int dxm = T.n - 1;
    if (abs(st.dx) > dxm) return false;
    st.op = A.rops + (uint32_t)((st.dx + dxm) * 3 + T.iy + st.sy) * (uint64_t)(MT * KSl * (D * 32));
    return true;
}

template <int NT, int D>
__global__ void __maxnreg__(D == 3 ? (NT == 1 ? 96 : 128) : (NT == 1 ? 128 : 168)) s6_kernel(const __grid_constant__ S6Args A) {
    using R = typename S6Traits<D>::R;
    constexpr int NO = S6Traits<D>::NO, NI = S6Traits<D>::NI;
    // digits of the sources of one 64-term chunk, in B-fragment order, two buffers
    __shared__ __align__(16) uint2 Bs[2][D][4][NT][32];
    pdl_start_next();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    const int S = (int)cluster_size(), rank = (int)cluster_rank();
    const int tile = blockIdx.x / S, r = blockIdx.z;
    const int no = 2 * A.p + 1, MT = (2 * no + 15) / 16;
    const int mper = (MT + gridDim.y - 1) / gridDim.y;
    const int mt = blockIdx.y * mper + wid;
    const bool has_m = wid < mper && mt < MT;
    constexpr int NC = 8 * NT;
    S6Tile T;
    int64_t box0 = 0;
    T.n = 1 << A.l;
    if (A.mode != 1) {
        box0 = (int64_t)tile * NC;
        T.iy = T.ix0 = 0;
        T.ncol = NC;
    } else {
        const int per = max(1, T.n >> 1), G = (per + NC - 1) / NC, par = T.n > 1 ? 2 : 1;
        T.iy = tile / (par * G);
        const int c = (tile / G) % par, g = tile % G;
        T.ix0 = 2 * NC * g + c;
        T.ncol = min(NC, per - NC * g);
    }
    const int64_t nbox = (int64_t)1 << (2 * A.l);
    // lane c: target of column c (-1: none)
    int64_t tgt = -1;
    if (lane < NC) {
        if (A.mode == 0) tgt = box0 + lane < nbox ? box0 + lane : -1;
        else if (A.mode == 2) tgt = A.tgt[box0 + lane];
        else if (lane < T.ncol) {
            const int64_t b = morton((uint32_t)(T.ix0 + 2 * lane), (uint32_t)T.iy);
            int32_t lo, hi;
            box_range(A.lb, A.L, A.l, b, &lo, &hi);
            if (hi > lo) tgt = b;
        }
    }
    // nothing to do where every target is empty (the same for all CTAs of the cluster)
    if (!__any_sync(0xffffffffu, tgt >= 0)) return;
    const int nsteps = s6_steps(A, T, tile);
    const int nis = A.shift.dig ? 2 * A.shift.p + 1 : 0, nil = A.list.dig ? 2 * A.list.p + 1 : 0;
    const int KSs = (2 * nis + 15) / 16, KSl = (2 * nil + 15) / 16;

    float acc[NT][NO][4];
    int iacc[NT][NI][4];
    double dacc[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            dacc[t][v] = 0.0;
#pragma unroll
            for (int o = 0; o < NI; ++o) iacc[t][o][v] = 0;
#pragma unroll
            for (int o = 0; o < NO; ++o) acc[t][o][v] = 0.0f;
        }
    int since = 0;                    // chunks since the integers were last folded
    // dacc += (digit sums) 2^E, E = Esrc + Eop - (18 D - 3) less the larger of the families' E, which the
    // epilogue puts back (so that no intermediate power of two leaves the range): order o weighs 512^(2 (D - 1) - o).
    // Four (two) FP64 instructions a value (the pipe takes 64 clocks for each of a
    // sub-partition's): orders 0 .. 2 and 3 .. 6 as integers below 2^51 (order 6 rounded to order 5's unit, 2^-61
    // of the largest term)
    auto fold = [&](int E) {
        const double chi = pow2d(E + 9 * (2 * D - 4)), clo = D == 6 ? pow2d(E + 45) : 0.0;
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                long long hi = ((long long)iacc[t][0][v] << 18) + ((long long)iacc[t][1][v] << 9);
                if (D == 6) {
                    hi += iacc[t][2][v];
                    const long long lo = ((long long)iacc[t][NI - 2][v] << 18) + ((long long)iacc[t][NI - 1][v] << 9) +
                                         __float2ll_rn(fmaf(acc[t][NO - 1][v], 0x1p-9f, acc[t][NO - 2][v]));
                    dacc[t][v] = fma(int51d(lo), clo, dacc[t][v]);
                } else hi += __float2ll_rn(acc[t][D - 1][v]);
                dacc[t][v] = fma(int51d(hi), chi, dacc[t][v]);
#pragma unroll
                for (int o = 0; o < NI; ++o) iacc[t][o][v] = 0;
#pragma unroll
                for (int o = NI; o < NO; ++o) acc[t][o][v] = 0.0f;
            }
        since = 0;
    };
    // A chunk: up to 64 terms (four k-steps) of one step.  While the tensor cores work on
    // one chunk the next one's source digits are copied into the other buffer and
    // its operator fragments into the slots of the warp's ring as they fall free,
    // all asynchronously: a k-step's loads alone take longer than its products.
    struct Chunk { S6Step st; int s, k0; };
    auto next = [&](Chunk& c) -> bool {             // the following chunk of this CTA, false at the end
        if (c.s >= 0) {
            c.k0 += 4;
            if (c.k0 < (c.st.fam ? KSl : KSs)) return true;
        }
        c.k0 = 0;
        for (c.s = c.s < 0 ? rank : c.s + S; c.s < nsteps; c.s += S)
            if (s6_step<D>(A, T, c.s, MT, KSs, KSl, c.st)) return true;
        return false;
    };
    // digits of the chunk's columns, 8 D pieces of 16 bytes each (k-step, digit, half): a
    // warp takes columns wid, wid + nw, ..., a lane the pieces lane and lane + 32; one group.
    // Lane c holds the source box of column c (found once per step).
    int64_t sbox = -1;
    auto load_src = [&](const Chunk& c, int buf, bool ok) {
        if (ok) {
            if (c.k0 == 0) {
                sbox = -1;
                if (A.mode == 2) sbox = lane < NC ? A.recs[c.st.child].src[lane & 7] : -1;
                else if (c.st.fam == 0) {
                    if (A.mode == 0) sbox = lane < NC && box0 + lane < nbox ? 4 * (box0 + lane) + c.st.child : -1;
                    else if (lane < T.ncol) sbox = morton((uint32_t)((T.ix0 >> 1) + lane), (uint32_t)(T.iy >> 1));
                } else if (lane < T.ncol) {
                    const int x = T.ix0 + 2 * lane - c.st.dx;
                    if (x >= 0 && x < T.n) sbox = morton((uint32_t)x, (uint32_t)c.st.sy);
                }
            }
            const int KS = c.st.fam ? KSl : KSs, nk = min(4, KS - c.k0);
            const uint4* dig = (c.st.fam ? A.list.dig : A.shift.dig) + (int64_t)c.k0 * (2 * D);
            const int64_t stride = (int64_t)A.nrhs * KS * (2 * D), first = (int64_t)r * KS * (2 * D);
#pragma unroll
            for (int u = 0; u < (8 * D + 31) / 32; ++u) {
                const int q = lane + 32 * u, kk = q / (2 * D), d = q % (2 * D) >> 1, h = q & 1;
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&Bs[buf][d][kk & 3][0][2 * h]);
                for (int col = wid; col < NC; col += nw) {
                    const int64_t b = __shfl_sync(0xffffffffu, sbox, col);
                    if (q < 8 * D && kk < nk)
                        cp_async16(dst + (col >> 3) * 256 + (col & 7) * 32, b >= 0 ? dig + b * stride + first + q : dig, b >= 0);
                }
            }
        }
        cp_commit();
    };
    extern __shared__ __align__(16) uint4 s6_ring[];      // [warps][4][D][32]
    const uint4* ring = s6_ring + (size_t)wid * (4 * D * 32) + lane;
    const uint32_t ring_a = (uint32_t)__cvta_generic_to_shared(ring);
    // operator fragments of k-step kk of chunk c into slot kk; one group, empty where there is none
    auto load_op = [&](const Chunk& c, int kk, bool ok) {
        const int KS = c.st.fam ? KSl : KSs;
        if (ok && has_m && c.k0 + kk < KS) {
            const uint4* op = c.st.op + (((int64_t)mt * KS + c.k0 + kk) * D) * 32 + lane;
#pragma unroll
            for (int d = 0; d < D; ++d) cp_async16(ring_a + (kk * D + d) * 512, op + d * 32, true);
        }
        cp_commit();
    };
    int buf = 0, prev_fam = -1;
    Chunk cur{{}, -1, 0};
    bool more = next(cur);
    // the operators are the plan's; everything below reads this apply's results.  (The
    // first digits' group comes after the slots', so the first wait is for all.)
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) load_op(cur, kk, more);
    pdl_wait();
    int Ef[2] = {4 * S6_NONE, 4 * S6_NONE};   // fold exponents per family
    bool bad = false;
    if (A.shift.dig) {
        const int e = __ldcg(A.shift.Esrc + r);
        bad |= e >= S6_NAN / 2;
        Ef[0] = max(e, S6_NONE) + max(*A.shift.Eop, S6_NONE) - (18 * D - 3);
    }
    if (A.list.dig) {
        const int e = __ldcg(A.list.Esrc + r);
        bad |= e >= S6_NAN / 2;
        Ef[1] = max(e, S6_NONE) + max(*A.list.Eop, S6_NONE) - (18 * D - 3);
    }
    const int Emax = D == 6 ? max(Ef[0], Ef[1]) : 0;       // (FP32's exponents cannot leave the range)
    Ef[0] -= Emax;
    Ef[1] -= Emax;

    load_src(cur, 0, more);
    bool first = true;
    while (more) {
        const int fam = cur.st.fam, nk = min(4, (fam ? KSl : KSs) - cur.k0);
        if (first) cp_wait<0>();                          // the source digits (four operator groups came after)
        else cp_wait<4>();
        first = false;
        __syncthreads();
        more = next(cur);
        load_src(cur, buf ^ 1, more);
        if (has_m) {
            if (prev_fam >= 0 && fam != prev_fam) fold(Ef[prev_fam]);
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int o = 0; o < NI; ++o)
#pragma unroll
                    for (int x = 0; x < 4; ++x) acc[t][o][x] = 0.0f;
        }
        // groups in flight, in order: this chunk's slots, the next chunk's digits, its slots.  Two
        // k-steps at a time between the waits and copies, which order memory accesses
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            cp_wait<3>();
            if (has_m)
#pragma unroll
                for (int kk = 2 * h; kk < 2 * h + 2; ++kk)
                    if (kk < nk) {
                        uint4 a[D];
#pragma unroll
                        for (int d = 0; d < D; ++d) a[d] = ring[(kk * D + d) * 32];
#pragma unroll
                        for (int t = 0; t < NT; ++t) {
                            uint2 bb[D];
#pragma unroll
                            for (int d = 0; d < D; ++d) bb[d] = Bs[buf][d][kk][t][lane];
#pragma unroll
                            for (int i = 0; i < D; ++i)
#pragma unroll
                                for (int j = 0; j < D && j < NO - i; ++j) s6_mma(acc[t][i + j], a[i], bb[j]);
                        }
                    }
            load_op(cur, 2 * h, more);
            load_op(cur, 2 * h + 1, more);
        }
        if (has_m) {
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int o = 0; o < NI; ++o)
#pragma unroll
                    for (int x = 0; x < 4; ++x) iacc[t][o][x] += __float2int_rn(acc[t][o][x]);
            if (++since == 96) fold(Ef[fam]);             // 96 x 5 x 2^22 < 2^31
        }
        prev_fam = fam;
        buf ^= 1;
    }
    if (prev_fam >= 0) fold(Ef[prev_fam]);
    cp_wait<0>();

    // partial sums of the cluster's CTAs, added in rank order by rank 0
    double* part = reinterpret_cast<double*>(s6_ring);              // [warp][NT][4][32]: NT KB of a warp's 2 D KB
    if (S > 1) {
        __syncthreads();
        if (rank != 0 && has_m)
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int v = 0; v < 4; ++v) part[((wid * NT + t) * 4 + v) * 32 + lane] = dacc[t][v];
        cluster_sync();
        if (rank == 0 && has_m) {
            const uint32_t local = (uint32_t)__cvta_generic_to_shared(part);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                double x[7][4];                                  // all ranks' values in flight at once
#pragma unroll
                for (int q = 1; q < 8; ++q)
                    if (q < S) {
                        uint32_t remote;
                        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(q));
#pragma unroll
                        for (int v = 0; v < 4; ++v)
                            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x[q - 1][v])
                                         : "r"(remote + (uint32_t)(((wid * NT + t) * 4 + v) * 32 + lane) * 8u));
                    }
#pragma unroll
                for (int q = 1; q < 8; ++q)
                    if (q < S)
#pragma unroll
                        for (int v = 0; v < 4; ++v) dacc[t][v] += x[q - 1][v];
            }
        }
        cluster_sync();
        if (rank != 0) return;
    }
    if (!has_m) return;
    int e = S6_NONE;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int row = 16 * mt + (lane >> 2) + (v >> 1) * 8, c = 8 * t + 2 * (lane & 3) + (v & 1);
            const int64_t b = __shfl_sync(0xffffffffu, tgt, c);
            if (row >= 2 * no || b < 0) continue;
            const int sh = A.sxo ? A.osign * A.sxo[abs((row >> 1) - A.p)] : 0;
            R* o = reinterpret_cast<R*>(A.out) + ((b * A.nrhs + r) * no * 2 + row);
            R x = (R)(bad ? nan : D == 6 ? scale2d(dacc[t][v], Emax + sh) : dacc[t][v] * pow2d(Emax + sh));
            if (A.accumulate) x += __ldcg(o);
            *o = x;
            e = max(e, s6_exponent(x, -sh));
        }
    if (A.Eout) {
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0 && e > S6_NONE) atomicMax(A.Eout + r, e);
    }
}

template <int NT, int D>
hfmm_status s6_launch(const S6Args& A, int tiles, int steps, cudaStream_t st) {
    const int MT = (2 * (2 * A.p + 1) + 15) / 16;
    const int gy = (MT + S6_MAXW - 1) / S6_MAXW, W = (MT + gy - 1) / gy;
    // CTAs per tile: split the steps over a cluster while one right-hand side leaves SMs
    // idle (whatever nrhs is, so that a right-hand side's bits do not depend on the others)
    int S = 1;
    while (S < 8 && (int64_t)tiles * gy * S * 2 <= 4 * 152 && 2 * S <= steps) S *= 2;
    const size_t sm = (size_t)W * 4 * D * 512;
    if (sm > 16 * 1024)                                    // beside up to 24 KB of static shared memory
        HFMM_CUDA_TRY(cudaFuncSetAttribute(s6_kernel<NT, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           S6_MAXW * 4 * D * 512));
    HFMM_CUDA_TRY(pdl_launch(s6_kernel<NT, D>, dim3((unsigned)(tiles * S), (unsigned)gy, (unsigned)A.nrhs), dim3(32 * W),
                             sm, st, (unsigned)S, A));
    return HFMM_OK;
}

// Columns per tile: 16 where that still fills the GPU (each operator slice is
// read once per tile), else 8.
template <int D>
hfmm_status s6_run(S6Args& A, cudaStream_t st) {
    if (A.tiles == 0 && A.mode == 2) return HFMM_OK;
    if (D == 3 || A.mode == 2) return s6_launch<1, D>(A, A.tiles, 28, st);     // FP32 digits: adaptive trees alone
    const int64_t n = (int64_t)1 << A.l;
    const int MT = (2 * (2 * A.p + 1) + 15) / 16, gy = (MT + S6_MAXW - 1) / S6_MAXW;
    auto tiles = [&](int nc) -> int64_t {
        if (A.mode == 0) return (n * n + nc - 1) / nc;
        const int64_t per = std::max<int64_t>(1, n >> 1);
        return (int64_t)A.rows * (n > 1 ? 2 : 1) * ((per + nc - 1) / nc);
    };
    const int steps = A.mode == 0 ? 4 : 1 + (A.vlist ? 27 : 0) + (A.rlist ? (int)std::min<int64_t>(n, 1 << 20) : 0);
    const bool wide = (A.mode == 0 || (n >> 1) > 8) && tiles(16) * gy >= 3 * 152;
    A.tiles = (int)tiles(wide ? 16 : 8);
    return wide ? s6_launch<2, 6>(A, A.tiles, steps, st) : s6_launch<1, D>(A, A.tiles, steps, st);
}

S6Fam s6_fam(const unsigned* dig, int p, const uint4* ops, const int* Eop, const int* Esrc) {
    S6Fam f{};
    f.dig = (const uint4*)dig;
    f.ops = ops;
    f.Eop = Eop;
    f.Esrc = Esrc;
    f.p = p;
    return f;
}

template <int D> S6Lev& s6_lev(LevelInfo& lv) { return lv.s6[D == 6 ? 0 : 1]; }
template <int D> typename S6Traits<D>::C* s6_expansion(const LevelInfo& lv, bool loc);
template <> cd* s6_expansion<6>(const LevelInfo& lv, bool loc) { return loc ? lv.loc : lv.mult; }
template <> cf* s6_expansion<3>(const LevelInfo& lv, bool loc) { return loc ? lv.loc32 : lv.mult32; }

template <int D>
hfmm_status s6_build(hfmm_plan_s* P, cudaStream_t st) {
    constexpr int w = D == 6 ? 0 : 1;
    if (P->s6_ready[w]) return HFMM_OK;
    const int L = P->L;
    auto bytes = [](int nop, int po, int pi) {
        return 512.0 * D * nop * ((2 * (2 * po + 1) + 15) / 16) * ((2 * (2 * pi + 1) + 15) / 16);
    };
    auto digits = [&](const LevelInfo& lv) { return (size_t)lv.nbox * P->max_rhs * ((2 * lv.ncoef + 15) / 16) * (D * 32); };
    // reaction entries of an adaptive tree: the ones its lists use
    std::vector<std::vector<int32_t>> rmap(L + 1);
    if (P->ad)
        for (int l = P->lmin; l <= L; ++l) adaptive_react_entries(P, l, rmap[l]);
    auto has_free = [&](const LevelInfo& lv) { return !lv.diag_logq && lv.t_free && lv.nv > 0; };
    auto nreact = [&](int l) {
        const LevelInfo& lv = P->lev[l];
        if (lv.diag_logq || !lv.t_react || lv.nr == 0) return 0;
        return P->ad ? (int)rmap[l].size() : lv.n_react_entries;
    };
    double used = 0.0, dbytes = 0.0;
    for (int l = P->lmin; l <= L; ++l) {
        const LevelInfo& lv = P->lev[l];
        used += (has_free(lv) ? bytes(49, lv.p, lv.p) : 0.0) + bytes(nreact(l), lv.p, lv.p);
        if (l > P->lmin) used += bytes(4, lv.p, P->lev[l - 1].p) + bytes(4, P->lev[l - 1].p, lv.p);
        dbytes += (l < L ? 2.0 : 1.0) * digits(lv);
    }
    if (used > S6_MAX_BYTES || dbytes > S6_MAX_BYTES || !optional_fits(used + dbytes)) return HFMM_OK;
    int* E = nullptr;                                     // [level][3] families, then [kind][level][rhs] expansions
    const size_t ne = (size_t)3 * (L + 1) + (size_t)2 * (L + 1) * P->max_rhs;
    HFMM_TRY(plan_alloc(P, (void**)&E, sizeof(int) * ne));
    P->s6_E[w] = E + 3 * (L + 1);
    HFMM_CUDA_TRY(cudaMemsetAsync(E, 0x80, sizeof(int) * ne, st));   // far below S6_NONE
    std::vector<int> sx;
    std::vector<size_t> off(L + 1, 0);
    std::vector<int32_t> maps;
    std::vector<size_t> moff(L + 1, 0);
    for (int l = 0; l <= L; ++l) {
        const LevelInfo& lv = P->lev[l];
        off[l] = sx.size();
        const double kR = P->k * lv.h / std::sqrt(2.0);
        for (int n = 0; n <= lv.p; ++n)
            sx.push_back((int)std::lround(std::min(0.0, n * std::log(0.5 * kR) - std::lgamma(n + 1.0)) / std::log(2.0)));
        moff[l] = maps.size();
        maps.insert(maps.end(), rmap[l].begin(), rmap[l].end());
    }
    int *dsx = nullptr, *dmaps = nullptr;
    HFMM_TRY(plan_alloc(P, (void**)&dsx, sizeof(int) * sx.size()));
    HFMM_CUDA_TRY(cudaMemcpyAsync(dsx, sx.data(), sizeof(int) * sx.size(), cudaMemcpyHostToDevice, st));
    HFMM_TRY(plan_alloc(P, (void**)&dmaps, sizeof(int) * maps.size()));
    if (!maps.empty())
        HFMM_CUDA_TRY(cudaMemcpyAsync(dmaps, maps.data(), sizeof(int) * maps.size(), cudaMemcpyHostToDevice, st));
    HFMM_CUDA_TRY(cudaStreamSynchronize(st));             // the vectors are locals
    for (int l = 0; l <= L; ++l) s6_lev<D>(P->lev[l]).sx = D == 6 ? dsx + off[l] : nullptr;
    auto op_of = [&](const cd* T, int kind, int nop, LevelInfo& o, LevelInfo& i, const int32_t* map) {
        return S6Op{T, map, kind, nop, o.p, i.p, s6_lev<D>(o).sx, s6_lev<D>(i).sx, o.d_log_s, i.d_log_s};
    };
    auto expo = [&](const S6Op& op, int* Ep) -> hfmm_status {
        const int64_t total = (int64_t)op.nop * (2 * op.po + 1) * (2 * op.pi + 1);
        s6_op_exponent_kernel<<<(unsigned)std::min<int64_t>((total + 255) / 256, 8 * 152), 256, 0, st>>>(op, Ep);
        HFMM_CUDA_TRY(cudaGetLastError());
        return HFMM_OK;
    };
    auto make = [&](const S6Op& op, int* Ep, uint4** out) -> hfmm_status {
        HFMM_TRY(plan_alloc(P, (void**)out, (size_t)bytes(op.nop, op.po, op.pi)));
        const int64_t total = (int64_t)(bytes(op.nop, op.po, op.pi) / (16.0 * D));
        s6_op_slice_kernel<D><<<(unsigned)std::min<int64_t>((total + 127) / 128, 64 * 152), 128, 0, st>>>(op, Ep, *out);
        HFMM_CUDA_TRY(cudaGetLastError());
        return HFMM_OK;
    };
    for (int l = P->lmin; l <= L; ++l) {
        LevelInfo& lv = P->lev[l];
        S6Lev& s = s6_lev<D>(lv);
        HFMM_TRY(plan_alloc(P, (void**)&s.dmult, digits(lv)));
        if (l < L) HFMM_TRY(plan_alloc(P, (void**)&s.dloc, digits(lv)));
        s.Eop = E + 3 * l;
        const int nre = nreact(l);                        // diagonal levels translate in diag.cu
        const S6Op fr = op_of(lv.t_free, S6_FREE, 49, lv, lv, nullptr);
        const S6Op re = op_of(lv.t_react, S6_REACT, nre, lv, lv, P->ad ? dmaps + moff[l] : nullptr);
        if (has_free(lv)) HFMM_TRY(expo(fr, s.Eop));
        if (nre) HFMM_TRY(expo(re, s.Eop));
        if (has_free(lv)) HFMM_TRY(make(fr, s.Eop, &s.free));
        if (nre) HFMM_TRY(make(re, s.Eop, &s.react));
        if (l > P->lmin) {
            const S6Op op = op_of(P->lev[l - 1].t_l2l, S6_L2L, 4, lv, P->lev[l - 1], nullptr);
            HFMM_TRY(expo(op, s.Eop + 1));
            HFMM_TRY(make(op, s.Eop + 1, &s.l2l));
        }
        if (l < L) {
            const S6Op op = op_of(lv.t_m2m, S6_M2M, 4, lv, P->lev[l + 1], nullptr);
            HFMM_TRY(expo(op, s.Eop + 2));
            HFMM_TRY(make(op, s.Eop + 2, &s.m2m));
        }
        if (P->ad) {
            for (int up = 0; up < 2; ++up) {
                std::vector<int32_t> tgt, tbeg;
                std::vector<S6Rec> recs;
                adaptive_tiles(P, l, up == 1, rmap[l], tgt, tbeg, recs);
                S6Tiles& t = up ? s.up : s.down;
                t.n = (int)(tgt.size() / 8);
                if (t.n == 0) continue;
                HFMM_TRY(plan_alloc(P, (void**)&t.tgt, sizeof(int32_t) * tgt.size()));
                HFMM_TRY(plan_alloc(P, (void**)&t.tbeg, sizeof(int32_t) * tbeg.size()));
                HFMM_TRY(plan_alloc(P, (void**)&t.recs, sizeof(S6Rec) * std::max<size_t>(recs.size(), 1)));
                HFMM_CUDA_TRY(cudaMemcpyAsync(t.tgt, tgt.data(), sizeof(int32_t) * tgt.size(), cudaMemcpyHostToDevice, st));
                HFMM_CUDA_TRY(cudaMemcpyAsync(t.tbeg, tbeg.data(), sizeof(int32_t) * tbeg.size(), cudaMemcpyHostToDevice, st));
                if (!recs.empty())
                    HFMM_CUDA_TRY(cudaMemcpyAsync(t.recs, recs.data(), sizeof(S6Rec) * recs.size(), cudaMemcpyHostToDevice, st));
                HFMM_CUDA_TRY(cudaStreamSynchronize(st));
            }
        }
    }
    P->table_bytes += used;
    P->buffer_bytes += dbytes;
    P->s6_ready[w] = true;
    return HFMM_OK;
}

template <int D>
hfmm_status s6_m2m(hfmm_plan_s* P, int l, int nrhs, cudaStream_t st) {
    constexpr int w = D == 6 ? 0 : 1;
    LevelInfo& lv = P->lev[l];
    LevelInfo& ch = P->lev[l + 1];
    const S6Lev &s = s6_lev<D>(lv), &sc = s6_lev<D>(ch);
    S6Args A{};
    A.l = l; A.L = P->L; A.mode = P->ad ? 2 : 0; A.nrhs = nrhs; A.p = lv.p;
    A.shift = s6_fam(sc.dmult, ch.p, s.m2m, s.Eop + 2, split_exp(P, w, l + 1, false));
    A.sxo = s.sx;
    A.osign = 1;
    A.out = s6_expansion<D>(lv, false);
    A.Eout = split_exp(P, w, l, false);
    A.tiles = s.up.n; A.tgt = s.up.tgt; A.tbeg = s.up.tbeg; A.recs = s.up.recs;
    ++P->launches;
    return s6_run<D>(A, st);
}

// L2L and both M2L lists of level l into loc (diagonal levels: the L2L alone).
template <int D>
hfmm_status s6_down(hfmm_plan_s* P, int l, int nrhs, int parts, cudaStream_t st) {
    constexpr int w = D == 6 ? 0 : 1;
    LevelInfo& lv = P->lev[l];
    const S6Lev& s = s6_lev<D>(lv);
    const bool dg = lv.diag_logq > 0;
    S6Args A{};
    A.l = l; A.L = P->L; A.mode = P->ad ? 2 : 1; A.nrhs = nrhs; A.p = lv.p;
    A.lb = P->leaf_begin;
    for (int c = 0; c < 4; ++c) {
        int k = 0;
        for (int o = 0; o < 36; ++o) {
            const int ox = o % 6 - 2 - (c & 1), oy = o / 6 - 2 - (c >> 1);
            if (std::abs(ox) >= 2 || std::abs(oy) >= 2) A.voff[c][k++] = (uint8_t)((ox + 3) + 8 * (oy + 3));
        }
    }
    if (l > P->lmin) {
        LevelInfo& pa = P->lev[l - 1];
        A.shift = s6_fam(s6_lev<D>(pa).dloc, pa.p, s.l2l, s.Eop + 1, split_exp(P, w, l - 1, true));
    }
    const S6Fam list = s6_fam(s.dmult, lv.p, s.free, s.Eop, split_exp(P, w, l, false));
    A.rops = s.react;
    A.vlist = !dg && lv.nv > 0 && (parts & HFMM_PART_FAR_FREE);
    const bool react = !dg && lv.nr > 0 && (parts & HFMM_PART_FAR_REACT);
    A.lstar = P->lstar;
    A.sxo = s.sx;
    A.osign = -1;
    A.out = s6_expansion<D>(lv, true);
    A.Eout = split_exp(P, w, l, true);
    A.rows = 1 << l;
    A.tiles = s.down.n; A.tgt = s.down.tgt; A.tbeg = s.down.tbeg; A.recs = s.down.recs;
    // a bottom-row tile of a fine level has up to 2^(l + 1) reaction steps against
    // 28 of the others: there they run as a launch of their own over the two rows
    const bool apart = react && l >= 5 && !P->ad;
    A.rlist = react && !apart;
    if (A.vlist || A.rlist) A.list = list;
    ++P->launches;
    HFMM_TRY(s6_run<D>(A, st));
    if (apart) {
        A.list = list;
        A.shift.dig = nullptr;
        A.vlist = 0;
        A.rlist = 1;
        A.rows = 2;
        A.accumulate = 1;
        ++P->launches;
        HFMM_TRY(s6_run<D>(A, st));
    }
    return HFMM_OK;
}

template <int D>
hfmm_status s6_slice(hfmm_plan_s* P, int l, bool loc, int nrhs, cudaStream_t st) {
    LevelInfo& lv = P->lev[l];
    const S6Lev& s = s6_lev<D>(lv);
    const int64_t total = lv.nbox * ((2 * lv.ncoef + 15) / 16 * 8);
    HFMM_CUDA_TRY(pdl_launch(s6_slice_kernel<D>,
                             dim3((unsigned)std::min<int64_t>((total + 127) / 128, 16 * 152), (unsigned)nrhs), dim3(128), 0,
                             st, 0, s6_expansion<D>(lv, loc), lv.nbox, nrhs, lv.p, s.sx, loc ? 1 : -1,
                             split_exp(P, D == 6 ? 0 : 1, l, loc), loc ? s.dloc : s.dmult));
    ++P->launches;
    return HFMM_OK;
}

}  // namespace

// w = 0: the FP64 expansions, 1: the mixed path's FP32 expansions.
// Operator slices of every level (plan time, or a mixed plan's first gradient).
// A plan whose slices or digits would pass the byte budget or the device's memory keeps the SIMT kernels.
hfmm_status build_split(hfmm_plan_s* P, int w, cudaStream_t st) {
    return plan_optional(P, [&] { return w ? s6_build<3>(P, st) : s6_build<6>(P, st); }, [&] { split_forget(P, w); });
}

// The plan's memory of its slices is gone.
void split_forget(hfmm_plan_s* P, int w) {
    P->s6_ready[w] = false;
    P->s6_E[w] = nullptr;
    for (LevelInfo& lv : P->lev) lv.s6[w] = S6Lev{};
}

// Start of a tree pass: no exponent is known.
hfmm_status split_begin(hfmm_plan_s* P, int w, cudaStream_t st) {
    HFMM_CUDA_TRY(cudaMemsetAsync(P->s6_E[w], 0x80, sizeof(int) * 2 * (P->L + 1) * P->max_rhs, st));
    return HFMM_OK;
}

int* split_exp(hfmm_plan_s* P, int w, int l, bool loc) {
    return P->s6_E[w] + ((size_t)(loc ? P->L + 1 : 0) + l) * P->max_rhs;
}

// Exponents of a level's FP64 expansions that another kernel wrote (uniform trees).
hfmm_status split_exponent(hfmm_plan_s* P, int l, bool loc, int nrhs, cudaStream_t st) {
    LevelInfo& lv = P->lev[l];
    const int64_t total = lv.nbox * lv.ncoef;
    HFMM_CUDA_TRY(pdl_launch(s6_exponent_kernel, dim3((unsigned)std::min<int64_t>((total + 255) / 256, 8 * 152), nrhs),
                             dim3(256), 0, st, 0, s6_expansion<6>(lv, loc), lv.nbox, nrhs, lv.p, P->leaf_begin, P->L, l,
                             lv.s6[0].sx, loc ? 1 : -1, split_exp(P, 0, l, loc)));
    ++P->launches;
    return HFMM_OK;
}

// Digits of a level's finished expansions, for the products that read them.
hfmm_status split_slice(hfmm_plan_s* P, int w, int l, bool loc, int nrhs, cudaStream_t st) {
    return w ? s6_slice<3>(P, l, loc, nrhs, st) : s6_slice<6>(P, l, loc, nrhs, st);
}

hfmm_status split_m2m(hfmm_plan_s* P, int w, int l, int nrhs, cudaStream_t st) {
    return w ? s6_m2m<3>(P, l, nrhs, st) : s6_m2m<6>(P, l, nrhs, st);
}

hfmm_status split_down(hfmm_plan_s* P, int w, int l, int nrhs, int parts, cudaStream_t st) {
    return w ? s6_down<3>(P, l, nrhs, parts, st) : s6_down<6>(P, l, nrhs, parts, st);
}
