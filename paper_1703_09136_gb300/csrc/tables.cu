// Plan-time translation tables, FP64 on the GPU (Algorithm 1, step 1:
// "precompute tables"; the paper used Mathematica, here quadrature kernels).
//
//  * free-space M2L:  C_n(D) = H_n(k|D|) e^{i n angle D}, n = -2p .. 2p, for the
//    49 offsets D = (dx, dy) h_l, |dx|, |dy| <= 3 (Graf, Sec. 3.3);
//  * M2M / L2L:       J_n(v) = J_n(k|v|) e^{i n angle v} for the four child
//    offsets v = +-(h_{l+1}/2, h_{l+1}/2);
//  * reaction M2L:    A_n(X, Y) of Eq. (eq:m2loperator) with sigma of the
//    medium (Sec. 5), n = -2p .. 2p, for every (dx, ysum) used by the
//    reaction lists, X = dx h_l, Y = 2 y0 + (ysum + 1) h_l;
//  * direct reaction: G^s(x_i - x_j, y_i + y_j) = (i/4) A_0 per point pair of
//    the leaf pairs whose images are not separated from the target leaf.
//
// Quadrature (written for this library): the propagating part is integrated
// over tau in [0, pi] with composite 16-point Gauss-Legendre panels; the
// evanescent part over t >= 0, where for layered media the path first dips
// below the real axis on [0, tb] (t = u - i c 4 u (tb - u) / tb^2) to pass
// the branch points of s2, s3 and the guided-mode poles on the radiating side,
// then follows the real axis to the point where the integrand envelope
// e^{-tY} ((xi + t)/k1)^nmax / xi has decayed by e^{-38}.
#include <algorithm>
#include <cmath>
#include <vector>

#include "bessel.cuh"
#include "hankel.cuh"
#include "plan.cuh"

namespace {

constexpr int GLN = 16;
// Largest accepted difference between a table and its node-doubled rule
// (weighted as in react_check_kernel).  Converged FP64 rules agree to a few
// 1e-14; the bound sits well above that and ten times below the FP64 path's
// 1e-11 parity bound.
constexpr double TABLE_RTOL = 1e-12;
__constant__ double c_glx[GLN];
__constant__ double c_glw[GLN];
double h_glx[GLN], h_glw[GLN];
bool gl_ready = false;

// Gauss-Legendre nodes on [-1, 1] by Newton's method on P_n.
void gauss_legendre(int n, double* x, double* w) {
    for (int i = 0; i < n; ++i) {
        double z = std::cos(HFMM_PI * (i + 0.75) / (n + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = 0.0;
            for (int j = 1; j <= n; ++j) {
                double p2 = p1;
                p1 = p0;
                p0 = ((2.0 * j - 1.0) * z * p1 - (j - 1.0) * p2) / j;
            }
            dp = n * (z * p0 - p1) / (z * z - 1.0);
            const double dz = p0 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        // derivative at the converged node
        double p0 = 1.0, p1 = 0.0;
        for (int j = 1; j <= n; ++j) {
            double p2 = p1;
            p1 = p0;
            p0 = ((2.0 * j - 1.0) * z * p1 - (j - 1.0) * p2) / j;
        }
        dp = n * (z * p0 - p1) / (z * z - 1.0);
        x[i] = -z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

hfmm_status ensure_gl() {
    if (!gl_ready) {
        gauss_legendre(GLN, h_glx, h_glw);
        gl_ready = true;
    }
    HFMM_CUDA_TRY(cudaMemcpyToSymbol(c_glx, h_glx, sizeof(h_glx)));
    HFMM_CUDA_TRY(cudaMemcpyToSymbol(c_glw, h_glw, sizeof(h_glw)));
    return HFMM_OK;
}

// quadrature segment: kind 0 tau (real panels on [a, b] in [0, pi]), 1 deformed
// t on [a, b] = [0, tb] with depth c, 2 real t on [a, b]
struct Seg {
    double a, b, c, tb;
    int kind, npan;
    int64_t node0;
};

struct Entry {
    double X, Y;
    int nmax;
    int seg0, seg1;
    int64_t nodes;
    int64_t out;      // offset of A_{-nmax} in the output
    int64_t wofs;     // offset of this level's weights w_n in the check's weight array
    int level, dx, ysum;
};

// real t >= 0 where sigma is not analytic (branch points of s_j, k_j > k1;
// guided-mode poles lie below the largest of them)
void singular_t(const hfmm_medium& m, std::vector<double>& out) {
    const double k1 = m.k[0];
    int nl = m.kind == HFMM_TWO_LAYER ? 1 : (m.kind == HFMM_THREE_LAYER ? 2 : 0);
    for (int j = 1; j <= nl; ++j) {
        double kj = m.k[j];
        if (kj > k1) out.push_back(std::sqrt(kj * kj - k1 * k1));
    }
}

void tau_kinks(const hfmm_medium& m, std::vector<double>& out) {
    const double k1 = m.k[0];
    int nl = m.kind == HFMM_TWO_LAYER ? 1 : (m.kind == HFMM_THREE_LAYER ? 2 : 0);
    for (int j = 1; j <= nl; ++j) {
        double kj = m.k[j];
        if (kj < k1) {
            out.push_back(std::acos(kj / k1));
            out.push_back(std::acos(-kj / k1));
        }
    }
}

double log_env(double t, double k1, double Y, int nmax) {
    double xi = std::sqrt(t * t + k1 * k1);
    return -t * Y + nmax * std::log((xi + t) / k1) - std::log(xi);
}

// end of the evanescent integral
double t_end(double k1, double Y, int nmax) {
    // peak of the envelope: derivative -Y + nmax / xi - t / xi^2 = 0
    double lo = 0.0, hi = std::max(1.0, (nmax + 1.0) / Y) * 4.0;
    auto d = [&](double t) {
        double xi = std::sqrt(t * t + k1 * k1);
        return -Y + nmax / xi - t / (xi * xi);
    };
    double tp = 0.0;
    if (d(0.0) > 0.0) {
        for (int it = 0; it < 200; ++it) {
            double mid = 0.5 * (lo + hi);
            if (d(mid) > 0.0) lo = mid; else hi = mid;
        }
        tp = 0.5 * (lo + hi);
    }
    const double target = log_env(tp, k1, Y, nmax) - 38.0;
    double a = tp, b = std::max(2.0 * tp, tp + 1.0);
    while (log_env(b, k1, Y, nmax) > target) b *= 2.0;
    for (int it = 0; it < 200; ++it) {
        double mid = 0.5 * (a + b);
        if (log_env(mid, k1, Y, nmax) > target) a = mid; else b = mid;
    }
    return b;
}

// Build the segments of one integral; returns the number of nodes.
// `scale` multiplies every panel count: 1 is the table's rule, 2 its
// node-doubled check, other values come from hfmm_options.quad_scale.
int64_t make_rule(const hfmm_medium& m, double xmax, double ymin, double ymax, int nmax,
                  std::vector<Seg>& segs, double scale) {
    const double k1 = m.k[0];
    const bool three = m.kind == HFMM_THREE_LAYER;
    const double dd = three ? m.d : 0.0;
    int64_t nodes = 0;
    auto push = [&](double a, double b, int kind, int npan, double c, double tb) {
        Seg s{a, b, c, tb, kind, std::max((int)std::ceil(npan * scale), 1), nodes};
        nodes += (int64_t)s.npan * GLN;
        segs.push_back(s);
    };
    // propagating part
    double rate = k1 * (std::fabs(xmax) + std::fabs(ymax)) + nmax + 1.0;
    if (three) rate += 2.0 * dd * std::max(m.k[1], k1);
    std::vector<double> brk{0.0};
    tau_kinks(m, brk);
    brk.push_back(HFMM_PI);
    std::sort(brk.begin(), brk.end());
    // impedance: sigma has a pole at s1 = i alpha, i.e. sin tau = -alpha / k1; for
    // 0 < alpha < k1 it lies on the real tau axis at -delta and pi + delta,
    // delta = asin(alpha / k1), so the panels near both ends are graded: no
    // panel is wider than 1.5 times its distance to the pole
    const bool imp_pole = m.kind == HFMM_IMPEDANCE && m.alpha > 0.0;
    const double delta = (imp_pole && m.alpha < k1) ? std::asin(m.alpha / k1) : -1.0;
    const double wu = 4.0 / rate;
    for (size_t i = 0; i + 1 < brk.size(); ++i) {
        const double A = brk[i], B = brk[i + 1];
        if (delta <= 0.0 || 1.5 * delta >= wu) {
            push(A, B, 0, (int)std::ceil((B - A) * rate / 4.0) + 1, 0.0, 0.0);
            continue;
        }
        const double M = 0.5 * (A + B);
        std::vector<std::pair<double, double>> right;
        for (double a = A; a < M;) {
            const double w = std::min(wu, 1.5 * (a + delta));
            const double b = w >= wu ? M : std::min(M, std::max(a + 8.0 * w, 2.0 * a + delta));
            push(a, b, 0, (int)std::ceil((b - a) / w), 0.0, 0.0);
            a = b;
        }
        for (double b = B; b > M;) {
            const double dist = HFMM_PI + delta - b;
            const double w = std::min(wu, 1.5 * dist);
            const double a = w >= wu ? M : std::max(M, std::min(b - 8.0 * w, b - dist));
            right.push_back({a, b});
            b = a;
        }
        for (auto it = right.rbegin(); it != right.rend(); ++it) {
            const double w = std::min(wu, 1.5 * (HFMM_PI + delta - it->second));
            push(it->first, it->second, 0, (int)std::ceil((it->second - it->first) / w), 0.0, 0.0);
        }
    }
    // evanescent part
    const double xa = std::max(std::fabs(xmax), 1e-12);
    double T = t_end(k1, ymin, nmax);
    std::vector<double> sing;
    singular_t(m, sing);
    double t0 = 0.0;
    if (!sing.empty()) {
        double ts = *std::max_element(sing.begin(), sing.end());
        double tb = 1.3 * ts + 0.1 * k1;
        double c = std::min(0.2 * tb, 0.8 / xa);
        double w = std::min({0.7 * c, 3.0 / std::max(ymax, 1e-12), 3.0 / xa});
        if (three && dd > 0) w = std::min(w, 1.5 / dd);
        push(0.0, tb, 1, (int)std::ceil(tb / w) + 2, c, tb);
        t0 = tb;
        T = std::max(T, tb + 1.0);
    }
    double wc = std::min(4.0 / std::max(ymin, 1e-300), 4.0 / xa);
    if (three && dd > 0) wc = std::min(wc, 2.0 / dd);
    const double wmin = wc / 16.0;
    double a = t0;
    while (a < T) {
        double wl = nmax > 0 ? 3.0 * a / nmax : wc;
        double w = std::min(wc, std::max(wmin, wl));
        // impedance pole at t = i alpha: panel width <= 1.5 x its distance
        if (imp_pole) w = std::min(w, 1.5 * std::sqrt(a * a + m.alpha * m.alpha));
        // branch points of 1/xi, xi = sqrt(t^2 + k1^2), at t = +-i k1 (close to
        // t = 0 at low frequency): the same grading
        w = std::min(w, 1.5 * std::sqrt(a * a + k1 * k1));
        double b = (w < wc) ? std::min(T, std::max(a + 16.0 * w, 2.0 * a)) : T;
        push(a, b, 2, (int)std::ceil((b - a) / w), 0.0, 0.0);
        a = b;
    }
    return nodes;
}

struct MedDev {
    int kind;
    double k1, k2sq, k3sq, d, alpha;
};

MedDev make_med(const hfmm_medium& m) {
    MedDev d;
    d.kind = m.kind;
    d.k1 = m.k[0];
    d.k2sq = m.k[1] * m.k[1];
    d.k3sq = m.k[2] * m.k[2];
    d.d = m.d;
    d.alpha = m.alpha;
    return d;
}

// s = -i sqrt(k^2 - lambda^2), principal root (Re s >= 0)
__device__ __forceinline__ cd s_branch(double kk, cd lam2) {
    cd r = csqrtz(cmk(kk - lam2.x, -lam2.y));
    return cmk(r.y, -r.x);
}

__device__ cd sigma_dev(const MedDev& m, cd lam2, cd s1) {
    if (m.kind == HFMM_IMPEDANCE) {
        return cdiv(cmk(s1.x, s1.y + m.alpha), cmk(s1.x, s1.y - m.alpha));
    }
    cd s2 = s_branch(m.k2sq, lam2);
    cd r12 = cdiv(csub(s1, s2), cadd(s1, s2));
    if (m.kind == HFMM_TWO_LAYER) return r12;
    cd s3 = s_branch(m.k3sq, lam2);
    cd r23 = cdiv(csub(s2, s3), cadd(s2, s3));
    cd e = cexpz(cscale(s2, -2.0 * m.d));
    cd re = cmul(r23, e);
    return cdiv(cadd(r12, re), cadd(cmk(1.0, 0.0), cmul(r12, re)));
}

// A node of a rule, without the pair's X and Y: tau (kind 0) carries its weight times
// sigma and sin, cos of tau; t (1 deformed, 2 real path) its weight times dt sigma / xi
// and t, xi (imaginary parts zero on the real path).
struct Node {
    int kind;
    cd c;
    double u;        // tau or the path parameter
    cd t, xi;        // kind 0: (sin tau, cos tau), unused
};

__device__ Node eval_node(const MedDev& m, const Seg* segs, int s0, int s1, int64_t nu) {
    int s = s0;
    while (s + 1 < s1 && segs[s + 1].node0 <= nu) ++s;
    const Seg sg = segs[s];
    const int64_t local = nu - sg.node0;
    const int pan = (int)(local / GLN), g = (int)(local % GLN);
    const double w = (sg.b - sg.a) / sg.npan;
    const double u = sg.a + (pan + 0.5 + 0.5 * c_glx[g]) * w;
    const double wu = 0.5 * w * c_glw[g];
    Node nd;
    nd.kind = sg.kind;
    nd.u = u;
    const double k1 = m.k1;
    if (sg.kind == 0) {
        double st, ct;
        sincos(u, &st, &ct);
        nd.t = cmk(st, ct);
        nd.xi = cmk(0.0, 0.0);
        nd.c = cscale(sigma_dev(m, cmk(k1 * k1 * ct * ct, 0.0), cmk(0.0, -k1 * st)), wu);
        return nd;
    }
    cd t = cmk(u, 0.0), dt = cmk(1.0, 0.0);
    if (sg.kind == 1) {
        const double tb = sg.tb;
        t.y = -sg.c * 4.0 * u * (tb - u) / (tb * tb);
        dt.y = -sg.c * 4.0 * (tb - 2.0 * u) / (tb * tb);
    }
    const cd lam2 = cadd(cmul(t, t), cmk(k1 * k1, 0.0));
    nd.t = t;
    nd.xi = csqrtz(lam2);
    nd.c = cdiv(cmul(cscale(dt, wu), sigma_dev(m, lam2, t)), nd.xi);
    return nd;
}

constexpr int CH = 8;                // orders n (and -n) per pass over a tile's nodes
constexpr int RT_THREADS = 128;
constexpr int RT_NODES = 512;        // nodes of a tile
constexpr int RT_NV = 10;            // doubles of a node in shared memory

// sums of v[0 .. 31] over the warp, value l in lane l (31 additions instead of 160)
__device__ __forceinline__ double warp_scatter32(double (&v)[32]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const bool up = lane & o;
            const double keep = up ? v[i + o] : v[i], give = up ? v[i] : v[i + o];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    return v[0];
}

// Sums over the nodes of one entry, for n = 0 .. nmax and both signs of the order:
//   tau nodes  C_n = sum c e^{i k1 (Y sin - X cos)} cos n tau, S_n = ... sin n tau
//              (order +-n: C_n -+ i S_n);
//   t nodes    T_n = sum e^{lp + n lz} + (-1)^n e^{lm - n lz},  T_{-n} likewise with -lz,
//              lp, lm = log c - t Y +- i xi X, lz = log(k1 / (xi + t)); on the real path lz
//              and the common real part of lp, lm are real, so P = e^{lr + n lz} and
//              Q = e^{lr - n lz} are real and multiply two constant phases.
// A tile's nodes (square roots, sigma, logarithms, the factors and phases that no order changes) are
// evaluated once into shared memory; each pass of eight orders serves both signs.  The t nodes'
// recurrences start every pass from exponentials (their range is that of the whole sum, not
// of one order).  The tau nodes' phases e^{i n tau} go on from pass to pass by e^{8 i tau},
// which errs less than the cosine of the rounded product n tau.  FP64 bound (1.0 TFLOP/s):
// nodes once per eight orders and complex recurrences for both signs, three layers, 1M points
// 612 ms per rule, impedance, 4099 points 16.2 ms; nodes once, 177 and 1.6 ms; factors and
// phases once too, 110 and 0.86 ms.
// blockIdx.y splits the tiles; chunks of eight orders c0 .. c0 + nwin; sums[entry][y][2][chunk][32] =
// (C, S | T_n, T_-n) x re, im.
__global__ void __launch_bounds__(RT_THREADS) react_sum_kernel(MedDev m, const Entry* __restrict__ ents,
                                                               const Seg* __restrict__ segs, int c0, int nwin,
                                                               double* __restrict__ sums) {
    extern __shared__ double rt_smem[];
    const Entry e = ents[blockIdx.x];
    const int nch = min((e.nmax + CH) / CH - c0, nwin);   // chunks of this launch's window, n = 0 .. nmax
    if (nch <= 0) return;
    double* nodes = rt_smem;                               // [RT_NV][RT_NODES]
    double* acc = nodes + RT_NV * RT_NODES;                  // [2][nch][32]
    double* red = acc + 2 * nch * 32;                      // [warps][32]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < 2 * nch * 32; i += RT_THREADS) acc[i] = 0.0;
    // tau nodes come first; the other group starts at the first t segment
    int64_t ntau = e.nodes;
    for (int s = e.seg0; s < e.seg1; ++s)
        if (segs[s].kind != 0) { ntau = segs[s].node0; break; }
    const double lk = log(m.k1);
    for (int grp = 0; grp < 2; ++grp) {
        const int64_t g0 = grp ? ntau : 0, g1 = grp ? e.nodes : ntau;
        for (int64_t t0 = g0 + (int64_t)blockIdx.y * RT_NODES; t0 < g1; t0 += (int64_t)gridDim.y * RT_NODES) {
            const int cnt = (int)(g1 - t0 < RT_NODES ? g1 - t0 : RT_NODES);
            __syncthreads();
            for (int i = tid; i < cnt; i += RT_THREADS) {
                const Node nd = eval_node(m, segs, e.seg0, e.seg1, t0 + i);
                double* o = nodes + i;
                if (grp == 0) {
                    // c e^{i k1 (...)}, e^{i tau}, e^{8 i tau}, e^{i n tau} of the next order
                    const cd b = cmul(nd.c, cexpi(m.k1 * (e.Y * nd.t.x - e.X * nd.t.y)));
                    const cd first = cexpi((double)(c0 * CH) * nd.u), step = cexpi(CH * nd.u);
                    o[0] = b.x; o[RT_NODES] = b.y;
                    o[2 * RT_NODES] = nd.t.y; o[3 * RT_NODES] = nd.t.x;
                    o[4 * RT_NODES] = step.x; o[5 * RT_NODES] = step.y;
                    o[6 * RT_NODES] = first.x; o[7 * RT_NODES] = first.y;
                } else {
                    const cd lc = csub(clogz(nd.c), cscale(nd.t, e.Y)), ix = cmuli(cscale(nd.xi, e.X));
                    const cd lx = clogz(cadd(nd.xi, nd.t));
                    const cd lp = cadd(lc, ix), lm = csub(lc, ix);
                    const cd lz = cmk(lk - lx.x, -lx.y);
                    cd f, g;
                    if (lz.y == 0.0 && lp.x == lm.x) {     // real path: z, 1 / z for the imaginary parts' places
                        o[RT_NODES] = exp(lz.x); o[3 * RT_NODES] = exp(-lz.x);
                        f = cexpi(lp.y); g = cexpi(lm.y);
                    } else {
                        o[RT_NODES] = lp.y; o[3 * RT_NODES] = lm.y;
                        f = cexpz(lz); g = cexpz(cneg(lz));
                    }
                    o[0] = lp.x; o[2 * RT_NODES] = lm.x;
                    o[4 * RT_NODES] = lz.x; o[5 * RT_NODES] = lz.y;
                    o[6 * RT_NODES] = f.x; o[7 * RT_NODES] = f.y;
                    o[8 * RT_NODES] = g.x; o[9 * RT_NODES] = g.y;
                }
            }
            __syncthreads();
            for (int c = 0; c < nch; ++c) {
                double v[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = 0.0;
                const double n0 = (c0 + c) * CH;
                for (int i = tid; i < cnt; i += RT_THREADS) {
                    double* o = nodes + i;                 // this thread's node in every pass
                    if (grp == 0) {
                        const double br = o[0], bi = o[RT_NODES], c1 = o[2 * RT_NODES], s1 = o[3 * RT_NODES];
                        double cn = o[6 * RT_NODES], sn = o[7 * RT_NODES];
                        const cd next = cmul(cmk(cn, sn), cmk(o[4 * RT_NODES], o[5 * RT_NODES]));
                        o[6 * RT_NODES] = next.x; o[7 * RT_NODES] = next.y;
#pragma unroll
                        for (int j = 0; j < CH; ++j) {
                            v[4 * j] = fma(br, cn, v[4 * j]);
                            v[4 * j + 1] = fma(bi, cn, v[4 * j + 1]);
                            v[4 * j + 2] = fma(br, sn, v[4 * j + 2]);
                            v[4 * j + 3] = fma(bi, sn, v[4 * j + 3]);
                            const double x = cn * c1 - sn * s1;
                            sn = sn * c1 + cn * s1;
                            cn = x;
                        }
                    } else if (o[5 * RT_NODES] == 0.0 && o[0] == o[2 * RT_NODES]) {   // real path
                        const double lr = o[0], lz = o[4 * RT_NODES], z = o[RT_NODES], zi = o[3 * RT_NODES];
                        const double pr = o[6 * RT_NODES], pi = o[7 * RT_NODES], mr = o[8 * RT_NODES], mi = o[9 * RT_NODES];
                        double P = exp(lr + n0 * lz), Q = exp(lr - n0 * lz);
#pragma unroll
                        for (int j = 0; j < CH; ++j) {
                            const double sP = (j & 1) ? -P : P, sQ = (j & 1) ? -Q : Q;    // n0 is even
                            v[4 * j] = fma(P, pr, fma(sQ, mr, v[4 * j]));
                            v[4 * j + 1] = fma(P, pi, fma(sQ, mi, v[4 * j + 1]));
                            v[4 * j + 2] = fma(Q, pr, fma(sP, mr, v[4 * j + 2]));
                            v[4 * j + 3] = fma(Q, pi, fma(sP, mi, v[4 * j + 3]));
                            P *= z;
                            Q *= zi;
                        }
                    } else {
                        const cd lp = cmk(o[0], o[RT_NODES]), lm = cmk(o[2 * RT_NODES], o[3 * RT_NODES]);
                        const cd nz = cscale(cmk(o[4 * RT_NODES], o[5 * RT_NODES]), n0);
                        const cd z = cmk(o[6 * RT_NODES], o[7 * RT_NODES]), zi = cmk(o[8 * RT_NODES], o[9 * RT_NODES]);
                        cd pu = cexpz(cadd(lp, nz)), pd = cexpz(csub(lp, nz));     // e^{lp +- n lz}
                        cd mu = cexpz(cadd(lm, nz)), md = cexpz(csub(lm, nz));
#pragma unroll
                        for (int j = 0; j < CH; ++j) {
                            const double sg = (j & 1) ? -1.0 : 1.0;
                            v[4 * j] += pu.x + sg * md.x;
                            v[4 * j + 1] += pu.y + sg * md.y;
                            v[4 * j + 2] += pd.x + sg * mu.x;
                            v[4 * j + 3] += pd.y + sg * mu.y;
                            pu = cmul(pu, z); mu = cmul(mu, z);
                            pd = cmul(pd, zi); md = cmul(md, zi);
                        }
                    }
                }
                const double x = warp_scatter32(v);
                red[wid * 32 + lane] = x;
                __syncthreads();
                if (wid == 0) {
                    double a = acc[(grp * nch + c) * 32 + lane];
                    for (int w = 0; w < RT_THREADS / 32; ++w) a += red[w * 32 + lane];
                    acc[(grp * nch + c) * 32 + lane] = a;
                }
                __syncthreads();
            }
        }
    }
    __syncthreads();
    double* out = sums + ((int64_t)blockIdx.x * gridDim.y + blockIdx.y) * (2 * nwin * 32);
    for (int i = tid; i < 2 * nch * 32; i += RT_THREADS) out[i] = acc[i];
}

// A_{+-n} = i^n / pi tau-sum + (-i)^n / (i pi) t-sum from the splits' sums.
__global__ void react_finish_kernel(const Entry* __restrict__ ents, const double* __restrict__ sums, int ny, int c0,
                                    int nwin, cd* __restrict__ out) {
    const Entry e = ents[blockIdx.x];
    const int nch = min((e.nmax + CH) / CH - c0, nwin);
    for (int n = c0 * CH + threadIdx.x; n <= e.nmax && n < (c0 + nch) * CH; n += blockDim.x) {
        double a[4] = {0, 0, 0, 0}, b[4] = {0, 0, 0, 0};
        for (int y = 0; y < ny; ++y) {
            const double* s = sums + ((int64_t)blockIdx.x * ny + y) * (2 * nwin * 32) + (n / CH - c0) * 32 + 4 * (n % CH);
            for (int q = 0; q < 4; ++q) {
                a[q] += s[q];
                b[q] += s[(int64_t)nch * 32 + q];
            }
        }
        for (int sg = 0; sg < (n > 0 ? 2 : 1); ++sg) {
            // tau: C - i S for +n, C + i S for -n; t: T_n, T_-n
            const cd ta = sg ? cmk(a[0] - a[3], a[1] + a[2]) : cmk(a[0] + a[3], a[1] - a[2]);
            const cd tb = sg ? cmk(b[2], b[3]) : cmk(b[0], b[1]);
            const int r = (sg ? 4 - (n & 3) : n) & 3;
            const cd in = (r == 0) ? cmk(1, 0) : (r == 1) ? cmk(0, 1) : (r == 2) ? cmk(-1, 0) : cmk(0, -1);
            const cd v = cadd(cscale(cmul(in, ta), 1.0 / HFMM_PI),
                              cscale(cmul(cconj(in), cmk(tb.y, -tb.x)), 1.0 / HFMM_PI));  // b / i = -i b
            out[e.out + e.nmax + (sg ? -n : n)] = v;
        }
    }
}

// Direct reaction blocks: one CTA per block of point pairs (i in T, j in S).
struct DirectJob {
    int32_t t_lo, t_n, s_lo, s_n;
    int seg0, seg1;
    int64_t nodes;
    int64_t blk;
};

constexpr int DB_NODES = 16;         // nodes of a tile
constexpr int DB_POINTS = 32;        // targets and sources of a tile
constexpr int DB_THREADS = 128;
constexpr int DB_PAIRS = DB_POINTS * DB_POINTS / DB_THREADS;

// The integrand factorises: with x, y from the block's first target and zero,
//   tau  c e^{i k1 (Y sin - X cos)} = c U_i V_j,  U = e^{i k1 (y sin - x cos)}, V = e^{i k1 (y sin + x cos)}
//   t    c e^{-t Y +- i xi X}       = c U_i V_j,  U = e^{-t y +- i xi x},        V = e^{-t y -+ i xi x}
// so a tile of 16 nodes takes one exponential per (node, point) and one complex product
// per (node, pair), instead of a node evaluation and two exponentials per (node, pair).
// GRAD: the X and Y derivatives instead (factors -i k1 cos, i k1 sin; +- i xi, -t).
// blockIdx.y walks the tiles of 32 targets x 32 sources; 1600 points near the interface, both rules:
// 449 -> 18 ms (one GB300).
template <bool GRAD>
__global__ void __launch_bounds__(DB_THREADS) direct_sum_kernel(MedDev m, const DirectJob* __restrict__ jobs,
                                                                const Seg* __restrict__ segs,
                                                                const double2* __restrict__ xs, cd* __restrict__ out,
                                                                cd* __restrict__ outy) {
    __shared__ cd U[2][DB_NODES][DB_POINTS], V[2][DB_NODES][DB_POINTS];   // [+, -]
    __shared__ cd fx[DB_NODES], fy[DB_NODES];                             // GRAD: derivative factors (+; - has -fx)
    __shared__ int kind[DB_NODES];
    const DirectJob jb = jobs[blockIdx.x];
    const int64_t nts = (jb.s_n + DB_POINTS - 1) / DB_POINTS, ntt = (jb.t_n + DB_POINTS - 1) / DB_POINTS;
    const int tid = threadIdx.x;
    for (int64_t tile = blockIdx.y; tile < nts * ntt; tile += gridDim.y) {
    const int ti = (int)(tile / nts) * DB_POINTS, tj = (int)(tile % nts) * DB_POINTS;
    const double xc = xs[jb.t_lo].x;
    cd at[DB_PAIRS], ae[DB_PAIRS], bt[GRAD ? DB_PAIRS : 1], be[GRAD ? DB_PAIRS : 1];
#pragma unroll
    for (int q = 0; q < DB_PAIRS; ++q) {
        at[q] = ae[q] = cmk(0, 0);
        if (GRAD) bt[q] = be[q] = cmk(0, 0);
    }
    for (int64_t n0 = 0; n0 < jb.nodes; n0 += DB_NODES) {
        const int cnt = (int)(jb.nodes - n0 < DB_NODES ? jb.nodes - n0 : DB_NODES);
        __syncthreads();
        __shared__ Node nd[DB_NODES];
        if (tid < cnt) {
            nd[tid] = eval_node(m, segs, jb.seg0, jb.seg1, n0 + tid);
            kind[tid] = nd[tid].kind;
            if (GRAD) {
                fx[tid] = nd[tid].kind == 0 ? cmk(0.0, -m.k1 * nd[tid].t.y) : cmuli(nd[tid].xi);
                fy[tid] = nd[tid].kind == 0 ? cmk(0.0, m.k1 * nd[tid].t.x) : cneg(nd[tid].t);
            }
        }
        __syncthreads();
        for (int w = tid; w < cnt * 2 * DB_POINTS; w += DB_THREADS) {
            const int q = w / (2 * DB_POINTS), pt = w % (2 * DB_POINTS);
            const bool tgt = pt < DB_POINTS;
            const int i = tgt ? ti + pt : tj + pt - DB_POINTS;
            if (i >= (tgt ? jb.t_n : jb.s_n)) continue;
            const double2 p = xs[(tgt ? jb.t_lo : jb.s_lo) + i];
            const double x = tgt ? p.x - xc : xc - p.x;      // X = x_i + x_j with this sign
            const Node& d = nd[q];
            cd a, b = cmk(0, 0);
            if (d.kind == 0) a = cexpi(m.k1 * (p.y * d.t.x - x * d.t.y));
            else {
                const cd ty = cscale(d.t, -p.y), ix = cmuli(cscale(d.xi, x));
                a = cexpz(cadd(ty, ix));
                b = d.kind == 2 ? cconj(a) : cexpz(csub(ty, ix));
            }
            if (tgt) { U[0][q][pt] = a; U[1][q][pt] = b; }
            else { V[0][q][pt - DB_POINTS] = cmul(a, d.c); V[1][q][pt - DB_POINTS] = cmul(b, d.c); }
        }
        __syncthreads();
        for (int q = 0; q < cnt; ++q) {
            const int kd = kind[q];
#pragma unroll
            for (int u = 0; u < DB_PAIRS; ++u) {
                const int id = tid + u * DB_THREADS, i = id / DB_POINTS, j = id % DB_POINTS;
                if (ti + i >= jb.t_n || tj + j >= jb.s_n) continue;
                if (kd == 0) {
                    if (GRAD) {
                        const cd vp = cmul(U[0][q][i], V[0][q][j]);
                        cfma(at[u], vp, fx[q]);
                        cfma(bt[u], vp, fy[q]);
                    } else cfma(at[u], U[0][q][i], V[0][q][j]);
                } else if (GRAD) {
                    const cd vp = cmul(U[0][q][i], V[0][q][j]), vm = cmul(U[1][q][i], V[1][q][j]);
                    cfma(ae[u], csub(vp, vm), fx[q]);
                    cfma(be[u], cadd(vp, vm), fy[q]);
                } else {
                    cfma(ae[u], U[0][q][i], V[0][q][j]);
                    cfma(ae[u], U[1][q][i], V[1][q][j]);
                }
            }
        }
    }
    // A_0 = tau-sum / pi + t-sum / (i pi);  G^s and its derivatives = (i/4) A
#pragma unroll
    for (int u = 0; u < DB_PAIRS; ++u) {
        const int id = tid + u * DB_THREADS, i = ti + id / DB_POINTS, j = tj + id % DB_POINTS;
        if (i >= jb.t_n || j >= jb.s_n) continue;
        const int64_t o = jb.blk + (int64_t)i * jb.s_n + j;
        out[o] = cmuli(cscale(cadd(at[u], cmk(ae[u].y, -ae[u].x)), 0.25 / HFMM_PI));
        if (GRAD) outy[o] = cmuli(cscale(cadd(bt[u], cmk(be[u].y, -be[u].x)), 0.25 / HFMM_PI));
    }
    }
}

// Node-doubling check of the tables.  The reaction entry A_n feeds the
// translation entries s(|m|) s(|p|) A_n (m + p = -n) that act on the
// normalised expansions (|J_m(k rho)| <= s(|m|) inside a box); its weight w_n
// is the largest such product, so a difference that no translated field can
// see (the tiny coefficients the expansions never reach) does not count.
// One CTA per entry: max_n w_n |A_n - A2_n| / max_n w_n |A2_n|.
__device__ double block_max(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

__global__ void react_check_kernel(const Entry* ents, const cd* a1, const cd* a2, const double* w,
                                   double* ratio) {
    __shared__ double red[32];
    const Entry e = ents[blockIdx.x];
    double dm = 0.0, am = 0.0;
    for (int i = threadIdx.x; i < 2 * e.nmax + 1; i += blockDim.x) {
        const cd x = a1[e.out + i], y = a2[e.out + i];
        const double wi = w[e.wofs + i];
        dm = fmax(dm, wi * hypot(x.x - y.x, x.y - y.y));
        am = fmax(am, wi * hypot(y.x, y.y));
    }
    dm = block_max(dm, red);
    am = block_max(am, red);
    if (threadIdx.x == 0) ratio[blockIdx.x] = am > 0.0 ? dm / am : (dm > 0.0 ? INFINITY : 0.0);
}

// Directly summed blocks: max |G - G2| / max |G2| over the block's point pairs.
__global__ void direct_check_kernel(const DirectJob* jobs, const cd* v1, const cd* v2, double* ratio) {
    __shared__ double red[32];
    const DirectJob jb = jobs[blockIdx.x];
    double dm = 0.0, am = 0.0;
    for (int64_t i = threadIdx.x; i < (int64_t)jb.t_n * jb.s_n; i += blockDim.x) {
        const cd x = v1[jb.blk + i], y = v2[jb.blk + i];
        dm = fmax(dm, hypot(x.x - y.x, x.y - y.y));
        am = fmax(am, hypot(y.x, y.y));
    }
    dm = block_max(dm, red);
    am = block_max(am, red);
    if (threadIdx.x == 0) ratio[blockIdx.x] = am > 0.0 ? dm / am : (dm > 0.0 ? INFINITY : 0.0);
}

// Mirrored reaction entries: out[dst + nmax + n] = out[src + nmax - n].
struct int64_t3 {
    int64_t dst, src, nmax;
};

__global__ void mirror_kernel(const int64_t3* mir, cd* out) {
    const int64_t3 m = mir[blockIdx.x];
    for (int64_t i = threadIdx.x; i <= 2 * m.nmax; i += blockDim.x) out[m.dst + i] = out[m.src + 2 * m.nmax - i];
}

// free-space M2L: a CTA per offset of one level.  One thread carries the recurrences in n, whose
// quotients and phases the others make: a lone thread's FP64 instructions take 64 clocks each (4,099 points,
// levels 2 .. 4: 494 us with a thread per offset for everything -> 126 us).
__global__ void __launch_bounds__(64) free_table_kernel(double k, double h, int p, cd* out) {
    const int o = blockIdx.x;
    const int dx = o / 7 - 3, dy = o % 7 - 3;
    const int w = 4 * p + 1;
    cd* T = out + (int64_t)o * w;
    if (abs(dx) < 2 && abs(dy) < 2) {
        for (int i = threadIdx.x; i < w; i += 64) T[i] = cmk(0, 0);
        return;
    }
    const double X = dx * h, Y = dy * h;
    const double r = hypot(X, Y), th = atan2(Y, X);
    const double x = k * r;
    for (int n = 1 + threadIdx.x; n <= 2 * p; n += 64) T[2 * p - n].x = 2.0 * n / x;   // until the phases
    __syncthreads();
    if (threadIdx.x == 0) {
        cd hm, hn;
        hankel_recurrence<true>(x, &hm, &hn);
        T[2 * p] = hm;
#pragma unroll 4
        for (int n = 1; n <= 2 * p; ++n) {
            T[2 * p + n] = hn;
            const cd hx = csub(cscale(hn, T[2 * p - n].x), hm);
            hm = hn;
            hn = hx;
        }
    }
    __syncthreads();
    for (int n = 1 + threadIdx.x; n <= 2 * p; n += 64) {
        const cd ph = cexpi(n * th), hn = T[2 * p + n];
        const double sg = (n & 1) ? -1.0 : 1.0;
        T[2 * p + n] = cmul(hn, ph);
        T[2 * p - n] = cscale(cmul(hn, cconj(ph)), sg);
    }
}

// M2M (P - c) and L2L (c - P) tables of parent level l: a CTA per child, one thread for the
// Bessel sequence (276 -> 121 us for the levels above)
__global__ void __launch_bounds__(64) shift_table_kernel(double k, double hc, int nmax, double* scratch, cd* m2m,
                                                         cd* l2l) {
    const int c = blockIdx.x;
    const int w = 2 * nmax + 1;
    const double vx = (0.5 - (c & 1)) * hc, vy = (0.5 - (c >> 1)) * hc;   // P - c
    const double r = hypot(vx, vy), th = atan2(vy, vx);
    double* J = scratch + (int64_t)c * (nmax + 1);
    if (threadIdx.x == 0) bessel_j_seq(k * r, nmax, J);
    __syncthreads();
    for (int n = threadIdx.x; n <= nmax; n += 64) {
        cd ph = cexpi(n * th);
        double sg = (n & 1) ? -1.0 : 1.0;
        cd vp = cscale(ph, J[n]);                  // J_n(v) e^{i n th}
        cd vn = cscale(cconj(ph), sg * J[n]);      // J_{-n} e^{-i n th}
        m2m[(int64_t)c * w + nmax + n] = vp;
        m2m[(int64_t)c * w + nmax - n] = vn;
        // c - P = -v: J_n(-v) = (-1)^n J_n(v)
        l2l[(int64_t)c * w + nmax + n] = cscale(vp, sg);
        l2l[(int64_t)c * w + nmax - n] = cscale(vn, sg);
    }
}

// A_n of every entry on its rule into out: the node sums split over enough CTAs per
// entry to fill the GPU, then the coefficients.
hfmm_status react_tables(const MedDev& md, const std::vector<Entry>& ents, const Entry* dents,
                         const Seg* dsegs, cd* out, cudaStream_t st) {
    int nmax = 0;
    int64_t most = 0;
    for (const Entry& e : ents) {
        nmax = std::max(nmax, e.nmax);
        most = std::max(most, e.nodes);
    }
    const int nch = (nmax + CH) / CH, nwin = std::min(nch, 128);   // chunks per launch: 64 KB of sums
    const size_t sm = sizeof(double) * (RT_NV * RT_NODES + 2 * (size_t)nwin * 32 + RT_THREADS);
    HFMM_CUDA_TRY(smem_limit(react_sum_kernel, sm));
    int ny = (int)std::max<int64_t>(1, std::min<int64_t>((most + RT_NODES - 1) / RT_NODES,
                                                         (8 * 152 + (int64_t)ents.size() - 1) / (int64_t)ents.size()));
    // the splits' sums, from the pool; where its granularity (32 MB) does not fit, one split's alone
    double* sums = nullptr;
    const size_t one = sizeof(double) * 2 * nwin * 32 * ents.size();
    const bool pooled = cudaMallocAsync((void**)&sums, one * ny, st) == cudaSuccess;
    if (!pooled) {
        cudaGetLastError();
        ny = 1;
        HFMM_CUDA_TRY(cudaMalloc((void**)&sums, one));
    }
    for (int c0 = 0; c0 < nch; c0 += nwin) {
        react_sum_kernel<<<dim3((unsigned)ents.size(), (unsigned)ny), RT_THREADS, sm, st>>>(md, dents, dsegs, c0, nwin, sums);
        react_finish_kernel<<<(unsigned)ents.size(), 128, 0, st>>>(dents, sums, ny, c0, nwin, out);
    }
    const cudaError_t err = cudaGetLastError();
    if (pooled) cudaFreeAsync(sums, st);
    else cudaFree(sums);
    HFMM_CUDA_TRY(err);
    return HFMM_OK;
}

}  // namespace

// G^s blocks of directly summed point-range pairs (target range x source
// range, row-major in the target) by quadrature on the panel rule for the
// pair's largest |X| and its range of Y, each block checked against the
// node-doubled rule (table_check).  Sets d_vals, nd_vals and the job list;
// blk[i] = offset of pair i's block.
hfmm_status build_direct_blocks(hfmm_plan_s* P, const std::vector<DirectSpec>& specs, std::vector<int64_t>& blk,
                                cudaStream_t st) {
    HFMM_TRY(ensure_gl());
    const MedDev md = make_med(P->med);
    const double qs = P->quad_scale;
    std::vector<Seg> dsg, dsg2;
    std::vector<DirectJob> jobs, jobs2;
    blk.assign(specs.size(), 0);
    int64_t off = 0;
    int64_t maxtiles = 0;
    for (size_t i = 0; i < specs.size(); ++i) {
        const DirectSpec& sp = specs[i];
        DirectJob jb;
        jb.t_lo = sp.t_lo; jb.t_n = sp.t_n;
        jb.s_lo = sp.s_lo; jb.s_n = sp.s_n;
        jb.blk = off;
        DirectJob jb2 = jb;
        jb.seg0 = (int)dsg.size();
        std::vector<Seg> tmp;
        jb.nodes = make_rule(P->med, sp.xmax, sp.ymin, sp.ymax, 0, tmp, qs);
        for (auto& sgm : tmp) dsg.push_back(sgm);
        jb.seg1 = (int)dsg.size();
        tmp.clear();
        jb2.seg0 = (int)dsg2.size();
        jb2.nodes = make_rule(P->med, sp.xmax, sp.ymin, sp.ymax, 0, tmp, 2.0 * qs);
        for (auto& sgm : tmp) dsg2.push_back(sgm);
        jb2.seg1 = (int)dsg2.size();
        blk[i] = off;
        off += (int64_t)jb.t_n * jb.s_n;
        maxtiles = std::max<int64_t>(maxtiles, (int64_t)((jb.t_n + DB_POINTS - 1) / DB_POINTS) *
                                                   ((jb.s_n + DB_POINTS - 1) / DB_POINTS));
        jobs.push_back(jb);
        jobs2.push_back(jb2);
    }
    P->nd_vals = off;
    HFMM_TRY(plan_alloc(P, (void**)&P->d_vals, sizeof(cd) * std::max<int64_t>(off, 1)));
    if (jobs.empty()) return HFMM_OK;
    Seg* dsegs = nullptr;
    DirectJob* djobs = nullptr;
    HFMM_TRY(plan_alloc(P, (void**)&dsegs, sizeof(Seg) * std::max<size_t>(dsg.size(), 1)));
    HFMM_TRY(plan_alloc(P, (void**)&djobs, sizeof(DirectJob) * jobs.size()));
    if (!dsg.empty())
        HFMM_CUDA_TRY(cudaMemcpyAsync(dsegs, dsg.data(), sizeof(Seg) * dsg.size(), cudaMemcpyHostToDevice, st));
    HFMM_CUDA_TRY(cudaMemcpyAsync(djobs, jobs.data(), sizeof(DirectJob) * jobs.size(), cudaMemcpyHostToDevice, st));
    P->dj_tiles = (int)std::min<int64_t>(maxtiles, 1024);
    if (maxtiles > 0) {
        const dim3 grid((unsigned)jobs.size(), (unsigned)P->dj_tiles);
        direct_sum_kernel<false><<<grid, DB_THREADS, 0, st>>>(md, djobs, dsegs, P->xy_sorted, P->d_vals, nullptr);
        HFMM_CUDA_TRY(cudaGetLastError());
        // node-doubled blocks for the check
        cd* vals2 = nullptr;
        Seg* dsegs2 = nullptr;
        DirectJob* djobs2 = nullptr;
        double* dratio = nullptr;
        HFMM_TRY(plan_alloc(P, (void**)&vals2, sizeof(cd) * off));
        HFMM_TRY(plan_alloc(P, (void**)&dsegs2, sizeof(Seg) * std::max<size_t>(dsg2.size(), 1)));
        HFMM_TRY(plan_alloc(P, (void**)&djobs2, sizeof(DirectJob) * jobs2.size()));
        HFMM_TRY(plan_alloc(P, (void**)&dratio, sizeof(double) * jobs.size()));
        if (!dsg2.empty())
            HFMM_CUDA_TRY(cudaMemcpyAsync(dsegs2, dsg2.data(), sizeof(Seg) * dsg2.size(), cudaMemcpyHostToDevice, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(djobs2, jobs2.data(), sizeof(DirectJob) * jobs2.size(), cudaMemcpyHostToDevice, st));
        direct_sum_kernel<false><<<grid, DB_THREADS, 0, st>>>(md, djobs2, dsegs2, P->xy_sorted, vals2, nullptr);
        direct_check_kernel<<<(unsigned)jobs.size(), 128, 0, st>>>(djobs, P->d_vals, vals2, dratio);
        HFMM_CUDA_TRY(cudaGetLastError());
        std::vector<double> ratio(jobs.size());
        HFMM_CUDA_TRY(cudaMemcpyAsync(ratio.data(), dratio, sizeof(double) * ratio.size(), cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        for (size_t i = 0; i < ratio.size(); ++i) {
            if (!(ratio[i] <= P->table_check)) {
                P->table_check = std::isnan(ratio[i]) ? INFINITY : ratio[i];
                P->table_check_where[0] = -1;      // a directly summed pair
                P->table_check_where[1] = (int)i;
                P->table_check_where[2] = 0;
            }
        }
    }
    P->dj_jobs = djobs;
    P->dj_segs = dsegs;
    P->dj_njobs = (int64_t)jobs.size();
    P->table_bytes += sizeof(cd) * (double)off;
    return HFMM_OK;
}

hfmm_status build_tables(hfmm_plan_s* P, cudaStream_t st) {
    HFMM_TRY(ensure_gl());
    const int L = P->L;
    const double k = P->k;
    const MedDev md = make_med(P->med);
    // free M2L and shift tables
    for (int l = 0; l <= L; ++l) {
        LevelInfo& lv = P->lev[l];
        if (l >= 2 && l >= P->lmin) {
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_free, sizeof(cd) * 49 * (4 * lv.p + 1)));
            free_table_kernel<<<49, 64, 0, st>>>(k, lv.h, lv.p, lv.t_free);
            HFMM_CUDA_TRY(cudaGetLastError());
            P->table_bytes += sizeof(cd) * 49.0 * (4 * lv.p + 1);
        }
        if (l < L && l >= P->lmin) {
            const int nmax = lv.p + P->lev[l + 1].p;
            const int w = 2 * nmax + 1;
            double* scratch = nullptr;
            HFMM_TRY(plan_alloc(P, (void**)&scratch, sizeof(double) * 4 * (nmax + 1)));
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_m2m, sizeof(cd) * 4 * w));
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_l2l, sizeof(cd) * 4 * w));
            shift_table_kernel<<<4, 64, 0, st>>>(k, P->lev[l + 1].h, nmax, scratch, lv.t_m2m, lv.t_l2l);
            HFMM_CUDA_TRY(cudaGetLastError());
            P->table_bytes += sizeof(cd) * 8.0 * w;
        }
    }
    // reaction tables (on the panel rule, and on the node-doubled rule for the check)
    const double qs = P->quad_scale;
    std::vector<Seg> segs, segs2;
    std::vector<Entry> ents, ents2;
    std::vector<int64_t3> mirrors;   // (destination, source, nmax) of mirrored entries
    std::vector<double> wts;
    int64_t total = 0;
    std::vector<int64_t> lev_off(L + 1, 0);
    for (int l = 0; l <= L; ++l) {
        LevelInfo& lv = P->lev[l];
        if (lv.nr == 0) continue;
        const int m = 1 << l;
        const int dxmax = l == 0 ? 0 : m - 1;
        lv.react_dx_max = dxmax;
        lv.n_react_entries = (2 * dxmax + 1) * 3;
        const int nmax = 2 * lv.p;
        lev_off[l] = total;
        // weights w_n = max over m + p = -n (|m|, |p| <= p_l) of s(|m|) s(|p|),
        // s(n) = min(1, (k R_l / 2)^n / n!)
        const int64_t wofs = (int64_t)wts.size();
        {
            const double kR = P->k * lv.h / std::sqrt(2.0);
            std::vector<double> ls(lv.p + 1);
            for (int j = 0; j <= lv.p; ++j)
                ls[j] = std::min(0.0, j * std::log(0.5 * kR) - std::lgamma(j + 1.0));
            for (int n = -nmax; n <= nmax; ++n) {
                double best = -1e300;
                for (int mm = -lv.p; mm <= lv.p; ++mm) {
                    const int pp = -n - mm;
                    if (pp < -lv.p || pp > lv.p) continue;
                    best = std::max(best, ls[std::abs(mm)] + ls[std::abs(pp)]);
                }
                wts.push_back(std::exp(std::max(best, -700.0)));
            }
        }
        for (int dx = -dxmax; dx <= dxmax; ++dx)
            for (int ys = 0; ys < 3; ++ys) {
                const int64_t idx = (int64_t)(dx + dxmax) * 3 + ys;
                bool used = (l == 0) ? (dx == 0 && ys == 0)
                                     : (ys <= 2 && reaction_admissible(ys, 0, P->y0, lv.h) && !(ys == 2 && m < 2));
                if (l == 0) used = used && P->lstar == 0;
                if (!used) continue;
                if (dx < 0) {
                    // sigma is even in lambda: A_n(-X, Y) = A_{-n}(X, Y), a copy of the dx > 0 entry
                    mirrors.push_back({total + idx * (2 * nmax + 1), total + ((int64_t)(-dx + dxmax) * 3 + ys) * (2 * nmax + 1),
                                       (int64_t)nmax});
                    continue;
                }
                Entry e;
                e.X = dx * lv.h;
                e.Y = 2.0 * P->y0 + (ys + 1) * lv.h;
                e.nmax = nmax;
                e.out = total + idx * (2 * nmax + 1);
                e.wofs = wofs;
                e.level = l;
                e.dx = dx;
                e.ysum = ys;
                Entry e2 = e;
                std::vector<Seg> tmp;
                e.seg0 = (int)segs.size();
                e.nodes = make_rule(P->med, e.X, e.Y, e.Y, nmax, tmp, qs);
                for (auto& sg : tmp) segs.push_back(sg);
                e.seg1 = (int)segs.size();
                ents.push_back(e);
                tmp.clear();
                e2.seg0 = (int)segs2.size();
                e2.nodes = make_rule(P->med, e2.X, e2.Y, e2.Y, nmax, tmp, 2.0 * qs);
                for (auto& sg : tmp) segs2.push_back(sg);
                e2.seg1 = (int)segs2.size();
                ents2.push_back(e2);
            }
        total += (int64_t)lv.n_react_entries * (2 * nmax + 1);
    }
    if (!ents.empty()) {
        cd* tab = nullptr;
        HFMM_TRY(plan_alloc(P, (void**)&tab, sizeof(cd) * total));
        HFMM_CUDA_TRY(cudaMemsetAsync(tab, 0, sizeof(cd) * total, st));
        for (int l = 0; l <= L; ++l)
            if (P->lev[l].nr > 0) P->lev[l].t_react = tab + lev_off[l];
        Seg* dsegs = nullptr;
        Entry* dents = nullptr;
        HFMM_TRY(plan_alloc(P, (void**)&dsegs, sizeof(Seg) * segs.size()));
        HFMM_TRY(plan_alloc(P, (void**)&dents, sizeof(Entry) * ents.size()));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dsegs, segs.data(), sizeof(Seg) * segs.size(), cudaMemcpyHostToDevice, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dents, ents.data(), sizeof(Entry) * ents.size(), cudaMemcpyHostToDevice, st));
        HFMM_TRY(react_tables(md, ents, dents, dsegs, tab, st));
        if (!mirrors.empty()) {
            int64_t3* dmir = nullptr;
            HFMM_TRY(plan_alloc(P, (void**)&dmir, sizeof(int64_t3) * mirrors.size()));
            HFMM_CUDA_TRY(cudaMemcpyAsync(dmir, mirrors.data(), sizeof(int64_t3) * mirrors.size(),
                                          cudaMemcpyHostToDevice, st));
            mirror_kernel<<<(unsigned)mirrors.size(), 128, 0, st>>>(dmir, tab);
            HFMM_CUDA_TRY(cudaGetLastError());
        }
        P->table_bytes += sizeof(cd) * (double)total;
        // the same entries on the node-doubled rule, compared entry by entry
        cd* tab2 = nullptr;
        Seg* dsegs2 = nullptr;
        Entry* dents2 = nullptr;
        double *dw = nullptr, *dratio = nullptr;
        HFMM_TRY(plan_alloc(P, (void**)&tab2, sizeof(cd) * total));
        HFMM_TRY(plan_alloc(P, (void**)&dsegs2, sizeof(Seg) * segs2.size()));
        HFMM_TRY(plan_alloc(P, (void**)&dents2, sizeof(Entry) * ents2.size()));
        HFMM_TRY(plan_alloc(P, (void**)&dw, sizeof(double) * wts.size()));
        HFMM_TRY(plan_alloc(P, (void**)&dratio, sizeof(double) * ents.size()));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dsegs2, segs2.data(), sizeof(Seg) * segs2.size(), cudaMemcpyHostToDevice, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dents2, ents2.data(), sizeof(Entry) * ents2.size(), cudaMemcpyHostToDevice, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dw, wts.data(), sizeof(double) * wts.size(), cudaMemcpyHostToDevice, st));
        HFMM_CUDA_TRY(cudaMemsetAsync(tab2, 0, sizeof(cd) * total, st));
        HFMM_TRY(react_tables(md, ents2, dents2, dsegs2, tab2, st));
        react_check_kernel<<<(unsigned)ents.size(), 128, 0, st>>>(dents, tab, tab2, dw, dratio);
        HFMM_CUDA_TRY(cudaGetLastError());
        std::vector<double> ratio(ents.size());
        HFMM_CUDA_TRY(cudaMemcpyAsync(ratio.data(), dratio, sizeof(double) * ratio.size(), cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        for (size_t i = 0; i < ratio.size(); ++i) {
            if (!(ratio[i] <= P->table_check)) {       // also catches NaN
                P->table_check = std::isnan(ratio[i]) ? INFINITY : ratio[i];
                P->table_check_where[0] = ents[i].level;
                P->table_check_where[1] = ents[i].dx;
                P->table_check_where[2] = ents[i].ysum;
            }
        }
    }
    // direct reaction blocks: leaf pairs of the bottom row (adaptive trees build theirs with their lists)
    if (P->nd > 0 && !P->ad) {
        const double h = P->lev[L].h;
        std::vector<int32_t> dbeg((size_t)P->lev[L].nbox + 1), dsrc(P->nd);
        HFMM_CUDA_TRY(cudaMemcpyAsync(dbeg.data(), P->d_begin, sizeof(int32_t) * dbeg.size(), cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaMemcpyAsync(dsrc.data(), P->d_src, sizeof(int32_t) * P->nd, cudaMemcpyDeviceToHost, st));
        HFMM_CUDA_TRY(cudaStreamSynchronize(st));
        const auto& lb = P->h_leaf_begin;
        std::vector<DirectSpec> specs;
        specs.reserve(P->nd);
        for (int64_t b = 0; b < P->lev[L].nbox; ++b)
            for (int32_t e = dbeg[b]; e < dbeg[b + 1]; ++e) {
                const int64_t s = dsrc[e];
                const int dx = (int)morton_x((uint32_t)b) - (int)morton_x((uint32_t)s);
                specs.push_back({lb[b], lb[b + 1] - lb[b], lb[s], lb[s + 1] - lb[s], (std::abs(dx) + 1) * h,
                                 2.0 * P->y0, 2.0 * P->y0 + 2.0 * h});
            }
        std::vector<int64_t> blk;
        HFMM_TRY(build_direct_blocks(P, specs, blk, st));
        HFMM_TRY(plan_alloc(P, (void**)&P->d_blk, sizeof(int64_t) * P->nd));
        HFMM_CUDA_TRY(cudaMemcpyAsync(P->d_blk, blk.data(), sizeof(int64_t) * P->nd, cudaMemcpyHostToDevice, st));
    }
    HFMM_CUDA_TRY(cudaStreamSynchronize(st));
    if (!(P->table_check <= TABLE_RTOL)) {
        if (P->table_check_where[0] >= 0)
            hfmm_set_error("reaction table quadrature not converged: level %d, dx %d, ysum %d differs from its "
                           "node-doubled rule by %.3g (bound %.1g)", P->table_check_where[0],
                           P->table_check_where[1], P->table_check_where[2], P->table_check, TABLE_RTOL);
        else
            hfmm_set_error("direct reaction quadrature not converged: leaf-pair block %d differs from its "
                           "node-doubled rule by %.3g (bound %.1g)", P->table_check_where[1], P->table_check,
                           TABLE_RTOL);
        return HFMM_ERR_NUMERICS;
    }
    return HFMM_OK;
}

// ---------------------------------------------------------------------------
// Mixed path: scaled FP32 translation matrices from the FP64 tables.
//   a~_n = a_n / s_l(|n|), b~_n = b_n s_l(|n|),  s_l(n) = min(1, (k R_l / 2)^n / n!)
// so that every stored matrix entry is O(1) or smaller (FP32 range).
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ cf to_cf(cd v) { return cfmk((float)v.x, (float)v.y); }

// Matrices are stored column-major (input coefficient outer, output inner),
// so that threads over output coefficients read consecutive entries.
// free-space M2L: F~[off][m][p] = s(p) s(m) C_{m-p}(off)
__global__ void free32_kernel(const cd* T, const double* ls, int p, cf* out) {
    const int nc = 2 * p + 1, w = 4 * p + 1;
    const int64_t total = (int64_t)49 * nc * nc;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int off = (int)(e / (nc * nc));
        const int r = (int)(e % (nc * nc));
        const int pp = r / nc - p, m = r % nc - p;
        const double sc = exp(ls[abs(pp)] + ls[abs(m)]);
        out[(int64_t)off * nc * nc + (int64_t)(m + p) * nc + (pp + p)] =
            to_cf(cscale(T[(int64_t)off * w + (m - pp) + 2 * p], sc));
    }
}

// reaction M2L on a (not a^im): H~[e][m][p] = s(p) s(m) (-1)^m A_{-m-p}
__global__ void react32_kernel(const cd* T, int nent, const double* ls, int p, cf* out) {
    const int nc = 2 * p + 1, w = 4 * p + 1;
    const int64_t total = (int64_t)nent * nc * nc;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int ent = (int)(e / (nc * nc));
        const int r = (int)(e % (nc * nc));
        const int pp = r / nc - p, m = r % nc - p;
        double sc = exp(ls[abs(pp)] + ls[abs(m)]);
        if (m & 1) sc = -sc;
        out[(int64_t)ent * nc * nc + (int64_t)(m + p) * nc + (pp + p)] =
            to_cf(cscale(T[(int64_t)ent * w + (-m - pp) + 2 * p], sc));
    }
}

// M2M child (level l+1, order pc) -> parent (level l, order pp):
//   T~[c][m][j] = J_{m-j}(P - c) s_{l+1}(m) / s_l(j)
// L2L parent -> child: L~[c][n][m] = J_{n-m}(c - P) s_{l+1}(m) / s_l(n)
__global__ void shift32_kernel(const cd* m2m, const cd* l2l, const double* lsp, const double* lsc,
                               int pp, int pc, cf* om2m, cf* ol2l) {
    const int np = 2 * pp + 1, nc = 2 * pc + 1, nmax = pp + pc, w = 2 * nmax + 1;
    const int64_t total = (int64_t)4 * np * nc;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(e / (np * nc));
        const int r = (int)(e % (np * nc));
        // M2M: row j (parent), column m (child)
        {
            const int j = r / nc - pp, m = r % nc - pc;
            const double sc = exp(lsc[abs(m)] - lsp[abs(j)]);
            om2m[(int64_t)c * np * nc + (int64_t)(m + pc) * np + (j + pp)] =
                to_cf(cscale(m2m[(int64_t)c * w + nmax + (m - j)], sc));
        }
        // L2L: row m (child), column n (parent)
        {
            const int m = r / np - pc, n = r % np - pp;
            const double sc = exp(lsc[abs(m)] - lsp[abs(n)]);
            ol2l[(int64_t)c * np * nc + (int64_t)(n + pp) * nc + (m + pc)] =
                to_cf(cscale(l2l[(int64_t)c * w + nmax + (n - m)], sc));
        }
    }
}

__global__ void vals32_kernel(const cd* v, int64_t n, cf* out) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = to_cf(v[e]);
}

}  // namespace

hfmm_status build_tables32(hfmm_plan_s* P, cudaStream_t st) {
    const int L = P->L;
    const int grid = 4 * 152, tb = 256;
    for (int l = P->lmin; l <= L; ++l) {
        LevelInfo& lv = P->lev[l];
        const double kR = P->k * lv.h / std::sqrt(2.0);
        lv.log_s.assign(lv.p + 1, 0.0);
        for (int n = 0; n <= lv.p; ++n) {
            double v = n * std::log(0.5 * kR) - std::lgamma(n + 1.0);
            lv.log_s[n] = std::max(-690.0, std::min(0.0, v));
        }
        HFMM_TRY(plan_alloc(P, (void**)&lv.d_log_s, sizeof(double) * (lv.p + 1)));
        HFMM_CUDA_TRY(cudaMemcpyAsync(lv.d_log_s, lv.log_s.data(), sizeof(double) * (lv.p + 1), cudaMemcpyHostToDevice, st));
    }
    for (int l = P->lmin; l <= L; ++l) {
        LevelInfo& lv = P->lev[l];
        const int nc = lv.ncoef;
        if (lv.t_free) {
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_free32, sizeof(cf) * 49 * nc * nc));
            free32_kernel<<<grid, tb, 0, st>>>(lv.t_free, lv.d_log_s, lv.p, lv.t_free32);
            HFMM_CUDA_TRY(cudaGetLastError());
            P->table_bytes += sizeof(cf) * 49.0 * nc * nc;
        }
        if (lv.t_react && lv.n_react_entries > 0) {
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_react32, sizeof(cf) * (size_t)lv.n_react_entries * nc * nc));
            react32_kernel<<<grid, tb, 0, st>>>(lv.t_react, lv.n_react_entries, lv.d_log_s, lv.p, lv.t_react32);
            HFMM_CUDA_TRY(cudaGetLastError());
            P->table_bytes += sizeof(cf) * (double)lv.n_react_entries * nc * nc;
        }
        if (l < L && lv.t_m2m) {
            const int ncc = P->lev[l + 1].ncoef;
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_m2m32, sizeof(cf) * 4 * nc * ncc));
            HFMM_TRY(plan_alloc(P, (void**)&lv.t_l2l32, sizeof(cf) * 4 * nc * ncc));
            shift32_kernel<<<grid, tb, 0, st>>>(lv.t_m2m, lv.t_l2l, lv.d_log_s, P->lev[l + 1].d_log_s, lv.p,
                                                P->lev[l + 1].p, lv.t_m2m32, lv.t_l2l32);
            HFMM_CUDA_TRY(cudaGetLastError());
            P->table_bytes += sizeof(cf) * 8.0 * nc * ncc;
        }
    }
    if (P->nd_vals > 0) {
        HFMM_TRY(plan_alloc(P, (void**)&P->d_vals32, sizeof(cf) * P->nd_vals));
        vals32_kernel<<<grid, tb, 0, st>>>(P->d_vals, P->nd_vals, P->d_vals32);
        HFMM_CUDA_TRY(cudaGetLastError());
    }
    HFMM_CUDA_TRY(cudaStreamSynchronize(st));
    return HFMM_OK;
}

// Gradient blocks of the directly summed reaction (built on the first
// position-gradient request).
hfmm_status build_direct_grad(hfmm_plan_s* P, cudaStream_t st) {
    if (P->nd == 0 || P->nd_vals == 0) return HFMM_OK;
    HFMM_TRY(ensure_gl());
    HFMM_TRY(plan_alloc(P, (void**)&P->d_gvals, sizeof(cd) * 2 * P->nd_vals));
    const MedDev md = make_med(P->med);
    direct_sum_kernel<true><<<dim3((unsigned)P->dj_njobs, (unsigned)P->dj_tiles), DB_THREADS, 0, st>>>(
        md, (const DirectJob*)P->dj_jobs, (const Seg*)P->dj_segs, P->xy_sorted, P->d_gvals, P->d_gvals + P->nd_vals);
    HFMM_CUDA_TRY(cudaGetLastError());
    return HFMM_OK;
}
