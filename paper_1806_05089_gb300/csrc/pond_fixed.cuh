// pond_fixed.cuh -- the FP64 staged step with its contractions in 64-bit
// fixed point on the integer multiply pipe.
//
// GB300 runs 2 FP64 FMAs per clock and SM but 32 integer multiply-adds with a
// 64-bit sum (mad.wide.s32; both measured).  The staged step
// (pond_staged.cuh) spends four fifths of its FP64 operations on dot products
// of 16 staged populations with 16 weights; here those run as
//   sum w g = 2^64 sum w1 g1 + 2^32 sum (w1 g0 + w0 g1) + sum w0 g0,
// with every operand v = 2^32 v1 + v0 split into a signed high word and a
// centred low word: three wide multiply-adds per product, exact 64-bit sums,
// and the last term (below 2^-58 of the operands' units, mean zero) dropped.
//
// Scales.  A tile's staged populations share one power of two: with M the
// largest population of the tile's centre node (each multiplied by
// 2^(s_k + s_l), s = 3 at the outer speeds of D2Q16, 2 at those of D2Q9, which
// brings W_q to one magnitude), R = 2^E >= 16 M, populations and sums are held
// to R 2^-60 and weights to 2^-60.  A row sum then carries about R 2^-59
// (2^-54 M or less), where the FP64 sum of 16 products rounds at 2^-53 of its
// terms: the fixed-point form is the more exact one as long as a tile's
// populations stay within its window of magnitudes.  So a group of 8 columns of a tile takes this
// path only if
//   - every staged |f| < R / 4 and |g| < R / 4, and at every staged node the
//     largest |g| is >= R / 128;
//   - the gauges of its nodes differ from the reference gauge by |xi_a - c_a|
//     <= 0.52, those of its sources by 1.2 (a node whose pass gauge goes beyond
//     0.58 is marked and computed again).  With S <= 4.4 the sum of the absolute
//     entries of a map's row at 0.58 and 1.25 that of the cubic weights, every
//     population stays below 0.4 S^2 R < 8 R and every middle sum below 2^63;
//   - its displacements are below 400 nodes.
// Any other group (strong shear at the window's scale, near-vacuum, NaN, the
// seed modes that start far from the reference) is put on a list, and
// k_step_staged<StagedFP64> runs the listed ones in a launch that follows.
//
// The staging, the maps' entries, the cubic weights and the closing re-gauge
// are in fixed point too: a product of two weights costs about ten
// integer instructions (a tenth of a clock and SM per node), an FP64 operation
// half a clock.  FP64 keeps what has no bounded range or needs a division or
// a root: gauge differences, displacements, conversions, the moments, the
// gauge update and its test, and BGK.
//
// Measured, GB300 (FP64: k_step_staged; contractions: only the dot products in
// fixed point; all: as here):
//                                  FP64  contractions      all
//   2048^2 supersonic, 1 step      69.8          36.8     22.1 ms
//   301 x 211, 4 steps              7.1           3.6      2.2 ms
//   1024^2 D2Q9, 2 steps           14.4           8.8      4.8 ms
//   64^2 Taylor-Green, 20 steps    14.0           7.3      1.7 ms
// It is bound by the integer multiplier: mad.wide runs at 32 a clock and SM
// (k_step_fixed at 2048^2: 62 % of the time in the row sweep, whose 192 of them
// per row alone take 192 of its 300 clocks).  Against a quadruple-precision
// step (three passes; populations, u_x, T on a smooth, a temperature-ratio-4
// and a shear field) the relative errors are 3.6-4.1e-16, 0.5-2.9e-16 and
// 3.1-3.4e-16 on D2Q16, where k_step_staged has 3.9-4.4e-16, 0.6-3.8e-16 and
// 3.4-3.6e-16.
#pragma once

#include "pond_staged.cuh"

namespace pond {

constexpr int kFix = 60;  // a weight of 1, or a population of R, is 2^60
constexpr float kFixTileDe = 0.52f, kFixNodeDe = 0.58f, kFixSourceDe = 1.2f;
constexpr double kFixOne = 1152921504606846976.0;         // 2^60
constexpr double kFixDisplacement = 18014398509481984.0;  // 2^54: |d| < 500 nodes

template <int N1>
__host__ __device__ constexpr int fix_shift(int k) {
    return (k == 0 || k == N1 - 1) ? (N1 == 4 ? 3 : 2) : 0;
}

struct Fix {
    int h, l;
};

// Lattice constants in fixed point (2^60): the speeds, and the Taylor
// coefficients of G[k][a] = L_k(c_a + de) times 2^(s_k - s_a), the factor between
// the scales of populations k and a.
struct LatticeFix {
    Fix c[4];
    long long d0[4][4], d1[4][4], d2[4][4];  // d0: the identity
    Fix d3[4][4];
};

// The split v = 2^32 h + l, l centred.
__host__ __device__ __forceinline__ Fix fix_split(long long v) {
    Fix f;
    f.l = (int)(unsigned)v;
    f.h = (int)((v + (1ll << 31)) >> 32);
    return f;
}

// (scaled = false: without those factors)
inline LatticeFix make_lattice_fix(const Lattice& L, bool scaled = true) {
    LatticeFix F{};
    auto fx = [](double v) { return (long long)std::llrint(v * kFixOne); };
    for (int k = 0; k < L.n1; ++k) {
        F.c[k] = fix_split(fx(L.c[k]));
        for (int a = 0; a < L.n1; ++a) {
            const int s = !scaled     ? 0
                          : L.n1 == 4 ? fix_shift<4>(k) - fix_shift<4>(a)
                                      : fix_shift<3>(k) - fix_shift<3>(a);
            F.d0[k][a] = k == a ? fx(1.0) : 0;
            F.d1[k][a] = fx(std::ldexp(L.d1[k][a], s));
            F.d2[k][a] = fx(std::ldexp(L.d2[k][a], s));
            F.d3[k][a] = fix_split(fx(std::ldexp(L.d3[k], s)));
        }
    }
    return F;
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// One product of a fixed-point dot product: h the 2^64 sum, m the 2^32 sum.
__device__ __forceinline__ void fix_mad(Fix w, int gh, int gl, long long& h, long long& m) {
    h = mad_wide(w.h, gh, h);
    m = mad_wide(w.h, gl, m);
    m = mad_wide(w.l, gh, m);
}

// The dot product h 2^64 + m 2^32 of weights and values, in the values' scale.
__device__ __forceinline__ long long fix_sum(long long h, long long m) {
    return (h << (64 - kFix)) + (m >> (kFix - 32));
}

// The same, rounded to nearest.
__device__ __forceinline__ long long fix_sum_rn(long long h, long long m) {
    return (h << (64 - kFix)) + ((m + (1ll << (kFix - 33))) >> (kFix - 32));
}

// Product of a weight and v, in v's scale.
__device__ __forceinline__ long long fix_mul(Fix w, Fix v) {
    long long h = 0, m = 0;
    fix_mad(w, v.h, v.l, h, m);
    return fix_sum(h, m);
}

// The 1D gauge map's entry for the offset de, in the scaled basis.
template <int N1>
__device__ __forceinline__ Fix fix_gauge(const LatticeFix& F, int k, int a, Fix de) {
    long long t = F.d2[k][a];
    if (N1 == 4) t += fix_mul(F.d3[k][a], de);
    t = F.d1[k][a] + fix_mul(de, fix_split(t));
    return fix_split(F.d0[k][a] + fix_mul(de, fix_split(t)));
}

// Floor of the displacement d 2^54 and the cubic weights at its
// fraction s.  With u = s (1 - s), v = u / 6, w = v s the weights of App. C at
// t = s + 1 are w - 2 v, 1 - s + 3 (v - w), s + 3 w, -(v + w); they sum to one
// exactly.
__device__ __forceinline__ int fix_departure(long long d, Fix (&l)[4]) {
    const long long s = (d & ((1ll << 54) - 1)) << (kFix - 54), one = 1ll << kFix;
    const Fix S = fix_split(s);
    const long long u = fix_mul(S, fix_split(one - s));
    const long long v = fix_mul(fix_split((one + 3) / 6), fix_split(u));
    const long long w = fix_mul(S, fix_split(v));
    l[0] = fix_split(w - 2 * v);
    l[1] = fix_split(one - s + 3 * (v - w));
    l[2] = fix_split(s + 3 * w);
    l[3] = fix_split(-(v + w));
    return (int)(d >> 54);
}

// fix_departure with the derivatives of the cubic weights by t, dl.
__device__ __forceinline__ int fix_departure_d(long long d, Fix (&l)[4], Fix (&dl)[4]) {
    const long long s = (d & ((1ll << 54) - 1)) << (kFix - 54), one = 1ll << kFix;
    const Fix S = fix_split(s), sixth = fix_split((one + 3) / 6);
    const Fix V = fix_split(fix_mul(sixth, fix_split(fix_mul(S, fix_split(one - s)))));
    const long long v = (long long)V.h * (1ll << 32) + V.l, w = fix_mul(S, V);
    l[0] = fix_split(w - 2 * v);
    l[1] = fix_split(one - s + 3 * (v - w));
    l[2] = fix_split(s + 3 * w);
    l[3] = fix_split(-(v + w));
    // v' = (1 - 2 s) / 6, w' = v' s + v
    const long long dv = fix_mul(sixth, fix_split(one - 2 * s)), dw = fix_mul(S, fix_split(dv)) + v;
    dl[0] = fix_split(dw - 2 * dv);
    dl[1] = fix_split(3 * (dv - dw) - one);
    dl[2] = fix_split(one + 3 * dw);
    dl[3] = fix_split(-(dv + dw));
    return (int)(d >> 54);
}

// The derivative of fix_gauge's entry by its offset.
template <int N1>
__device__ __forceinline__ long long fix_gauge_d(const LatticeFix& F, int k, int a, Fix de) {
    long long t = 2 * F.d2[k][a];
    if (N1 == 4) t += 3 * fix_mul(F.d3[k][a], de);
    return F.d1[k][a] + fix_mul(de, fix_split(t));
}

// A weight as a double.
__device__ __forceinline__ double fix_to_double(Fix w) {
    return (double)((long long)w.h * (1ll << 32) + w.l) * (1.0 / kFixOne);
}

// 2^e for |e| < 1000.
__device__ __forceinline__ double pow2d(int e) {
    return __hiloint2double((1023 + e) << 20, 0);
}

// x 2^e rounded to an integer; `big` is set when |x| 2^e >= 2^58 (R / 4; or x is not
// finite).  The exponent is added on the integer pipe.
__device__ __forceinline__ long long fix_population(double x, int e, bool& big) {
    const int hi = __double2hiint(x);
    const int ex = (hi >> 20 & 0x7ff) + e;
    big = big || ex >= 1023 + kFix - 2;
    const double y = __hiloint2double((hi & 0x800fffff) | ex << 20, __double2loint(x));
    return __double2ll_rn(ex > 0 && ex < 1023 + kFix - 2 ? y : 0.0);
}

// The largest |de_a| the gauge offsets r, dx, dy give (in units of 1).
__device__ __forceinline__ float fix_offset(long long r, long long dx, long long dy, float c_max) {
    const float u = 1.0f / (float)(1 << (kFix - 32));  // the high words' unit
    return u * fmaf(c_max, fabsf((float)(int)(r >> 32)),
                    fmaxf(fabsf((float)(int)(dx >> 32)), fabsf((float)(int)(dy >> 32))));
}

// Stage the window as stage_window does, the sources rounded to the tile's
// fixed point (2^e = 2^60 / R) and re-expressed there: high words in s_h, low
// words in s_l, row a at [a * WN + i].  Two planes, so that a quarter warp's
// 16-byte reads are contiguous.  Returns whether every value this thread
// staged is in range.
constexpr int kFixBadSource = (int)0x80000000;  // no staged high word is this

template <int N1, bool WIDE>
__device__ __forceinline__ bool stage_window_fixed(const StateBuf<double>& in, long long plane,
                                                   const GridDesc& G, long long base, int wx0,
                                                   int wy0, int ww, int wh, int WN, double rux,
                                                   double ruy, double rst, int scale_e, int4* s_h,
                                                   int4* s_l, const LatticeFix& F, float c_max,
                                                   DevStats* stats, int tid, int nt) {
    constexpr int Q = N1 * N1;
    const double inv_rst = kFixOne / rst;
    bool ok = true;
    (void)stats;
    const float inv_ww = 1.0f / (float)ww;
    for (int i = tid; i < ww * wh; i += nt) {
        const int cy = window_row(i, inv_ww), cx = i - cy * ww;
        const int gx = wrap_near(wx0 + cx, G.nx);
        const int gy = wrap_near(wy0 + cy, G.ny);
        const long long gi = base + (long long)gy * G.nx + gx;
        if (!POND_INDEX_OK(gx >= 0 && gx < G.nx && gy >= 0 && gy < G.ny && i < WN, stats))
            continue;
        const long long r = __double2ll_rn((__ldg(in.st + gi) - rst) * inv_rst);
        const long long dx = __double2ll_rn((__ldg(in.ux + gi) - rux) * inv_rst);
        const long long dy = __double2ll_rn((__ldg(in.uy + gi) - ruy) * inv_rst);
        bool big = !(fix_offset(r, dx, dy, c_max) <= kFixSourceDe);
        long long f[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q)
            f[q] = fix_population(__ldg(in.f + gi + (long long)q * plane),
                                  scale_e + fix_shift<N1>(q / N1) + fix_shift<N1>(q % N1), big);
        // g = G_x (x) G_y f, one y-speed l at a time: unrolled, with whole-row
        // stores, at 255 registers a thread (WIDE), else rolled
        Fix v[Q], gx_[N1][N1], dey[N1];
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = fix_split(f[q]);
        {
            const Fix R = fix_split(r);
            Fix dex[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const long long ca = fix_mul(F.c[a], R);
                dex[a] = fix_split(dx + ca);
                dey[a] = fix_split(dy + ca);
            }
#pragma unroll
            for (int k = 0; k < N1; ++k)
#pragma unroll
                for (int a = 0; a < N1; ++a) gx_[k][a] = fix_gauge<N1>(F, k, a, dex[a]);
        }
        int top = 0;
        int* dh = reinterpret_cast<int*>(s_h + i);
        int* dl = reinterpret_cast<int*>(s_l + i);
        Fix out[N1][4];
#pragma unroll(WIDE ? N1 : 1)
        for (int l = 0; l < N1; ++l) {
            Fix g[N1], H[N1];
#pragma unroll
            for (int b = 0; b < N1; ++b) g[b] = fix_gauge<N1>(F, l, b, dey[b]);
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                long long h = 0, m = 0;
#pragma unroll
                for (int b = 0; b < N1; ++b) fix_mad(g[b], v[N1 * a + b].h, v[N1 * a + b].l, h, m);
                H[a] = fix_split(fix_sum(h, m));
            }
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                long long h = 0, m = 0;
#pragma unroll
                for (int a = 0; a < N1; ++a) fix_mad(gx_[k][a], H[a].h, H[a].l, h, m);
                const Fix o = fix_split(fix_sum(h, m));
                top = max(top, abs(o.h));
                if constexpr (WIDE) {
                    out[k][l] = o;
                } else {
                    dh[(size_t)k * WN * 4 + l] = o.h;
                    dl[(size_t)k * WN * 4 + l] = o.l;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            if constexpr (WIDE) {
                if (N1 == 3) out[k][3] = Fix{0, 0};
                s_h[(size_t)k * WN + i] = make_int4(out[k][0].h, out[k][1].h, out[k][2].h, out[k][3].h);
                s_l[(size_t)k * WN + i] = make_int4(out[k][0].l, out[k][1].l, out[k][2].l, out[k][3].l);
            } else if (N1 == 3) {
                dh[(size_t)k * WN * 4 + 3] = dl[(size_t)k * WN * 4 + 3] = 0;
            }
        }
        // |g| < R / 4, and the node's largest >= R / 128; else the source is marked
        if (big || !(top < (1 << (kFix - 2 - 32)) && top >= (1 << (kFix - 7 - 32)))) {
            ok = false;
            s_h[i].x = kFixBadSource;
        }
    }
    return ok;
}

// The 8-column groups of a CTA's TXS columns whose own window -- the one a CTA of
// that group alone stages -- holds a source out of range (kFixBadSource in the
// staged window at wx0, wy0).  Every thread of the CTA calls it, with its node's
// velocity and largest thermal speed where `valid`; s_bad is zero on entry.
template <int TXS, int TYS, int NT>
__device__ __noinline__ unsigned fixed_bad_groups(const int4* s_h, int wx0, int wy0, int ww, int wh,
                                                  int tx0, int ty0, float m, float fdt, bool valid,
                                                  float ux, float uy, float sp, int n,
                                                  unsigned* s_bad) {
    constexpr int NG = TXS / 8;
    __shared__ int s_v[NG][4];  // xlo, xhi, ylo, yhi of a group's nodes, as ordered integers
    const int tid = threadIdx.x;
    auto key = [](float v) {
        const int i = __float_as_int(v);
        return i >= 0 ? i : i ^ 0x7fffffff;
    };
    auto val = [](int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); };
    if (tid < NG) {
        s_v[tid][0] = s_v[tid][2] = key(3.0e38f);
        s_v[tid][1] = s_v[tid][3] = key(-3.0e38f);
    }
    __syncthreads();
    if (valid) {
        const int g = n % TXS / 8;
        atomicMin(&s_v[g][0], key(ux - sp));
        atomicMax(&s_v[g][1], key(ux + sp));
        atomicMin(&s_v[g][2], key(uy - sp));
        atomicMax(&s_v[g][3], key(uy + sp));
    }
    __syncthreads();
    for (int i = tid; i < ww * wh; i += NT) {
        if (s_h[i].x != kFixBadSource) continue;
        const int x = wx0 + i % ww, y = wy0 + i / ww;
        for (int g = 0; g < NG; ++g) {
            const int gx = tx0 + 8 * g;
            if (x >= (int)floorf((float)gx - val(s_v[g][1]) * fdt - m) - 1 &&
                x <= (int)floorf((float)(gx + 7) - val(s_v[g][0]) * fdt + m) + 2 &&
                y >= (int)floorf((float)ty0 - val(s_v[g][3]) * fdt - m) - 1 &&
                y <= (int)floorf((float)(ty0 + TYS - 1) - val(s_v[g][2]) * fdt + m) + 2)
                atomicOr(s_bad, 1u << g);
        }
    }
    __syncthreads();
    return *s_bad;
}

// The step with its contractions in fixed point: k_step_staged's tile, window,
// pass loop and fallbacks (its comments hold here), over CTAs of TXS x TYS
// target nodes of the LTX x LTY tiles that fix the reference gauge and scale,
// so that every shape gives a node the same staged values and sums, bit for
// bit.  A 32 x 8 window takes most of an SM's shared memory, so one CTA of 256
// threads runs per SM, a thread per node (KS = 1, 255 registers: two threads
// per node at 128 registers, splitting the components b, spilled and measured
// 26 ms against 22.7 for a 2048^2 step).  With fewer tiles than SMs, parts of 8
// x LTY nodes run with KS = 4 lanes per node, lane `part` sweeping the x-speed k
// = part and computing the y-stencil and y-map row l = part; eight nodes stand
// side by side in a quarter warp, whose 16-byte reads are then contiguous.
// The gauge update runs in all lanes of a node.  A pass's populations (64-bit
// integers) wait in the output planes for the closing re-gauge.  What is out of
// range goes to A.redo_list, by groups of 8 columns whose nodes and window decide
// for themselves: which nodes the FP64 form computes does not depend on the shape
// either, and a steep spot takes 8 columns with it, not a tile.
template <class Tr, int LTX, int LTY, int TXS, int TYS, int KS, int N1, int MINB>
__global__ void __launch_bounds__(TXS* TYS* KS, MINB) k_step_fixed(StagedArgs<double> A) {
    constexpr int NN = TXS * TYS, NT = NN * KS, Q = N1 * N1;
    constexpr int SUB = LTX / TXS, NG = TXS / 8;
    constexpr unsigned FULL = 0xffffffffu;
    static_assert(NT % 32 == 0 && (KS == 1 || KS == 4) && LTX % TXS == 0 && LTY == TYS && TXS % 8 == 0,
                  "whole warps, the lanes of a node in one");
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int WN = A.wn;
    int4* s_h = reinterpret_cast<int4*>(smem_raw);                 // [N1][WN] high words
    int4* s_l = s_h + (size_t)N1 * WN;                             // [N1][WN] low words
    int2* s_gy = reinterpret_cast<int2*>(s_l + (size_t)N1 * WN);   // [Q][NN] y-map of the pass
    int2* s_ly = s_gy + (size_t)Q * NN;                            // [4 N1][NN] y-weights
    int* s_top = reinterpret_cast<int*>(s_ly + (size_t)4 * N1 * NN);  // [N1][NN]
    __shared__ float s_red[4][NT / 32];
    __shared__ long long s_item;
    __shared__ unsigned long long s_passes, s_nc, s_np, s_fb;
    __shared__ unsigned int s_max, s_bad, s_late;
    const Lattice& L = Tr::template lat<N1>();
    const LatticeFix& F = Tr::template lat_fix<N1>();
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_passes = 0ull;
        s_nc = 0ull;
        s_np = 0ull;
        s_fb = 0ull;
        s_max = 0u;
    }
    const int lane = tid & 31, part = lane / (32 / KS);
    const int n = tid / 32 * (32 / KS) + lane % (32 / KS);
    // the value of lane `part` = k of this lane's node
    auto from_part = [&](double v, int k) {
        return KS == 1 ? v : __shfl_sync(FULL, v, k * (32 / KS) + lane % (32 / KS));
    };
    const double dt54 = A.P.dt * kFixDisplacement;
    const float c_max = (float)A.c_max;
    const unsigned long long t_begin = (A.work_counter && tid == 0) ? pond_globaltimer() : 0ull;

    long long item = blockIdx.x;
    for (;;) {
        if (A.work_counter) {
            __syncthreads();
            if (tid == 0) s_item = (long long)atomicAdd(A.work_counter, 1u);
            __syncthreads();
            item = s_item;
        }
        if (item >= A.n_tiles * SUB) break;

        const long long tile = item / SUB;
        const int sub = (int)(item % SUB);
        int g = 0;
        if (A.n_grids > 1) {
            int lo = 0, hi = A.n_grids - 1;  // largest g with prefix[g] <= tile
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (A.tile_prefix[mid] <= tile) lo = mid; else hi = mid - 1;
            }
            g = lo;
        }
        const GridDesc G = A.n_grids == 1 ? A.grid0 : A.grids[g];
        const long long t = A.n_grids == 1 ? tile : tile - A.tile_prefix[g];
        const int tiles_x = (G.iw + LTX - 1) / LTX;
        const int ltx0 = G.ix0 + (int)(t % tiles_x) * LTX;
        const int lty0 = G.iy0 + (int)(t / tiles_x) * LTY;
        const int tx0 = ltx0 + sub * TXS, ty0 = lty0;
        if (SUB > 1 && tx0 >= G.ix0 + G.iw) {  // nothing of a ragged tile
            if (!A.work_counter) break;
            continue;
        }
        if (tid == 0) s_bad = s_late = 0u;
        const int X = tx0 + n % TXS, Y = ty0 + n / TXS;
        const unsigned group = 1u << (n % TXS / 8);
        bool valid = X < G.ix0 + G.iw && Y < G.iy0 + G.ih;
        const long long base = G.offset;
        const long long node = base + (long long)Y * G.nx + X;
        const long long rnode = base + (long long)min(lty0 + LTY / 2, G.iy0 + G.ih - 1) * G.nx +
                                min(ltx0 + LTX / 2, G.ix0 + G.iw - 1);
        const double rux = A.in.ux[rnode], ruy = A.in.uy[rnode], rst = A.in.st[rnode];

        // the tile's scale: the exponent of the centre node's largest scaled
        // population (each warp finds it for itself)
        unsigned mh = 0u;
        if (lane < Q) {
            const int s = fix_shift<N1>(lane / N1) + fix_shift<N1>(lane % N1);
            const double v = fabs(A.in.f[(long long)lane * A.plane + rnode]) * (double)(1 << s);
            mh = (unsigned)__double2hiint(v);
        }
        mh = __reduce_max_sync(FULL, mh);
        const int me = (int)(mh >> 20) - 1023;    // M in [2^me, 2^(me + 1))
        const int rexp = me + 5;                  // R = 2^rexp
        bool in_range = me > -900 && me < 900;    // rules out 0, Inf and NaN

        PassGauge pg;
        pg.ux = 0.0;
        pg.uy = 0.0;
        pg.st = 1.0;
        float vxlo = 3.0e38f, vxhi = -3.0e38f, vylo = 3.0e38f, vyhi = -3.0e38f;
        if (valid) {
            pg.ux = A.in.ux[node];
            pg.uy = A.in.uy[node];
            pg.st = A.in.st[node];
            if (A.P.seed_mode == 1) {
                pg.ux = 0.0;
                pg.uy = 0.0;
                pg.st = 1.0;
            } else if (A.P.seed_mode == 2) {
                pg.ux = -pg.ux;
                pg.uy = -pg.uy;
            }
            const float sp = (float)(A.c_max * pg.st);
            vxlo = (float)pg.ux - sp;
            vxhi = (float)pg.ux + sp;
            vylo = (float)pg.uy - sp;
            vyhi = (float)pg.uy + sp;
            const float de = fmaf(c_max, fabsf((float)(rst - pg.st)),
                                  fmaxf(fabsf((float)(rux - pg.ux)), fabsf((float)(ruy - pg.uy))));
            in_range = in_range && de <= kFixTileDe * (float)pg.st;
        }
        const float fdt = (float)A.P.dt;
        // (finite, and displacements in the fixed-point range of fix_departure)
        in_range = in_range && (!valid || (vxlo * fdt > -400.0f && vxhi * fdt < 400.0f &&
                                           vylo * fdt > -400.0f && vyhi * fdt < 400.0f));
        staged_block_minmax4<Tr, NT>(vxlo, vxhi, vylo, vyhi, s_red);
        unsigned bad = 0u;  // groups out of range (uniform)
        if (__syncthreads_or(!in_range)) {
            if (!in_range) atomicOr(&s_bad, group);
            __syncthreads();
            bad = s_bad;
            if (NG > 1) {  // the window of the others
                valid = valid && !(bad & group);
                const float sp = (float)(A.c_max * pg.st);
                vxlo = valid ? (float)pg.ux - sp : 3.0e38f;
                vxhi = valid ? (float)pg.ux + sp : -3.0e38f;
                vylo = valid ? (float)pg.uy - sp : 3.0e38f;
                vyhi = valid ? (float)pg.uy + sp : -3.0e38f;
                staged_block_minmax4<Tr, NT>(vxlo, vxhi, vylo, vyhi, s_red);
            }
        }
        constexpr unsigned ALL = (1u << NG) - 1u;

        // staged window in unwrapped grid coordinates (departure = x - v dt); with
        // no node left in range it is empty and not staged
        const float m = A.margin;
        const bool any = vxlo <= vxhi;
        const int wx0 = any ? (int)floorf((float)tx0 - vxhi * fdt - m) - 1 : 0;
        const int wx1 = any ? (int)floorf((float)(tx0 + TXS - 1) - vxlo * fdt + m) + 2 : 0;
        const int wy0 = any ? (int)floorf((float)ty0 - vyhi * fdt - m) - 1 : 0;
        const int wy1 = any ? (int)floorf((float)(ty0 + TYS - 1) - vylo * fdt + m) + 2 : 0;
        const int ww = max(1, min(wx1 - wx0 + 1, A.ww));
        const int wh = max(1, min(min(wy1 - wy0 + 1, A.wh), WN / ww));
        if (bad != ALL) {
            const bool ok = stage_window_fixed<N1, KS == 1>(A.in, A.plane, G, base, wx0, wy0, ww, wh, WN,
                                                            rux, ruy, rst, kFix - rexp, s_h, s_l, F,
                                                            c_max, A.stats, tid, NT);
            if (__syncthreads_or(!ok)) {  // also: the window is staged
                if (NG > 1) {
                    bad |= fixed_bad_groups<TXS, TYS, NT>(s_h, wx0, wy0, ww, wh, tx0, ty0, m, fdt, valid,
                                                          (float)pg.ux, (float)pg.uy,
                                                          (float)(A.c_max * pg.st), n, &s_bad);
                    valid = valid && !(bad & group);
                } else {
                    bad = ALL;
                }
            }
        }
        if (bad) {
            if (tid < NG && (bad >> tid & 1u) && tx0 + 8 * tid < G.ix0 + G.iw)
                A.redo_list[atomicAdd(A.redo_count, 1u)] = (unsigned)(item * NG + tid);
            if (bad == ALL) {
                if (!A.work_counter) break;
                continue;
            }
        }

        // ---------------------------------------------------- pass loop
        const double f_unit = pow2d(rexp - kFix);  // a scaled population's unit
        pg.nux = pg.ux;
        pg.nuy = pg.uy;
        pg.nst = pg.st;
        pg.rho = 0.0;
        pg.pass = 0;
        pg.flag = 0u;
        unsigned int fallbacks = 0u;
        unsigned int offwin = 0u, off_last = 0u;  // populations of a pass read from global memory
        bool done = !valid;
        while (__any_sync(FULL, !done)) {
            const double st = pg.st, ux = pg.ux, uy = pg.uy;
            // target gauge of this pass: its offsets from lambda_r
            const double inv = kFixOne / st;
            const long long rt = __double2ll_rn((rst - st) * inv);
            const long long dxt = __double2ll_rn((rux - ux) * inv);
            const long long dyt = __double2ll_rn((ruy - uy) * inv);
            if (!done && !(fix_offset(rt, dxt, dyt, c_max) <= kFixNodeDe)) {
                // the node left the range on the way: to the FP64 form, by its
                // mark (staged_fallback took it at first, 16 populations one
                // after the other: 15 such nodes held a step for 4 ms)
                done = true;
                valid = false;
                if (part == 0) {
                    A.out.st[node] = __longlong_as_double(kRedoMark);
                    if (!(atomicOr(&s_late, group) & group))
                        A.redo_list[atomicAdd(A.redo_count, 1u)] =
                            kRedoMarked | (unsigned)(item * NG + n % TXS / 8);
                }
            }
            const bool work = !done;
            const Fix Rt = fix_split(rt);
            __syncwarp();  // the tables are written again
            if (work) {
                // y-map r -> lambda of the pass, and the y-stencils: top row in
                // the window and weights
                Fix de[N1];
#pragma unroll
                for (int b = 0; b < N1; ++b) de[b] = fix_split(dyt + fix_mul(F.c[b], Rt));
#pragma unroll 1
                for (int l = part; l < N1; l += KS) {
#pragma unroll
                    for (int b = 0; b < N1; ++b) {
                        const Fix gw = fix_gauge<N1>(F, l, b, de[b]);
                        s_gy[(N1 * l + b) * NN + n] = make_int2(gw.h, gw.l);
                    }
                    const double d = -fma(st, L.c[l], uy) * dt54;
                    Fix ly[4];
                    int top = Y - wy0 - 1 + fix_departure(__double2ll_rn(d), ly);
#pragma unroll
                    for (int j = 0; j < 4; ++j) s_ly[(4 * l + j) * NN + n] = make_int2(ly[j].h, ly[j].l);
                    if (!(fabs(d) < 500.0 * kFixDisplacement && top >= 0 && top + 3 < wh))
                        top = -1;
                    s_top[l * NN + n] = top;
                }
            }
            __syncwarp();
            int last[N1];  // the row that completes population l's stencil
            int lo = 0x7fffffff, hi = -1;
            offwin = 0u;
#pragma unroll
            for (int l = 0; l < N1; ++l) {
                const int top = work ? s_top[l * NN + n] : -1;
                last[l] = top >= 0 ? top + 3 : -1;
                if (top >= 0) {
                    lo = min(lo, top);
                    hi = max(hi, top + 3);
                }
            }
            double m0 = 0, m1 = 0, m2 = 0, m3 = 0;
#pragma unroll 1
            for (int k0 = 0; k0 < N1; k0 += KS) {
                const int k = KS == 1 ? k0 : min(part, N1 - 1);
                const bool mine = KS == 1 || part < N1;  // D2Q9: the fourth lane idles
                const double ck = L.c[k];
                const bool outer = k == 0 || k == N1 - 1;
                const double d = -fma(st, ck, ux) * dt54;
                // the row's weights, cxa[jx][a] = lx[jx] G_x(r -> lambda)[k][a]
                Fix cxa[4][N1];
                int col;
                {
                    Fix lx[4];
                    col = X - wx0 - 1 + fix_departure(__double2ll_rn(d), lx);
#pragma unroll
                    for (int a = 0; a < N1; ++a) {
                        const Fix gw = fix_gauge<N1>(F, k, a, fix_split(dxt + fix_mul(F.c[a], Rt)));
#pragma unroll
                        for (int jx = 0; jx < 4; ++jx) cxa[jx][a] = fix_split(fix_mul(lx[jx], gw));
                    }
                }
                const bool on = work && mine && hi >= 0 && fabs(d) < 500.0 * kFixDisplacement && col >= 0 &&
                                col + 3 < ww;
                // the sweep over the rows of the union of the y-stencils keeps
                // the last four rows' P; population l takes its rows when the
                // sweep reaches its last one
                Fix Pb[4][N1];
                long long f[N1];  // the populations (k, l)
#pragma unroll
                for (int l = 0; l < N1; ++l) f[l] = 0;
#pragma unroll 1
                for (int y = lo; on && y <= hi; ++y) {
                    const int4* sh = s_h + y * ww + col;
                    const int4* sl = s_l + y * ww + col;
                    const bool rowok = POND_INDEX_OK(y >= 0 && col >= 0 && y < wh && col + 3 < ww &&
                                                         y * ww + col + 3 < WN,
                                                     A.stats);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int b = 0; b < N1; ++b) Pb[i][b] = Pb[i + 1][b];
                    long long h[4], mm[4];
#pragma unroll
                    for (int b = 0; b < 4; ++b) h[b] = mm[b] = 0;
#pragma unroll
                    for (int jx = 0; jx < 4; ++jx) {
#pragma unroll
                        for (int a = 0; a < N1; ++a) {
                            int4 gh = make_int4(0, 0, 0, 0), gl = make_int4(0, 0, 0, 0);
                            if (rowok) {
                                gh = sh[(size_t)a * WN + jx];
                                gl = sl[(size_t)a * WN + jx];
                            }
                            fix_mad(cxa[jx][a], gh.x, gl.x, h[0], mm[0]);
                            fix_mad(cxa[jx][a], gh.y, gl.y, h[1], mm[1]);
                            fix_mad(cxa[jx][a], gh.z, gl.z, h[2], mm[2]);
                            if (N1 == 4) fix_mad(cxa[jx][a], gh.w, gl.w, h[3], mm[3]);
                        }
                    }
#pragma unroll
                    for (int b = 0; b < N1; ++b) Pb[3][b] = fix_split(fix_sum(h[b], mm[b]));
                    unsigned todo = 0u;
#pragma unroll
                    for (int l = 0; l < N1; ++l) todo |= y == last[l] ? 1u << l : 0u;
                    while (todo) {
                        const int l = __ffs(todo) - 1;
                        todo &= todo - 1;
                        long long fh = 0, fm = 0;
                        Fix ly[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int2 v = s_ly[(4 * l + j) * NN + n];
                            ly[j] = Fix{v.x, v.y};
                        }
#pragma unroll
                        for (int b = 0; b < N1; ++b) {
                            long long zh = 0, zm = 0;
#pragma unroll
                            for (int j = 0; j < 4; ++j) fix_mad(ly[j], Pb[j][b].h, Pb[j][b].l, zh, zm);
                            const Fix z = fix_split(fix_sum(zh, zm));
                            const int2 gw = s_gy[(N1 * l + b) * NN + n];
                            fix_mad(Fix{gw.x, gw.y}, z.h, z.l, fh, fm);
                        }
                        const long long v = fix_sum(fh, fm);
#pragma unroll
                        for (int i = 0; i < N1; ++i) f[i] = i == l ? v : f[i];
                    }
                }
#pragma unroll
                for (int l = 0; l < N1; ++l) {
                    const bool in = on && last[l] >= 0;
                    if (work && mine && !in) offwin |= 1u << (N1 * k + l);
                    if (in) A.out.f[(long long)(N1 * k + l) * A.plane + node] = __longlong_as_double(f[l]);
                }
                // sums over l of f (A), c_l f (B) and c_l^2 f (C), of two at half
                // the scale, added up in the order of k
                constexpr double dn = 1.0 / (double)(1 << fix_shift<N1>(0));
                const double u = 2.0 * f_unit * (outer ? dn : 1.0);
                const long long f0 = f[0] >> 1, f3 = f[N1 - 1] >> 1;
                const double so = (double)(f0 + f3) * (u * dn), c_out = L.c[N1 - 1];
                double sa, sb = c_out * ((double)(f3 - f0) * (u * dn)), sc = c_out * c_out * so;
                if (N1 == 4) {
                    const long long f1 = f[1] >> 1, f2 = f[N1 - 2] >> 1;
                    const double si = (double)(f1 + f2) * u, c_in = L.c[2];
                    sa = si + so;
                    sb = fma(c_in, (double)(f2 - f1) * u, sb);
                    sc = fma(c_in * c_in, si, sc);
                } else {
                    sa = fma((double)f[1], 0.5 * u, so);
                }
#pragma unroll
                for (int i = 0; i < (KS == 1 ? 1 : N1); ++i) {
                    const double ci = KS == 1 ? ck : L.c[i], ai = from_part(sa, i);
                    m0 += ai;
                    m1 = fma(ci, ai, m1);
                    m2 += from_part(sb, i);
                    m3 += fma(ci * ci, ai, from_part(sc, i));
                }
            }
            if (KS > 1) {
#pragma unroll
                for (int o = 32 / KS; o < 32; o <<= 1) offwin |= __shfl_xor_sync(FULL, offwin, o);
            }
            if (work) {
                // populations whose stencil leaves the staged window, from global
                // memory; kept as doubles in their slots
                for (unsigned int left = offwin; left; left &= left - 1) {
                    const int q = __ffs(left) - 1;
                    const int k = q / N1, l = q - N1 * k;
                    const double acc = staged_fallback<Tr, N1>(A, G, base, X, Y, k, l, ux, uy, st);
                    ++fallbacks;
                    if (part == 0) A.out.f[(long long)q * A.plane + node] = acc;
                    const double ck = L.c[k], cl = L.c[l];
                    m0 += acc;
                    m1 = fma(ck, acc, m1);
                    m2 = fma(cl, acc, m2);
                    m3 = fma(fma(ck, ck, cl * cl), acc, m3);
                }
                off_last = offwin;
                done = Tr::update(A.P, pg, m0, m1, m2, m3);
            }
        }

        // the node's last populations into its co-moving gauge, BGK and the
        // store, as Tr::finish -- which takes the nodes out of the fixed-point
        // range: populations read from global memory, a large last increment,
        // non-physical moments.  A lane takes its y-speeds l = part, ...
        __syncwarp();
        unsigned passes = 0u;
        const bool store = valid && POND_INDEX_OK(node >= base && node < base + (long long)G.nx * G.ny, A.stats);
        Fix v[Q];
        int top = 0;
        if (store) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                v[q] = fix_split(__double_as_longlong(A.out.f[(long long)q * A.plane + node]));
                top = max(top, abs(v[q].h));
            }
        }
        __syncwarp();  // all lanes of a node have read its populations
        if (store) {
            const double finv = kFixOne / pg.nst;
            const long long fr = __double2ll_rn((pg.st - pg.nst) * finv);
            const long long fdx = __double2ll_rn((pg.ux - pg.nux) * finv);
            const long long fdy = __double2ll_rn((pg.uy - pg.nuy) * finv);
            const bool fixed = off_last == 0u && !(pg.flag & 2u) && top < (1 << (kFix - 32)) &&
                               fix_offset(fr, fdx, fdy, c_max) <= kFixNodeDe;
            if (fixed) {
                const Fix FR = fix_split(fr);
                const double two_beta = 2.0 * A.P.beta;
                const double keep = (1.0 - two_beta) * f_unit, eq = two_beta * pg.rho;
                Fix gx[N1][N1], dey[N1];
#pragma unroll
                for (int a = 0; a < N1; ++a) {
                    const long long ca = fix_mul(F.c[a], FR);
                    const Fix de = fix_split(fdx + ca);
                    dey[a] = fix_split(fdy + ca);
#pragma unroll
                    for (int k = 0; k < N1; ++k) gx[k][a] = fix_gauge<N1>(F, k, a, de);
                }
#pragma unroll 1
                for (int l = part; l < N1; l += KS) {
                    Fix gw[N1], H[N1];
#pragma unroll
                    for (int b = 0; b < N1; ++b) gw[b] = fix_gauge<N1>(F, l, b, dey[b]);
#pragma unroll
                    for (int a = 0; a < N1; ++a) {
                        long long h = 0, mm = 0;
#pragma unroll
                        for (int b = 0; b < N1; ++b) fix_mad(gw[b], v[N1 * a + b].h, v[N1 * a + b].l, h, mm);
                        H[a] = fix_split(fix_sum(h, mm));
                    }
                    constexpr double dn = 1.0 / (double)(1 << fix_shift<N1>(0));
                    const double ul = l == 0 || l == N1 - 1 ? keep * dn : keep;
                    const double el = eq * L.w[l];
#pragma unroll
                    for (int k = 0; k < N1; ++k) {
                        long long h = 0, mm = 0;
#pragma unroll
                        for (int a = 0; a < N1; ++a) fix_mad(gx[k][a], H[a].h, H[a].l, h, mm);
                        A.out.f[(long long)(N1 * k + l) * A.plane + node] =
                            fma((double)fix_sum(h, mm), fix_shift<N1>(k) ? ul * dn : ul, el * L.w[k]);
                    }
                }
                if (part == 0) {
                    A.out.ux[node] = pg.nux;
                    A.out.uy[node] = pg.nuy;
                    A.out.st[node] = pg.nst;
                }
            } else if (part == 0) {
                // the populations as doubles, in the node's column of the y-map table
                double* acc = reinterpret_cast<double*>(s_gy);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const double us = 1.0 / (double)(1 << (fix_shift<N1>(q / N1) + fix_shift<N1>(q % N1)));
                    const long long w = (long long)v[q].h * (1ll << 32) + v[q].l;
                    acc[q * NN + n] = (off_last >> q & 1u) ? __longlong_as_double(w) : (double)w * (f_unit * us);
                }
                Tr::template finish<N1>(A, acc, NN, n, node, pg);
            }
            if (part == 0) {
                if (A.iters) A.iters[node] = pg.pass;
                passes = (unsigned)pg.pass;
                if (pg.flag & 1u) atomicAdd(&s_nc, 1ull);
                if (pg.flag & 2u) atomicAdd(&s_np, 1ull);
                if (fallbacks) atomicAdd(&s_fb, (unsigned long long)fallbacks);
            }
        }
        __syncwarp();
        const unsigned wsum = __reduce_add_sync(FULL, passes), wmax = __reduce_max_sync(FULL, passes);
        if (lane == 0) {
            atomicAdd(&s_passes, (unsigned long long)wsum);
            atomicMax(&s_max, wmax);
        }
        if (!A.work_counter) break;
        __syncthreads();  // the next item restages the window
    }
    __syncthreads();
    if (tid == 0 && A.stats) {
        if (s_passes) {
            atomicAdd(&A.stats->passes, s_passes);
            atomicMax(&A.stats->max_passes, s_max);
        }
        if (s_nc) atomicAdd(&A.stats->nonconverged, s_nc);
        if (s_np) atomicAdd(&A.stats->nonphysical, s_np);
        if (s_fb) atomicAdd(&A.stats->halo_fallback, s_fb);
        if (A.work_counter) persistent_exit(A.stats, t_begin);
    }
}

// Dynamic shared memory of k_step_fixed: the staged planes, and per node the
// y-map and y-weight tables and the stencil tops.
inline size_t fixed_smem_bytes(int n1, int wn, int nodes) {
    return (size_t)n1 * wn * 32 + (size_t)nodes * (8 * (n1 * n1 + 4 * n1) + 4 * n1);
}

}  // namespace pond
