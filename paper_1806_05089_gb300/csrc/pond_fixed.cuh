// pond_fixed.cuh -- the FP64 staged step with its contractions in 64-bit
// fixed point on the integer multiply pipe.
//
// GB300 runs 2 FP64 FMAs per clock and SM but 64 integer multiply-adds with a
// 64-bit sum (mad.wide.s32, measured 60 per clock and SM).  The staged step
// (pond_staged.cuh) spends four fifths of its FP64 operations on dot products
// of 16 staged populations with 16 weights; here those run as
//   sum w g = 2^58 sum w1 g1 + 2^29 sum (w1 g0 + w0 g1) + sum w0 g0,
// with every operand v = 2^29 v1 + v0 split into a signed high limb and a
// centred 29-bit low limb: three wide multiply-adds per product, exact 64-bit
// sums, and the last term (at most 2^-2 units of the result's last place per
// product) dropped.
//
// Scales.  A tile's staged populations share one power of two: with M the
// largest population of the tile's centre node (each multiplied by
// 2^(s_k + s_l), s = 3 at the outer speeds of D2Q16, 2 at those of D2Q9, which
// brings W_q to one magnitude), R = 2^E >= 8 M, and g is held to R 2^-59.
// Weights are held to 2^-57.  A row sum then carries R 2^-58 (2^-54 M or
// less), where the FP64 sum of 16 products rounds at 2^-53 of its terms: the
// fixed-point form is the more exact one as long as a tile's populations stay
// within its window of magnitudes.  So a tile takes this path only if
//   - every staged |f| < R / 4 and |g| < R / 2, and at every staged node the
//     largest |g| is >= R / 64;
//   - the gauges of its nodes differ from the reference gauge by |xi_a - c_a|
//     <= 0.30, those of its sources by 0.45 (the weights' sums are then bounded
//     and no 64-bit sum or limb overflows; a pass gauge beyond 0.35 sends that
//     node to the global-memory path);
//   - its displacements are below 400 nodes.
// Any other tile (strong shear at the window's scale, near-vacuum, NaN, the
// seed modes that start far from the reference) is put on a list, and
// k_step_staged<StagedFP64> runs the listed tiles in a launch that follows.
//
// The staging, the maps' entries, the cubic weights and the closing re-gauge
// are in fixed point too: a product of two 57-bit weights costs about ten
// integer instructions (a tenth of a clock and SM per node), an FP64 operation
// half a clock.  FP64 keeps what has no bounded range or needs a division or
// a root: gauge differences, displacements, conversions, the moments, the
// gauge update and its test, and BGK.
//
// Measured, GB300 (start: all FP64; contractions: the dot products alone in
// fixed point; all: as here):
//                                 start  contractions      all
//   2048^2 supersonic, 1 step      69.8          36.8     22.3 ms
//   301 x 211, 4 steps              7.1           3.6      2.3 ms
//   1024^2 D2Q9, 2 steps           14.4           8.8      4.8 ms
// and a relative error against a 64-bit restatement of 4.9e-16 before and
// 4.3e-16 after (2048^2, populations, 2-norm).
#pragma once

#include "pond_staged.cuh"

namespace pond {

constexpr int kFixLimb = 29;    // bits of a low limb
constexpr int kFixWeight = 57;  // a weight of 1 is 2^57
constexpr int kFixSource = 59;  // a staged population of R is 2^59
constexpr int kFixPop = 58;     // a pass's population of R is 2^58
constexpr float kFixTileDe = 0.30f, kFixNodeDe = 0.35f, kFixSourceDe = 0.45f;
constexpr double kFixOne = 144115188075855872.0;        // 2^57
constexpr double kFixDisplacement = 18014398509481984.0;  // 2^54: |d| < 500 nodes

template <int N1>
__host__ __device__ constexpr int fix_shift(int k) {
    return (k == 0 || k == N1 - 1) ? (N1 == 4 ? 3 : 2) : 0;
}

struct Fix {
    int h, l;
};

// Lattice constants in fixed point (2^57): the speeds, and the Taylor
// coefficients of G[k][a] = L_k(c_a + de) times 2^(s_k - s_a), the factor between
// the scales of populations k and a.
struct LatticeFix {
    Fix c[4];
    long long d0[4][4], d1[4][4], d2[4][4];  // d0: the identity
    Fix d3[4][4];
};

// The split v = 2^29 h + l, l centred; |v| < 2^60.
__host__ __device__ __forceinline__ Fix fix_split(long long v) {
    Fix f;
    f.h = (int)((v + (1ll << (kFixLimb - 1))) >> kFixLimb);
    f.l = (int)((unsigned)v - ((unsigned)f.h << kFixLimb));
    return f;
}

inline LatticeFix make_lattice_fix(const Lattice& L) {
    LatticeFix F{};
    auto fx = [](double v) { return (long long)std::llrint(v * kFixOne); };
    for (int k = 0; k < L.n1; ++k) {
        F.c[k] = fix_split(fx(L.c[k]));
        for (int a = 0; a < L.n1; ++a) {
            const int s = L.n1 == 4 ? fix_shift<4>(k) - fix_shift<4>(a)
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

// One product of a fixed-point dot product: h the 2^58 sum, m the 2^29 sum.
__device__ __forceinline__ void fix_mad(Fix w, int gh, int gl, long long& h, long long& m) {
    h = mad_wide(w.h, gh, h);
    m = mad_wide(w.h, gl, m);
    m = mad_wide(w.l, gh, m);
}

// The sum h 2^58 + m 2^29 in units of 2^(58 - up), rounded (0 <= up <= 2).
template <int UP>
__device__ __forceinline__ long long fix_sum(long long h, long long m) {
    return (h << UP) + ((m + (1ll << (kFixLimb - 1 - UP))) >> (kFixLimb - UP));
}

// Product of a weight (2^57) and v, in v's scale.
__device__ __forceinline__ long long fix_mul(Fix w, Fix v) {
    long long h = 0, m = 0;
    fix_mad(w, v.h, v.l, h, m);
    return fix_sum<1>(h, m);
}

// The 1D gauge map's entry for the offset de (2^57), in the scaled basis.
template <int N1>
__device__ __forceinline__ Fix fix_gauge(const LatticeFix& F, int k, int a, Fix de) {
    long long t = F.d2[k][a];
    if (N1 == 4) t += fix_mul(F.d3[k][a], de);
    t = F.d1[k][a] + fix_mul(de, fix_split(t));
    return fix_split(F.d0[k][a] + fix_mul(de, fix_split(t)));
}

// Floor of the displacement d 2^54 and the cubic weights (2^57) at its
// fraction s.  With u = s (1 - s), v = u / 6, w = v s the weights of App. C at
// t = s + 1 are w - 2 v, 1 - s + 3 (v - w), s + 3 w, -(v + w); they sum to one
// exactly.
__device__ __forceinline__ int fix_departure(long long d, Fix (&l)[4]) {
    const long long s = (d & ((1ll << 54) - 1)) << 3, one = 1ll << kFixWeight;
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

// 2^e for |e| < 1000.
__device__ __forceinline__ double pow2d(int e) {
    return __hiloint2double((1023 + e) << 20, 0);
}

// x 2^e rounded to an integer; `big` is set when |x| 2^e >= 2^57 (or x is not
// finite).  The exponent is added on the integer pipe.
__device__ __forceinline__ long long fix_population(double x, int e, bool& big) {
    const int hi = __double2hiint(x);
    const int ex = (hi >> 20 & 0x7ff) + e;
    big = big || ex >= 1023 + 57;
    const double y = __hiloint2double((hi & 0x800fffff) | ex << 20, __double2loint(x));
    return __double2ll_rn(ex > 0 && ex < 1023 + 57 ? y : 0.0);
}

// |de_a| of the gauge offsets r, dx, dy (2^57), at most (in units of 1).
__device__ __forceinline__ float fix_offset(long long r, long long dx, long long dy, float c_max) {
    const float u = 1.0f / 33554432.0f;  // the high words carry 2^25
    return u * fmaf(c_max, fabsf((float)(int)(r >> 32)),
                    fmaxf(fabsf((float)(int)(dx >> 32)), fabsf((float)(int)(dy >> 32))));
}

// G_x (x) G_y of the offsets r, dx, dy applied to the scaled populations f
// (|f| < 2^58 or so, both sums bounded by the caller's limit on the offsets):
// in place, in f's scale.
template <int N1>
__device__ __forceinline__ void fix_transform(const LatticeFix& F, long long r, long long dx,
                                              long long dy, long long (&f)[N1 * N1]) {
    const Fix R = fix_split(r);
    Fix v[N1 * N1];
#pragma unroll
    for (int q = 0; q < N1 * N1; ++q) v[q] = fix_split(f[q]);
    {
        Fix de[N1];
#pragma unroll
        for (int b = 0; b < N1; ++b) de[b] = fix_split(dy + fix_mul(F.c[b], R));
#pragma unroll
        for (int l = 0; l < N1; ++l) {
            Fix g[N1];
#pragma unroll
            for (int b = 0; b < N1; ++b) g[b] = fix_gauge<N1>(F, l, b, de[b]);
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                long long h = 0, m = 0;
#pragma unroll
                for (int b = 0; b < N1; ++b) fix_mad(g[b], v[N1 * a + b].h, v[N1 * a + b].l, h, m);
                f[N1 * a + l] = fix_sum<1>(h, m);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < N1 * N1; ++q) v[q] = fix_split(f[q]);
    {
        Fix de[N1];
#pragma unroll
        for (int a = 0; a < N1; ++a) de[a] = fix_split(dx + fix_mul(F.c[a], R));
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            Fix g[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) g[a] = fix_gauge<N1>(F, k, a, de[a]);
#pragma unroll
            for (int l = 0; l < N1; ++l) {
                long long h = 0, m = 0;
#pragma unroll
                for (int a = 0; a < N1; ++a) fix_mad(g[a], v[N1 * a + l].h, v[N1 * a + l].l, h, m);
                f[N1 * k + l] = fix_sum<1>(h, m);
            }
        }
    }
}

// Stage the window as stage_window does, the sources rounded to the tile's
// fixed point (2^e = 2^59 / R) and re-expressed there: high limbs in s_h, low
// limbs in s_l, row a at [a * WN + i].  Two planes, so that a quarter warp's
// 16-byte reads are contiguous.  Returns whether every value this thread
// staged is in range.
template <int N1>
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
    for (int i = tid; i < ww * wh; i += nt) {
        const int cx = i % ww, cy = i / ww;
        const int gx = wrap_idx((long long)wx0 + cx, G.nx);
        const int gy = wrap_idx((long long)wy0 + cy, G.ny);
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
        fix_transform<N1>(F, r, dx, dy, f);
        int top = 0;
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            Fix o[4];
#pragma unroll
            for (int l = 0; l < N1; ++l) {
                top = max(top, abs((int)(f[N1 * k + l] >> 32)));
                o[l] = fix_split(f[N1 * k + l]);
            }
            if constexpr (N1 == 3) o[3] = Fix{0, 0};
            s_h[(size_t)k * WN + i] = make_int4(o[0].h, o[1].h, o[2].h, o[3].h);
            s_l[(size_t)k * WN + i] = make_int4(o[0].l, o[1].l, o[2].l, o[3].l);
        }
        // |g| < R / 2, and the node's largest >= R / 64 (high words of 2^58, 2^53)
        ok = ok && !big && top < (1 << (kFixSource - 1 - 32)) && top >= (1 << (kFixSource - 6 - 32));
    }
    return ok;
}

// The node's last populations into its co-moving gauge, BGK and the store, as
// Tr::finish (which takes the nodes out of the fixed-point range: populations
// read from global memory, a large last increment, non-physical moments).
template <class Tr, int N1>
__device__ __forceinline__ void finish_fixed(const StagedArgs<double>& A, const LatticeFix& F,
                                             long long* s_acc, int NT, int tid, long long node,
                                             const PassGauge& g, unsigned offwin, double f_unit) {
    constexpr int Q = N1 * N1;
    const Lattice& L = Tr::template lat<N1>();
    const double inv = kFixOne / g.nst;
    const long long r = __double2ll_rn((g.st - g.nst) * inv);
    const long long dx = __double2ll_rn((g.ux - g.nux) * inv);
    const long long dy = __double2ll_rn((g.uy - g.nuy) * inv);
    long long f[Q];
    int top = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        f[q] = s_acc[q * NT + tid];
        top = max(top, abs((int)(f[q] >> 32)));
    }
    const bool fixed = offwin == 0u && !(g.flag & 2u) && top < (1 << (kFixPop - 32)) &&
                       fix_offset(r, dx, dy, (float)A.c_max) <= kFixNodeDe;
    if (!fixed) {
        double* acc = reinterpret_cast<double*>(s_acc);
#pragma unroll 1
        for (int q = 0; q < Q; ++q) {
            const double us = 1.0 / (double)(1 << (fix_shift<N1>(q / N1) + fix_shift<N1>(q % N1)));
            const long long v = s_acc[q * NT + tid];
            acc[q * NT + tid] = (offwin >> q & 1u) ? __longlong_as_double(v)
                                                   : (double)v * (f_unit * us);
        }
        Tr::template finish<N1>(A, acc, NT, tid, node, g);
        return;
    }
    fix_transform<N1>(F, r, dx, dy, f);
    const double two_beta = 2.0 * A.P.beta;
    const double keep = (1.0 - two_beta) * f_unit, eq = two_beta * g.rho;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const double us = 1.0 / (double)(1 << (fix_shift<N1>(q / N1) + fix_shift<N1>(q % N1)));
        A.out.f[q * A.plane + node] = fma((double)f[q], keep * us, eq * (L.w[q / N1] * L.w[q % N1]));
    }
    A.out.ux[node] = g.nux;
    A.out.uy[node] = g.nuy;
    A.out.st[node] = g.nst;
}

// One CTA per 32 x TY tile as k_step_staged (whose comments on the window,
// the passes and the fallbacks hold here), the contractions in fixed point.
// Tiles out of its range go to A.redo_list.
template <class Tr, int TY, int N1>
__global__ void __launch_bounds__(32 * TY, TY >= 8 ? 1 : 2) k_step_fixed(StagedArgs<double> A) {
    constexpr int TX = 32, NT = TX * TY, Q = N1 * N1;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int WN = A.ww * A.wh;
    int4* s_h = reinterpret_cast<int4*>(smem_raw);                 // [N1][WN] high limbs
    int4* s_l = s_h + (size_t)N1 * WN;                             // [N1][WN] low limbs
    long long* s_acc = reinterpret_cast<long long*>(s_l + (size_t)N1 * WN);  // [Q][NT]
    int2* s_gy = reinterpret_cast<int2*>(s_acc + (size_t)Q * NT);  // [Q][NT] y-map of the pass
    __shared__ float s_red[4][NT / 32];
    __shared__ long long s_item;
    __shared__ unsigned long long s_passes, s_nc, s_np, s_fb;
    __shared__ unsigned int s_max;
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
    const int lxi = tid % TX, lyi = tid / TX;
    const double dt57 = A.P.dt * kFixDisplacement;
    const unsigned long long t_begin = (A.work_counter && tid == 0) ? pond_globaltimer() : 0ull;

    long long item = blockIdx.x;
    for (;;) {
        if (A.work_counter) {
            __syncthreads();
            if (tid == 0) s_item = (long long)atomicAdd(A.work_counter, 1u);
            __syncthreads();
            item = s_item;
        }
        if (item >= A.n_tiles) break;

        int g = 0;
        if (A.n_grids > 1) {
            int lo = 0, hi = A.n_grids - 1;  // largest g with prefix[g] <= item
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (A.tile_prefix[mid] <= item) lo = mid; else hi = mid - 1;
            }
            g = lo;
        }
        const GridDesc G = A.grids[g];
        const long long t = item - A.tile_prefix[g];
        const int tiles_x = (G.iw + TX - 1) / TX;
        const int tx0 = G.ix0 + (int)(t % tiles_x) * TX;
        const int ty0 = G.iy0 + (int)(t / tiles_x) * TY;
        const int X = tx0 + lxi, Y = ty0 + lyi;
        const bool valid = X < G.ix0 + G.iw && Y < G.iy0 + G.ih;
        const long long base = G.offset;
        const long long node = base + (long long)Y * G.nx + X;
        const long long rnode = base + (long long)min(ty0 + TY / 2, G.iy0 + G.ih - 1) * G.nx +
                                min(tx0 + TX / 2, G.ix0 + G.iw - 1);
        const double rux = A.in.ux[rnode], ruy = A.in.uy[rnode], rst = A.in.st[rnode];

        // the tile's scale: the exponent of the centre node's largest scaled
        // population (each warp finds it for itself)
        const int lane = tid & 31;
        unsigned mh = 0u;
        if (lane < Q) {
            const int s = fix_shift<N1>(lane / N1) + fix_shift<N1>(lane % N1);
            const double v = fabs(A.in.f[(long long)lane * A.plane + rnode]) * (double)(1 << s);
            mh = (unsigned)__double2hiint(v);
        }
        mh = __reduce_max_sync(FULL, mh);
        const int me = (int)(mh >> 20) - 1023;    // M in [2^me, 2^(me + 1))
        const int rexp = me + 4;                  // R = 2^rexp
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
            const float de = fmaf((float)A.c_max, fabsf((float)(rst - pg.st)),
                                  fmaxf(fabsf((float)(rux - pg.ux)), fabsf((float)(ruy - pg.uy))));
            in_range = in_range && de <= kFixTileDe * (float)pg.st;
        }
        staged_block_minmax4<Tr, NT>(vxlo, vxhi, vylo, vyhi, s_red);

        // staged window in unwrapped grid coordinates (departure = x - v dt)
        const float m = A.margin;
        const float fdt = (float)A.P.dt;
        const float bxl = fminf(fmaxf(vxlo, -1.0e6f), 1.0e6f), bxh = fminf(fmaxf(vxhi, -1.0e6f), 1.0e6f);
        const float byl = fminf(fmaxf(vylo, -1.0e6f), 1.0e6f), byh = fminf(fmaxf(vyhi, -1.0e6f), 1.0e6f);
        const int wx0 = (int)floorf((float)tx0 - bxh * fdt - m) - 1;
        const int wx1 = (int)floorf((float)(tx0 + TX - 1) - bxl * fdt + m) + 2;
        const int wy0 = (int)floorf((float)ty0 - byh * fdt - m) - 1;
        const int wy1 = (int)floorf((float)(ty0 + TY - 1) - byl * fdt + m) + 2;
        const bool fin = isfinite(vxlo) && isfinite(vxhi) && isfinite(vylo) && isfinite(vyhi) &&
                         vxlo > -1.0e6f && vxhi < 1.0e6f && vylo > -1.0e6f && vyhi < 1.0e6f;
        const int ww = fin ? max(1, min(wx1 - wx0 + 1, A.ww)) : 1;
        const int wh = fin ? max(1, min(wy1 - wy0 + 1, A.wh)) : 1;
        // (displacements in the fixed-point range of fix_departure)
        in_range = in_range && fin &&
                   fmaxf(fmaxf(fabsf(vxlo), fabsf(vxhi)), fmaxf(fabsf(vylo), fabsf(vyhi))) * fdt < 400.0f;

        in_range = stage_window_fixed<N1>(A.in, A.plane, G, base, wx0, wy0, ww, wh, WN, rux, ruy,
                                          rst, kFixSource - rexp, s_h, s_l, F,
                                          (float)A.c_max, A.stats, tid, NT) &&
                   in_range;
        if (__syncthreads_or(!in_range)) {  // also: the window is staged
            if (tid == 0) A.redo_list[atomicAdd(A.redo_count, 1u)] = (unsigned)item;
            if (!A.work_counter) break;
            continue;
        }

        // ---------------------------------------------------- pass loop
        const double f_unit = pow2d(rexp - kFixPop);  // a scaled population's unit
        pg.nux = pg.ux;
        pg.nuy = pg.uy;
        pg.nst = pg.st;
        pg.rho = 0.0;
        pg.pass = 0;
        pg.flag = 0u;
        unsigned int fallbacks = 0u;
        unsigned int offwin = 0u;  // populations of the pass read from global memory
        bool done = !valid;
        while (!done) {
            // target gauge of this pass, and its offsets from lambda_r
            const double st = pg.st, ux = pg.ux, uy = pg.uy;
            const double inv = kFixOne / st;
            const long long rt = __double2ll_rn((rst - st) * inv);
            const long long dxt = __double2ll_rn((rux - ux) * inv);
            const long long dyt = __double2ll_rn((ruy - uy) * inv);
            const bool near_r = fix_offset(rt, dxt, dyt, (float)A.c_max) <= kFixNodeDe;
            const Fix Rt = fix_split(rt);
            // y-map r -> lambda of the pass, and the y-stencils: top row in
            // the window and weights
            int top[N1];
            Fix ly[N1][4];
            {
                Fix de[N1];
#pragma unroll
                for (int b = 0; b < N1; ++b) de[b] = fix_split(dyt + fix_mul(F.c[b], Rt));
#pragma unroll
                for (int l = 0; l < N1; ++l) {
#pragma unroll
                    for (int b = 0; b < N1; ++b) {
                        const Fix gw = fix_gauge<N1>(F, l, b, de[b]);
                        s_gy[(N1 * l + b) * NT + tid] = make_int2(gw.h, gw.l);
                    }
                    const double d = -fma(st, L.c[l], uy) * dt57;
                    top[l] = Y - wy0 - 1 + fix_departure(__double2ll_rn(d), ly[l]);
                    if (!(near_r && fabs(d) < 500.0 * kFixDisplacement && top[l] >= 0 &&
                          top[l] + 3 < wh))
                        top[l] = -1;
                }
            }
            Fix dex[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) dex[a] = fix_split(dxt + fix_mul(F.c[a], Rt));
            int lo = 0x7fffffff, hi = -1;
#pragma unroll
            for (int l = 0; l < N1; ++l)
                if (top[l] >= 0) {
                    lo = min(lo, top[l]);
                    hi = max(hi, top[l] + 3);
                }
            double m0 = 0, m1 = 0, m2 = 0, m3 = 0;
            offwin = 0u;
#pragma unroll 1
            for (int k = 0; k < N1; ++k) {
                const double ck = L.c[k];
                const bool outer = k == 0 || k == N1 - 1;
                Fix lx[4];
                const double d = -fma(st, ck, ux) * dt57;
                const int col = X - wx0 - 1 + fix_departure(__double2ll_rn(d), lx);
                if (!(fabs(d) < 500.0 * kFixDisplacement && col >= 0 && col + 3 < ww) || hi < 0) {
                    offwin |= ((1u << N1) - 1u) << (N1 * k);
                    continue;
                }
                // the row's weights, cxa[jx][a] = lx[jx] G_x(r -> lambda)[k][a]
                Fix cxa[4][N1];
#pragma unroll
                for (int a = 0; a < N1; ++a) {
                    const Fix gw = fix_gauge<N1>(F, k, a, dex[a]);
#pragma unroll
                    for (int jx = 0; jx < 4; ++jx) cxa[jx][a] = fix_split(fix_mul(lx[jx], gw));
                }
                // the sweep over the rows of the union of the y-stencils keeps
                // the last four rows' P; population l takes its rows when the
                // sweep reaches its last one
                Fix Pb[4][N1];
                long long e_in = 0, e_out = 0, y_in = 0, y_out = 0;
#pragma unroll 1
                for (int y = lo; y <= hi; ++y) {
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
                    for (int b = 0; b < N1; ++b) Pb[3][b] = fix_split(fix_sum<0>(h[b], mm[b]));
#pragma unroll
                    for (int l = 0; l < N1; ++l) {
                        if (top[l] < 0 || y != top[l] + 3) continue;
                        long long fh = 0, fm = 0;
#pragma unroll
                        for (int b = 0; b < N1; ++b) {
                            long long zh = 0, zm = 0;
#pragma unroll
                            for (int j = 0; j < 4; ++j) fix_mad(ly[l][j], Pb[j][b].h, Pb[j][b].l, zh, zm);
                            const Fix z = fix_split(fix_sum<1>(zh, zm));
                            const int2 gw = s_gy[(N1 * l + b) * NT + tid];
                            fix_mad(Fix{gw.x, gw.y}, z.h, z.l, fh, fm);
                        }
                        const long long f = fix_sum<1>(fh, fm);
                        s_acc[(N1 * k + l) * NT + tid] = f;
                        if (fix_shift<N1>(l)) {
                            e_out += f;
                            y_out += l == 0 ? -f : f;
                        } else {
                            e_in += f;
                            if (N1 == 4) y_in += l == 1 ? -f : f;
                        }
                    }
                }
#pragma unroll
                for (int l = 0; l < N1; ++l)
                    if (top[l] < 0) offwin |= 1u << (N1 * k + l);
                // sums over l of f, c_l f and c_l^2 f
                constexpr double dn = 1.0 / (double)(1 << fix_shift<N1>(0));
                const double u = f_unit * (outer ? dn : 1.0);
                const double si = (double)e_in * u, so = (double)e_out * (u * dn);
                const double c_in = N1 == 4 ? L.c[2] : 0.0, c_out = L.c[N1 - 1];
                const double s = si + so;
                m0 += s;
                m1 = fma(ck, s, m1);
                m2 = fma(c_out, (double)y_out * (u * dn), m2);
                if (N1 == 4) m2 = fma(c_in, (double)y_in * u, m2);
                m3 = fma(ck * ck, s, m3);
                m3 = fma(c_out * c_out, so, m3);
                if (N1 == 4) m3 = fma(c_in * c_in, si, m3);
            }
            // populations whose stencil leaves the staged window, from global
            // memory; kept as doubles in their slots
            for (unsigned int left = offwin; left; left &= left - 1) {
                const int q = __ffs(left) - 1;
                const int k = q / N1, l = q - N1 * k;
                const double acc = staged_fallback<Tr, N1>(A, G, base, X, Y, k, l, ux, uy, st);
                ++fallbacks;
                s_acc[q * NT + tid] = __double_as_longlong(acc);
                const double ck = L.c[k], cl = L.c[l];
                m0 += acc;
                m1 = fma(ck, acc, m1);
                m2 = fma(cl, acc, m2);
                m3 = fma(fma(ck, ck, cl * cl), acc, m3);
            }
            done = Tr::update(A.P, pg, m0, m1, m2, m3);
        }
        __syncwarp();
        unsigned passes = 0u;
        if (valid && POND_INDEX_OK(node >= base && node < base + (long long)G.nx * G.ny, A.stats)) {
            finish_fixed<Tr, N1>(A, F, s_acc, NT, tid, node, pg, offwin, f_unit);
            if (A.iters) A.iters[node] = pg.pass;
            passes = (unsigned)pg.pass;
            if (pg.flag & 1u) atomicAdd(&s_nc, 1ull);
            if (pg.flag & 2u) atomicAdd(&s_np, 1ull);
            if (fallbacks) atomicAdd(&s_fb, (unsigned long long)fallbacks);
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

}  // namespace pond
