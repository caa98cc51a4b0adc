// pond_adjoint.cu -- vector-Jacobian product of one PonD step (FP64).
//
// The step maps the input state S = {f_s, lambda_s} to, at every node x,
//   lambda*(x) = the fixed point of Phi(lambda) = M(A(lambda), lambda)
//                (Eqs. conservation_*, density..T),
//   A*(x)      = A(lambda*), A_q(lambda) = sum_j a_j(lambda) (G_{lambda_j}^{lambda} f_j)_q
//                (Eqs. advection, interpolation, transform),
//   f_out      = A* + 2 beta (rho W - A*)   (Eq. postcollision),  gauge_out = lambda*.
// The fixed point is differentiated implicitly.  In the parametrisation
// lambda = (u_x, u_y, s = sqrt(theta)) the moment map M has, at the fixed point,
// dM/dlambda = I (its explicit gauge dependence cancels there), so
// I - dPhi/dlambda = -M_A A_lambda, a 3 x 3 matrix per node, with
//   M_A[u_x][q] = s c_k / rho,  M_A[u_y][q] = s c_l / rho,
//   M_A[s][q]   = s (|c_q|^2 - 2 T_L) / (4 rho T_L).
// Given cotangents (fbar, lambdabar) of the output:
//   Abar   = (1 - 2 beta) fbar + 2 beta (W . fbar) 1,   betabar = sum 2 (rho W - A) fbar
//   g      = A_lambda^T Abar + lambdabar
//   mu     = (I - dPhi/dlambda)^{-T} g = -(M_A A_lambda)^{-T} g
//   w      = Abar + M_A^T mu
//   Sbar   = A_S^T w   (transpose of the reconstruction: onto the source
//                       populations f_j and source gauges lambda_j)
// The seed gauge gets no gradient: the limit does not depend on it.
//
// Phase A forms A*, the JVP A_lambda in three directions, the 3 x 3 solve
// and w.  Contexts on the staged forward kernel run it staged, the sources
// staged per tile in a reference gauge and one thread per target node
// (k_adjoint_jvp_fixed in fixed point, k_adjoint_jvp_staged in FP64 for the
// tiles out of its range, then k_adjoint_epilogue); contexts on the direct
// kernels run k_adjoint_targets (one warp per target node, lane = population).
// Phase B is the transpose: the staged contexts scatter each target's cotangent
// over its stencils in fixed point (k_adjoint_scatter, whole-number sums in
// shared memory, so the order of the additions does not matter and the result
// is deterministic, then k_adjoint_reduce), and gather over the targets of the
// tiles out of range (k_adjoint_sources_t: one warp per source node, per target
// the hit set K x L); the direct contexts gather per population
// (k_adjoint_sources).
#include <cmath>

#include "pond_device.cuh"
#include "pond_fixed.cuh"

namespace pond {

// Lattice constants of the adjoint kernels, slot lattice_slot(n1).
__constant__ Lattice c_La[2];
__constant__ LatticeFix c_Lafix[2], c_Lafix1[2];  // scaled, and not

cudaError_t upload_lattice_adjoint() {
    const Lattice L[2] = {make_lattice(POND_D2Q16), make_lattice(POND_D2Q9)};
    const LatticeFix F[2] = {make_lattice_fix(L[0]), make_lattice_fix(L[1])};
    cudaError_t e = cudaMemcpyToSymbol(c_La, L, sizeof(L));
    const LatticeFix F1[2] = {make_lattice_fix(L[0], false), make_lattice_fix(L[1], false)};
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_Lafix, F, sizeof(F));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_Lafix1, F1, sizeof(F1));
    return e;
}

struct ScatterTile;
struct AdjointScratch {
    int64_t N = 0;
    StateBuf<double> fwd{};   // forward step output: gauge = lambda*
    double* w = nullptr;      // [Q][N] (allocated for 16)
    int32_t* iters = nullptr;
    DevStats* stats = nullptr;
    double* beta_bar = nullptr;  // device accumulator
    double* minmax = nullptr;    // 6 doubles: min/max of ux*, uy*, s*
    int2* org = nullptr;         // [16][N] stencil origin of (q, t), relative to t
    double* lw = nullptr;        // [16][N][8] cubic weights of (q, t): x 0..3, y 0..3
    // staged contexts keep org and lw per speed and direction instead
    int* org1 = nullptr;         // [2][4][N]
    double* lw1 = nullptr;       // [2][4][N][4]
    unsigned int* redo = nullptr;  // {count, tiles, marks} left to the FP64 kernels (phase A, then B)
    double* win = nullptr;         // phase B: the tiles' windows of f_bar
    ScatterTile* tiles = nullptr;
    double* inv_st = nullptr;    // [N] 1 / s* at every target
    double* jvp = nullptr;       // [4][16][N] A*, dA/du_x, dA/du_y, dA/ds (staged phase A)
    double* nu_dev = nullptr;    // nu cotangent of calls with nu_bar_accum == NULL
    double host_minmax[6];
};

// Cubic Lagrange weights on 0..3 and their derivatives at t (App. C).
__device__ __forceinline__ void lagrange4_d(double t, double l[4], double dl[4]) {
    const double a = t, b = t - 1.0, c = t - 2.0, d = t - 3.0;
    l[0] = -(b * c * d) / 6.0;
    l[1] = (a * c * d) / 2.0;
    l[2] = -(a * b * d) / 2.0;
    l[3] = (a * b * c) / 6.0;
    dl[0] = -(c * d + b * d + b * c) / 6.0;
    dl[1] = (c * d + a * d + a * c) / 2.0;
    dl[2] = -(b * d + a * d + a * b) / 2.0;
    dl[3] = (b * c + a * c + a * b) / 6.0;
}

// L_k(c_a + de) and its derivative in xi, from the Taylor coefficients.
__device__ __forceinline__ void lag_taylor(const Lattice& L, int k, int a, double de, double& g,
                                          double& gd) {
    const double d1 = L.d1[k][a], d2 = L.d2[k][a], d3 = L.d3[k];
    g = fma(fma(fma(d3, de, d2), de, d1), de, (k == a) ? 1.0 : 0.0);
    gd = fma(fma(3.0 * d3, de, 2.0 * d2), de, d1);
}

struct AdjArgs {
    StateBuf<double> in;     // input state S
    const double* ux_s;      // lambda* (forward output gauge)
    const double* uy_s;
    const double* st_s;
    const double* fbar;      // [Q][N]
    const double* gbar;      // [3][N]  (u_x, u_y, T)
    double* w;               // [Q][N]
    double* fbar_in;         // [Q][N]
    double* gbar_in;         // [3][N]
    double* beta_bar;
    // per (population, target), written by the target kernel for the gather:
    // stencil origin relative to the target, cubic weights, and 1 / s*
    // (staged contexts: per speed and direction)
    int2* org;
    double* lw;
    int *org_x, *org_y;      // [n1][N]
    double *lw_x, *lw_y;     // [n1][N][4]
    double* inv_st;
    int nx, ny;
    long long N;
    double beta, dt, T_L;
    double vlo_x[4], vhi_x[4], vlo_y[4], vhi_y[4];  // particle-velocity bounds per speed
};

constexpr int ADJ_WARPS = 4;
constexpr int ADJ_TY = 8;  // tiles of targets of the staged kernels: 32 x 8

template <int N1>
__global__ void __launch_bounds__(ADJ_WARPS * 32, 2) k_adjoint_targets(AdjArgs A) {
    constexpr int Q = N1 * N1;
    const Lattice& L = c_La[lattice_slot(N1)];
    const int lane = threadIdx.x & 31;
    const long long node = (long long)blockIdx.x * ADJ_WARPS + (threadIdx.x >> 5);
    if (node >= A.N) return;  // warp-uniform
    const int X = (int)(node % A.nx), Y = (int)(node / A.nx);
    // lane = (population q, half); on D2Q9 lanes with q >= 9 hold no
    // population: they contribute zeros to the 16-lane sums and read nothing
    const int q = lane & 15, half = lane >> 4;
    const bool act = q < Q;
    const int qa = act ? q : 0, k = qa / N1, l = qa % N1;
    const double ck = act ? L.c[k] : 0.0, cl = act ? L.c[l] : 0.0;
    const double ux = A.ux_s[node], uy = A.uy_s[node], st = A.st_s[node];
    const double inv = 1.0 / st;

    // departure of population q at lambda*
    const double vx = fma(st, ck, ux), vy = fma(st, cl, uy);
    const double depx = (double)X - vx * A.dt, depy = (double)Y - vy * A.dt;
    const double flx = floor(depx), fly = floor(depy);
    double lx[4], dlx[4], ly[4], dly[4];
    lagrange4_d(depx - flx + 1.0, lx, dlx);
    lagrange4_d(depy - fly + 1.0, ly, dly);
    const int x0 = wrap_idx((long long)flx - 1, A.nx);
    const int y0 = wrap_idx((long long)fly - 1, A.ny);
    // what the gather needs of (q, target): the stencil origin relative to
    // the target and the cubic weights; and 1 / s* of the target
    if (act) {
        const long long o = (long long)q * A.N + node;
        double2* pw = reinterpret_cast<double2*>(A.lw + 8 * o + 4 * half);
        if (half == 0) {
            A.org[o] = make_int2((int)((long long)flx - 1 - X), (int)((long long)fly - 1 - Y));
            pw[0] = make_double2(lx[0], lx[1]);
            pw[1] = make_double2(lx[2], lx[3]);
        } else {
            pw[0] = make_double2(ly[0], ly[1]);
            pw[1] = make_double2(ly[2], ly[3]);
        }
    }
    if (lane == 0) A.inv_st[node] = inv;

    double Aq = 0.0, dAux = 0.0, dAuy = 0.0, dAst = 0.0;
    if (act) {
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
        const int jy = 2 * half + jj;
        const double wy = half ? ly[2 + jj] : ly[jj];
        const double dwy = half ? dly[2 + jj] : dly[jj];
        const int sy = wrap_inc(y0, jy, A.ny);
#pragma unroll
        for (int jx = 0; jx < 4; ++jx) {
            const int sx = wrap_inc(x0, jx, A.nx);
            const long long s = (long long)sy * A.nx + sx;
            const double r = fma(A.in.st[s], inv, -1.0);
            const double dx = (A.in.ux[s] - ux) * inv;
            const double dy = (A.in.uy[s] - uy) * inv;
            double gx[N1], gdx[N1], gy[N1], gdy[N1], xix[N1], xiy[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const double ex = fma(L.c[a], r, dx), ey = fma(L.c[a], r, dy);
                xix[a] = L.c[a] + ex;
                xiy[a] = L.c[a] + ey;
                lag_taylor(L, k, a, ex, gx[a], gdx[a]);
                lag_taylor(L, l, a, ey, gy[a], gdy[a]);
            }
            double g = 0.0, gux = 0.0, guy = 0.0, gst = 0.0;
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                double h = 0.0, hp = 0.0, hq = 0.0;
#pragma unroll
                for (int b = 0; b < N1; ++b) {
                    const double fv = A.in.f[(long long)(N1 * a + b) * A.N + s];
                    h = fma(gy[b], fv, h);
                    hp = fma(gdy[b], fv, hp);
                    hq = fma(gdy[b] * xiy[b], fv, hq);
                }
                g = fma(gx[a], h, g);
                gux = fma(gdx[a], h, gux);
                guy = fma(gx[a], hp, guy);
                gst = fma(gdx[a] * xix[a], h, fma(gx[a], hq, gst));
            }
            // d xi / d(target u) = -1/s ; d xi / d(target s) = -xi / s
            gux *= -inv;
            guy *= -inv;
            gst *= -inv;
            const double wx = lx[jx], dwx = dlx[jx];
            const double a_w = wx * wy;
            // d t / d u = -dt ; d t / d s = -c dt
            const double da_ux = -A.dt * dwx * wy;
            const double da_uy = -A.dt * wx * dwy;
            const double da_st = -A.dt * (ck * dwx * wy + cl * wx * dwy);
            Aq = fma(a_w, g, Aq);
            dAux = fma(a_w, gux, fma(da_ux, g, dAux));
            dAuy = fma(a_w, guy, fma(da_uy, g, dAuy));
            dAst = fma(a_w, gst, fma(da_st, g, dAst));
        }
    }
    }
    Aq += __shfl_xor_sync(0xffffffffu, Aq, 16);
    dAux += __shfl_xor_sync(0xffffffffu, dAux, 16);
    dAuy += __shfl_xor_sync(0xffffffffu, dAuy, 16);
    dAst += __shfl_xor_sync(0xffffffffu, dAst, 16);

    auto sum16 = [](double v) {
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    const double Wq = act ? L.w[k] * L.w[l] : 0.0;
    const double fb = act ? A.fbar[(long long)q * A.N + node] : 0.0;
    const double rho = sum16(Aq);
    const double wf = sum16(Wq * fb);
    const double Abar = (1.0 - 2.0 * A.beta) * fb + 2.0 * A.beta * wf;
    const double bb = sum16(2.0 * (rho * Wq - Aq) * fb);

    // moment-map rows at the fixed point
    const double c2 = ck * ck + cl * cl;
    const double mux = st * ck / rho, muy = st * cl / rho;
    const double mst = st * (c2 - 2.0 * A.T_L) / (4.0 * rho * A.T_L);
    double J[3][3];
    J[0][0] = sum16(mux * dAux);
    J[0][1] = sum16(mux * dAuy);
    J[0][2] = sum16(mux * dAst);
    J[1][0] = sum16(muy * dAux);
    J[1][1] = sum16(muy * dAuy);
    J[1][2] = sum16(muy * dAst);
    J[2][0] = sum16(mst * dAux);
    J[2][1] = sum16(mst * dAuy);
    J[2][2] = sum16(mst * dAst);
    // output-gauge cotangent, T -> s: dL/ds = dL/dT * 2 s T_L
    double g0 = sum16(Abar * dAux) + A.gbar[node];
    double g1 = sum16(Abar * dAuy) + A.gbar[A.N + node];
    double g2 = sum16(Abar * dAst) + A.gbar[2 * A.N + node] * 2.0 * st * A.T_L;
    // solve J^T mu = -g (Cramer's rule on the transpose)
    const double a00 = J[0][0], a01 = J[1][0], a02 = J[2][0];
    const double a10 = J[0][1], a11 = J[1][1], a12 = J[2][1];
    const double a20 = J[0][2], a21 = J[1][2], a22 = J[2][2];
    const double det = a00 * (a11 * a22 - a12 * a21) - a01 * (a10 * a22 - a12 * a20) +
                       a02 * (a10 * a21 - a11 * a20);
    const double idet = 1.0 / det;
    const double r0 = -g0, r1 = -g1, r2 = -g2;
    const double mu0 = (r0 * (a11 * a22 - a12 * a21) - a01 * (r1 * a22 - a12 * r2) +
                        a02 * (r1 * a21 - a11 * r2)) * idet;
    const double mu1 = (a00 * (r1 * a22 - a12 * r2) - r0 * (a10 * a22 - a12 * a20) +
                        a02 * (a10 * r2 - r1 * a20)) * idet;
    const double mu2 = (a00 * (a11 * r2 - r1 * a21) - a01 * (a10 * r2 - r1 * a20) +
                        r0 * (a10 * a21 - a11 * a20)) * idet;
    const double wq = Abar + mux * mu0 + muy * mu1 + mst * mu2;
    if (half == 0 && act) A.w[(long long)q * A.N + node] = wq;
    if (lane == 0) atomicAdd(A.beta_bar, bb);
}

// Warp reduce-scatter of 16 per-lane partial sums by recursive halving: at
// distance 2h each lane keeps the h slots its lane bit selects and adds its
// partner's copy of them.  Returns, in lanes 2p and 2p + 1, the warp total of
// slot p (16 additions per lane, against 16 x 5 for a full all-reduce).
__device__ __forceinline__ double warp_reduce_scatter16(double (&v)[16], int lane) {
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = (lane & (2 * h)) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double keep = up ? v[i + h] : v[i];
            const double send = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Transpose of the reconstruction, gathered at each source node.
template <int N1>
__global__ void __launch_bounds__(ADJ_WARPS * 32, 2) k_adjoint_sources(AdjArgs A) {
    constexpr int Q = N1 * N1;
    const Lattice& L = c_La[lattice_slot(N1)];
    const int lane = threadIdx.x & 31;
    const long long src = (long long)blockIdx.x * ADJ_WARPS + (threadIdx.x >> 5);
    if (src >= A.N) return;  // warp-uniform
    const int JX = (int)(src % A.nx), JY = (int)(src / A.nx);
    // lane = (population q, half); on D2Q9 lanes with q >= 9 hold no
    // population: they contribute zeros to the 16-lane sums and read nothing
    const int q = lane & 15, half = lane >> 4;
    const bool act = q < Q;
    const int qa = act ? q : 0, k = qa / N1, l = qa % N1;
    double fj[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) fj[i] = A.in.f[(long long)i * A.N + src];
    const double uxj = A.in.ux[src], uyj = A.in.uy[src], stj = A.in.st[src];

    double fb[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) fb[i] = 0.0;
    double bux = 0.0, buy = 0.0, bst = 0.0;

    // candidate targets: J is in the stencil of the target at x when
    // floor(x - v dt) is in [J - 2, J + 1], i.e. x in [J - 2 + v dt, J + 2 + v dt);
    // over v in [vlo, vhi] the integers x from ceil(J - 2 + vlo dt) to
    // ceil(J + 2 + vhi dt) - 1, widened by a rounding margin (the exact test
    // below decides).  ceil(J + a) = J + ceil(a) for integer J, so the bounds
    // are formed relative to J.
    const double ex = 1e-9 * (1.0 + fabs(A.vlo_x[k]) + fabs(A.vhi_x[k])) * A.dt;
    const double ey = 1e-9 * (1.0 + fabs(A.vlo_y[l]) + fabs(A.vhi_y[l])) * A.dt;
    const int xlo = JX + (int)ceil(-2.0 + A.vlo_x[k] * A.dt - ex);
    const int xhi = JX + (int)ceil(2.0 + A.vhi_x[k] * A.dt + ex) - 1;
    const int ylo = JY + (int)ceil(-2.0 + A.vlo_y[l] * A.dt - ey);
    const int yhi = JY + (int)ceil(2.0 + A.vhi_y[l] * A.dt + ey) - 1;
    for (int yy = ylo + half; act && yy <= yhi; yy += 2) {
        const int ty = wrap_idx(yy, A.ny);
        for (int xx = xlo; xx <= xhi; ++xx) {
            const int tx = wrap_idx(xx, A.nx);
            const long long t = (long long)ty * A.nx + tx;
            // the target's stencil origin for population q, as the target
            // kernel found it (at the target's own, wrapped position)
            const long long o = (long long)q * A.N + t;
            const int2 og = A.org[o];
            const int jx = JX - (xx + og.x), jy = JY - (yy + og.y);
            if (jx < 0 || jx > 3 || jy < 0 || jy > 3) continue;
            const double wgt = A.lw[8 * o + jx] * A.lw[8 * o + 4 + jy];
            const double coef = A.w[o] * wgt;
            const double ux = A.ux_s[t], uy = A.uy_s[t];
            const double inv = A.inv_st[t];
            const double r = fma(stj, inv, -1.0);
            const double dx = (uxj - ux) * inv, dy = (uyj - uy) * inv;
            double gx[N1], gdx[N1], gy[N1], gdy[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                lag_taylor(L, k, a, fma(L.c[a], r, dx), gx[a], gdx[a]);
                lag_taylor(L, l, a, fma(L.c[a], r, dy), gy[a], gdy[a]);
            }
            double sux = 0.0, suy = 0.0, sst = 0.0;
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const double cgx = coef * gx[a];
                double h = 0.0, hp = 0.0, hq = 0.0;
#pragma unroll
                for (int b = 0; b < N1; ++b) {
                    fb[N1 * a + b] = fma(cgx, gy[b], fb[N1 * a + b]);
                    const double fv = fj[N1 * a + b];
                    h = fma(gy[b], fv, h);
                    hp = fma(gdy[b], fv, hp);
                    hq = fma(gdy[b] * L.c[b], fv, hq);
                }
                sux = fma(gdx[a], h, sux);
                suy = fma(gx[a], hp, suy);
                sst = fma(gdx[a] * L.c[a], h, fma(gx[a], hq, sst));
            }
            // d xi / d(source u) = 1/s ; d xi / d(source s) = c / s
            const double ci = coef * inv;
            bux = fma(ci, sux, bux);
            buy = fma(ci, suy, buy);
            bst = fma(ci, sst, bst);
        }
    }
    // reduce over the warp (all populations and both halves): lanes 2p and
    // 2p + 1 get population p's total, every lane the gauge cotangents
    double v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = i < Q ? fb[i] : 0.0;
    const double tot = warp_reduce_scatter16(v, lane);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        bux += __shfl_xor_sync(0xffffffffu, bux, o);
        buy += __shfl_xor_sync(0xffffffffu, buy, o);
        bst += __shfl_xor_sync(0xffffffffu, bst, o);
    }
    const int p = lane >> 1;
    if ((lane & 1) == 0 && p < Q) A.fbar_in[(long long)p * A.N + src] = tot;
    if (lane == 1) {
        A.gbar_in[src] = bux;
        A.gbar_in[A.N + src] = buy;
        // s = sqrt(T / T_L): dL/dT = dL/ds / (2 s T_L)
        A.gbar_in[2 * A.N + src] = bst / (2.0 * stj * A.T_L);
    }
}

// The gather of the staged contexts takes the source-gauge derivatives out
// of the hit loop.  G(j -> t) = G(r -> t) G(j -> r) for any fixed r (the matched
// moments determine the populations), so with r held at the source's own
// gauge lambda_j,
//   d/dlambda_j [G(j -> t) f_j]_q = [G(r -> t) dG(j -> r)/dlambda_j f_j]_q,
// and summed over the hits (target t, population q) with their weights,
//   lambda_j_bar = sum_{a,b} h[a][b] (dG(j -> r)/dlambda_j f_j)[a][b],
//   h = sum_hits coef G(j -> t)[q, :]  (= the populations' cotangent f_j_bar).
// At r = lambda_j the map G(j -> r) is the identity and its derivatives are
// the constants L_k'(c_a) = d1[k][a] over s_j (x: d xi/d u = 1/s_j; s:
// d xi/d s = c_a/s_j).  A hit then needs only the two rows of G(j -> t) and a
// rank-one update, about a third of the direct gather's FP64 work.
//
// It is organised by target.  For a source j and a candidate
// target t, population (k, l) hits when j lies in both its x-stencil and its
// y-stencil; the x-stencil's origin depends on k alone and the y-stencil's
// on l alone, so the hits of (j, t) are a product set K x L.  The rows
// G(j -> t)_x[k][.] (k in K) and G_y[l][.] (l in L) are then evaluated once
// per target, not once per hit, and a hit costs its weight and a rank-one
// update.  Each round, every lane of the source's warp takes one candidate
// target and writes its gauge offsets and stencil positions to a
// shared-memory slot, its rows to a job queue and its hits to a hit queue
// (offsets by a warp prefix sum); the warp then evaluates the rows and does
// the hits 32 at a time.  Work per lane thus does not depend on how many
// rows and hits its own target has: the FP64 pipe serves full warps.
constexpr int ADJ_GATHER_WARPS = 2;

struct GatherSlot {
    double gx[4][4];   // G_x(j -> t)[k][a]
    double gy[4][4];   // G_y(j -> t)[l][b]
    double lx[4];      // x-weight of j in the stencil of x-speed k
    double ly[4];      // y-weight of j in the stencil of y-speed l
    double r, dx, dy;  // gauge offsets of j from t (r: s_j / s_t - 1)
    long long t;
    signed char jx[4], jy[4];  // j's position in the x- and y-stencils
};

template <int N1>
__global__ void __launch_bounds__(ADJ_GATHER_WARPS * 32)
k_adjoint_sources_t(AdjArgs A, const unsigned int* __restrict__ left) {
    constexpr int Q = N1 * N1;
    constexpr unsigned FULL = 0xffffffffu;
    // only the targets of the tiles that k_adjoint_scatter left (left: {count,
    // a mark per tile}), added to what its reduction stored
    if (left[0] == 0u) return;
    const int tiles_x = (A.nx + 31) / 32;
    __shared__ GatherSlot s_slot[ADJ_GATHER_WARPS][32];
    __shared__ unsigned short s_hit[ADJ_GATHER_WARPS][32 * Q];
    __shared__ unsigned short s_job[ADJ_GATHER_WARPS][32 * 2 * N1];
    const Lattice& L = c_La[lattice_slot(N1)];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    GatherSlot& my = s_slot[wid][lane];
    for (long long src = (long long)blockIdx.x * ADJ_GATHER_WARPS + wid; src < A.N;
         src += (long long)gridDim.x * ADJ_GATHER_WARPS) {  // warp-uniform
    const int JX = (int)(src % A.nx), JY = (int)(src / A.nx);
    const double uxj = A.in.ux[src], uyj = A.in.uy[src], stj = A.in.st[src];
    unsigned short* hitq = s_hit[wid];
    unsigned short* jobq = s_job[wid];

    // candidate targets: the union over the speeds of the windows of
    // k_adjoint_sources (J in the stencil of the target at x when
    // floor(x - v dt) is in [J - 2, J + 1], v within the speed's bounds)
    int xlo = 0x7fffffff, xhi = -0x7fffffff, ylo = 0x7fffffff, yhi = -0x7fffffff;
#pragma unroll
    for (int i = 0; i < N1; ++i) {
        const double ex = 1e-9 * (1.0 + fabs(A.vlo_x[i]) + fabs(A.vhi_x[i])) * A.dt;
        const double ey = 1e-9 * (1.0 + fabs(A.vlo_y[i]) + fabs(A.vhi_y[i])) * A.dt;
        xlo = min(xlo, (int)ceil(-2.0 + A.vlo_x[i] * A.dt - ex));
        xhi = max(xhi, (int)ceil(2.0 + A.vhi_x[i] * A.dt + ex) - 1);
        ylo = min(ylo, (int)ceil(-2.0 + A.vlo_y[i] * A.dt - ey));
        yhi = max(yhi, (int)ceil(2.0 + A.vhi_y[i] * A.dt + ey) - 1);
    }
    const int wx = xhi - xlo + 1;
    const int nc = wx * (yhi - ylo + 1);

    double fb[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) fb[i] = 0.0;
    for (int c0 = 0; c0 < nc; c0 += 32) {
        // 1. this lane's candidate: its hit set K x L and gauge offsets
        const int c = c0 + lane;
        unsigned kmask = 0u, lmask = 0u;
        const int xx = JX + xlo + c % wx, yy = JY + ylo + c / wx;
        const int wy_ = wrap_near(yy, A.ny), wx_ = wrap_near(xx, A.nx);
        if (c < nc && left[1 + wy_ / ADJ_TY * tiles_x + wx_ / 32] != 0u) {
            const long long t = (long long)wy_ * A.nx + wx_;
#pragma unroll
            for (int i = 0; i < N1; ++i) {
                const int jx = JX - (xx + A.org_x[(long long)i * A.N + t]);
                const int jy = JY - (yy + A.org_y[(long long)i * A.N + t]);
                my.jx[i] = (signed char)jx;
                my.jy[i] = (signed char)jy;
                kmask |= (jx >= 0 && jx <= 3) ? 1u << i : 0u;
                lmask |= (jy >= 0 && jy <= 3) ? 1u << i : 0u;
            }
            if (kmask && lmask) {
                my.t = t;
                const double inv = A.inv_st[t];
                my.r = fma(stj, inv, -1.0);
                my.dx = (uxj - A.ux_s[t]) * inv;
                my.dy = (uyj - A.uy_s[t]) * inv;
            } else {
                kmask = lmask = 0u;
            }
        }
        // 2. the round's row jobs and hits into the warp's queues: one scan
        //    of (jobs << 16 | hits)
        const int nk = __popc(kmask), nl = __popc(lmask);
        const int mine = ((nk + nl) << 16) | (nk * nl);
        int incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += v;
        }
        const int tot = __shfl_sync(FULL, incl, 31);
        const int ex = incl - mine;
        int hoff = ex & 0xffff, joff = ex >> 16;
        const int nhit = tot & 0xffff, njob = tot >> 16;
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            if (!(kmask >> k & 1u)) continue;
            jobq[joff++] = (unsigned short)((lane << 3) | k);
#pragma unroll
            for (int l = 0; l < N1; ++l)
                if (lmask >> l & 1u) hitq[hoff++] = (unsigned short)((lane << 4) | (k << 2) | l);
        }
#pragma unroll
        for (int l = 0; l < N1; ++l)
            if (lmask >> l & 1u) jobq[joff++] = (unsigned short)((lane << 3) | 4 | l);
        __syncwarp();
        // 3. the rows on full warps: G_x[k][.] or G_y[l][.] and the weight
        for (int j = lane; j < njob; j += 32) {
            const unsigned code = jobq[j];
            GatherSlot& g = s_slot[wid][code >> 3];
            const int i = (int)code & 3;
            const bool yrow = (code & 4u) != 0;
            const double base = yrow ? g.dy : g.dx, r = g.r;
            double row[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a)
                row[a] = gauge_poly<N1>(L.d3[i], L.d2[i][a], L.d1[i][a], a == i ? 1.0 : 0.0,
                                        fma(L.c[a], r, base));
            if (yrow) {
                g.ly[i] = A.lw_y[4 * ((long long)i * A.N + g.t) + g.jy[i]];
#pragma unroll
                for (int a = 0; a < N1; ++a) g.gy[i][a] = row[a];
            } else {
                g.lx[i] = A.lw_x[4 * ((long long)i * A.N + g.t) + g.jx[i]];
#pragma unroll
                for (int a = 0; a < N1; ++a) g.gx[i][a] = row[a];
            }
        }
        __syncwarp();
        // 4. the hits on full warps: weight, then the rank-one update
        for (int h = lane; h < nhit; h += 32) {
            const unsigned code = hitq[h];
            const GatherSlot& g = s_slot[wid][code >> 4];
            const int k = (int)(code >> 2) & 3, l = (int)code & 3;
            const double coef = A.w[(long long)(N1 * k + l) * A.N + g.t] * g.lx[k] * g.ly[l];
            double gy[N1];
#pragma unroll
            for (int b = 0; b < N1; ++b) gy[b] = g.gy[l][b];
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const double cgx = coef * g.gx[k][a];
#pragma unroll
                for (int b = 0; b < N1; ++b) fb[N1 * a + b] = fma(cgx, gy[b], fb[N1 * a + b]);
            }
        }
        __syncwarp();  // the slots and the queues are rewritten next round
    }

    // reduce over the warp: lanes 2p and 2p + 1 get population p's total
    double v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = i < Q ? fb[i] : 0.0;
    const double tot = warp_reduce_scatter16(v, lane);
    // the source-gauge cotangent from h = fb, one population per even lane:
    // dg/du_x [k][l] = sum_a d1[k][a] f[a][l] / s_j, dg/du_y [k][l] =
    // sum_b d1[l][b] f[k][b] / s_j, dg/ds the same with c_a, c_b inside
    const int p = lane >> 1;
    double pux = 0.0, puy = 0.0, pst = 0.0;
    if ((lane & 1) == 0 && p < Q) {
        const int kk = p / N1, ll = p % N1;
        double gxu = 0.0, gyu = 0.0, gsx = 0.0, gsy = 0.0;
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            // the source's populations f_j[a][ll] and f_j[kk][a]
            const double fx = A.in.f[(long long)(N1 * a + ll) * A.N + src];
            const double fy = A.in.f[(long long)(N1 * kk + a) * A.N + src];
            gxu = fma(L.d1[kk][a], fx, gxu);
            gsx = fma(L.d1[kk][a] * L.c[a], fx, gsx);
            gyu = fma(L.d1[ll][a], fy, gyu);
            gsy = fma(L.d1[ll][a] * L.c[a], fy, gsy);
        }
        pux = tot * gxu;
        puy = tot * gyu;
        pst = tot * (gsx + gsy);
        A.fbar_in[(long long)p * A.N + src] += tot;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        pux += __shfl_xor_sync(FULL, pux, o);
        puy += __shfl_xor_sync(FULL, puy, o);
        pst += __shfl_xor_sync(FULL, pst, o);
    }
    if (lane == 0) {
        const double is = 1.0 / stj;
        A.gbar_in[src] += pux * is;
        A.gbar_in[A.N + src] += puy * is;
        // s = sqrt(T / T_L): dL/dT = dL/ds / (2 s T_L)
        A.gbar_in[2 * A.N + src] += pst * is / (2.0 * stj * A.T_L);
    }
    }
}

// Bounds {min ux, max ux, min uy, max uy, min s, max s} of a gauge field,
// exact in FP64: a grid-stride pass, warp reductions, and 64-bit integer
// atomics on an order-preserving encoding of the doubles (one per warp and
// value), decoded in place into out6.
__device__ __forceinline__ unsigned long long d2ord(double d) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__global__ void k_minmax3_reset(unsigned long long* o) {
    const int j = threadIdx.x;
    if (j < 6) o[j] = (j & 1) ? 0ull : ~0ull;
}

__global__ void k_minmax3(const double* __restrict__ ux, const double* __restrict__ uy,
                          const double* __restrict__ st, long long N, unsigned long long* o) {
    double v[6] = {1e300, -1e300, 1e300, -1e300, 1e300, -1e300};
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        const double a = ux[i], b = uy[i], c = st[i];
        v[0] = fmin(v[0], a);
        v[1] = fmax(v[1], a);
        v[2] = fmin(v[2], b);
        v[3] = fmax(v[3], b);
        v[4] = fmin(v[4], c);
        v[5] = fmax(v[5], c);
    }
    // warp, then block reduction: one atomic per block and value
    __shared__ double s_b[6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int j = 0; j < 6; ++j) {
                const double u = __shfl_xor_sync(0xffffffffu, v[j], off);
                v[j] = (j & 1) ? fmax(v[j], u) : fmin(v[j], u);
            }
        if (pass == 1) break;
        if (lane == 0)
#pragma unroll
            for (int j = 0; j < 6; ++j) s_b[j][warp] = v[j];
        __syncthreads();
        if (warp != 0) return;
        const bool in = lane < (int)(blockDim.x >> 5);
#pragma unroll
        for (int j = 0; j < 6; ++j) v[j] = in ? s_b[j][lane] : ((j & 1) ? -1e300 : 1e300);
    }
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j & 1) atomicMax(o + j, d2ord(v[j]));
            else atomicMin(o + j, d2ord(v[j]));
        }
}

__global__ void k_minmax3_decode(unsigned long long* o) {
    const int j = threadIdx.x;
    if (j < 6) {
        const unsigned long long u = o[j];
        const unsigned long long b = (u >> 63) ? (u & 0x7fffffffffffffffull) : ~u;
        reinterpret_cast<double*>(o)[j] = __longlong_as_double((long long)b);
    }
}

cudaError_t launch_minmax3(const double* ux, const double* uy, const double* st, long long N,
                           double* out6, cudaStream_t s) {
    unsigned long long* o = reinterpret_cast<unsigned long long*>(out6);
    k_minmax3_reset<<<1, 32, 0, s>>>(o);
    long long nb = (N + 255) / 256;
    if (nb > 256) nb = 256;
    if (nb < 1) nb = 1;
    k_minmax3<<<(unsigned)nb, 256, 0, s>>>(ux, uy, st, N, o);
    k_minmax3_decode<<<1, 32, 0, s>>>(o);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Phase A in the staged form of the forward step (pond_staged.cuh): the
// sources are re-expressed once per tile in a reference gauge lambda_r (the
// tile's centre node of the input state), g = G(s -> r) f_s, and for each
// target population (k, l)
//   A_q(lambda) = sum_b (I + Ey)[l][b] sum_jy ly[jy] P(jy)[b],
//   P(jy)[b]    = sum_a (I + Ex)[k][a] Fi[a][b],  Fi = sum_jx lx[jx] g(x0 + jx, y0 + jy),
// with Ex, Ey the maps r -> lambda.  Its tangents at lambda* follow term by
// term: the cubic weights move with the departure point (d t / d u = -dt,
// d t / d s = -c dt) and the maps with xi_a = (s_r c_a + u_r - u) / s
// (d xi / d u = -1/s, d xi / d s = -xi / s), so one sweep of the stencil rows
// gives A and its three tangents from the interpolated rows Fi and their
// weight derivatives Fd = sum_jx lx'[jx] g.  About a third of the FP64
// arithmetic of the per-(population, source) form.

struct StagedAdj64 {
    using Real = double;
    using Real4 = Double4;
    template <int N1>
    static __device__ __forceinline__ const Lattice& lat() {
        return c_La[lattice_slot(N1)];
    }
    static __device__ __forceinline__ void load4(const Real4* p, double (&v)[4]) {
        const double2 a = reinterpret_cast<const double2*>(p)[0];
        const double2 b = reinterpret_cast<const double2*>(p)[1];
        v[0] = a.x;
        v[1] = a.y;
        v[2] = b.x;
        v[3] = b.y;
    }
    static __device__ __forceinline__ void store4(Real4* p, const double (&v)[4]) {
        reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
    }
};

// L_k(c_a + de) - [k == a] in correction form, and L_k'(c_a + de).
__device__ __forceinline__ void lag_taylor_e(const Lattice& L, int k, int a, double de, double& e,
                                            double& gd) {
    const double d1 = L.d1[k][a], d2 = L.d2[k][a], d3 = L.d3[k];
    e = fma(fma(d3, de, d2), de, d1) * de;
    gd = fma(fma(3.0 * d3, de, 2.0 * d2), de, d1);
}

// One population's A and tangents in the direct form, read from global
// memory: for a stencil that leaves the staged window.
template <int N1>
__device__ __noinline__ void adj_population_direct(const AdjArgs& A, int X, int Y, int k, int l,
                                                   double ux, double uy, double st,
                                                   double* out4) {
    const Lattice& L = c_La[lattice_slot(N1)];
    const double ck = L.c[k], cl = L.c[l];
    const double inv = 1.0 / st;
    const double vx = fma(st, ck, ux), vy = fma(st, cl, uy);
    const double depx = (double)X - vx * A.dt, depy = (double)Y - vy * A.dt;
    const double flx = floor(depx), fly = floor(depy);
    double lx[4], dlx[4], ly[4], dly[4];
    lagrange4_d(depx - flx + 1.0, lx, dlx);
    lagrange4_d(depy - fly + 1.0, ly, dly);
    const int x0 = wrap_idx((long long)flx - 1, A.nx);
    const int y0 = wrap_idx((long long)fly - 1, A.ny);
    double Aq = 0.0, dAux = 0.0, dAuy = 0.0, dAst = 0.0;
    for (int jy = 0; jy < 4; ++jy) {
        const int sy = wrap_inc(y0, jy, A.ny);
        for (int jx = 0; jx < 4; ++jx) {
            const int sx = wrap_inc(x0, jx, A.nx);
            const long long s = (long long)sy * A.nx + sx;
            const double r = fma(A.in.st[s], inv, -1.0);
            const double dx = (A.in.ux[s] - ux) * inv;
            const double dy = (A.in.uy[s] - uy) * inv;
            double gx[N1], gdx[N1], gy[N1], gdy[N1], xix[N1], xiy[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const double ex = fma(L.c[a], r, dx), ey = fma(L.c[a], r, dy);
                xix[a] = L.c[a] + ex;
                xiy[a] = L.c[a] + ey;
                lag_taylor(L, k, a, ex, gx[a], gdx[a]);
                lag_taylor(L, l, a, ey, gy[a], gdy[a]);
            }
            double g = 0.0, gux = 0.0, guy = 0.0, gst = 0.0;
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                double h = 0.0, hp = 0.0, hq = 0.0;
#pragma unroll
                for (int b = 0; b < N1; ++b) {
                    const double fv = A.in.f[(long long)(N1 * a + b) * A.N + s];
                    h = fma(gy[b], fv, h);
                    hp = fma(gdy[b], fv, hp);
                    hq = fma(gdy[b] * xiy[b], fv, hq);
                }
                g = fma(gx[a], h, g);
                gux = fma(gdx[a], h, gux);
                guy = fma(gx[a], hp, guy);
                gst = fma(gdx[a] * xix[a], h, fma(gx[a], hq, gst));
            }
            gux *= -inv;
            guy *= -inv;
            gst *= -inv;
            const double wx = lx[jx], dwx = dlx[jx], wy = ly[jy], dwy = dly[jy];
            const double a_w = wx * wy;
            const double da_ux = -A.dt * dwx * wy;
            const double da_uy = -A.dt * wx * dwy;
            const double da_st = -A.dt * (ck * dwx * wy + cl * wx * dwy);
            Aq = fma(a_w, g, Aq);
            dAux = fma(a_w, gux, fma(da_ux, g, dAux));
            dAuy = fma(a_w, guy, fma(da_uy, g, dAuy));
            dAst = fma(a_w, gst, fma(da_st, g, dAst));
        }
    }
    out4[0] = Aq;
    out4[1] = dAux;
    out4[2] = dAuy;
    out4[3] = dAst;
}


// Phase A, staged: A*, its tangents at lambda* into jvp[4][Q][N], the
// gather's per-(population, target) stencil origin and weights, and 1 / s*.
template <int N1>
__global__ void __launch_bounds__(32 * ADJ_TY, 1)
k_adjoint_jvp_staged(AdjArgs A, int wwa, int wha, double c_max, double* __restrict__ jvp,
                     const unsigned int* __restrict__ redo) {
    constexpr int TX = 32, NT = TX * ADJ_TY, Q = N1 * N1;
    extern __shared__ __align__(32) unsigned char smem_raw[];
    Double4* s_f = reinterpret_cast<Double4*>(smem_raw);  // [N1][WN]
    __shared__ float s_red[4][NT / 32];
    const Lattice& L = c_La[lattice_slot(N1)];
    const int WN = wwa * wha;
    const int tid = threadIdx.x;
    const int tiles_x = (A.nx + TX - 1) / TX;
    // the tiles that k_adjoint_jvp_fixed left: {count, tiles}
    const unsigned int left = redo[0];
    for (unsigned int it = blockIdx.x; it < left; it += gridDim.x) {
    __syncthreads();  // the last tile's staged rows are done with
    const int tile = (int)redo[1 + it];
    const int tx0 = tile % tiles_x * TX;
    const int ty0 = tile / tiles_x * ADJ_TY;
    const int X = tx0 + tid % TX, Y = ty0 + tid / TX;
    const bool valid = X < A.nx && Y < A.ny;
    const long long node = (long long)Y * A.nx + X;

    // reference gauge: the tile's centre node of the input state
    const long long rnode = (long long)min(ty0 + ADJ_TY / 2, A.ny - 1) * A.nx +
                            min(tx0 + TX / 2, A.nx - 1);
    const double rux = A.in.ux[rnode], ruy = A.in.uy[rnode], rst = A.in.st[rnode];

    double ux = 0.0, uy = 0.0, st = 1.0;
    float vxlo = 3.0e38f, vxhi = -3.0e38f, vylo = 3.0e38f, vyhi = -3.0e38f;
    if (valid) {
        ux = A.ux_s[node];
        uy = A.uy_s[node];
        st = A.st_s[node];
        const float sp = (float)(c_max * st);
        vxlo = (float)ux - sp;
        vxhi = (float)ux + sp;
        vylo = (float)uy - sp;
        vyhi = (float)uy + sp;
    }
    staged_block_minmax4<StagedAdj64, NT>(vxlo, vxhi, vylo, vyhi, s_red);
    const float m = 1.0f, fdt = (float)A.dt;
    const float bxl = fminf(fmaxf(vxlo, -1.0e6f), 1.0e6f), bxh = fminf(fmaxf(vxhi, -1.0e6f), 1.0e6f);
    const float byl = fminf(fmaxf(vylo, -1.0e6f), 1.0e6f), byh = fminf(fmaxf(vyhi, -1.0e6f), 1.0e6f);
    const int wx0 = (int)floorf((float)tx0 - bxh * fdt - m) - 1;
    const int wx1 = (int)floorf((float)(tx0 + TX - 1) - bxl * fdt + m) + 2;
    const int wy0 = (int)floorf((float)ty0 - byh * fdt - m) - 1;
    const int wy1 = (int)floorf((float)(ty0 + ADJ_TY - 1) - byl * fdt + m) + 2;
    const bool fin = isfinite(vxlo) && isfinite(vxhi) && isfinite(vylo) && isfinite(vyhi) &&
                     vxlo > -1.0e6f && vxhi < 1.0e6f && vylo > -1.0e6f && vyhi < 1.0e6f;
    const int ww = fin ? max(1, min(wx1 - wx0 + 1, wwa)) : 1;
    const int wh = fin ? max(1, min(wy1 - wy0 + 1, wha)) : 1;
    GridDesc G;
    G.nx = A.nx;
    G.ny = A.ny;
    G.offset = 0;
    G.ix0 = 0;
    G.iy0 = 0;
    G.iw = A.nx;
    G.ih = A.ny;
    stage_window<StagedAdj64, N1>(A.in, A.N, G, 0, wx0, wy0, ww, wh, WN, rux, ruy, rst, s_f,
                                  nullptr, tid, NT);
    __syncthreads();
    if (!valid) continue;

    const double inv = 1.0 / st;
    A.inv_st[node] = inv;
    // offsets of the maps r -> lambda*
    const double rt = (rst - st) * inv, dxt = (rux - ux) * inv, dyt = (ruy - uy) * inv;
    const double dt = A.dt;
#pragma unroll 1
    for (int k = 0; k < N1; ++k) {
        const double ck = L.c[k];
        const double depx = (double)X - fma(st, ck, ux) * dt;
        const double flx = floor(depx);
        double lx[4], dlx[4];
        lagrange4_d(depx - flx + 1.0, lx, dlx);
        const int col = (int)flx - 1 - wx0;  // flx is the absolute departure floor
        double ex[N1], gdx[N1], gdxx[N1];
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            const double de = fma(L.c[a], rt, dxt);
            lag_taylor_e(L, k, a, de, ex[a], gdx[a]);
            gdxx[a] = gdx[a] * (L.c[a] + de);
        }
        const bool colok = col >= 0 && col + 3 < ww;
        // The y-speeds in pairs (l0, l0 + 1): one sweep over the union of
        // the pair's two y-stencils, so a row both stencils hold is
        // interpolated once.  Each row is taken one component b at a time
        // (Fi, Fd of that column of the staged rows), which keeps the two
        // populations' accumulators in registers; every sum runs in the
        // order of the single-population sweep, so the results are the same.
#pragma unroll 1
        for (int l0 = 0; l0 < N1; l0 += 2) {
            const int np = l0 + 1 < N1 ? 2 : 1;
            double ly[2][4], dly[2][4];
            int top[2] = {0, 0};
            bool in[2] = {false, false};
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (p >= np) break;
                const int l = l0 + p;
                const double depy = (double)Y - fma(st, L.c[l], uy) * dt;
                const double fly = floor(depy);
                lagrange4_d(depy - fly + 1.0, ly[p], dly[p]);
                top[p] = (int)fly - 1 - wy0;
                in[p] = colok && top[p] >= 0 && top[p] + 3 < wh;
                if (l == 0) {
                    A.org_x[(long long)k * A.N + node] = (int)((long long)flx - 1 - X);
                    double2* pw = reinterpret_cast<double2*>(A.lw_x + 4 * ((long long)k * A.N + node));
                    pw[0] = make_double2(lx[0], lx[1]);
                    pw[1] = make_double2(lx[2], lx[3]);
                }
                if (k == 0) {
                    A.org_y[(long long)l * A.N + node] = (int)((long long)fly - 1 - Y);
                    double2* pw = reinterpret_cast<double2*>(A.lw_y + 4 * ((long long)l * A.N + node));
                    pw[0] = make_double2(ly[p][0], ly[p][1]);
                    pw[1] = make_double2(ly[p][2], ly[p][3]);
                }
            }
            double Z[2][N1], Zux[2][N1], Zuy[2][N1], Zs[2][N1];
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int b = 0; b < N1; ++b) Z[p][b] = Zux[p][b] = Zuy[p][b] = Zs[p][b] = 0.0;
            if (in[0] || in[1]) {
                const int r0 = in[0] && in[1] ? min(top[0], top[1]) : (in[0] ? top[0] : top[1]);
                const int r1 = (in[0] && in[1] ? max(top[0], top[1]) : (in[0] ? top[0] : top[1])) + 3;
#pragma unroll 1
                for (int row = r0; row <= r1; ++row) {
                    bool cov[2];
                    double w[2], dw[2];
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        const int j = row - top[p];
                        cov[p] = in[p] && j >= 0 && j < 4;
                        w[p] = j == 0 ? ly[p][0] : j == 1 ? ly[p][1] : j == 2 ? ly[p][2] : ly[p][3];
                        dw[p] = j == 0 ? dly[p][0] : j == 1 ? dly[p][1] : j == 2 ? dly[p][2] : dly[p][3];
                    }
                    if (!cov[0] && !cov[1]) continue;  // a gap between the two stencils
                    // the row's weights in the four accumulators, per population
                    double cwux[2], cwdy[2], cwi[2], cckwux[2], cclwdy[2];
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        cwux[p] = -dt * w[p];
                        cwdy[p] = -dt * dw[p];
                        cwi[p] = -w[p] * inv;
                        cckwux[p] = ck * cwux[p];
                        cclwdy[p] = L.c[l0 + p] * cwdy[p];
                    }
                    const Double4* src = s_f + row * ww + col;
#pragma unroll
                    for (int b = 0; b < N1; ++b) {
                        double Fi[N1], Fd[N1];
#pragma unroll
                        for (int a = 0; a < N1; ++a) Fi[a] = Fd[a] = 0.0;
#pragma unroll
                        for (int jx = 0; jx < 4; ++jx) {
#pragma unroll
                            for (int a = 0; a < N1; ++a) {
                                const double v =
                                    reinterpret_cast<const double*>(src + (size_t)a * WN + jx)[b];
                                Fi[a] = fma(lx[jx], v, Fi[a]);
                                Fd[a] = fma(dlx[jx], v, Fd[a]);
                            }
                        }
                        // the row's contributions: value, and the tangents
                        // through the x-weights (Fd), the x-map (gdx) and
                        // the row weight (dw)
                        // the identity part of the x-map, Fi[k] (k is a
                        // loop variable: taken by selection, in registers)
                        double P = Fi[0], P1 = Fd[0], Pd = 0.0, Pdx = 0.0;
#pragma unroll
                        for (int a = 1; a < N1; ++a) {
                            P = k == a ? Fi[a] : P;
                            P1 = k == a ? Fd[a] : P1;
                        }
#pragma unroll
                        for (int a = 0; a < N1; ++a) {
                            P = fma(ex[a], Fi[a], P);
                            P1 = fma(ex[a], Fd[a], P1);
                            Pd = fma(gdx[a], Fi[a], Pd);
                            Pdx = fma(gdxx[a], Fi[a], Pdx);
                        }
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            if (!cov[p]) continue;
                            Z[p][b] = fma(w[p], P, Z[p][b]);
                            Zux[p][b] = fma(cwux[p], P1, fma(cwi[p], Pd, Zux[p][b]));
                            Zuy[p][b] = fma(cwdy[p], P, Zuy[p][b]);
                            Zs[p][b] = fma(cckwux[p], P1, fma(cwi[p], Pdx, fma(cclwdy[p], P, Zs[p][b])));
                        }
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (p >= np) break;
                const int l = l0 + p;
                const int q = N1 * k + l;
                double R[4];
                if (in[p]) {
                    // the y-map r -> lambda* and its derivatives; its
                    // identity part exactly
                    double Al = 0.0, Axl = 0.0, Ayl = 0.0, Asl = 0.0;
#pragma unroll
                    for (int b = 0; b < N1; ++b) {
                        const bool id = b == l;
                        Al += id ? Z[p][b] : 0.0;
                        Axl += id ? Zux[p][b] : 0.0;
                        Ayl += id ? Zuy[p][b] : 0.0;
                        Asl += id ? Zs[p][b] : 0.0;
                    }
                    double Ae = 0.0, Axe = 0.0, Aye = 0.0, Ase = 0.0, Dy = 0.0, Ds = 0.0;
#pragma unroll
                    for (int b = 0; b < N1; ++b) {
                        const double de = fma(L.c[b], rt, dyt);
                        double ey, gdy;
                        lag_taylor_e(L, l, b, de, ey, gdy);
                        Ae = fma(ey, Z[p][b], Ae);
                        Axe = fma(ey, Zux[p][b], Axe);
                        Aye = fma(ey, Zuy[p][b], Aye);
                        Ase = fma(ey, Zs[p][b], Ase);
                        Dy = fma(gdy, Z[p][b], Dy);
                        Ds = fma(gdy * (L.c[b] + de), Z[p][b], Ds);
                    }
                    R[0] = Al + Ae;
                    R[1] = Axl + Axe;
                    R[2] = fma(-inv, Dy, Ayl + Aye);
                    R[3] = fma(-inv, Ds, Asl + Ase);
                } else {
                    adj_population_direct<N1>(A, X, Y, k, l, ux, uy, st, R);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) jvp[((long long)i * Q + q) * A.N + node] = R[i];
            }
        }
    }
    }
}

// Phase A with its contractions in fixed point (pond_fixed.cuh: the staged
// window, its scale and range, the row sweep).  Each of the sums over a row's
// sources that the three tangents need is one sweep of its own, with its
// weights folded ahead of it,
//   P = sum lx G_x g,  U = sum (-tau lx' G_x - lx G_x') g,
//   S = sum (-c_k tau lx' G_x - lx G_x' xi) g    (tau = s dt; U, S times s),
// so that the sweep's registers are the forward step's.  Per population, with
// Z = sum_j ly P, D = sum_j ly' P,
//   A = G_y Z,  dA/du_x = G_y sum ly U / s,  dA/du_y = -dt G_y D - G_y' Z / s,
//   dA/ds = (G_y sum ly S - G_y' xi Z) / s - dt c_l G_y D.
// Scales (units of R): P, Z 2^-60; U, G_y' Z, G_y' xi Z, D 2^-57; S 2^-56, with
// tau <= 1.9 so that every sum stays below 2^63.  Tiles out of range go to
// redo.  Also per target: the gather's stencil origins and weights (one set
// per speed and direction) and 1 / s*.
// Measured against k_adjoint_jvp_staged: see launch_adjoint_phase_a_staged.
template <int N1, int TY>
__global__ void __launch_bounds__(32 * TY, TY == 8 ? 1 : 2)
k_adjoint_jvp_fixed(AdjArgs A, int wwa, int wha, double c_max_d, double* __restrict__ jvp,
                    unsigned int* __restrict__ redo) {
    constexpr int TX = 32, NT = TX * TY, Q = N1 * N1;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int WN = wwa * wha;
    int4* s_h = reinterpret_cast<int4*>(smem_raw);                // [N1][WN] high words
    int4* s_l = s_h + (size_t)N1 * WN;                            // [N1][WN] low words
    int2* s_gy = reinterpret_cast<int2*>(s_l + (size_t)N1 * WN);  // [Q][NT] y-map
    int2* s_ly = s_gy + (size_t)Q * NT;                           // [4 N1][NT] y-weights
    int2* s_dy = s_ly + (size_t)4 * N1 * NT;                      // [4 N1][NT] their derivatives, 2^57
    __shared__ float s_red[4][NT / 32];
    const Lattice& L = c_La[lattice_slot(N1)];
    const LatticeFix& F = c_Lafix[lattice_slot(N1)];
    const int tid = threadIdx.x, lane = tid & 31;
    const int tiles_x = (A.nx + TX - 1) / TX;
    const int tx0 = (int)(blockIdx.x % tiles_x) * TX;
    const int ty0 = (int)(blockIdx.x / tiles_x) * TY;
    const int X = tx0 + tid % TX, Y = ty0 + tid / TX;
    const bool valid = X < A.nx && Y < A.ny;
    const long long node = (long long)Y * A.nx + X;
    const float c_max = (float)c_max_d;

    // reference gauge and scale: the tile's centre node of the input state
    const long long rnode = (long long)min(ty0 + TY / 2, A.ny - 1) * A.nx + min(tx0 + TX / 2, A.nx - 1);
    const double rux = A.in.ux[rnode], ruy = A.in.uy[rnode], rst = A.in.st[rnode];
    unsigned mh = 0u;
    if (lane < Q) {
        const int sh = fix_shift<N1>(lane / N1) + fix_shift<N1>(lane % N1);
        mh = (unsigned)__double2hiint(fabs(A.in.f[(long long)lane * A.N + rnode]) * (double)(1 << sh));
    }
    mh = __reduce_max_sync(FULL, mh);
    const int me = (int)(mh >> 20) - 1023, rexp = me + 5;
    bool in_range = me > -900 && me < 900;

    double ux = 0.0, uy = 0.0, st = 1.0;
    float vxlo = 3.0e38f, vxhi = -3.0e38f, vylo = 3.0e38f, vyhi = -3.0e38f;
    if (valid) {
        ux = A.ux_s[node];
        uy = A.uy_s[node];
        st = A.st_s[node];
        const float sp = (float)(c_max_d * st);
        vxlo = (float)ux - sp;
        vxhi = (float)ux + sp;
        vylo = (float)uy - sp;
        vyhi = (float)uy + sp;
        const float de = fmaf(c_max, fabsf((float)(rst - st)),
                              fmaxf(fabsf((float)(rux - ux)), fabsf((float)(ruy - uy))));
        in_range = in_range && de <= kFixTileDe * (float)st && (float)(st * A.dt) <= 1.9f;
    }
    staged_block_minmax4<StagedAdj64, NT>(vxlo, vxhi, vylo, vyhi, s_red);
    const float m = 1.0f, fdt = (float)A.dt;
    const float bxl = fminf(fmaxf(vxlo, -1.0e6f), 1.0e6f), bxh = fminf(fmaxf(vxhi, -1.0e6f), 1.0e6f);
    const float byl = fminf(fmaxf(vylo, -1.0e6f), 1.0e6f), byh = fminf(fmaxf(vyhi, -1.0e6f), 1.0e6f);
    const int wx0 = (int)floorf((float)tx0 - bxh * fdt - m) - 1;
    const int wx1 = (int)floorf((float)(tx0 + TX - 1) - bxl * fdt + m) + 2;
    const int wy0 = (int)floorf((float)ty0 - byh * fdt - m) - 1;
    const int wy1 = (int)floorf((float)(ty0 + TY - 1) - byl * fdt + m) + 2;
    in_range = in_range && isfinite(vxlo) && isfinite(vxhi) && isfinite(vylo) && isfinite(vyhi) &&
               fmaxf(fmaxf(fabsf(vxlo), fabsf(vxhi)), fmaxf(fabsf(vylo), fabsf(vyhi))) * fdt < 400.0f;
    const int ww = max(1, min(wx1 - wx0 + 1, wwa)), wh = max(1, min(wy1 - wy0 + 1, wha));
    GridDesc G;
    G.nx = A.nx;
    G.ny = A.ny;
    G.offset = 0;
    G.ix0 = 0;
    G.iy0 = 0;
    G.iw = A.nx;
    G.ih = A.ny;
    if (!__syncthreads_or(!in_range))
        in_range = stage_window_fixed<N1, true>(A.in, A.N, G, 0, wx0, wy0, ww, wh, WN, rux, ruy, rst,
                                                kFix - rexp, s_h, s_l, F, c_max, nullptr, tid, NT);
    else
        in_range = false;
    if (__syncthreads_or(!in_range)) {  // also: the window is staged
        // the FP64 kernel's tiles are 32 x ADJ_TY: a tile holds ADJ_TY / TY of these
        if (tid == 0) {
            const unsigned tile = (unsigned)(ty0 / ADJ_TY * tiles_x + tx0 / TX);
            if (TY == ADJ_TY || atomicExch(redo + 1 + gridDim.x + tile, 1u) == 0u)
                redo[1 + atomicAdd(redo, 1u)] = tile;
        }
        return;
    }
    if (!valid) return;

    const double inv = 1.0 / st, inv60 = kFixOne / st, dt54 = A.dt * kFixDisplacement;
    A.inv_st[node] = inv;
    const long long rt = __double2ll_rn((rst - st) * inv60);
    const long long dxt = __double2ll_rn((rux - ux) * inv60), dyt = __double2ll_rn((ruy - uy) * inv60);
    const Fix Rt = fix_split(rt), tau = fix_split(__double2ll_rn(st * A.dt * (kFixOne / 8.0)));
    Fix dex[N1], dey[N1];
    int last[N1];  // the row that completes population l's stencil, else -1
#pragma unroll
    for (int a = 0; a < N1; ++a) {
        const long long ca = fix_mul(F.c[a], Rt);
        dex[a] = fix_split(dxt + ca);
        dey[a] = fix_split(dyt + ca);
    }
    int lo = 0x7fffffff, hi = -1;
#pragma unroll
    for (int l = 0; l < N1; ++l) {
        Fix ly[4], dy[4];
        const int fy = fix_departure_d(__double2ll_rn(-fma(st, L.c[l], uy) * dt54), ly, dy);
        const int top = Y - wy0 - 1 + fy;
        last[l] = top >= 0 && top + 3 < wh ? top + 3 : -1;
        if (last[l] >= 0) {
            lo = min(lo, top);
            hi = max(hi, top + 3);
        }
        A.org_y[(long long)l * A.N + node] = fy - 1;
        double w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            s_ly[(4 * l + j) * NT + tid] = make_int2(ly[j].h, ly[j].l);
            const Fix d8 = fix_split(((long long)dy[j].h * (1ll << 32) + dy[j].l) >> 3);
            s_dy[(4 * l + j) * NT + tid] = make_int2(d8.h, d8.l);
            w[j] = fix_to_double(ly[j]);
        }
        double2* pw = reinterpret_cast<double2*>(A.lw_y + 4 * ((long long)l * A.N + node));
        pw[0] = make_double2(w[0], w[1]);
        pw[1] = make_double2(w[2], w[3]);
#pragma unroll
        for (int b = 0; b < N1; ++b) {
            const Fix gw = fix_gauge<N1>(F, l, b, dey[b]);
            s_gy[(N1 * l + b) * NT + tid] = make_int2(gw.h, gw.l);
        }
    }
    const double f_unit = pow2d(rexp - kFix);
    constexpr double dn = 1.0 / (double)(1 << fix_shift<N1>(0));
#pragma unroll 1
    for (int k = 0; k < N1; ++k) {
        Fix lx[4], dlx[4];
        const int fx = fix_departure_d(__double2ll_rn(-fma(st, L.c[k], ux) * dt54), lx, dlx);
        const int col = X - wx0 - 1 + fx;
        A.org_x[(long long)k * A.N + node] = fx - 1;
        double2* pw = reinterpret_cast<double2*>(A.lw_x + 4 * ((long long)k * A.N + node));
        pw[0] = make_double2(fix_to_double(lx[0]), fix_to_double(lx[1]));
        pw[1] = make_double2(fix_to_double(lx[2]), fix_to_double(lx[3]));
        const bool on = col >= 0 && col + 3 < ww;
        const double uk = k == 0 || k == N1 - 1 ? f_unit * dn : f_unit;
        // mode 0: U, 1: S, 2: P (which completes what the others left)
#pragma unroll 1
        for (int mode = 0; on && mode < 3; ++mode) {
            Fix cw[4][N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const Fix g = fix_gauge<N1>(F, k, a, dex[a]);
                Fix gd{0, 0};
                if (mode != 2) {
                    long long d = fix_gauge_d<N1>(F, k, a, dex[a]);
                    if (mode == 1) {
                        const long long xi = ((long long)F.c[a].h * (1ll << 32) + F.c[a].l) +
                                             ((long long)dex[a].h * (1ll << 32) + dex[a].l);
                        d = fix_mul(fix_split(xi), fix_split(d));
                    }
                    gd = fix_split(d);
                }
#pragma unroll
                for (int jx = 0; jx < 4; ++jx) {
                    if (mode == 2) {
                        cw[jx][a] = fix_split(fix_mul(lx[jx], g));
                    } else {
                        long long tb = fix_mul(fix_split(fix_mul(dlx[jx], g)), tau);
                        long long lg = fix_mul(lx[jx], gd) >> 3;
                        if (mode == 1) {
                            tb = fix_mul(F.c[k], fix_split(tb)) >> 1;
                            lg >>= 1;
                        }
                        cw[jx][a] = fix_split(-tb - lg);
                    }
                }
            }
            Fix Pb[4][N1];
#pragma unroll 1
            for (int y = lo; y <= hi; ++y) {
                const int4* sh = s_h + y * ww + col;
                const int4* sl = s_l + y * ww + col;
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
                        const int4 gh = sh[(size_t)a * WN + jx], gl = sl[(size_t)a * WN + jx];
                        fix_mad(cw[jx][a], gh.x, gl.x, h[0], mm[0]);
                        fix_mad(cw[jx][a], gh.y, gl.y, h[1], mm[1]);
                        fix_mad(cw[jx][a], gh.z, gl.z, h[2], mm[2]);
                        if (N1 == 4) fix_mad(cw[jx][a], gh.w, gl.w, h[3], mm[3]);
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
                    long long fh = 0, fm = 0, eh = 0, em = 0, ph = 0, pm = 0, qh = 0, qm = 0;
                    Fix ly[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int2 v = s_ly[(4 * l + j) * NT + tid];
                        ly[j] = Fix{v.x, v.y};
                    }
#pragma unroll
                    for (int b = 0; b < N1; ++b) {
                        long long zh = 0, zm = 0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) fix_mad(ly[j], Pb[j][b].h, Pb[j][b].l, zh, zm);
                        const Fix z = fix_split(fix_sum(zh, zm));
                        const int2 v = s_gy[(N1 * l + b) * NT + tid];
                        const Fix gw{v.x, v.y};
                        fix_mad(gw, z.h, z.l, fh, fm);  // G_y sum ly (P, U or S)
                        if (mode == 2) {
                            long long dh = 0, dm = 0;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int2 w = s_dy[(4 * l + j) * NT + tid];
                                fix_mad(Fix{w.x, w.y}, Pb[j][b].h, Pb[j][b].l, dh, dm);
                            }
                            const Fix d = fix_split(fix_sum(dh, dm));
                            fix_mad(gw, d.h, d.l, eh, em);  // G_y D
                            const long long gd = fix_gauge_d<N1>(F, l, b, dey[b]);
                            const long long xi = ((long long)F.c[b].h * (1ll << 32) + F.c[b].l) +
                                                 ((long long)dey[b].h * (1ll << 32) + dey[b].l);
                            const long long gx = fix_mul(fix_split(xi), fix_split(gd));
                            fix_mad(fix_split(gd >> 3), z.h, z.l, ph, pm);  // G_y' Z
                            fix_mad(fix_split(gx >> 3), z.h, z.l, qh, qm);  // G_y' xi Z
                        }
                    }
                    const long long q = (long long)(N1 * k + l) * A.N + node;
                    const long long plane = (long long)Q * A.N;
                    const double u = l == 0 || l == N1 - 1 ? uk * dn : uk;
                    const double f = (double)fix_sum(fh, fm);
                    if (mode == 0) {
                        jvp[plane + q] = f * (8.0 * u * inv);
                    } else if (mode == 1) {
                        jvp[3 * plane + q] = f * (16.0 * u * inv);
                    } else {
                        jvp[q] = f * u;
                        const double d = (double)fix_sum(eh, em) * (8.0 * u * A.dt);
                        const double ui = 8.0 * u * inv;
                        jvp[2 * plane + q] = -fma((double)fix_sum(ph, pm), ui, d);
                        const double qx = fma((double)fix_sum(qh, qm), ui, L.c[l] * d);
                        jvp[3 * plane + q] -= qx;
                    }
                }
            }
        }
        // stencils off the window
#pragma unroll 1
        for (int l = 0; l < N1; ++l) {
            int la = last[0];
#pragma unroll
            for (int i = 1; i < N1; ++i) la = i == l ? last[i] : la;
            if (on && la >= 0) continue;
            double R[4];
            adj_population_direct<N1>(A, X, Y, k, l, ux, uy, st, R);
#pragma unroll
            for (int i = 0; i < 4; ++i) jvp[((long long)i * Q + N1 * k + l) * A.N + node] = R[i];
        }
    }
}

// The rest of phase A from A* and its tangents: the collision cotangent,
// beta_bar, the 3 x 3 implicit solve at the fixed point and w, one thread
// per target node.  Every sum the solve needs is linear in the populations'
// values, so the node's populations are read once and folded into running
// sums (tangent d^i, i = u_x, u_y, s; e_q = |c_q|^2 - 2 T_L):
//   rho = sum A_q,  wf = sum W_q fbar_q,  af = sum A_q fbar_q,
//   sk_i = sum c_k d^i_q,  sl_i = sum c_l d^i_q,  se_i = sum e_q d^i_q,
//   sf_i = sum fbar_q d^i_q,  s1_i = sum d^i_q.
// Then J = M_A A_lambda has rows (s/rho) sk, (s/rho) sl, s/(4 rho T_L) se;
// g_i = (1 - 2 beta) sf_i + 2 beta wf s1_i + lambdabar_i (the s component
// of lambdabar taken from T: dT/ds = 2 s T_L); betabar = 2 rho wf - 2 af;
// and w_q = Abar_q + (M_A^T mu)_q.
template <int N1>
__global__ void __launch_bounds__(256) k_adjoint_epilogue(AdjArgs A, const double* __restrict__ jvp) {
    constexpr int Q = N1 * N1;
    const Lattice& L = c_La[lattice_slot(N1)];
    const long long node = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = node < A.N;
    double bb = 0.0;
    if (valid) {
        const long long N = A.N;
        double rho = 0.0, wf = 0.0, af = 0.0;
        double sk[3], sl[3], se[3], sf[3], s1[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) sk[i] = sl[i] = se[i] = sf[i] = s1[i] = 0.0;
        double fb[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int k = q / N1, l = q % N1;
            const double ck = L.c[k], cl = L.c[l];
            const double e = fma(ck, ck, cl * cl) - 2.0 * A.T_L;
            const double a = jvp[(long long)q * N + node];
            fb[q] = A.fbar[(long long)q * N + node];
            rho += a;
            wf = fma(L.w[k] * L.w[l], fb[q], wf);
            af = fma(a, fb[q], af);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const double d = jvp[((long long)(1 + i) * Q + q) * N + node];
                sk[i] = fma(ck, d, sk[i]);
                sl[i] = fma(cl, d, sl[i]);
                se[i] = fma(e, d, se[i]);
                sf[i] = fma(fb[q], d, sf[i]);
                s1[i] += d;
            }
        }
        const double st = A.st_s[node];
        const double sr = st / rho, ss = st / (4.0 * rho * A.T_L);
        bb = 2.0 * (rho * wf - af);
        // J[m][i]: moment m (u_x, u_y, s), tangent i
        double J[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            J[0][i] = sr * sk[i];
            J[1][i] = sr * sl[i];
            J[2][i] = ss * se[i];
        }
        const double b1 = 1.0 - 2.0 * A.beta, b2 = 2.0 * A.beta * wf;
        const double g0 = fma(b1, sf[0], b2 * s1[0]) + A.gbar[node];
        const double g1 = fma(b1, sf[1], b2 * s1[1]) + A.gbar[N + node];
        const double g2 = fma(b1, sf[2], b2 * s1[2]) + A.gbar[2 * N + node] * 2.0 * st * A.T_L;
        // solve J^T mu = -g by Cramer's rule (a = J^T)
        const double a00 = J[0][0], a01 = J[1][0], a02 = J[2][0];
        const double a10 = J[0][1], a11 = J[1][1], a12 = J[2][1];
        const double a20 = J[0][2], a21 = J[1][2], a22 = J[2][2];
        const double det = a00 * (a11 * a22 - a12 * a21) - a01 * (a10 * a22 - a12 * a20) +
                           a02 * (a10 * a21 - a11 * a20);
        const double idet = 1.0 / det;
        const double r0 = -g0, r1 = -g1, r2 = -g2;
        const double mu0 = (r0 * (a11 * a22 - a12 * a21) - a01 * (r1 * a22 - a12 * r2) +
                            a02 * (r1 * a21 - a11 * r2)) * idet;
        const double mu1 = (a00 * (r1 * a22 - a12 * r2) - r0 * (a10 * a22 - a12 * a20) +
                            a02 * (a10 * r2 - r1 * a20)) * idet;
        const double mu2 = (a00 * (a11 * r2 - r1 * a21) - a01 * (a10 * r2 - r1 * a20) +
                            r0 * (a10 * a21 - a11 * a20)) * idet;
        const double m0 = sr * mu0, m1 = sr * mu1, m2 = ss * mu2;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int k = q / N1, l = q % N1;
            const double ck = L.c[k], cl = L.c[l];
            const double e = fma(ck, ck, cl * cl) - 2.0 * A.T_L;
            A.w[(long long)q * N + node] = fma(b1, fb[q], b2) + fma(ck, m0, fma(cl, m1, e * m2));
        }
    }
    // beta_bar: one atomic per warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bb += __shfl_xor_sync(0xffffffffu, bb, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(A.beta_bar, bb);
}

// Launch of the staged phase A: the fixed-point kernel, the FP64 kernel over the
// tiles it left (windows of wwa x wha staged nodes), the epilogue.  The fixed
// kernel takes 32 x 8 tiles, or 32 x 4 where the window of those does not fit.
// 256^2: 2.12 ms for the FP64 kernel alone, 0.44 ms so (4 steps forward and back:
// 21.6 -> 14.9 ms).
cudaError_t launch_adjoint_phase_a_staged(const AdjArgs& A, int n1, int ex, int ey, double c_max,
                                          double* jvp, unsigned int* redo, int sms, cudaStream_t s) {
    static int s_set[64][2] = {{0}}, s_fix[64][4] = {{0}};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    auto raise = [](const void* kern, size_t smem, int* set) {
        if ((int)smem <= *set) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) *set = (int)smem;
        return e;
    };
    const size_t cap = 220 * 1024, cap64 = 200 * 1024;
    int ty = 8, w = 32 + ex, h = 8 + ey;
    auto bytes = [&] { return (size_t)n1 * w * h * 32 + (size_t)32 * ty * 8 * (n1 * n1 + 8 * n1); };
    if (bytes() > cap) {
        ty = 4;
        h = 4 + ey;
    }
    while (bytes() > cap) {
        if (w - 32 >= h - ty) --w; else --h;
    }
    const long long tiles_x = (A.nx + 31) / 32, tiles = tiles_x * ((A.ny + ty - 1) / ty);
    const long long tiles8 = tiles_x * ((A.ny + ADJ_TY - 1) / ADJ_TY);
    void (*fixed)(AdjArgs, int, int, double, double*, unsigned int*) =
        n1 == 3 ? (ty == 8 ? k_adjoint_jvp_fixed<3, 8> : k_adjoint_jvp_fixed<3, 4>)
                : (ty == 8 ? k_adjoint_jvp_fixed<4, 8> : k_adjoint_jvp_fixed<4, 4>);
    e = raise((const void*)fixed, bytes(), &s_fix[dev][(n1 == 3 ? 2 : 0) + (ty == 8 ? 1 : 0)]);
    // the count, and (32 x 4) the marks behind the list
    if (e == cudaSuccess) e = cudaMemsetAsync(redo, 0, sizeof(unsigned int), s);
    if (e == cudaSuccess && ty != ADJ_TY)
        e = cudaMemsetAsync(redo + 1 + tiles, 0, sizeof(unsigned int) * tiles8, s);
    if (e != cudaSuccess) return e;
    fixed<<<(unsigned)tiles, 32 * ty, bytes(), s>>>(A, w, h, c_max, jvp, redo);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;

    w = 32 + ex;
    h = ADJ_TY + ey;
    while ((size_t)n1 * w * h * sizeof(Double4) > cap64) {
        if (w - 32 >= h - ADJ_TY) --w; else --h;
    }
    const size_t smem = (size_t)n1 * w * h * sizeof(Double4);
    void (*kern)(AdjArgs, int, int, double, double*, const unsigned int*) =
        n1 == 3 ? k_adjoint_jvp_staged<3> : k_adjoint_jvp_staged<4>;
    e = raise((const void*)kern, smem, &s_set[dev][n1 == 3 ? 1 : 0]);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)(tiles8 < sms ? tiles8 : sms), 32 * ADJ_TY, smem, s>>>(A, w, h, c_max, jvp, redo);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)((A.N + 255) / 256);
    if (n1 == 3) k_adjoint_epilogue<3><<<nb, 256, 0, s>>>(A, jvp);
    else k_adjoint_epilogue<4><<<nb, 256, 0, s>>>(A, jvp);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Phase B in fixed point.  Per source and target the gather evaluates gauge maps
// and visits some 80 targets; the transpose of the staged reconstruction
// instead runs over the targets, in the frame of their tile's reference gauge r:
//   h(s)[a][b] = sum_{t, k} lx_k(s) G_x(r -> t)[k][a] V_k(y_s)[b],
//   V_k(y)[b]  = sum_l ly_l(y) w_(k,l) G_y(r -> t)[l][b]  over the stencils with row y,
// 2304 products per target (D2Q16) as in a pass of the step, scattered into
// the tile's window of sources in shared memory.  The sums are 64-bit integers
// (the largest |w| of the tile is held to 2^55 .. 2^56; every sum of a source
// stays below 2^63), added as two 32-bit atomics with the carry taken from the
// first one's result, so their order does not matter and the result is the
// same in every run.  (A 64-bit shared-memory atomic takes 14.6 clocks per warp
// and SM, two 32-bit ones 3 to 4.)  Then each source's h is taken back to its
// own frame, G(s -> r)^T h, in FP64, and stored per tile; k_adjoint_reduce adds the
// tiles that reach a source in a fixed order and forms the gauge cotangent.
// Tiles whose gauges, displacements or cotangents are out of range, or with a
// stencil off the window, are marked and left to k_adjoint_sources_t.
struct ScatterTile {
    int x0, y0, w, h;  // the window in unwrapped coordinates; w = 0: left
};
constexpr int ADJ_SCATTER_WN = 1248;  // window nodes (160 KB of sums on D2Q16)

__device__ __forceinline__ void atomic_add64(unsigned int* lo, unsigned int* hi, long long v) {
    const unsigned int vl = (unsigned int)v;
    const unsigned int old = atomicAdd(lo, vl);
    atomicAdd(hi, (unsigned int)((unsigned long long)v >> 32) + (old + vl < old ? 1u : 0u));
}

template <int N1>
__global__ void __launch_bounds__(32 * ADJ_TY, 1)
k_adjoint_scatter(AdjArgs A, double c_max_d, double* __restrict__ win, ScatterTile* __restrict__ tiles,
                  unsigned int* __restrict__ left) {
    constexpr int TX = 32, TY = ADJ_TY, NT = TX * TY, Q = N1 * N1, WN = ADJ_SCATTER_WN;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(32) unsigned char smem_raw[];
    unsigned int* s_lo = reinterpret_cast<unsigned int*>(smem_raw);  // [Q][WN]
    unsigned int* s_hi = s_lo + (size_t)Q * WN;                      // [Q][WN]
    int2* s_gy = reinterpret_cast<int2*>(s_hi + (size_t)Q * WN);     // [Q][NT] G_y(r -> t)
    int2* s_ly = s_gy + (size_t)Q * NT;                              // [4 N1][NT] y-weights
    __shared__ float s_red[4][NT / 32];
    __shared__ unsigned int s_max;
    const Lattice& L = c_La[lattice_slot(N1)];
    const LatticeFix& F = c_Lafix1[lattice_slot(N1)];
    const int tid = threadIdx.x;
    const int tiles_x = (A.nx + TX - 1) / TX;
    const int tx0 = (int)(blockIdx.x % tiles_x) * TX, ty0 = (int)(blockIdx.x / tiles_x) * TY;
    const int X = tx0 + tid % TX, Y = ty0 + tid / TX;
    const bool valid = X < A.nx && Y < A.ny;
    const long long node = (long long)Y * A.nx + X, N = A.N;
    const float c_max = (float)c_max_d;
    if (tid == 0) s_max = 0u;
    const long long rnode = (long long)min(ty0 + TY / 2, A.ny - 1) * A.nx + min(tx0 + TX / 2, A.nx - 1);
    const double rux = A.in.ux[rnode], ruy = A.in.uy[rnode], rst = A.in.st[rnode];

    bool in_range = true;
    double ux = 0.0, uy = 0.0, st = 1.0;
    unsigned int mh = 0u;
    float vxlo = 3.0e38f, vxhi = -3.0e38f, vylo = 3.0e38f, vyhi = -3.0e38f;
    if (valid) {
        ux = A.ux_s[node];
        uy = A.uy_s[node];
        st = A.st_s[node];
        const float sp = (float)(c_max_d * st);
        vxlo = (float)ux - sp;
        vxhi = (float)ux + sp;
        vylo = (float)uy - sp;
        vyhi = (float)uy + sp;
        const float de = fmaf(c_max, fabsf((float)(rst - st)),
                              fmaxf(fabsf((float)(rux - ux)), fabsf((float)(ruy - uy))));
        in_range = de <= kFixTileDe * (float)st;
#pragma unroll
        for (int q = 0; q < Q; ++q)
            mh = max(mh, (unsigned)__double2hiint(A.w[(long long)q * N + node]) & 0x7fffffffu);
    }
    mh = __reduce_max_sync(FULL, mh);
    staged_block_minmax4<StagedAdj64, NT>(vxlo, vxhi, vylo, vyhi, s_red);  // (orders s_max = 0)
    if ((tid & 31) == 0) atomicMax(&s_max, mh);
    const float m = 1.0f, fdt = (float)A.dt;
    const float bxl = fminf(fmaxf(vxlo, -1.0e6f), 1.0e6f), bxh = fminf(fmaxf(vxhi, -1.0e6f), 1.0e6f);
    const float byl = fminf(fmaxf(vylo, -1.0e6f), 1.0e6f), byh = fminf(fmaxf(vyhi, -1.0e6f), 1.0e6f);
    const int wx0 = (int)floorf((float)tx0 - bxh * fdt - m) - 1;
    const int wx1 = (int)floorf((float)(tx0 + TX - 1) - bxl * fdt + m) + 2;
    const int wy0 = (int)floorf((float)ty0 - byh * fdt - m) - 1;
    const int wy1 = (int)floorf((float)(ty0 + TY - 1) - byl * fdt + m) + 2;
    const int ww = max(1, min(wx1 - wx0 + 1, WN)), wh = max(1, min(wy1 - wy0 + 1, WN / ww));
    in_range = in_range && isfinite(vxlo) && isfinite(vxhi) && isfinite(vylo) && isfinite(vyhi) &&
               fmaxf(fmaxf(fabsf(vxlo), fabsf(vxhi)), fmaxf(fabsf(vylo), fabsf(vyhi))) * fdt < 400.0f;
    __syncthreads();
    mh = s_max;
    // the scale: |w| 2^scale < 2^56 (all zero: any)
    const int scale = mh == 0u ? 0 : 55 - ((int)(mh >> 20) - 1023);
    in_range = in_range && mh < 0x7ff00000u && (mh == 0u || (scale > -900 && scale < 900));

    // this target's map and stencils (all in the window, or the tile is left)
    const double inv60 = kFixOne / st, dt54 = A.dt * kFixDisplacement;
    const long long rt = __double2ll_rn((rst - st) * inv60);
    const long long dxt = __double2ll_rn((rux - ux) * inv60), dyt = __double2ll_rn((ruy - uy) * inv60);
    const Fix Rt = fix_split(rt);
    Fix dex[N1];
    int top[N1];
    if (valid) {
        Fix dey[N1];
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            const long long ca = fix_mul(F.c[a], Rt);
            dex[a] = fix_split(dxt + ca);
            dey[a] = fix_split(dyt + ca);
        }
#pragma unroll
        for (int l = 0; l < N1; ++l) {
            Fix w[4];
            top[l] = Y - wy0 - 1 + fix_departure(__double2ll_rn(-fma(st, L.c[l], uy) * dt54), w);
            const int col = X - wx0 - 1 + fix_departure(__double2ll_rn(-fma(st, L.c[l], ux) * dt54), w);
            in_range = in_range && top[l] >= 0 && top[l] + 3 < wh && col >= 0 && col + 3 < ww;
        }
#pragma unroll
        for (int l = 0; l < N1; ++l) {
            Fix w[4];
            fix_departure(__double2ll_rn(-fma(st, L.c[l], uy) * dt54), w);
#pragma unroll
            for (int j = 0; j < 4; ++j) s_ly[(4 * l + j) * NT + tid] = make_int2(w[j].h, w[j].l);
#pragma unroll
            for (int b = 0; b < N1; ++b) {
                const Fix g = fix_gauge<N1>(F, l, b, dey[b]);
                s_gy[(N1 * l + b) * NT + tid] = make_int2(g.h, g.l);
            }
        }
    }
    const int wn = ww * wh;
    for (int i = tid; i < Q * WN; i += NT) s_lo[i] = s_hi[i] = 0u;
    if (__syncthreads_or(!in_range)) {  // also: the sums are zero
        if (tid == 0) {
            tiles[blockIdx.x] = ScatterTile{0, 0, 0, 0};
            left[1 + blockIdx.x] = 1u;
            atomicAdd(left, 1u);
        }
        return;
    }
    if (tid == 0) {
        tiles[blockIdx.x] = ScatterTile{wx0, wy0, ww, wh};
        left[1 + blockIdx.x] = 0u;
    }

    if (valid) {
        int lo = top[0], hi = top[0] + 3;
#pragma unroll
        for (int l = 1; l < N1; ++l) {
            lo = min(lo, top[l]);
            hi = max(hi, top[l] + 3);
        }
#pragma unroll 1
        for (int k = 0; k < N1; ++k) {
            Fix cxa[4][N1];
            int col;
            {
                Fix lx[4];
                col = X - wx0 - 1 + fix_departure(__double2ll_rn(-fma(st, L.c[k], ux) * dt54), lx);
#pragma unroll
                for (int a = 0; a < N1; ++a) {
                    const Fix g = fix_gauge<N1>(F, k, a, dex[a]);
#pragma unroll
                    for (int jx = 0; jx < 4; ++jx) cxa[jx][a] = fix_split(fix_mul(lx[jx], g));
                }
            }
            Fix wg[N1][N1];  // w_(k,l) G_y[l][b]
#pragma unroll
            for (int l = 0; l < N1; ++l) {
                bool big = false;
                const Fix w = fix_split(fix_population(A.w[(long long)(N1 * k + l) * N + node], scale, big));
#pragma unroll
                for (int b = 0; b < N1; ++b) {
                    const int2 v = s_gy[(N1 * l + b) * NT + tid];
                    wg[l][b] = fix_split(fix_mul(Fix{v.x, v.y}, w));
                }
            }
#pragma unroll 1
            for (int y = lo; y <= hi; ++y) {
                long long vh[N1], vm[N1];
#pragma unroll
                for (int b = 0; b < N1; ++b) vh[b] = vm[b] = 0;
                bool any = false;
#pragma unroll
                for (int l = 0; l < N1; ++l) {
                    const unsigned j = (unsigned)(y - top[l]);
                    if (j > 3u) continue;
                    any = true;
                    const int2 v = s_ly[(4 * l + (int)j) * NT + tid];
#pragma unroll
                    for (int b = 0; b < N1; ++b) fix_mad(Fix{v.x, v.y}, wg[l][b].h, wg[l][b].l, vh[b], vm[b]);
                }
                if (!any) continue;
                Fix V[N1];
#pragma unroll
                for (int b = 0; b < N1; ++b) V[b] = fix_split(fix_sum_rn(vh[b], vm[b]));
                const int at = y * ww + col;
#pragma unroll
                for (int jx = 0; jx < 4; ++jx)
#pragma unroll
                    for (int a = 0; a < N1; ++a)
#pragma unroll
                        for (int b = 0; b < N1; ++b) {
                            long long h = 0, mm = 0;
                            fix_mad(cxa[jx][a], V[b].h, V[b].l, h, mm);
                            const int i = (N1 * a + b) * WN + at + jx;
                            atomic_add64(s_lo + i, s_hi + i, fix_sum_rn(h, mm));
                        }
            }
        }
    }
    __syncthreads();

    // the sources' sums into their own frames
    const double inv_rst = 1.0 / rst;
    double* out = win + (size_t)blockIdx.x * Q * WN;
    const float inv_ww = 1.0f / (float)ww;
    for (int i = tid; i < wn; i += NT) {
        const int cy = window_row(i, inv_ww), cx = i - cy * ww;
        const long long s = (long long)wrap_near(wy0 + cy, A.ny) * A.nx + wrap_near(wx0 + cx, A.nx);
        const double r = (A.in.st[s] - rst) * inv_rst;
        const double dx = (A.in.ux[s] - rux) * inv_rst, dy = (A.in.uy[s] - ruy) * inv_rst;
        double h[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const double v = (double)((long long)((unsigned long long)s_hi[q * WN + i] << 32 | s_lo[q * WN + i]));
            h[q] = v * pow2d(-scale);
        }
        double e[N1][N1];  // [k][a] of G(s -> r) - I, by y, then by x
        double H[Q];
#pragma unroll
        for (int b = 0; b < N1; ++b) {
            const double de = fma(L.c[b], r, dy);
#pragma unroll
            for (int l = 0; l < N1; ++l) e[l][b] = gauge_tail<N1>(L.d3[l], L.d2[l][b], L.d1[l][b], de) * de;
        }
#pragma unroll
        for (int a = 0; a < N1; ++a)
#pragma unroll
            for (int b = 0; b < N1; ++b) {
                double v = h[N1 * a + b];
#pragma unroll
                for (int l = 0; l < N1; ++l) v = fma(e[l][b], h[N1 * a + l], v);
                H[N1 * a + b] = v;
            }
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            const double de = fma(L.c[a], r, dx);
#pragma unroll
            for (int k = 0; k < N1; ++k) e[k][a] = gauge_tail<N1>(L.d3[k], L.d2[k][a], L.d1[k][a], de) * de;
        }
#pragma unroll
        for (int a = 0; a < N1; ++a)
#pragma unroll
            for (int b = 0; b < N1; ++b) {
                double v = H[N1 * a + b];
#pragma unroll
                for (int k = 0; k < N1; ++k) v = fma(e[k][a], H[N1 * k + b], v);
                out[(N1 * a + b) * WN + i] = v;
            }
    }
}

// f_bar of every source from the tiles whose windows hold it (an image of it,
// where the grid is narrower than a window), and its gauge cotangent, from
//   d g / d u_x [k][l] = sum_a d1[k][a] f[a][l] / s  and so on (k_adjoint_sources_t),
// through M[k][a] = sum_l f_bar[k][l] f[a][l] and its y-counterpart.
template <int N1>
__global__ void __launch_bounds__(128)
k_adjoint_reduce(AdjArgs A, const double* __restrict__ win, const ScatterTile* __restrict__ tiles) {
    constexpr int Q = N1 * N1, WN = ADJ_SCATTER_WN;
    const Lattice& L = c_La[lattice_slot(N1)];
    const long long src = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (src >= A.N) return;
    const int JX = (int)(src % A.nx), JY = (int)(src / A.nx);
    const int tiles_x = (A.nx + 31) / 32, tiles_y = (A.ny + ADJ_TY - 1) / ADJ_TY;
    double fb[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) fb[q] = 0.0;
    // tile origins t0 whose window can hold x: x + vlo dt - 31 - 5 <= t0 <= x + vhi dt + 5
    double vx0 = A.vlo_x[0], vx1 = A.vhi_x[0], vy0 = A.vlo_y[0], vy1 = A.vhi_y[0];
#pragma unroll
    for (int i = 1; i < N1; ++i) {
        vx0 = fmin(vx0, A.vlo_x[i]);
        vx1 = fmax(vx1, A.vhi_x[i]);
        vy0 = fmin(vy0, A.vlo_y[i]);
        vy1 = fmax(vy1, A.vhi_y[i]);
    }
    // (a left tile has no window: bounds beyond its 400 nodes are not needed)
    const int xa = (int)floor(fmax(vx0 * A.dt, -500.0)) - 36, xb = (int)ceil(fmin(vx1 * A.dt, 500.0)) + 5;
    const int ya = (int)floor(fmax(vy0 * A.dt, -500.0)) - (ADJ_TY + 4), yb = (int)ceil(fmin(vy1 * A.dt, 500.0)) + 5;
    // images x + m n with a tile origin in [0, n - 1] in reach
    const int my0 = -(JY + yb) / A.ny - 1, my1 = (A.ny - 1 - JY - ya) / A.ny + 1;
    const int mx0 = -(JX + xb) / A.nx - 1, mx1 = (A.nx - 1 - JX - xa) / A.nx + 1;
    for (int my = my0; my <= my1; ++my) {
        const int y = JY + my * A.ny;
        const int tya = max(0, (y + ya) / ADJ_TY - 1), tyb = min(tiles_y - 1, (y + yb) / ADJ_TY);
        for (int ty = tya; y + yb >= 0 && ty <= tyb; ++ty)
            for (int mx = mx0; mx <= mx1; ++mx) {
                const int x = JX + mx * A.nx;
                const int txa = max(0, (x + xa) / 32 - 1), txb = min(tiles_x - 1, (x + xb) / 32);
                for (int tx = txa; x + xb >= 0 && tx <= txb; ++tx) {
                    const long long t = (long long)ty * tiles_x + tx;
                    const ScatterTile w = tiles[t];
                    const int cx = x - w.x0, cy = y - w.y0;
                    if (cx < 0 || cx >= w.w || cy < 0 || cy >= w.h) continue;
                    const double* p = win + (size_t)t * Q * WN + cy * w.w + cx;
#pragma unroll
                    for (int q = 0; q < Q; ++q) fb[q] += p[(size_t)q * WN];
                }
            }
    }
    double f[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        f[q] = A.in.f[(long long)q * A.N + src];
        A.fbar_in[(long long)q * A.N + src] = fb[q];
    }
    double bux = 0.0, buy = 0.0, bst = 0.0;
#pragma unroll
    for (int k = 0; k < N1; ++k)
#pragma unroll
        for (int a = 0; a < N1; ++a) {
            double mx = 0.0, my = 0.0;
#pragma unroll
            for (int i = 0; i < N1; ++i) {
                mx = fma(fb[N1 * k + i], f[N1 * a + i], mx);
                my = fma(fb[N1 * i + k], f[N1 * i + a], my);
            }
            const double d = L.d1[k][a];
            bux = fma(d, mx, bux);
            buy = fma(d, my, buy);
            bst = fma(d * L.c[a], mx + my, bst);
        }
    const double stj = A.in.st[src], is = 1.0 / stj;
    A.gbar_in[src] = bux * is;
    A.gbar_in[A.N + src] = buy * is;
    // s = sqrt(T / T_L): dL/dT = dL/ds / (2 s T_L)
    A.gbar_in[2 * A.N + src] = bst * is / (2.0 * stj * A.T_L);
}

// Phase B of the staged contexts: the scatter, its reduction, and the gather
// over the tiles the scatter left (usually none: its CTAs then end at once).
// 256^2: 2.02 ms for the gather alone, 0.37 ms so (scatter 310, reduction 58 us); 4
// steps forward and back 14.9 -> 8.4 ms.
cudaError_t launch_adjoint_phase_b_staged(const AdjArgs& A, int n1, double c_max, double* win,
                                          ScatterTile* tiles, unsigned int* left, int sms,
                                          cudaStream_t s) {
    static int s_set[64][2] = {{0}};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const size_t smem = (size_t)8 * n1 * n1 * ADJ_SCATTER_WN + (size_t)32 * ADJ_TY * 8 * (n1 * n1 + 4 * n1);
    void (*kern)(AdjArgs, double, double*, ScatterTile*, unsigned int*) =
        n1 == 3 ? k_adjoint_scatter<3> : k_adjoint_scatter<4>;
    int& set = s_set[dev][n1 == 3 ? 1 : 0];
    if ((int)smem > set) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        set = (int)smem;
    }
    e = cudaMemsetAsync(left, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    const unsigned n_tiles = (unsigned)(((A.nx + 31) / 32) * ((A.ny + ADJ_TY - 1) / ADJ_TY));
    kern<<<n_tiles, 32 * ADJ_TY, smem, s>>>(A, c_max, win, tiles, left);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const unsigned nb = (unsigned)((A.N + 127) / 128);
    if (n1 == 3) k_adjoint_reduce<3><<<nb, 128, 0, s>>>(A, win, tiles);
    else k_adjoint_reduce<4><<<nb, 128, 0, s>>>(A, win, tiles);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long all = (A.N + ADJ_GATHER_WARPS - 1) / ADJ_GATHER_WARPS;
    const unsigned ng = (unsigned)(all < 16 * sms ? all : 16 * sms);
    if (n1 == 3) k_adjoint_sources_t<3><<<ng, ADJ_GATHER_WARPS * 32, 0, s>>>(A, left);
    else k_adjoint_sources_t<4><<<ng, ADJ_GATHER_WARPS * 32, 0, s>>>(A, left);
    return cudaGetLastError();
}

template <int N1>
__global__ void k_rho_bar(const double* __restrict__ fbar, double* __restrict__ rbar, long long N) {
    const Lattice& L = c_La[lattice_slot(N1)];
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double r = 0.0;
#pragma unroll
    for (int q = 0; q < N1 * N1; ++q) r = fma(L.w[q / N1] * L.w[q % N1], fbar[q * N + i], r);
    rbar[i] = r;
}

}  // namespace pond

using namespace pond;

void destroy_adjoint(pond_ctx* ctx) {
    AdjointScratch* a = ctx->adj;
    if (!a) return;
    cudaFree(a->fwd.f);
    cudaFree(a->fwd.ux);
    cudaFree(a->fwd.uy);
    cudaFree(a->fwd.st);
    cudaFree(a->w);
    cudaFree(a->iters);
    cudaFree(a->stats);
    cudaFree(a->beta_bar);
    cudaFree(a->minmax);
    cudaFree(a->org);
    cudaFree(a->lw);
    cudaFree(a->org1);
    cudaFree(a->lw1);
    cudaFree(a->redo);
    cudaFree(a->win);
    cudaFree(a->tiles);
    cudaFree(a->inv_st);
    cudaFree(a->jvp);
    cudaFree(a->nu_dev);
    delete a;
    ctx->adj = nullptr;
}

static pond_status adj_fail(pond_ctx* ctx, cudaError_t e, const char* where) {
    ctx->err = std::string(where) + ": " + cudaGetErrorString(e);
    (void)cudaGetLastError();  // clear a non-sticky error (a failed allocation) for the next call
    return e == cudaErrorMemoryAllocation ? POND_ERR_OOM : POND_ERR_CUDA;
}

#define ACK(call, where)                                           \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return adj_fail(ctx, e_, where);    \
    } while (0)

namespace pond {

// The step's output gauge (u_x, u_y, T) given by the caller, stored as the
// scratch forward gauge (u_x, u_y, sqrt(T / T_L)), the form the forward step
// itself stores.
__global__ void k_gauge_from_T(const double* __restrict__ ux, const double* __restrict__ uy,
                               const double* __restrict__ T, double* __restrict__ ux_o,
                               double* __restrict__ uy_o, double* __restrict__ st_o, long long N,
                               double T_L) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) {
        ux_o[i] = ux[i];
        uy_o[i] = uy[i];
        st_o[i] = sqrt(T[i] / T_L);
    }
}

cudaError_t launch_gauge_from_T(const double* ux, const double* uy, const double* T,
                                double* ux_o, double* uy_o, double* st_o, long long N,
                                double T_L, cudaStream_t s) {
    if (N == 0) return cudaSuccess;
    k_gauge_from_T<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(ux, uy, T, ux_o, uy_o, st_o, N, T_L);
    return cudaGetLastError();
}

}  // namespace pond

// d(loss)/d(nu) of one adjoint step from its beta cotangent on the device:
// beta = 1 / (2 nu / (T_ref dt) + 1)  =>  d beta / d nu = -2 beta^2 / (T_ref dt).
// To the host accumulator when one is given (a copy and a synchronisation),
// else to the context's device accumulator (stream-ordered, no
// synchronisation), which pond_adjoint_nu_bar reads.
__global__ void k_nu_accum(const double* __restrict__ beta_bar, double* __restrict__ nu_dev,
                           double dbeta_dnu) {
    if (threadIdx.x == 0) *nu_dev += *beta_bar * dbeta_dnu;
}

static cudaError_t accumulate_nu_bar(pond_ctx* ctx, AdjointScratch* a, double* nu_bar_accum) {
    const double beta = ctx->P.beta;
    const double dbeta = -2.0 * beta * beta / (ctx->cfg.T_ref * ctx->cfg.dt);
    if (!nu_bar_accum) {
        k_nu_accum<<<1, 32, 0, ctx->stream>>>(a->beta_bar, a->nu_dev, dbeta);
        return cudaGetLastError();
    }
    double bb = 0.0;
    cudaError_t e = cudaMemcpyAsync(&bb, a->beta_bar, sizeof(double), cudaMemcpyDeviceToHost,
                                    ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) *nu_bar_accum += bb * dbeta;
    return e;
}

// Both entry points: out_gauge = {u_x, u_y, T} of the step's output when
// the caller has it (pond_adjoint_step_given), else NULLs and the forward
// step is recomputed here.
static pond_status adjoint_step_impl(pond_ctx* ctx, const double* const out_gauge[3],
                                     const void* f_bar_in, const void* gauge_bar_in,
                                     void* f_bar_out, void* gauge_bar_out,
                                     double* nu_bar_accum) {
    if (!ctx) return POND_ERR_ARG;
    if (!f_bar_in || !gauge_bar_in || !f_bar_out || !gauge_bar_out) {
        ctx->err = "adjoint: NULL argument";
        return POND_ERR_ARG;
    }
    if (ctx->n_grids != 1 || !ctx->cfg.thermal) {
        ctx->err = "adjoint: single-grid thermal contexts only";
        return POND_ERR_ARG;
    }
    if (!ctx->grid_set[0]) {
        ctx->err = "adjoint before pond_set_state";
        return POND_ERR_STATE;
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != ctx->device) cudaSetDevice(ctx->device);
    struct Restore {
        int p, d;
        ~Restore() {
            if (p >= 0 && p != d) cudaSetDevice(p);
        }
    } restore{prev, ctx->device};

    const int64_t N = ctx->N;
    const bool fp64 = ctx->cfg.precision == POND_FP64;
    if (!ctx->adj) {
        AdjointScratch* a = new AdjointScratch();
        ctx->adj = a;
        a->N = N;
        ACK(cudaMalloc(&a->beta_bar, sizeof(double)), "adjoint alloc");
        ACK(cudaMalloc(&a->nu_dev, sizeof(double)), "adjoint alloc");
        ACK(cudaMemsetAsync(a->nu_dev, 0, sizeof(double), ctx->stream), "adjoint alloc");
        ACK(cudaMalloc(&a->minmax, sizeof(double) * 6), "adjoint alloc");
        if (fp64) {
            ACK(cudaMalloc(&a->inv_st, sizeof(double) * N), "adjoint alloc");
            if (ctx_staged(ctx)) {
                // the list and marks of the finer (32 x 4) tiles
                const GridDesc& G0 = ctx->grids_host[0];
                const size_t tiles = ((size_t)(G0.nx + 31) / 32) * (((size_t)G0.ny + 3) / 4);
                ACK(cudaMalloc(&a->org1, sizeof(int) * 2 * 4 * N), "adjoint alloc");
                ACK(cudaMalloc(&a->lw1, sizeof(double) * 2 * 4 * 4 * N), "adjoint alloc");
                const size_t tiles8 = ((size_t)(G0.nx + 31) / 32) * (((size_t)G0.ny + ADJ_TY - 1) / ADJ_TY);
                ACK(cudaMalloc(&a->redo, sizeof(unsigned int) * (1 + 2 * tiles)), "adjoint alloc");
                ACK(cudaMalloc(&a->win, sizeof(double) * ctx->L.q * ADJ_SCATTER_WN * tiles8), "adjoint alloc");
                ACK(cudaMalloc(&a->tiles, sizeof(ScatterTile) * tiles8), "adjoint alloc");
            } else {
                ACK(cudaMalloc(&a->org, sizeof(int2) * 16 * N), "adjoint alloc");
                ACK(cudaMalloc(&a->lw, sizeof(double) * 8 * 16 * N), "adjoint alloc");
            }
            ACK(cudaMalloc(&a->fwd.f, sizeof(double) * 16 * N), "adjoint alloc");
            ACK(cudaMalloc(&a->fwd.ux, sizeof(double) * N), "adjoint alloc");
            ACK(cudaMalloc(&a->fwd.uy, sizeof(double) * N), "adjoint alloc");
            ACK(cudaMalloc(&a->fwd.st, sizeof(double) * N), "adjoint alloc");
            ACK(cudaMalloc(&a->w, sizeof(double) * 16 * N), "adjoint alloc");
            ACK(cudaMalloc(&a->iters, sizeof(int32_t) * N), "adjoint alloc");
            ACK(cudaMalloc(&a->stats, sizeof(DevStats)), "adjoint alloc");
        }
    }
    AdjointScratch* a = ctx->adj;
    if (!fp64) {
        // FP32 populations: pond_adjoint_mixed.cu
        ACK(adjoint_step_mixed(ctx, out_gauge, static_cast<const double*>(f_bar_in),
                               static_cast<const double*>(gauge_bar_in),
                               static_cast<double*>(f_bar_out), static_cast<double*>(gauge_bar_out),
                               a->beta_bar, a->minmax),
            "adjoint (mixed)");
        ACK(accumulate_nu_bar(ctx, a, nu_bar_accum), "adjoint nu cotangent");
        return POND_OK;
    }
    const GridDesc& G = ctx->grids_host[0];
    StateBuf<double> in;
    in.f = static_cast<double*>(ctx->f[ctx->cur]);
    in.ux = ctx->ux[ctx->cur];
    in.uy = ctx->uy[ctx->cur];
    in.st = ctx->st[ctx->cur];
    cudaStream_t s = ctx->stream;

    NvtxRange nv("pond_adjoint_step (FP64)");
    // 1. the fixed point lambda*: the gauge the forward step stores, given by
    //    the caller or recomputed into scratch
    if (out_gauge[0]) {
        ACK(launch_gauge_from_T(out_gauge[0], out_gauge[1], out_gauge[2], a->fwd.ux, a->fwd.uy,
                                a->fwd.st, N, ctx->L.T_L, s),
            "adjoint given gauge");
    } else {
        ACK(launch_ctx_step_fp64(ctx, in, a->fwd, a->iters, a->stats), "adjoint forward");
    }
    // 2. velocity bounds for the transpose gather
    ACK(launch_minmax3(a->fwd.ux, a->fwd.uy, a->fwd.st, N, a->minmax, s), "adjoint bounds");
    ACK(cudaMemcpyAsync(a->host_minmax, a->minmax, sizeof(double) * 6, cudaMemcpyDeviceToHost, s),
        "adjoint bounds copy");
    ACK(cudaMemsetAsync(a->beta_bar, 0, sizeof(double), s), "adjoint reset");
    ACK(cudaStreamSynchronize(s), "adjoint sync");

    AdjArgs A{};
    A.in = in;
    A.ux_s = a->fwd.ux;
    A.uy_s = a->fwd.uy;
    A.st_s = a->fwd.st;
    A.fbar = static_cast<const double*>(f_bar_in);
    A.gbar = static_cast<const double*>(gauge_bar_in);
    A.w = a->w;
    A.fbar_in = static_cast<double*>(f_bar_out);
    A.gbar_in = static_cast<double*>(gauge_bar_out);
    A.beta_bar = a->beta_bar;
    A.org = a->org;
    A.lw = a->lw;
    A.org_x = a->org1;
    A.org_y = a->org1 ? a->org1 + 4 * N : nullptr;
    A.lw_x = a->lw1;
    A.lw_y = a->lw1 ? a->lw1 + 16 * N : nullptr;
    A.inv_st = a->inv_st;
    A.nx = G.nx;
    A.ny = G.ny;
    A.N = N;
    A.beta = ctx->P.beta;
    A.dt = ctx->P.dt;
    A.T_L = ctx->L.T_L;
    const double* mm = a->host_minmax;
    for (int i = 0; i < 4; ++i) {
        const double c = ctx->L.c[i];
        const double slo = c >= 0 ? c * mm[4] : c * mm[5];
        const double shi = c >= 0 ? c * mm[5] : c * mm[4];
        A.vlo_x[i] = slo + mm[0];
        A.vhi_x[i] = shi + mm[1];
        A.vlo_y[i] = slo + mm[2];
        A.vhi_y[i] = shi + mm[3];
    }
    const unsigned nb = (unsigned)((N + ADJ_WARPS - 1) / ADJ_WARPS);
    nvtxRangePushA("adjoint targets + transpose gather");
    if (ctx_staged(ctx)) {
        // phase A in the staged form: a window per tile of targets sized from the bounds of the particle velocities at lambda*
        if (!a->jvp) ACK(cudaMalloc(&a->jvp, sizeof(double) * 4 * 16 * N), "adjoint alloc");
        const double cm = ctx->L.c_max;
        const double sx = (mm[1] - mm[0]) + 2.0 * cm * mm[5];
        const double sy = (mm[3] - mm[2]) + 2.0 * cm * mm[5];
        int sms = 0;
        ACK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device), "SM count");
        ACK(launch_adjoint_phase_a_staged(A, ctx->L.n1, window_extent(sx, A.dt, 2.0) + 5,
                                          window_extent(sy, A.dt, 2.0) + 5, cm, a->jvp, a->redo, sms, s),
            "adjoint targets (staged)");
    } else {
        if (ctx->L.n1 == 3) k_adjoint_targets<3><<<nb, ADJ_WARPS * 32, 0, s>>>(A);
        else k_adjoint_targets<4><<<nb, ADJ_WARPS * 32, 0, s>>>(A);
    }
    ACK(cudaGetLastError(), "adjoint targets");
    if (ctx_staged(ctx)) {
        int sms = 0;
        ACK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device), "SM count");
        ACK(launch_adjoint_phase_b_staged(A, ctx->L.n1, ctx->L.c_max, a->win, a->tiles, a->redo, sms, s),
            "adjoint sources (staged)");
    } else {
        if (ctx->L.n1 == 3) k_adjoint_sources<3><<<nb, ADJ_WARPS * 32, 0, s>>>(A);
        else k_adjoint_sources<4><<<nb, ADJ_WARPS * 32, 0, s>>>(A);
    }
    nvtxRangePop();
    ACK(cudaGetLastError(), "adjoint sources");
    ACK(accumulate_nu_bar(ctx, a, nu_bar_accum), "adjoint nu cotangent");
    return POND_OK;
}

extern "C" pond_status pond_adjoint_nu_bar(pond_ctx* ctx, double* nu_bar) {
    if (!ctx || !nu_bar) {
        if (ctx) ctx->err = "adjoint_nu_bar: NULL argument";
        return POND_ERR_ARG;
    }
    *nu_bar = 0.0;
    AdjointScratch* a = ctx->adj;
    if (!a) return POND_OK;
    DeviceGuard dg(ctx->device);
    ACK(cudaMemcpyAsync(nu_bar, a->nu_dev, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream),
        "adjoint_nu_bar copy");
    ACK(cudaMemsetAsync(a->nu_dev, 0, sizeof(double), ctx->stream), "adjoint_nu_bar reset");
    ACK(cudaStreamSynchronize(ctx->stream), "adjoint_nu_bar sync");
    return POND_OK;
}

extern "C" pond_status pond_adjoint_step(pond_ctx* ctx, const void* f_bar_in,
                                         const void* gauge_bar_in, void* f_bar_out,
                                         void* gauge_bar_out, double* nu_bar_accum) {
    const double* none[3] = {nullptr, nullptr, nullptr};
    return adjoint_step_impl(ctx, none, f_bar_in, gauge_bar_in, f_bar_out, gauge_bar_out,
                             nu_bar_accum);
}

extern "C" pond_status pond_adjoint_step_given(pond_ctx* ctx, const void* ux_out,
                                               const void* uy_out, const void* T_out,
                                               const void* f_bar_in, const void* gauge_bar_in,
                                               void* f_bar_out, void* gauge_bar_out,
                                               double* nu_bar_accum) {
    if (!ctx) return POND_ERR_ARG;
    if (!ux_out || !uy_out || !T_out) {
        ctx->err = "adjoint: NULL output gauge";
        return POND_ERR_ARG;
    }
    const double* given[3] = {static_cast<const double*>(ux_out), static_cast<const double*>(uy_out),
                              static_cast<const double*>(T_out)};
    return adjoint_step_impl(ctx, given, f_bar_in, gauge_bar_in, f_bar_out, gauge_bar_out,
                             nu_bar_accum);
}

extern "C" pond_status pond_adjoint_init(pond_ctx* ctx, const void* f_bar, void* rho_bar) {
    if (!ctx) return POND_ERR_ARG;
    if (!f_bar || !rho_bar || ctx->n_grids != 1) {
        ctx->err = "adjoint_init: NULL argument or batched context";
        return POND_ERR_ARG;
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != ctx->device) cudaSetDevice(ctx->device);
    const long long N = ctx->N;
    const unsigned nb = (unsigned)((N + 255) / 256);
    if (ctx->L.n1 == 3)
        k_rho_bar<3><<<nb, 256, 0, ctx->stream>>>(static_cast<const double*>(f_bar),
                                                   static_cast<double*>(rho_bar), N);
    else
        k_rho_bar<4><<<nb, 256, 0, ctx->stream>>>(static_cast<const double*>(f_bar),
                                                   static_cast<double*>(rho_bar), N);
    const cudaError_t e = cudaGetLastError();
    if (prev >= 0 && prev != ctx->device) cudaSetDevice(prev);
    if (e != cudaSuccess) return adj_fail(ctx, e, "adjoint_init");
    return POND_OK;
}
