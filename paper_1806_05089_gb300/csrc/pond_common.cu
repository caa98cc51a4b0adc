// pond_common.cu -- lattice constants, state initialisation / read-out and
// displacement bounds for the PonD library.
#include <cmath>
#include <cstring>

#include "pond_device.cuh"

namespace pond {

// Lattice constants from their closed forms -- D2Q16: He4 roots and their
// Gauss-Hermite weights; D2Q9: c = -1, 0, 1, W = 1/6, 2/3, 1/6, T_L = 1/3
// (App. A) -- and the Taylor coefficients of the Lagrange basis polynomials
// L_k(x) = prod_{j != k} (x - c_j)/(c_k - c_j) around each speed c_a.
Lattice make_lattice(int kind) {
    Lattice L{};
    if (kind == POND_D2Q9) {
        L.n1 = 3;
        L.c[0] = -1.0;
        L.c[1] = 0.0;
        L.c[2] = 1.0;
        L.w[0] = L.w[2] = 1.0 / 6.0;
        L.w[1] = 2.0 / 3.0;
        L.T_L = 1.0 / 3.0;
    } else {
        const double s6 = std::sqrt(6.0);
        L.n1 = 4;
        L.c[0] = -std::sqrt(3.0 + s6);
        L.c[1] = -std::sqrt(3.0 - s6);
        L.c[2] = std::sqrt(3.0 - s6);
        L.c[3] = std::sqrt(3.0 + s6);
        L.w[0] = L.w[3] = (3.0 - s6) / 12.0;
        L.w[1] = L.w[2] = (3.0 + s6) / 12.0;
        L.T_L = 1.0;
    }
    const int n1 = L.n1;
    L.q = n1 * n1;
    L.c_max = L.c[n1 - 1];
    for (int k = 0; k < n1; ++k) {
        double p[4] = {1.0, 0.0, 0.0, 0.0};  // coefficients of x^0..x^3
        double den = 1.0;
        for (int j = 0; j < n1; ++j) {
            if (j == k) continue;
            double np[4] = {0.0, 0.0, 0.0, 0.0};
            for (int i = 0; i < 4; ++i) {
                if (i + 1 < 4) np[i + 1] += p[i];
                np[i] -= L.c[j] * p[i];
            }
            for (int i = 0; i < 4; ++i) p[i] = np[i];
            den *= (L.c[k] - L.c[j]);
        }
        for (int i = 0; i < 4; ++i) p[i] /= den;
        for (int a = 0; a < n1; ++a) {
            const double x = L.c[a];
            L.d1[k][a] = p[1] + 2.0 * p[2] * x + 3.0 * p[3] * x * x;
            L.d2[k][a] = p[2] + 3.0 * p[3] * x;
        }
        L.d3[k] = p[3];
    }
    // W-dual basis of {1, |c|^2}: inverse of [[1, 2 T_L], [2 T_L, g]]
    double K4 = 0.0;
    for (int a = 0; a < n1; ++a) K4 += L.w[a] * L.c[a] * L.c[a] * L.c[a] * L.c[a];
    const double g = 2.0 * K4 + 2.0 * L.T_L * L.T_L;
    const double det = g - 4.0 * L.T_L * L.T_L;
    L.pe0 = g / det;
    L.pe2 = -2.0 * L.T_L / det;
    L.pt0 = -2.0 * L.T_L / det;
    L.pt2 = 1.0 / det;
    L.inv_TL = 1.0 / L.T_L;
    return L;
}

LatticeF to_float(const Lattice& L) {
    LatticeF F{};
    for (int i = 0; i < 4; ++i) {
        F.c[i] = (float)L.c[i];
        F.w[i] = (float)L.w[i];
        F.d3[i] = (float)L.d3[i];
        for (int j = 0; j < 4; ++j) {
            F.d1[i][j] = (float)L.d1[i][j];
            F.d2[i][j] = (float)L.d2[i][j];
        }
    }
    F.pe0 = (float)L.pe0;
    F.pe2 = (float)L.pe2;
    F.pt0 = (float)L.pt0;
    F.pt2 = (float)L.pt2;
    F.inv_TL = (float)L.inv_TL;
    return F;
}

// FP64 <-> FP32 on the integer pipe.  The conversion instructions share the
// FP64 pipe (2 a clock and SM), which held the state I/O below at a third of
// the memory rate.  Exact; to FP32 rounded to nearest even.  Zeros, FP32
// subnormals, infinities and NaN take the instruction.
__device__ __forceinline__ double widen(float v) {
    const unsigned int b = __float_as_uint(v);
    if ((b & 0x7f800000u) - 0x00800000u >= 0x7f000000u) return (double)v;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))),
                            (int)(b << 29));
}

__device__ __forceinline__ float narrow(double v) {
    const unsigned int hi = (unsigned int)__double2hiint(v), lo = (unsigned int)__double2loint(v);
    const unsigned int e = hi >> 20 & 0x7ffu;
    if (e - 897u >= 253u) return (float)v;
    const unsigned int m = (e - 896u) << 23 | (hi & 0xfffffu) << 3 | lo >> 29;
    // the first bit below, and a tie to even
    const unsigned int up = (lo >> 28 & 1u) & (((lo & 0x0fffffffu) | (m & 1u)) != 0u ? 1u : 0u);
    return __uint_as_float((hi & 0x80000000u) | (m + up));
}
__device__ __forceinline__ double widen(double v) { return v; }
template <typename Real>
__device__ __forceinline__ Real narrow_to(double v) {
    if constexpr (sizeof(Real) == 4) return narrow(v);
    else return v;
}

__device__ __forceinline__ bool finite_bits(double v) {
    return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}

// Order-preserving encoding of a float, larger for a larger value; never 0 for
// a number, so that a zeroed word is below all.
__device__ __forceinline__ unsigned int f2ord(float f) {
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Block reduction of the particle-velocity bounds {min x, max x, min y, max y}
// and of the count of bad nodes into out5: the maxima encoded by f2ord, the
// minima as the complement of it (all five words start at zero; decode_bounds
// reads them).  Warp, then block: one atomic per block and value, as atomics on
// one address serialise.  All threads of the block take part.
__device__ __forceinline__ void reduce_bounds(float lo_x, float hi_x, float lo_y, float hi_y,
                                              unsigned int bad, unsigned int* out5) {
    __shared__ float s_b[4][32];
    __shared__ unsigned int s_bad[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int pass = 0; pass < 2; ++pass) {
        for (int o = 16; o > 0; o >>= 1) {
            lo_x = fminf(lo_x, __shfl_xor_sync(0xffffffffu, lo_x, o));
            hi_x = fmaxf(hi_x, __shfl_xor_sync(0xffffffffu, hi_x, o));
            lo_y = fminf(lo_y, __shfl_xor_sync(0xffffffffu, lo_y, o));
            hi_y = fmaxf(hi_y, __shfl_xor_sync(0xffffffffu, hi_y, o));
        }
        bad = __reduce_add_sync(0xffffffffu, bad);
        if (pass == 1) break;
        if (lane == 0) {
            s_b[0][warp] = lo_x;
            s_b[1][warp] = hi_x;
            s_b[2][warp] = lo_y;
            s_b[3][warp] = hi_y;
            s_bad[warp] = bad;
        }
        __syncthreads();
        if (warp != 0) return;
        const bool in = lane < (int)(blockDim.x >> 5);
        lo_x = in ? s_b[0][lane] : 3.0e38f;
        hi_x = in ? s_b[1][lane] : -3.0e38f;
        lo_y = in ? s_b[2][lane] : 3.0e38f;
        hi_y = in ? s_b[3][lane] : -3.0e38f;
        bad = in ? s_bad[lane] : 0u;
    }
    if (lane == 0) {
        atomicMax(out5 + 0, ~f2ord(lo_x));
        atomicMax(out5 + 1, f2ord(hi_x));
        atomicMax(out5 + 2, ~f2ord(lo_y));
        atomicMax(out5 + 3, f2ord(hi_y));
        if (bad) atomicAdd(out5 + 4, bad);
    }
}

void decode_bounds(const unsigned int in5[5], float out4[4], unsigned int* bad) {
    for (int i = 0; i < 4; ++i) {
        const unsigned int u = (i & 1) ? in5[i] : ~in5[i];
        const unsigned int b = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
        std::memcpy(&out4[i], &b, sizeof b);
    }
    *bad = in5[4];
}

// f_q = rho W_q in the node's own gauge (Eq. equilibrium), or a copy of the
// given FP64 populations; T -> sqrt(theta).  The same pass bounds the particle
// velocities (in FP32: they size the staged windows, which have a node of
// margin) and counts the nodes with T <= 0 or a non-finite gauge, into out5.
// Of FP64 arithmetic a node needs the root, 2 + 4 products (the weights take two
// values per dimension) and, on D2Q9, the division by T_L: 2048^2 mixed, with
// the former pass for the bounds, 597 -> 185 us.
template <typename Real, int N1>
__global__ void __launch_bounds__(256)
k_init_state(const double* __restrict__ rho, const double* __restrict__ ux,
             const double* __restrict__ uy, const double* __restrict__ T,
             const double* __restrict__ f_given, StateBuf<Real> st, int64_t N, int64_t plane,
             Lattice L, unsigned int* __restrict__ out5) {
    constexpr int Q = N1 * N1;
    float lo_x = 3.0e38f, hi_x = -3.0e38f, lo_y = 3.0e38f, hi_y = -3.0e38f;
    unsigned int bad = 0u;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) {
        const double x = ux[i], y = uy[i];
        const double t = sqrt(N1 == 4 ? T[i] : T[i] / L.T_L);  // T_L = 1 on D2Q16
        st.ux[i] = x;
        st.uy[i] = y;
        st.st[i] = t;
        if (f_given) {
#pragma unroll
            for (int q = 0; q < Q; ++q) st.f[q * plane + i] = narrow_to<Real>(f_given[q * N + i]);
        } else {
            // populations (k, l) by the classes of k and l: inner, outer speed
            const double r = rho[i], ri = r * L.w[1], ro = r * L.w[0];
            const Real ii = narrow_to<Real>(ri * L.w[1]), io = narrow_to<Real>(ri * L.w[0]);
            const Real oi = narrow_to<Real>(ro * L.w[1]), oo = narrow_to<Real>(ro * L.w[0]);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const bool ko = q / N1 == 0 || q / N1 == N1 - 1, lo = q % N1 == 0 || q % N1 == N1 - 1;
                st.f[q * plane + i] = ko ? (lo ? oo : oi) : (lo ? io : ii);
            }
        }
        bad = __double2hiint(t) >= 0 && t != 0.0 && finite_bits(t) && finite_bits(x) && finite_bits(y) ? 0u : 1u;
        const float xf = narrow(x), yf = narrow(y), s = (float)L.c_max * narrow(t);
        lo_x = xf - s;
        hi_x = xf + s;
        lo_y = yf - s;
        hi_y = yf + s;
    }
    reduce_bounds(lo_x, hi_x, lo_y, hi_y, bad, out5);
}

template <typename Real>
cudaError_t launch_init_state(const double* rho, const double* ux, const double* uy,
                              const double* T, const double* f_given, StateBuf<Real> st,
                              int64_t N, int64_t plane, const Lattice& L, unsigned int* out5,
                              cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out5, 0, 5 * sizeof(unsigned int), s);
    if (e != cudaSuccess || N == 0) return e;
    const int bs = 256;
    const unsigned nb = (unsigned)((N + bs - 1) / bs);
    if (L.n1 == 4)
        k_init_state<Real, 4><<<nb, bs, 0, s>>>(rho, ux, uy, T, f_given, st, N, plane, L, out5);
    else
        k_init_state<Real, 3><<<nb, bs, 0, s>>>(rho, ux, uy, T, f_given, st, N, plane, L, out5);
    return cudaGetLastError();
}

// Bound by memory: the density's sum (16 dependent FP64 additions) is formed
// only where it is asked for, and FP32 populations are widened on the integer
// pipe.  2048^2 mixed, populations and gauge: 271 -> 148 us (6.8 TB/s).
template <typename Real, int N1, bool RHO>
__global__ void __launch_bounds__(256)
k_read_state(StateBuf<Real> st, int64_t N, int64_t plane, double* __restrict__ rho,
             double* __restrict__ ux, double* __restrict__ uy, double* __restrict__ T,
             double* __restrict__ f, double T_L) {
    constexpr int Q = N1 * N1;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    if (RHO || f) {
        double r = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const double v = widen(st.f[q * plane + i]);
            if (RHO) r += v;
            if (f) f[q * N + i] = v;
        }
        if (RHO) rho[i] = r;
    }
    if (ux) ux[i] = st.ux[i];
    if (uy) uy[i] = st.uy[i];
    if (T) {
        const double s = st.st[i];
        T[i] = s * s * T_L;
    }
}

template <typename Real>
cudaError_t launch_read_state(StateBuf<Real> st, int64_t N, int64_t plane, double* rho,
                              double* ux, double* uy, double* T, double* f, const Lattice& L,
                              cudaStream_t s) {
    if (N == 0) return cudaSuccess;
    const int bs = 256;
    const unsigned nb = (unsigned)((N + bs - 1) / bs);
    if (L.n1 == 4) {
        if (rho) k_read_state<Real, 4, true><<<nb, bs, 0, s>>>(st, N, plane, rho, ux, uy, T, f, L.T_L);
        else k_read_state<Real, 4, false><<<nb, bs, 0, s>>>(st, N, plane, rho, ux, uy, T, f, L.T_L);
    } else {
        if (rho) k_read_state<Real, 3, true><<<nb, bs, 0, s>>>(st, N, plane, rho, ux, uy, T, f, L.T_L);
        else k_read_state<Real, 3, false><<<nb, bs, 0, s>>>(st, N, plane, rho, ux, uy, T, f, L.T_L);
    }
    return cudaGetLastError();
}

template cudaError_t launch_init_state<double>(const double*, const double*, const double*,
                                               const double*, const double*, StateBuf<double>,
                                               int64_t, int64_t, const Lattice&, unsigned int*,
                                               cudaStream_t);
template cudaError_t launch_init_state<float>(const double*, const double*, const double*,
                                              const double*, const double*, StateBuf<float>,
                                              int64_t, int64_t, const Lattice&, unsigned int*,
                                              cudaStream_t);
template cudaError_t launch_read_state<double>(StateBuf<double>, int64_t, int64_t, double*,
                                               double*, double*, double*, double*,
                                               const Lattice&, cudaStream_t);
template cudaError_t launch_read_state<float>(StateBuf<float>, int64_t, int64_t, double*,
                                              double*, double*, double*, double*,
                                              const Lattice&, cudaStream_t);

// Bounds of the particle velocities over a grid, from the FP64 values.
__global__ void k_disp_bounds(const double* __restrict__ ux, const double* __restrict__ uy,
                              const double* __restrict__ st, int64_t N, double cmax,
                              unsigned int* out5) {
    float lo_x = 3.0e38f, hi_x = -3.0e38f, lo_y = 3.0e38f, hi_y = -3.0e38f;
    unsigned int bad = 0u;  // nodes with s <= 0 or a non-finite gauge
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double x = ux[i], y = uy[i], t = st[i];
        bad += (t > 0.0 && isfinite(t) && isfinite(x) && isfinite(y)) ? 0u : 1u;
        const double s = cmax * t;
        lo_x = fminf(lo_x, (float)(x - s));
        hi_x = fmaxf(hi_x, (float)(x + s));
        lo_y = fminf(lo_y, (float)(y - s));
        hi_y = fmaxf(hi_y, (float)(y + s));
    }
    reduce_bounds(lo_x, hi_x, lo_y, hi_y, bad, out5);
}

// Halo strips of a domain decomposition: a rectangle of the state to or from
// a contiguous device buffer.  The stored representation moves unchanged
// (populations widened to FP64 exactly, the gauge as stored), so a state
// split over sub-domains and reassembled is bit-identical.
template <typename Real>
__global__ void k_pack_rect(StateBuf<Real> st, int nx, int x0, int y0, int w, int h, int q,
                            long long plane, double* __restrict__ buf) {
    const long long n = (long long)w * h;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long long node = (long long)(y0 + i / w) * nx + x0 + i % w;
    for (int c = 0; c < q; ++c) buf[c * n + i] = (double)st.f[c * plane + node];
    buf[q * n + i] = st.ux[node];
    buf[(q + 1) * n + i] = st.uy[node];
    buf[(q + 2) * n + i] = st.st[node];
}

template <typename Real>
__global__ void k_unpack_rect(StateBuf<Real> st, int nx, int x0, int y0, int w, int h, int q,
                              long long plane, const double* __restrict__ buf) {
    const long long n = (long long)w * h;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long long node = (long long)(y0 + i / w) * nx + x0 + i % w;
    for (int c = 0; c < q; ++c) st.f[c * plane + node] = (Real)buf[c * n + i];
    st.ux[node] = buf[q * n + i];
    st.uy[node] = buf[(q + 1) * n + i];
    st.st[node] = buf[(q + 2) * n + i];
}

template <typename Real>
cudaError_t launch_pack_rect(StateBuf<Real> st, int nx, int x0, int y0, int w, int h, int q,
                             int64_t plane, double* buf, cudaStream_t s) {
    const long long n = (long long)w * h;
    if (n == 0) return cudaSuccess;
    k_pack_rect<Real><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(st, nx, x0, y0, w, h, q, plane, buf);
    return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_unpack_rect(StateBuf<Real> st, int nx, int x0, int y0, int w, int h, int q,
                               int64_t plane, const double* buf, cudaStream_t s) {
    const long long n = (long long)w * h;
    if (n == 0) return cudaSuccess;
    k_unpack_rect<Real><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(st, nx, x0, y0, w, h, q, plane, buf);
    return cudaGetLastError();
}

template cudaError_t launch_pack_rect<double>(StateBuf<double>, int, int, int, int, int, int,
                                              int64_t, double*, cudaStream_t);
template cudaError_t launch_pack_rect<float>(StateBuf<float>, int, int, int, int, int, int,
                                             int64_t, double*, cudaStream_t);
template cudaError_t launch_unpack_rect<double>(StateBuf<double>, int, int, int, int, int, int,
                                                int64_t, const double*, cudaStream_t);
template cudaError_t launch_unpack_rect<float>(StateBuf<float>, int, int, int, int, int, int,
                                               int64_t, const double*, cudaStream_t);

cudaError_t launch_disp_bounds(const double* ux, const double* uy, const double* st, int64_t N,
                               double c_max, unsigned int* out5, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out5, 0, 5 * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    const int bs = 256;
    int64_t nb = (N + bs - 1) / bs;
    if (nb > 256) nb = 256;
    if (nb < 1) nb = 1;
    k_disp_bounds<<<(unsigned)nb, bs, 0, s>>>(ux, uy, st, N, c_max, out5);
    return cudaGetLastError();
}

}  // namespace pond
