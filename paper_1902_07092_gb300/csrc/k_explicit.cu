// Explicit stage of one IMEX step (Sections 2, 3 and 3.2 of Gastine, pizza,
// GJI 2019): spectral -> radial grid per azimuthal mode m, grid products per
// radius, radial grid -> integrated right-hand sides per m.
//
// Layouts (double2 = complex):
//   state   Psi_hat, theta_hat  [M][nc]  (paper f_hat convention, Eq. cheb)
//   G1      [n_r][4][M]  radial-grid Fourier coefficients of
//           v = dPsi/dphi, u_phi, omega, theta            (radius-major)
//   G2      [n_r][4][M]  Fourier coefficients of the products
//           v*omega, u_phi*omega, v*theta, u_phi*theta     (radius-major)
//   e       [M][nc] integrated explicit right-hand sides
// The change from mode-major to radius-major order (the paper's MPI transpose)
// is folded into the stores of spec_to_grid and the loads of grid_to_spec.
#include <algorithm>

#include "device_common.cuh"
#include "fixfft.cuh"

namespace pz {

namespace {

constexpr int NTHREADS_R = 256;  // radial kernels
constexpr int MAXPER = 12;       // azimuthal points per thread held in registers

__device__ __forceinline__ int g_index(int k, int f, int m, int M) { return (k * 4 + f) * M + m; }

// number of radial transforms batched together in shared memory (the
// autotuner's choice, else four in FP64 up to n_r = 257 -- all four synthesised
// fields of a mode in one pass -- and two in FP32 and at n_r = 513: measured
// fastest at n_r = 257 and, 99 against 107 us for a1 at 513 x 1536, at 513)
__host__ __device__ inline int radial_batch(const StepParams& P) {
    if (P.nb_r > 0) return P.nb_r;
    if (2 * P.K > 1024) return 1;
    return (P.fp32 || P.K > 256) ? 2 : 4;
}
// threads of the per-radius azimuthal kernels
inline int phi_threads(const StepParams& P) {
    if (P.phi_threads > 0) return P.phi_threads;
    return P.n_phi > 256 * MAXPER ? 512 : 256;
}

// of the fixed-point one: a divisor of the n_phi/2 radix-4 butterflies of a pass over
// both pairs (96 2^j of them), at most 384 (two CTAs share an SM's registers); 512 where
// shared memory leaves one CTA an SM (1025 x 3072: 336 -> 327 us)
inline int phi_threads_fx(const StepParams& P) {
    if (P.phi_threads > 0 || P.n_phi > 256 * MAXPER) return phi_threads(P);
    return P.n_phi >= 3072 ? 512 : P.n_phi >= 768 ? 384 : 192;
}

// ---------------------------------------------------------------------------
// K1: per m, Chebyshev coefficients -> values on the Gauss-Lobatto grid.
//   v = i m Psi,  u_phi = -h^2 Psi' + 3 s Psi,
//   omega = -[h^2 Psi'' + (h^2/s - 5 s) Psi' - (6 + m^2 h^2/s^2) Psi]   (m >= 1)
//   m = 0:  v = 0, u_phi = u_bar, omega = u_bar' + u_bar/s
// (Section 3.2: u_s = (h^2/s) dPsi/dphi, u_phi = u_bar - h^2 dPsi/ds + 3 s Psi,
//  omega = (1/s) d(s u_bar)/ds - L_I Psi.)
// u_phi and omega are built up over the passes of Psi, Psi' and Psi''.  Their partial
// sums wait in W[m][2][n_r] (contiguous for a mode; the grid array's columns are
// strided by 4 M entries, and rereading and rewriting those took 175 of the 305
// thousand cycles of a mode at 2049 x 6144): the grid array is only written, once.
// With Ekman pumping it also writes P.pump_F[m][k]: for m >= 1 the approximate
// pumping of Eq. approx_pump,
//   F_eps = Ups_eps [ -omega + (s/2) Psi' - (3 s^2/(2 h_eps^2) + m^2 + i m 5 s_o/(2 h_eps)) Psi ]
// (L_I Psi = -omega), built up over the passes of Psi, Psi' and omega; for m = 0
// the zonal-flow terms Ups_eps u_bar (1 + (E/2) omega_0) of Eqs. uphi_int and
// uphicoll.
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(NTHREADS_R) k_spec_to_grid(StepParams P, VecSet y, T* __restrict__ G1, T* __restrict__ W) {
    chain_wait();
    using RT = typename Cx<T>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    T* sm = reinterpret_cast<T*>(smraw);
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, L = 2 * K, N = P.n_r, nc = P.nc, M = P.M;
    const int NB = radial_batch(P);
    T* bufA = sm;
    T* bufB = bufA + NB * L;
    T* cc0 = bufB + NB * L;  // Psi (or u_bar) plain coefficients, length N
    T* cc1 = cc0 + N;        // first derivative
    T* cc2 = cc1 + N;        // second derivative
    const int tid = threadIdx.x, nth = blockDim.x;
    // C w_n of Eq. cheb in the working precision (the state is converted first)
    const RT Cw = (RT)P.cnorm, Cw0 = (RT)(0.5 * P.cnorm);

    for (int n = tid; n < N; n += nth) {
        T a = Cx<T>::make(0.0, 0.0);
        if (n < nc) {
            const RT w = (n == 0) ? Cw0 : Cw;
            if (m > 0)
                a = cscale(Cx<T>::from(y.psi[(size_t)m * nc + n]), w);
            else
                a = Cx<T>::make((RT)y.u[n] * w, 0.0);
        }
        cc0[n] = a;
    }
    __syncthreads();
    cheb_derivative_scan(cc0, cc1, bufA, N, P.inv_a);
    if (m > 0) cheb_derivative_scan(cc1, cc2, bufA, N, P.inv_a);

    // field list: 0 Psi, 1 Psi', 2 Psi'', 3 theta, 4 packed u_bar + i lam u_bar'
    // (lam a power of two balancing the two parts).  The reduction's 16 doubles
    // live in bufB (at least 128 bytes: n_r >= 9), unused until the first
    // transform: without static shared memory two FP32 CTAs fit an SM at
    // n_r = 2049.
    RT lam = 1;
    if (m == 0) {
        double* red = reinterpret_cast<double*>(bufB);  // [warp][2]
        double a0 = 0.0, a1 = 0.0;
        for (int i = tid; i < N; i += nth) {
            a0 = fmax(a0, (double)(fabs(cc0[i].x) + fabs(cc0[i].y)));
            a1 = fmax(a1, (double)(fabs(cc1[i].x) + fabs(cc1[i].y)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a0 = fmax(a0, __shfl_xor_sync(0xffffffffu, a0, o));
            a1 = fmax(a1, __shfl_xor_sync(0xffffffffu, a1, o));
        }
        const int w = tid >> 5;
        if ((tid & 31) == 0) {
            red[2 * w] = a0;
            red[2 * w + 1] = a1;
        }
        __syncthreads();
        double r0 = 0.0, r1 = 0.0;
        for (int q = 0; q < (nth >> 5); ++q) {
            r0 = fmax(r0, red[2 * q]);
            r1 = fmax(r1, red[2 * q + 1]);
        }
        lam = (RT)pow2_ratio(r0, r1);
    }
    int fields[4];
    int nf;
    if (m > 0) {
        fields[0] = 0; fields[1] = 1; fields[2] = 2; fields[3] = 3; nf = 4;
    } else {
        fields[0] = 4; fields[1] = 3; nf = 2;
    }
    const RT dm = (RT)m;
    T* PF = P.pump ? reinterpret_cast<T*>(P.pump_F) + (size_t)m * N : nullptr;
    T* wu = W + (size_t)m * 2 * N;
    T* wo = wu + N;
    for (int f0 = 0; f0 < nf; f0 += NB) {
        const int nb = min(NB, nf - f0);
        for (int b = 0; b < nb; ++b) {
            const int fid = fields[f0 + b];
            T* z = bufA + b * L;
            for (int j = tid; j <= K; j += nth) {
                T v;
                if (fid == 0) v = cc0[j];
                else if (fid == 1) v = cc1[j];
                else if (fid == 2) v = cc2[j];
                else if (fid == 3)
                    v = (j < nc) ? cscale(Cx<T>::from(y.th[(size_t)m * nc + j]), (j == 0) ? Cw0 : Cw)
                                 : Cx<T>::make(0.0, 0.0);
                else {
                    v.x = cc0[j].x;
                    v.y = lam * cc1[j].x;
                }
                if (j == 0 || j == K) v = cscale(v, (RT)2);
                even_extend_store(z, K, j, v);
            }
        }
        T* R = radial_dct1(bufA, bufB, P, nb);
        for (int b = 0; b < nb; ++b) {
            const int fid = fields[f0 + b];
            const T* Z = R + b * L;
            for (int k = tid; k < N; k += nth) {
                const T g = cscale(Z[k], (RT)0.5);  // value of the series at x_k
                const RT s = Tab<T>::s(P, k), h2 = Tab<T>::h2(P, k), is = Tab<T>::is(P, k);
                T* out = G1 + g_index(k, 0, m, M);
                // out[0] = v, out[M] = u_phi, out[2M] = omega, out[3M] = theta
                if (fid == 0) {
                    out[0] = cmul_i(g, dm);
                    wu[k] = cscale(g, (RT)3 * s);
                    wo[k] = cscale(g, (RT)6 + dm * dm * h2 * is * is);
                    if (PF) {
                        const RT U = (RT)P.pump_ups[k];
                        PF[k] = cadd(cscale(g, -U * ((RT)P.pump_cr[k] + dm * dm)), cmul_i(g, -U * dm * (RT)P.pump_ci[k]));
                    }
                } else if (fid == 1) {
                    out[M] = csub(wu[k], cscale(g, h2));
                    wo[k] = csub(wo[k], cscale(g, h2 * is - (RT)5 * s));
                    if (PF) PF[k] = cadd(PF[k], cscale(g, (RT)P.pump_ups[k] * (RT)0.5 * s));
                } else if (fid == 2) {
                    const T om = csub(wo[k], cscale(g, h2));
                    out[2 * M] = om;
                    if (PF) PF[k] = csub(PF[k], cscale(om, (RT)P.pump_ups[k]));
                } else if (fid == 3) {
                    out[3 * M] = g;
                } else {
                    out[0] = Cx<T>::make(0.0, 0.0);
                    out[M] = Cx<T>::make(g.x, 0.0);
                    out[2 * M] = Cx<T>::make(g.y / lam + g.x * is, 0.0);
                    if (PF) {
                        const RT w0 = g.y / lam + g.x * is;
                        PF[k] = Cx<T>::make((RT)P.pump_ups[k] * g.x * ((RT)1 + (RT)(0.5 * P.E) * w0), 0.0);
                    }
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// K2: per radius, Eq. fft to the N_phi-point azimuthal grid, the four products,
// Eq. ifft back (modes m <= N_m kept).  Two real fields travel in one complex
// transform: g1 = v + i u_phi, g2 = omega + i theta; then
//   g1 * Re(g2) = v omega + i u_phi omega,  g1 * Im(g2) = v theta + i u_phi theta.
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ void load_packed_spectrum(T* Z, const T* src, int M, int Pn, int n_m,
                                                     typename Cx<T>::R sa, typename Cx<T>::R sb) {
    // src points at G1/G2 row (k, f): field a = src[0..M), field b = src[M..2M);
    // packed as sa a + i sb b
    for (int j = threadIdx.x; j < Pn; j += blockDim.x) {
        T z = Cx<T>::make(0.0, 0.0);
        if (j == 0) {
            z.x = sa * src[0].x;
            z.y = sb * src[M].x;
        } else if (j <= n_m) {
            const T a = cscale(src[j], sa), b = cscale(src[M + j], sb);
            z.x = a.x - b.y;  // a + i b
            z.y = a.y + b.x;
        } else if (j >= Pn - n_m) {
            const int mm = Pn - j;
            const T a = cscale(src[mm], sa), b = cscale(src[M + mm], sb);
            z.x = a.x + b.y;  // conj(a) + i conj(b)
            z.y = -a.y + b.x;
        }
        Z[j] = z;
    }
}

// Split the transform Y of a + i b (a, b real fields) into the spectra of a and
// b, scaled by ia and ib (1/Pn times the inverse packing weights).
template <class T>
__device__ __forceinline__ void store_split_spectrum(const T* Y, T* __restrict__ dst, int M, int Pn, int n_m,
                                                     typename Cx<T>::R ia, typename Cx<T>::R ib) {
    using RT = typename Cx<T>::R;
    const RT h = (RT)0.5;
    for (int m = threadIdx.x; m <= n_m; m += blockDim.x) {
        T a, b;
        if (m == 0) {
            a = Cx<T>::make(Y[0].x * ia, 0.0);
            b = Cx<T>::make(Y[0].y * ib, 0.0);
        } else {
            const T y1 = Y[m], y2 = Y[Pn - m];
            // a = (y1 + conj(y2))/2,  b = (y1 - conj(y2))/(2i)
            a.x = h * (y1.x + y2.x) * ia;
            a.y = h * (y1.y - y2.y) * ia;
            b.x = h * (y1.y + y2.y) * ib;
            b.y = -h * (y1.x - y2.x) * ib;
        }
        dst[m] = a;
        dst[M + m] = b;
    }
}

// exact powers of two in the working precision; balancing exponents are
// limited further in FP32 (exponent range of float)
template <class T>
struct P2;
template <>
struct P2<double2> {
    static constexpr int lim = 400;
    __device__ static double v(int e) { return pow2d(e); }
};
template <>
struct P2<float2> {
    static constexpr int lim = 40;
    __device__ static float v(int e) { return pow2f(e); }
};

// Courant rates of Eq. cfl at radius k from the synthesised packed pair
// g1 = v + i l1 u_phi on the n_phi points (v = d Psi/d phi, u_s = (h^2/s) v in
// the integration formulation, v/s in collocation): max |u_s|/ds_k and
// max |u_phi|/(s_k dphi), folded into P.cfl_max[0..1] as atomic maxima of their
// bit patterns (non-negative doubles order like their bits).  Called by every
// thread of the block; uses red[0 .. 2 * warps).
__device__ __forceinline__ double re_abs(float2 z) { return fabs((double)z.x); }
__device__ __forceinline__ double im_abs(float2 z) { return fabs((double)z.y); }
__device__ __forceinline__ double re_abs(double2 z) { return fabs(z.x); }
__device__ __forceinline__ double im_abs(double2 z) { return fabs(z.y); }

template <class T>
__device__ void cfl_rates(const StepParams& P, const T* R, int Pn, double l1, int k, double* red) {
    double a = 0.0, b = 0.0;
    for (int j = threadIdx.x; j < Pn; j += blockDim.x) {
        a = fmax(a, re_abs(R[j]));
        b = fmax(b, im_abs(R[j]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = fmax(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[2 * w] = a;
        red[2 * w + 1] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < nw; ++i) {
            a = fmax(a, red[2 * i]);
            b = fmax(b, red[2 * i + 1]);
        }
        const double s = P.s[k];
        const double fs = P.coll ? 1.0 / s : P.h2[k] / s;
        const double rs = fs * a / P.cfl_ds[k];
        const double rp = b / l1 / (s * P.cfl_dphi);
        atomicMax(reinterpret_cast<unsigned long long*>(P.cfl_max), (unsigned long long)__double_as_longlong(rs));
        atomicMax(reinterpret_cast<unsigned long long*>(P.cfl_max + 1),
                  (unsigned long long)__double_as_longlong(rp));
    }
    __syncthreads();
}

template <class T>
__global__ void __launch_bounds__(512, 1) k_phi_products(StepParams P, const T* G1,
                                                         T* __restrict__ G2, int pair) {
    chain_wait();
    using RT = typename Cx<T>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    T* sm = reinterpret_cast<T*>(smraw);
    const int k = P.k_lo + blockIdx.x;
    const int Pn = P.n_phi, M = P.M, n_m = P.n_m;
    T* X = sm;
    T* Y = sm + Pn;
    const int tid = threadIdx.x, nth = blockDim.x;
    T reg[MAXPER];
    // exact power-of-two weights that balance the packed pairs:
    // g1 = v + i l1 u_phi, g2 = omega + i l2 theta
    __shared__ double red[4 * 32], mx[4];
    block_max_abs(G1 + g_index(k, 0, 0, M), M, 4, n_m + 1, mx, red);
    const int e1 = pow2_exponent(mx[0], mx[1], P2<T>::lim), e2 = pow2_exponent(mx[2], mx[3], P2<T>::lim);
    const RT l1 = P2<T>::v(e1), l2 = P2<T>::v(e2);
    const RT iP = (RT)P.inv_nphi;  // 1/n_phi, a power of two divided by 3

    if (pair) {
        // both packed pairs in one batched transform each way (X, Y hold 2 Pn)
        Y = X + 2 * Pn;
        load_packed_spectrum(X, G1 + g_index(k, 0, 0, M), M, Pn, n_m, (RT)1, l1);
        load_packed_spectrum(X + Pn, G1 + g_index(k, 2, 0, M), M, Pn, n_m, (RT)1, l2);
        T* R = fft_batched<+1>(X, Y, P.plan_p, 2);
        if (P.cfl_max) cfl_rates(P, R, Pn, (double)l1, k, red);
        T* O = (R == X) ? Y : X;
        for (int j = tid; j < Pn; j += nth) {
            const T g1 = R[j], g2 = R[Pn + j];
            O[j] = cscale(g1, g2.x);
            O[Pn + j] = cscale(g1, g2.y);
        }
        T* S = fft_batched<-1>(O, R, P.plan_p, 2);
        store_split_spectrum(S, G2 + g_index(k, 0, 0, M), M, Pn, n_m, iP, iP * P2<T>::v(-e1));
        store_split_spectrum(S + Pn, G2 + g_index(k, 2, 0, M), M, Pn, n_m, iP * P2<T>::v(-e2),
                             iP * P2<T>::v(-e1 - e2));
        return;
    }
    load_packed_spectrum(X, G1 + g_index(k, 0, 0, M), M, Pn, n_m, (RT)1, l1);
    T* R = fft_batched<+1>(X, Y, P.plan_p, 1);
    if (P.cfl_max) cfl_rates(P, R, Pn, (double)l1, k, red);
#pragma unroll
    for (int i = 0; i < MAXPER; ++i) {
        const int j = tid + i * nth;
        if (j < Pn) reg[i] = R[j];
    }
    __syncthreads();
    load_packed_spectrum(X, G1 + g_index(k, 2, 0, M), M, Pn, n_m, (RT)1, l2);
    R = fft_batched<+1>(X, Y, P.plan_p, 1);
#pragma unroll
    for (int i = 0; i < MAXPER; ++i) {
        const int j = tid + i * nth;
        if (j < Pn) {
            const T g2 = R[j], g1 = reg[i];
            R[j] = cscale(g1, g2.x);
            reg[i] = cscale(g1, g2.y);
        }
    }
    T* other = (R == X) ? Y : X;
    T* S = fft_batched<-1>(R, other, P.plan_p, 1);
    // g1 Re(g2) = v omega + i l1 u_phi omega
    store_split_spectrum(S, G2 + g_index(k, 0, 0, M), M, Pn, n_m, iP, iP * P2<T>::v(-e1));
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MAXPER; ++i) {
        const int j = tid + i * nth;
        if (j < Pn) X[j] = reg[i];
    }
    S = fft_batched<-1>(X, Y, P.plan_p, 1);
    // g1 Im(g2) = l2 (v theta + i l1 u_phi theta)
    store_split_spectrum(S, G2 + g_index(k, 2, 0, M), M, Pn, n_m, iP * P2<T>::v(-e2), iP * P2<T>::v(-e1 - e2));
}

// ---------------------------------------------------------------------------
// K3: per m, radial divergences of the fluxes, Eq. icheb, truncation to n < N_c
// (dealiasing), and the integrated right-hand sides
//   N_omega = (1/s) d/ds(h^2 [v omega]_m) + (i m/s) [u_phi omega]_m
//   N_theta = (1/s) d/ds(h^2 [v theta]_m) + (i m/s) [u_phi theta]_m - [v theta]_m
//   N_u     = (h^2/s) [v omega]_0
//   e_psi   = C^I [ (Ra/Pr)(i m/s_o) theta_hat_m + N_omega_hat ]        (m >= 1)
//   e_theta = -D^I N_theta_hat - (alpha/ln eta) i m G^I Psi_hat_m
//   e_u     = -D^I N_u_hat
// (Eqs. vort, temp, uphi; psi_int, temp_int, uphi_int; u_s = (h^2/s) v and
//  beta u_s = -v.)  The radial derivative is that of the n_r-point interpolant.
// ---------------------------------------------------------------------------
template <int H, class V>
__device__ __forceinline__ double2 band_row(const double* __restrict__ band, const V* x, int k, int nc) {
    const double* row = band + (size_t)k * (2 * H + 1);
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int d = 0; d <= 2 * H; ++d) {
        const int n = k - H + d;
        if (n >= 0 && n < nc) {
            const double c = __ldg(&row[d]);
            const double2 v = to_d2(x[n]);
            acc.x = fma(c, v.x, acc.x);
            acc.y = fma(c, v.y, acc.y);
        }
    }
    return acc;
}

template <class T>
__global__ void __launch_bounds__(NTHREADS_R) k_grid_to_spec(StepParams P, const T* G2, VecSet y,
                                                             VecSet e) {
    chain_wait();
    using RT = typename Cx<T>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    T* sm = reinterpret_cast<T*>(smraw);
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, L = 2 * K, N = P.n_r, nc = P.nc, M = P.M;
    const int NB = radial_batch(P);
    T* bufA = sm;
    T* bufB = bufA + NB * L;
    T* cc0 = bufB + NB * L;
    T* cc1 = cc0 + N;
    T* cc2 = cc1 + N;
    const int tid = threadIdx.x, nth = blockDim.x;
    const RT dm = (RT)m;

    // pass A: plain Chebyshev coefficients of F1 = h^2 [v omega]_m, F2 = h^2 [v theta]_m
    for (int b0 = 0; b0 < 2; b0 += NB) {
        const int nb = min(NB, 2 - b0);
        for (int b = 0; b < nb; ++b) {
            const int f = (b0 + b == 0) ? 0 : 2;
            T* z = bufA + b * L;
            for (int j = tid; j <= K; j += nth)
                even_extend_store(z, K, j, cscale(G2[g_index(j, f, m, M)], Tab<T>::h2(P, j)));
        }
        T* R = radial_dct1(bufA, bufB, P, nb);
        const RT iK = (RT)(1.0 / (double)K), hK = (RT)(0.5 / (double)K);
        for (int b = 0; b < nb; ++b) {
            T* dst = (b0 + b == 0) ? cc0 : cc1;
            const T* Z = R + b * L;
            for (int n = tid; n <= K; n += nth) dst[n] = cscale(Z[n], (n == 0 || n == K) ? hK : iK);
        }
        __syncthreads();
    }
    // d/ds of both, in place, the two scans side by side (bufA, bufB: scratch)
    cheb_derivative_scan2(cc0, bufA, cc1, bufB, N, P.inv_a);

    // pass B: derivative values on the grid, then N_omega (or N_u) and N_theta;
    // with Ekman pumping N_omega - F_eps and N_u + Ups_eps u_bar (1 + (E/2) omega_0)
    const T* PF = P.pump ? reinterpret_cast<const T*>(P.pump_F) + (size_t)m * N : nullptr;
    for (int b0 = 0; b0 < 2; b0 += NB) {
        const int nb = min(NB, 2 - b0);
        for (int b = 0; b < nb; ++b) {
            const T* c = (b0 + b == 0) ? cc0 : cc1;
            T* z = bufA + b * L;
            for (int j = tid; j <= K; j += nth) {
                T v = c[j];
                if (j == 0 || j == K) v = cscale(v, (RT)2);
                even_extend_store(z, K, j, v);
            }
        }
        T* R = radial_dct1(bufA, bufB, P, nb);
        // the grid values of N go to cc2 (omega) and cc0 (theta): cc0 was consumed
        // by the loads above (for NB == 1 the theta pass runs after the omega one)
        for (int b = 0; b < nb; ++b) {
            const int fld = b0 + b;  // 0: omega, 1: theta
            const T* Z = R + b * L;
            T* dst = (fld == 0) ? cc2 : cc0;
            for (int k = tid; k <= K; k += nth) {
                const T dF = cscale(Z[k], (RT)0.5);
                const RT is = Tab<T>::is(P, k);
                T val;
                if (fld == 0) {
                    if (m > 0) {
                        const T uw = G2[g_index(k, 1, m, M)];
                        val = cscale(cadd(dF, cmul_i(uw, dm)), is);
                        if (PF) val = csub(val, PF[k]);
                    } else {
                        const T vw = G2[g_index(k, 0, m, M)];
                        val = cscale(vw, Tab<T>::h2(P, k) * is);
                        if (PF) val = cadd(val, PF[k]);
                    }
                } else {
                    const T ut = G2[g_index(k, 3, m, M)];
                    const T vt = G2[g_index(k, 2, m, M)];
                    val = csub(cscale(cadd(dF, cmul_i(ut, dm)), is), vt);
                }
                dst[k] = val;
            }
        }
        __syncthreads();
    }
    // pass C: Eq. icheb of N_omega (cc2) and N_theta (cc0), truncated to n < nc
    for (int b0 = 0; b0 < 2; b0 += NB) {
        const int nb = min(NB, 2 - b0);
        for (int b = 0; b < nb; ++b) {
            const T* src = (b0 + b == 0) ? cc2 : cc0;
            T* z = bufA + b * L;
            for (int j = tid; j <= K; j += nth) even_extend_store(z, K, j, src[j]);
        }
        T* R = radial_dct1(bufA, bufB, P, nb);
        for (int b = 0; b < nb; ++b) {
            T* dst = (b0 + b == 0) ? cc1 : cc2;  // N_omega_hat -> cc1, N_theta_hat -> cc2
            const T* Z = R + b * L;
            // for NB == 1 the theta pass reads cc0 and writes cc2, which holds
            // nothing needed any more (N_omega_hat went to cc1)
            const RT hc = (RT)(0.5 * P.cnorm);
            for (int n = tid; n < nc; n += nth) dst[n] = cscale(Z[n], hc);
        }
        __syncthreads();
    }
    // integrated right-hand sides; the linear couplings read the FP64 state
    //   e_psi = C^I N_omega_hat + (Ra/Pr)(i m/s_o) C^I theta_hat
    //   e_theta = -D^I N_theta_hat - (alpha/ln eta) i m G^I Psi_hat,  e_u = -D^I N_u_hat
    const double bfac = P.Ra / P.Pr * (double)m / P.s_o;
    const double2* th_m = y.th + (size_t)m * nc;
    const double2* ps_m = y.psi + (size_t)m * nc;
    for (int k = tid; k < nc; k += nth) {
        double2 ep = make_double2(0.0, 0.0), et = make_double2(0.0, 0.0);
        if (k >= 4 && m > 0) {
            ep = band_row<8>(P.ops.band[OP_C], cc1, k, nc);
            if (!P.buoy_imp) ep = cadd(ep, cmul_i(band_row<8>(P.ops.band[OP_C], th_m, k, nc), bfac));
        }
        if (k >= 2) {
            const double2 dn = band_row<4>(P.ops.band[OP_D], cc2, k, nc);
            if (m > 0) {
                const double2 gp = band_row<4>(P.ops.band[OP_G], ps_m, k, nc);
                et = csub(cmul_i(gp, -P.tc * (double)m), dn);
            } else {
                et = cscale(dn, -1.0);
            }
        }
        e.psi[(size_t)m * nc + k] = ep;
        e.th[(size_t)m * nc + k] = et;
        if (m == 0) {
            double eu = 0.0;
            if (k >= 2) eu = -band_row<4>(P.ops.band[OP_D], cc1, k, nc).x;
            e.u[k] = eu;
        }
    }
}

// ---------------------------------------------------------------------------
// Radial DCT-I in fixed point (fixfft.cuh), the FP64 stage's transform: the even
// extension of K + 1 FP64 values as 64-bit integers, one complex transform of
// length 2K for each vector, the outputs back in FP64.
//
// A vector's components are normalised separately by the exponents of their
// largest magnitudes; FxScale keeps the exponents and the transforms' schedules of
// up to FX_VEC vectors of a kernel.  The work around the transforms is split by
// component (task t: entry t/2, part t & 1): an FP64 instruction of a warp takes
// 64 cycles, so twice the warps with half the instructions each is twice as fast
// until all four sub-partitions issue FP64 without a pause.
// ---------------------------------------------------------------------------
constexpr int FX_VEC = 6;
constexpr int FX_L1 = 43;  // 1-norms are summed in units of 2^FX_L1 (up to 2^13 points)
struct FxScale {
    unsigned e[FX_VEC][2];  // biased exponent of the largest |re|, |im|
    unsigned l1[FX_VEC];    // 1-norm of the extension in units of 2^FX_L1
    unsigned back[FX_VEC];  // fx_schedule
    int S[FX_VEC];
};
// threads of the fixed-point radial kernels: every (entry, part) at once, at
// least eight warps (the derivative scans' roles)
constexpr int NTHREADS_FX = 544;
inline int fx_threads(const StepParams& P) { return std::max(256, std::min(NTHREADS_FX, (2 * P.n_r + 31) / 32 * 32)); }

// Whole CTA, before the first use; the caller's next barrier publishes it.
__device__ __forceinline__ void fx_scale_clear(FxScale& sc) {
    for (int i = threadIdx.x; i < (int)(sizeof(FxScale) / 4); i += blockDim.x) reinterpret_cast<unsigned*>(&sc)[i] = 0u;
}
// exponent ex of part of vector v joins the block's; whole warps
__device__ __forceinline__ void fx_scale_max(FxScale& sc, int v, int part, unsigned ex) {
    const unsigned x = __reduce_max_sync(0xffffffffu, part ? 0u : ex), y = __reduce_max_sync(0xffffffffu, part ? ex : 0u);
    if ((threadIdx.x & 31) == 0) {
        if (x) atomicMax(&sc.e[v][0], x);
        if (y) atomicMax(&sc.e[v][1], y);
    }
}
// at least |q| 2^-FX_L1, from the leading word
__device__ __forceinline__ unsigned fx_l1_part(fx64 q) {
    int h, l;
    fx_words(q, h, l);
    return (unsigned)abs(h) / (1u << (FX_L1 - 32)) + 1u;
}
__device__ __forceinline__ int fx_l1_bits(unsigned l1) { return FX_L1 + 32 - __clz((int)l1); }

// DCT-I of vectors v0 .. v0 + nb - 1 of the kernel, val(i, t) the FP64 part t & 1 of
// entry t / 2 of vector v0 + i for t < 2 n (entries from n to K are zero), whose
// exponents have been gathered before a barrier.  twice: the entries at both ends
// count twice (a synthesis).  a, b: 2K nb points each.  Vector i's transform Z_n
// (n <= K) is at the returned pointer + 2K i; dct_part gives it in FP64.  Ends with
// a barrier.
template <class V>
__device__ __forceinline__ fxc* dct1_fx(const StepParams& P, FxScale& sc, int v0, int nb, int n, bool twice, fxc* a,
                                        fxc* b, V val) {
    const int K = P.K, L = 2 * K;
    for (int i = 0; i < nb; ++i) {
        fx64* z = reinterpret_cast<fx64*>(a + (size_t)i * L);
        unsigned l1 = 0u;
        for (int t = threadIdx.x; t < 2 * (K + 1); t += blockDim.x) {
            const int j = t >> 1, part = t & 1;
            const int e = (int)sc.e[v0 + i][part];
            fx64 q = 0;
            if (j < n && e && e != 0x7ff) {  // (zero, or with an infinity or NaN in the block: outputs are NaN)
                q = fx_from(val(i, t), e);
                if (twice && (j == 0 || j == K)) q = 2 * q;  // its exponent entered e plus one
            }
            z[t] = q;
            const unsigned w = fx_l1_part(q);
            if (j > 0 && j < K) {
                z[2 * (L - j) + part] = q;
                l1 += 2u * w;
            } else {
                l1 += w;
            }
        }
        l1 = __reduce_add_sync(0xffffffffu, l1);
        if ((threadIdx.x & 31) == 0) atomicAdd(&sc.l1[v0 + i], l1);
    }
    __syncthreads();
    const int lg = 32 - __clz(K);  // L = 2^lg
    if ((int)threadIdx.x < nb) {
        const int v = v0 + threadIdx.x;
        int S;
        sc.back[v] = fx_schedule(lg, false, fx_l1_bits(sc.l1[v]), S);
        sc.S[v] = S;
    }
    return fx_fft<true>(a, b, reinterpret_cast<const fxw*>(P.fx_r), 1, lg, false, nb, sc.back + v0);
}
// 2^p times part of an output of vector v
__device__ __forceinline__ double dct_part(const FxScale& sc, int v, const fxc* z, int part, int p) {
    const int ex = (int)sc.e[v][part];
    return fx_to(part ? z->y : z->x, sc.S[v] - 1022 - FX_BITS + p + ex, ex == 0x7ff);
}

// Chebyshev derivative of FP64 plain coefficients c[0 .. n-1] into d (another
// array), the sums of cheb_derivative_scan, by four warps: role 0..3 takes one
// index parity of one component, -1 none.  The exponents of d (as a synthesis's
// input: the first entry twice) join vector v.  The caller's next barrier publishes d.
__device__ __forceinline__ void cheb_derivative_part(const double2* c, double2* d, int n, double scale, int role,
                                                     FxScale& sc, int v) {
    if (role < 0) return;
    const int lane = threadIdx.x & 31;
    const int q = role & 1, part = role >> 1;
    const double* cs = reinterpret_cast<const double*>(c) + part;
    double* ds = reinterpret_cast<double*>(d) + part;
    const int len = (n - q + 1) / 2;
    const int per = (len + 31) / 32;
    const int i0 = lane * per, i1 = min(i0 + per, len);
    double acc = 0.0;
    for (int i = i1 - 1; i >= i0; --i) {
        const int k = 2 * i + q;
        if (k > 0) {
            acc = fma((double)(2 * k), cs[2 * k], acc);
            ds[2 * (k - 1)] = acc;
        }
    }
    double sfx = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double x = __shfl_down_sync(0xffffffffu, sfx, o);
        if (lane + o < 32) sfx += x;
    }
    const double off = sfx - acc;
    unsigned ex = 0u;
    for (int i = i0; i < i1; ++i) {
        const int k = 2 * i + q;
        if (k > 0) {
            const double x = (ds[2 * (k - 1)] + off) * ((k == 1) ? 0.5 * scale : scale);
            ds[2 * (k - 1)] = x;
            ex = max(ex, fx_exponent(x) + (k == 1 && fx_exponent(x) ? 1u : 0u));
        }
    }
    if (q == 0 && lane == 0) ds[2 * (n - 1)] = 0.0;
    ex = __reduce_max_sync(0xffffffffu, min(ex, 0x7ffu));
    if (lane == 0) atomicMax(&sc.e[v][part], ex);
}

// K1 of the FP64 stage in the batched layout: the equations of k_spec_to_grid with
// the DCT-I in fixed point.  Bound by the latency of its phases (39 % of the issue
// slots, 42 % of the FP64 pipe's at 257 x 768, where the FP64 transforms kept
// that pipe 60 % busy): 50 -> 24.8 us there, 23 -> 14.8 us at 129 x 384, 67 -> 35 us
// at 513 x 384 (against the double-float lean layout it replaces at that size).
__global__ void __launch_bounds__(NTHREADS_FX, 2) k_spec_to_grid_fx(StepParams P, VecSet y, double2* __restrict__ G1,
                                                                   double2* __restrict__ W) {
    chain_wait();
    __shared__ FxScale sc;
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, L = 2 * K, N = P.n_r, nc = P.nc, M = P.M;
    const int NB = radial_batch(P);
    fxc* bufA = fx_shared;
    fxc* bufB = bufA + NB * L;
    double2* cc0 = reinterpret_cast<double2*>(bufB + NB * L);  // Psi (or u_bar) plain coefficients, length nc
    double2* cc1 = cc0 + N;                                    // first derivative
    double2* cc2 = cc1 + N;                                    // second derivative
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5;
    const double Cw = P.cnorm, Cw0 = 0.5 * P.cnorm;
    // vectors: 0 Psi, 1 Psi', 2 Psi'', 3 theta (m >= 1); 0 u_bar, 1 u_bar', 3 theta (m = 0)
    const int th_v = 3;
    const double* ps = reinterpret_cast<const double*>(y.psi + (size_t)m * nc);
    const double* th = reinterpret_cast<const double*>(y.th + (size_t)m * nc);
    fx_scale_clear(sc);
    __syncthreads();
    for (int b = 0; b < 2; ++b) {
        unsigned ex = 0u;
        for (int t = tid; t < 2 * nc; t += nth) {
            const double w = (t < 2) ? Cw0 : Cw;
            double x;
            if (b) {
                x = th[t] * w;  // (formed again when it is converted)
            } else {
                x = (m > 0) ? ps[t] * w : (t & 1) ? 0.0 : y.u[t >> 1] * w;
                reinterpret_cast<double*>(cc0)[t] = x;
            }
            const unsigned e = fx_exponent(x);
            ex = max(ex, (t < 2 && e) ? min(e + 1u, 0x7ffu) : e);  // the first entry counts twice
        }
        fx_scale_max(sc, b ? th_v : 0, tid & 1, ex);
    }
    __syncthreads();
    cheb_derivative_part(cc0, cc1, nc, P.inv_a, warp < 4 ? warp : -1, sc, 1);
    __syncthreads();
    if (m > 0) {
        cheb_derivative_part(cc1, cc2, nc, P.inv_a, warp < 4 ? warp : -1, sc, 2);
        __syncthreads();
    }
    auto value = [&](int v, int t) -> double {
        if (v == th_v) return th[t] * ((t < 2) ? Cw0 : Cw);
        return reinterpret_cast<const double*>(v == 0 ? cc0 : v == 1 ? cc1 : cc2)[t];
    };
    const double dm = (double)m;
    double* PF = P.pump ? reinterpret_cast<double*>(P.pump_F + (size_t)m * N) : nullptr;
    double* wu = reinterpret_cast<double*>(W + (size_t)m * 2 * N);  // partial sums of u_phi, then of omega
    for (int f0 = 0; f0 < 4; f0 += NB) {
        const fxc* R = dct1_fx(P, sc, f0, NB, nc, true, bufA, bufB, [&](int i, int t) { return value(f0 + i, t); });
        for (int t = tid; t < 2 * N; t += nth) {
            const int k = t >> 1, part = t & 1;
            const double s = P.s[k], h2 = P.h2[k], is = P.inv_s[k];
            double* out = reinterpret_cast<double*>(G1 + g_index(k, 0, m, M));
            // out: fields v, u_phi, omega, theta, 2M doubles apart.  u_phi and omega are summed
            // over the vectors of a batch in a register, over batches in W.
            double up = 0.0, om = 0.0, pf = 0.0;
            if (f0 > 0) {
                up = wu[t];
                om = wu[2 * N + t];
                if (PF) pf = PF[t];
            }
            for (int i = 0; i < NB; ++i) {
                const int v = f0 + i;
                const double g = dct_part(sc, v, R + (size_t)i * L + k, part, -1);  // value of the series at x_k
                if (v == th_v) {
                    out[6 * M + part] = g;
                } else if (m == 0) {
                    if (v == 0) {
                        out[part] = 0.0;
                        up = g;
                        om = __dmul_rn(g, is);
                    } else if (v == 1) {
                        om += g;
                        if (PF) pf = part ? 0.0 : P.pump_ups[k] * up * (1.0 + (0.5 * P.E) * om);
                    }
                } else if (v == 0) {
                    const double c = fma(__dmul_rn(dm * dm, h2), __dmul_rn(is, is), 6.0);
                    out[part ^ 1] = part ? -dm * g : dm * g;
                    up = __dmul_rn(__dmul_rn(3.0, s), g);
                    om = __dmul_rn(c, g);
                    if (PF) {
                        const double go = dct_part(sc, v, R + (size_t)i * L + k, part ^ 1, -1), U = P.pump_ups[k];
                        const double ci = __dmul_rn(__dmul_rn(U, dm), P.pump_ci[k]);
                        pf = fma(part ? -ci : ci, go, __dmul_rn(__dmul_rn(-U, fma(dm, dm, P.pump_cr[k])), g));
                    }
                } else if (v == 1) {
                    const double c = fma(-5.0, s, __dmul_rn(h2, is));
                    up = fma(-h2, g, up);
                    om = fma(-c, g, om);
                    if (PF) pf = fma(__dmul_rn(P.pump_ups[k], __dmul_rn(0.5, s)), g, pf);
                } else {
                    om = fma(-h2, g, om);
                    if (PF) pf = fma(-P.pump_ups[k], om, pf);
                }
            }
            // u_phi is complete after vector 1, omega after vector 2 (1 for m = 0, whose
            // vector 2 is zero)
            if (f0 <= 1 && f0 + NB > 1) out[2 * M + part] = up;
            if (f0 <= 2 && f0 + NB > 2) out[4 * M + part] = om;
            if (f0 + NB < 3) {
                wu[t] = up;
                wu[2 * N + t] = om;
            }
            if (PF) PF[t] = pf;
        }
        __syncthreads();
    }
}

// row k of a real band applied to one component of complex values: x points at
// that component (stride 2)
template <int H>
__device__ __forceinline__ double band_part(const double* __restrict__ band, const double* x, int k, int nc) {
    const double* row = band + (size_t)k * (2 * H + 1);
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d <= 2 * H; ++d) {
        const int n = k - H + d;
        if (n >= 0 && n < nc) acc = fma(__ldg(&row[d]), x[2 * n], acc);
    }
    return acc;
}

// K3 of the FP64 stage in the batched layout: the equations of k_grid_to_spec with
// the DCT-I in fixed point, the buoyancy added to N_omega_hat before the one C^I
// apply (Eq. psi_int applies C^I to their sum), and the banded applies spread
// over (row, component, operator) so that every warp issues FP64.  257 x 768:
// 75 -> 43 us (50 % of the FP64 pipe's slots, 33 % of the issue slots), 129 x 384: 43 ->
// 24.0, 513 x 384: 114 -> 49 us (from the double-float lean layout).
// Vectors 0, 1: F1, F2 (to coefficients); 2, 3: their derivatives (to the grid);
// 4, 5: N_omega (N_u), N_theta (to coefficients).
__global__ void __launch_bounds__(NTHREADS_FX, 2) k_grid_to_spec_fx(StepParams P, const double2* G2,
                                                                    VecSet y, VecSet e) {
    chain_wait();
    __shared__ FxScale sc;
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, L = 2 * K, N = P.n_r, nc = P.nc, M = P.M;
    const int NB = min(2, radial_batch(P));
    fxc* bufA = fx_shared;
    fxc* bufB = bufA + NB * L;
    double2* cc0 = reinterpret_cast<double2*>(bufB + NB * L);
    double2* cc1 = cc0 + N;
    double2* cc2 = cc1 + N;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5;
    const double dm = (double)m;
    const int lgK = 31 - __clz(K);
    const double* g2 = reinterpret_cast<const double*>(G2);
    auto flat = [](double2* c) { return reinterpret_cast<double*>(c); };
    fx_scale_clear(sc);
    __syncthreads();
    // pass A: plain Chebyshev coefficients of F1 = h^2 [v omega]_m, F2 = h^2 [v theta]_m
    for (int b = 0; b < 2; ++b) {
        double* dst = flat(b ? cc1 : cc0);
        unsigned ex = 0u;
        for (int t = tid; t < 2 * N; t += nth) {
            const double v = g2[2 * (size_t)g_index(t >> 1, 2 * b, m, M) + (t & 1)] * P.h2[t >> 1];
            dst[t] = v;
            ex = max(ex, fx_exponent(v));
        }
        fx_scale_max(sc, b, tid & 1, ex);
    }
    __syncthreads();
    for (int b0 = 0; b0 < 2; b0 += NB) {
        const fxc* R = dct1_fx(P, sc, b0, NB, N, false, bufA, bufB,
                               [&](int i, int t) { return flat((b0 + i) ? cc1 : cc0)[t]; });
        for (int i = 0; i < NB; ++i) {
            double* dst = flat((b0 + i) ? cc1 : cc0);
            for (int t = tid; t < 2 * N; t += nth) {
                const int n = t >> 1;
                dst[t] = dct_part(sc, b0 + i, R + (size_t)i * L + n, t & 1, (n == 0 || n == K) ? -lgK - 1 : -lgK);
            }
        }
        __syncthreads();
    }
    // d/ds of both: F1' -> cc2, F2' -> the free transform buffer beside it (two
    // vectors in it) or, one vector at a time, cc0 once F1 is done with
    double2* d1 = cc0;
    if (NB == 2) {
        d1 = reinterpret_cast<double2*>(bufB);
        if (warp < 4)
            cheb_derivative_part(cc0, cc2, N, P.inv_a, warp, sc, 2);
        else
            cheb_derivative_part(cc1, d1, N, P.inv_a, warp < 8 ? warp - 4 : -1, sc, 3);
    } else {
        cheb_derivative_part(cc0, cc2, N, P.inv_a, warp < 4 ? warp : -1, sc, 2);
        __syncthreads();
        cheb_derivative_part(cc1, d1, N, P.inv_a, warp < 4 ? warp : -1, sc, 3);
    }
    __syncthreads();
    // pass B: derivative values on the grid, then N_omega (or N_u) -> cc1 and N_theta
    // -> cc2; with Ekman pumping N_omega - F_eps and N_u + Ups_eps u_bar (1 + (E/2) omega_0)
    const double* PF = P.pump ? reinterpret_cast<const double*>(P.pump_F + (size_t)m * N) : nullptr;
    for (int b0 = 0; b0 < 2; b0 += NB) {
        // (the last coefficient of a derivative is zero)
        const fxc* R = dct1_fx(P, sc, 2 + b0, NB, K, true, bufA, bufB,
                               [&](int i, int t) { return flat((b0 + i) ? d1 : cc2)[t]; });
        for (int i = 0; i < NB; ++i) {
            const int fld = b0 + i;  // 0: omega, 1: theta
            double* dst = flat(fld ? cc2 : cc1);
            unsigned ex = 0u;
            for (int t = tid; t < 2 * N; t += nth) {
                const int k = t >> 1, part = t & 1;
                const double dF = dct_part(sc, 2 + fld, R + (size_t)i * L + k, part, -1);
                const double is = P.inv_s[k];
                const double* g = g2 + 2 * (size_t)g_index(k, 0, m, M);  // fields 2M doubles apart
                double val;
                if (fld == 0 && m == 0) {
                    val = g[part] * (P.h2[k] * is);
                    if (PF) val += PF[t];
                } else {  // dF + i m [u_phi omega] (or [u_phi theta]), over s
                    const double u = g[(fld ? 6 : 2) * M + (part ^ 1)];
                    const double w = fma(part ? dm : -dm, u, dF);
                    if (fld == 0) {
                        val = w * is;
                        if (PF) val -= PF[t];
                    } else {
                        val = fma(w, is, -g[4 * M + part]);
                    }
                }
                dst[t] = val;
                ex = max(ex, fx_exponent(val));
            }
            fx_scale_max(sc, 4 + fld, tid & 1, ex);
        }
        __syncthreads();
    }
    // pass C: Eq. icheb of N_omega (cc1) and N_theta (cc2), truncated to n < nc:
    // N_omega_hat, with the buoyancy, -> cc0, N_theta_hat -> cc1
    const double hc = 0.5 * P.cnorm, bfac = P.Ra / P.Pr * dm / P.s_o;
    const bool buoy = m > 0 && !P.buoy_imp;
    const double* th = reinterpret_cast<const double*>(y.th + (size_t)m * nc);
    for (int b0 = 0; b0 < 2; b0 += NB) {
        const fxc* R = dct1_fx(P, sc, 4 + b0, NB, N, false, bufA, bufB,
                               [&](int i, int t) { return flat((b0 + i) ? cc2 : cc1)[t]; });
        for (int i = 0; i < NB; ++i)
            for (int t = tid; t < 2 * nc; t += nth) {
                const int part = t & 1;
                double v = dct_part(sc, 4 + b0 + i, R + (size_t)i * L + (t >> 1), part, 0) * hc;
                if (b0 + i) {
                    flat(cc1)[t] = v;
                } else {
                    if (buoy) v = fma(part ? bfac : -bfac, th[t ^ 1], v);
                    flat(cc0)[t] = v;
                }
            }
        __syncthreads();
    }
    // integrated right-hand sides; the linear couplings read the FP64 state
    //   e_psi = C^I N_omega_hat,  e_theta = -D^I N_theta_hat - (alpha/ln eta) i m G^I Psi_hat,
    //   e_u = -D^I N_u_hat
    double* eps = reinterpret_cast<double*>(e.psi + (size_t)m * nc);
    double* eth = reinterpret_cast<double*>(e.th + (size_t)m * nc);
    const double* ps = reinterpret_cast<const double*>(y.psi + (size_t)m * nc);
    for (int t = tid; t < 4 * nc; t += nth) {
        const int r = (t < 2 * nc) ? t : t - 2 * nc;
        const int k = r >> 1, part = r & 1;
        if (t < 2 * nc) {
            double v = 0.0;
            if (m > 0) {
                if (k >= 4) v = band_part<8>(P.ops.band[OP_C], flat(cc0) + part, k, nc);
            } else if (part == 0) {
                e.u[k] = (k >= 2) ? -band_part<4>(P.ops.band[OP_D], flat(cc0), k, nc) : 0.0;
            }
            eps[r] = v;
        } else {
            double v = 0.0;
            if (k >= 2) {
                v = -band_part<4>(P.ops.band[OP_D], flat(cc1) + part, k, nc);
                if (m > 0) {
                    const double gp = band_part<4>(P.ops.band[OP_G], ps + (part ^ 1), k, nc);
                    v = fma(part ? -P.tc * dm : P.tc * dm, gp, v);
                }
            }
            eth[r] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// K2 of the FP64 stage in fixed point: the steps of k_phi_products on 64-bit
// integers.  Each field is normalised by the exponent of its largest
// coefficient on load; the physical values of each field are shifted up by the
// free leading bits of their largest before the products, whose 60-bit results
// are transformed back.  FP64 is used for conversions only.  The means of the
// products (m = 0), which cancel, are summed over the modes in FP64 (13 us of 327 at
// 1025 x 3072, 100 of 1363 at 2049 x 6144).  Bound by instruction issue (43 to 49 % of
// the slots at 257 x 768 .. 1025 x 1536; 16 warps an SM at n_phi = 6144, where two buffers
// fill its shared memory).  Against the double-float kernel: 257 x 768 37 -> 26.8 us, 33 x
// 96 22 -> 12.2, 1025 x 3072 443 -> 334, 2049 x 6144 1706 -> 1364 us.
// ---------------------------------------------------------------------------
constexpr int PHI_SUMS = 12;
struct PhiScale {
    unsigned e[4];      // biased exponents of v, u_phi, omega, theta
    unsigned top[4];    // OR of the leading words of the fields' physical values
    unsigned l1[4];     // 1-norms of the packed spectra, then of the packed products
    unsigned back[4];
    int S[4];
    double mean[PHI_SUMS][4];  // partial sums of the four products over the modes
    double mean0[4];     // the products' means
    double cfl[2 * 16];
};

// 2/3 of a: 1/n_phi = (2/3) 2^-(lg + 1) for n_phi = 3 2^lg
__device__ __forceinline__ fx64 fx_two_thirds(fx64 a) {
    constexpr long long c = 3074457345618258603ll;  // in units of 2^-62
    constexpr int lo = (int)(unsigned)(unsigned long long)c;
    return fx_mulc(a, (int)((c - lo) >> 32), lo);
}
// a b 2^-62, |a|, |b| < 2^61
__device__ __forceinline__ fx64 fx_mul62(fx64 a, fx64 b) {
    int ah, al, bh, bl;
    fx_split(a, ah, al);
    fx_split(b, bh, bl);
    return (fx64)((unsigned long long)fx_mulw(ah, bh) << 2) + ((fx_mad(al, bh, fx_mulw(ah, bl)) + ((fx64)1 << 29)) >> 30);
}
__device__ __forceinline__ unsigned fx_top(fx64 a) { return (unsigned)((a < 0 ? ~a : a) >> 32); }

// a field's coefficient in fixed point, components up to 2^FX_BITS
__device__ __forceinline__ fxc phi_coef(double2 v, unsigned e) {
    return (e == 0x7ff) ? fxc{0, 0} : fxc{fx_from(v.x, (int)e), fx_from(v.y, (int)e)};
}
// mode m of the fields a and b packed as a + i b into Z, halved (the packed values
// stay within 2^FX_BITS) and with the components exchanged (fx_fft then runs the
// backward transform); returns the 1-norm written
__device__ __forceinline__ unsigned phi_pack(fxc a, fxc b, int m, int Pn, fxc* Z) {
    a = fx_half(a);
    b = fx_half(b);
    if (m == 0) {
        Z[0] = fxc{b.x, a.x};
        return fx_l1_part(a.x) + fx_l1_part(b.x);
    }
    const fxc z1 = fxc{a.y + b.x, a.x - b.y};  // (im, re) of a + i b
    const fxc z2 = fxc{b.x - a.y, a.x + b.y};  // of conj(a) + i conj(b)
    Z[m] = z1;
    Z[Pn - m] = z2;
    return fx_l1_part(z1.x) + fx_l1_part(z1.y) + fx_l1_part(z2.x) + fx_l1_part(z2.y);
}
// the spectra of a + i b from its transform Y (scaled by 2^-S), over n_phi
__device__ __forceinline__ void phi_split(const fxc* Y, double2* __restrict__ dst, int M, int Pn, int n_m, bool three,
                                          int exa, int exb, bool bada, bool badb) {
    for (int m = threadIdx.x; m <= n_m; m += blockDim.x) {
        const fxc y1 = Y[m], y2 = Y[m ? Pn - m : 0];
        // a = (y1 + conj(y2))/2,  b = (y1 - conj(y2))/(2i)
        const fx64 v[4] = {fx_avg(y1.x, y2.x), fx_avg(y1.y, -y2.y), fx_avg(y1.y, y2.y), fx_avg(y2.x, -y1.x)};
        double d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            d[i] = fx_to(three ? fx_two_thirds(v[i]) : v[i], i < 2 ? exa : exb, i < 2 ? bada : badb);
        dst[m] = make_double2(d[0], d[1]);
        dst[M + m] = make_double2(d[2], d[3]);
    }
}

// Courant rates (cfl_rates) from the packed physical pair (u_phi, v) in R.  A radius
// whose fields hold an infinity or NaN (bad) adds no rate, as in cfl_rates, whose
// maxima pass over NaNs: the rates of the radii and states before it stay to be
// reported (a NaN, above every number as a bit pattern, would replace them).
__device__ void cfl_rates_fx(const StepParams& P, const fxc* R, int k, int sv, int su, bool bad, double* red) {
    if (bad) return;
    fx64 a = 0, b = 0;
    for (int j = threadIdx.x; j < P.n_phi; j += blockDim.x) {
        const fxc g = R[j];
        a = max(a, g.y < 0 ? -g.y : g.y);
        b = max(b, g.x < 0 ? -g.x : g.x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[2 * w] = fx_to(a, sv, false);
        red[2 * w + 1] = fx_to(b, su, false);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ra = red[0], rb = red[1];
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
            ra = fmax(ra, red[2 * i]);
            rb = fmax(rb, red[2 * i + 1]);
        }
        const double s = P.s[k];
        const double fs = P.coll ? 1.0 / s : P.h2[k] / s;
        const double rs = fs * ra / P.cfl_ds[k], rp = rb / (s * P.cfl_dphi);
        atomicMax(reinterpret_cast<unsigned long long*>(P.cfl_max), (unsigned long long)__double_as_longlong(rs));
        atomicMax(reinterpret_cast<unsigned long long*>(P.cfl_max + 1), (unsigned long long)__double_as_longlong(rp));
    }
    __syncthreads();
}

// PAIR: both packed pairs in one batched transform each way (buffers of 2 n_phi
// points each); else one after the other, the first pair's physical values
// and the second products waiting in registers.  MANY: several modes a lane in the means'
// sums, read ahead (1025 x 3072 334 us, 340 without); with a mode or two the longer code
// alone costs 1 us (65 x 192 12.4 -> 13.6, 257 x 768 26.7 -> 28.1).
template <bool PAIR, bool MANY>
__global__ void __launch_bounds__(512, PAIR ? 2 : 1) k_phi_products_fx(StepParams P, const double2* G1,
                                                            double2* __restrict__ G2) {
    chain_wait();
    __shared__ PhiScale sc;
    const int k = P.k_lo + blockIdx.x;
    const int Pn = P.n_phi, M = P.M, n_m = P.n_m;
    const int tid = threadIdx.x, nth = blockDim.x;
    const bool three = Pn % 3 == 0;
    const int lg = 31 - __clz(three ? Pn / 3 : Pn);
    const fxw* tw = reinterpret_cast<const fxw*>(P.fx_p);
    fxc* X = fx_shared;
    fxc* Y = X + (PAIR ? 2 : 1) * Pn;
    const double2* src = G1 + g_index(k, 0, 0, M);
    double2* dst = G2 + g_index(k, 0, 0, M);
    if (tid < (int)(offsetof(PhiScale, mean) / 4)) reinterpret_cast<unsigned*>(&sc)[tid] = 0u;
    __syncthreads();
    {
        // exponents of the fields and, in FP64 (its pipe is idle here), the means of the
        // products, a_0 b_0 + 2 sum_{m >= 1} Re(a_m conj(b_m)), exact for these band-limited fields:
        // they cancel (the zonal forcing [v omega]_0 down to 1e-7 of its terms), where even a
        // few units of rounding of the transforms' m = 0 entries show.  In the same order for
        // any number of threads (a launch shape, which changes no bit of a result): partial
        // sum w takes the modes of warp w of PHI_SUMS, and a smaller CTA's warps take several.
        // (Twelve are what the 384 threads of n_phi = 768 and 1536 have: 83.5 us at 513 x
        // 1536 as with one sum a warp, 85.7 with sixteen.)
        unsigned ex[4] = {0u, 0u, 0u, 0u};
        const int lane = tid & 31;
        for (int w = tid >> 5; w < PHI_SUMS && 32 * w <= n_m; w += nth >> 5) {
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll (MANY ? 4 : 1)
            for (int m = 32 * w + lane; m <= n_m; m += 32 * PHI_SUMS) {
                double2 f[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    f[q] = src[q * M + m];
                    ex[q] = max(ex[q], max(fx_exponent(f[q].x), fx_exponent(f[q].y)));
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {  // (v, omega), (u_phi, omega), (v, theta), (u_phi, theta)
                    const double2 a = f[q & 1], b = f[2 + (q >> 1)];
                    acc[q] = m ? fma(a.x, b.x, fma(a.y, b.y, acc[q])) : 0.5 * (a.x * b.x);
                }
            }
            // four sums over the warp: halves exchanged twice, then lanes of equal l >> 3 added up
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int o = 16 >> s, half = 2 >> s;
                const bool up = lane & o;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const double send = up ? acc[i] : acc[i + half];
                    acc[i] = (up ? acc[i + half] : acc[i]) + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
            if ((lane & 7) == 0) sc.mean[w][lane >> 3] = acc[0];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ex[q] = __reduce_max_sync(0xffffffffu, ex[q]);
            if (lane == 0) atomicMax(&sc.e[q], ex[q]);
        }
    }
    __syncthreads();
    if (tid >= nth - 32) {  // one warp: lane 4 w + q adds partial sums w and w + 8 of product q
        const int q = tid & 3, w = (tid & 31) >> 2;
        const int ns = min(PHI_SUMS, n_m / 32 + 1);
        double v = (w < ns ? sc.mean[w][q] : 0.0) + (w + 8 < ns ? sc.mean[w + 8][q] : 0.0);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (w == 0) sc.mean0[q] = 2.0 * v;
    }
    const unsigned ev = sc.e[0], eu = sc.e[1], ew = sc.e[2], et = sc.e[3];
    // schedules of transforms i0 .. i0 + n - 1 from their 1-norms
    auto schedule = [&](int i0, int n) {
        __syncthreads();
        if (tid < n) {
            int S;
            sc.back[i0 + tid] = fx_schedule(lg, three, fx_l1_bits(sc.l1[i0 + tid]), S);
            sc.S[i0 + tid] = S;
        }
    };
    // leading bits in use of the fields of pair i, from the physical values
    auto tops = [&](int i, unsigned x, unsigned yv) {
        x = __reduce_or_sync(0xffffffffu, x);
        yv = __reduce_or_sync(0xffffffffu, yv);
        if ((tid & 31) == 0) {
            atomicOr(&sc.top[2 * i], yv);  // first field of the pair: the exchanged y
            atomicOr(&sc.top[2 * i + 1], x);
        }
    };
    fxc reg[PAIR ? 1 : MAXPER];
    const fxc *R1 = nullptr, *R2 = nullptr;
    for (int j = n_m + 1 + tid; j < Pn - n_m; j += nth) {
        X[j] = fxc{0, 0};
        if (PAIR) X[Pn + j] = fxc{0, 0};
    }
    {
        unsigned w0 = 0u, w1 = 0u;
        for (int m = tid; m <= n_m; m += nth) {
            w0 += phi_pack(phi_coef(src[m], ev), phi_coef(src[M + m], eu), m, Pn, X);
            if (PAIR) w1 += phi_pack(phi_coef(src[2 * M + m], ew), phi_coef(src[3 * M + m], et), m, Pn, X + Pn);
        }
        w0 = __reduce_add_sync(0xffffffffu, w0);
        if ((tid & 31) == 0) atomicAdd(&sc.l1[0], w0);
        if (PAIR) {
            w1 = __reduce_add_sync(0xffffffffu, w1);
            if ((tid & 31) == 0) atomicAdd(&sc.l1[1], w1);
        }
    }
    if (PAIR) {
        schedule(0, 2);
        R1 = fx_fft<false>(X, Y, tw, 1, lg, three, 2, sc.back);
        R2 = R1 + Pn;
        for (int i = 0; i < 2; ++i) {
            unsigned x = 0u, yv = 0u;
            for (int j = tid; j < Pn; j += nth) {
                x |= fx_top(R1[i * Pn + j].x);
                yv |= fx_top(R1[i * Pn + j].y);
            }
            tops(i, x, yv);
        }
    } else {
        for (int i = 0; i < 2; ++i) {
            if (i) {
                unsigned w1 = 0u;
                for (int m = tid; m <= n_m; m += nth)
                    w1 += phi_pack(phi_coef(src[2 * M + m], ew), phi_coef(src[3 * M + m], et), m, Pn, X);
                for (int j = n_m + 1 + tid; j < Pn - n_m; j += nth) X[j] = fxc{0, 0};
                w1 = __reduce_add_sync(0xffffffffu, w1);
                if ((tid & 31) == 0) atomicAdd(&sc.l1[1], w1);
            }
            schedule(i, 1);
            R2 = fx_fft<false>(X, Y, tw, 1, lg, three, 1, sc.back + i);
            unsigned x = 0u, yv = 0u;
            for (int j = tid; j < Pn; j += nth) {
                x |= fx_top(R2[j].x);
                yv |= fx_top(R2[j].y);
            }
            tops(i, x, yv);
            if (i == 0) {
                if (P.cfl_max)
                    cfl_rates_fx(P, R2, k, sc.S[0] + (int)ev - 1022 - FX_BITS + 1, sc.S[0] + (int)eu - 1022 - FX_BITS + 1,
                                 ev == 0x7ff || eu == 0x7ff, sc.cfl);
#pragma unroll
                for (int n = 0; n < (PAIR ? 1 : MAXPER); ++n) {
                    const int j = tid + n * nth;
                    if (j < Pn) reg[n] = R2[j];
                }
                __syncthreads();
            }
        }
    }
    __syncthreads();
    if (PAIR && P.cfl_max)
        cfl_rates_fx(P, R1, k, sc.S[0] + (int)ev - 1022 - FX_BITS + 1, sc.S[0] + (int)eu - 1022 - FX_BITS + 1,
                     ev == 0x7ff || eu == 0x7ff, sc.cfl);
    // free leading bits: |value| < 2^(32 + bits of top), shifted up to below 2^61
    int sh[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) sh[q] = __clz((int)sc.top[q]) - 3;  // (-2 at least)
    // exponents of the shifted physical fields: value = integer 2^x
    const int xv = sc.S[0] + (int)ev - 1022 - FX_BITS + 1 - sh[0], xu = sc.S[0] + (int)eu - 1022 - FX_BITS + 1 - sh[1];
    const int xw = sc.S[1] + (int)ew - 1022 - FX_BITS + 1 - sh[2], xt = sc.S[1] + (int)et - 1022 - FX_BITS + 1 - sh[3];
    unsigned l0 = 0u, l1 = 0u;
    auto up = [](fx64 a, int s) { return s >= 0 ? (fx64)((unsigned long long)a << s) : fx_shr(a, -s); };
    // (v omega, u_phi omega) and (v theta, u_phi theta), each 2^-62 of the integers' product
    auto prods = [&](fxc g1, fxc g2, fxc& p, fxc& r) {
        const fx64 v = up(g1.y, sh[0]), u = up(g1.x, sh[1]), w = up(g2.y, sh[2]), t = up(g2.x, sh[3]);
        p = fxc{fx_mul62(v, w), fx_mul62(u, w)};
        r = fxc{fx_mul62(v, t), fx_mul62(u, t)};
        l0 += fx_l1_part(p.x) + fx_l1_part(p.y);
        l1 += fx_l1_part(r.x) + fx_l1_part(r.y);
    };
    auto norms = [&]() {
        l0 = __reduce_add_sync(0xffffffffu, l0);
        l1 = __reduce_add_sync(0xffffffffu, l1);
        if ((tid & 31) == 0) {
            atomicAdd(&sc.l1[2], l0);
            atomicAdd(&sc.l1[3], l1);
        }
    };
    const bool bv = ev == 0x7ff, bu = eu == 0x7ff, bw = ew == 0x7ff, bt = et == 0x7ff;
    const int ln = three ? -(lg + 1) : -lg;  // 1/n_phi
    // after the stores of phi_split: the means in the place of the transforms' m = 0 entries
    auto means = [&]() {
        __syncthreads();
        if (tid < 4) dst[tid * M] = make_double2(sc.mean0[tid], 0.0);
    };
    if (PAIR) {
        fxc* O = (R1 == X) ? Y : X;
        for (int j = tid; j < Pn; j += nth) {
            fxc p, r;
            prods(R1[j], R2[j], p, r);
            O[j] = p;
            O[Pn + j] = r;
        }
        norms();
        schedule(2, 2);
        const fxc* Z = fx_fft<false>(O, const_cast<fxc*>(R1), tw, 1, lg, three, 2, sc.back + 2);
        phi_split(Z, dst, M, Pn, n_m, three, xv + xw + 62 + sc.S[2] + ln, xu + xw + 62 + sc.S[2] + ln, bv || bw, bu || bw);
        phi_split(Z + Pn, dst + 2 * M, M, Pn, n_m, three, xv + xt + 62 + sc.S[3] + ln, xu + xt + 62 + sc.S[3] + ln,
                  bv || bt, bu || bt);
        means();
    } else {
        fxc* O = (R2 == X) ? Y : X;
#pragma unroll
        for (int n = 0; n < (PAIR ? 1 : MAXPER); ++n) {
            const int j = tid + n * nth;
            if (j < Pn) {
                fxc p;
                prods(reg[n], R2[j], p, reg[n]);
                O[j] = p;
            }
        }
        norms();
        schedule(2, 2);
        const fxc* Z = fx_fft<false>(O, const_cast<fxc*>(R2), tw, 1, lg, three, 1, sc.back + 2);
        phi_split(Z, dst, M, Pn, n_m, three, xv + xw + 62 + sc.S[2] + ln, xu + xw + 62 + sc.S[2] + ln, bv || bw, bu || bw);
        __syncthreads();
#pragma unroll
        for (int n = 0; n < (PAIR ? 1 : MAXPER); ++n) {
            const int j = tid + n * nth;
            if (j < Pn) X[j] = reg[n];
        }
        Z = fx_fft<false>(X, Y, tw, 1, lg, three, 1, sc.back + 3);
        phi_split(Z, dst + 2 * M, M, Pn, n_m, three, xv + xt + 62 + sc.S[3] + ln, xu + xt + 62 + sc.S[3] + ln, bv || bt,
                  bu || bt);
        means();
    }
}

// ---------------------------------------------------------------------------
// Diagnostics from G1 (radial-grid Fourier coefficients written by K1):
// per mode, sums over the Gauss-Lobatto points with quadrature weights q_k
// (int f s ds ~ sum_k q_k f_k) of |u_s|^2 + |u_phi|^2 and |omega|^2;
// u_s = (h^2/s) v.  out[m*2 + 0], out[m*2 + 1].
// ---------------------------------------------------------------------------
__global__ void k_diag_modes(StepParams P, const double2* __restrict__ G1, const double* __restrict__ q,
                             double* __restrict__ out) {
    const int m = blockIdx.x, M = P.M;
    double e = 0.0, z = 0.0;
    for (int k = threadIdx.x; k < P.n_r; k += blockDim.x) {
        const double f = P.coll ? P.inv_s[k] : P.h2[k] * P.inv_s[k];
        const double2 v = G1[g_index(k, 0, m, M)], up = G1[g_index(k, 1, m, M)], w = G1[g_index(k, 2, m, M)];
        const double us2 = f * f * (v.x * v.x + v.y * v.y);
        e += q[k] * (us2 + up.x * up.x + up.y * up.y);
        z += q[k] * (w.x * w.x + w.y * w.y);
    }
    __shared__ double red[2][32];
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = e;
        red[1][threadIdx.x >> 5] = z;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            a += red[0][i];
            b += red[1][i];
        }
        out[2 * m] = a;
        out[2 * m + 1] = b;
    }
}

// per radius: max |u_s| and max |u_phi| over the azimuthal grid (Eq. fft of
// g = u_s + i l u_phi, l a balancing power of two); out[k*2 + 0], out[k*2 + 1].
__global__ void __launch_bounds__(512) k_phi_cfl(StepParams P, const double2* __restrict__ G1,
                                                 double* __restrict__ out) {
    extern __shared__ double2 sm[];
    const int k = blockIdx.x;
    const int Pn = P.n_phi, M = P.M, n_m = P.n_m;
    double2* X = sm;
    double2* Y = sm + Pn;
    const double f = P.coll ? P.inv_s[k] : P.h2[k] * P.inv_s[k];
    const double2* src = G1 + g_index(k, 0, 0, M);
    __shared__ double red4[4 * 32], mx[4];
    block_max_abs(src, M, 2, n_m + 1, mx, red4);
    const double l = pow2_ratio(f * mx[0], mx[1]);
    load_packed_spectrum(X, src, M, Pn, n_m, f, l);
    double2* R = fft_batched<+1>(X, Y, P.plan_p, 1);
    double ms = 0.0, mp = 0.0;
    for (int j = threadIdx.x; j < Pn; j += blockDim.x) {
        ms = fmax(ms, fabs(R[j].x));
        mp = fmax(mp, fabs(R[j].y));
    }
    __shared__ double red[2][32];
    for (int o = 16; o > 0; o >>= 1) {
        ms = fmax(ms, __shfl_xor_sync(0xffffffffu, ms, o));
        mp = fmax(mp, __shfl_xor_sync(0xffffffffu, mp, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = ms;
        red[1][threadIdx.x >> 5] = mp;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            a = fmax(a, red[0][i]);
            b = fmax(b, red[1][i]);
        }
        out[2 * k] = a;
        out[2 * k + 1] = b / l;
    }
}

// per radius: the physical-grid values (Eq. fft) of u_s, u_phi, omega and theta,
// out[k * n_phi + j]; u_s = (h^2/s) v (integration) or v/s (collocation).  The
// pairs (u_s, u_phi) and (omega, theta) travel in one complex transform each,
// balanced by powers of two.
__global__ void __launch_bounds__(512) k_phi_fields(StepParams P, const double2* __restrict__ G1,
                                                    double* __restrict__ us, double* __restrict__ uphi,
                                                    double* __restrict__ omega, double* __restrict__ theta) {
    extern __shared__ double2 sm[];
    const int k = blockIdx.x;
    const int Pn = P.n_phi, M = P.M, n_m = P.n_m;
    double2* X = sm;
    double2* Y = sm + Pn;
    const double f = P.coll ? P.inv_s[k] : P.h2[k] * P.inv_s[k];
    __shared__ double red4[4 * 32], mx[4];
    block_max_abs(G1 + g_index(k, 0, 0, M), M, 4, n_m + 1, mx, red4);
    for (int pass = 0; pass < 2; ++pass) {
        const double2* src = G1 + g_index(k, 2 * pass, 0, M);
        const double fa = (pass == 0) ? f : 1.0;
        const double l = pow2_ratio(fa * mx[2 * pass], mx[2 * pass + 1]);
        load_packed_spectrum(X, src, M, Pn, n_m, fa, l);
        double2* R = fft_batched<+1>(X, Y, P.plan_p, 1);
        double* oa = (pass == 0) ? us : omega;
        double* ob = (pass == 0) ? uphi : theta;
        const double il = 1.0 / l;
        for (int j = threadIdx.x; j < Pn; j += blockDim.x) {
            oa[(size_t)k * Pn + j] = R[j].x;
            ob[(size_t)k * Pn + j] = R[j].y * il;
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_diagnostics(const StepParams& P, const double2* G1, const double* q, double* mode_sums,
                               double* radius_max, cudaStream_t st) {
    k_diag_modes<<<P.M, 128, 0, st>>>(P, G1, q, mode_sums);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    const size_t sm = smem_phi_products(P);
    const int nth = P.n_phi > 256 * MAXPER ? 512 : 256;
    err = cudaFuncSetAttribute(k_phi_cfl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    k_phi_cfl<<<P.n_r, nth, sm, st>>>(P, G1, radius_max);
    return cudaGetLastError();
}

cudaError_t launch_phi_fields(const StepParams& P, const double2* G1, double* us, double* uphi, double* omega,
                              double* theta, cudaStream_t st) {
    const size_t sm = smem_phi_products(P);
    cudaError_t err = cudaFuncSetAttribute(k_phi_fields, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    k_phi_fields<<<P.n_r, 256, sm, st>>>(P, G1, us, uphi, omega, theta);
    return cudaGetLastError();
}

size_t smem_spec_to_grid(const StepParams& P) {
    const int L = 2 * P.K;
    const size_t c = P.fp32 ? sizeof(float2) : sizeof(double2);
    return c * (2 * radial_batch(P) * L + 3 * P.n_r);
}
size_t smem_phi_products(const StepParams& P) {
    return (P.fp32 ? sizeof(float2) : sizeof(double2)) * 2 * P.n_phi;
}
// a3: two vectors at a time at most in the fixed-point kernel
size_t smem_grid_to_spec(const StepParams& P) {
    if (P.fp32) return smem_spec_to_grid(P);
    return sizeof(double2) * (2 * (size_t)std::min(2, radial_batch(P)) * 2 * P.K + 3 * P.n_r);
}

// The explicit stage runs on double2 (FP64) or float2 (option "precision" =
// mixed) grid arrays; G1, G2 hold either type.
// ---------------------------------------------------------------------------
// Large radial grids (K = n_r - 1 >= LEAN_K, the half-length DCT-I):
// a1 and a3 with three shared arrays of K + 1 entries, X, C, Y (98 KB at
// n_r = 2049), instead of the batched layout's 2 x 2K + 3 n_r entries (229 KB),
// so that two CTAs share an SM and hide each other's barrier and shared-memory
// latency (one CTA left the FP64 pipe ~50 % idle).  The fields of a mode go
// through the transform one after another; the derivative scans run in place on
// C with X as scratch; the DCT-I works in place on the pair (X, Y).  The same
// equations, in the same precision, as k_spec_to_grid / k_grid_to_spec.
// ---------------------------------------------------------------------------
constexpr int LEAN_K = 1024;

__device__ __forceinline__ double2 warp_sum(double2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// The mixed-precision (FP32) stage takes the lean layout only when asked
// (radial_lean = 1): at n_r = 2049 it ran the mixed step 5.99 against 6.53 ms,
// but the half-length DCT-I builds its odd outputs from a prefix sum over the
// FP32 transform's outputs, which accumulates their rounding: 2.2e-7 from the
// FP64 path after 20 steps against 1.1e-8 with the batched layout's
// even-extension transform.
__host__ __device__ inline bool lean_radial(const StepParams& P) {
    if (P.plan_h.L != P.K || P.K < 128 || P.radial_lean == 0) return false;
    if (P.fp32) return P.radial_lean > 0;
    return P.radial_lean > 0 || P.K >= LEAN_K;
}

// fixed-point radial transforms of the FP64 stage (option "radial_dd"): 1 always, 0
// never (FP64 transforms in either layout), -1 (default) in the batched layout and, in
// the lean one, from its own default size
inline bool radial_fx(const StepParams& P) {
    if (!P.fx_r || P.radial_dd == 0) return false;
    return P.radial_dd > 0 || !lean_radial(P) || P.K >= LEAN_K;
}

// The FP64 accumulators of dct1_pair: exact widening of FP32 values by their
// bits (no FP64-unit conversion), the nearest float on the way back
__device__ __forceinline__ double acc_of(double v) { return v; }
__device__ __forceinline__ double acc_of(float v) { return f2d_bits(v); }
__device__ __forceinline__ double2 acc_of(double2 v) { return v; }
__device__ __forceinline__ double2 acc_of(float2 v) { return make_double2(f2d_bits(v.x), f2d_bits(v.y)); }
template <class T>
__device__ __forceinline__ T from_acc(double2 v);
template <>
__device__ __forceinline__ double2 from_acc<double2>(double2 v) { return v; }
template <>
__device__ __forceinline__ float2 from_acc<float2>(double2 v) { return make_float2(f32_from_bits(v.x), f32_from_bits(v.y)); }

// DCT-I of x_0..x_K in X (K + 1 entries):
//   C_k = x_0 + (-1)^k x_K + 2 sum_{j=1}^{K-1} x_j cos(pi j k / K),  k = 0..K,
// by one complex FFT of length K, as dct1_batched: y_j = (x_j + x_{K-j})/2
// - sin(pi j/K)(x_j - x_{K-j}) formed in place pair by pair (j, K - j),
// F = FFT(y), C_{2k} = F_k + F_{K-k}, and the odd outputs from
// C_1 = sum_j (x_j - x_{K-j}) cos(pi j/K) by C_{2k+1} = C_{2k-1} - i(F_k - F_{K-k}),
// the prefix sum taken by the whole CTA in FP64 (also for FP32 data, whose
// transform and pair arithmetic stay FP32).  The FFT ping-pongs between X and Y;
// the outputs go to the buffer that does not hold F, which is returned.
// Starts and ends with __syncthreads().
template <class T>
__device__ T* dct1_pair(T* X, T* Y, const StepParams& P) {
    using RT = typename Cx<T>::R;
    const int K = P.plan_h.L, H = K / 2;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nth >> 5;
    const T* tw = Cx<T>::tw(P.plan_r);  // tw[j] = (cos(pi j/K), -sin(pi j/K))
    __shared__ double2 wsum[NTHREADS_R / 32];
    __shared__ double2 c1;
    __syncthreads();
    double2 acc = make_double2(0.0, 0.0);
    for (int j = tid; j < H; j += nth) {
        if (j == 0) {
            const T a = X[0], b = X[K];
            T h = a;
            h.x = (RT)0.5 * (a.x + b.x);
            h.y = (RT)0.5 * (a.y + b.y);
            X[0] = h;
            acc = acc_of(csub(a, b));
        } else {
            const T a = X[j], b = X[K - j];
            const RT sn = -tw[j].y, cs = tw[j].x;
            const T sum = cadd(a, b), dif = csub(a, b);
            T lo = sum, hi = sum;
            lo.x = fmat(-sn, dif.x, (RT)0.5 * sum.x);
            lo.y = fmat(-sn, dif.y, (RT)0.5 * sum.y);
            hi.x = fmat(sn, dif.x, (RT)0.5 * sum.x);
            hi.y = fmat(sn, dif.y, (RT)0.5 * sum.y);
            X[j] = lo;
            X[K - j] = hi;
            const double2 dd = acc_of(dif);
            const double c2 = 2.0 * acc_of(cs);
            acc.x = fma(c2, dd.x, acc.x);
            acc.y = fma(c2, dd.y, acc.y);
        }
    }
    // (j = H: y_H = x_H, and its term of C_1 vanishes)
    acc = warp_sum(acc);
    if (lane == 0) wsum[warp] = acc;
    __syncthreads();
    if (tid == 0) {
        double2 t = wsum[0];
        for (int w = 1; w < nw; ++w) t = cadd(t, wsum[w]);
        c1 = t;
    }
    T* F = fft_batched<+1>(X, Y, P.plan_h, 1);  // begins with a barrier
    T* O = (F == X) ? Y : X;
    for (int k = tid; k <= H; k += nth) O[2 * k] = cadd(F[k], F[k == 0 ? 0 : K - k]);
    // odd outputs: each thread a contiguous chunk of k in [0, H), its sum of
    // d_k = -i (F_k - F_{K-k}) (d_0 = 0), a block-wide exclusive scan, then the chunk
    const int chunk = (H + nth - 1) / nth;
    const int lo = min(tid * chunk, H), hi = min(lo + chunk, H);
    double2 tot = make_double2(0.0, 0.0);
    for (int k = max(lo, 1); k < hi; ++k) {
        const double2 df = acc_of(csub(F[k], F[K - k]));
        tot.x += df.y;
        tot.y -= df.x;
    }
    double2 inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double ux = __shfl_up_sync(0xffffffffu, inc.x, o);
        const double uy = __shfl_up_sync(0xffffffffu, inc.y, o);
        if (lane >= o) {
            inc.x += ux;
            inc.y += uy;
        }
    }
    __syncthreads();  // c1 and the even outputs are published; wsum is free again
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    double2 run = c1;
    for (int w = 0; w < warp; ++w) run = cadd(run, wsum[w]);
    run.x += inc.x - tot.x;
    run.y += inc.y - tot.y;
    for (int k = lo; k < hi; ++k) {
        if (k > 0) {
            const double2 df = acc_of(csub(F[k], F[K - k]));
            run.x += df.y;
            run.y -= df.x;
        }
        O[2 * k + 1] = from_acc<T>(run);
    }
    __syncthreads();
    return O;
}

// The FP64 coefficients as the lean kernels' element type: unchanged in FP64,
// the nearest float in FP32 (bit-level, off the FP64 unit)
template <class T>
__device__ __forceinline__ T to_elem(double2 v);
template <>
__device__ __forceinline__ double2 to_elem<double2>(double2 v) { return v; }
template <>
__device__ __forceinline__ float2 to_elem<float2>(double2 v) { return make_float2(f32_from_bits(v.x), f32_from_bits(v.y)); }

// CTAs per SM of the lean kernels: two in FP64 (98 KB of shared memory at
// n_r = 2049), three in FP32 (the FP32 arrays and the FP64 coefficients of a3)
template <class T>
constexpr int lean_ctas() { return sizeof(T) == sizeof(double2) ? 2 : 3; }

// T = double2: the FP64 stage; T = float2: the mixed-precision stage (FP32
// transforms and field arithmetic, grid arrays in FP32, the FP64 state read and
// the analysed coefficients widened to FP64 for the banded applies).
template <class T>
__global__ void __launch_bounds__(NTHREADS_R, lean_ctas<T>()) k_spec_to_grid_lean(StepParams P, VecSet y,
                                                                                  T* __restrict__ G1) {
    chain_wait();
    using RT = typename Cx<T>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, N = P.n_r, nc = P.nc, M = P.M;
    T* X = reinterpret_cast<T*>(smraw);
    T* C = X + N;   // plain coefficients (Psi, then its derivatives; u_bar)
    T* Y = C + N;   // second DCT buffer (u_bar' for m = 0)
    const int tid = threadIdx.x, nth = blockDim.x;
    const double Cw = P.cnorm, Cw0 = 0.5 * P.cnorm;
    const RT dm = (RT)m;
    const T zero = Cx<T>::make(0.0, 0.0);

    for (int n = tid; n < N; n += nth) {
        double2 a = make_double2(0.0, 0.0);
        if (n < nc) {
            const double w = (n == 0) ? Cw0 : Cw;
            a = (m > 0) ? cscale(y.psi[(size_t)m * nc + n], w) : make_double2(y.u[n] * w, 0.0);
        }
        C[n] = to_elem<T>(a);
    }
    __syncthreads();
    T* PF = P.pump ? reinterpret_cast<T*>(P.pump_F) + (size_t)m * N : nullptr;
    __shared__ double red[4 * 32], mx[4];
    RT lam = (RT)1;
    if (m == 0) {  // u_bar and lam u_bar' packed into one transform (lam a power of two)
        cheb_derivative_scan(C, Y, X, N, P.inv_a);
        block_max_abs(C, N, 2, N, mx, red);
        lam = (RT)pow2_ratio(mx[0], mx[1]);
    }
    // fields: 0 Psi, 1 Psi', 2 Psi'', 3 theta (m >= 1); 4 packed u_bar, 3 theta (m = 0)
    const int nf = (m > 0) ? 4 : 2;
    for (int i = 0; i < nf; ++i) {
        const int fid = (m > 0) ? i : (i == 0 ? 4 : 3);
        if (m > 0 && (fid == 1 || fid == 2)) cheb_derivative_scan(C, C, X, N, P.inv_a);  // C <- dC/ds
        for (int j = tid; j <= K; j += nth) {
            T v;
            if (fid <= 2) {
                v = C[j];
            } else if (fid == 3) {
                v = (j < nc) ? to_elem<T>(cscale(y.th[(size_t)m * nc + j], (j == 0) ? Cw0 : Cw)) : zero;
            } else {
                v = C[j];
                v.y = lam * Y[j].x;
            }
            X[j] = (j == 0 || j == K) ? cscale(v, (RT)2) : v;
        }
        T* Z = dct1_pair(X, Y, P);
        for (int k = tid; k < N; k += nth) {
            const T g = cscale(Z[k], (RT)0.5);  // value of the series at x_k
            const RT s = Tab<T>::s(P, k), h2 = Tab<T>::h2(P, k), is = Tab<T>::is(P, k);
            T* out = G1 + g_index(k, 0, m, M);
            if (fid == 0) {
                out[0] = cmul_i(g, dm);
                out[M] = cscale(g, (RT)3 * s);
                out[2 * M] = cscale(g, (RT)6 + dm * dm * h2 * is * is);
                if (PF) {
                    const RT U = (RT)P.pump_ups[k];
                    PF[k] = cadd(cscale(g, -U * ((RT)P.pump_cr[k] + dm * dm)), cmul_i(g, -U * dm * (RT)P.pump_ci[k]));
                }
            } else if (fid == 1) {
                out[M] = csub(out[M], cscale(g, h2));
                out[2 * M] = csub(out[2 * M], cscale(g, h2 * is - (RT)5 * s));
                if (PF) PF[k] = cadd(PF[k], cscale(g, (RT)P.pump_ups[k] * (RT)0.5 * s));
            } else if (fid == 2) {
                out[2 * M] = csub(out[2 * M], cscale(g, h2));
                if (PF) PF[k] = csub(PF[k], cscale(out[2 * M], (RT)P.pump_ups[k]));
            } else if (fid == 3) {
                out[3 * M] = g;
            } else {
                T o = zero;
                out[0] = o;
                o.x = g.x;
                out[M] = o;
                o.x = g.y / lam + g.x * is;
                out[2 * M] = o;
                if (PF) {
                    const RT w0 = g.y / lam + g.x * is;
                    T pf = zero;
                    pf.x = (RT)P.pump_ups[k] * g.x * ((RT)1 + (RT)(0.5 * P.E) * w0);
                    PF[k] = pf;
                }
            }
        }
        __syncthreads();
    }
}

// byte offset of a3's FP64 coefficient array behind the three T arrays (16-byte
// aligned); in FP64 the coefficients overwrite C instead
template <class T>
__host__ __device__ inline size_t lean_cd_offset(int n_r) {
    return sizeof(T) == sizeof(double2) ? sizeof(T) * (size_t)n_r : (sizeof(T) * 3 * (size_t)n_r + 15) / 16 * 16;
}

template <class T>
__global__ void __launch_bounds__(NTHREADS_R, lean_ctas<T>()) k_grid_to_spec_lean(StepParams P, const T* G2,
                                                                                  VecSet y, VecSet e) {
    chain_wait();
    using RT = typename Cx<T>::R;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, N = P.n_r, nc = P.nc, M = P.M;
    T* X = reinterpret_cast<T*>(smraw);
    T* C = X + N;
    T* Y = C + N;
    double2* Cd = reinterpret_cast<double2*>(smraw + lean_cd_offset<T>(N));  // FP64 coefficients
    const int tid = threadIdx.x, nth = blockDim.x;
    const RT dm = (RT)m, iK = (RT)(1.0 / (double)K), hK = (RT)(0.5 / (double)K);
    const double dmd = (double)m, hc = 0.5 * P.cnorm;
    const T* PF = P.pump ? reinterpret_cast<const T*>(P.pump_F) + (size_t)m * N : nullptr;
    const double bfac = P.Ra / P.Pr * (double)m / P.s_o;
    // field 0: N_omega (m >= 1) or N_u (m = 0); field 1: N_theta
    for (int fld = 0; fld < 2; ++fld) {
        T* W = X;  // the buffer holding the grid values to analyse
        if (fld == 1 || m > 0) {
            // plain coefficients of F = h^2 [v omega]_m (or h^2 [v theta]_m), d/ds of them
            const int f = (fld == 0) ? 0 : 2;
            for (int j = tid; j <= K; j += nth) X[j] = cscale(G2[g_index(j, f, m, M)], Tab<T>::h2(P, j));
            const T* Z = dct1_pair(X, Y, P);
            for (int n = tid; n <= K; n += nth) C[n] = cscale(Z[n], (n == 0 || n == K) ? hK : iK);
            __syncthreads();
            cheb_derivative_scan(C, C, X, N, P.inv_a);
            for (int j = tid; j <= K; j += nth) X[j] = (j == 0 || j == K) ? cscale(C[j], (RT)2) : C[j];
            const T* D = dct1_pair(X, Y, P);
            W = (D == X) ? Y : X;
            for (int k = tid; k <= K; k += nth) {
                const T dF = cscale(D[k], (RT)0.5);
                const RT is = Tab<T>::is(P, k);
                T val;
                if (fld == 0) {
                    val = cscale(cadd(dF, cmul_i(G2[g_index(k, 1, m, M)], dm)), is);
                    if (PF) val = csub(val, PF[k]);
                } else {
                    val = csub(cscale(cadd(dF, cmul_i(G2[g_index(k, 3, m, M)], dm)), is), G2[g_index(k, 2, m, M)]);
                }
                W[k] = val;
            }
        } else {  // N_u = (h^2/s) [v omega]_0 (+ pumping)
            for (int k = tid; k <= K; k += nth) {
                T val = cscale(G2[g_index(k, 0, m, M)], Tab<T>::h2(P, k) * Tab<T>::is(P, k));
                if (PF) val = cadd(val, PF[k]);
                W[k] = val;
            }
        }
        // Eq. icheb of the grid values, truncated to n < nc
        const T* Z = dct1_pair(W, (W == X) ? Y : X, P);
        // N_omega_hat, with the buoyancy (Ra/Pr)(i m/s_o) theta_hat added before the
        // one C^I apply (Eq. psi_int applies C^I to their sum); Z lives in X or Y,
        // never where the FP64 coefficients go
        const bool buoy = (fld == 0 && m > 0 && !P.buoy_imp);
        for (int n = tid; n < nc; n += nth) {
            const double2 v = cscale(acc_of(Z[n]), hc);
            Cd[n] = buoy ? cadd(v, cmul_i(y.th[(size_t)m * nc + n], bfac)) : v;
        }
        __syncthreads();
        // integrated right-hand sides; the linear couplings read the FP64 state
        for (int k = tid; k < nc; k += nth) {
            if (fld == 0) {
                if (m > 0) {
                    double2 ep = make_double2(0.0, 0.0);
                    if (k >= 4) ep = band_row<8>(P.ops.band[OP_C], Cd, k, nc);
                    e.psi[(size_t)m * nc + k] = ep;
                } else {
                    e.psi[k] = make_double2(0.0, 0.0);
                    e.u[k] = (k >= 2) ? -band_row<4>(P.ops.band[OP_D], Cd, k, nc).x : 0.0;
                }
            } else {
                double2 et = make_double2(0.0, 0.0);
                if (k >= 2) {
                    const double2 dn = band_row<4>(P.ops.band[OP_D], Cd, k, nc);
                    if (m > 0) {
                        const double2 gp = band_row<4>(P.ops.band[OP_G], y.psi + (size_t)m * nc, k, nc);
                        et = csub(cmul_i(gp, -P.tc * dmd), dn);
                    } else {
                        et = cscale(dn, -1.0);
                    }
                }
                e.th[(size_t)m * nc + k] = et;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The lean layout in fixed point (option "radial_dd", the FP64 stage's default from
// n_r = 1025): two buffers of K fixed-point entries and one array of n_r FP64 values
// (98 KB at n_r = 2049: two CTAs of 512 threads share an SM), the vectors of a mode
// one after another through a half-length DCT-I.  Against double-float transforms
// in the same layout: 1025 x 3072 343 -> 263 (a1) and 581 -> 440 us (a3), 2049 x 6144
// 1124 -> 889 and 1607 -> 1633 us (1598 with shifts that round down); the derivative of
// 2049 grid values 1.4e-7 -> 4e-9 off (1.3e-9 by the FP64 transform of this form); from n_r =
// 1025, since at 513 the batched layout is faster (a1 52 -> 35, a3 90 -> 49 us at 513 x 384).
// ---------------------------------------------------------------------------
constexpr int NTHREADS_LX = 512;

struct DctHalf {
    long long c1h[NTHREADS_LX / 32][2], c1l[NTHREADS_LX / 32][2];  // partial sums of C_1
    long long c1[2];                                              // C_1 2^-(S + 1)
    long long run[NTHREADS_LX / 32][2];                           // odd outputs' increments of a warp
    double tot[NTHREADS_LX / 32];                                 // derivative sums of a warp
};

// DCT-I of K + 1 values by one complex transform of length K, as dct1_pair: y_j = (x_j + x_{K-j})/2
// - sin(pi j/K)(x_j - x_{K-j}), F = FFT(y), C_{2k} = F_k + F_{K-k}, and the odd outputs
// from C_1 = sum_j (x_j - x_{K-j}) cos(pi j/K) by prefix sums of -i (F_k - F_{K-k})
// (the transform here is the forward one, F_{K-k} in the place of F_k, which
// changes the sign).  The integer prefix sums are exact; what accumulates is the
// rounding of F, about 2^-55 of its largest value a term.
// The schedule takes the 1-norms of x and y together: the outputs are bounded by
// x's, and y's can be far below it (sin(pi j/K) is small near the ends).
// val(t): FP64 part t & 1 of entry t / 2, t < 2 n, exponents gathered before a
// barrier; twice: the end entries count twice.  X, Y: K points each.  On return F holds
// the transform and O[k] the odd outputs C_{2k+1}; half_part reads an output.
// Ends with a barrier.
template <class V>
__device__ __forceinline__ void dct1_half_fx(const StepParams& P, FxScale& sc, DctHalf& dh, int v, int n, bool twice,
                                             fxc* X, fxc* Y, fxc*& F, fxc*& O, V val) {
    const int K = P.K, H = K >> 1;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nth >> 5;
    const fxw* tw = reinterpret_cast<const fxw*>(P.fx_r);  // (cos(pi j/K), -sin(pi j/K))
    {
        const int part = tid & 1;
        const int e = (int)sc.e[v][part];
        fx64* x = reinterpret_cast<fx64*>(X) + part;
        unsigned l1 = 0u;
        fx64 ch = 0, cl = 0;
        auto get = [&](int j) -> fx64 {
            if (j >= n || e == 0x7ff) return 0;
            const fx64 q = fx_shr(fx_from(val(2 * j + part), e), 2);  // pairs grow by less than four
            return (twice && (j == 0 || j == K)) ? 2 * q : q;
        };
        for (int j = tid >> 1; j <= H; j += nth >> 1) {
            const fx64 a = get(j);
            l1 += fx_l1_part(a);
            if (j == H) {
                x[2 * H] = a;
                continue;
            }
            const fx64 b = get(K - j);
            l1 += fx_l1_part(b);
            const fx64 hs = fx_half(a + b), dif = a - b;
            fx64 c;
            if (j == 0) {
                x[0] = hs;
                c = dif;
            } else {
                const fxw w = fx_ldw(tw + j);
                const fx64 sd = fx_mulc(dif, w.y1, w.y0);  // -sin(pi j/K) dif
                x[2 * j] = hs + sd;
                x[2 * (K - j)] = hs - sd;
                l1 += fx_l1_part(hs + sd) + fx_l1_part(hs - sd);
                c = 2 * fx_mulc(dif, w.x1, w.x0);
            }
            ch += c >> 32;
            cl += (fx64)(unsigned)c;
        }
        l1 = __reduce_add_sync(0xffffffffu, l1);
        if (lane == 0) atomicAdd(&sc.l1[v], l1);
#pragma unroll
        for (int o = 2; o < 32; o <<= 1) {
            ch += __shfl_xor_sync(0xffffffffu, ch, o);
            cl += __shfl_xor_sync(0xffffffffu, cl, o);
        }
        if (lane < 2) {
            dh.c1h[warp][lane] = ch;
            dh.c1l[warp][lane] = cl;
        }
    }
    __syncthreads();
    const int lg = 31 - __clz(K);  // transform length 2^lg
    if (tid < 2) {
        int S;
        const unsigned bk = fx_schedule(lg, false, fx_l1_bits(sc.l1[v]), S);
        if (tid == 0) {
            sc.back[v] = bk;
            sc.S[v] = S;
        }
        fx64 h = 0, l = 0;
        for (int w = 0; w < nw; ++w) {
            h += dh.c1h[w][tid];
            l += dh.c1l[w][tid];
        }
        h += l >> 32;
        l &= 0xffffffffll;
        dh.c1[tid] = (fx64)((unsigned long long)h << (31 - S)) + fx_shr(l, S + 1);  // (S < 31)
    }
    F = fx_fft<true>(X, Y, tw, 2, lg, false, 1, sc.back + v);
    O = (F == X) ? Y : X;
    // odd outputs: each thread a run of k, its increments, a scan over the CTA
    const int chunk = (H + nth - 1) / nth;
    const int lo = min(tid * chunk, H), hi = min(lo + chunk, H);
    auto inc = [&](int k) {  // (the roundings of the two halves cancel on average)
        const fxc p = F[k], q = F[K - k];
        return fxc{(q.y >> 1) - (p.y >> 1), (p.x >> 1) - (q.x >> 1)};
    };
    fxc tot = fxc{0, 0};
    for (int k = max(lo, 1); k < hi; ++k) tot = fx_add(tot, inc(k));
    fxc sum = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const fx64 ux = __shfl_up_sync(0xffffffffu, sum.x, o), uy = __shfl_up_sync(0xffffffffu, sum.y, o);
        if (lane >= o) sum = fx_add(sum, fxc{ux, uy});
    }
    if (lane == 31) {
        dh.run[warp][0] = sum.x;
        dh.run[warp][1] = sum.y;
    }
    __syncthreads();
    // C_1 and the runs of the warps below: lane l those of warp l
    fxc run = fxc{0, 0};
    if (lane < warp) run = fxc{dh.run[lane][0], dh.run[lane][1]};
#pragma unroll
    for (int o = 1; o < NTHREADS_LX / 32; o <<= 1)
        run = fx_add(run, fxc{__shfl_xor_sync(0xffffffffu, run.x, o), __shfl_xor_sync(0xffffffffu, run.y, o)});
    run.x = __shfl_sync(0xffffffffu, run.x, 0) + dh.c1[0];
    run.y = __shfl_sync(0xffffffffu, run.y, 0) + dh.c1[1];
    run = fx_add(run, fx_sub(sum, tot));
    for (int k = lo; k < hi; ++k) {
        if (k > 0) run = fx_add(run, inc(k));
        O[k] = run;
    }
    __syncthreads();
}
// 2^p times part of output C_k of vector v
__device__ __forceinline__ double half_part(const FxScale& sc, int v, const fxc* F, const fxc* O, int K, int k, int part,
                                            int p) {
    const int kk = k >> 1;
    fx64 c;
    if (k & 1) {
        c = part ? O[kk].y : O[kk].x;
    } else {
        const fxc* f0 = F + kk;
        const fxc* f1 = F + (kk ? K - kk : 0);
        c = part ? fx_avg(f0->y, f1->y) : fx_avg(f0->x, f1->x);
    }
    const int ex = (int)sc.e[v][part];
    return fx_to(c, sc.S[v] + 1 - 1022 - (FX_BITS - 2) + p + ex, ex == 0x7ff);
}

// Chebyshev derivative of FP64 plain coefficients (the sums of cheb_derivative_scan)
// by the whole CTA: warp w takes one index parity of one component (w & 3) in
// the w >> 2-th of nw / 4 segments.  The exponents of d join vector v.  Ends
// with a barrier.
__device__ __forceinline__ void cheb_derivative_cta(const double2* c, double2* d, int n, int nd, double scale, DctHalf& dh,
                                                    FxScale& sc, int v) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nseg = blockDim.x >> 7;
    const int q = warp & 1, part = (warp >> 1) & 1, seg = warp >> 2;
    const double* cs = reinterpret_cast<const double*>(c) + part;
    double* ds = reinterpret_cast<double*>(d) + part;
    const int len = (n - q + 1) / 2;
    const int per = (len + 32 * nseg - 1) / (32 * nseg);
    const int i0 = min((seg * 32 + lane) * per, len), i1 = min(i0 + per, len);
    double acc = 0.0;
    for (int i = i1 - 1; i >= i0; --i) {
        const int k = 2 * i + q;
        if (k > 0) {
            acc = fma((double)(2 * k), cs[2 * k], acc);
            ds[2 * (k - 1)] = acc;
        }
    }
    double sfx = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double x = __shfl_down_sync(0xffffffffu, sfx, o);
        if (lane + o < 32) sfx += x;
    }
    if (lane == 0) dh.tot[warp] = sfx;
    __syncthreads();
    double off = sfx - acc;
    for (int s = seg + 1; s < nseg; ++s) off += dh.tot[4 * s + (warp & 3)];
    unsigned ex = 0u;
    for (int i = i0; i < i1; ++i) {
        const int k = 2 * i + q;
        if (k > 0) {
            const double x = (ds[2 * (k - 1)] + off) * ((k == 1) ? 0.5 * scale : scale);
            ds[2 * (k - 1)] = x;
            const unsigned e = fx_exponent(x);
            ex = max(ex, (k == 1 && e) ? e + 1u : e);
        }
    }
    if (n <= nd && q == 0 && seg == 0 && lane == 0) ds[2 * (n - 1)] = 0.0;  // (unless d ends before it)
    ex = __reduce_max_sync(0xffffffffu, min(ex, 0x7ffu));
    if (lane == 0) atomicMax(&sc.e[v][part], ex);
    __syncthreads();
}

__global__ void __launch_bounds__(NTHREADS_LX, 2) k_spec_to_grid_lean_fx(StepParams P, VecSet y,
                                                                         double2* __restrict__ G1,
                                                                         double2* __restrict__ W) {
    chain_wait();
    __shared__ FxScale sc;
    __shared__ DctHalf dh;
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, N = P.n_r, nc = P.nc, M = P.M;
    fxc* X = fx_shared;
    fxc* Y = X + K;
    double2* C = reinterpret_cast<double2*>(Y + K);  // plain coefficients of Psi and then of its derivatives (u_bar)
    const int tid = threadIdx.x, nth = blockDim.x;
    const double Cw = P.cnorm, Cw0 = 0.5 * P.cnorm, dm = (double)m;
    const double* ps = reinterpret_cast<const double*>(y.psi + (size_t)m * nc);
    const double* th = reinterpret_cast<const double*>(y.th + (size_t)m * nc);
    double* PF = P.pump ? reinterpret_cast<double*>(P.pump_F + (size_t)m * N) : nullptr;
    double* wu = reinterpret_cast<double*>(W + (size_t)m * 2 * N);  // partial sums of u_phi
    double* wo = wu + 2 * N;                                         // and of omega
    fx_scale_clear(sc);
    __syncthreads();
    for (int b = 0; b < 2; ++b) {
        unsigned ex = 0u;
        for (int t = tid; t < 2 * nc; t += nth) {
            const double w = (t < 2) ? Cw0 : Cw;
            double x;
            if (b) {
                x = th[t] * w;
            } else {
                x = (m > 0) ? ps[t] * w : (t & 1) ? 0.0 : y.u[t >> 1] * w;
                reinterpret_cast<double*>(C)[t] = x;
            }
            const unsigned e = fx_exponent(x);
            ex = max(ex, (t < 2 && e) ? min(e + 1u, 0x7ffu) : e);
        }
        fx_scale_max(sc, b ? 3 : 0, tid & 1, ex);
    }
    __syncthreads();
    // vectors 0 Psi, 1 Psi', 2 Psi'' (u_bar, u_bar' for m = 0), 3 theta
    for (int v = 0; v < 4; ++v) {
        if (m == 0 && v == 2) continue;
        double2* D = C;
        if (v == 1 || v == 2) {
            D = reinterpret_cast<double2*>(Y);
            cheb_derivative_cta(C, D, nc, nc, P.inv_a, dh, sc, v);
            for (int t = tid; t < 2 * nc; t += nth) reinterpret_cast<double*>(C)[t] = reinterpret_cast<double*>(D)[t];
        }
        fxc *F, *O;
        if (v == 3)
            dct1_half_fx(P, sc, dh, v, nc, true, X, Y, F, O, [&](int t) { return th[t] * ((t < 2) ? Cw0 : Cw); });
        else
            dct1_half_fx(P, sc, dh, v, nc, true, X, Y, F, O, [&](int t) { return reinterpret_cast<const double*>(D)[t]; });
        for (int t = tid; t < 2 * N; t += nth) {
            const int k = t >> 1, part = t & 1;
            const double g = half_part(sc, v, F, O, K, k, part, -1);  // value of the series at x_k
            double* out = reinterpret_cast<double*>(G1 + g_index(k, 0, m, M));  // fields 2M doubles apart
            if (v == 3) {
                out[6 * M + part] = g;
                continue;
            }
            const double s = P.s[k], h2 = P.h2[k], is = P.inv_s[k];
            if (m == 0) {
                if (v == 0) {
                    out[part] = 0.0;
                    out[2 * M + part] = g;
                    wu[t] = g;
                    wo[t] = g * is;
                } else {
                    const double om = wo[t] + g;
                    out[4 * M + part] = om;
                    if (PF) PF[t] = part ? 0.0 : P.pump_ups[k] * wu[t] * (1.0 + (0.5 * P.E) * om);
                }
            } else if (v == 0) {
                out[part ^ 1] = part ? -dm * g : dm * g;
                wu[t] = (3.0 * s) * g;
                wo[t] = fma(dm * dm * h2, is * is, 6.0) * g;
                if (PF) {
                    const double go = half_part(sc, v, F, O, K, k, part ^ 1, -1), U = P.pump_ups[k];
                    const double ci = U * dm * P.pump_ci[k];
                    PF[t] = fma(part ? -ci : ci, go, -U * fma(dm, dm, P.pump_cr[k]) * g);
                }
            } else if (v == 1) {
                out[2 * M + part] = fma(-h2, g, wu[t]);
                wo[t] = fma(-fma(-5.0, s, h2 * is), g, wo[t]);
                if (PF) PF[t] = fma(P.pump_ups[k] * (0.5 * s), g, PF[t]);
            } else {
                const double om = fma(-h2, g, wo[t]);
                out[4 * M + part] = om;
                if (PF) PF[t] = fma(-P.pump_ups[k], om, PF[t]);
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(NTHREADS_LX, 2) k_grid_to_spec_lean_fx(StepParams P, const double2* G2,
                                                                         VecSet y, VecSet e) {
    chain_wait();
    __shared__ FxScale sc;
    __shared__ DctHalf dh;
    const int m = P.m_lo + blockIdx.x;
    const int K = P.K, N = P.n_r, nc = P.nc, M = P.M;
    fxc* X = fx_shared;
    fxc* Y = X + K;
    double* C = reinterpret_cast<double*>(Y + K);  // n_r complex values
    double* D = reinterpret_cast<double*>(Y);      // derivative coefficients 0 .. K-1 (the last one is zero)
    const int tid = threadIdx.x, nth = blockDim.x;
    const double dm = (double)m, hc = 0.5 * P.cnorm;
    const int lgK = 31 - __clz(K);
    const double* PF = P.pump ? reinterpret_cast<const double*>(P.pump_F + (size_t)m * N) : nullptr;
    const double bfac = P.Ra / P.Pr * dm / P.s_o;
    const double* g2 = reinterpret_cast<const double*>(G2);
    const double* th = reinterpret_cast<const double*>(y.th + (size_t)m * nc);
    const double* ps = reinterpret_cast<const double*>(y.psi + (size_t)m * nc);
    double* eps = reinterpret_cast<double*>(e.psi + (size_t)m * nc);
    double* eth = reinterpret_cast<double*>(e.th + (size_t)m * nc);
    fx_scale_clear(sc);
    __syncthreads();
    fxc *F, *O;
    auto coef = [&](int t) { return C[t]; };
    // field 0: N_omega (m >= 1) or N_u (m = 0); field 1: N_theta; vectors 3 fld ..: the flux, its
    // derivative, N
    for (int fld = 0; fld < 2; ++fld) {
        const int v = 3 * fld;
        unsigned ex = 0u;
        if (fld == 1 || m > 0) {
            for (int t = tid; t < 2 * N; t += nth) {
                const double x = g2[2 * (size_t)g_index(t >> 1, 2 * fld, m, M) + (t & 1)] * P.h2[t >> 1];
                C[t] = x;
                ex = max(ex, fx_exponent(x));
            }
            fx_scale_max(sc, v, tid & 1, ex);
            __syncthreads();
            dct1_half_fx(P, sc, dh, v, N, false, X, Y, F, O, coef);
            for (int t = tid; t < 2 * N; t += nth) {
                const int n = t >> 1;
                C[t] = half_part(sc, v, F, O, K, n, t & 1, (n == 0 || n == K) ? -lgK - 1 : -lgK);
            }
            __syncthreads();
            cheb_derivative_cta(reinterpret_cast<double2*>(C), reinterpret_cast<double2*>(D), N, K, P.inv_a, dh, sc, v + 1);
            dct1_half_fx(P, sc, dh, v + 1, K, true, X, Y, F, O, [&](int t) { return D[t]; });
        }
        ex = 0u;
        for (int t = tid; t < 2 * N; t += nth) {
            const int k = t >> 1, part = t & 1;
            const double is = P.inv_s[k];
            const double* g = g2 + 2 * (size_t)g_index(k, 0, m, M);  // fields 2M doubles apart
            double val;
            if (fld == 0 && m == 0) {
                val = g[part] * (P.h2[k] * is);
                if (PF) val += PF[t];
            } else {
                const double dF = half_part(sc, v + 1, F, O, K, k, part, -1);
                const double w = fma(part ? dm : -dm, g[(fld ? 6 : 2) * M + (part ^ 1)], dF);
                if (fld == 0) {
                    val = w * is;
                    if (PF) val -= PF[t];
                } else {
                    val = fma(w, is, -g[4 * M + part]);
                }
            }
            C[t] = val;
            ex = max(ex, fx_exponent(val));
        }
        fx_scale_max(sc, v + 2, tid & 1, ex);
        __syncthreads();
        // Eq. icheb of the grid values, truncated to n < nc, N_omega_hat with the buoyancy
        dct1_half_fx(P, sc, dh, v + 2, N, false, X, Y, F, O, coef);
        const bool buoy = (fld == 0 && m > 0 && !P.buoy_imp);
        for (int t = tid; t < 2 * nc; t += nth) {
            const int part = t & 1;
            double x = half_part(sc, v + 2, F, O, K, t >> 1, part, 0) * hc;
            if (buoy) x = fma(part ? bfac : -bfac, th[t ^ 1], x);
            C[t] = x;
        }
        __syncthreads();
        for (int t = tid; t < 2 * nc; t += nth) {
            const int k = t >> 1, part = t & 1;
            double x = 0.0;
            if (fld == 0) {
                if (m > 0) {
                    if (k >= 4) x = band_part<8>(P.ops.band[OP_C], C + part, k, nc);
                } else if (part == 0) {
                    e.u[k] = (k >= 2) ? -band_part<4>(P.ops.band[OP_D], C, k, nc) : 0.0;
                }
                eps[t] = x;
            } else {
                if (k >= 2) {
                    x = -band_part<4>(P.ops.band[OP_D], C + part, k, nc);
                    if (m > 0) {
                        const double gp = band_part<4>(P.ops.band[OP_G], ps + (part ^ 1), k, nc);
                        x = fma(part ? -P.tc * dm : P.tc * dm, gp, x);
                    }
                }
                eth[t] = x;
            }
        }
        __syncthreads();
    }
}

size_t smem_radial_lean(const StepParams& P) { return sizeof(double2) * 3 * (size_t)P.n_r; }
// the FP32 lean kernels: three float2 arrays; a3 also the FP64 coefficients
static size_t smem_radial_lean32(const StepParams& P, bool analysis) {
    return analysis ? lean_cd_offset<float2>(P.n_r) + sizeof(double2) * (size_t)P.nc : sizeof(float2) * 3 * (size_t)P.n_r;
}

template <class T>
static cudaError_t spec_to_grid_t(const StepParams& P, VecSet y, void* G1, void* W, cudaStream_t st) {
    const size_t sm = smem_spec_to_grid(P);
    cudaError_t err = cudaFuncSetAttribute(k_spec_to_grid<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(k_spec_to_grid<T>, slab_modes(P), NTHREADS_R, sm, st, P, y, static_cast<T*>(G1),
                          static_cast<T*>(W));
}

// 1 when the azimuthal kernels can hold both packed pairs at once (twice
// smem_phi_products: n_phi <= 3072 in FP64), else 0
static int phi_pair(const StepParams& P, cudaError_t& err) {
    int dev = 0, smax = 0;
    err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return (err == cudaSuccess && 2 * smem_phi_products(P) <= (size_t)smax) ? 1 : 0;
}

template <class T>
static cudaError_t phi_products_t(const StepParams& P, const void* G1, void* G2, cudaStream_t st) {
    const int nth = phi_threads(P);
    if (P.n_phi > nth * MAXPER || nth > 512) return cudaErrorInvalidValue;
    cudaError_t err;
    const int pair = phi_pair(P, err);
    if (err != cudaSuccess) return err;
    const size_t sm = (pair ? 2 : 1) * smem_phi_products(P);
    err = cudaFuncSetAttribute(k_phi_products<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(k_phi_products<T>, slab_radii(P), nth, sm, st, P, static_cast<const T*>(G1),
                          static_cast<T*>(G2), pair);
}

template <class T>
static cudaError_t grid_to_spec_t(const StepParams& P, const void* G2, VecSet y, VecSet e, cudaStream_t st) {
    const size_t sm = smem_spec_to_grid(P);  // (its buffers are those of the synthesis)
    cudaError_t err = cudaFuncSetAttribute(k_grid_to_spec<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(k_grid_to_spec<T>, slab_modes(P), NTHREADS_R, sm, st, P, static_cast<const T*>(G2), y, e);
}

cudaError_t launch_spec_to_grid(const StepParams& P, VecSet y, double2* G1, double2* W, cudaStream_t st) {
    if (lean_radial(P) && P.fp32) {
        const size_t sm = smem_radial_lean32(P, false);
        cudaError_t err =
            cudaFuncSetAttribute(k_spec_to_grid_lean<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (err != cudaSuccess) return err;
        return launch_chained(k_spec_to_grid_lean<float2>, slab_modes(P), NTHREADS_R, sm, st, P, y,
                              reinterpret_cast<float2*>(G1));
    }
    if (lean_radial(P)) {
        const size_t sm = smem_radial_lean(P);
        const bool fx = radial_fx(P);
        cudaError_t err = fx ? cudaFuncSetAttribute(k_spec_to_grid_lean_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)
                             : cudaFuncSetAttribute(k_spec_to_grid_lean<double2>,
                                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (err != cudaSuccess) return err;
        if (fx) return launch_chained(k_spec_to_grid_lean_fx, slab_modes(P), NTHREADS_LX, sm, st, P, y, G1, W);
        return launch_chained(k_spec_to_grid_lean<double2>, slab_modes(P), NTHREADS_R, sm, st, P, y, G1);
    }
    if (P.fp32) return spec_to_grid_t<float2>(P, y, G1, W, st);
    if (!radial_fx(P)) return spec_to_grid_t<double2>(P, y, G1, W, st);
    const size_t sm = smem_spec_to_grid(P);
    cudaError_t err = cudaFuncSetAttribute(k_spec_to_grid_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(k_spec_to_grid_fx, slab_modes(P), fx_threads(P), sm, st, P, y, G1, W);
}

cudaError_t launch_phi_products(const StepParams& P, const double2* G1, double2* G2, cudaStream_t st) {
    if (P.fp32) return phi_products_t<float2>(P, G1, G2, st);
    if (P.phi_dd && P.fx_p) {
        const int nth = phi_threads_fx(P);
        if (P.n_phi > nth * MAXPER || nth > 512) return cudaErrorInvalidValue;
        // the batched pair of transforms needs twice the buffers (n_phi <= 3072)
        cudaError_t err;
        const int pair = phi_pair(P, err);
        if (err != cudaSuccess) return err;
        const size_t sm = (pair ? 2 : 1) * smem_phi_products(P);
        auto kern = !pair ? k_phi_products_fx<false, true>
                    : P.n_m < 768 ? k_phi_products_fx<true, false> : k_phi_products_fx<true, true>;
        err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (err != cudaSuccess) return err;
        return launch_chained(kern, slab_radii(P), nth, sm, st, P, G1, G2);
    }
    return phi_products_t<double2>(P, G1, G2, st);
}

cudaError_t launch_grid_to_spec(const StepParams& P, const double2* G2, VecSet y, VecSet e, cudaStream_t st) {
    if (lean_radial(P) && P.fp32) {
        const size_t sm = smem_radial_lean32(P, true);
        cudaError_t err =
            cudaFuncSetAttribute(k_grid_to_spec_lean<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (err != cudaSuccess) return err;
        return launch_chained(k_grid_to_spec_lean<float2>, slab_modes(P), NTHREADS_R, sm, st, P,
                              reinterpret_cast<const float2*>(G2), y, e);
    }
    if (lean_radial(P)) {
        const size_t sm = smem_radial_lean(P);
        const bool fx = radial_fx(P);
        auto kern = fx ? k_grid_to_spec_lean_fx : k_grid_to_spec_lean<double2>;
        cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (err != cudaSuccess) return err;
        return launch_chained(kern, slab_modes(P), fx ? NTHREADS_LX : NTHREADS_R, sm, st, P, G2, y, e);
    }
    if (P.fp32) return grid_to_spec_t<float2>(P, G2, y, e, st);
    if (!radial_fx(P)) return grid_to_spec_t<double2>(P, G2, y, e, st);
    const size_t sm = smem_grid_to_spec(P);
    cudaError_t err = cudaFuncSetAttribute(k_grid_to_spec_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(k_grid_to_spec_fx, slab_modes(P), fx_threads(P), sm, st, P, G2, y, e);
}

}  // namespace pz
