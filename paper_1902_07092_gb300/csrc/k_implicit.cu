// Implicit stage of one IMEX step: right-hand-side assembly (Eqs. multistep1
// and dirks of Section 4) and the bordered banded solve of Appendix A of
// Gastine, pizza, GJI 2019.
//
// For each mode the tau system  [tau rows; Mass - gamma dt Lin] y = [0; r]  is
//   (A B; C D)(y1; y2) = (g; h),   D banded (half width 8 for Psi, 4 for theta
//   and u_bar), factored at set-up without pivoting,
//   x = D^{-1} h,  y1 = S^{-1}(g - B x) with S = A - B D^{-1} C,  y2 = x - Y y1,
//   Y = D^{-1} C precomputed.
// The unpivoted factorisation of the streamfunction block loses digits as n_r
// grows, so its solution is refined once: the residual of the assembled system
// is formed in FP64 and solved again with the same factors.
//
// The banded block is solved through its two-sided block-tridiagonal
// factorisation (blocks of 8 rows; the temperature and zonal-flow bands, half
// width 4, are padded to that: twice the block size halves their chains and keeps
// all 32 lanes busy; host_ops.h, block_lu_twisted): a pair of warps walks the top and
// the bottom half towards the middle block and back.  On GB300 an FP64 instruction
// of a warp holds its sub-partition ~64 cycles, dependent or not, so a phase costs
// the FP64 instructions of its longest warp: the chains have as few of them as the
// lanes allow, and everything else (right-hand side, Schur sums and updates,
// residual, the banded mass applies for later stages) is cut into tasks of one
// component of one row over the whole CTA.
#include "device_common.cuh"

namespace pz {

namespace {

constexpr int NTHREADS_S = 256;

template <class T>
__device__ __forceinline__ T zero();
template <>
__device__ __forceinline__ double2 zero<double2>() { return make_double2(0.0, 0.0); }
template <>
__device__ __forceinline__ double zero<double>() { return 0.0; }

// x - a*z in fused form
__device__ __forceinline__ double2 fms(double2 x, double a, double2 z) {
    return make_double2(fma(-a, z.x, x.x), fma(-a, z.y, x.y));
}
__device__ __forceinline__ double2 mul(double2 a, double2 b) { return cmul(a, b); }
__device__ __forceinline__ double2 mul(double a, double2 b) { return cscale(b, a); }

template <class TX>
__device__ __forceinline__ TX shfl_idx(TX v, int src);
template <>
__device__ __forceinline__ double shfl_idx<double>(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
template <>
__device__ __forceinline__ double2 shfl_idx<double2>(double2 v, int src) {
    return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 fms_x(double2 a, double2 b, double2 acc) {
    return make_double2(fma(-a.x, b.x, fma(a.y, b.y, acc.x)), fma(-a.x, b.y, fma(-a.y, b.x, acc.y)));
}
__device__ __forceinline__ double2 fms_x(double a, double2 b, double2 acc) {
    return make_double2(fma(-a, b.x, acc.x), fma(-a, b.y, acc.y));
}
__device__ __forceinline__ double fms_x(double a, double b, double acc) { return fma(-a, b, acc); }

// FP32 counterparts for the refined FP32 temperature solves
template <>
__device__ __forceinline__ float2 zero<float2>() { return make_float2(0.f, 0.f); }
template <>
__device__ __forceinline__ float2 shfl_idx<float2>(float2 v, int src) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
// conversions between the FP32 chains and FP64 on the integer and FP32 pipes
// (GB300 issues float <-> double conversions on its FP64 unit)
__device__ __forceinline__ float2 to_f2(double2 v) { return make_float2(f32_from_bits(v.x), f32_from_bits(v.y)); }
__device__ __forceinline__ double2 to_d2_bits(float2 v) { return make_double2(f2d_bits(v.x), f2d_bits(v.y)); }

// Double-float chains of the streamfunction solve.  The block chains of the
// Appendix A solve need about 44 significant bits: with the Schur step, the
// residual and the refinement in FP64, chains in 44- to 48-bit arithmetic leave
// the refined solution as close to the oracle's as FP64 chains do (measured on the
// tau systems at n_r = 257, 1025 and 2049), while FP32 chains need two and more
// corrections at n_r = 1025 and do not converge at 2049.  A double-float value
// (ddfloat.cuh) carries 48 bits on the FP32 pipe, which issues 64 times the FP64
// rate on GB300.
//
// Factors and chain values are complex double-floats (ddc, 16 bytes like a
// double2).  A row sum runs in leading sums s and trailing sums e: every product a b of double-floats adds its leading part
// p = a.hi b.hi to s by a two-sum and its trailing parts (the two-product error
// fma(a.hi, b.hi, -p), a.hi b.lo + a.lo b.hi, and the two-sum's error) to e; the
// value is s + e, renormalised once at the end of the row (Ogita, Rump and
// Oishi's compensated dot product, applied to double-float inputs).
// s + p = s' + t exactly (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float s, float p, float& t) {
    const float r = __fadd_rn(s, p);
    const float bb = __fsub_rn(r, s);
    t = __fadd_rn(__fsub_rn(s, __fsub_rn(r, bb)), __fsub_rn(p, bb));
    return r;
}
// (s, e) += (ah + al)(bh + bl)
__device__ __forceinline__ void dd_acc(float& s, float& e, float ah, float al, float bh, float bl) {
    const float p = __fmul_rn(ah, bh);
    const float pe = __fmaf_rn(ah, bh, -p);
    const float cr = __fmaf_rn(ah, bl, __fmul_rn(al, bh));
    float t;
    s = two_sum(s, p, t);
    e = __fadd_rn(e, __fadd_rn(t, __fadd_rn(pe, cr)));
}
// sum over a pair of lanes; the two-sum's result and error do not depend
// on the order of its operands, so every lane gets the same bits
__device__ __forceinline__ void dd_pair_sum(float& s, float& e, int o) {
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o), e2 = __shfl_xor_sync(0xffffffffu, e, o);
    float t;
    s = two_sum(s, s2, t);
    e = __fadd_rn(__fadd_rn(e, e2), t);
}
// (s + e) as a normalised double-float: two-sum, since e may exceed a cancelled s
__device__ __forceinline__ ddf dd_norm(float s, float e) {
    float t;
    const float h = two_sum(s, e, t);
    return ddf{h, t};
}
// Asynchronous 16-byte copies global -> shared (cp.async), committed in groups;
// cp_async_wait<N> returns when at most N of the calling thread's groups are
// still in flight.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_wait1() { cp_async_wait<1>(); }

// ---------------------------------------------------------------------------
// Block chains.  D x = b by the two-sided block factorisation (host_ops.h,
// block_lu_twisted) with blocks of 8 rows: a pair of warps walks the two halves,
//   forward   Z_k = b_k - [0]_k Z_prev            (half 0 down from the top, half 1 up from the bottom),
//   middle    x_c = [1]_c (b_c - [0]_c Z_{c-1} - [2]_c Z_{c+1})   (both warps),
//   diagonal  W_k = [1]_k Z_k for every other block (no chain depends on it: every warp of the CTA),
//   backward  x_k = W_k - [2]_k x_prev,
// with a barrier of the CTA between the phases.  Everything may run in place (Z, W
// and x over b): a block's row is read before it is written, the middle block's
// rows after the barrier that ends the middle phase.
//
// Lane (r, part, g) owns row r = lane/4 of a block, one component (part) of its
// value and columns 4 g .. 4 g + 3: a step is four multiply-adds a lane (eight with
// complex coefficients) and one exchange, the right-hand side being the sum's start.
// With a lane per (row, two columns) and both components a step took 10 and 18 FP64
// instructions of 64 cycles where it now takes 5 and 9.  The previous block's values
// come by shuffles (real coefficients) or through shared memory (complex ones, whose
// lanes need both components of four rows).
//
// The matrices of a walk stream through a ring of slots in shared memory, filled by
// asynchronous copies one slot short of its length ahead and kept filled across the phases' barriers:
// forward, the middle block's three, backward.  (Six slots measured the same as four.)
// ---------------------------------------------------------------------------
// Component, accumulator and arithmetic of a chain by its coefficient type: double2
// (complex, FP64), ddc (complex double-float), double and float (real coefficients).
// An accumulator starts from the value the products are taken from, in one of the two
// lanes that share a row's component: no subtraction afterwards.  The double-float
// one keeps the products of the coefficients' real and imaginary parts apart: two
// shorter strings of dependent sums, and one sign for the second.
struct ddacc {
    float s, e, t, f;
};
template <class C>
struct Chain;
template <>
struct Chain<double2> {
    using V = double;
    using A = double;
    static constexpr bool cplx = true;
};
template <>
struct Chain<double> {
    using V = double;
    using A = double;
    static constexpr bool cplx = false;
};
template <>
struct Chain<float> {
    using V = float;
    using A = float;
    static constexpr bool cplx = false;
};
template <>
struct Chain<ddc> {
    using V = ddf;
    using A = ddacc;
    static constexpr bool cplx = true;
};
__device__ __forceinline__ void ch_zero(double& a) { a = 0.0; }
__device__ __forceinline__ void ch_zero(float& a) { a = 0.f; }
__device__ __forceinline__ void ch_zero(ddf& a) { a = ddf{0.f, 0.f}; }
__device__ __forceinline__ void ch_start(double& a, double b) { a = b; }
__device__ __forceinline__ void ch_start(float& a, float b) { a = b; }
__device__ __forceinline__ void ch_start(ddacc& a, ddf b) { a = ddacc{b.hi, b.lo, 0.f, 0.f}; }
// acc -= (SUB) or += component part of a (x + i y); p, q: that component and the other
template <bool SUB>
__device__ __forceinline__ void ch_mac(double& acc, double2 a, double p, double q, int part) {
    q = (part != 0) == SUB ? -q : q;  // operands chosen, not instructions: one path for all lanes
    acc = fma(SUB ? -a.x : a.x, p, fma(a.y, q, acc));
}
template <bool SUB>
__device__ __forceinline__ void ch_mac(ddacc& acc, ddc a, ddf p, ddf q, int) {
    dd_acc(acc.s, acc.e, SUB ? -a.x.hi : a.x.hi, SUB ? -a.x.lo : a.x.lo, p.hi, p.lo);
    dd_acc(acc.t, acc.f, a.y.hi, a.y.lo, q.hi, q.lo);
}
// acc -= or += a x
template <bool SUB>
__device__ __forceinline__ void ch_mac(double& acc, double a, double x) { acc = fma(SUB ? -a : a, x, acc); }
template <bool SUB>
__device__ __forceinline__ void ch_mac(float& acc, float a, float x) { acc = fmaf(SUB ? -a : a, x, acc); }
// the value: both lanes' sums (g = 0, 1) of a row's component
template <bool SUB>
__device__ __forceinline__ double ch_value(double a, int) { return a + __shfl_xor_sync(0xffffffffu, a, 1); }
template <bool SUB>
__device__ __forceinline__ float ch_value(float a, int) { return a + __shfl_xor_sync(0xffffffffu, a, 1); }
template <bool SUB>
__device__ __forceinline__ ddf ch_value(ddacc a, int part) {
    const float sg = (part != 0) == SUB ? -1.f : 1.f;
    float u, s = two_sum(a.s, sg * a.t, u), e = __fadd_rn(__fadd_rn(a.e, sg * a.f), u);
    dd_pair_sum(s, e, 1);
    return dd_norm(s, e);
}
// the sum over 4 columns: coefficients a[4], this lane's component p[4] of the values
// and (complex coefficients) the other q[4]
template <bool SUB, class C>
__device__ __forceinline__ void ch_row(typename Chain<C>::A& acc, const C (&a)[4], const typename Chain<C>::V (&p)[4],
                                       const typename Chain<C>::V (&q)[4], int part) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if constexpr (Chain<C>::cplx)
            ch_mac<SUB>(acc, a[j], p[j], q[j], part);
        else
            ch_mac<SUB>(acc, a[j], p[j]);
    }
}
// its values from a vector with NP components a row
template <class C, int NP>
__device__ __forceinline__ void ch_values(const typename Chain<C>::V* v, int c0, int part, typename Chain<C>::V (&p)[4],
                                          typename Chain<C>::V (&q)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        p[j] = v[NP * (c0 + j) + (NP == 2 ? part : 0)];
        if constexpr (Chain<C>::cplx) q[j] = v[2 * (c0 + j) + 1 - part];
    }
}
// or from a walk's previous block, stored component by component (8 rows each):
// 16-byte reads
template <class V>
__device__ __forceinline__ void ch_four(const V* v, V (&p)[4]) {
    struct __align__(16) Q {
        V x[16 / sizeof(V)];
    };
    constexpr int K = 16 / (int)sizeof(V);
#pragma unroll
    for (int i = 0; i < 4 / K; ++i) {
        const Q w = reinterpret_cast<const Q*>(v)[i];
#pragma unroll
        for (int j = 0; j < K; ++j) p[i * K + j] = w.x[j];
    }
}
template <class C, int NP>
__device__ __forceinline__ void ch_prev(const typename Chain<C>::V* v, int c0, int part, typename Chain<C>::V (&p)[4],
                                        typename Chain<C>::V (&q)[4]) {
    ch_four(v + (NP == 2 ? 8 * part : 0) + c0, p);
    if constexpr (Chain<C>::cplx) ch_four(v + 8 * (1 - part) + c0, q);
}

// slots of a walk's ring (a power of two): 4 KB of complex or double-float matrices,
// 2 KB of real FP64, 1 KB of FP32 ones (eight of these measured the same)
constexpr int RING = 4;
template <class C>
__host__ __device__ constexpr int ring_bytes() { return RING * 64 * (int)sizeof(C); }

struct ChainGeom {
    int nb, cm, len, k_fw, k_bw, dir;  // blocks, middle block, blocks of this half, its first blocks, forward direction
    __device__ __forceinline__ ChainGeom(int n, int half) {
        nb = (n + 7) / 8;
        cm = nb / 2;
        dir = half ? -1 : 1;
        len = half ? (nb - 1 - cm) : cm;
        k_fw = half ? nb - 1 : 0;
        k_bw = half ? cm + 1 : cm - 1;
    }
};

// One warp's walk (one set of registers whatever its system) and its stream of matrices
// through a ring: entry e (issued in order) to slot e % RING.  A walking warp is mostly alone
// on its sub-partition and pays for every instruction of a step, so its arrays are
// offsets into shared memory (read and written as such, 32-bit arithmetic), and the
// loops run on a pointer that moves by a constant for as long as the entries stay in
// one direction (far), instead of 64-bit pointers of unknown space and a choice of the
// source in every step.  Solve, us: 257 x 768 67.7 -> 63.1, 513 x 1536 254 -> 233,
// 1025 x 3072 770 -> 688, 2049 x 6144 2834 -> 2505; implicit buoyancy, whose temperature
// and streamfunction chains follow one another, 1025 x 384 305 -> 268 (277 with the
// real coefficients' previous block through shared memory too).  Real matrices straight
// to registers, 8 ahead, with unrolled steps: 343 (the code no longer fits the
// instruction cache next to a lone warp).
extern __shared__ __align__(16) char walk_shared[];
template <class V>
__device__ __forceinline__ V* walk_at(int off) {
    return reinterpret_cast<V*>(walk_shared + off);
}
__device__ __forceinline__ int walk_off(const void* p) { return (int)(reinterpret_cast<const char*>(p) - walk_shared); }
struct Walk {
    int b, Z, x, ring;  // offsets
    const char* blk;
    int n, half, e;
    ChainGeom g;
    template <class C>
    __device__ __forceinline__ void copy(const char* src) {
        constexpr int MAT = 64 * (int)sizeof(C);
        const int lane = threadIdx.x & 31;
        char* dst = walk_at<char>(ring + (e & (RING - 1)) * MAT + 16 * lane);
#pragma unroll
        for (int j = 0; j < MAT; j += 512)
            if (j + 512 <= MAT || lane < 16) cp_async16(dst + j, src + j + 16 * lane);
        cp_async_commit();
        ++e;
    }
    // entry i: the blocks forward, the middle one's three matrices, the blocks backward
    template <class C>
    __device__ __forceinline__ const char* entry(int i) const {
        const int j = i - g.len;
        const int mat = j < 0    ? (g.k_fw + g.dir * i) * 3
                        : j < 3  ? g.cm * 3 + (j == 0 ? 0 : j == 1 ? 2 : 1)
                                 : (g.k_bw - g.dir * (j - 3)) * 3 + 2;
        return blk + (ptrdiff_t)mat * (64 * (int)sizeof(C));
    }
    template <class C>
    __device__ __forceinline__ void issue() {
        if (e < 2 * g.len + 3) {
            copy<C>(entry<C>(e));
        } else {
            cp_async_commit();
            ++e;
        }
    }
    // the four coefficients of this lane of entry e - RING + 1, the oldest in flight
    template <class C>
    __device__ __forceinline__ void take(C (&a)[4]) {
        const int lane = threadIdx.x & 31;
        cp_async_wait<RING - 2>();
        __syncwarp();  // also: every lane has read the slot before, which issue refills
        ch_four(walk_at<C>(ring + ((e + 1) & (RING - 1)) * 64 * (int)sizeof(C)) + (lane >> 2) * 8 + (lane & 1) * 4, a);
    }
};
// A walk over the blocks of one direction: step(i, next) for i < len, next() asking for
// the matrix that takes the slot of the one just read
template <class C, class Step>
__device__ __forceinline__ void walk_blocks(Walk& w, int stride, Step step) {
    const int len = w.g.len, far = len - (RING - 1);
    int i = 0;
    if (far > 0) {
        const char* src = w.entry<C>(w.e);
        for (; i < far; ++i)
            step(i, [&]() {
                w.copy<C>(src);
                src += stride;
            });
    }
    for (; i < len; ++i) step(i, [&]() { w.issue<C>(); });
}

// Forward walk of one warp.  b: n rows (NP components each), Z: 8 nb rows.  prev:
// this warp's 2 x 16 components in shared memory.
template <class C, int NP>
__device__ __forceinline__ void chain_forward(Walk& w, typename Chain<C>::V* prev) {
    using V = typename Chain<C>::V;
    const ChainGeom& g = w.g;
    const int n = w.n;
    const int lane = threadIdx.x & 31, r = lane >> 2, part = (lane >> 1) & 1, gcol = lane & 1;
    const bool own = gcol == 0 && part < NP;
#pragma unroll 1
    for (int e = 0; e < RING - 1; ++e) w.issue<C>();
    if (lane < 16) ch_zero(prev[lane]);
    V pv;
    ch_zero(pv);
    int row = g.k_fw * 8 + r;
    const V* b = walk_at<const V>(w.b) + row * NP + part;
    V* Z = walk_at<V>(w.Z) + row * NP + part;
    walk_blocks<C>(w, g.dir * 3 * 64 * (int)sizeof(C), [&](int i, auto next) {
        V bv, p[4], q[4];
        C a[4];
        w.take<C>(a);
        if constexpr (Chain<C>::cplx) ch_prev<C, NP>(prev + (i & 1) * 16, 4 * gcol, part, p, q);
        else {
#pragma unroll
            for (int j = 0; j < 4; ++j) p[j] = __shfl_sync(0xffffffffu, pv, (4 * gcol + j) * 4 + 2 * part);
        }
        ch_zero(bv);
        if (row < n && own) bv = *b;
        next();
        typename Chain<C>::A acc;
        ch_start(acc, bv);
        ch_row<true>(acc, a, p, q, part);
        const V z = ch_value<true>(acc, part);
        if constexpr (!Chain<C>::cplx) pv = z;
        if (own) {
            if constexpr (Chain<C>::cplx) prev[((i + 1) & 1) * 16 + 8 * part + r] = z;
            *Z = z;
        }
        row += 8 * g.dir;
        b += 8 * NP * g.dir;
        Z += 8 * NP * g.dir;
    });
}
// middle block by both warps of the pair; returns the lane's component of it, also
// left in prev[0 .. 16) for the backward walk.  The caller stores it after a barrier.
template <class C, int NP>
__device__ __forceinline__ typename Chain<C>::V chain_middle(Walk& w, typename Chain<C>::V* prev) {
    using V = typename Chain<C>::V;
    const V *b = walk_at<const V>(w.b), *Z = walk_at<const V>(w.Z);
    const ChainGeom& g = w.g;
    const int n = w.n;
    const int lane = threadIdx.x & 31, r = lane >> 2, part = (lane >> 1) & 1, gcol = lane & 1;
    const bool own = gcol == 0 && part < NP;
    const int row = g.cm * 8 + r;
    V bv;
    ch_zero(bv);
    if (row < n && own) bv = b[row * NP + part];
    typename Chain<C>::A acc;
    ch_start(acc, bv);
    C a[4];
    V p[4], q[4];
    w.take<C>(a);
    w.issue<C>();
    if (g.cm > 0) {
        ch_values<C, NP>(Z + (g.cm - 1) * 8 * NP, 4 * gcol, part, p, q);
        ch_row<true>(acc, a, p, q, part);
    }
    w.take<C>(a);
    w.issue<C>();
    if (g.cm < g.nb - 1) {
        ch_values<C, NP>(Z + (g.cm + 1) * 8 * NP, 4 * gcol, part, p, q);
        ch_row<true>(acc, a, p, q, part);
    }
    const V y = ch_value<true>(acc, part);
    __syncwarp();  // the lanes' reads of the last block
    if (own) prev[16 + 8 * part + r] = y;
    w.take<C>(a);  // (synchronises the warp)
    w.issue<C>();
    ch_prev<C, NP>(prev + 16, 4 * gcol, part, p, q);
    ch_zero(bv);
    ch_start(acc, bv);
    ch_row<false>(acc, a, p, q, part);
    const V x = ch_value<false>(acc, part);
    if (own) prev[8 * part + r] = x;
    return x;
}
template <int NP, class V>
__device__ __forceinline__ void chain_middle_store(const Walk& w, V xv) {
    const int lane = threadIdx.x & 31, part = (lane >> 1) & 1;
    const int row = w.g.cm * 8 + (lane >> 2);
    if (w.half == 0 && (lane & 1) == 0 && part < NP && row < w.n) walk_at<V>(w.x)[row * NP + part] = xv;
}
// W_k = [1]_k Z_k in place for every block but the middle one, blocks w, w + nw, ...
// by warp w, DU of them in flight (their loads before any product)
template <class C, int NP, int DU>
__device__ __forceinline__ void chain_diag(typename Chain<C>::V* Z, int n, const C* __restrict__ blk, int w, int nw) {
    using V = typename Chain<C>::V;
    const int lane = threadIdx.x & 31, r = lane >> 2, part = (lane >> 1) & 1, gcol = lane & 1;
    const bool own = gcol == 0 && part < NP;
    const int nb = (n + 7) / 8, cm = nb / 2;
    for (int k0 = w; k0 < nb; k0 += nw * DU) {
        C a[DU][4];
#pragma unroll
        for (int u = 0; u < DU; ++u) {
            const int k = k0 + u * nw;
            if (k < nb) ch_four(blk + (k * 3 + 1) * 64 + r * 8 + 4 * gcol, a[u]);
        }
#pragma unroll
        for (int u = 0; u < DU; ++u) {
            const int k = k0 + u * nw;
            if (k >= nb || k == cm) continue;
            V v;
            ch_zero(v);
            typename Chain<C>::A acc;
            ch_start(acc, v);
            V p[4], q[4];
            ch_values<C, NP>(Z + k * 8 * NP, 4 * gcol, part, p, q);
            ch_row<false>(acc, a[u], p, q, part);
            v = ch_value<false>(acc, part);
            __syncwarp();
            if (own && k * 8 + r < n) Z[(k * 8 + r) * NP + part] = v;
        }
    }
}
// backward walk away from the middle block (prev[0 .. 16) holds it)
template <class C, int NP>
__device__ __forceinline__ void chain_backward(Walk& w, typename Chain<C>::V* prev, typename Chain<C>::V mid) {
    using V = typename Chain<C>::V;
    const ChainGeom& g = w.g;
    const int n = w.n;
    const int lane = threadIdx.x & 31, r = lane >> 2, part = (lane >> 1) & 1, gcol = lane & 1;
    const bool own = gcol == 0 && part < NP;
    int row = g.k_bw * 8 + r;
    V pv = mid;
    const V* W = walk_at<const V>(w.Z) + row * NP + part;
    V* x = walk_at<V>(w.x) + row * NP + part;
    walk_blocks<C>(w, -g.dir * 3 * 64 * (int)sizeof(C), [&](int i, auto next) {
        V wv, p[4], q[4];
        C a[4];
        w.take<C>(a);
        if constexpr (Chain<C>::cplx) ch_prev<C, NP>(prev + (i & 1) * 16, 4 * gcol, part, p, q);
        else {
#pragma unroll
            for (int j = 0; j < 4; ++j) p[j] = __shfl_sync(0xffffffffu, pv, (4 * gcol + j) * 4 + 2 * part);
        }
        ch_zero(wv);
        if (row < n && own) wv = *W;
        next();
        typename Chain<C>::A acc;
        ch_start(acc, wv);
        ch_row<true>(acc, a, p, q, part);
        const V xv = ch_value<true>(acc, part);
        if constexpr (!Chain<C>::cplx) pv = xv;
        if (own) {
            if constexpr (Chain<C>::cplx) prev[((i + 1) & 1) * 16 + 8 * part + r] = xv;
            if (row < n) *x = xv;
        }
        row -= 8 * g.dir;
        W -= 8 * NP * g.dir;
        x -= 8 * NP * g.dir;
    });
    cp_async_wait<0>();
    __syncwarp();
}

// One system's chain, for the phases below: b, Z and x as flattened components.
template <class C, int NP>
struct ChainJob {
    typename Chain<C>::V *b, *Z, *x;
    int n;  // 0: no such system
    const C* blk;
    int w;       // first warp of its pair
    char* ring;  // the pair's two rings
};
// Whole-CTA driver: ja, jb two halves of one system or one alone, jt and ju others, on
// disjoint warp pairs.  prevs: 16 doubles x 2 a warp in shared memory.  Z may be b
// and x where it has room for whole blocks; ends with a barrier that publishes x.
// With the walks, the diagonal products and the phases above: solve by mode at n_r x
// n_phi = 129 x 384, 257 x 768, 513 x 1536 46 -> 35, 71 -> 63, 270 -> 233 us; 513 x 384
// with implicit buoyancy 136 -> 123 us.
template <int DU, class CP, int NPP, class CT, int NPT, class CU, int NPU>
__device__ __forceinline__ void run_chains(const ChainJob<CP, NPP>& ja, const ChainJob<CP, NPP>& jb, const ChainJob<CT, NPT>& jt,
                                           const ChainJob<CU, NPU>& ju, double (*prevs)[32]) {
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Walk w{0, 0, 0, 0, nullptr, 0, warp & 1, 0, ChainGeom(0, 0)};
    auto pick = [&]<class C, int NP>(const ChainJob<C, NP>& j) {
        if (j.n == 0 || (warp & ~1) != j.w) return false;
        w.b = walk_off(j.b);
        w.Z = walk_off(j.Z);
        w.x = walk_off(j.x);
        w.ring = walk_off(j.ring) + (warp & 1) * ring_bytes<C>();
        w.blk = reinterpret_cast<const char*>(j.blk);
        w.n = j.n;
        w.g = ChainGeom(j.n, warp & 1);
        return true;
    };
    bool inp = pick(ja);
    if (pick(jb)) inp = true;
    const bool in_t = pick(jt), in_u = pick(ju);
    using VP = typename Chain<CP>::V;
    using VT = typename Chain<CT>::V;
    using VU = typename Chain<CU>::V;
    VP* pp = reinterpret_cast<VP*>(prevs[warp]);
    VT* pt = reinterpret_cast<VT*>(prevs[warp]);
    VU* pu = reinterpret_cast<VU*>(prevs[warp]);
    if (inp) chain_forward<CP, NPP>(w, pp);
    if (in_t) chain_forward<CT, NPT>(w, pt);
    if (in_u) chain_forward<CU, NPU>(w, pu);
    __syncthreads();
    VP xp;
    VT xt;
    VU xu;
    if (inp) xp = chain_middle<CP, NPP>(w, pp);
    if (in_t) xt = chain_middle<CT, NPT>(w, pt);
    if (in_u) xu = chain_middle<CU, NPU>(w, pu);
    __syncthreads();
    if (inp) chain_middle_store<NPP>(w, xp);
    if (in_t) chain_middle_store<NPT>(w, xt);
    if (in_u) chain_middle_store<NPU>(w, xu);
    for (int h = 0; h < 2; ++h) {
        const int n = h ? jb.n : ja.n;
        if (n > 0) chain_diag<CP, NPP, DU>(h ? jb.Z : ja.Z, n, h ? jb.blk : ja.blk, warp, nw);
    }
    if (jt.n > 0) chain_diag<CT, NPT, DU>(jt.Z, jt.n, jt.blk, nw - 1 - warp, nw);
    if (ju.n > 0) chain_diag<CU, NPU, DU>(ju.Z, ju.n, ju.blk, warp, nw);
    __syncthreads();
    if (inp) chain_backward<CP, NPP>(w, pp, xp);
    if (in_t) chain_backward<CT, NPT>(w, pt, xt);
    if (in_u) chain_backward<CU, NPU>(w, pu, xu);
    __syncthreads();
}
template <class C, int NP>
__device__ __forceinline__ ChainJob<C, NP> no_job() { return ChainJob<C, NP>{nullptr, nullptr, nullptr, 0, nullptr, 0, nullptr}; }

// acc - a z, component part
__device__ __forceinline__ double fms_part(double acc, double2 a, double2 z, int part) {
    const double p = part ? z.y : z.x, q = part ? -z.x : z.y;
    return fma(-a.x, p, fma(a.y, q, acc));
}
// Join of the streamfunction block solved in two halves (rows [0, nA) by warps
// 0-1, [nA, n) by warps 6-7; DevFactors psplit): x holds each half's own solution
// g.  The interface unknowns, A's last block and B's first, are
// [x_A,last; x_B,first] = Rj [g_A,last; g_B,first], Rj the inverse of
// [[I, V_last], [W_first, I]]; then x_A = g_A - V x_B,first and
// x_B = g_B - W x_A,last with the spikes V = D_A^{-1} E, W = D_B^{-1} F (spk rows
// < nA: V, the rest: W).  Whole CTA, after a __syncthreads that published x;
// ends with one.  act = false: no memory accesses.
__device__ void split_join(double2* x, int n, int nA, const double2* __restrict__ spk, const double2* __restrict__ rj,
                           bool act) {
    __shared__ double2 xi[16];
    const int tid = threadIdx.x;
    if (act && tid < 256) {  // (output, component, two columns)
        const int o = tid >> 4, part = (tid >> 3) & 1, c = 2 * (tid & 7);
        const double2* v = x + (c < 8 ? nA - 8 + c : nA + c - 8);
        double acc = fms_part(fms_part(0.0, __ldg(&rj[o * 16 + c]), v[0], part), __ldg(&rj[o * 16 + c + 1]), v[1], part);
#pragma unroll
        for (int h = 1; h < 8; h <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, h);
        if ((tid & 7) == 0) reinterpret_cast<double*>(xi)[tid >> 3] = -acc;
    }
    __syncthreads();
    if (act)
        for (int t = tid; t < 2 * n; t += blockDim.x) {
            const double2* row = spk + (size_t)(t >> 1) * 8;
            const double2* v = ((t >> 1) < nA) ? xi + 8 : xi;
            double* xt = reinterpret_cast<double*>(x) + t;
            double acc = *xt;
#pragma unroll
            for (int c = 0; c < 8; ++c) acc = fms_part(acc, __ldg(&row[c]), v[c], t & 1);
            *xt = acc;
        }
    __syncthreads();
}

// The same join in double-float arithmetic on the FP32 pipe (double-float
// chains): x, the spikes and the interface inverse as complex double-floats.  The
// 16 interface values are summed by 64 threads (four partial sums each, joined
// by shuffles).
__device__ void split_join_dd(ddc* x, int n, int nA, const ddc* __restrict__ spk, const ddc* __restrict__ rj,
                              bool act) {
    __shared__ __align__(16) ddf xi[2][16];  // by component
    const int tid = threadIdx.x;
    if (act && tid < 256) {  // (output, component, two columns)
        const int o = tid >> 4, part = (tid >> 3) & 1, c = 2 * (tid & 7);
        const ddf* v = reinterpret_cast<const ddf*>(x + (c < 8 ? nA - 8 + c : nA + c - 8));
        ddacc acc{0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 2; ++j) ch_mac<false>(acc, rj[o * 16 + c + j], v[2 * j + part], v[2 * j + 1 - part], part);
        float u, s = two_sum(acc.s, part ? acc.t : -acc.t, u), e = __fadd_rn(__fadd_rn(acc.e, part ? acc.f : -acc.f), u);
#pragma unroll
        for (int h = 1; h < 8; h <<= 1) dd_pair_sum(s, e, h);
        if ((tid & 7) == 0) xi[part][o] = dd_norm(s, e);
    }
    __syncthreads();
    if (act)
        for (int t = tid; t < 2 * n; t += blockDim.x) {
            const int part = t & 1, c0 = ((t >> 1) < nA) ? 8 : 0;
            ddc sp[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) sp[c] = spk[(size_t)(t >> 1) * 8 + c];
            ddf* xt = reinterpret_cast<ddf*>(x) + t;
            ddacc acc;
            ch_start(acc, *xt);
#pragma unroll
            for (int c = 0; c < 8; ++c) ch_mac<true>(acc, sp[c], xi[part][c0 + c], xi[1 - part][c0 + c], part);
            float u, s = two_sum(acc.s, part ? -acc.t : acc.t, u);
            *xt = dd_norm(s, __fadd_rn(__fadd_rn(acc.e, part ? -acc.f : acc.f), u));
        }
    __syncthreads();
}

// The same join for the FP32 temperature block split in halves (real spikes
// and interface inverse, complex FP32 values).
__device__ void split_join32(float2* x, int n, int nA, const float* __restrict__ spk, const float* __restrict__ rj) {
    __shared__ float2 xi[16];
    const int tid = threadIdx.x;
    if (tid < 16) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int c = 0; c < 16; ++c) {
            const float r = __ldg(&rj[tid * 16 + c]);
            const float2 v = x[c < 8 ? nA - 8 + c : nA + c - 8];
            acc.x = fmaf(r, v.x, acc.x);
            acc.y = fmaf(r, v.y, acc.y);
        }
        xi[tid] = acc;
    }
    __syncthreads();
    for (int i = tid; i < n; i += blockDim.x) {
        const float* row = spk + (size_t)i * 8;
        const float2* v = (i < nA) ? xi + 8 : xi;
        float2 t = x[i];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float r = __ldg(&row[c]);
            t.x = fmaf(-r, v[c].x, t.x);
            t.y = fmaf(-r, v[c].y, t.y);
        }
        x[i] = t;
    }
    __syncthreads();
}

__device__ __forceinline__ double2 warp_sum(double2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// Row-block dot products by the whole CTA: t_r = sum_{j < nj} R[r nj + j] x[j]
// for the PB rows r of a real row block R (tau rows restricted to some columns)
// against a complex vector, FP64 or FP32.  Each thread takes a stride of j (a few
// loads in flight per thread instead of one warp walking all of them), a
// butterfly per warp, then the warp partials summed in warp order.  Lane r < PB
// of warp 0 gets t_r (every other thread zero).  Contains one __syncthreads; the
// caller's next barrier must come before any thread calls it again.
__device__ __forceinline__ void acc_rx(double2& t, double b, double2 x) {
    t.x = fma(b, x.x, t.x);
    t.y = fma(b, x.y, t.y);
}
__device__ __forceinline__ void acc_rx(float2& t, float b, float2 x) {
    t.x = fmaf(b, x.x, t.x);
    t.y = fmaf(b, x.y, t.y);
}
__device__ __forceinline__ float2 warp_sum(float2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}
__device__ __forceinline__ float2 add_x(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 add_x(double2 a, double2 b) { return cadd(a, b); }

template <int PB, class TX, class TR>
__device__ TX block_rows_dot(const TX* x, int nj, const TR* __restrict__ R) {
    __shared__ TX part[NTHREADS_S / 32][PB];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    TX t[PB];
#pragma unroll
    for (int r = 0; r < PB; ++r) t[r] = zero<TX>();
    for (int j = tid; j < nj; j += blockDim.x) {
        const TX xv = x[j];
#pragma unroll
        for (int r = 0; r < PB; ++r) acc_rx(t[r], __ldg(&R[(size_t)r * nj + j]), xv);
    }
#pragma unroll
    for (int r = 0; r < PB; ++r) t[r] = warp_sum(t[r]);
    if (lane == 0)
#pragma unroll
        for (int r = 0; r < PB; ++r) part[warp][r] = t[r];
    __syncthreads();
    TX v = zero<TX>();
    if (warp == 0 && lane < PB)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = add_x(v, part[w][lane]);
    return v;
}

// FP32 Schur step of the temperature system by the whole CTA: sol[2..] = D^{-1} r
// on entry, sol[0..2) = S^{-1}(g - B sol[2..]) on exit, g = the residual's tau
// rows; B: 2 x (nc-2) tau rows in FP32, Sinv real 2 x 2.  Ends with __syncthreads.
__device__ void block_schur32_dir(float2* sol, const float2* g, int nc, const float* __restrict__ B,
                                  const float* __restrict__ Sinv) {
    const float2 t = block_rows_dot<2>(sol + 2, nc - 2, B);
    if ((threadIdx.x >> 5) == 0) {
        const int lane = threadIdx.x & 31;
        const float2 gv = (lane < 2) ? make_float2(g[lane].x - t.x, g[lane].y - t.y) : make_float2(0.f, 0.f);
        const float2 g0 = shfl_idx(gv, 0), g1 = shfl_idx(gv, 1);
        if (lane < 2) {
            const float a = Sinv[lane * 2], b = Sinv[lane * 2 + 1];
            sol[lane] = make_float2(fmaf(a, g0.x, b * g1.x), fmaf(a, g0.y, b * g1.y));
        }
    }
    __syncthreads();
}

// FP32 Schur step of the temperature system by one warp: sol[2..] = D^{-1} r on
// entry, sol[0..2) = S^{-1}(g - B sol[2..]) on exit, g = the residual's tau rows;
// B: 2 x (nc-2) tau rows in FP32, Sinv real 2 x 2.
__device__ void warp_schur32_dir(float2* sol, const float2* g, int nc, const float* __restrict__ B,
                                 const float* __restrict__ Sinv) {
    const int lane = threadIdx.x & 31;
    const int n = nc - 2;
    float2 t[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    for (int j = lane; j < n; j += 32) {
        const float2 xv = sol[2 + j];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float b = __ldg(&B[(size_t)r * n + j]);
            t[r].x = fmaf(b, xv.x, t[r].x);
            t[r].y = fmaf(b, xv.y, t[r].y);
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            t[r].x += __shfl_xor_sync(0xffffffffu, t[r].x, o);
            t[r].y += __shfl_xor_sync(0xffffffffu, t[r].y, o);
        }
        t[r] = make_float2(g[r].x - t[r].x, g[r].y - t[r].y);
    }
    __syncwarp();
    if (lane < 2) {
        const float a = Sinv[lane * 2], b = Sinv[lane * 2 + 1];
        sol[lane] = make_float2(fmaf(a, t[0].x, b * t[1].x), fmaf(a, t[0].y, b * t[1].y));
    }
    __syncwarp();
}

// FP32 y2 -= Y y1 for the temperature system, threads [t0, t0 + nt)
__device__ void schur_update32_dir(float2* sol, int nc, const float* __restrict__ Y, int t0, int nt) {
    const int n = nc - 2;
    const float2 y0 = sol[0], y1 = sol[1];
    for (int j = threadIdx.x - t0; j < n; j += nt) {
        const float a = Y[(size_t)j * 2], b = Y[(size_t)j * 2 + 1];
        float2 acc = sol[2 + j];
        acc.x -= fmaf(a, y0.x, b * y1.x);
        acc.y -= fmaf(a, y0.y, b * y1.y);
        sol[2 + j] = acc;
    }
}

template <int H>
__device__ __forceinline__ double2 band_row_c(const double* __restrict__ band, const double2* x, int k, int nc) {
    const double* row = band + (size_t)k * (2 * H + 1);
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int d = 0; d <= 2 * H; ++d) {
        const int n = k - H + d;
        if (n >= 0 && n < nc) {
            const double c = __ldg(&row[d]);
            acc.x = fma(c, x[n].x, acc.x);
            acc.y = fma(c, x[n].y, acc.y);
        }
    }
    return acc;
}

// mass / implicit operators applied to one mode's new state
__device__ void apply_row(const StepParams& P, int m, int k, const double2* xp, const double2* xt, const double* xu,
                          VecSet mass_out, VecSet imp_out, bool want_mass, bool want_imp) {
    const int nc = P.nc;
    const double mu = (double)m * m;
    const double dm = (double)m;
    double2 mp = make_double2(0.0, 0.0), ip = make_double2(0.0, 0.0);
    double2 mt = make_double2(0.0, 0.0), it = make_double2(0.0, 0.0);
    if (m > 0 && k >= 4) {
        if (want_mass) {
            const double2 a0 = band_row_c<8>(P.ops.band[OP_A0], xp, k, nc);
            const double2 a2 = band_row_c<8>(P.ops.band[OP_A2], xp, k, nc);
            mp = make_double2(fma(mu, a2.x, a0.x), fma(mu, a2.y, a0.y));
        }
        if (want_imp) {
            const double2 b0 = band_row_c<6>(P.ops.band[OP_B0], xp, k, nc);
            const double2 b2 = band_row_c<6>(P.ops.band[OP_B2], xp, k, nc);
            const double2 b4 = band_row_c<6>(P.ops.band[OP_B4], xp, k, nc);
            const double2 c = band_row_c<8>(P.ops.band[OP_C], xp, k, nc);
            const double ce = 2.0 * dm / P.E;
            ip.x = b0.x + mu * (b2.x + mu * b4.x) - ce * c.y;
            ip.y = b0.y + mu * (b2.y + mu * b4.y) + ce * c.x;
            if (P.buoy_imp)  // (Ra/Pr)(i m/s_o) C^I theta
                ip = cadd(ip, cmul_i(band_row_c<8>(P.ops.band[OP_C], xt, k, nc), P.Ra / P.Pr * dm / P.s_o));
        }
    }
    if (k >= 2) {
        if (want_mass) mt = band_row_c<4>(P.ops.band[OP_D], xt, k, nc);
        if (want_imp) {
            const double2 f0 = band_row_c<2>(P.ops.band[OP_F0], xt, k, nc);
            const double2 f2 = band_row_c<2>(P.ops.band[OP_F2], xt, k, nc);
            const double ip_ = 1.0 / P.Pr;
            it = make_double2((f0.x + mu * f2.x) * ip_, (f0.y + mu * f2.y) * ip_);
        }
    }
    if (want_mass) {
        mass_out.psi[(size_t)m * nc + k] = mp;
        mass_out.th[(size_t)m * nc + k] = mt;
    }
    if (want_imp) {
        imp_out.psi[(size_t)m * nc + k] = ip;
        imp_out.th[(size_t)m * nc + k] = it;
    }
    if (m == 0) {
        double mu_ = 0.0, iu = 0.0;
        if (k >= 2) {
            const double* rd = P.ops.band[OP_D] + (size_t)k * 9;
            const double* re = P.ops.band[OP_EZ] + (size_t)k * 5;
            for (int d = 0; d < 9; ++d) {
                const int n = k - 4 + d;
                if (n >= 0 && n < nc) mu_ = fma(__ldg(&rd[d]), xu[n], mu_);
            }
            for (int d = 0; d < 5; ++d) {
                const int n = k - 2 + d;
                if (n >= 0 && n < nc) iu = fma(__ldg(&re[d]), xu[n], iu);
            }
        }
        if (want_mass) mass_out.u[k] = mu_;
        if (want_imp) imp_out.u[k] = iu;
    }
}

// Epilogue of a solve for row k of mode m: the mass term of the new state
// (A^I_m Psi, D^I theta, D^I u) and, from the solved equation
// (Mass - gamma dt Lin) y = f on the rows below the tau rows, its implicit term
// Lin y = (Mass y - f)/(gamma dt), which saves the banded B^I, C^I, F^I, E^I
// applies.  f is the right-hand side of the solve (recomputed here from the
// same terms in the same order).
__device__ void epilogue_row(const StepParams& P, const RhsSpec& R, double gdt, int m, int k, const double2* xp,
                             const double2* xt, const double* xu, VecSet mass_out, VecSet imp_out, bool want_mass,
                             bool want_imp) {
    const int nc = P.nc;
    const double mu = (double)m * m;
    double2 mp = make_double2(0.0, 0.0), mt = make_double2(0.0, 0.0);
    double muu = 0.0;
    if (m > 0 && k >= 4) {
        const double* r0 = P.ops.band[OP_A0] + (size_t)k * 17;
        const double* r2 = P.ops.band[OP_A2] + (size_t)k * 17;
#pragma unroll
        for (int d = 0; d < 17; ++d) {
            const int n = k - 8 + d;
            if (n >= 0 && n < nc) {
                const double c = fma(mu, __ldg(&r2[d]), __ldg(&r0[d]));
                mp.x = fma(c, xp[n].x, mp.x);
                mp.y = fma(c, xp[n].y, mp.y);
            }
        }
    }
    if (k >= 2) {
        mt = band_row_c<4>(P.ops.band[OP_D], xt, k, nc);
        if (m == 0) {
            const double* rd = P.ops.band[OP_D] + (size_t)k * 9;
            for (int d = 0; d < 9; ++d) {
                const int n = k - 4 + d;
                if (n >= 0 && n < nc) muu = fma(__ldg(&rd[d]), xu[n], muu);
            }
        }
    }
    const size_t idx = (size_t)m * nc + k;
    if (want_imp) {  // before any store: an output may be one of the terms of f
        double2 fp = make_double2(0.0, 0.0), ft = make_double2(0.0, 0.0);
        double fu = 0.0;
        for (int t = 0; t < R.nterms; ++t) {
            const double c = R.t[t].c;
            const double2 vp = R.t[t].v.psi[idx];
            const double2 vt = R.t[t].v.th[idx];
            fp.x = fma(c, vp.x, fp.x);
            fp.y = fma(c, vp.y, fp.y);
            ft.x = fma(c, vt.x, ft.x);
            ft.y = fma(c, vt.y, ft.y);
            if (m == 0) fu = fma(c, R.t[t].v.u[k], fu);
        }
        const double ig = 1.0 / gdt;
        imp_out.psi[idx] = (m > 0 && k >= 4) ? cscale(csub(mp, fp), ig) : make_double2(0.0, 0.0);
        imp_out.th[idx] = (k >= 2) ? cscale(csub(mt, ft), ig) : make_double2(0.0, 0.0);
        if (m == 0) imp_out.u[k] = (k >= 2) ? (muu - fu) * ig : 0.0;
    }
    if (want_mass) {
        mass_out.psi[idx] = mp;
        mass_out.th[idx] = mt;
        if (m == 0) mass_out.u[k] = muu;
    }
}

// ---------------------------------------------------------------------------
// The same steps spread over the CTA by component (k_solve).  An FP64 instruction
// of a warp takes 64 cycles of its sub-partition whatever it does, so a phase costs
// its longest warp's FP64 instructions: one warp adding 4 complex sums over its
// lanes one by one spent 40 of them (2600 cycles), the rows of a system one thread
// each left most warps idle.  Here a task is (row, component), and the sums of
// a row block over the CTA are added by exchanging halves of the values.
// ---------------------------------------------------------------------------
// v[0 .. 2^LOG): each lane's partial sums; returns the sum over the warp of value
// (lane >> (5 - LOG)), the same in the lanes that share it.
template <int LOG>
__device__ __forceinline__ double warp_sums(double (&v)[1 << LOG]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int s = 0; s < LOG; ++s) {
        const int o = 16 >> s, half = 1 << (LOG - 1 - s);
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const double send = up ? v[i] : v[i + half];
            const double keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 16 >> LOG; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}
// Partial sums of the PB rows R (PB x nj, real) against a complex vector x, one
// value per (row, component): part[warp][2 row + component].
template <int PB>
__device__ __forceinline__ void rows_dot_part(const double2* x, int nj, const double* __restrict__ R,
                                              double (*part)[8]) {
    constexpr int LOG = PB == 4 ? 3 : 2;
    const int tid = threadIdx.x, lane = tid & 31;
    double t[1 << LOG];
#pragma unroll
    for (int i = 0; i < 2 * PB; ++i) t[i] = 0.0;
    for (int j = tid; j < nj; j += blockDim.x) {
        const double2 xv = x[j];
#pragma unroll
        for (int r = 0; r < PB; ++r) {
            const double b = __ldg(&R[(size_t)r * nj + j]);
            t[2 * r] = fma(b, xv.x, t[2 * r]);
            t[2 * r + 1] = fma(b, xv.y, t[2 * r + 1]);
        }
    }
    const double v = warp_sums<LOG>(t);
    if ((lane & ((32 >> LOG) - 1)) == 0) part[tid >> 5][lane >> (5 - LOG)] = v;
}
// the sums over the CTA's eight warps: lane l of the calling warp gets value l & 7
__device__ __forceinline__ double rows_dot_sum(const double (*part)[8], int nval) {
    const int lane = threadIdx.x & 31, i = lane & 7, w = lane >> 3;
    double v = (i < nval) ? part[w][i] + part[w + 4][i] : 0.0;
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}
// sol[0 .. PB) = S^{-1} (g - t) by one warp, t the sums of rows_dot_sum (value 2 r +
// component in lane 2 r + component), g = 0 when null.  Lane (row, component, c)
// takes one term.
__device__ __forceinline__ double2 as_complex(double2 a) { return a; }
__device__ __forceinline__ double2 as_complex(double a) { return make_double2(a, 0.0); }
template <int PB, class TS>
__device__ __forceinline__ void schur_apply(double2* sol, const double2* g, double t, const TS* __restrict__ Sinv) {
    const int lane = threadIdx.x & 31;
    double gv = 0.0;
    if (lane < 2 * PB) gv = (g ? reinterpret_cast<const double*>(g)[lane] : 0.0) - t;
    const int c = lane % PB, p = (lane / PB) & 1, r = lane / (2 * PB);
    const double gx = __shfl_sync(0xffffffffu, gv, 2 * c), gy = __shfl_sync(0xffffffffu, gv, 2 * c + 1);
    const bool on = r < PB;
    const double2 a = on ? as_complex(Sinv[r * PB + c]) : make_double2(0.0, 0.0);
    double v = fma(a.x, p ? gy : gx, a.y * (p ? gx : -gy));
#pragma unroll
    for (int o = 1; o < PB; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (on && c == 0) reinterpret_cast<double*>(sol)[2 * r + p] = v;
}
// component part of y2 -= Y y1, every (row, component) of the CTA
__device__ __forceinline__ double fms_part(double acc, double a, double2 z, int part) {
    return fma(-a, part ? z.y : z.x, acc);
}
template <int PB, class TF>
__device__ __forceinline__ void schur_update_parts(double2* sol, int nc, const TF* __restrict__ Y) {
    const int part = threadIdx.x & 1;
    double2 y1[PB];
#pragma unroll
    for (int c = 0; c < PB; ++c) y1[c] = sol[c];
    for (int t = threadIdx.x; t < 2 * (nc - PB); t += blockDim.x) {
        double* x = reinterpret_cast<double*>(sol + PB) + t;
        double acc = *x;
#pragma unroll
        for (int c = 0; c < PB; ++c) acc = fms_part(acc, Y[(size_t)(t >> 1) * PB + c], y1[c], part);
        *x = acc;
    }
}
// component part of f_k - (L x)_k, a complex band row of half width 8
__device__ __forceinline__ double residual_part(double acc, const double2* __restrict__ row, const double2* x, int k, int nc,
                                                int part) {
#pragma unroll
    for (int d = 0; d < 17; ++d) {
        const int n = k - 8 + d;
        if (n >= 0 && n < nc) acc = fms_part(acc, __ldg(&row[d]), x[n], part);
    }
    return acc;
}
// row k, one component, of a real band applied to complex values (x: that component, stride 2)
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
// Epilogue of a solve (epilogue_row) for one component of row k: the streamfunction's
// mass term A^I_m Psi and its implicit term (mass - f)/(gamma dt), f the component
// of the assembled right-hand side (fps) or, null, its terms summed again.
__device__ __forceinline__ void epilogue_psi_part(const StepParams& P, const RhsSpec& R, double gdt, int m, int k, int part,
                                                  const double2* xp, VecSet mass_out, VecSet imp_out, bool want_mass,
                                                  bool want_imp, const double2* fps) {
    const int nc = P.nc;
    const size_t idx = 2 * ((size_t)m * nc + k) + part;
    const double mu = (double)m * m;
    double mp = 0.0, im = 0.0;
    if (m > 0 && k >= 4) {
        const double* r0 = P.ops.band[OP_A0] + (size_t)k * 17;
        const double* r2 = P.ops.band[OP_A2] + (size_t)k * 17;
        const double* x = reinterpret_cast<const double*>(xp) + part;
        // the row's coefficients, half of them by each component's lane
        const unsigned both = 3u << (threadIdx.x & 30);
        double c[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int d = min(2 * i + part, 16);
            c[i] = fma(mu, __ldg(&r2[d]), __ldg(&r0[d]));
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double o = __shfl_xor_sync(both, c[i], 1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int n = k - 8 + 2 * i + h;
                if (2 * i + h < 17 && n >= 0 && n < nc) mp = fma(h == part ? c[i] : o, x[2 * n], mp);
            }
        }
        if (want_imp) {  // before any store: an output may be one of the terms of f
            double f = 0.0;
            if (fps)
                f = reinterpret_cast<const double*>(fps)[2 * k + part];
            else
                for (int t = 0; t < R.nterms; ++t) f = fma(R.t[t].c, reinterpret_cast<const double*>(R.t[t].v.psi)[idx], f);
            im = (mp - f) * (1.0 / gdt);
        }
    }
    if (want_imp) reinterpret_cast<double*>(imp_out.psi)[idx] = im;
    if (want_mass) reinterpret_cast<double*>(mass_out.psi)[idx] = mp;
}
// the same for the temperature (fts always kept) and, for m = 0 and component 0,
// the zonal flow (fus kept, or null)
__device__ __forceinline__ void epilogue_theta_part(const StepParams& P, const RhsSpec& R, double gdt, int m, int k,
                                                    int part, const double2* xt, const double* xu, VecSet mass_out,
                                                    VecSet imp_out, bool want_mass, bool want_imp, const double2* fts,
                                                    const double* fus) {
    const int nc = P.nc;
    const size_t idx = 2 * ((size_t)m * nc + k) + part;
    const double ig = 1.0 / gdt;
    const double mt = (k >= 2) ? band_part<4>(P.ops.band[OP_D], reinterpret_cast<const double*>(xt) + part, k, nc) : 0.0;
    if (want_imp)
        reinterpret_cast<double*>(imp_out.th)[idx] =
            (k >= 2) ? (mt - reinterpret_cast<const double*>(fts)[2 * k + part]) * ig : 0.0;
    if (want_mass) reinterpret_cast<double*>(mass_out.th)[idx] = mt;
    if (m == 0 && part == 0) {
        double mu = 0.0;
        if (k >= 2) {
            const double* rd = P.ops.band[OP_D] + (size_t)k * 9;
            for (int d = 0; d < 9; ++d) {
                const int n = k - 4 + d;
                if (n >= 0 && n < nc) mu = fma(__ldg(&rd[d]), xu[n], mu);
            }
        }
        if (want_imp) {
            double f = 0.0;
            if (fus)
                f = fus[k];
            else
                for (int t = 0; t < R.nterms; ++t) f = fma(R.t[t].c, R.t[t].v.u[k], f);
            imp_out.u[k] = (k >= 2) ? (mu - f) * ig : 0.0;
        }
        if (want_mass) mass_out.u[k] = mu;
    }
}

// shared-memory layout of one CTA (chains run in place in the solution's array):
//   streamfunction: pf rhs (then the refinement residual), px solution, pd correction
//   temperature:    tf rhs, tx solution
// and for the zonal flow (the CTA holding m = 0): uf rhs, ux solution (real).
struct SolveSmem {
    double2 *pf, *px, *pd, *tf, *tx;
    double *uf, *ux;
    float2 *tr, *td;  // refined FP32 temperature solves: residual, correction
    char *ring_p, *ring_t, *ring_u;  // the walks' rings of matrices (the zonal flow's over the streamfunction's)
    double (*prevs)[32];             // the walking warps' previous blocks
    // the streamfunction and zonal-flow right-hand sides as assembled (pf and uf
    // become residuals), for the epilogue
    double2* fp;
    double* fu;
};

__host__ __device__ inline int round8(int n) { return (n + 7) / 8 * 8; }

// rows of an array that a chain solves in place: whole blocks past an offset of up to 4
__host__ __device__ inline int chain_rows(int nc) { return round8(nc) + 8; }

// shared_d: the streamfunction's correction over the temperature's FP32 arrays, which are
// done with before it is formed when the buoyancy is implicit: two CTAs on an SM
// instead of one at N_c = 682 (solve at 1025 x 1536 1100 -> 788 us)
__host__ __device__ inline size_t solve_smem_doubles(int nc, bool shared_d) {
    return (size_t)(shared_d ? 12 : 14) * chain_rows(nc) + (4 * ring_bytes<double2>() + 2 * ring_bytes<double>()) / 8 +
           3 * (size_t)round8(nc);  // (208 KB at N_c = 1365, the largest)
}

__device__ __forceinline__ SolveSmem carve(double2* base, int nc, bool shared_d) {
    SolveSmem s;
    const int b = chain_rows(nc);
    s.pf = base;
    s.px = base + b;
    s.tf = base + 2 * b;
    s.tx = base + 3 * b;
    s.uf = reinterpret_cast<double*>(base + 4 * b);
    s.ux = s.uf + b;
    s.tr = reinterpret_cast<float2*>(s.ux + b);
    s.td = s.tr + b;
    s.pd = reinterpret_cast<double2*>(s.tr) + (shared_d ? 0 : b);
    s.ring_p = reinterpret_cast<char*>(s.pd + b);
    s.ring_t = s.ring_p + 4 * ring_bytes<double2>();
    s.ring_u = s.ring_p;
    s.fp = reinterpret_cast<double2*>(s.ring_t + 2 * ring_bytes<double>());
    s.fu = reinterpret_cast<double*>(s.fp + round8(nc));
    return s;
}

// The zonal flow's chain (the CTA of m = 0) by warps 4-5
__device__ void zonal_chains(const DevFactors& F, SolveSmem& s, double* b, double* x, int nt) {
    run_chains<2>(no_job<double, 1>(), no_job<double, 1>(), no_job<float, 2>(),
                      ChainJob<double, 1>{b, x, x, nt, F.uBlk, 4, s.ring_u}, s.prevs);
}

// One FP64 refinement step of the zonal-flow solve (the CTA of m = 0, large N_c):
// r = f - L u over the assembled rows and the tau rows, solved with the same
// factors, u += correction.  The residual replaces the right-hand side; the
// correction uses a streamfunction array, which mode 0 leaves unused.
__device__ void refine_zonal_flow(const StepParams& P, const DevFactors& F, SolveSmem& s) {
    const int nc = P.nc, nt = nc - 2;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
    for (int k = 2 + tid; k < nc; k += nth) {
        const double* row = F.uBand + (size_t)(k - 2) * 9;
        double acc = s.uf[k];
        for (int d = 0; d < 9; ++d) {
            const int n = k - 4 + d;
            if (n >= 0 && n < nc) acc = fma(-__ldg(&row[d]), s.ux[n], acc);
        }
        s.uf[k] = acc;
    }
    if (warp == 0) {  // tau rows: r = 0 - tau u
        double t0 = 0.0, t1 = 0.0;
        for (int j = lane; j < nc; j += 32) {
            t0 = fma(__ldg(&P.ops.tau_dir[j]), s.ux[j], t0);
            t1 = fma(__ldg(&P.ops.tau_dir[nc + j]), s.ux[j], t1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            t0 += __shfl_xor_sync(0xffffffffu, t0, o);
            t1 += __shfl_xor_sync(0xffffffffu, t1, o);
        }
        if (lane < 2) s.uf[lane] = -(lane ? t1 : t0);
    }
    __syncthreads();
    double* du = reinterpret_cast<double*>(s.pd);
    zonal_chains(F, s, s.uf + 2, du + 2, nt);
    {
        if (warp == 4) {
            double t0 = 0.0, t1 = 0.0;
            for (int j = lane; j < nt; j += 32) {
                t0 = fma(__ldg(&P.ops.tau_dir_B[j]), du[2 + j], t0);
                t1 = fma(__ldg(&P.ops.tau_dir_B[nt + j]), du[2 + j], t1);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t0 += __shfl_xor_sync(0xffffffffu, t0, o);
                t1 += __shfl_xor_sync(0xffffffffu, t1, o);
            }
            const double g0 = s.uf[0], g1 = s.uf[1];
            __syncwarp();
            if (lane < 2) du[lane] = F.uSinv[lane * 2] * (g0 - t0) + F.uSinv[lane * 2 + 1] * (g1 - t1);
            __syncwarp();
        }
    }
    __syncthreads();
    {
        const double u0 = du[0], u1 = du[1];
        for (int j = tid; j < nt; j += nth) du[2 + j] -= F.uY[(size_t)j * 2] * u0 + F.uY[(size_t)j * 2 + 1] * u1;
    }
    __syncthreads();
    for (int n = tid; n < nc; n += nth) s.ux[n] += du[n];
    __syncthreads();
}

// FP64 residual r = f - L x of the temperature system of mode m0,
// rounded to FP32 into s.tr: the assembled rows by the whole CTA, the two tau
// rows (r = 0 - tau x) by warp tw.  The caller synchronises.
__device__ void temperature_residual(const StepParams& P, const DevFactors& F, SolveSmem& s, int m0, int tw) {
    const int nc = P.nc, nt = nc - 2;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
    for (int k = 2 + tid; k < nc; k += nth) {
        const double* row = F.tBand + ((size_t)m0 * nt + (k - 2)) * 9;
        double2 acc = s.tf[k];
#pragma unroll
        for (int d = 0; d < 9; ++d) {
            const int n = k - 4 + d;
            if (n >= 0 && n < nc) acc = fms(acc, __ldg(&row[d]), s.tx[n]);
        }
        s.tr[k] = to_f2(acc);
    }
    if (warp == tw) {
        double2 t0 = make_double2(0.0, 0.0), t1 = t0;
        for (int j = lane; j < nc; j += 32) {
            const double2 xv = s.tx[j];
            const double b0 = __ldg(&P.ops.tau_dir[j]), b1 = __ldg(&P.ops.tau_dir[nc + j]);
            t0.x = fma(b0, xv.x, t0.x);
            t0.y = fma(b0, xv.y, t0.y);
            t1.x = fma(b1, xv.x, t1.x);
            t1.y = fma(b1, xv.y, t1.y);
        }
        t0 = warp_sum(t0);
        t1 = warp_sum(t1);
        if (lane < 2) s.tr[lane] = to_f2(lane ? make_double2(-t1.x, -t1.y) : make_double2(-t0.x, -t0.y));
    }
}

// The FP32 temperature solve D td = tr of the kernel with one CTA per system:
// one block walked by warps 2-3, or (tsplit) its two halves by warps 2-3 and 4-5
// joined through the spikes.  Whole CTA; ends with a barrier.
__device__ __forceinline__ void theta32_chains(const DevFactors& F, SolveSmem& s, int m, int nt, int nbt) {
    const float* tb = (F.tsplit ? F.tBlk32S : F.tBlk32) + (size_t)m * nbt * 192;
    float *b = reinterpret_cast<float*>(s.tr + 2), *x = reinterpret_cast<float*>(s.td + 2);
    const int ntA = F.tsplit ? 8 * (nbt / 2) : nt;
    run_chains<4>(ChainJob<float, 2>{b, x, x, ntA, tb, 2, s.ring_t},
                      ChainJob<float, 2>{b + 2 * ntA, x + 2 * ntA, x + 2 * ntA, nt - ntA, tb + (size_t)(nbt / 2) * 192, 4,
                                         s.ring_t + 2 * ring_bytes<float>()},
                      no_job<double, 1>(), no_job<double, 1>(), s.prevs);
    if (F.tsplit) split_join32(s.td + 2, nt, ntA, F.tSpk32 + (size_t)m * nt * 8, F.tRj32 + (size_t)m * 256);
}

// The same residual with the tau rows summed by the whole CTA (kernel with one
// CTA per system, where no other system's warps run beside it).  Contains one
// __syncthreads; the caller's next barrier publishes s.tr.
__device__ void temperature_residual_block(const StepParams& P, const DevFactors& F, SolveSmem& s, int m0) {
    const int nc = P.nc, nt = nc - 2;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
    for (int k = 2 + tid; k < nc; k += nth) {
        const double* row = F.tBand + ((size_t)m0 * nt + (k - 2)) * 9;
        double2 acc = s.tf[k];
#pragma unroll
        for (int d = 0; d < 9; ++d) {
            const int n = k - 4 + d;
            if (n >= 0 && n < nc) acc = fms(acc, __ldg(&row[d]), s.tx[n]);
        }
        s.tr[k] = to_f2(acc);
    }
    const double2 t = block_rows_dot<2>(s.tx, nc, P.ops.tau_dir);
    if (warp == 0 && lane < 2) s.tr[lane] = to_f2(make_double2(-t.x, -t.y));
}

// The FP32-refined temperature solve of the kernel with one CTA per system:
// ir_t corrections x += S32^{-1}(f - L x), every reduction by the whole CTA.
__device__ __forceinline__ void temperature_corrections_roles(const StepParams& P, const DevFactors& F, SolveSmem& s, int m0) {
    const int nc = P.nc, nt = nc - 2, nbt = (nt + 7) / 8;
    const int tid = threadIdx.x, nth = blockDim.x;
    for (int it = 0; it < F.ir_t; ++it) {
        temperature_residual_block(P, F, s, m0);
        __syncthreads();
        theta32_chains(F, s, m0, nt, nbt);
        block_schur32_dir(s.td, s.tr, nc, P.ops.tau_dir_B32, F.tSinv32 + (size_t)m0 * 4);
        schur_update32_dir(s.td, nc, F.tY32 + (size_t)m0 * nt * 2, 0, nth);
        __syncthreads();
        for (int n = tid; n < nc; n += nth) s.tx[n] = cadd(s.tx[n], to_d2_bits(s.td[n]));
        __syncthreads();
    }
}

// the whole FP32 temperature block, walked by warps w, w + 1
__device__ __forceinline__ ChainJob<float, 2> theta32_job(const DevFactors& F, const SolveSmem& s, int m0, int nt, int nbt, int w) {
    return ChainJob<float, 2>{reinterpret_cast<float*>(s.tr + 2), reinterpret_cast<float*>(s.td + 2),
                              reinterpret_cast<float*>(s.td + 2), nt, F.tBlk32 + (size_t)m0 * nbt * 192, w, s.ring_t};
}

// The FP32-refined temperature solve (F.ir_t > 0, MB == 1): x += S32^{-1}(f - L x)
// for the passes it0 .. ir_t - 1 (pass 0 may have run beside the streamfunction
// refinement), then the FP64 refinement of the zonal flow (mode 0).
template <bool IMP>
__device__ __forceinline__ void temperature_corrections(const StepParams& P, const DevFactors& F, SolveSmem& s, int m0, bool has_u,
                                        int it0) {
    const int nc = P.nc, nt = nc - 2, nbt = (nt + 7) / 8;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5;
    if (F.ir_t) {
        if constexpr (IMP) temperature_corrections_roles(P, F, s, m0);
        for (int it = IMP ? F.ir_t : it0; it < F.ir_t; ++it) {
            temperature_residual(P, F, s, m0, 0);
            __syncthreads();
            run_chains<4>(no_job<float, 2>(), no_job<float, 2>(), theta32_job(F, s, m0, nt, nbt, 2), no_job<double, 1>(), s.prevs);
            if (warp == 2) warp_schur32_dir(s.td, s.tr, nc, P.ops.tau_dir_B32, F.tSinv32 + (size_t)m0 * 4);
            __syncthreads();
            schur_update32_dir(s.td, nc, F.tY32 + (size_t)m0 * nt * 2, 0, nth);
            __syncthreads();
            for (int n = tid; n < nc; n += nth) s.tx[n] = cadd(s.tx[n], to_d2_bits(s.td[n]));
            __syncthreads();
        }
        if (has_u) refine_zonal_flow(P, F, s);  // FP64
    }
}

// T32: the temperature by FP32 chains refined from FP64 residuals (F.ir_t); DDP:
// double-float streamfunction chains (explicit buoyancy); IMP: implicit buoyancy
template <bool T32, bool DDP, bool IMP>
__global__ void __launch_bounds__(NTHREADS_S, 2) k_solve(StepParams P, RhsSpec R, DevFactors F, VecSet y_out,
                                                      VecSet mass_out, VecSet imp_out, int want_mass,
                                                      int want_imp) {
    chain_wait();
    extern __shared__ double2 sm[];
    __shared__ double part_p[NTHREADS_S / 32][8], part_t[NTHREADS_S / 32][8];
    const int nc = P.nc;
    const int m0 = P.m_lo + blockIdx.x;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
    const int part = tid & 1;  // the component of this thread's tasks
    const int np = nc - 4, nt = nc - 2;
    const int nbp = (np + 7) / 8, nbt = (nt + 7) / 8;
    const int nA = 8 * (nbp / 2);  // first half of a split streamfunction block (F.psplit)
    SolveSmem s = carve(sm, nc, T32 && IMP);
    __shared__ __align__(16) double prevs[NTHREADS_S / 32][32];
    s.prevs = prevs;
    const bool has_u = (m0 == 0);
    // Warps w, w + 4 of a CTA run on the same sub-partition, and so do the same warps of
    // the two CTAs of an SM, whose chains then wait for one FP64 pipe: the CTA in the
    // odd slot swaps its warp pairs (a hint only; any value gives the same results).
    __shared__ int flip_s;
    if (tid == 0) {
        unsigned w;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(w));
        flip_s = (w >> 3) & 1 ? 2 : 0;
    }
    __syncthreads();
    const int flip = flip_s;
    using CP = std::conditional_t<DDP, ddc, double2>;  // the streamfunction chain's coefficients and components
    using VP = typename Chain<CP>::V;
    const CP* blk_p = DDP ? reinterpret_cast<const CP*>(F.pBlkDD) : reinterpret_cast<const CP*>(F.pBlk);
    blk_p += (size_t)m0 * nbp * 192;
    const ddc* spk_dd = reinterpret_cast<const ddc*>(F.pSpkDD) + (size_t)m0 * np * 8;
    const ddc* rj_dd = reinterpret_cast<const ddc*>(F.pRjDD) + (size_t)m0 * 256;
    // the streamfunction block, one or (psplit) two halves: right-hand side b to x
    auto job_p = [&](double2* b, double2* x, bool second) {
        const int n0 = second ? nA : 0, n = m0 == 0 ? 0 : second ? (F.psplit ? np - nA : 0) : F.psplit ? nA : np;
        return ChainJob<CP, 2>{reinterpret_cast<VP*>(b + 4 + n0), reinterpret_cast<VP*>(x + 4 + n0), reinterpret_cast<VP*>(x + 4 + n0), n,
                               blk_p + (second ? (size_t)(nbp / 2) * 192 : 0), (second ? 6 : 0) ^ flip,
                               s.ring_p + (second ? 2 * ring_bytes<CP>() : 0)};
    };
    // the temperature: FP32, or FP64
    using CT = std::conditional_t<T32, float, double>;
    auto job_t = [&]() {
        if constexpr (T32)
            return theta32_job(F, s, m0, nt, nbt, 2 ^ flip);
        else
            return ChainJob<double, 2>{reinterpret_cast<double*>(s.tf + 2), reinterpret_cast<double*>(s.tx + 2),
                                       reinterpret_cast<double*>(s.tx + 2), nt, F.tBlk + (size_t)m0 * nbt * 192, 2 ^ flip, s.ring_t};
    };
    auto job_u = [&]() {
        return ChainJob<double, 1>{s.uf + 2, s.ux + 2, s.ux + 2, nt, F.uBlk, 4 ^ flip, s.ring_u};
    };
    auto flat = [](double2* v) { return reinterpret_cast<double*>(v); };

    // 1. right-hand side sum_t c_t V_t (tau rows zero)
    for (int q = tid; q < 2 * nc; q += nth) {
        const int n = q >> 1;
        const size_t idx = (size_t)m0 * 2 * nc + q;
        double ap = 0.0, at = 0.0, au = 0.0;
#pragma unroll 4
        for (int t = 0; t < R.nterms; ++t) {
            const double c = R.t[t].c;
            ap = fma(c, reinterpret_cast<const double*>(R.t[t].v.psi)[idx], ap);
            at = fma(c, reinterpret_cast<const double*>(R.t[t].v.th)[idx], at);
            if (has_u) au = fma(c, R.t[t].v.u[n], au);
        }
        if (n < 4 || m0 == 0) ap = 0.0;
        if (n < 2) at = 0.0;
        flat(s.pf)[q] = ap;
        // double-float streamfunction chains (explicit buoyancy): the right-hand side
        // as double-floats in pd, which the correction fills later
        if (DDP && m0 > 0) reinterpret_cast<ddf*>(s.pd)[q] = dd_from_bits(ap);
        flat(s.tf)[q] = at;
        if (T32) reinterpret_cast<float*>(s.tr)[q] = f32_from_bits(at);
        if (has_u && part == 0) s.uf[n] = (n < 2) ? 0.0 : au;
        flat(s.fp)[q] = ap;  // for the epilogue: pf and uf become residuals
        if (has_u && part == 0) s.fu[n] = s.uf[n];
    }
    __syncthreads();

    // 2.-4. banded solves, Schur steps and Y updates.  With explicit buoyancy the
    //    streamfunction and temperature systems are independent and run together;
    //    with implicit buoyancy (Section 4) the temperature (and zonal flow) goes
    //    first, then g (Ra/Pr)(i m/s_o) C^I theta_new joins the streamfunction rows.
    const int npass = IMP ? 2 : 1;
    for (int pass = 0; pass < npass; ++pass) {
        const bool do_p = !IMP || pass == 1;
        const bool do_t = !IMP || pass == 0;
        if (IMP && pass == 1) {
            if (m0 > 0) {
                const double cb = F.gdt * P.Ra / P.Pr * (double)m0 / P.s_o;
                for (int q = 8 + tid; q < 2 * nc; q += nth) {
                    const double v = band_part<8>(P.ops.band[OP_C], flat(s.tx) + (part ^ 1), q >> 1, nc);
                    flat(s.pf)[q] = fma(part ? cb : -cb, v, flat(s.pf)[q]);
                }
            }
            __syncthreads();
        }
        // 2. banded solves by warp pairs: warps 0-1 the streamfunction (6-7 its second
        //    half), 2-3 the temperature, 4-5 the zonal flow (m = 0 only)
        // implicit buoyancy: the FP32 temperature solve has the CTA to itself, so its block
        // goes in halves and its sums over every warp, as in k_solve_roles (1025 x 384:
        // 268 -> 257 us, 2049 x 384: 516 -> 470)
        const bool alone_t = T32 && IMP && do_t;
        if (alone_t) {
            theta32_chains(F, s, m0, nt, nbt);
            if (has_u) zonal_chains(F, s, s.uf + 2, s.ux + 2, nt);
        } else {
            run_chains<2>(do_p ? job_p(DDP ? s.pd : s.pf, s.px, false) : no_job<CP, 2>(),
                          do_p ? job_p(DDP ? s.pd : s.pf, s.px, true) : no_job<CP, 2>(),
                          do_t ? job_t() : no_job<CT, 2>(), do_t && has_u ? job_u() : no_job<double, 1>(), s.prevs);
        }
        if (DDP && do_p && m0 > 0) {  // the solution back from double-floats
            if (F.psplit) split_join_dd(reinterpret_cast<ddc*>(s.px) + 4, np, nA, spk_dd, rj_dd, true);
            const ddf* xd = reinterpret_cast<const ddf*>(s.px);
            for (int q = 8 + tid; q < 2 * nc; q += nth) flat(s.px)[q] = dd_compose(xd[q]);
            __syncthreads();
        }
        if (!DDP && do_p && F.psplit)
            split_join(s.px + 4, np, nA, F.pSpk + (size_t)(m0 > 0 ? m0 : 0) * np * 8,
                       F.pRj + (size_t)(m0 > 0 ? m0 : 0) * 256, m0 > 0);

        // 3. Schur steps: the tau rows' sums by the CTA, then warp 0 the streamfunction,
        //    2 the temperature, 4 the zonal flow
        if (do_p && m0 > 0) rows_dot_part<4>(s.px + 4, np, P.ops.tau_psi_B, part_p);
        if (do_t && !T32) rows_dot_part<2>(s.tx + 2, nt, P.ops.tau_dir_B, part_t);
        if (alone_t) block_schur32_dir(s.td, s.tr, nc, P.ops.tau_dir_B32, F.tSinv32 + (size_t)m0 * 4);
        __syncthreads();
        if (warp == 0) {
            if (do_p && m0 > 0) schur_apply<4>(s.px, nullptr, rows_dot_sum(part_p, 8), F.pSinv + (size_t)m0 * 16);
        } else if (warp == 2) {
            if (do_t && !alone_t) {
                if (T32)
                    warp_schur32_dir(s.td, s.tr, nc, P.ops.tau_dir_B32, F.tSinv32 + (size_t)m0 * 4);
                else
                    schur_apply<2>(s.tx, nullptr, rows_dot_sum(part_t, 4), F.tSinv + (size_t)m0 * 4);
            }
        } else if (warp == 4 && has_u && do_t) {
            double t0 = 0.0, t1 = 0.0;
            for (int j = lane; j < nt; j += 32) {
                t0 = fma(__ldg(&P.ops.tau_dir_B[j]), s.ux[2 + j], t0);
                t1 = fma(__ldg(&P.ops.tau_dir_B[nt + j]), s.ux[2 + j], t1);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t0 += __shfl_xor_sync(0xffffffffu, t0, o);
                t1 += __shfl_xor_sync(0xffffffffu, t1, o);
            }
            if (lane < 2) s.ux[lane] = -(F.uSinv[lane * 2] * t0 + F.uSinv[lane * 2 + 1] * t1);
            __syncwarp();
        }
        __syncthreads();
        // 4. y2 -= Y y1
        if (do_p && m0 > 0) schur_update_parts<4>(s.px, nc, F.pY + (size_t)m0 * np * 4);
        if (do_t) {
            if (T32)
                schur_update32_dir(s.td, nc, F.tY32 + (size_t)m0 * nt * 2, 0, nth);
            else
                schur_update_parts<2>(s.tx, nc, F.tY + (size_t)m0 * nt * 2);
            if (has_u) {
                const double u0 = s.ux[0], u1 = s.ux[1];
                for (int j = tid; j < nt; j += nth)
                    s.ux[2 + j] -= F.uY[(size_t)j * 2] * u0 + F.uY[(size_t)j * 2 + 1] * u1;
            }
        }
        __syncthreads();
        if (T32 && do_t) {  // the FP32 temperature solve becomes the FP64 iterate
            for (int n = tid; n < nc; n += nth) s.tx[n] = to_d2_bits(s.td[n]);
            __syncthreads();
        }
        if (IMP && pass == 0) temperature_corrections<IMP>(P, F, s, m0, has_u, 0);
    }

    // 5. one refinement step of the streamfunction solve: r = f - L x (a second
    //    step gains nothing: FP64 residuals limit the accuracy to ~cond * eps).
    //    With the FP32-refined temperature solve and explicit buoyancy the first
    //    temperature correction runs beside it: its chain (FP32, warps 2-3) beside
    //    the streamfunction chains (FP64), on disjoint arrays.
    const bool fuse_t = T32 && !IMP;
    if (m0 > 0) {
        for (int q = 8 + tid; q < 2 * nc; q += nth) {
            const int k = q >> 1;
            const double acc = residual_part(flat(s.pf)[q], F.pBand + ((size_t)m0 * np + (k - 4)) * 17, s.px, k, nc, part);
            if (DDP)  // the residual replaces the right-hand side, as double-floats
                reinterpret_cast<ddf*>(s.pf)[q] = dd_from_bits(acc);
            else
                flat(s.pf)[q] = acc;
        }
        rows_dot_part<4>(s.px, nc, P.ops.tau_psi, part_p);  // tau rows: r = 0 - tau x
    }
    if (fuse_t) temperature_residual(P, F, s, m0, 1);
    __syncthreads();
    if (warp == 2 && m0 > 0) {
        const double t = rows_dot_sum(part_p, 8);
        if (lane < 8) flat(s.pf)[lane] = -t;  // read by the Schur step below, past the next barrier
    }
    if (fuse_t)
        run_chains<2>(job_p(s.pf, s.pd, false), job_p(s.pf, s.pd, true), job_t(), no_job<double, 1>(), s.prevs);
    else if (m0 > 0)
        run_chains<2>(job_p(s.pf, s.pd, false), job_p(s.pf, s.pd, true), no_job<CT, 2>(), no_job<double, 1>(),
                          s.prevs);
    if (fuse_t) {
        if (warp == 2) warp_schur32_dir(s.td, s.tr, nc, P.ops.tau_dir_B32, F.tSinv32 + (size_t)m0 * 4);
        __syncthreads();
    }
    if (m0 > 0) {
        if (DDP) {  // the correction back from double-floats
            if (F.psplit) split_join_dd(reinterpret_cast<ddc*>(s.pd) + 4, np, nA, spk_dd, rj_dd, true);
            const ddf* xd = reinterpret_cast<const ddf*>(s.pd);
            for (int q = 8 + tid; q < 2 * nc; q += nth) flat(s.pd)[q] = dd_compose(xd[q]);
            __syncthreads();
        }
        if (!DDP && F.psplit) split_join(s.pd + 4, np, nA, F.pSpk + (size_t)m0 * np * 8, F.pRj + (size_t)m0 * 256, true);
        rows_dot_part<4>(s.pd + 4, np, P.ops.tau_psi_B, part_p);
        __syncthreads();
        if (warp == 0) schur_apply<4>(s.pd, s.pf, rows_dot_sum(part_p, 8), F.pSinv + (size_t)m0 * 16);
        __syncthreads();
        schur_update_parts<4>(s.pd, nc, F.pY + (size_t)m0 * np * 4);
    }
    if (fuse_t) schur_update32_dir(s.td, nc, F.tY32 + (size_t)m0 * nt * 2, 0, nth);
    __syncthreads();
    for (int q = tid; q < 2 * nc; q += nth) flat(s.px)[q] = m0 ? flat(s.px)[q] + flat(s.pd)[q] : 0.0;
    if (fuse_t)
        for (int n = tid; n < nc; n += nth) s.tx[n] = cadd(s.tx[n], to_d2_bits(s.td[n]));
    __syncthreads();
    if (!IMP) temperature_corrections<IMP>(P, F, s, m0, has_u, fuse_t ? 1 : 0);

    // 6. store, then mass / implicit operators for later stages
    for (int q = tid; q < 2 * nc; q += nth) {
        reinterpret_cast<double*>(y_out.psi)[(size_t)m0 * 2 * nc + q] = flat(s.px)[q];
        reinterpret_cast<double*>(y_out.th)[(size_t)m0 * 2 * nc + q] = flat(s.tx)[q];
        if (has_u && part == 0) y_out.u[q >> 1] = s.ux[q >> 1];
    }
    if (want_mass || want_imp)
        for (int q = tid; q < 4 * nc; q += nth) {
            if (q < 2 * nc)
                epilogue_psi_part(P, R, F.gdt, m0, q >> 1, part, s.px, mass_out, imp_out, want_mass, want_imp,
                                  s.fp);
            else
                epilogue_theta_part(P, R, F.gdt, m0, (q - 2 * nc) >> 1, part, s.tx, s.ux, mass_out, imp_out, want_mass,
                                    want_imp, s.tf, s.fu);
        }
}

// ---------------------------------------------------------------------------
// The tau solve at small N_c (up to DENSE_NC) with the dense inverses of the whole
// systems: x = G f, one refinement of the streamfunction from the FP64 residual of
// the assembled band and the tau rows.  At this size a block chain is a handful of
// steps, each a string of dependent FP64 instructions on one warp (35 us a solve at
// N_c = 21, of which the chains, Schur sums and single-warp phases were 25); a
// dense apply has 2 N_c independent sums, cut into up to 6 pieces each, on every
// warp.  Column-major inverses (pInv [M][N_c][N_c] complex, tInv real, uInv): lanes of
// consecutive rows read consecutive entries.
// ---------------------------------------------------------------------------
constexpr int DENSE_GROUPS = 6;
__host__ __device__ inline int dense_groups(int nc) {
    const int g = NTHREADS_S / (2 * nc);
    return g < 1 ? 1 : g > DENSE_GROUPS ? DENSE_GROUPS : g;
}
__host__ __device__ inline size_t dense_smem_doubles(int nc) { return (size_t)nc * (12 + 4 * dense_groups(nc)); }

__global__ void __launch_bounds__(NTHREADS_S) k_solve_dense(StepParams P, RhsSpec R, DevFactors F, VecSet y_out,
                                                            VecSet mass_out, VecSet imp_out, int want_mass,
                                                            int want_imp) {
    chain_wait();
    extern __shared__ double2 sm[];
    const int nc = P.nc, n2 = 2 * nc, np = nc - 4;
    const int m = P.m_lo + blockIdx.x;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int ng = dense_groups(nc);
    double* fp = reinterpret_cast<double*>(sm);  // assembled right-hand sides (f of the zonal flow in fp for m = 0)
    double* ft = fp + n2;
    double* xp = ft + n2;  // solutions (the zonal flow's in xp for m = 0)
    double* xt = xp + n2;
    double* rp = xt + n2;  // residual, then correction
    double* xu = rp + n2;  // (m = 0) the zonal flow
    double* fu = xu + nc;
    double* red_p = fu + nc;  // [group][2 N_c] pieces of the sums
    double* red_t = red_p + ng * n2;
    const double dm = (double)m;

    // right-hand sides sum_t c_t V_t (tau rows zero)
    for (int t = tid; t < 2 * n2 + (m == 0 ? nc : 0); t += nth) {
        double acc = 0.0;
        if (t < n2) {
            if (t >= 8 && m > 0)
                for (int i = 0; i < R.nterms; ++i)
                    acc = fma(R.t[i].c, reinterpret_cast<const double*>(R.t[i].v.psi)[(size_t)m * n2 + t], acc);
            fp[t] = acc;
        } else if (t < 2 * n2) {
            const int q = t - n2;
            if (q >= 4)
                for (int i = 0; i < R.nterms; ++i)
                    acc = fma(R.t[i].c, reinterpret_cast<const double*>(R.t[i].v.th)[(size_t)m * n2 + q], acc);
            ft[q] = acc;
        } else {
            const int n = t - 2 * n2;
            if (n >= 2)
                for (int i = 0; i < R.nterms; ++i) acc = fma(R.t[i].c, R.t[i].v.u[n], acc);
            fu[n] = acc;
        }
    }
    __syncthreads();
    // pieces of G r: group g takes the columns n0 + g, n0 + g + ng, ...
    auto pieces = [&](auto&& term, int n0, double* red) {
        for (int t = tid; t < ng * n2; t += nth) {
            const int g = t / n2, q = t - g * n2;
            double acc = 0.0;
            for (int n = n0 + g; n < nc; n += ng) acc = term(q, n, acc);
            red[t] = acc;
        }
    };
    auto joined = [&](const double* red, int q) {
        double v = red[q];
        for (int g = 1; g < ng; ++g) v += red[g * n2 + q];
        return v;
    };
    const double2* gp = F.pInv + (size_t)m * nc * nc;
    const double* gt = F.tInv + (size_t)m * nc * nc;
    auto psi_term = [&](const double* r) {
        return [=](int q, int n, double acc) {
            const double2 a = __ldg(&gp[(size_t)n * nc + (q >> 1)]);
            const double o = r[2 * n + 1 - (q & 1)];
            return fma(a.x, r[2 * n + (q & 1)], fma(a.y, (q & 1) ? o : -o, acc));
        };
    };
    auto theta_term = [&](int q, int n, double acc) { return fma(__ldg(&gt[(size_t)n * nc + (q >> 1)]), ft[2 * n + (q & 1)], acc); };
    auto zonal_term = [&](int q, int n, double acc) { return q < nc ? fma(__ldg(&F.uInv[(size_t)n * nc + q]), fu[n], acc) : acc; };
    // temperature (and zonal flow); with implicit buoyancy (Section 4) its
    // g (Ra/Pr)(i m/s_o) C^I theta_new then joins the streamfunction rows
    pieces(theta_term, 2, red_t);
    if (m == 0)
        pieces(zonal_term, 2, red_p);
    else if (!P.buoy_imp)
        pieces(psi_term(fp), 4, red_p);
    __syncthreads();
    for (int q = tid; q < 2 * n2; q += nth) {
        if (q < n2) {
            if (m == 0) {
                xp[q] = 0.0;
                if (q < nc) xu[q] = joined(red_p, q);
            } else if (!P.buoy_imp) {
                xp[q] = joined(red_p, q);
            }
        } else {
            xt[q - n2] = joined(red_t, q - n2);
        }
    }
    __syncthreads();
    if (m > 0) {
        if (P.buoy_imp) {
            const double cb = F.gdt * P.Ra / P.Pr * dm / P.s_o;
            for (int q = 8 + tid; q < n2; q += nth) {
                const double v = band_part<8>(P.ops.band[OP_C], xt + ((q & 1) ^ 1), q >> 1, nc);
                fp[q] = fma((q & 1) ? cb : -cb, v, fp[q]);
            }
            __syncthreads();
            pieces(psi_term(fp), 4, red_p);
            __syncthreads();
            for (int q = tid; q < n2; q += nth) xp[q] = joined(red_p, q);
            __syncthreads();
        }
        // residual r = f - L x: the band's 17 taps in pieces; tau rows r = -tau x
        const double2* band = F.pBand + (size_t)m * np * 17;
        for (int t = tid; t < ng * n2; t += nth) {
            const int g = t / n2, q = t - g * n2, k = q >> 1;
            double acc = 0.0;
            if (k < 4) {
                for (int n = g; n < nc; n += ng) acc = fma(-__ldg(&P.ops.tau_psi[k * nc + n]), xp[2 * n + (q & 1)], acc);
            } else {
                if (g == 0) acc = fp[q];
                for (int d = g; d < 17; d += ng) {
                    const int n = k - 8 + d;
                    if (n >= 0 && n < nc)
                        acc = fms_part(acc, __ldg(&band[(size_t)(k - 4) * 17 + d]), make_double2(xp[2 * n], xp[2 * n + 1]), q & 1);
                }
            }
            red_p[t] = acc;
        }
        __syncthreads();
        for (int q = tid; q < n2; q += nth) rp[q] = joined(red_p, q);
        __syncthreads();
        pieces(psi_term(rp), 0, red_p);
        __syncthreads();
        for (int q = tid; q < n2; q += nth) xp[q] += joined(red_p, q);
        __syncthreads();
    }
    // store, then mass / implicit terms for later stages (epilogue_psi_part, epilogue_theta_part)
    for (int q = tid; q < n2; q += nth) {
        reinterpret_cast<double*>(y_out.psi)[(size_t)m * n2 + q] = xp[q];
        reinterpret_cast<double*>(y_out.th)[(size_t)m * n2 + q] = xt[q];
        if (m == 0 && q < nc) y_out.u[q] = xu[q];
    }
    if (want_mass || want_imp)
        for (int q = tid; q < 2 * n2; q += nth) {
            if (q < n2)
                epilogue_psi_part(P, R, F.gdt, m, q >> 1, q & 1, reinterpret_cast<const double2*>(xp), mass_out, imp_out,
                                  want_mass, want_imp, P.buoy_imp ? nullptr : reinterpret_cast<const double2*>(fp));
            else
                epilogue_theta_part(P, R, F.gdt, m, (q - n2) >> 1, q & 1, reinterpret_cast<const double2*>(xt), xu, mass_out,
                                    imp_out, want_mass, want_imp, reinterpret_cast<const double2*>(ft), fu);
        }
}

// ---------------------------------------------------------------------------
// The same solve split by system over two CTAs per mode (large N_c, explicit
// buoyancy): role 0 the streamfunction system, role 1 the temperature system (and,
// for m = 0, the zonal flow after it).  The streamfunctions' CTAs come first: they
// take twice as long, so the short ones fill the end of the launch.  (Interleaved,
// block 2m + role, the 152 SMs got only one role each per pass over them: 875 and 2949
// us against 780 and 2786 at 1025 x 3072 and 2049 x 6144; interleaved with the roles
// exchanged from pass to pass 858 and 2906.)  The same arithmetic as k_solve with
// fuse_t = 0.
//
// A CTA alternates between block chains (two to four walking warps, latency) and
// phases of the whole CTA (FP64 and the factors' HBM reads), so it takes several on
// an SM to keep either busy: three, by holding two vectors a system.  Chains run in
// place and the assembled right-hand side f waits in y_out, which the solution
// replaces in the end: each element of y_out is written, read and written by this
// CTA alone, first after the terms of f at that element have been read.  60 KB at
// N_c = 1365 where five vectors a system took 109 KB (two CTAs).  Bound by FP64 (43%
// of its rate) and the latency of the chains; with two CTAs an SM 3231 and 1005 us at
// n_r x n_phi = 2049 x 6144 and 1025 x 3072, with three 2949 and 875, 2834 and 770 in the
// order above, 2505 and 688 with the slimmer steps of Walk.
// ---------------------------------------------------------------------------
__host__ __device__ inline size_t solve_roles_smem_bytes(int nc) {
    const size_t b = (size_t)chain_rows(nc);
    const size_t psi = 2 * b * 16 + 4 * (size_t)ring_bytes<ddc>();          // work vector, solution
    const size_t th = 5 * b * 8 + 4 * (size_t)ring_bytes<double>();         // solution, FP32 work vector, uf, ux
    return psi > th ? psi : th;
}

template <bool DDP>
__global__ void __launch_bounds__(NTHREADS_S, 3) k_solve_roles(StepParams P, RhsSpec R, DevFactors F, VecSet y_out,
                                                                VecSet mass_out, VecSet imp_out, int want_mass,
                                                                int want_imp) {
    chain_wait();
    extern __shared__ double2 sm[];
    __shared__ double part_s[NTHREADS_S / 32][8];
    __shared__ __align__(16) double prevs[NTHREADS_S / 32][32];
    const int nc = P.nc;
    const int nm = gridDim.x >> 1, role = (int)blockIdx.x >= nm, m = P.m_lo + (int)blockIdx.x - role * nm;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31;
    const int part = tid & 1;  // the component of this thread's tasks
    const int np = nc - 4, nt = nc - 2;
    const int b = chain_rows(nc);
    auto flat = [](double2* v) { return reinterpret_cast<double*>(v); };
    SolveSmem s{};
    s.prevs = prevs;
    if (role == 0) {
        // ---------------------------------------------------- streamfunction
        if (m == 0) {  // Psi_0 = 0
            for (int n = tid; n < nc; n += nth) {
                y_out.psi[n] = make_double2(0.0, 0.0);
                if (want_mass) mass_out.psi[n] = make_double2(0.0, 0.0);
                if (want_imp) imp_out.psi[n] = make_double2(0.0, 0.0);
            }
            return;
        }
        const int nbp = (np + 7) / 8, nA = 8 * (nbp / 2);
        using C = std::conditional_t<DDP, ddc, double2>;
        using V = typename Chain<C>::V;
        double2 *work = sm, *x = sm + b, *f = y_out.psi + (size_t)m * nc;
        char* ring = reinterpret_cast<char*>(sm + 2 * b);
        const C* blk = (DDP ? reinterpret_cast<const C*>(F.pBlkDD) : reinterpret_cast<const C*>(F.pBlk)) + (size_t)m * nbp * 192;
        const ddc* spk_dd = reinterpret_cast<const ddc*>(F.pSpkDD) + (size_t)m * np * 8;
        for (int q = tid; q < 2 * nc; q += nth) {
            double acc = 0.0;
#pragma unroll 4
            for (int t = 0; t < R.nterms; ++t)
                acc = fma(R.t[t].c, reinterpret_cast<const double*>(R.t[t].v.psi)[(size_t)m * 2 * nc + q], acc);
            if (q < 8) acc = 0.0;
            flat(f)[q] = acc;
            if constexpr (DDP)
                reinterpret_cast<ddf*>(work)[q] = dd_from_bits(acc);
            else
                flat(work)[q] = acc;
        }
        __syncthreads();
        // the block in place, one or (psplit) two halves by warps 0-1 and 6-7
        auto job = [&](bool second) {
            const int n0 = second ? nA : 0, n = second ? (F.psplit ? np - nA : 0) : F.psplit ? nA : np;
            V* v = reinterpret_cast<V*>(work + 4 + n0);
            return ChainJob<C, 2>{v, v, v, n, blk + (second ? (size_t)(nbp / 2) * 192 : 0), second ? 6 : 0,
                                  ring + (second ? 2 * ring_bytes<C>() : 0)};
        };
        for (int it = 0; it < 2; ++it) {  // solve, then one refinement step
            double2* sol = it ? work : x;
            run_chains<2>(job(false), job(true), no_job<float, 2>(), no_job<double, 1>(), prevs);
            if constexpr (DDP) {
                if (F.psplit)
                    split_join_dd(reinterpret_cast<ddc*>(work) + 4, np, nA, spk_dd,
                                  reinterpret_cast<const ddc*>(F.pRjDD) + (size_t)m * 256, true);
                for (int q = 8 + tid; q < 2 * nc; q += nth) flat(sol)[q] = dd_compose(reinterpret_cast<const ddf*>(work)[q]);
            } else {
                if (F.psplit) split_join(work + 4, np, nA, F.pSpk + (size_t)m * np * 8, F.pRj + (size_t)m * 256, true);
                if (!it)
                    for (int q = 8 + tid; q < 2 * nc; q += nth) flat(x)[q] = flat(work)[q];
            }
            __syncthreads();
            rows_dot_part<4>(sol + 4, np, P.ops.tau_psi_B, part_s);
            __syncthreads();
            if (warp == 0) schur_apply<4>(sol, it ? work : nullptr, rows_dot_sum(part_s, 8), F.pSinv + (size_t)m * 16);
            __syncthreads();
            schur_update_parts<4>(sol, nc, F.pY + (size_t)m * np * 4);
            __syncthreads();
            if (it == 0) {  // residual r = f - L x over the assembled rows, and the tau rows (f = 0)
                for (int q = 8 + tid; q < 2 * nc; q += nth) {
                    const int k = q >> 1;
                    const double acc = residual_part(flat(f)[q], F.pBand + ((size_t)m * np + (k - 4)) * 17, x, k, nc, part);
                    if constexpr (DDP)
                        reinterpret_cast<ddf*>(work)[q] = dd_from_bits(acc);
                    else
                        flat(work)[q] = acc;
                }
                rows_dot_part<4>(x, nc, P.ops.tau_psi, part_s);
                __syncthreads();
                if (warp == 2) {
                    const double t = rows_dot_sum(part_s, 8);
                    if (lane < 8) flat(work)[lane] = -t;  // read by the Schur step, past the chains' barriers
                }
            }
        }
        for (int q = tid; q < 2 * nc; q += nth) flat(x)[q] += flat(work)[q];
        __syncthreads();
        for (int q = tid; q < 2 * nc; q += nth) {
            if (want_mass || want_imp)
                epilogue_psi_part(P, R, F.gdt, m, q >> 1, part, x, mass_out, imp_out, want_mass, want_imp, f);
            flat(f)[q] = flat(x)[q];
        }
        return;
    }
    // ------------------------------------------- temperature (and zonal flow)
    s.tx = sm;
    s.tr = s.td = reinterpret_cast<float2*>(sm + b);  // FP32 residual, then (in place) correction
    s.uf = reinterpret_cast<double*>(s.tr + b);
    s.ux = s.uf + b;
    s.ring_t = s.ring_u = reinterpret_cast<char*>(s.ux + b);
    s.tf = y_out.th + (size_t)m * nc;
    const int nbt = (nt + 7) / 8;
    for (int q = tid; q < 2 * nc; q += nth) {
        const int n = q >> 1;
        double acc = 0.0, au = 0.0;
#pragma unroll 4
        for (int t = 0; t < R.nterms; ++t) {
            acc = fma(R.t[t].c, reinterpret_cast<const double*>(R.t[t].v.th)[(size_t)m * 2 * nc + q], acc);
            if (m == 0) au = fma(R.t[t].c, R.t[t].v.u[n], au);
        }
        if (n < 2) acc = au = 0.0;
        flat(s.tf)[q] = acc;
        if (F.ir_t)
            reinterpret_cast<float*>(s.tr)[q] = f32_from_bits(acc);
        else
            flat(s.tx)[q] = acc;
        if (m == 0 && part == 0) s.uf[n] = au;
    }
    __syncthreads();
    if (F.ir_t) {
        theta32_chains(F, s, m, nt, nbt);
        block_schur32_dir(s.td, s.tr, nc, P.ops.tau_dir_B32, F.tSinv32 + (size_t)m * 4);
        schur_update32_dir(s.td, nc, F.tY32 + (size_t)m * nt * 2, 0, nth);
        __syncthreads();
        for (int n = tid; n < nc; n += nth) s.tx[n] = to_d2_bits(s.td[n]);
        __syncthreads();
        temperature_corrections_roles(P, F, s, m);
    } else {
        double* v = flat(s.tx + 2);
        run_chains<2>(no_job<double, 1>(), no_job<double, 1>(),
                          ChainJob<double, 2>{v, v, v, nt, F.tBlk + (size_t)m * nbt * 192, 2, s.ring_t}, no_job<double, 1>(),
                          prevs);
        rows_dot_part<2>(s.tx + 2, nt, P.ops.tau_dir_B, part_s);
        __syncthreads();
        if (warp == 0) schur_apply<2>(s.tx, nullptr, rows_dot_sum(part_s, 4), F.tSinv + (size_t)m * 4);
        __syncthreads();
        schur_update_parts<2>(s.tx, nc, F.tY + (size_t)m * nt * 2);
        __syncthreads();
    }
    if (m == 0) {
        // the zonal flow after the temperature, whose FP32 array takes the
        // refinement's correction
        s.pd = reinterpret_cast<double2*>(s.td);
        zonal_chains(F, s, s.uf + 2, s.ux + 2, nt);
        if (warp == 4) {
            double t0 = 0.0, t1 = 0.0;
            for (int j = lane; j < nt; j += 32) {
                t0 = fma(__ldg(&P.ops.tau_dir_B[j]), s.ux[2 + j], t0);
                t1 = fma(__ldg(&P.ops.tau_dir_B[nt + j]), s.ux[2 + j], t1);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t0 += __shfl_xor_sync(0xffffffffu, t0, o);
                t1 += __shfl_xor_sync(0xffffffffu, t1, o);
            }
            if (lane < 2) s.ux[lane] = -(F.uSinv[lane * 2] * t0 + F.uSinv[lane * 2 + 1] * t1);
            __syncwarp();
        }
        __syncthreads();
        {
            const double u0 = s.ux[0], u1 = s.ux[1];
            for (int j = tid; j < nt; j += nth) s.ux[2 + j] -= F.uY[(size_t)j * 2] * u0 + F.uY[(size_t)j * 2 + 1] * u1;
        }
        __syncthreads();
        if (F.ir_t) refine_zonal_flow(P, F, s);
    }
    for (int q = tid; q < 2 * nc; q += nth) {
        const int n = q >> 1;
        if (want_mass || want_imp)
            epilogue_theta_part(P, R, F.gdt, m, n, part, s.tx, s.ux, mass_out, imp_out, want_mass, want_imp, s.tf, nullptr);
        flat(s.tf)[q] = flat(s.tx)[q];
        if (m == 0 && part == 0) y_out.u[n] = s.ux[n];
    }
}

// ---------------------------------------------------------------------------
// Galerkin-basis solve (Appendix B; option "radial" = 2).  Per mode the square
// systems P_4 (A - g dt B) S_Psi x = P_4 r and P_2 (D - g dt F/Pr) S_D x = P_2 r
// (and the zonal-flow one) are solved with their banded LU factors with partial
// pivoting (host_ops.h, band_lu_pivot), then expanded to Chebyshev coefficients:
// f_hat_k = (1/(C w_k)) sum_i S(k, n) x_n.  The same discrete problem as the tau
// solve, without border rows, Schur steps or refinement.
//
// A system is solved by one warp in two sweeps of n dependent steps each.  The
// rows the next steps touch sit in a register window across the lanes:
//   forward (L, interchanges interleaved): lanes 0..KL hold b[j..j+KL]; step j
//     swaps row j with row j + piv[j], lanes 1..KL subtract l_t b_j, the window
//     shifts down one lane and lane KL takes b[j+KL+1];
//   backward (U, column by column, with U's columns divided by their diagonal
//     entries): lanes 0..KK hold y[i..i-KK]; step i takes y_i final, lanes
//     1..KK subtract (U(i-t, i)/U_ii) y_i, the window shifts; x_i = y_i / U_ii
//     is formed afterwards by the whole CTA (off the chain).
// A step's chain is two shuffles and one or two dependent FMAs; the factors are
// staged through shared memory in chunks of GCH rows by asynchronous copies, the
// next chunk in flight while the current one is used.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double shfl_down_x(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double2 shfl_down_x(double2 v) {
    return make_double2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}

// Asynchronous 16-byte global -> shared copies (cp.async): a lane's copies
// complete at cp.async.wait_group; __syncwarp then publishes them to the warp.

constexpr int GCH = 32;  // rows of factors staged per chunk

// Copy rows [r0, r1) of a row-major factor array (W entries of TF per row, W *
// sizeof(TF) a multiple of 16 bytes, the array 16-byte aligned) to dst, by one warp.
template <int W, class TF>
__device__ __forceinline__ void stage_rows(TF* dst, const TF* src, int r0, int r1) {
    constexpr int PER = W * (int)sizeof(TF) / 16;
    static_assert(PER * 16 == W * (int)sizeof(TF), "factor rows must be whole 16-byte pieces");
    const char* s = reinterpret_cast<const char*>(src + (size_t)r0 * W);
    char* d = reinterpret_cast<char*>(dst);
    for (int q = threadIdx.x & 31; q < (r1 - r0) * PER; q += 32) cp_async16(d + 16 * q, s + 16 * q);
}

// b: right-hand side (n entries, row-scaled), overwritten by the forward result;
// x: y = U_ii x_i (n entries; the caller multiplies by Uc[i][0] = 1/U_ii).
// Lm [n][KL], Uc [n][UW] (UW >= KK+1, padded to whole 16-byte rows):
// band_lu_pivot's factors; pv: the pivot offsets in shared memory.
// stg: shared staging of 2 GCH rows of Uc (which also holds 2 GCH rows of Lm):
// chunk k+1 of the factors is copied while chunk k is used.
template <int KL, int KK, int UW, class TF, class TX>
__device__ void warp_band_solve(TX* b, TX* x, int n, const TF* __restrict__ Lm, const TF* __restrict__ Uc,
                                const unsigned char* pv, TF* stg) {
    static_assert(KK < 32 && KL <= KK && UW >= KK + 1, "window wider than a warp");
    const int lane = threadIdx.x & 31;
    const bool lrow = lane >= 1 && lane <= KL, urow = lane >= 1 && lane <= KK;
    // forward: L z = P b
    TX w = (lane <= KL && lane < n) ? b[lane] : zero<TX>();
    stage_rows<KL>(stg, Lm, 0, min(n, GCH));
    cp_async_commit();
    for (int c0 = 0, k = 0; c0 < n; c0 += GCH, k ^= 1) {
        const int c1 = min(n, c0 + GCH);
        if (c1 < n) stage_rows<KL>(stg + (k ^ 1) * GCH * KL, Lm, c1, min(n, c1 + GCH));
        cp_async_commit();
        cp_async_wait1();
        __syncwarp();
        const TF* sl = stg + k * GCH * KL;
        for (int j = c0; j < c1; ++j) {
            const int p = pv[j];
            const TF l = lrow ? sl[(j - c0) * KL + lane - 1] : zero<TF>();
            const TX in = (lane == KL && j + KL + 1 < n) ? b[j + KL + 1] : zero<TX>();
            const TX bj = shfl_idx(w, p);
            const TX w0 = shfl_idx(w, 0);
            if (lane == p) w = w0;
            if (lrow) w = fms_x(l, bj, w);
            if (lane == 0) b[j] = bj;
            w = shfl_down_x(w);
            if (lane == KL) w = in;
        }
        __syncwarp();
    }
    // backward: U x = z, chunks of rows taken from the bottom
    TX v = (lane <= KK && n - 1 - lane >= 0) ? b[n - 1 - lane] : zero<TX>();
    stage_rows<UW>(stg, Uc, max(0, n - GCH), n);
    cp_async_commit();
    for (int c1 = n, k = 0; c1 > 0; c1 -= GCH, k ^= 1) {
        const int c0 = max(0, c1 - GCH);
        if (c0 > 0) stage_rows<UW>(stg + (k ^ 1) * GCH * UW, Uc, max(0, c0 - GCH), c0);
        cp_async_commit();
        cp_async_wait1();
        __syncwarp();
        const TF* su = stg + k * GCH * UW;
        for (int i = c1 - 1; i >= c0; --i) {
            const TF u = urow ? su[(i - c0) * UW + lane] : zero<TF>();
            const TX in2 = (lane == KK && i - KK - 1 >= 0) ? b[i - KK - 1] : zero<TX>();
            const TX yi = shfl_idx(v, 0);
            if (lane == 0) x[i] = yi;
            if (urow) v = fms_x(u, yi, v);
            v = shfl_down_x(v);
            if (lane == KK) v = in2;
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(NTHREADS_S) k_solve_galerkin(StepParams P, RhsSpec R, DevFactors F, VecSet y_out,
                                                               VecSet mass_out, VecSet imp_out, int want_mass,
                                                               int want_imp) {
    chain_wait();
    extern __shared__ double2 sm[];
    const int nc = P.nc, m = P.m_lo + blockIdx.x;
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5;
    const int np = nc - 4, nt = nc - 2;
    const bool has_u = (m == 0);
    const int b = round8(nc);
    double2 *pf = sm, *xp = sm + b, *px = sm + 2 * b, *tf = sm + 4 * b, *xt = sm + 5 * b, *tx = sm + 6 * b;
    double* xu = reinterpret_cast<double*>(sm + 3 * b);
    SolveSmem s{};
    s.uf = reinterpret_cast<double*>(sm + 7 * b);
    s.ux = s.uf + b;
    // after the FP64 solve arrays (over the FP32 refinement arrays of the tau
    // path, unused here): factor staging (2 GCH rows per system) and pivots
    double2* stp = sm + 8 * round8(nc);
    double* stt = reinterpret_cast<double*>(stp + 2 * GCH * 21);
    double* stu = stt + 2 * GCH * 12;
    unsigned char* pvp = reinterpret_cast<unsigned char*>(stu + 2 * GCH * 12);
    unsigned char* pvt = pvp + round8(nc);
    unsigned char* pvu = pvt + round8(nc);
    for (int n = tid; n < nt; n += nth) {
        if (n < np && m > 0) pvp[n] = F.gpPiv[(size_t)m * np + n];
        pvt[n] = F.gtPiv[(size_t)m * nt + n];
        if (has_u) pvu[n] = F.guPiv[n];
    }

    // right-hand side sum_t c_t V_t; the rows of the integrated equations
    // (k >= 4 for Psi, k >= 2 otherwise) times the row scales of the factors
    for (int n = tid; n < nc; n += nth) {
        double2 ap = make_double2(0.0, 0.0), at = make_double2(0.0, 0.0);
        double au = 0.0;
#pragma unroll 4
        for (int t = 0; t < R.nterms; ++t) {
            const double c = R.t[t].c;
            const double2 vp = R.t[t].v.psi[(size_t)m * nc + n];
            const double2 vt = R.t[t].v.th[(size_t)m * nc + n];
            ap.x = fma(c, vp.x, ap.x);
            ap.y = fma(c, vp.y, ap.y);
            at.x = fma(c, vt.x, at.x);
            at.y = fma(c, vt.y, at.y);
            if (has_u) au = fma(c, R.t[t].v.u[n], au);
        }
        pf[n] = (n < 4 || m == 0) ? make_double2(0.0, 0.0) : ap;
        tf[n] = (n < 2) ? make_double2(0.0, 0.0) : cscale(at, F.gtR[(size_t)m * nt + n - 2]);
        if (has_u) s.uf[n] = (n < 2) ? 0.0 : au * F.guR[n - 2];
    }
    __syncthreads();
    const double ic = 1.0 / P.cnorm;  // 1/(C w_k), w_0 = 1/2
    // implicit buoyancy (Section 4): temperature first, then the streamfunction
    // rows with g dt (Ra/Pr)(i m/s_o) C^I theta_new; otherwise all in one pass
    const int npass = P.buoy_imp ? 2 : 1;
    for (int pass = 0; pass < npass; ++pass) {
        const bool do_p = !P.buoy_imp || pass == 1, do_t = !P.buoy_imp || pass == 0;
        if (do_p && m > 0) {
            if (P.buoy_imp) {
                const double cb = F.gdt * P.Ra / P.Pr * (double)m / P.s_o;
                for (int k = 4 + tid; k < nc; k += nth)
                    pf[k] = cadd(pf[k], cmul_i(band_row_c<8>(P.ops.band[OP_C], tx, k, nc), cb));
                __syncthreads();
            }
            for (int k = 4 + tid; k < nc; k += nth) pf[k] = cscale(pf[k], F.gpR[(size_t)m * np + k - 4]);
            __syncthreads();
        }
        if (warp == 0) {
            if (do_p && m > 0)
                warp_band_solve<8, 20, 21>(pf + 4, xp, np, F.gpL + (size_t)m * np * 8,
                                           F.gpU + (size_t)m * np * 21, pvp, stp);
        } else if (warp == 1) {
            if (do_t)
                warp_band_solve<4, 10, 12>(tf + 2, xt, nt, F.gtL + (size_t)m * nt * 4,
                                           F.gtU + (size_t)m * nt * 12, pvt, stt);
        } else if (warp == 2) {
            if (do_t && has_u) warp_band_solve<4, 10, 12>(s.uf + 2, xu, nt, F.guL, F.guU, pvu, stu);
        }
        __syncthreads();
        // x_n = y_n / U_nn
        for (int n = tid; n < nt; n += nth) {
            if (do_p && m > 0 && n < np) xp[n] = mul(F.gpU[((size_t)m * np + n) * 21], xp[n]);
            if (do_t) {
                xt[n] = mul(F.gtU[((size_t)m * nt + n) * 12], xt[n]);
                if (has_u) xu[n] *= F.guU[(size_t)n * 12];
            }
        }
        __syncthreads();
        // expansion to f_hat: Psi_k = sum_i gamma_i^{k-i} x_{k-i}, f_k = x_{k-2} - x_k
        for (int k = tid; k < nc; k += nth) {
            const double h = (k == 0) ? 2.0 * ic : ic;
            if (do_p) {
                double2 a = make_double2(0.0, 0.0);
                if (m > 0) {
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const int n = k - i;
                        if (n >= 0 && n < np) {
                            const double g = __ldg(&F.gam[n * 5 + i]);
                            a.x = fma(g, xp[n].x, a.x);
                            a.y = fma(g, xp[n].y, a.y);
                        }
                    }
                }
                px[k] = cscale(a, h);
            }
            if (do_t) {
                double2 a = (k < nt) ? make_double2(-xt[k].x, -xt[k].y) : make_double2(0.0, 0.0);
                if (k >= 2) a = cadd(a, xt[k - 2]);
                tx[k] = cscale(a, h);
                if (has_u) s.ux[k] = h * (((k >= 2) ? xu[k - 2] : 0.0) - ((k < nt) ? xu[k] : 0.0));
            }
        }
        __syncthreads();
    }

    // store, then mass / implicit operators for later stages
    for (int n = tid; n < nc; n += nth) {
        y_out.psi[(size_t)m * nc + n] = px[n];
        y_out.th[(size_t)m * nc + n] = tx[n];
        if (has_u) y_out.u[n] = s.ux[n];
        if (want_mass || want_imp)
            epilogue_row(P, R, F.gdt, m, n, px, tx, s.ux, mass_out, imp_out, want_mass, want_imp);
    }
}

__global__ void __launch_bounds__(NTHREADS_S) k_apply(StepParams P, VecSet y, VecSet mass_out, VecSet imp_out,
                                                      int want_mass, int want_imp) {
    chain_wait();
    extern __shared__ double2 sm[];
    const int m = P.m_lo + blockIdx.x;
    const int nc = P.nc;
    double2* xp = sm;
    double2* xt = xp + nc;
    double* xu = reinterpret_cast<double*>(xt + nc);
    for (int n = threadIdx.x; n < nc; n += blockDim.x) {
        xp[n] = (m > 0) ? y.psi[(size_t)m * nc + n] : make_double2(0.0, 0.0);
        xt[n] = y.th[(size_t)m * nc + n];
        if (m == 0) xu[n] = y.u[n];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nc; k += blockDim.x) apply_row(P, m, k, xp, xt, xu, mass_out, imp_out, want_mass, want_imp);
}

// Sets *flag when any entry of the state (Psi, theta, u_bar and, for
// collocation, omega) is NaN or infinite.
__global__ void k_check_finite(VecSet y, size_t n2, int nu, int* __restrict__ flag) {
    chain_wait();
    bool bad = false;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x) {
        const double2 a = y.psi[i], b = y.th[i];
        bad |= !(isfinite(a.x) && isfinite(a.y) && isfinite(b.x) && isfinite(b.y));
        if (y.w) {
            const double2 c = y.w[i];
            bad |= !(isfinite(c.x) && isfinite(c.y));
        }
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += gridDim.x * blockDim.x) bad |= !isfinite(y.u[i]);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

}  // namespace


cudaError_t launch_solve(const StepParams& P, const RhsSpec& rhs, const DevFactors& F, VecSet y_out,
                         VecSet mass_out, VecSet imp_out, bool want_mass, bool want_imp, cudaStream_t st) {
    if (F.gal) {
        // the FP64 solve arrays (16 round8(nc) doubles), the staging of the factors
        // (double2 x 2 GCH x 21, double x 2 GCH x 12 twice) and 3 pivot rows
        const size_t smg = sizeof(double) * 16 * round8(P.nc) + sizeof(double2) * 2 * GCH * 21 +
                           sizeof(double) * 2 * 2 * GCH * 12 + 3 * round8(P.nc);
        cudaError_t err = cudaFuncSetAttribute(k_solve_galerkin, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smg);
        if (err != cudaSuccess) return err;
        return launch_chained(k_solve_galerkin, slab_modes(P), NTHREADS_S, smg, st, P, rhs, F, y_out, mass_out, imp_out,
                              want_mass ? 1 : 0, want_imp ? 1 : 0);
    }
    // small systems (N_c <= DENSE_NC): the dense inverses, 35 -> 16 us at N_c = 21.
    // Their operations and bytes grow as N_c^2: at N_c = 85 (n_r = 129) the applies
    // alone are 2300 FP64 instructions a warp and mode, 19 us of an SM's FP64 units for
    // each mode on it, where the chains take 35 us for two.  The options that pick a
    // form of the chains keep them.
    if (F.pInv && P.psi_dd < 0 && P.solve_roles <= 0 && !F.ir_t) {
        return launch_chained(k_solve_dense, slab_modes(P), NTHREADS_S, sizeof(double) * dense_smem_doubles(P.nc), st, P, rhs,
                              F, y_out, mass_out, imp_out, want_mass ? 1 : 0, want_imp ? 1 : 0);
    }
    // double-float streamfunction chains with explicit buoyancy (option psi_chain_dd),
    // by default from N_c > 64: by mode at 129 x 384 and 257 x 768 45.3 and 84.8 us with
    // FP64 ones, 35.4 and 63.0 with these
    const bool ddp = !P.buoy_imp && F.pBlkDD && (P.psi_dd > 0 || (P.psi_dd < 0 && P.nc > 64));
    // With explicit buoyancy one CTA per system or one per mode.  N_c > 600 (an
    // FP32-refined temperature): per system.  Below, per system for up to a mode an SM,
    // whose two systems then run on two SMs, and from four modes an SM on, where three
    // CTAs of two vectors an SM beat two of seven; between, the modes fit one or two
    // passes of two CTAs an SM, the systems need part of another.  Solve, us, per mode /
    // per system: n_r = 129, 257, 513 with 129 modes 35.4 / 34.2, 50.4 / 49.4, 78.8 / 71.9; with
    // 257 modes 43.1 / 51.5, 63.0 / 75.6, 112.4 / 128.9; with 513 modes 86.3 / 92.4, 132.7 /
    // 139.2, 233.4 / 224.9; with 1025 modes 173.3 / 141.3, 263.4 / 218.5, 461.4 / 369.1.  (By
    // the whole number of modes: a slab solves as the whole step does.)
    const bool per_system = P.nc > 600 || (P.nc > 64 && (P.M <= P.sms || P.M > 4 * P.sms));
    if (!P.buoy_imp && (P.solve_roles > 0 || (P.solve_roles < 0 && per_system))) {
        const size_t smr = solve_roles_smem_bytes(P.nc);
        auto kern = ddp ? k_solve_roles<true> : k_solve_roles<false>;
        cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smr);
        // three CTAs per SM need the largest shared-memory carveout
        if (err == cudaSuccess)
            err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
        if (err != cudaSuccess) return err;
        return launch_chained(kern, 2 * slab_modes(P), NTHREADS_S, smr, st, P, rhs, F, y_out, mass_out, imp_out,
                              want_mass ? 1 : 0, want_imp ? 1 : 0);
    }
    auto kern = P.buoy_imp ? (F.ir_t ? k_solve<true, false, true> : k_solve<false, false, true>)
                : F.ir_t   ? (ddp ? k_solve<true, true, false> : k_solve<true, false, false>)
                           : (ddp ? k_solve<false, true, false> : k_solve<false, false, false>);
    const size_t sm = sizeof(double) * solve_smem_doubles(P.nc, F.ir_t && P.buoy_imp);
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(kern, slab_modes(P), NTHREADS_S, sm, st, P, rhs, F, y_out, mass_out, imp_out, want_mass ? 1 : 0,
                          want_imp ? 1 : 0);
}

// acc[0] += sum_n w_n Re theta_hat_0n = Nu - 1 of the state (one warp, a fixed
// summation order: the lane sums, then a butterfly of shuffles)
__global__ void k_nusselt_accumulate(const double2* th0, const double* __restrict__ w, int nc,
                                     double* acc) {
    chain_wait();
    double t = 0.0;
    for (int n = threadIdx.x; n < nc; n += 32) t = fma(w[n], th0[n].x, t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) acc[0] += t;
}

cudaError_t launch_nusselt_accumulate(const StepParams& P, VecSet y, const double* w, double* acc,
                                      cudaStream_t st) {
    return launch_chained(k_nusselt_accumulate, 1, 32, 0, st, y.th, w, P.nc, acc);
}

cudaError_t launch_check_finite(const StepParams& P, VecSet y, int* flag, cudaStream_t st) {
    return launch_chained(k_check_finite, 152, 256, 0, st, y, (size_t)P.M * P.nc, P.nc, flag);
}

cudaError_t launch_apply(const StepParams& P, VecSet y, VecSet mass_out, VecSet imp_out, bool want_mass,
                         bool want_imp, cudaStream_t st) {
    const size_t sm = sizeof(double2) * 2 * P.nc + sizeof(double) * P.nc;
    cudaError_t err = cudaFuncSetAttribute(k_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    return launch_chained(k_apply, slab_modes(P), NTHREADS_S, sm, st, P, y, mass_out, imp_out, want_mass ? 1 : 0, want_imp ? 1 : 0);
}

}  // namespace pz
