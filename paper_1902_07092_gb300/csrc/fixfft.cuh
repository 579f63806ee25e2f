// Fixed-point Fourier transforms on the integer pipes.
//
// GB300 issues an FP64 instruction of a warp every 64 cycles per SM
// sub-partition (1.6 lane operations per clock per SM measured), 32-bit integer
// additions at about 64 and 32 x 32 -> 64 bit multiply-adds at about 25 per clock
// per SM.  A complex point held as two 64-bit integers is added in 4
// instructions and multiplied by a twiddle factor in about 18, so a radix-4
// butterfly costs ~120 integer instructions where FP64 needs 34 instructions of
// 64 cycles and double-floats ~400; the code is also short enough to stay in the
// instruction cache.  One rounding of a value x with block maximum 2^e is
// 2^(e - 60) or finer, so a transform is no worse than an FP64 one (compared with
// long double in the tests, as it is and through a Chebyshev derivative).
//
// Scaling.  Each real component of a vector is normalised by the power of two
// above its largest magnitude (|x| <= 2^60 on entry).  The first pass grows the
// magnitude by at most its radix and is not scaled.  A later radix-4 or radix-3
// pass is either scaled by 1/4 -- a twiddle product comes out as a w / 4 without
// a shift, so this costs one shift of the untwiddled point -- or, where the
// 1-norm of the vector shows that no intermediate can leave 62 bits, not scaled:
// the products are shifted back (fx_schedule).  A vector whose 1-norm is close to its
// maximum (a decaying spectrum) so keeps almost all 60 bits; a flat one loses only
// the bits its transform can grow by.
#pragma once
#include <cuda_runtime.h>

namespace pz {

#define FX_HD __host__ __device__ __forceinline__

typedef long long fx64;
struct __align__(16) fxc {
    fx64 x, y;
};
// exp(-2 pi i j/L) in units of 2^-62, each component split as hi 2^32 + lo with
// a signed lo (|lo| < 2^31)
struct __align__(16) fxw {
    int x1, x0, y1, y0;
};

constexpr int FX_BITS = 60;  // |component| <= 2^FX_BITS on entry to a transform

// The widening multiply-adds and the word accesses are written out: from plain C
// the compiler spends 40 instructions on a complex product instead of 29.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ fx64 fx_mad(int a, int b, fx64 c) {
    fx64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
__device__ __forceinline__ fx64 fx_mulw(int a, int b) {
    fx64 d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ void fx_words(fx64 a, int& h, int& l) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(a));
}
#else
inline fx64 fx_mad(int a, int b, fx64 c) { return c + (fx64)a * b; }
inline fx64 fx_mulw(int a, int b) { return (fx64)a * b; }
inline void fx_words(fx64 a, int& h, int& l) {
    l = (int)(unsigned)(unsigned long long)a;
    h = (int)(a >> 32);
}
#endif
// a = h 2^32 + l with l signed
FX_HD void fx_split(fx64 a, int& h, int& l) {
    fx_words(a, h, l);
    h += (int)((unsigned)l >> 31);
}
// a 2^-32 rounded
FX_HD fx64 fx_round32(fx64 a) {
    int h, l;
    fx_split(a, h, l);
    return (fx64)h;
}
FX_HD fxc fx_add(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
FX_HD fxc fx_sub(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }
// Shifts to the right without a preferred direction.  One that rounds down moves every
// butterfly of a pass the same way, by 3/8 of a unit (1/8 rounding halves up), and such
// a constant survives the sums of a transform and of a Chebyshev derivative, where
// unbiased roundings cancel: a derivative from 2049 grid values comes out 2.7e-11 wrong
// rounding down, 7.2e-12 with halves up, 2.3e-12 unbiased (7.0e-12 in FP64).  The radial
// transforms round so (RND); the azimuthal ones, whose spectra no sum differentiates,
// shift down (no worse than FP64 either; rounding there too, a step took 0.3 to 0.6 % more).
// a 2^-s to nearest, halves to even (s >= 1)
FX_HD fx64 fx_shr(fx64 a, int s) { return (a + ((((fx64)1 << (s - 1)) - 1) + ((a >> s) & 1))) >> s; }
// a/2 and (a + b)/2, a half to the odd neighbour: one instruction beside the shift
FX_HD fx64 fx_half(fx64 a) { return (a >> 1) | (a & 1); }
FX_HD fxc fx_half(fxc a) { return fxc{fx_half(a.x), fx_half(a.y)}; }
FX_HD fx64 fx_avg(fx64 a, fx64 b) { return ((a >> 1) + (b >> 1) + (a & b & 1)) | ((a ^ b) & 1); }
// a/2 and a/4 of the passes
template <bool RND>
FX_HD fxc fx_scale2(fxc a) {
    return RND ? fx_half(a) : fxc{a.x >> 1, a.y >> 1};
}
template <bool RND>
FX_HD fxc fx_scale4(fxc a) {
    return RND ? fxc{fx_shr(a.x, 2), fx_shr(a.y, 2)} : fxc{a.x >> 2, a.y >> 2};
}
FX_HD fxc fx_shl2(fxc a) {
    return fxc{(fx64)((unsigned long long)a.x << 2), (fx64)((unsigned long long)a.y << 2)};
}

// a w / 4.  The four cross products of a component (below 2^63 together for
// |a| <= 2^62.5) are summed and rounded to 2^32 before they join the leading
// products; the products of the two low words are left out (below 2^-1 units).
FX_HD fxc fx_mul4(fxc a, fxw w) {
    int xh, xl, yh, yl;
    fx_split(a.x, xh, xl);
    fx_split(a.y, yh, yl);
    const int ny1 = -w.y1, ny0 = -w.y0;
    const fx64 c = fx_mad(yl, ny1, fx_mad(xl, w.x1, fx_mad(yh, ny0, fx_mulw(xh, w.x0))));
    const fx64 d = fx_mad(yl, w.x1, fx_mad(xl, w.y1, fx_mad(yh, w.x0, fx_mulw(xh, w.y0))));
    return fxc{fx_mad(yh, ny1, fx_mad(xh, w.x1, fx_round32(c))), fx_mad(yh, w.x1, fx_mad(xh, w.y1, fx_round32(d)))};
}

// a c for a real constant c = hi 2^-30 + lo 2^-62 (split as a twiddle), to the last place
FX_HD fx64 fx_mulc(fx64 a, int hi, int lo) {
    int h, l;
    fx_split(a, h, l);
    const fx64 c = fx_mad(l, hi, fx_mulw(h, lo));
    return (fx64)((unsigned long long)fx_mulw(h, hi) << 2) + ((c + ((fx64)1 << 29)) >> 30);
}
// sqrt(3)/2 and sqrt(1/2)
#define FX_H3_1 929887697
#define FX_H3_0 (-1332128537)
#define FX_R2_1 759250125
#define FX_R2_0 (-25716447)

// One butterfly t < L/R of a pass over one vector (src, dst of length L).
// q: log2 of the sub-transform length Ns before the pass.  Forward transform
// sum_j x_j exp(-2 pi i j k / L); the backward one is the forward transform of the
// vector with its components exchanged, components exchanged again.
FX_HD void fx_bfly4(fxc v0, fxc v1, fxc v2, fxc v3, fxc& o0, fxc& o1, fxc& o2, fxc& o3) {
    const fxc t0 = fx_add(v0, v2), t1 = fx_sub(v0, v2), t2 = fx_add(v1, v3), t3 = fx_sub(v1, v3);
    const fxc r = fxc{t3.y, -t3.x};  // -i t3
    o0 = fx_add(t0, t2);
    o2 = fx_sub(t0, t2);
    o1 = fx_add(t1, r);
    o3 = fx_sub(t1, r);
}
// Place of entry i in the buffer between the first and the second pass: the first
// pass writes runs of 4 or 8 entries a thread, which fall on the same shared-memory
// banks (4- and 8-way conflicts) unless the position within eight entries is
// exchanged by the index of the eight.
FX_HD int fx_swz(int i) { return i ^ ((i >> 3) & 7); }
FX_HD void fx_first4(const fxc* src, fxc* dst, int quarter, int t) {
    fxc o0, o1, o2, o3;
    fx_bfly4(src[t], src[t + quarter], src[t + 2 * quarter], src[t + 3 * quarter], o0, o1, o2, o3);
    const int x = (t >> 1) & 7;
    dst[(4 * t) ^ x] = o0;
    dst[(4 * t + 1) ^ x] = o1;
    dst[(4 * t + 2) ^ x] = o2;
    dst[(4 * t + 3) ^ x] = o3;
}
// radix 8 as the first pass (L = 8^a 4^b with an odd log2): two 4-point transforms of
// the even and the odd points, halved, and one radix-2 level.  Scaled by 1/2.
template <bool RND>
FX_HD void fx_first8(const fxc* src, fxc* dst, int eighth, int t) {
    fxc e0, e1, e2, e3, o0, o1, o2, o3;
    fx_bfly4(src[t], src[t + 2 * eighth], src[t + 4 * eighth], src[t + 6 * eighth], e0, e1, e2, e3);
    fx_bfly4(src[t + eighth], src[t + 3 * eighth], src[t + 5 * eighth], src[t + 7 * eighth], o0, o1, o2, o3);
    e0 = fx_scale2<RND>(e0);
    e1 = fx_scale2<RND>(e1);
    e2 = fx_scale2<RND>(e2);
    e3 = fx_scale2<RND>(e3);
    o0 = fx_scale2<RND>(o0);
    o1 = fx_scale2<RND>(o1);
    o2 = fx_scale2<RND>(o2);
    o3 = fx_scale2<RND>(o3);
    // o1 (1 - i)/sqrt 2, o2 (-i), o3 (-1 - i)/sqrt 2
    o1 = fxc{fx_mulc(o1.x + o1.y, FX_R2_1, FX_R2_0), fx_mulc(o1.y - o1.x, FX_R2_1, FX_R2_0)};
    o2 = fxc{o2.y, -o2.x};
    o3 = fxc{fx_mulc(o3.y - o3.x, FX_R2_1, FX_R2_0), -fx_mulc(o3.x + o3.y, FX_R2_1, FX_R2_0)};
    const int x = t & 7;
    fxc* d = dst + 8 * t;
    d[0 ^ x] = fx_add(e0, o0);
    d[1 ^ x] = fx_add(e1, o1);
    d[2 ^ x] = fx_add(e2, o2);
    d[3 ^ x] = fx_add(e3, o3);
    d[4 ^ x] = fx_sub(e0, o0);
    d[5 ^ x] = fx_sub(e1, o1);
    d[6 ^ x] = fx_sub(e2, o2);
    d[7 ^ x] = fx_sub(e3, o3);
}
#ifdef __CUDA_ARCH__
FX_HD fxw fx_ldw(const fxw* p) {
    const int4 v = __ldg(reinterpret_cast<const int4*>(p));
    return fxw{v.x, v.y, v.z, v.w};
}
#else
FX_HD fxw fx_ldw(const fxw* p) { return *p; }
#endif
// twstep: stride of the twiddle table times L / (4 Ns)
template <bool RND>
FX_HD void fx_pass4(const fxc* src, fxc* dst, int quarter, int q, const fxw* tw, int twstep, bool back, bool swz, int t) {
    const int k = t & ((1 << q) - 1);
    const int i0 = k * twstep;
    const int p0 = swz ? fx_swz(t) : t, p1 = swz ? fx_swz(t + quarter) : t + quarter;
    const int p2 = swz ? fx_swz(t + 2 * quarter) : t + 2 * quarter, p3 = swz ? fx_swz(t + 3 * quarter) : t + 3 * quarter;
    fxc v0 = src[p0];
    fxc v1 = fx_mul4(src[p1], fx_ldw(tw + i0));
    fxc v2 = fx_mul4(src[p2], fx_ldw(tw + 2 * i0));
    fxc v3 = fx_mul4(src[p3], fx_ldw(tw + 3 * i0));
    if (back) {
        v1 = fx_shl2(v1);
        v2 = fx_shl2(v2);
        v3 = fx_shl2(v3);
    } else {
        v0 = fx_scale4<RND>(v0);
    }
    fxc o0, o1, o2, o3;
    fx_bfly4(v0, v1, v2, v3, o0, o1, o2, o3);
    fxc* d = dst + (((t >> q) << (q + 2)) + k);
    d[0] = o0;
    d[1 << q] = o1;
    d[2 << q] = o2;
    d[3 << q] = o3;
}
// the last pass of a length 3 * 2^p (azimuthal): sub-transforms of length third = L/3
FX_HD void fx_pass3(const fxc* src, fxc* dst, int third, const fxw* tw, int tws, bool back, bool swz, int t) {
    const int p1 = t + third, p2 = t + 2 * third;
    fxc v0 = src[swz ? fx_swz(t) : t];
    fxc v1 = fx_mul4(src[swz ? fx_swz(p1) : p1], fx_ldw(tw + t * tws));
    fxc v2 = fx_mul4(src[swz ? fx_swz(p2) : p2], fx_ldw(tw + 2 * t * tws));
    if (back) {
        v1 = fx_shl2(v1);
        v2 = fx_shl2(v2);
    } else {
        v0 = fx_scale4<false>(v0);
    }
    const fxc s = fx_add(v1, v2), e = fx_sub(v1, v2);
    const fxc m = fx_sub(v0, fx_scale2<false>(s));
    const fxc r = fxc{fx_mulc(e.y, FX_H3_1, FX_H3_0), -fx_mulc(e.x, FX_H3_1, FX_H3_0)};  // -i (sqrt 3/2) e
    dst[t] = fx_add(v0, s);
    dst[t + third] = fx_add(m, r);
    dst[t + 2 * third] = fx_sub(m, r);
}

// Passes of a transform of length (three ? 3 : 1) << lg (lg >= 2): radix 8 first when
// lg is odd, else radix 4; radix 4; then radix 3.
FX_HD int fx_passes(int lg, bool three) { return lg / 2 + (three ? 1 : 0); }

// Which passes are not scaled (bit p of the result) and the bits S lost by the whole
// transform (the outputs hold X 2^-S), for inputs with components up to
// 2^FX_BITS and 1-norm (sum of |re| + |im|) below 2^l1.  Every intermediate of
// the transform is at most the 1-norm and at most the growth of its passes times
// the largest input.
FX_HD unsigned fx_schedule(int lg, bool three, int l1, int& S) {
    const int np = fx_passes(lg, three);
    int grown = FX_BITS + ((lg & 1) ? 3 : 2);
    unsigned back = 0;
    S = (lg & 1) ? 1 : 0;
    for (int p = 1; p < np; ++p) {
        grown += 2;
        if ((grown < l1 ? grown : l1) - S > 62)
            S += 2;
        else
            back |= 1u << p;
    }
    return back;
}

#ifdef __CUDACC__
// v 2^(FX_BITS - e) rounded, for |v| < 2^e with e = emax - 1022 given through the
// biased exponent emax of the block maximum; zero for emax = 0 (a zero or subnormal
// block) or a subnormal v.  The exponent moves on the integer pipe; the conversion
// issues once on the FP64 pipe (64 cycles of a sub-partition, against about 24 integer
// instructions, and 40 for fx_to).
__device__ __forceinline__ fx64 fx_from(double v, int emax) {
    const int h = __double2hiint(v), s = FX_BITS + 1022 - emax;
    const int E = (h >> 20) & 0x7ff;
    const fx64 r = __double2ll_rn(__hiloint2double(h + (s << 20), __double2loint(v)));
    return (E == 0 || E + s <= 0) ? 0 : r;
}
// a 2^ex as a double, rounded to nearest; 0 below the normal range, infinity above it;
// NaN for a bad block (an infinity or NaN in it)
__device__ __forceinline__ double fx_to(fx64 a, int ex, bool bad) {
    const double d = __ll2double_rn(a);
    int h = __double2hiint(d);
    const int E = ((h >> 20) & 0x7ff) + ex;
    int l = __double2loint(d);
    h += ex << 20;
    if (a == 0 || E <= 0) h = l = 0;
    if (E >= 2047 && a != 0) {
        h = (a < 0) ? 0xfff00000 : 0x7ff00000;
        l = 0;
    }
    if (bad) h = 0x7ff80000;
    return __hiloint2double(h, l);
}
// biased exponent of |v|
__device__ __forceinline__ unsigned fx_exponent(double v) { return ((unsigned)__double2hiint(v) >> 20) & 0x7ffu; }

// nb transforms stored contiguously in a (each L = (three ? 3 : 1) << lg), b scratch
// of the same size, both in dynamic shared memory; back[i] the schedule of vector
// i.  Whole CTA; begins and ends with __syncthreads(); returns the buffer holding
// the result.  Not inlined, with the buffers as offsets into shared memory (so
// that they are read and written as such): one copy of the passes serves every
// transform of a kernel and stays in the instruction cache.
extern __shared__ __align__(16) fxc fx_shared[];
template <bool RND>
__device__ __noinline__ int fx_fft_off(int a, int b, const fxw* __restrict__ tw, int tws, int lg, bool three, int nb,
                                       const unsigned* back) {
    const int L = (three ? 3 : 1) << lg;
    const int tid = threadIdx.x, nth = blockDim.x;
    // bit 8 i + p: pass p of vector i is not scaled (at most four vectors of eight passes)
    unsigned bk = 0u;
    __syncthreads();
    for (int i = 0; i < nb; ++i) bk |= back[i] << (8 * i);
    {
        const int n = (lg & 1) ? L >> 3 : L >> 2;
        for (int u = tid; u < nb * n; u += nth) {
            const int i = three ? (u >= n) : u >> (lg - ((lg & 1) ? 3 : 2));  // (three: at most two vectors)
            const fxc* s = fx_shared + (a + i * L);
            fxc* d = fx_shared + (b + i * L);
            if (lg & 1)
                fx_first8<RND>(s, d, n, u - i * n);
            else
                fx_first4(s, d, n, u - i * n);
        }
    }
    const int n = L >> 2;
    int p = 1;
    for (int q = (lg & 1) ? 3 : 2; q < lg; q += 2, ++p) {
        __syncthreads();
        const int x = a;
        a = b;
        b = x;
        const int twstep = (L >> (q + 2)) * tws;
        for (int u = tid; u < nb * n; u += nth) {
            const int i = three ? (u >= n) : u >> (lg - 2);
            fx_pass4<RND>(fx_shared + (a + i * L), fx_shared + (b + i * L), n, q, tw, twstep, (bk >> (8 * i + p)) & 1u, p == 1,
                          u - i * n);
        }
    }
    if (three) {
        __syncthreads();
        const int x = a;
        a = b;
        b = x;
        for (int u = tid; u < nb << lg; u += nth) {
            const int i = u >> lg;
            fx_pass3(fx_shared + (a + i * L), fx_shared + (b + i * L), 1 << lg, tw, tws, (bk >> (8 * i + p)) & 1u, p == 1,
                     u & ((1 << lg) - 1));
        }
    }
    __syncthreads();
    return b;
}
template <bool RND>
__device__ __forceinline__ fxc* fx_fft(fxc* a, fxc* b, const fxw* __restrict__ tw, int tws, int lg, bool three, int nb,
                                       const unsigned* back) {
    return fx_shared + fx_fft_off<RND>((int)(a - fx_shared), (int)(b - fx_shared), tw, tws, lg, three, nb, back);
}
#endif

}  // namespace pz
