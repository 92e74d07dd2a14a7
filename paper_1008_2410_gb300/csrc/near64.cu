// near64.cu -- Fig. 1 stage 9 in the plain form: the near field of Eq. 6 in (at least) FP64 accuracy.
//
// GB300 has 2 FP64 multiply-adds per SM and clock against 128 in FP32 and 30 wide (32 x 32 -> 64) integer ones, so
// the pairs run in 64-bit fixed point on the integer pipe: coordinates as integers in units of 2^-60 of a leaf's width
// (FP64 positions exactly, but for those within 2^-7 widths of a coordinate axis: differences carry no other rounding
// error), products from three wide multiplications each, sums in 64-bit integers.
//   * r > sqrt(75) sigma (x = r^2 / 2 sigma^2 > 37.5): 1 - e^-x is 1 in FP64 and the pair is the point vortex
//     gamma (-dy, dx) / r^2, with 1 / r^2 by one Newton step of second order from the SFU's FP32 reciprocal.
//   * closer pairs go to a list per thread (index in shared memory) and run once the list is full or the sources are
//     done, every lane with a pair of its own: F(x) = (1 - e^-x) / x from a table of polynomials of degree 5 (no
//     exponential, no division). Where nearly every adjacent pair is close, all take this path, without the list.
// A block whose charges span a wide range (so that a fixed unit could lose digits of a small sum) or that has few
// sources runs all pairs in FP64, with a table of polynomials of degree 6; so do close pairs in leaves wider than about
// 100 sigma. A target whose sums turn out small against the fixed unit (its velocity is that of weak charges among strong
// ones without weight there, or of particles much closer together than sigma) is summed in FP64 instead.
#include <math.h>

#include <mutex>

#include "near64.cuh"

namespace fmm {

namespace {

constexpr double kTwoPi = 6.283185307179586476925;

// ------------------------------------------------------------------ table of F(x) = (1 - e^-x) / x

// Row i: the polynomial in t = x - c, c = (i + 1/2) / 16, that interpolates F on [i / 16, (i + 1) / 16) at Chebyshev
// nodes, truncated to degree 6 (its error there is below (1/32)^7 / (2^6 7! 8) = 2e-17), then c itself. x < 37.5.
constexpr int kTabN = 600;
constexpr double kXCut = N64_XCUT;
__device__ double2 g_blob_f[kTabN * 4], g_blob_d[kTabN * 4];  // F and F'

// Double-double numbers for the tables, h + l with |l| <= ulp(h) / 2 (Knuth's two-sum, products by fma): about 2^-102 relative.
struct DD {
    double h, l;
};
__device__ __forceinline__ DD dd_fast(double a, double b)  // |a| >= |b|
{
    const double s = __dadd_rn(a, b);
    return {s, __dadd_rn(b, -__dadd_rn(s, -a))};
}
__device__ __forceinline__ DD operator+(DD a, DD b)
{
    const double s = __dadd_rn(a.h, b.h), t = __dadd_rn(s, -a.h);
    const double e = __dadd_rn(__dadd_rn(a.h, -__dadd_rn(s, -t)), __dadd_rn(b.h, -t));
    return dd_fast(s, __dadd_rn(e, __dadd_rn(a.l, b.l)));
}
__device__ __forceinline__ DD operator-(DD a) { return {-a.h, -a.l}; }
__device__ __forceinline__ DD operator*(DD a, DD b)
{
    const double p = __dmul_rn(a.h, b.h), e = __fma_rn(a.h, b.h, -p);
    return dd_fast(p, __fma_rn(a.h, b.l, __fma_rn(a.l, b.h, e)));
}
__device__ __forceinline__ DD operator/(DD a, DD b)
{
    const double q = a.h / b.h;
    const DD r = a + -(b * DD{q, 0.0});
    return dd_fast(q, r.h / b.h);
}
__device__ __forceinline__ DD scaled(DD a, int k) { return {ldexp(a.h, k), ldexp(a.l, k)}; }
__device__ __forceinline__ long long rounded(DD a)
{
    const long long i = __double2ll_rn(a.h);
    return i + __double2ll_rn(__dadd_rn(__dadd_rn(a.h, -(double)i), a.l));
}

__device__ DD dd_cos(DD x)  // by its Taylor series; |x| <= pi / 2
{
    const DD x2 = x * x;
    DD s = {1.0, 0.0};
    for (int k = 28; k >= 2; k -= 2)
        s = DD{1.0, 0.0} + -(x2 * s / DD{(double)(k * (k - 1)), 0.0});
    return s;
}

__device__ DD dd_exp_neg(DD x)  // e^-x, 0 <= x < 128: the Taylor series at x / 4096, squared twelve times
{
    const DD t = scaled(x, -12);
    DD s = {1.0, 0.0};
    for (int k = 14; k >= 1; --k)
        s = DD{1.0, 0.0} + -(t * s / DD{(double)k, 0.0});
    for (int k = 0; k < 12; ++k)
        s = s * s;
    return s;
}

// F(x) = (1 - e^-x) / x = sum_k (-x)^k / (k+1)!, or F'(x) = ((1 + x) e^-x - 1) / x^2 = sum_k (-1)^(k+1) (k+1) x^k / (k+2)!:
// the series below x = 1.5.
__device__ DD blob_value(bool derivative, DD x)
{
    const DD one = {1.0, 0.0};
    if (x.h < 1.5) {
        DD s = {0.0, 0.0};
        for (int k = 36; k >= 0; --k)  // s = c_k - x s / (k + 2 or 3), c_k = 1 or k + 1
            s = DD{derivative ? k + 1.0 : 1.0, 0.0} + -(x * s / DD{k + (derivative ? 3.0 : 2.0), 0.0});
        return derivative ? scaled(-s, -1) : s;
    }
    const DD e = dd_exp_neg(x);
    return derivative ? ((one + x) * e + -one) / (x * x) : (one + -e) / x;
}

// The same functions for the fixed point on [0, 128): rows of degree-5 polynomials of F and of -F' in u = (x - c) / h
// about the row's centre c. Below x = 8 the rows are 1 / 64 wide, above it twice as wide from octave to octave (256 rows
// each): interpolation error below 2^-59. 32 bytes: c0 2^62, c1 2^64, c2 2^66 (50 bits, |c5| 2^58 above them), c3 2^56,
// c4 2^58. Both functions are completely monotone, so the signs alternate: c2 > 0 > c5.
constexpr int kFixN = 1536;
__device__ int4 g_fix_f[kFixN * 2], g_fix_d[kFixN * 2];

// cos(pi m / 32) from its values for m <= 16.
__device__ DD cosine(const DD *cosines, int m)
{
    m &= 63;
    m = m > 32 ? 64 - m : m;
    return m > 16 ? -cosines[32 - m] : cosines[m];
}

// Sixteen threads per row of the four tables, one per Chebyshev node: the interpolant of F or F' about c at the nodes
// c + h cos(pi (2 j + 1) / 32), truncated to degree 6 (5), as a polynomial in t / h, |t| <= h. Filled once per process and
// device, in 0.33 ms (in long double on the host, which Arm has in software, they took 0.7 s of every first call).
constexpr int kRows = 2 * (kTabN + kFixN);
__constant__ signed char c_cheb[7][7] = {{1}, {0, 1}, {-1, 0, 2}, {0, -3, 0, 4}, {1, 0, -8, 0, 8}, {0, 5, 0, -20, 0, 16}, {-1, 0, 18, 0, -48, 0, 32}};
__global__ void __launch_bounds__(64) k_near64_tables()  // grid: kRows / 4
{
    __shared__ DD cosines[17], val[4][16], coef[4][7], mono[4][7];
    if (threadIdx.x < 17)
        cosines[threadIdx.x] = dd_cos(DD{3.141592653589793116, 1.2246467991473532e-16} * DD{threadIdx.x / 32.0, 0.0});
    __syncthreads();
    const int sub = threadIdx.x >> 4, j = threadIdx.x & 15, row = 4 * blockIdx.x + sub;
    const bool derivative = row & 1, fixed = row >= 2 * kTabN;
    const int i = (row >> 1) - (fixed ? kTabN : 0), deg = fixed ? 5 : 6;
    const int o = i < 512 ? 0 : (i >> 8) - 1;  // fixed: octave [4 2^o, 8 2^o) for i >= 256
    const double c = fixed ? ldexp((i - 256 * o + 0.5) / 64.0, o) : (i + 0.5) / 16.0;
    const double h = fixed ? ldexp(1.0 / 128.0, o) : 1.0 / 32.0;
    val[sub][j] = blob_value(derivative, DD{c, 0.0} + DD{h, 0.0} * cosine(cosines, 2 * j + 1));
    __syncthreads();
    if (j <= deg) {
        DD a = {0.0, 0.0};
        for (int n = 0; n < 16; ++n)
            a = a + val[sub][n] * cosine(cosines, j * (2 * n + 1));
        coef[sub][j] = scaled(a, j == 0 ? -4 : -3);
    }
    __syncthreads();
    if (j <= deg) {
        DD a = {0.0, 0.0};
        for (int k = deg; k >= j; --k)
            a = a + coef[sub][k] * DD{(double)c_cheb[k][j], 0.0};
        mono[sub][j] = fixed && derivative ? -a : a;
    }
    __syncthreads();
    if (j != 0)
        return;
    const DD *a = mono[sub];
    if (!fixed) {
        double v[8];
        for (int m = 0; m <= 6; ++m)
            v[m] = ldexp(a[m].h, 5 * m);  // t in place of t / h
        v[7] = c;
        for (int m = 0; m < 4; ++m)
            (derivative ? g_blob_d : g_blob_f)[4 * i + m] = make_double2(v[2 * m], v[2 * m + 1]);
    } else {
        const long long c0 = rounded(scaled(a[0], 62)), c1 = rounded(scaled(a[1], 64)),
                        c2 = rounded(scaled(a[2], 66)) | (rounded(scaled(-a[5], 58)) << 50);
        int4 *r = (derivative ? g_fix_d : g_fix_f) + 2 * i;
        r[0] = make_int4((int)c0, (int)(c0 >> 32), (int)c1, (int)(c1 >> 32));
        r[1] = make_int4((int)c2, (int)(c2 >> 32), (int)rounded(scaled(a[3], 56)), (int)rounded(scaled(a[4], 58)));
    }
}

std::mutex g_tab_mu;
bool g_tab_ready[64];
const double2 *g_tab_f[64];  // device address of g_blob_f

// ------------------------------------------------------------------ fixed point

// round(v * 2^-k) modulo 2^64.
__device__ __forceinline__ long long to_fixed(double v, int k)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int be = (int)((b >> 52) & 0x7ff);
    const unsigned long long m = (b & 0xfffffffffffffull) | (be ? 1ull << 52 : 0ull);
    const int sh = max(be, 1) - 1075 - k;
    unsigned long long r;
    if (sh >= 0)
        r = sh < 64 ? m << sh : 0ull;
    else
        r = sh > -64 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull;
    return (long long)((b >> 63) ? 0ull - r : r);
}

// X = h 2^31 + l with |l| <= 2^30 (h modulo 2^32): differences of two such numbers are formed limb by limb, without
// a carry.
__device__ __forceinline__ int2 limbs31(long long X)
{
    const unsigned long long s = (unsigned long long)X + (1ull << 30);
    return make_int2((int)(s >> 31), (int)(s & 0x7fffffffu) - (1 << 30));
}

__device__ __forceinline__ long long wide(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long wide_u(unsigned a, unsigned b) { return (unsigned long long)a * b; }
__device__ __forceinline__ int hi_of(long long v) { return (int)(v >> 32); }
__device__ __forceinline__ unsigned lo_of(long long v) { return (unsigned)v; }
// Signed limbs of a 64-bit number in base 2^32: v = h 2^32 + l, l = the low word read as signed.
__device__ __forceinline__ int hi_bal(long long v) { return (int)(v >> 32) + (int)(lo_of(v) >> 31); }

// Near-field geometry of one target leaf: its source rows, contiguous runs of the sorted particles (rows iy - 1, iy,
// iy + 1 of columns ix - 1 .. ix + 1).
struct Rows64 {
    int a[3], pre[4];  // first particle of row k, prefix of the rows' counts
    __device__ __forceinline__ Rows64(const Work &w, const SysDev &d, int leaf)
    {
        const int L = d.depth, ns = 1 << L, local = leaf - (int)d.leaf0;
        const int ix = local & (ns - 1), iy = local >> L;
        const int jx0 = ix > 0 ? ix - 1 : 0, jx1 = ix < ns - 1 ? ix + 1 : ns - 1;
        pre[0] = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int row = iy + k - 1;
            int n = 0;
            a[k] = 0;
            if (row >= 0 && row < ns) {
                a[k] = w.start[d.leaf0 + row * ns + jx0];
                n = w.start[d.leaf0 + row * ns + jx1 + 1] - a[k];
            }
            pre[k + 1] = pre[k] + n;
        }
    }
    __device__ __forceinline__ int global(int q) const
    {
        int g = a[0] + q;
        g = q >= pre[1] ? a[1] + (q - pre[1]) : g;
        return q >= pre[2] ? a[2] + (q - pre[2]) : g;
    }
};

constexpr int N64_THREADS = 256;
constexpr int N64_TILE = 640;   // sources staged at a time
constexpr int N64_CAP = 48;     // close pairs listed per thread before they are run
constexpr int N64_SPILL = 96;   // terms a 64-bit sum holds: 96 * 2^56.2 < 2^63
constexpr int N64_CSPILL = 16;  // close terms a 64-bit sum holds: 16 * 2^59 at most
constexpr int N64_FEW = 96;     // fewer sources than this run in FP64
// The smallest e with every charge of the neighbourhood below 2^e (1 - 2^-12), or kNoFixed where the fixed point is not
// for them: where the sum of the charges' squares, the largest left out, is below a quarter of the largest one's. A
// term's rounding is about 0.3 2^-54 of a term of the largest charge, an FP64 sum of N such terms of size V takes about
// sqrt(N) 2^-55 V, and V may leave out the target's own charge, so that from there on the fixed point is no worse for a
// target that the large charges act on (the others: see the kernels' ends).
// Subnormal, infinite and NaN charges run in FP64. b, if given, is a second array of charges of the same kind.
// Block-uniform (integer sums, so the choice is the same in every run).
constexpr int kNoFixed = -1000000;
struct Stats64 {
    unsigned max, sum;
};
__device__ __forceinline__ int charge_exponent(const Rows64 &R, int ntot, const double *__restrict__ a,
                                               const double *__restrict__ b, Stats64 &st)
{
    const int tid = threadIdx.x;
    auto mag = [&](int q) {  // high word of |charge|: the exponent and 20 bits
        const int j = R.global(q);
        const unsigned h = (unsigned)__double2hiint(a[j]) & 0x7fffffffu;
        return b ? max(h, (unsigned)__double2hiint(b[j]) & 0x7fffffffu) : h;
    };
    __syncthreads();
    if (tid == 0)
        st.max = st.sum = 0;
    __syncthreads();
    unsigned gm = 0;
    for (int q = tid; q < ntot; q += blockDim.x)
        gm = max(gm, mag(q));
    gm = __reduce_max_sync(0xffffffffu, gm);
    if ((tid & 31) == 0)
        atomicMax(&st.max, gm);
    __syncthreads();
    gm = st.max;
    const int ge = (int)(gm >> 20);  // biased exponent of the largest charge
    if (ge <= 100 || ge == 0x7ff)
        return kNoFixed;
    unsigned sum = 0;  // of (charge / 2^ge)^2 2^18; enough is enough at 2^20
    for (int q = tid; q < ntot && sum < (1u << 20); q += blockDim.x) {
        const unsigned h = mag(q), v = (((h & 0xfffffu) | 0x100000u) >> 6) >> min(ge - (int)(h >> 20), 31);
        sum += (v * v) >> 10;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((tid & 31) == 0)
        atomicAdd(&st.sum, sum);
    __syncthreads();
    const unsigned big = ((gm & 0xfffffu) | 0x100000u) >> 6, big2 = (big * big) >> 10;
    if (st.sum < big2 + big2 / 4)
        return kNoFixed;
    return ge - 1022 + ((gm & 0xfffffu) < 0xfff00u ? 0 : 1);
}

// Far pair at displacement (dxh 2^31 + dxl, dyh 2^31 + dyl): r2 = r^2 2^-62.
__device__ __forceinline__ long long r2_fixed(int dxh, int dxl, int dyh, int dyl)
{
    // the high products and the cross terms 2 h l 2^-31
    const long long cr = wide(dyh, dyl, wide(dxh, dxl, 0));
    return wide(dyh, dyh, wide(dxh, dxh, cr >> 30));
}
// 2^116 / r2 for a high word of r2 in [N64_RMIN, 2^31): the SFU's seed y0 ~ 2^84 / r2; r2 y0 = 2^84 (1 + e) modulo
// 2^64 with |e| < 2^-21, and 1 / (1 + e) = 1 - e + e^2 to 2^-63. Any other r2 gives an arbitrary value.
__device__ __forceinline__ long long recip_fixed(long long r2)
{
    const int rh = hi_of(r2);
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__int2float_rn(rh) + 0.5f));
    const unsigned y0 = __float2uint_rn(yf * 0x1p52f);
    const unsigned long long P = wide_u(lo_of(r2), y0);
    const int eh = (int)((unsigned)(P >> 32) + (unsigned)rh * y0);
    const int es = eh >> 15;
    const unsigned e2 = (unsigned)es * (unsigned)es;  // e^2 2^74
    // c = e^2 - e with 84 fraction bits; y0 2^32 (1 + c)
    const long long c = (long long)(((unsigned long long)e2 << 10) -
                                    (((unsigned long long)(unsigned)eh << 32) | (unsigned)P));
    const long long T = wide(hi_of(c), (int)y0, (long long)(unsigned long long)__umulhi(lo_of(c), y0));
    return (long long)((unsigned long long)(T >> 20) + ((unsigned long long)y0 << 32));
}
// Rounded high half of (ah 2^32 + al) (bh 2^32 + bl), limbs signed.
__device__ __forceinline__ long long mul_hi(int ah, int al, int bh, int bl)
{
    return wide(ah, bh, (long long)hi_of(wide(al, bh, wide(ah, bl, 1ll << 31))));
}

// Close pairs in fixed point: displacements D = dx 2^s (at most 2^62, s >= 1) as signed limbs, D = x 2^32 + y.
__device__ __forceinline__ int2 close_limbs(int h, int l, int s)
{
    const long long t = wide(l, 1 << s, 0);
    return make_int2(hi_bal(t) + (h << (s - 1)), (int)lo_of(t));
}
// z = x 2^56 from r2 = r^2 2^-64, or -1 beyond the tables
__device__ __forceinline__ long long z_close(const Near64 &c, long long r2)
{
    const long long v = mul_hi(hi_bal(r2), (int)lo_of(r2), c.kmh, c.kml);
    return hi_of(v) >= c.vmax ? -1 : v << c.e;
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }  // normal range only
// r^2 2^-64 of a displacement (X, Y).
__device__ __forceinline__ long long r2_close(int2 X, int2 Y)
{
    return wide(X.x, X.x, wide(Y.x, Y.x, wide(X.x, X.y, wide(Y.x, Y.y, 1 << 30)) >> 31));
}
__device__ __forceinline__ long long square_hi(int2 X)
{
    return wide(X.x, X.x, wide(X.x, X.y, 1 << 30) >> 31);
}
// v (h 2^32 + l) / 2^55, to its last bit.
__device__ __forceinline__ long long mul_55(long long v, int h, int l)
{
    const int vh = hi_bal(v), vl = (int)lo_of(v);
    return (wide(vh, h, 0) << 9) + (wide(vl, h, wide(vh, l, (long long)__mulhi(vl, l) + (1 << 22))) >> 23);
}
// The share of z that a part of r2 gives (a square or a product of displacements), to its last bit (e < 32).
__device__ __forceinline__ long long scale_z(const Near64 &c, long long v)
{
    const int h = hi_bal(v), l = (int)lo_of(v);
    return (wide(h, c.kmh, 0) << c.e) + (wide(l, c.kmh, wide(h, c.kml, (long long)__mulhi(l, c.kml))) >> (32 - c.e));
}
// F 2^62 (or -F' 2^62) at z = x 2^56 < 2^63.
__device__ __forceinline__ long long blob_fixed(const int4 *__restrict__ tab, long long z)
{
    const int o = max(5 - __clz(hi_of(z)), 0);  // octave: 0 below x = 8, then x in [4 2^o, 8 2^o)
    const int i = (hi_of(z) >> (18 + o)) + 256 * o;
    const int4 a = __ldg(tab + 2 * i), b = __ldg(tab + 2 * i + 1);
    const long long U = (long long)(((unsigned long long)z << (14 - o)) ^ 0x8000000000000000ull) >> 1;  // u 2^62
    const int uh = hi_bal(U), ul = (int)lo_of(U);
    const int e4 = b.w - (__mulhi(uh, (int)((unsigned)b.y >> 18) << 2));
    const int e3 = b.z + __mulhi(uh, e4);
    const long long c2 = ((long long)(b.y & 0x3ffff) << 32) | (unsigned)b.x;
    const long long e2 = c2 + (wide(uh, e3, 1 << 19) >> 20);
    const long long e1 = (((long long)a.w << 32) | (unsigned)a.z) + mul_hi(uh, ul, hi_bal(e2), (int)lo_of(e2));
    return (((long long)a.y << 32) | (unsigned)a.x) + mul_hi(uh, ul, hi_bal(e1), (int)lo_of(e1));
}

// Passes over a leaf of c targets: the number of passes (at most 2 more than needed) that keeps most of the 256
// threads busy, threads = (targets of the pass) x (source groups).
__device__ __forceinline__ int pick_passes(int c)
{
    const int np0 = (c + N64_THREADS - 1) / N64_THREADS;
    int best = np0, bs = 0;
    for (int np = np0; np < np0 + 3; ++np) {
        const int cp = (c + np - 1) / np;
        const int used = N64_THREADS / cp * c / np;  // busy threads of an average pass
        if (used > bs + 8) {
            bs = used;
            best = np;
        }
    }
    return best;
}

// Sums of 64-bit sums, one per thread: 96 bits, carried in shared memory (a conversion to FP64 and an addition on that
// pipe cost as much as half a pair).
// big: the largest magnitude that a sum has had when it was marked, in units of 2^32 (to 2^-24 of it or 2^8; 0 only if it
// was always zero).
struct Acc64 {
    unsigned long long lo[N64_THREADS];
    int hi[N64_THREADS];
    float big[N64_THREADS];
    __device__ __forceinline__ void clear(int t) { lo[t] = 0, hi[t] = 0, big[t] = 0.0f; }
    __device__ __forceinline__ void mark(int t)
    {
        const unsigned long long l = lo[t];
        const int h = hi[t];
        big[t] = fmaxf(big[t], fmaxf(fabsf(fmaf((float)h, 0x1p32f, (float)(unsigned)(l >> 32))), (l | (unsigned)h) ? 1.0f : 0.0f));
    }
    __device__ __forceinline__ void add(int t, long long v)
    {
        const unsigned long long a = lo[t], b = a + (unsigned long long)v;
        lo[t] = b;
        hi[t] += (int)(v >> 63) + (b < a ? 1 : 0);
    }
    __device__ __forceinline__ void add(int t, long long h, long long l)  // h 2^24 + l
    {
        const unsigned long long a = lo[t], b = a + ((unsigned long long)h << 24), d = b + (unsigned long long)l;
        lo[t] = d;
        hi[t] += (int)(h >> 40) + (b < a ? 1 : 0) + (int)(l >> 63) + (d < b ? 1 : 0);
    }
    __device__ __forceinline__ void meet(int t, const Acc64 &o) { big[t] = fmaxf(big[t], o.big[t]); }
    __device__ __forceinline__ float biggest(int t, int step, int n) const  // of threads t, t + step, ...
    {
        float m = big[t];
#pragma unroll 4
        for (int k = 1; k < n; ++k)
            m = fmaxf(m, big[t + k * step]);
        return m;
    }
    // the sum over threads t, t + step, ... (n of them), as FP64
    __device__ __forceinline__ double total(int t, int step, int n) const
    {
        unsigned long long a = 0;
        int h = 0;
        for (int k = 0; k < n; ++k) {
            const unsigned long long b = a + lo[t + k * step];
            h += hi[t + k * step] + (b < a ? 1 : 0);
            a = b;
        }
        return fma((double)(h + (int)(a >> 63)), 0x1p64, (double)(long long)a);
    }
};
// v, without the compiler's knowledge that it is the same in every pass: what is derived from it is not kept in registers
// through the loops over the sources (in the adjoint 3% of the kernel).
__device__ __forceinline__ int fresh(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}
constexpr size_t N64_SMEM = N64_TILE * 24 + 4 * sizeof(Acc64) + N64_CAP * N64_THREADS * 2;

// The line below which a target's far and near sums are too small: the larger of those of the kinds that take part.
__device__ __forceinline__ float line_of(float far, float near, float far_line, float near_line)
{
    const bool none = far == 0.0f && near == 0.0f;
    return fmaxf(far != 0.0f || none ? far_line : 0.0f, near != 0.0f || none ? near_line : 0.0f);
}

// Source j in FP64: au, av in units of k2.
__device__ __forceinline__ void near_pair(const Work &w, int j, double xt, double yt, double k2, double &au, double &av)
{
    const double ax = xt - w.sx[j], ay = yt - w.sy[j];
    const double x = fma(ax, ax, ay * ay) * k2;
    double f = x < kXCut ? blob_poly(g_blob_f, blob_row(x), x) : recip64(x);
    // a particle and itself, or coincident ones: nothing, whatever the charge
    f = __double_as_longlong(x) != 0 ? f * w.sg[j] : 0.0;
    au = fma(-ay, f, au);
    av = fma(ax, f, av);
}

// The sum of v over the block, added in a fixed order; for thread 0. red: 2 x 8 values.
__device__ __forceinline__ double block_sum(double v, double *red)
{
#pragma unroll
    for (int o = 16; o; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // red is free
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < N64_THREADS / 32; ++i)
            v += red[i];
    return v;
}

// Persistent blocks take units from a counter: a leaf, or one of `parts` shares of a leaf's targets (launch_near64). Thread =
// (target t, source group g of G): a pass's targets run over the threads, and the groups take the sources in turn; the
// groups' sums of a target are added at the end in a fixed order.
// Measured at 2^20 uniform particles (leaves of 64, 16 sigma wide): 39.0 ms with every pair by expm1 and a division
// in FP64, 3.25 ms so, issue and integer pipes about 65 % busy. The error of the near field against quad precision fell
// from 8.6e-16 to 1.9e-16 relative L2 (integer differences and sums).
// Line of the fixed point: fewer than 96 sources in the neighbourhood have no time in it (4 to 24 particles a leaf
// agree to 2.5e-16 either way).
__global__ void __launch_bounds__(N64_THREADS, 4) k_near64(Work w, int parts)
{
    __shared__ int s_leaf, s_weak;
    __shared__ float2 s_line;
    extern __shared__ __align__(16) unsigned char sm[];  // N64_SMEM bytes
    int4 *pos = reinterpret_cast<int4 *>(sm);                        // x and y limbs
    int2 *gam = reinterpret_cast<int2 *>(pos + N64_TILE);            // gamma limbs, base 2^32
    Acc64 *acc = reinterpret_cast<Acc64 *>(gam + N64_TILE);          // far u, far v, close u, close v
    unsigned short *lst = reinterpret_cast<unsigned short *>(acc + 4);
    __shared__ Stats64 st;
    const int tid = threadIdx.x;
    for (;;) {
    if (tid == 0)
        s_leaf = atomicAdd(&w.cnt[w.nleaf + 1], 1);
    __syncthreads();
    const int leaf = s_leaf / parts, part = s_leaf - leaf * parts;
    __syncthreads();
    if (leaf >= w.nleaf)
        return;
    int s0 = w.start[leaf], c = w.start[leaf + 1] - s0;
    {  // this unit's share of the leaf's targets
        const int a = (int)((long long)part * c / parts), b = (int)((long long)(part + 1) * c / parts);
        s0 += a;
        c = b - a;
    }
    if (c == 0)
        continue;
    const int k = w.nsys == 1 ? 0 : find_sys_by_leaf(w.sys, w.nsys, leaf);
    const SysDev &d = w.sys[k];
    const Rows64 R(w, d, leaf);
    const int ntot = R.pre[3];
    const Near64 cl = near64_of(d);
    const double k2 = cl.k2;
    const int ku = cl.ku, thr = cl.thr;
    const bool ranges = cl.ranges;
    bool fixed = ranges && ntot >= N64_FEW;
    const int ge = fixed ? charge_exponent(R, ntot, w.sg, nullptr, st) : kNoFixed;
    fixed = ge != kNoFixed;
    const int ka = ge - 63;  // charges in units of 2^ka: below 2^63 - 2^50, so that their high limb fits
    if (tid == 0 && fixed) {  // cs / fs and the close sums' line (see the sums' end): here for the registers' sake
        const float ratio = cl.lim ? (float)(k2 * pow2(117 - cl.s + 2 * ku)) : 0.0f;
        s_line = make_float2(ratio, ratio * (cl.s > 3 ? 0x1p20f : 0x1p19f));  // s > 3: positions next to an axis (2^(s - 3) units)
    }

    const int npass = pick_passes(c);
    for (int pass = 0; pass < npass; ++pass) {
        const int t0 = (int)((long long)pass * c / npass), cp = (int)((long long)(pass + 1) * c / npass) - t0;
        const int G = N64_THREADS / cp;
        const int grp = tid / cp, tpos = s0 + t0 + (tid - grp * cp);
        const bool active = grp < G;
        const double xt = w.sx[tpos], yt = w.sy[tpos];
        double au = 0.0, av = 0.0;    // FP64 pairs: sums of gamma F(x) (-dy, dx), in units of k2
        for (int q = 0; q < 4; ++q)
            acc[q].clear(tid);        // pairs in fixed point
        auto pair64 = [&](int q) { near_pair(w, R.global(q), xt, yt, k2, au, av); };
        if (!ranges) {
            if (active)
                for (int q = grp; q < ntot; q += G) {
                    const int j = R.global(q);
                    const double ax = xt - w.sx[j], ay = yt - w.sy[j], r2 = ax * ax + ay * ay;
                    if (r2 > 0.0) {
                        const double f = -expm1(-r2 * k2) / r2 * w.sg[j];
                        au -= ay * f;
                        av += ax * f;
                    }
                }
        } else if (!fixed) {
            double tu = 0.0, tv = 0.0;
            for (int q = grp, i = 0; active && q < ntot; q += G) {
                pair64(q);
                if (++i % 32 == 0) {  // sums of 32 terms, then their sum
                    tu += au;
                    tv += av;
                    au = av = 0.0;
                }
            }
            au += tu;
            av += tv;
        } else {
            const int2 tx = limbs31(to_fixed(xt, ku)), ty = limbs31(to_fixed(yt, ku));
            int cnt = 0, terms = 0, cterms = 0;
            long long su = 0, sv = 0, wu = 0, wv = 0;
            auto close = [&](int q0, int q) {
                const int4 p = pos[q];
                const int2 g = gam[q];
                const int dxh = tx.x - p.x, dyh = ty.x - p.z;
                const int2 X = close_limbs(dxh, tx.y - p.y, cl.s), Y = close_limbs(dyh, ty.y - p.w, cl.s);
                const long long z = z_close(cl, r2_close(X, Y));
                if (max(abs(dxh), abs(dyh)) >= cl.lim || z < 0) {  // leaves so wide that far pairs are listed too
                    pair64(q0 + q);
                    return;
                }
                const long long F = blob_fixed(g_fix_f, z);
                const long long f = mul_hi(g.x, g.y, hi_bal(F), (int)lo_of(F));
                const int fh = hi_bal(f), fl = (int)lo_of(f);
                wu += mul_hi(fh, fl, Y.x, Y.y);
                wv += mul_hi(fh, fl, X.x, X.y);
            };
            auto spill_close = [&]() {
                acc[2].add(tid, wu);
                acc[3].add(tid, wv);
                wu = wv = 0;
            };
            for (int q0 = 0; q0 < ntot; q0 += N64_TILE) {
                const int m = min(N64_TILE, ntot - q0);
                if (q0 > 0)
                    for (int q = 0; q < 4; ++q)
                        acc[q].mark(tid);
                __syncthreads();
                for (int q = tid; q < m; q += N64_THREADS) {
                    const int j = R.global(q0 + q);
                    const int2 lx = limbs31(to_fixed(w.sx[j], ku)), ly = limbs31(to_fixed(w.sy[j], ku));
                    const long long g = to_fixed(w.sg[j], ka);
                    pos[q] = make_int4(lx.x, lx.y, ly.x, ly.y);
                    gam[q] = make_int2(hi_bal(g), (int)lo_of(g));
                }
                __syncthreads();
                const int nj = active ? (m - grp + G - 1) / G : 0;  // this thread's sources: grp, grp + G, ...
                const int nmax = __reduce_max_sync(0xffffffffu, nj);
                if (thr == 0) {  // every pair is close
                    for (int i = 0; i < nj; ++i) {
                        close(q0, grp + G * i);
                        if (i % N64_CSPILL == N64_CSPILL - 1)
                            spill_close();
                    }
                    spill_close();
                    continue;
                }
                for (int i0 = 0; i0 < nmax;) {
                    // as many sources as the fullest list of the warp still takes
                    const int used = __reduce_max_sync(0xffffffffu, cnt);
                    const int i1 = min(nmax, i0 + N64_CAP - used);
                    const int ie = min(i1, nj);
#pragma unroll 2
                    for (int i = i0; i < ie; ++i) {
                        const int q = grp + G * i;
                        const int4 p = pos[q];
                        int2 g = gam[q];
                        const int dxh = tx.x - p.x, dxl = tx.y - p.y, dyh = ty.x - p.z, dyl = ty.y - p.w;
                        const long long r2 = r2_fixed(dxh, dxl, dyh, dyl);
                        if (hi_of(r2) < thr) {
                            lst[cnt * N64_THREADS + tid] = (unsigned short)q;
                            ++cnt;
                            g = make_int2(0, 0);
                        }
                        const long long Y = recip_fixed(r2);
                        const long long f = mul_hi(g.x, g.y, hi_bal(Y), (int)lo_of(Y));  // gamma Y 2^-64
                        const int fh = hi_bal(f), fl = (int)lo_of(f) >> 1;
                        su += wide(fh, dyh, wide(fl, dyh, wide(fh, dyl, 1ll << 30)) >> 31);
                        sv += wide(fh, dxh, wide(fl, dxh, wide(fh, dxl, 1ll << 30)) >> 31);
                    }
                    terms += i1 - i0;
                    if (terms > N64_SPILL - N64_CAP) {
                        acc[0].add(tid, su);
                        acc[1].add(tid, sv);
                        su = sv = 0;
                        terms = 0;
                    }
                    i0 = i1;
                    const int full = __reduce_max_sync(0xffffffffu, cnt);
                    if (full > N64_CAP - 12 || (i0 >= nmax && full > 0)) {
                        for (int e = 0; e < full; ++e)
                            if (e < cnt)
                                close(q0, lst[e * N64_THREADS + tid]);
                        cnt = 0;
                        cterms += full;  // here F D is at most 0.64 sqrt(2) / 12.2 2^124: 96 terms fit, as for far pairs
                        if (cterms > N64_SPILL - N64_CAP) {
                            spill_close();
                            cterms = 0;
                        }
                    }
                }
            }
            acc[0].add(tid, su);
            acc[1].add(tid, sv);
            spill_close();
            for (int q = 0; q < 4; ++q)
                acc[q].mark(tid);
            acc[0].meet(tid, acc[1]);
            acc[2].meet(tid, acc[3]);
        }
        // sums of a target's groups, in order; the FP64 pairs' through the (now idle) source limbs
        double2 *red = reinterpret_cast<double2 *>(pos);
        if (tid == 0)
            s_weak = 0;
        const bool some64 = __syncthreads_or(au != 0.0 || av != 0.0);
        if (some64) {
            red[tid] = make_double2(au, av);
            __syncthreads();
        }
        if (tid < cp) {
            const int ng = min(G, ntot);  // groups with sources
            double u = 0.0, v = 0.0;
            for (int g = 0; some64 && g < ng; ++g) {
                const double2 a = red[tid + g * cp];
                u += a.x;
                v += a.y;
            }
            if (ranges) {
                u *= k2;
                v *= k2;
            }
            if (fixed) {
                // a far term is gamma dx / r^2 2^(51 + ku - ka), a close one gamma F dx 2^(s - 66 - ku - ka)
                const int kq = fresh(ku);
                const double gs = pow2(fresh(ka)), fs = pow2(-51 - kq), cs = k2 * pow2(66 - cl.s + kq);
                // A term's rounding is about 0.4 of its unit (fs or cs, times gs) however small the term is, in FP64 it is
                // relative to it: a target whose sums are all small against the unit, because the strong sources have no
                // weight there, is left to FP64 below. At this line the error is a few times that of FP64 sums. What counts is the
                // largest that a sum has been at the tiles' ends, so that a velocity that is small by cancellation does not count.
                const float far = acc[0].biggest(tid, cp, ng), near = acc[2].biggest(tid, cp, ng);
                const float line = line_of(far, near, 0x1p19f, s_line.y);
                if (fmaxf(far, near * s_line.x) < line && (!some64 || fmax(fabs(u), fabs(v)) < line * 0x1p32 * fs * gs))
                    lst[atomicAdd(&s_weak, 1)] = (unsigned short)tid;
                u -= fma(acc[2].total(tid, cp, ng), cs, acc[0].total(tid, cp, ng) * fs) * gs;
                v += fma(acc[3].total(tid, cp, ng), cs, acc[1].total(tid, cp, ng) * fs) * gs;
            }
            w.near64[tpos] = make_double2(u / kTwoPi, v / kTwoPi);
        }
        __syncthreads();
        const int nweak = s_weak;
        for (int e = 0; e < nweak; ++e) {  // the whole block on each weak target
            const int t = s0 + t0 + lst[e];
            const double xw = w.sx[t], yw = w.sy[t];
            double bu = 0.0, bv = 0.0;
            for (int q = tid; q < ntot; q += N64_THREADS)
                near_pair(w, R.global(q), xw, yw, k2, bu, bv);
            bu = block_sum(bu, &red->x);
            bv = block_sum(bv, &red->x);
            if (tid == 0)
                w.near64[t] = make_double2(bu * k2 / kTwoPi, bv * k2 / kTwoPi);
        }
        if (nweak > 0)
            __syncthreads();
    }
    }
}

// ------------------------------------------------------------------ adjoint

__device__ __forceinline__ unsigned position_hash(double x, double y)  // the same for 0 and -0
{
    const unsigned long long a = (unsigned long long)__double_as_longlong(x), b = (unsigned long long)__double_as_longlong(y);
    const unsigned ah = (a << 1) ? (unsigned)(a >> 32) : 0u, bh = (b << 1) ? (unsigned)(b >> 32) : 0u;
    return (((unsigned)a * 0x9e3779b1u + ah) * 0x85ebca77u + (unsigned)b) * 0xc2b2ae3du + bh;
}

// A particle of the adjoint, and its pair with source j in FP64: g (dgamma), x and y (dx, dy) in units of k2.
struct Adj64 {
    double x, y, g, gu, gv;
    __device__ __forceinline__ Adj64(const Work &w, int t) : x(w.sx[t]), y(w.sy[t]), g(w.sg[t]), gu(w.sgu[t]), gv(w.sgv[t]) {}
    __device__ __forceinline__ void pair(const Work &w, int j, double k2, double &ag, double &ax, double &ay) const
    {
        const double a = x - w.sx[j], b = y - w.sy[j];
        const double r2 = fma(a, a, b * b), xx = r2 * k2;
        if (__double_as_longlong(r2) == 0)
            return;  // a particle and itself, or coincident ones: K and its Jacobian count as zero
        double f, h;     // f / k2 and 2 f' / k2
        if (xx < kXCut) {
            const int i = blob_row(xx);
            f = blob_poly(g_blob_f, i, xx);
            h = 2.0 * k2 * blob_poly(g_blob_d, i, xx);
        } else {
            f = recip64(xx);
            h = -2.0 * k2 * (f * f);
        }
        const double gj = w.sg[j], guj = w.sgu[j], gvj = w.sgv[j];
        const double ah = a * h, bh = b * h, ab = a * bh;
        const double J2 = fma(a, ah, f), J1 = fma(b, bh, f);  // dKv/da, -dKu/db; dKv/db = -dKu/da = ab
        const double cu = gj * gu - g * guj, cv = gj * gv - g * gvj;
        ag = fma(f, guj * b - gvj * a, ag);
        ax += fma(cv, J2, -cu * ab);  // one rounding at the size of the sum
        ay += fma(cv, ab, -cu * J1);
    }
};

// For target k and neighbour m (z = (a, b) = z_k - z_m), with K = (Ku, Kv) = (-b, a) f of Eq. 6 and its Jacobian J:
//   dgamma_k += -(gu_m Ku + gv_m Kv) = f (gu_m b - gv_m a)
//   dx_k     += cu dKu/da + cv dKv/da,  cu = gamma_m gu_k - gamma_k gu_m
//   dy_k     += cu dKu/db + cv dKv/db,  cv = gamma_m gv_k - gamma_k gv_m
// (K is odd and its Jacobian even in z). The same split as the forward kernel's. A far pair has f = 1 / r^2 and, with
// P = 2 a b / r^4 and Q = (b^2 - a^2) / r^4, contributes cu P + cv Q to dx and cu Q - cv P to dy: 54 wide integer
// multiplications in fixed point (22 operations in FP64, several times the time); sums in two 64-bit parts, high
// products and cross terms. A close one takes F and -F' from their tables, 86 wide multiplications (37 operations in
// FP64). Measured at 2^20 uniform particles (leaves of 64, 16 sigma wide): 103 ms with exp, expm1 and divisions in FP64
// for every pair; the whole adjoint (near field beside both sweeps) 108 ms then, 8.9 ms now. 104 to 128 registers keep
// the sweeps' blocks out (11.6 to 12.0 ms), 80 spill (10.9). Errors against quad precision are below the former ones.
// Writes the near part in caller order (the far part is added later). Targets for whom the fixed unit is too coarse, or
// with coincident particles, are listed in slot (free after the binning) and summed in FP64 at the end.
constexpr int A64_REGS = 96, A64_B = 2;  // registers a thread, blocks an SM: room for the sweep's blocks beside them
constexpr int A64_TILE = 640;
constexpr int A64_CAP = 48;  // terms between two hand-overs to the 96-bit sums
constexpr size_t A64_SMEM = A64_TILE * 40 + 6 * sizeof(Acc64) + A64_CAP * N64_THREADS * 2;

// The near part of target t in FP64, by the whole block.
__device__ __noinline__ void adjoint_block64(const Work &w, int t, double *red, double *odg, double *odx, double *ody)
{
    const int leaf = w.sleaf[t], i = w.perm[t];
    const SysDev &d = w.sys[w.nsys == 1 ? 0 : find_sys_by_leaf(w.sys, w.nsys, leaf)];
    const Rows64 R(w, d, leaf);
    const double k2 = near64_of(d).k2;
    const Adj64 me(w, t);
    double ag = 0.0, ax = 0.0, ay = 0.0;
    for (int q = threadIdx.x; q < R.pre[3]; q += N64_THREADS)
        me.pair(w, R.global(q), k2, ag, ax, ay);
    ag = block_sum(ag, red);
    ax = block_sum(ax, red);
    ay = block_sum(ay, red);
    if (threadIdx.x == 0) {
        if (odg)
            odg[i] = ag * k2 / kTwoPi;
        if (odx)
            odx[i] = ax * k2 / kTwoPi;
        if (ody)
            ody[i] = ay * k2 / kTwoPi;
    }
}

__global__ void __maxnreg__(A64_REGS) k_adjoint_near64(const __grid_constant__ Work w, int parts, double *__restrict__ odg,
                                                                                double *__restrict__ odx,
                                                                                double *__restrict__ ody, int skip_plain)
{
    extern __shared__ __align__(16) unsigned char sm[];  // A64_SMEM bytes
    int4 *pos = reinterpret_cast<int4 *>(sm);                // x and y limbs
    int4 *ggr = pos + A64_TILE;                              // gu and gv limbs
    int2 *gam = reinterpret_cast<int2 *>(ggr + A64_TILE);    // gamma limbs, base 2^32
    Acc64 *acc = reinterpret_cast<Acc64 *>(gam + A64_TILE);  // dgamma, dx, dy of the far pairs, of the close ones
    unsigned short *lst = reinterpret_cast<unsigned short *>(acc + 6);
    __shared__ Stats64 st;
    __shared__ int s_leaf, s_weak;  // s_weak: head of the block's list of weak targets, linked by slot
    __shared__ float4 s_line;
    const int tid = threadIdx.x;
    if (skip_plain && w.nsys == 1 && !(w.sys[0].s_unit > P2P_SPLIT_S))
        return;  // the only system's near field is the FP32 kernel's
    if (tid == 0)
        s_weak = -1;
    for (;;) {
    if (tid == 0)
        s_leaf = atomicAdd(&w.cnt[w.nleaf + 1], 1);
    __syncthreads();
    const int leaf = s_leaf / parts, part = s_leaf - leaf * parts;
    __syncthreads();
    if (leaf >= w.nleaf)
        break;
    int s0 = w.start[leaf], c = w.start[leaf + 1] - s0;
    {  // this unit's share of the leaf's targets
        const int a = (int)((long long)part * c / parts), b = (int)((long long)(part + 1) * c / parts);
        s0 += a;
        c = b - a;
    }
    if (c == 0)
        continue;
    const int k = w.nsys == 1 ? 0 : find_sys_by_leaf(w.sys, w.nsys, leaf);
    const SysDev &d = w.sys[k];
    if (skip_plain && !(d.s_unit > P2P_SPLIT_S))
        continue;  // this system's near field is the FP32 kernel's
    const Rows64 R(w, d, leaf);
    const int ntot = R.pre[3];
    const Near64 cl = near64_of(d);
    const double k2 = cl.k2;
    const int ku = cl.ku, thr = cl.thr;
    const bool ranges = cl.ranges;
    bool fixed = ranges && ntot >= N64_FEW;
    int ka = 0, kb = 0;  // units 2^ka of gamma (below 2^62), 2^kb of gu and gv (below 2^58)
    if (fixed) {
        const int ea = charge_exponent(R, ntot, w.sg, nullptr, st);
        const int eb = ea != kNoFixed ? charge_exponent(R, ntot, w.sgu, w.sgv, st) : kNoFixed;
        fixed = eb != kNoFixed;
        ka = ea - 62;
        kb = eb - 58;
        if (tid == 0) {  // cg / fg, the close sums' line, cx / fx, the line (see the sums' end)
            const float axis = cl.s > 3 ? 2.0f : 1.0f;
            const float rg = cl.lim ? (float)(k2 * pow2(121 - cl.s + 2 * ku)) : 0.0f;
            const float rx = cl.lim ? (float)(k2 * pow2(112 + 2 * ku)) : 0.0f;
            s_line = make_float4(rg, axis * rg * (thr ? 0x1p38f : 0x1p41f), rx, axis * rx * (thr ? 0x1p38f : 0x1p40f));
        }
    }
    const int npass = pick_passes(c);
    for (int pass = 0; pass < npass; ++pass) {
        const int t0 = (int)((long long)pass * c / npass), cp = (int)((long long)(pass + 1) * c / npass) - t0;
        const int G = N64_THREADS / cp;
        const int grp = tid / cp, tpos = s0 + t0 + (tid - grp * cp);
        const bool active = grp < G;
        const Adj64 me(w, tpos);
        const double xt = me.x, yt = me.y, gt = me.g, gut = me.gu, gvt = me.gv;
        for (int q = 0; q < 6; ++q)
            acc[q].clear(tid);
        int tau = 0;
        double ag = 0.0, ax = 0.0, ay = 0.0;  // FP64 pairs: dgamma in units of k2, dx and dy in units of k2
        auto pair64 = [&](int q) { me.pair(w, R.global(q), k2, ag, ax, ay); };
        if (!ranges) {
            if (active)
                for (int q = grp; q < ntot; q += G) {
                    const int j = R.global(q);
                    const double a = xt - w.sx[j], b = yt - w.sy[j], s = a * a + b * b;
                    if (s == 0.0)
                        continue;
                    const double e = exp(-s * k2), om = -expm1(-s * k2);
                    const double f = om / s, fp = (k2 * e * s - om) / (s * s);
                    const double cu = w.sg[j] * gut - gt * w.sgu[j], cv = w.sg[j] * gvt - gt * w.sgv[j];
                    ag += f * (w.sgu[j] * b - w.sgv[j] * a);
                    ax += cv * (f + 2.0 * a * a * fp) - cu * (2.0 * a * b * fp);
                    ay += cv * (2.0 * a * b * fp) - cu * (f + 2.0 * b * b * fp);
                }
        } else if (!fixed) {
            double tg = 0.0, tx = 0.0, ty = 0.0;
            for (int q = grp, i = 0; active && q < ntot; q += G) {
                pair64(q);
                if (++i % 32 == 0) {  // sums of 32 terms, then their sum
                    tg += ag;
                    tx += ax;
                    ty += ay;
                    ag = ax = ay = 0.0;
                }
            }
            ag += tg;
            ax += tx;
            ay += ty;
        } else {
            const int2 tx = limbs31(to_fixed(xt, ku)), ty = limbs31(to_fixed(yt, ku));
            // cu and cv are linear in the target's charges: scaled up together, so that a weak target keeps its digits
            const int te = max(exponent_of(gt) - (ka + 61), max(exponent_of(gut), exponent_of(gvt)) - (kb + 57));
            tau = te < -900 ? 0 : -te;
            // Coincident particles (whose Jacobian counts as zero) are of one leaf. Looking for them here, by hashes of the
            // positions, costs nothing that shows; a test in the loop over the close pairs 2.5% of the kernel.
            unsigned *hash = reinterpret_cast<unsigned *>(lst);
            constexpr int kHashes = A64_CAP * N64_THREADS / 2;
            const unsigned mine = position_hash(xt, yt);
            bool same = false;
            const int own = fresh(leaf), own1 = w.start[own + 1];
            for (int h0 = w.start[own]; h0 < own1; h0 += kHashes) {
                const int m = min(kHashes, own1 - h0);
                if (h0 > w.start[own])
                    __syncthreads();
                for (int j = tid; j < m; j += N64_THREADS)
                    hash[j] = position_hash(w.sx[h0 + j], w.sy[h0 + j]);
                __syncthreads();
                for (int j = active ? grp : m; j < m; j += G)
                    same |= hash[j] == mine && h0 + j != tpos;
            }
            if (same)
                acc[0].big[tid] = INFINITY;
            const long long tg = to_fixed(gt, ka - tau), tgu = to_fixed(gut, kb - tau), tgv = to_fixed(gvt, kb - tau);
            const int tgh = -hi_bal(tg), tgl = (int)lo_of(tg) >> 1;  // low limb halved: it can be negated
            const int tuh = hi_bal(tgu), tul = (int)lo_of(tgu), tvh = hi_bal(tgv), tvl = (int)lo_of(tgv);
            int cnt = 0;
            long long hg = 0, lg = 0, hx = 0, lx = 0, hy = 0, ly = 0;  // high products, cross terms / 2^8
            auto spill = [&](Acc64 *a) {  // units of 2^40
                a[0].add(tid, hg, lg);
                a[1].add(tid, hx, lx);
                a[2].add(tid, hy, ly);
                hg = lg = hx = lx = hy = ly = 0;
            };
            // listed pairs beyond x = 40 in FP64: J falls as 1 / x, and few closer ones may be there to outweigh it
            const int vmax = (thr ? cl.vmax / 3 : cl.vmax) - 2;
            // cu, cv / 2^64 of a source: gamma_m gu_k - gamma_k gu_m; the target's negated limbs are (tgh, -2 tgl)
            auto cross = [&](int2 g, int gh, int gl, int th, int tl) {
                return wide(g.x, th, wide(tgh, gh, (long long)hi_of(wide(g.y, th, wide(g.x, tl, 1ll << 31)) +
                                                                    wide(tgh, gl, -2 * wide(tgl, gh, 0)))));
            };
            // dx += cu A + cv B, dy += cu C + cv D, with the low halves' products (the range of the terms takes up
            // most of the high ones)
            auto grad = [&](long long cu, long long cv, long long A, long long B, long long C, long long D) {
                const int cuh = hi_bal(cu), cul = (int)lo_of(cu), cvh = hi_bal(cv), cvl = (int)lo_of(cv);
                const int Ah = hi_bal(A), Al = (int)lo_of(A), Bh = hi_bal(B), Bl = (int)lo_of(B);
                hx = wide(cuh, Ah, wide(cvh, Bh, hx));
                lx += wide(cuh, Al, wide(cul, Ah, wide(cvh, Bl, wide(cvl, Bh, (long long)__mulhi(cul, Al) + __mulhi(cvl, Bl))))) >> 8;
                const int Ch = hi_bal(C), Cl = (int)lo_of(C), Dh = hi_bal(D), Dl = (int)lo_of(D);
                hy = wide(cuh, Ch, wide(cvh, Dh, hy));
                ly += wide(cuh, Cl, wide(cul, Ch, wide(cvh, Dl, wide(cvl, Dh, (long long)__mulhi(cul, Cl) + __mulhi(cvl, Dl))))) >> 8;
            };
            // a close pair: with alpha^2 = a^2 k2 and so on, in units of k2,
            //   J = dKv/da = F - 2 alpha^2 H, -dKu/db = F - 2 beta^2 H, dKv/db = -dKu/da = -2 alpha beta H, H = -F'
            auto close = [&](int q0, int q) {
                const int4 p = pos[q];
                const int dxh = tx.x - p.x, dyh = ty.x - p.z;
                const int2 X = close_limbs(dxh, tx.y - p.y, cl.s), Y = close_limbs(dyh, ty.y - p.w, cl.s);
                const long long sxx = square_hi(X), syy = square_hi(Y), sxy = mul_hi(X.x, X.y, Y.x, Y.y);
                if (max(abs(dxh), abs(dyh)) >= cl.lim || __mulhi(hi_bal(sxx + syy), cl.kmh) >= vmax) {
                    pair64(q0 + q);  // leaves so wide that far pairs are listed too
                    return;
                }
                const long long zx = scale_z(cl, sxx), zy = scale_z(cl, syy), zxy = scale_z(cl, sxy);
                const long long F = blob_fixed(g_fix_f, zx + zy), H = blob_fixed(g_fix_d, zx + zy);
                const int hh = hi_bal(H), hl = (int)lo_of(H);
                const long long Pxx = mul_55(zx, hh, hl), Pyy = mul_55(zy, hh, hl), Pxy = mul_55(zxy, hh, hl);
                const int2 g = gam[q];
                const int4 gg = ggr[q];
                // dgamma: (gu_m b - gv_m a) F
                const long long t = wide(gg.x, Y.x, wide(-gg.z, X.x, (long long)hi_of(wide(gg.y, Y.x, wide(gg.x, Y.y, 1ll << 31)) -
                                                                                      wide(gg.w, X.x, wide(gg.z, X.y, 0)))));
                const int th = hi_bal(t), tl = (int)lo_of(t), fh = hi_bal(F), fl = (int)lo_of(F);
                hg = wide(th, fh, hg);
                lg += wide(th, fl, wide(tl, fh, (long long)__mulhi(tl, fl))) >> 8;
                grad(cross(g, gg.x, gg.y, tuh, tul), cross(g, gg.z, gg.w, tvh, tvl), Pxy, F - Pxx, Pyy - F, -Pxy);
            };
            for (int q0 = 0; q0 < ntot; q0 += A64_TILE) {
                const int m = min(A64_TILE, ntot - q0);
                if (q0 > 0)
                    for (int q = 0; q < 6; ++q)
                        acc[q].mark(tid);
                __syncthreads();
                for (int q = tid; q < m; q += N64_THREADS) {
                    const int j = R.global(q0 + q);
                    const int2 px = limbs31(to_fixed(w.sx[j], ku)), py = limbs31(to_fixed(w.sy[j], ku));
                    const long long g = to_fixed(w.sg[j], ka), gu = to_fixed(w.sgu[j], kb), gv = to_fixed(w.sgv[j], kb);
                    pos[q] = make_int4(px.x, px.y, py.x, py.y);
                    gam[q] = make_int2(hi_bal(g), (int)lo_of(g));
                    ggr[q] = make_int4(hi_bal(gu), (int)lo_of(gu), hi_bal(gv), (int)lo_of(gv));
                }
                __syncthreads();
                const int nj = active ? (m - grp + G - 1) / G : 0;  // this thread's sources: grp, grp + G, ...
                const int nmax = __reduce_max_sync(0xffffffffu, nj);
                if (thr == 0) {  // every pair is close
                    for (int i = 0; i < nj; ++i) {
                        close(q0, grp + G * i);
                        if (i % A64_CAP == A64_CAP - 1)
                            spill(acc + 3);
                    }
                    spill(acc + 3);
                    continue;
                }
                for (int i0 = 0; i0 < nmax;) {
                    const int used = __reduce_max_sync(0xffffffffu, cnt);
                    const int i1 = min(nmax, i0 + A64_CAP - used);
                    for (int i = i0; i < min(i1, nj); ++i) {
                        const int q = grp + G * i;
                        const int4 p = pos[q];
                        const int dxh = tx.x - p.x, dxl = tx.y - p.y, dyh = ty.x - p.z, dyl = ty.y - p.w;
                        const long long r2 = r2_fixed(dxh, dxl, dyh, dyl);
                        if (hi_of(r2) < thr) {
                            lst[cnt * N64_THREADS + tid] = (unsigned short)q;
                            ++cnt;
                            continue;
                        }
                        // a / r^2 and b / r^2: displacement times Y, / 2^59 (at most 2^61.2)
                        const long long Y = recip_fixed(r2);
                        const int yh = hi_bal(Y), yl = (int)lo_of(Y), y2 = yl >> 1;
                        const long long ca = (wide(dxh, yh, 0) << 4) + (wide(dxl, yh, wide(dxh, y2, 1 << 26)) >> 27);
                        const long long cb = (wide(dyh, yh, 0) << 4) + (wide(dyl, yh, wide(dyh, y2, 1 << 26)) >> 27);
                        // P = 2 ca cb, Q = (cb - ca) (cb + ca), / 2^64
                        const long long cb2 = cb * 2, cs = cb + ca, cd = cb - ca;
                        const int cah = hi_bal(ca), cal = (int)lo_of(ca), cbh = hi_bal(cb), cbl = (int)lo_of(cb);
                        const long long P = mul_hi(cah, cal, hi_bal(cb2), (int)lo_of(cb2));
                        const long long Q = mul_hi(hi_bal(cs), (int)lo_of(cs), hi_bal(cd), (int)lo_of(cd));
                        const int2 g = gam[q];
                        const int4 gg = ggr[q];
                        // dgamma: gu_m b - gv_m a
                        hg = wide(gg.x, cbh, wide(-gg.z, cah, hg));
                        lg += (wide(gg.y, cbh, wide(gg.x, cbl, 0)) - wide(gg.w, cah, wide(gg.z, cal, 0))) >> 8;
                        grad(cross(g, gg.x, gg.y, tuh, tul), cross(g, gg.z, gg.w, tvh, tvl), P, Q, Q, -P);
                    }
                    spill(acc);
                    i0 = i1;
                    const int full = __reduce_max_sync(0xffffffffu, cnt);
                    if (full > A64_CAP - 12 || (i0 >= nmax && full > 0)) {
                        for (int e = 0; e < full; ++e)
                            if (e < cnt)
                                close(q0, lst[e * N64_THREADS + tid]);
                        spill(acc + 3);
                        cnt = 0;
                    }
                }
            }
            for (int q = 0; q < 6; ++q)
                acc[q].mark(tid);
            acc[1].meet(tid, acc[2]);
            acc[4].meet(tid, acc[5]);
        }
        // sums of a target's groups, in order; the FP64 pairs' through the (now idle) source limbs
        double *red = reinterpret_cast<double *>(pos);
        const bool some64 = __syncthreads_or(ag != 0.0 || ax != 0.0 || ay != 0.0);
        if (some64) {
            red[tid] = ag;
            red[N64_THREADS + tid] = ax;
            red[2 * N64_THREADS + tid] = ay;
            __syncthreads();
        }
        if (tid < cp) {
            const int ng = min(G, ntot);  // groups with sources
            double out[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                for (int g = 0; some64 && g < ng; ++g)
                    out[q] += red[q * N64_THREADS + tid + g * cp];
                if (ranges)
                    out[q] *= k2;
            }
            if (fixed) {
                // sums in units of 2^40: far a / r^2 2^(119 + ku) per ca, close F 2^62 in units of k2, a 2^(s - ku);
                // charges 2^-ka and 2^-kb, the target's 2^tau up (in one exponent: 2^(ka - tau) alone may be below FP64's range)
                const int kq = fresh(ku);
                const double fg = pow2(-79 - kq), cg = k2 * pow2(42 - cl.s + kq), fx = pow2(-70 - 2 * kq), cx = k2 * 0x1p42;
                // A target whose sums are all small against the rounding of their terms is left to FP64 (as in k_near64): a
                // far pair's dgamma is off by 2^20 (the charges' last bits, the low halves left out), its gradient by 2^16
                // (P and Q); a close pair's by about 2^18 and 2^19, by up to 2^21 where all pairs are close. So is one with a
                // coincident particle.
                const float far_g = acc[0].biggest(tid, cp, ng), near_g = acc[3].biggest(tid, cp, ng);
                const float far_x = acc[1].biggest(tid, cp, ng), near_x = acc[4].biggest(tid, cp, ng);
                const float4 line = s_line;
                bool small = fmaxf(far_g, near_g * line.x) < line_of(far_g, near_g, 0x1p42f, line.y) || far_g == INFINITY;
                if (gt != 0.0 || gut != 0.0 || gvt != 0.0)
                    small |= fmaxf(far_x, near_x * line.z) < line_of(far_x, near_x, 0x1p37f, line.w);
                if (small)
                    w.slot[tpos] = atomicExch(&s_weak, tpos);
                out[0] += ldexp(fma(acc[3].total(tid, cp, ng), cg, acc[0].total(tid, cp, ng) * fg), fresh(kb));
#pragma unroll
                for (int q = 1; q < 3; ++q)
                    out[q] += ldexp(fma(acc[3 + q].total(tid, cp, ng), cx, acc[q].total(tid, cp, ng) * fx), fresh(ka) + fresh(kb) - fresh(tau));
            }
            const int i = w.perm[tpos];
            if (odg)
                odg[i] = out[0] / kTwoPi;
            if (odx)
                odx[i] = out[1] / kTwoPi;
            if (ody)
                ody[i] = out[2] / kTwoPi;
        }
        __syncthreads();
    }
    }
    // the weak targets, in FP64 by the whole block (out of the loop over the leaves: within it, or in line, this takes
    // registers from the loops over the sources and 3% of the kernel)
    for (int t = s_weak; t >= 0; t = w.slot[t])
        adjoint_block64(w, t, reinterpret_cast<double *>(pos), odg, odx, ody);
}

}  // namespace

int prepare_near64(cudaStream_t s)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return -1;
    std::lock_guard<std::mutex> lk(g_tab_mu);
    if (g_tab_ready[dev])
        return 0;
    k_near64_tables<<<kRows / 4, 64, 0, s>>>();
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    if (cudaFuncSetAttribute(k_adjoint_near64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A64_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_adjoint_near64, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_near64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)N64_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_near64, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess)
        return -1;
    void *f = nullptr;
    if (cudaGetSymbolAddress(&f, g_blob_f) != cudaSuccess)
        return -1;
    g_tab_f[dev] = (const double2 *)f;
    g_tab_ready[dev] = true;
    return 0;
}

const double2 *near64_table()
{
    int dev = 0;
    return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? g_tab_f[dev] : nullptr;
}

// Persistent blocks, three to an SM, that take leaves from a counter: the register file (3 x 16 K of 64 K registers)
// and the shared memory left over hold blocks of the multipole sweep, which runs beside this kernel on the FP64 pipe
// (pending blocks of a plain grid would keep them out, and so would a smaller shared-memory carveout). Measured at 2^20:
// near field 3.05 ms with four blocks an SM and 3.25 with three; whole evaluation 4.38 and 3.50 ms (sweep alone 1.5).
// Where there are fewer leaves than resident blocks, each leaf's targets are shared out over up to eight units.
int launch_near64(const Work &w, cudaStream_t s)
{
    const int resident = 3 * kSMs;
    const int parts = max(1, min(8, resident / w.nleaf));
    k_near64<<<min(w.nleaf * parts, resident), N64_THREADS, N64_SMEM, s>>>(w, parts);
    return 1;
}

int launch_adjoint_near64(const Work &w, double *dg, double *dx, double *dy, int skip_plain, cudaStream_t s)
{
    const int resident = A64_B * kSMs;
    const int parts = max(1, min(8, resident / w.nleaf));
    k_adjoint_near64<<<min(w.nleaf * parts, resident), N64_THREADS, A64_SMEM, s>>>(w, parts, dg, dx, dy, skip_plain);
    return 1;
}

}  // namespace fmm
