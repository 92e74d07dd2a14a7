// near64.cu -- Fig. 1 stage 9 in the plain form: the near field of Eq. 6 in (at least) FP64 accuracy.
//
// GB300 has 2 FP64 multiply-adds per SM and clock against 128 in FP32 and 30 wide (32 x 32 -> 64) integer ones, so
// the pairs are split by what they need:
//   * r > sqrt(75) sigma (x = r^2 / 2 sigma^2 > 37.5): 1 - e^-x is 1 in FP64 and the pair is the point vortex
//     gamma (-dy, dx) / r^2. It runs in 64-bit fixed point on the integer pipe: coordinates as exact integers (their
//     differences carry no rounding error), 1 / r^2 by one Newton step of second order from the SFU's FP32
//     reciprocal, products from three wide multiplications each, sums in 64-bit integers.
//   * closer pairs go to a list per thread (index in shared memory) and run in FP64 once the list is full or the
//     sources are done, every lane with a pair of its own: F(x) = (1 - e^-x) / x comes from a table of 600
//     polynomials of degree 6 (no exponential, no division), 15 FP64 operations a pair.
// A block whose charges span a wide range (so that a fixed unit could lose digits of a small sum), and trees whose
// leaves are so narrow that every adjacent pair is close, run all pairs in FP64.
#include <math.h>

#include <mutex>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

constexpr double kTwoPi = 6.283185307179586476925;

// ------------------------------------------------------------------ table of F(x) = (1 - e^-x) / x

// Row i: the polynomial in t = x - c, c = (i + 1/2) / 16, that interpolates F on [i / 16, (i + 1) / 16) at Chebyshev
// nodes, truncated to degree 6 (its error there is below (1/32)^7 / (2^6 7! 8) = 2e-17), then c itself. x < 37.5.
constexpr int kTabN = 600;
constexpr double kXCut = 37.5;  // e^-37.5 < 2^-54: beyond it 1 - e^-x rounds to 1
__device__ double2 g_blob_f[kTabN * 4];

long double blob_f(long double x) { return x == 0.0L ? 1.0L : -expm1l(-x) / x; }

// Coefficients (monomial in t, |t| <= h) of the degree-6 truncation of the Chebyshev interpolant of fn about c.
void cheb6(long double (*fn)(long double), long double c, long double h, double *out)
{
    constexpr int N = 16, D = 6;
    const long double pi = 3.141592653589793238462643383279502884L;
    long double a[D + 1];
    for (int k = 0; k <= D; ++k) {
        a[k] = 0.0L;
        for (int j = 0; j < N; ++j)
            a[k] += fn(c + h * cosl(pi * (j + 0.5L) / N)) * cosl(pi * k * (j + 0.5L) / N);
        a[k] *= (k == 0 ? 1.0L : 2.0L) / N;
    }
    long double T[D + 1][D + 1] = {};  // T_k(s) = sum_m T[k][m] s^m
    T[0][0] = 1.0L;
    T[1][1] = 1.0L;
    for (int k = 2; k <= D; ++k)
        for (int m = 0; m <= k; ++m)
            T[k][m] = (m ? 2.0L * T[k - 1][m - 1] : 0.0L) - T[k - 2][m];
    long double hm = 1.0L;
    for (int m = 0; m <= D; ++m) {
        long double s = 0.0L;
        for (int k = D; k >= m; --k)
            s += a[k] * T[k][m];
        out[m] = (double)(s / hm);
        hm *= h;
    }
}

std::mutex g_tab_mu;
bool g_tab_ready[64];

// F(x) for 0 <= x < kXCut: the row from the bit pattern of x (integer operations), then one subtraction and six
// multiply-adds.
__device__ __forceinline__ int blob_row(double x)
{
    const int hi = __double2hiint(x);
    const int e = (hi >> 20) - 1023;
    return e >= -4 ? ((hi & 0xfffff) | 0x100000) >> (16 - e) : 0;
}
__device__ __forceinline__ double blob_poly(const double2 *__restrict__ tab, int i, double x)
{
    const double2 c01 = __ldg(tab + 4 * i), c23 = __ldg(tab + 4 * i + 1), c45 = __ldg(tab + 4 * i + 2),
                  c6c = __ldg(tab + 4 * i + 3);
    const double t = x - c6c.y;
    double f = fma(c6c.x, t, c45.y);
    f = fma(f, t, c45.x);
    f = fma(f, t, c23.y);
    f = fma(f, t, c23.x);
    f = fma(f, t, c01.y);
    return fma(f, t, c01.x);
}

// 1 / x to FP64 rounding for a normal x > 0: the SFU's seed (relative error below 2^-20) and one Newton step of third
// order, y (1 + e + e^2) with e = 1 - x y.
__device__ __forceinline__ double recip64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// ------------------------------------------------------------------ fixed point

// round(v * 2^-k) modulo 2^64 (v = 0 for zeros and subnormals).
__device__ __forceinline__ long long to_fixed(double v, int k)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int be = (int)((b >> 52) & 0x7ff);
    if (be == 0)
        return 0;
    const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
    const int sh = be - 1075 - k;
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

// Near-field geometry of one target leaf: its source rows (contiguous runs of the sorted particles) and the fixed
// point scales.
struct Rows64 {
    int a[3], pre[4];  // first particle of row k, prefix of the rows' counts
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
constexpr int N64_FEW = 96;     // fewer sources than this run in FP64
// smallest high word of r^2 (62 fraction bits dropped) that the fixed point takes: 1 / r^2 below 2^31 as a seed and
// r^2 to 2^-53 relative
constexpr int N64_RMIN = 3410000;

__device__ __forceinline__ int exponent_of(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff) - 1023; }

// Smallest k with v <= 2^k, v > 0 normal.
__device__ __forceinline__ int ceil_log2(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return exponent_of(v) + ((b & 0xfffffffffffffull) ? 1 : 0);
}

// Passes over a leaf of c targets: the number of passes (at most 4 more than needed) that keeps most of the 256
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

// One block per leaf. Thread = (target t, source group g of G): the pass's targets run over the threads, and the
// groups take the sources in turn; the groups' sums of a target are added at the end in a fixed order.
// Measured at 2^20 uniform particles (leaves of 64, 16 sigma wide): 39.0 ms with every pair by expm1 and a division
// in FP64, 4.1 ms so; bound by the FP64 pipe (77 % busy) on the tenth of the pairs that are close. The error of the
// near field against quad precision fell from 8.6e-16 to 2.2e-16 relative L2 (exact differences, integer sums).
// Line of the fixed point: fewer than 96 sources in the neighbourhood have no time in it (4 to 24 particles a leaf
// agree to 2.5e-16 either way).
__global__ void __launch_bounds__(N64_THREADS, 4) k_near64(Work w)
{
    __shared__ int4 pos[N64_TILE];   // x and y limbs
    __shared__ int2 gam[N64_TILE];   // gamma limbs, base 2^32
    __shared__ unsigned short lst[N64_CAP * N64_THREADS];
    __shared__ unsigned s_max;
    __shared__ unsigned long long s_sum;
    __shared__ int s_cnt;
    const int leaf = blockIdx.x, tid = threadIdx.x;
    const int s0 = w.start[leaf], c = w.start[leaf + 1] - s0;
    if (c == 0)
        return;
    const int k = w.nsys == 1 ? 0 : find_sys_by_leaf(w.sys, w.nsys, leaf);
    const SysDev &d = w.sys[k];
    const int L = d.depth, ns = 1 << L, local = leaf - (int)d.leaf0;
    const int ix = local & (ns - 1), iy = local >> L;
    const int jx0 = ix > 0 ? ix - 1 : 0, jx1 = ix < ns - 1 ? ix + 1 : ns - 1;
    Rows64 R;
    R.pre[0] = 0;
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) {
        const int row = iy + dy - 1;
        int a = 0, n = 0;
        if (row >= 0 && row < ns) {
            a = w.start[d.leaf0 + row * ns + jx0];
            n = w.start[d.leaf0 + row * ns + jx1 + 1] - a;
        }
        R.a[dy] = a;
        R.pre[dy + 1] = R.pre[dy] + n;
    }
    const int ntot = R.pre[3];
    const double k2 = 1.0 / (2.0 * d.sigma * d.sigma);

    // fixed-point unit 2^ku: two leaf widths are at most 2^61 of it; r^2 >= rc2 units of 2^94 is the far range
    const int ku = ceil_log2(2.0 * d.wl) - 61;
    const double cut = ldexp(2.0 * kXCut * d.sigma * d.sigma, -2 * ku - 94);
    // lengths whose squares and their ratios stay well inside FP64's range (else every pair by expm1 and division)
    const bool ranges = abs(exponent_of(d.sigma)) < 200 && abs(exponent_of(d.wl)) < 200;
    bool fixed = ranges && cut < 0x1p30 && ntot >= N64_FEW;  // some adjacent pair is far
    const int thr = fixed ? max((int)cut + 2, N64_RMIN) : 0;
    // the charges' largest magnitude and mean (of the non-zero ones): the fixed point is kept for sums whose terms
    // are not all far below its unit's range
    if (tid == 0) {
        s_max = 0;
        s_sum = 0;
        s_cnt = 0;
    }
    __syncthreads();
    unsigned gm = 0;
    if (fixed) {
        for (int q = tid; q < ntot; q += N64_THREADS)
            gm = max(gm, (unsigned)__double2hiint(w.sg[R.global(q)]) & 0x7fffffffu);
        gm = __reduce_max_sync(0xffffffffu, gm);
        if ((tid & 31) == 0)
            atomicMax(&s_max, gm);
    }
    __syncthreads();
    gm = s_max;
    const int ge = (int)(gm >> 20);  // biased exponent of the largest charge
    fixed = fixed && ge > 100 && ge < 0x7ff;
    if (fixed) {
        unsigned sum = 0;
        int cnt = 0;
        for (int q = tid; q < ntot; q += N64_THREADS) {
            const unsigned h = (unsigned)__double2hiint(w.sg[R.global(q)]) & 0x7fffffffu;
            sum += ((h & 0xfffffu) | 0x100000u) >> min(ge - (int)(h >> 20), 31);
            cnt += h != 0;
            if (sum > 0x40000000u) {
                atomicAdd(&s_sum, (unsigned long long)sum);
                sum = 0;
            }
        }
        sum = __reduce_add_sync(0xffffffffu, sum >> 5) << 5;  // the low bits do not matter here
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if ((tid & 31) == 0) {
            atomicAdd(&s_sum, (unsigned long long)sum);
            atomicAdd(&s_cnt, cnt);
        }
    }
    __syncthreads();
    if (fixed) {
        const unsigned long long big = (gm & 0xfffffu) | 0x100000u;
        fixed = s_sum > big && (s_sum - big) * 16 >= big * (unsigned long long)max(s_cnt - 1, 1);
    }
    // charges in units of 2^ka: below 2^63 - 2^50, so that their high limb fits
    const int ka = ge - 1023 + 1 - ((gm & 0xfffffu) < 0xfff00u ? 63 : 62);

    const int npass = pick_passes(c);
    for (int pass = 0; pass < npass; ++pass) {
        const int t0 = (int)((long long)pass * c / npass), cp = (int)((long long)(pass + 1) * c / npass) - t0;
        const int G = N64_THREADS / cp;
        const int grp = tid / cp, tpos = s0 + t0 + (tid - grp * cp);
        const bool active = grp < G;
        const double xt = w.sx[tpos], yt = w.sy[tpos];
        double au = 0.0, av = 0.0;    // FP64 pairs: sums of gamma F(x) (-dy, dx), in units of k2
        double iu = 0.0, iv = 0.0;    // fixed-point pairs, in units of 2^-(...) (scaled at the end)
        auto pair64 = [&](int q) {
            const int j = R.global(q);
            const double ax = xt - w.sx[j], ay = yt - w.sy[j];
            const double x = fma(ax, ax, ay * ay) * k2;
            double f = x < kXCut ? blob_poly(g_blob_f, blob_row(x), x) : recip64(x);
            // a particle and itself, or coincident ones: nothing, whatever the charge
            f = __double_as_longlong(x) != 0 ? f * w.sg[j] : 0.0;
            au = fma(-ay, f, au);
            av = fma(ax, f, av);
        };
        if (!ranges) {
            if (active)
                for (int q = grp; q < ntot; q += G) {
                    const int j = R.global(q);
                    const double ax = xt - w.sx[j], ay = yt - w.sy[j], r2 = ax * ax + ay * ay;
                    if (r2 > 0.0) {
                        const double f = -expm1(-r2 * k2) / r2 * w.sg[j];
                        iu += ay * f;
                        iv += ax * f;
                    }
                }
        } else if (!fixed) {
            if (active)
                for (int q = grp; q < ntot; q += G)
                    pair64(q);
        } else {
            const int2 tx = limbs31(to_fixed(xt, ku)), ty = limbs31(to_fixed(yt, ku));
            int cnt = 0, terms = 0;
            long long su = 0, sv = 0;
            for (int q0 = 0; q0 < ntot; q0 += N64_TILE) {
                const int m = min(N64_TILE, ntot - q0);
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
                for (int i0 = 0; i0 < nmax;) {
                    // as many sources as the fullest list of the warp still takes
                    const int used = __reduce_max_sync(0xffffffffu, cnt);
                    const int i1 = min(nmax, i0 + N64_CAP - used);
                    for (int i = i0; i < min(i1, nj); ++i) {
                        const int q = grp + G * i;
                        const int4 p = pos[q];
                        int2 g = gam[q];
                        const int dxh = tx.x - p.x, dxl = tx.y - p.y, dyh = ty.x - p.z, dyl = ty.y - p.w;
                        // r^2 2^-62: high products and the cross terms 2 h l 2^-31
                        const long long cr = wide(dyh, dyl, wide(dxh, dxl, 0));
                        const long long r2 = wide(dyh, dyh, wide(dxh, dxh, cr >> 30));
                        const int rh = hi_of(r2);
                        if (rh < thr) {
                            lst[cnt * N64_THREADS + tid] = (unsigned short)q;
                            ++cnt;
                            g = make_int2(0, 0);
                        }
                        // Y0 ~ 2^84 / r^2 from the SFU; r^2 Y0 = 2^84 (1 + e) modulo 2^64, |e| < 2^-21
                        float yf;
                        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__int2float_rn(rh) + 0.5f));
                        const unsigned y0 = __float2uint_rn(yf * 0x1p52f);
                        const unsigned long long P = wide_u(lo_of(r2), y0);
                        const int eh = (int)((unsigned)(P >> 32) + (unsigned)rh * y0);
                        const int es = eh >> 15;
                        const unsigned e2 = (unsigned)(es * es);  // e^2 2^74
                        // c = e^2 - e, 84 fraction bits; Y = 2^32 Y0 (1 + c) = 2^116 / r^2
                        const long long cc = (long long)((unsigned long long)e2 << 10) -
                                             (long long)(((unsigned long long)(unsigned)eh << 32) | (unsigned)P);
                        const long long T = wide(hi_of(cc), (int)y0, (long long)(unsigned long long)__umulhi(lo_of(cc), y0));
                        const long long Y = (T >> 20) + ((long long)y0 << 32);
                        // f = gamma Y 2^-64
                        const int yh = hi_bal(Y), yl = (int)lo_of(Y);
                        const long long f = wide(g.x, yh, (long long)hi_of(wide(g.y, yh, wide(g.x, yl, 1ll << 31))));
                        const int fh = hi_bal(f), fl = (int)lo_of(f) >> 1;
                        su += wide(fh, dyh, wide(fl, dyh, wide(fh, dyl, 1ll << 30)) >> 31);
                        sv += wide(fh, dxh, wide(fl, dxh, wide(fh, dxl, 1ll << 30)) >> 31);
                    }
                    terms += i1 - i0;
                    if (terms > N64_SPILL - N64_CAP) {
                        iu += (double)su;
                        iv += (double)sv;
                        su = sv = 0;
                        terms = 0;
                    }
                    i0 = i1;
                    const int full = __reduce_max_sync(0xffffffffu, cnt);
                    if (full > N64_CAP - 12 || (i0 >= nmax && full > 0)) {
                        for (int e = 0; e < full; ++e)
                            if (e < cnt)
                                pair64(q0 + lst[e * N64_THREADS + tid]);
                        cnt = 0;
                    }
                }
            }
            iu += (double)su;
            iv += (double)sv;
            // a fixed-point term is gamma dx / r^2 * 2^(51 + ku - ka)
            const double sc = scalbn(1.0, -51 - ku) ;
            iu = scalbn(iu * sc, ka);
            iv = scalbn(iv * sc, ka);
        }
        // groups of a target, in order, through the (now idle) list
        double2 *red = reinterpret_cast<double2 *>(pos);
        const double pu = ranges ? fma(au, k2, -iu) : -iu, pv = ranges ? fma(av, k2, iv) : iv;
        __syncthreads();
        if (active)
            red[tid] = make_double2(pu, pv);
        __syncthreads();
        if (tid < cp) {
            double u = 0.0, v = 0.0;
            for (int g = 0; g < G; ++g) {
                const double2 a = red[tid + g * cp];
                u += a.x;
                v += a.y;
            }
            w.near64[tpos] = make_double2(u / kTwoPi, v / kTwoPi);
        }
    }
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
    static double tab[kTabN][8];
    for (int i = 0; i < kTabN; ++i) {
        const long double c = (i + 0.5L) / 16.0L;
        cheb6(blob_f, c, 1.0L / 32.0L, tab[i]);
        tab[i][7] = (double)c;
    }
    if (cudaMemcpyToSymbolAsync(g_blob_f, tab, sizeof tab, 0, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    g_tab_ready[dev] = true;
    return 0;
}

int launch_near64(const Work &w, cudaStream_t s)
{
    k_near64<<<w.nleaf, N64_THREADS, 0, s>>>(w);
    return 1;
}

}  // namespace fmm
