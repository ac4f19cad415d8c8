// gauge.cu -- the gauge part of the molecular dynamics step (Sec. 2.1, the
// tree-level Symanzik improved action; Sec. 4.2 and Algorithm 2, the gauge
// cycle; Listing lst:rect_staples, the staples; Table md-norm, its cost per
// site) in FP64 and in FP32 (Algorithm 1, step 5: "possibly in single
// precision").
//
//   S_g = -(beta/3) sum_x [ c0 sum_{mu<nu} Re Tr P_{mu nu}(x) + c1 sum_{mu!=nu} Re Tr R_{mu nu}(x) ]
//   c0 = 5/3, c1 = -1/12;  P: 1x1 plaquette, R: 2 links along mu, 1 along nu
//   force:  F_mu(x) = traceless part of -(i beta/6)(M - M^dag), M = U_mu(x) A_mu(x)
//   momenta: H <- H - eps F          links: U <- exp(i eps H) U
// where A_mu(x) is the sum of the staples of U_mu(x): c0 times the 3-link
// paths and c1 times the 5-link paths that close the plaquettes and
// rectangles through U_mu(x), for nu != mu and both signs of nu.
//
// Storage: links in the context's SoA formats, [4 mu][2 parity][9 comp][V/2]
// (double2 for FP64 -- the master copy -- and float2 for FP32); momenta as 8
// reals per link (traceless Hermitian: h00, h11, re/im of h01, h02, h12),
// [4][2][8][V/2].  One thread per link.  Neighbour links are gathered through
// L1/L2 (every link is read by ~80 threads of nearby sites).
#include <cmath>
#include <mutex>

#include "deo_core.cuh"
#include "internal.h"

namespace lqcd {

constexpr double kSymC0 = 5.0 / 3.0;
constexpr double kSymC1 = -1.0 / 12.0;
constexpr int kGaugeThreads = 128;

template <class T> struct Cplx { T re, im; };
template <class T> struct Mat3 { Cplx<T> e[9]; };
template <class T> struct Vec2T;
template <> struct Vec2T<double> { using t = double2; };
template <> struct Vec2T<float> { using t = float2; };

template <class T>
__device__ __forceinline__ void mat_mul(const Mat3<T> &a, const Mat3<T> &b, Mat3<T> &c)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T re = 0, im = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Cplx<T> x = a.e[i * 3 + k], y = b.e[k * 3 + j];
                re = fma(x.re, y.re, fma(-x.im, y.im, re));
                im = fma(x.re, y.im, fma(x.im, y.re, im));
            }
            c.e[i * 3 + j] = {re, im};
        }
}

// c = a b^dag
template <class T>
__device__ __forceinline__ void mat_mul_dag(const Mat3<T> &a, const Mat3<T> &b, Mat3<T> &c)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T re = 0, im = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Cplx<T> x = a.e[i * 3 + k], y = b.e[j * 3 + k];  // conj(b_jk)
                re = fma(x.re, y.re, fma(x.im, y.im, re));
                im = fma(-x.re, y.im, fma(x.im, y.re, im));
            }
            c.e[i * 3 + j] = {re, im};
        }
}

// c += a b, c += a b^dag, c += (a b)^dag: sums without a pass of their own
// (FP64, 16^4: stout level 851 -> 798 us, local pass of the chain 1652 -> 1567)
template <class T>
__device__ __forceinline__ void mat_mul_add(const Mat3<T> &a, const Mat3<T> &b, Mat3<T> &c)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            Cplx<T> s = c.e[i * 3 + j];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Cplx<T> x = a.e[i * 3 + k], y = b.e[k * 3 + j];
                s.re = fma(x.re, y.re, fma(-x.im, y.im, s.re));
                s.im = fma(x.re, y.im, fma(x.im, y.re, s.im));
            }
            c.e[i * 3 + j] = s;
        }
}
template <class T>
__device__ __forceinline__ void mat_mul_dag_add(const Mat3<T> &a, const Mat3<T> &b, Mat3<T> &c)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            Cplx<T> s = c.e[i * 3 + j];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Cplx<T> x = a.e[i * 3 + k], y = b.e[j * 3 + k];  // conj(b_jk)
                s.re = fma(x.re, y.re, fma(x.im, y.im, s.re));
                s.im = fma(-x.re, y.im, fma(x.im, y.re, s.im));
            }
            c.e[i * 3 + j] = s;
        }
}
template <class T>
__device__ __forceinline__ void mat_mul_add_dag(const Mat3<T> &a, const Mat3<T> &b, Mat3<T> &c)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            Cplx<T> s = c.e[j * 3 + i];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Cplx<T> x = a.e[i * 3 + k], y = b.e[k * 3 + j];
                s.re = fma(x.re, y.re, fma(-x.im, y.im, s.re));
                s.im = fma(-x.re, y.im, fma(-x.im, y.re, s.im));
            }
            c.e[j * 3 + i] = s;
        }
}

template <class T>
__device__ __forceinline__ void mat_dag(Mat3<T> &a)
{
    Mat3<T> t = a;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) a.e[i * 3 + j] = {t.e[j * 3 + i].re, -t.e[j * 3 + i].im};
}

template <class T>
__device__ __forceinline__ void mat_axpy(T s, const Mat3<T> &x, Mat3<T> &y)
{
#pragma unroll
    for (int i = 0; i < 9; ++i) y.e[i] = {fma(s, x.e[i].re, y.e[i].re), fma(s, x.e[i].im, y.e[i].im)};
}

// ------------------------------------------------------------------ geometry of links
struct LinkGeo {
    int N[4];
    int Vh;
};

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// (parity, half index) of x + d, |d_m| <= 2 <= N_m
__device__ __forceinline__ void site_of(const LinkGeo &g, const int (&x)[4], int d0, int d1, int d2, int d3, int &par,
                                        int &idx)
{
    const int y0 = wrap(x[0] + d0, g.N[0]), y1 = wrap(x[1] + d1, g.N[1]);
    const int y2 = wrap(x[2] + d2, g.N[2]), y3 = wrap(x[3] + d3, g.N[3]);
    par = (y0 + y1 + y2 + y3) & 1;
    idx = bound_index((y0 + g.N[0] * (y1 + g.N[1] * (y2 + g.N[2] * y3))) >> 1, g.Vh);
}

template <class T>
__device__ __forceinline__ void load_link_soa(const typename Vec2T<T>::t *__restrict__ L, int mu, int par, int idx,
                                              int Vh, Mat3<T> &U)
{
    const typename Vec2T<T>::t *p = L + (size_t)((mu * 2 + par) * 9) * Vh + idx;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const typename Vec2T<T>::t v = __ldg(p + (size_t)c * Vh);
        U.e[c] = {v.x, v.y};
    }
}

struct SiteIdx { int par, idx; };
__device__ __forceinline__ SiteIdx site_step(const LinkGeo &g, const int (&x)[4], int a, int sa, int b = 0, int sb = 0)
{
    int d[4] = {0, 0, 0, 0};
#pragma unroll
    for (int m = 0; m < 4; ++m) d[m] = (m == a ? sa : 0) + (m == b ? sb : 0);
    SiteIdx s;
    site_of(g, x, d[0], d[1], d[2], d[3], s.par, s.idx);
    return s;
}

// Lexicographic offset of d steps in direction m from x.  Offsets of different
// directions add, so a site of a staple costs one addition.
__device__ __forceinline__ int step_delta(const LinkGeo &g, const int (&x)[4], int m, int d)
{
    const int n = g.N[m], v = m == 0 ? x[0] : m == 1 ? x[1] : m == 2 ? x[2] : x[3];
    const int stride = m == 0 ? 1 : g.N[0] * (m == 1 ? 1 : g.N[1] * (m == 2 ? 1 : g.N[2]));
    return (wrap(v + d, n) - v) * stride;
}

// Links on their way from L2 to a thread: D slots of nine components per thread
// of the block, filled with cp.async.  A thread reads only what it copied.
struct LinkRing {
    static constexpr int D = 4;
    float2 e[D + 1][9][kGaugeThreads];   // slot D: the link that every side takes
};

// Element 0 of U_dir at a site in an array of link layout.  64 bits: the last
// component of a lattice of 2^26 even sites lies beyond 2^32.
__host__ __device__ constexpr size_t link_offset(int dir, int par, int idx, int Vh)
{
    return (size_t)((dir * 2 + par) * 9) * (size_t)Vh + (size_t)idx;
}
static_assert(link_offset(3, 1, (1 << 30) - 1, 1 << 30) + 8 * (size_t)(1 << 30) == ((size_t)72 << 30) - 1,
              "the largest lattice that lqcd_create takes");

// U_dir at a site into slot (one group; an empty one if !live)
__device__ __forceinline__ void ring_fetch(LinkRing &R, int slot, const float2 *__restrict__ L, int dir, SiteIdx s, int Vh,
                                           bool live = true)
{
    if (live) {
        const float2 *p = L + link_offset(dir, s.par, s.idx, Vh);
        const unsigned d = (unsigned)__cvta_generic_to_shared(&R.e[slot][0][threadIdx.x]);
#pragma unroll
        for (int c = 0; c < 9; ++c)
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d + c * (unsigned)(kGaugeThreads * sizeof(float2))),
                         "l"(p + (size_t)c * Vh), "n"
                         (sizeof(float2))
                         : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The link in a slot, or its conjugate transpose (read transposed, imaginary
// parts negated).
__device__ __forceinline__ void ring_read(const LinkRing &R, int slot, bool dag, Mat3<float> &U)
{
    const int row = dag ? 1 : 3, col = dag ? 3 : 1;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const float2 v = R.e[slot][(c / 3) * row + (c % 3) * col][threadIdx.x];
        U.e[c] = {v.x, dag ? -v.y : v.y};
    }
}

__device__ __forceinline__ void coords_of(const LinkGeo &g, int P, int i, int (&x)[4])
{
    const int n0h = g.N[0] >> 1;
    int r = i / n0h;
    const int x0h = i - r * n0h;
    x[1] = r % g.N[1];
    r /= g.N[1];
    x[2] = r % g.N[2];
    x[3] = r / g.N[2];
    x[0] = 2 * x0h + ((x[1] + x[2] + x[3] + P) & 1);
}

// Staple sum A of the link U_mu(x) (see the file header).  Prefix sharing
// per (nu, s): P1 = step +s nu from x+mu, Q = P1 U_mu(x+s nu)^dag,
// E = step from x+s nu back to x; plaquette = Q E, rectangle (b) =
// Q U_mu(x-mu+s nu)^dag (step -s nu) U_mu(x-mu), rectangles (a) and (c)
// end in E, so c0 Q + c1 (a' + c') is multiplied by E once.
// A step in direction -nu starting at y is U_nu(y - nu)^dag.
// Twelve links of a side come through the ring in the order of their use, D - 1
// links ahead, across sides.
constexpr int kSideLinks = 12;
__device__ __forceinline__ void staple_sum_f32(const LinkGeo &g, const float2 *__restrict__ L, LinkRing &R,
                                               const int (&x)[4], int P, int i, int mu, Mat3<float> &A)
{
    using T = float;
    constexpr int D = LinkRing::D;
    const int Vh = g.Vh;
#pragma unroll
    for (int k = 0; k < 9; ++k) A.e[k] = {T(0), T(0)};
    const T c0 = T(kSymC0), c1 = T(kSymC1);
    const int full = x[0] + g.N[0] * (x[1] + g.N[1] * (x[2] + g.N[2] * x[3]));
    const int dm1 = step_delta(g, x, mu, 1), dm2 = step_delta(g, x, mu, 2), db1 = step_delta(g, x, mu, -1);
    // the site at lexicographic offset d, an odd or even number of steps away
    auto at = [&](int d, int odd) { return SiteIdx{P ^ odd, bound_index((full + d) >> 1, Vh)}; };
    // link k of the side (nu, up); d1, d2: offsets of one and two steps s nu
    auto fetch = [&](int slot, int k, int nu, bool up, int d1, int d2, bool live) {
        SiteIdx s;
        int dir = mu;
        switch (k) {
            case 0: dir = nu; s = up ? at(dm1, 1) : at(dm1 + d1, 0); break;
            case 1: s = at(d1, 1); break;
            case 2: s = at(db1 + d1, 0); break;
            case 3: dir = nu; s = up ? at(db1, 1) : at(db1 + d1, 0); break;
            case 4: dir = nu; s = up ? at(dm1 + d1, 0) : at(dm1 + d2, 1); break;
            case 5: s = at(d2, 0); break;
            case 6: dir = nu; s = up ? at(d1, 1) : at(d2, 0); break;
            case 7: s = at(dm1, 1); break;
            case 8: dir = nu; s = up ? at(dm2, 0) : at(dm2 + d1, 1); break;
            case 9: s = at(dm1 + d1, 0); break;
            case 10: s = at(d1, 1); break;
            default: dir = nu; s = up ? SiteIdx{P, i} : at(d1, 1); break;
        }
        ring_fetch(R, slot, L, dir, s, Vh, live);
    };
    int w = mu == 0 ? 2 : 0;
    int d1 = step_delta(g, x, w >> 1, -1);
    const SiteIdx b1 = at(db1, 1);
    ring_fetch(R, D, L, mu, b1, Vh);   // U_mu(x - mu)
#pragma unroll
    for (int k = 0; k < D - 1; ++k) fetch(k, k, w >> 1, false, d1, 0, true);
#pragma unroll 1
    while (w < 8) {
        const int nu = w >> 1;
        const bool up = (w & 1) != 0;   // s = -1, then +1
        const int d2 = step_delta(g, x, nu, up ? 2 : -2);
        int wn = w + 1;
        if ((wn >> 1) == mu) wn += 2;
        const int nn = min(wn, 7) >> 1;
        const bool un = (wn & 1) != 0;
        // nothing after the last side (nn may be mu there, whose offsets do not add)
        const int dn = wn < 8 ? step_delta(g, x, nn, un ? 1 : -1) : 0;
        // link k into U, and the one D - 1 further on into the slot of link k - 1
        auto take = [&](int k, bool dag, Mat3<T> &U) {
            asm volatile("cp.async.wait_group %0;" ::"n"(D - 2) : "memory");
            ring_read(R, k % D, dag, U);
            const int f = k + D - 1;
            if (f < kSideLinks) fetch(f % D, f, nu, up, d1, d2, true);
            else fetch(f % D, f - kSideLinks, nn, un, dn, 0, wn < 8);
        };
        Mat3<T> P1, Q, W, t1, t2;
        // P1 = step(x+mu, s nu)
        take(0, !up, P1);
        // Q = P1 U_mu(x + s nu)^dag
        take(1, true, t1);
        mat_mul(P1, t1, Q);
        // rectangle (b): Q U_mu(x - mu + s nu)^dag step(x-mu+s nu, -s nu) U_mu(x - mu)
        take(2, true, t1);
        mat_mul(Q, t1, t2);
        take(3, up, t1);
        mat_mul(t2, t1, W);
        ring_read(R, D, false, t1);
        mat_mul(W, t1, t2);
        mat_axpy(c1, t2, A);
        // W = c0 Q + c1 (a' + c'), multiplied by E below
#pragma unroll
        for (int k = 0; k < 9; ++k) W.e[k] = {c0 * Q.e[k].re, c0 * Q.e[k].im};
        // c' = P1 step(x+mu+s nu, s nu) U_mu(x + 2 s nu)^dag step(x + 2 s nu, -s nu)
        take(4, !up, t1);
        mat_mul(P1, t1, t2);
        take(5, true, t1);
        mat_mul(t2, t1, Q);
        take(6, up, t1);
        mat_mul(Q, t1, t2);
        mat_axpy(c1, t2, W);
        // a' = U_mu(x + mu) step(x + 2 mu, s nu) U_mu(x + mu + s nu)^dag U_mu(x + s nu)^dag
        take(7, false, P1);
        take(8, !up, t1);
        mat_mul(P1, t1, t2);
        take(9, true, t1);
        mat_mul(t2, t1, Q);
        take(10, true, t1);
        mat_mul(Q, t1, t2);
        mat_axpy(c1, t2, W);
        // E = step(x + s nu, -s nu);  A += W E
        take(11, up, t1);
        mat_mul(W, t1, t2);
        mat_axpy(T(1), t2, A);
        w = wn;
        d1 = dn;
    }
}

// ------------------------------------------------------------------ double-float (FP64 on FP32 pipes)
// The FP64 MD step in double-float arithmetic: an SU(3) element is 9
// complex numbers of (hi, lo) float pairs (the context's df64 link copy, one
// float4 per complex), products summed Dot2-style (common.cuh), so the
// result carries ~48 significant bits on the FP32 pipes, which GB300 issues
// 64 times faster than FP64.
using DC = Cplx<float2>;
using DM3 = Mat3<float2>;

__device__ __forceinline__ void dm_load(const float4 *__restrict__ L, int mu, int par, int idx, int Vh, DM3 &U)
{
    const float4 *p = L + (size_t)((mu * 2 + par) * 9) * Vh + idx;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const float4 v = __ldg(p + (size_t)c * Vh);
        U.e[c].re = make_float2(v.x, v.y);
        U.e[c].im = make_float2(v.z, v.w);
    }
}

// c = a b
__device__ __forceinline__ void dm_mul(const DM3 &a, const DM3 &b, DM3 &c)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            Acc2 re, im;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const DC x = a.e[i * 3 + k];
                const DC y = b.e[k * 3 + j];
                if (k == 0) {
                    acc_first(re, x.re.x, x.re.y, y.re.x, y.re.y);
                    acc_first(im, x.re.x, x.re.y, y.im.x, y.im.y);
                } else {
                    acc_prod(re, x.re.x, x.re.y, y.re.x, y.re.y);
                    acc_prod(im, x.re.x, x.re.y, y.im.x, y.im.y);
                }
                acc_prod(re, -x.im.x, -x.im.y, y.im.x, y.im.y);
                acc_prod(im, x.im.x, x.im.y, y.re.x, y.re.y);
            }
            c.e[i * 3 + j].re = acc_result(re);
            c.e[i * 3 + j].im = acc_result(im);
        }
}

// r = x b for a row x.  The first product of a sum skips the addition to zero
// (8 of 78 instructions of a component).
__device__ __forceinline__ void mm_row(const DC (&x)[3], const DM3 &b, DC (&r)[3])
{
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        Acc2 re, im;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const DC y = b.e[k * 3 + j];
            if (k == 0) {
                acc_first(re, x[k].re.x, x[k].re.y, y.re.x, y.re.y);
                acc_first(im, x[k].re.x, x[k].re.y, y.im.x, y.im.y);
            } else {
                acc_prod(re, x[k].re.x, x[k].re.y, y.re.x, y.re.y);
                acc_prod(im, x[k].re.x, x[k].re.y, y.im.x, y.im.y);
            }
            acc_prod(re, -x[k].im.x, -x[k].im.y, y.im.x, y.im.y);
            acc_prod(im, x[k].im.x, x[k].im.y, y.re.x, y.re.y);
        }
        r[j].re = acc_result(re);
        r[j].im = acc_result(im);
    }
}
__device__ __forceinline__ void mm_row(const Cplx<double> (&x)[3], const Mat3<double> &b, Cplx<double> (&r)[3])
{
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        double re = 0, im = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const Cplx<double> y = b.e[k * 3 + j];
            re = fma(x[k].re, y.re, fma(-x[k].im, y.im, re));
            im = fma(x[k].re, y.im, fma(x[k].im, y.re, im));
        }
        r[j] = {re, im};
    }
}

// a <- a b, row by row (a row of the product needs only that row of a), so that
// no third matrix is live
template <class R>
__device__ __forceinline__ void mm_inplace(Mat3<R> &a, const Mat3<R> &b)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        Cplx<R> r[3];
        const Cplx<R> x[3] = {a.e[i * 3], a.e[i * 3 + 1], a.e[i * 3 + 2]};
        mm_row(x, b, r);
#pragma unroll
        for (int j = 0; j < 3; ++j) a.e[i * 3 + j] = r[j];
    }
}

// H -= eps F at one link from M = U A (FP64, about 20 operations): F = traceless
// part of -(i beta / 6)(M - M^dag), 8 reals with stride Vh.
__device__ __forceinline__ void gauge_kick(const double (&mre)[9], const double (&mim)[9], double *h, int Vh,
                                           double beta6, double eps)
{
    double f[8];
    const double d0 = 2.0 * beta6 * mim[0], d1 = 2.0 * beta6 * mim[4], d2 = 2.0 * beta6 * mim[8];
    const double tr = (d0 + d1 + d2) / 3.0;
    f[0] = d0 - tr;
    f[1] = d1 - tr;
    f[2] = beta6 * (mim[1] + mim[3]);
    f[3] = beta6 * (mre[3] - mre[1]);
    f[4] = beta6 * (mim[2] + mim[6]);
    f[5] = beta6 * (mre[6] - mre[2]);
    f[6] = beta6 * (mim[5] + mim[7]);
    f[7] = beta6 * (mre[7] - mre[5]);
#pragma unroll
    for (int k = 0; k < 8; ++k) h[(size_t)k * Vh] = fma(-eps, f[k], h[(size_t)k * Vh]);
}

// ------------------------------------------------------------------ scalar arithmetic
// One spelling for FP64 and double-float (float2 = hi, lo) reals.
__device__ __forceinline__ double r_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float2 r_fma(float2 a, float2 b, float2 c) { return df_fma(a, b, c); }
__device__ __forceinline__ double r_mul(double a, double b) { return a * b; }
__device__ __forceinline__ float2 r_mul(float2 a, float2 b) { return df_mul(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 r_add(float2 a, float2 b) { return df_add(a, b); }
__device__ __forceinline__ double r_neg(double a) { return -a; }
__device__ __forceinline__ float2 r_neg(float2 a) { return df_neg(a); }
// times a power of two (exact)
__device__ __forceinline__ double r_scale(double a, float p) { return a * (double)p; }
__device__ __forceinline__ float2 r_scale(float2 a, float p) { return make_float2(a.x * p, a.y * p); }
__device__ __forceinline__ float r_hi(double a) { return (float)a; }
__device__ __forceinline__ float r_hi(float2 a) { return a.x; }
template <class R> __device__ __forceinline__ R r_of(double v);
template <> __device__ __forceinline__ double r_of<double>(double v) { return v; }
template <> __device__ __forceinline__ float2 r_of<float2>(double v) { return f64_to_df_slow(v); }

__device__ __forceinline__ double r_double(double a) { return a; }
__device__ __forceinline__ double r_double(float2 a) { return df_to_f64(a); }
__device__ __forceinline__ void mm(const Mat3<double> &a, const Mat3<double> &b, Mat3<double> &c) { mat_mul(a, b, c); }
__device__ __forceinline__ void mm(const DM3 &a, const DM3 &b, DM3 &c) { dm_mul(a, b, c); }

// 1 / n!, rounded to FP64 and split into double-float pairs
constexpr int kExpDegMax = 20;
constexpr double inv_fact(int n) { return n <= 1 ? 1.0 : inv_fact(n - 1) / n; }
__constant__ double c_ifact64[kExpDegMax + 1] = {
    inv_fact(0), inv_fact(1), inv_fact(2), inv_fact(3), inv_fact(4), inv_fact(5), inv_fact(6),
    inv_fact(7), inv_fact(8), inv_fact(9), inv_fact(10), inv_fact(11), inv_fact(12), inv_fact(13),
    inv_fact(14), inv_fact(15), inv_fact(16), inv_fact(17), inv_fact(18), inv_fact(19), inv_fact(20)};
#define LQCD_IFACT_DF(n) {(float)inv_fact(n), (float)(inv_fact(n) - (double)(float)inv_fact(n))}
__constant__ float2 c_ifact_df[kExpDegMax + 1] = {
    LQCD_IFACT_DF(0), LQCD_IFACT_DF(1), LQCD_IFACT_DF(2), LQCD_IFACT_DF(3), LQCD_IFACT_DF(4), LQCD_IFACT_DF(5),
    LQCD_IFACT_DF(6), LQCD_IFACT_DF(7), LQCD_IFACT_DF(8), LQCD_IFACT_DF(9), LQCD_IFACT_DF(10), LQCD_IFACT_DF(11),
    LQCD_IFACT_DF(12), LQCD_IFACT_DF(13), LQCD_IFACT_DF(14), LQCD_IFACT_DF(15), LQCD_IFACT_DF(16),
    LQCD_IFACT_DF(17), LQCD_IFACT_DF(18), LQCD_IFACT_DF(19), LQCD_IFACT_DF(20)};
#undef LQCD_IFACT_DF
template <class R> __device__ __forceinline__ R inv_factorial(int n);
template <> __device__ __forceinline__ double inv_factorial<double>(int n) { return c_ifact64[n]; }
template <> __device__ __forceinline__ float2 inv_factorial<float2>(int n) { return c_ifact_df[n]; }

// ------------------------------------------------------------------ exponential
// exp(iQ) of a traceless Hermitian Q.  By Cayley-Hamilton Q^3 = c1 Q + c0 with
// c1 = Tr Q^2 / 2 and c0 = det Q, so every power series in Q is f0 + f1 Q +
// f2 Q^2: the Taylor series runs on three complex coefficients instead of on
// matrices (multiplying a + b Q + c Q^2 by iQ gives i c c0 + i (a + c c1) Q +
// i b Q^2).  Horner with the coefficients 1/n!, 4 multiply-adds a step; no
// division by eigenvalue differences, so nothing is lost near degenerate
// eigenvalues.  |eigenvalue| <= sqrt(4 c1 / 3) =: r; Q is scaled by 2^-k to
// r <= 1 and the result squared k times.  Degrees: the first term left out
// is below 2^-64 (1/21! at r = 1).
// Horner on matrices instead (17 products and the squarings from norm 1/4)
// took, at 16^4: double-float link update 256 us, now 73 (20 us of memory
// traffic; the rest double-float arithmetic); stout level 1884, now 851, and
// with the block-matrix derivative the local pass of the force chain 5966,
// now 1652 (both bound by the FP64 pipe).
template <class R> struct Herm {
    R d0, d1, d2;                    // diagonal
    Cplx<R> a, b, c;                 // entries 01, 02, 12
};
template <class R> struct ExpF { R ar, ai, br, bi, cr, ci; };   // f0, f1, f2

template <class R>
__device__ __forceinline__ R norm2(const Cplx<R> &z) { return r_fma(z.re, z.re, r_mul(z.im, z.im)); }

template <class R>
__device__ __forceinline__ Herm<R> herm_square(const Herm<R> &q)
{
    Herm<R> s;
    const R na = norm2(q.a), nb = norm2(q.b), nc = norm2(q.c);
    s.d0 = r_fma(q.d0, q.d0, r_add(na, nb));
    s.d1 = r_fma(q.d1, q.d1, r_add(na, nc));
    s.d2 = r_fma(q.d2, q.d2, r_add(nb, nc));
    const R t01 = r_add(q.d0, q.d1), t02 = r_add(q.d0, q.d2), t12 = r_add(q.d1, q.d2);
    // 01: (d0 + d1) a + b conj(c);  02: (d0 + d2) b + a c;  12: (d1 + d2) c + conj(a) b
    s.a.re = r_fma(t01, q.a.re, r_fma(q.b.re, q.c.re, r_mul(q.b.im, q.c.im)));
    s.a.im = r_fma(t01, q.a.im, r_fma(q.b.im, q.c.re, r_neg(r_mul(q.b.re, q.c.im))));
    s.b.re = r_fma(t02, q.b.re, r_fma(q.a.re, q.c.re, r_neg(r_mul(q.a.im, q.c.im))));
    s.b.im = r_fma(t02, q.b.im, r_fma(q.a.re, q.c.im, r_mul(q.a.im, q.c.re)));
    s.c.re = r_fma(t12, q.c.re, r_fma(q.a.re, q.b.re, r_mul(q.a.im, q.b.im)));
    s.c.im = r_fma(t12, q.c.im, r_fma(q.a.re, q.b.im, r_neg(r_mul(q.a.im, q.b.re))));
    return s;
}

template <class R>
__device__ __forceinline__ R herm_det(const Herm<R> &q)
{
    // d0 (d1 d2 - |c|^2) - d1 |b|^2 - d2 |a|^2 + 2 Re(a c conj(b))
    const R m = r_fma(q.d1, q.d2, r_neg(norm2(q.c)));
    R t = r_fma(q.d0, m, r_neg(r_fma(q.d1, norm2(q.b), r_mul(q.d2, norm2(q.a)))));
    const R xr = r_fma(q.a.re, q.c.re, r_neg(r_mul(q.a.im, q.c.im)));
    const R xi = r_fma(q.a.re, q.c.im, r_mul(q.a.im, q.c.re));
    const R y = r_fma(xr, q.b.re, r_mul(xi, q.b.im));
    return r_add(t, r_add(y, y));
}

template <class R>
__device__ __forceinline__ void herm_scale(Herm<R> &q, float p)
{
    q.d0 = r_scale(q.d0, p); q.d1 = r_scale(q.d1, p); q.d2 = r_scale(q.d2, p);
    q.a = {r_scale(q.a.re, p), r_scale(q.a.im, p)};
    q.b = {r_scale(q.b.re, p), r_scale(q.b.im, p)};
    q.c = {r_scale(q.c.re, p), r_scale(q.c.im, p)};
}

// Q scaled to r <= 1 (k halvings), its square S, c0 and c1 of the scaled Q,
// and the degree of the series.
template <class R>
struct ExpArg {
    Herm<R> Q, S;
    R c0, c1;
    int k, deg;
};

template <class R>
__device__ __forceinline__ ExpArg<R> exp_arg(const Herm<R> &q)
{
    ExpArg<R> X;
    X.Q = q;
    X.S = herm_square(q);
    X.c1 = r_scale(r_add(X.S.d0, r_add(X.S.d1, X.S.d2)), 0.5f);
    X.c0 = herm_det(q);
    float r2 = 1.3333334f * r_hi(X.c1);
    X.k = 0;
    while (r2 > 1.f && X.k < 60) {
        r2 *= 0.25f;
        herm_scale(X.Q, 0.5f);
        herm_scale(X.S, 0.25f);
        X.c1 = r_scale(X.c1, 0.25f);
        X.c0 = r_scale(X.c0, 0.125f);
        ++X.k;
    }
    X.deg = r2 <= 1.f / 256 ? 10 : (r2 <= 1.f / 16 ? 13 : kExpDegMax);
    return X;
}

template <class R>
__device__ __forceinline__ ExpF<R> exp_coef(const ExpArg<R> &X)
{
    ExpF<R> f;
    const R zero = r_of<R>(0.0);
    f.ar = inv_factorial<R>(X.deg);
    f.ai = f.br = f.bi = f.cr = f.ci = zero;
#pragma unroll 1
    for (int n = X.deg - 1; n >= 0; --n) {
        const R ar = r_fma(r_neg(f.ci), X.c0, inv_factorial<R>(n)), ai = r_mul(f.cr, X.c0);
        const R br = r_neg(r_fma(f.ci, X.c1, f.ai)), bi = r_fma(f.cr, X.c1, f.ar);
        f.cr = r_neg(f.bi);
        f.ci = f.br;
        f.ar = ar;
        f.ai = ai;
        f.br = br;
        f.bi = bi;
    }
    return f;
}

// E = f0 + f1 Q + f2 S for the entry pair (ij, ji) with Q_ij = q, S_ij = s
template <class R>
__device__ __forceinline__ void exp_pair(const ExpF<R> &f, const Cplx<R> &q, const Cplx<R> &s, Cplx<R> &u, Cplx<R> &l)
{
    const R t1 = r_fma(f.br, q.re, r_mul(f.cr, s.re)), t2 = r_fma(f.bi, q.im, r_mul(f.ci, s.im));
    const R t3 = r_fma(f.br, q.im, r_mul(f.cr, s.im)), t4 = r_fma(f.bi, q.re, r_mul(f.ci, s.re));
    u = {r_add(t1, r_neg(t2)), r_add(t3, t4)};
    l = {r_add(t1, t2), r_add(t4, r_neg(t3))};
}

template <class R>
__device__ __forceinline__ void exp_matrix(const ExpArg<R> &X, const ExpF<R> &f, Mat3<R> &E)
{
    E.e[0] = {r_fma(f.br, X.Q.d0, r_fma(f.cr, X.S.d0, f.ar)), r_fma(f.bi, X.Q.d0, r_fma(f.ci, X.S.d0, f.ai))};
    E.e[4] = {r_fma(f.br, X.Q.d1, r_fma(f.cr, X.S.d1, f.ar)), r_fma(f.bi, X.Q.d1, r_fma(f.ci, X.S.d1, f.ai))};
    E.e[8] = {r_fma(f.br, X.Q.d2, r_fma(f.cr, X.S.d2, f.ar)), r_fma(f.bi, X.Q.d2, r_fma(f.ci, X.S.d2, f.ai))};
    exp_pair(f, X.Q.a, X.S.a, E.e[1], E.e[3]);
    exp_pair(f, X.Q.b, X.S.b, E.e[2], E.e[6]);
    exp_pair(f, X.Q.c, X.S.c, E.e[5], E.e[7]);
}

// E = exp(iQ)
template <class R>
__device__ __forceinline__ void exp_herm(const Herm<R> &Q, Mat3<R> &E)
{
    const ExpArg<R> X = exp_arg(Q);
    const ExpF<R> f = exp_coef(X);
    exp_matrix(X, f, E);
#pragma unroll 1
    for (int q = 0; q < X.k; ++q) {
        Mat3<R> T;
        mm(E, E, T);
        E = T;
    }
}

// t H of 8 reals
template <class R, class T>
__device__ __forceinline__ Herm<R> herm_from(const T (&h)[8], T t)
{
    Herm<R> q;
    q.d0 = r_of<R>((double)(t * h[0]));
    q.d1 = r_of<R>((double)(t * h[1]));
    q.d2 = r_of<R>((double)(-t * (h[0] + h[1])));
    q.a = {r_of<R>((double)(t * h[2])), r_of<R>((double)(t * h[3]))};
    q.b = {r_of<R>((double)(t * h[4])), r_of<R>((double)(t * h[5]))};
    q.c = {r_of<R>((double)(t * h[6])), r_of<R>((double)(t * h[7]))};
    return q;
}

// U <- exp(i eps H) U in double-float (eps H formed in FP64); the product is
// written to the IEEE master and to the df64 copy.
__global__ void __launch_bounds__(kGaugeThreads)
    k_gauge_link_update_df(int Vh, double2 *__restrict__ nat, float4 *__restrict__ Ldf,
                           const double *__restrict__ mom, double eps)
{
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 8L * Vh) return;
    const int i = (int)(t % Vh);
    const int mp = (int)(t / Vh);
    double h[8];
    const double *hp = mom + (size_t)(mp * 8) * Vh + i;
#pragma unroll
    for (int k = 0; k < 8; ++k) h[k] = hp[(size_t)k * Vh];
    DM3 E, U, W;
    exp_herm(herm_from<float2>(h, eps), E);
    dm_load(Ldf, mp >> 1, mp & 1, i, Vh, U);
    dm_mul(E, U, W);
    double2 *pn = nat + (size_t)(mp * 9) * Vh + i;
    float4 *pd = Ldf + (size_t)(mp * 9) * Vh + i;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const float2 re = W.e[c].re, im = W.e[c].im;
        pn[(size_t)c * Vh] = make_double2(df_to_f64(re), df_to_f64(im));
        pd[(size_t)c * Vh] = make_float4(re.x, re.y, im.x, im.y);
    }
}

// ------------------------------------------------------------------ force from stored staples
// The staple sum of the Symanzik action with the plaquette staples as
// intermediates.  For ordered directions (m, n):
//   up_mn(x)   = U_n(x) U_m(x+n) U_n(x+m)^dag            (a path from x to x+m)
//   down_mn(x) = U_n(x-n)^dag U_m(x-n) U_n(x-n+m)
// and the two sides of a link (mu, x) in the plane of nu, as paths X Y Z from
// x + mu back to x, carry their three rectangles as one side bent outwards:
//   c0 X Y Z + c1 (X' Y Z + X Y' Z + X Y Z')
//     = c1 [ (X Y) (Z' - 20 Z) + (X' Y + X Y') Z ]          5 products
// (c0 / c1 = -20; c1 goes into the factor beta / 6)
//   upper: X = U_nu(x+mu), Y = U_mu(x+nu)^dag, Z = U_nu(x)^dag,
//          X' = up_{nu mu}(x+mu), Y' = up_{mu nu}(x+nu)^dag, Z' = down_{nu mu}(x)^dag
//   lower: X = U_nu(x+mu-nu)^dag, Y = U_mu(x-nu)^dag, Z = U_nu(x-nu),
//          X' = up_{nu mu}(x+mu-nu)^dag, Y' = down_{mu nu}(x-nu)^dag, Z' = down_{nu mu}(x-nu)
// A site's 24 staples cost 36 products (a pair shares its first one), its
// links' 24 sides 120: 160 products per site with U A, where the separate
// paths take 340, and 5 neighbour sites per plane instead of 17.  Bound by the
// FP32 pipes (double-float) or the FP64 pipe (native).  Momentum update,
// separate paths -> stored staples: double-float 1542 -> 645 us at 16^4, 7.44 ->
// 3.06 ms at 24^4, 23.2 -> 11.8 at 32^4; native 3750 -> 2207 us at 16^4.
// The staples of np of the six planes at a time are kept (576 bytes per site
// and plane); the force is linear in A, so planes may be added one pass after
// another.
template <class R> struct SideT;
template <> struct SideT<float2> { using t = float4; };
template <> struct SideT<double> { using t = double2; };

struct PlaneRange { int p0, np; };
__device__ __forceinline__ int plane_of(int m, int n)
{
    const int a = m < n ? m : n, b = m < n ? n : m;   // 01 02 03 12 13 23
    return a == 0 ? b - 1 : (a == 1 ? b + 1 : 5);
}
// array number of up_mn (down_mn: + 1) among the stored staples
__device__ __forceinline__ int side_of(const PlaneRange &pr, int m, int n)
{
    return ((plane_of(m, n) - pr.p0) * 2 + (m < n ? 0 : 1)) * 2;
}

// Matrix number k of an array of link layout at a site, or its conjugate
// transpose (read transposed, imaginary parts negated).
__device__ __forceinline__ void load_side(const float4 *__restrict__ L, int k, SiteIdx s, int Vh, bool dag, DM3 &U)
{
    const float4 *p = L + (size_t)((k * 2 + s.par) * 9) * Vh + s.idx;
    const uint32_t neg = dag ? 0x80000000u : 0u;
    const size_t row = (size_t)(dag ? 1 : 3) * Vh, col = (size_t)(dag ? 3 : 1) * Vh;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const float4 v = __ldg(p + (c / 3) * row + (c % 3) * col);
        U.e[c].re = make_float2(v.x, v.y);
        U.e[c].im = xor_sign(make_float2(v.z, v.w), neg);
    }
}
__device__ __forceinline__ void load_side(const double2 *__restrict__ L, int k, SiteIdx s, int Vh, bool dag,
                                          Mat3<double> &U)
{
    const double2 *p = L + (size_t)((k * 2 + s.par) * 9) * Vh + s.idx;
    const uint32_t neg = dag ? 0x80000000u : 0u;
    const size_t row = (size_t)(dag ? 1 : 3) * Vh, col = (size_t)(dag ? 3 : 1) * Vh;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const double2 v = __ldg(p + (c / 3) * row + (c % 3) * col);
        U.e[c] = {v.x, flip_sign(v.y, neg)};
    }
}
__device__ __forceinline__ void store_side(float4 *L, int k, SiteIdx s, int Vh, const DM3 &U)
{
    float4 *p = L + (size_t)((k * 2 + s.par) * 9) * Vh + s.idx;
#pragma unroll
    for (int c = 0; c < 9; ++c) p[(size_t)c * Vh] = make_float4(U.e[c].re.x, U.e[c].re.y, U.e[c].im.x, U.e[c].im.y);
}
__device__ __forceinline__ void store_side(double2 *L, int k, SiteIdx s, int Vh, const Mat3<double> &U)
{
    double2 *p = L + (size_t)((k * 2 + s.par) * 9) * Vh + s.idx;
#pragma unroll
    for (int c = 0; c < 9; ++c) p[(size_t)c * Vh] = make_double2(U.e[c].re, U.e[c].im);
}

// a - 20 b
__device__ __forceinline__ double minus20(double a, double b) { return fma(-20.0, b, a); }
__device__ __forceinline__ float2 minus20(float2 a, float2 b)
{
    float p, e, t, f, h, l;
    two_prod(-20.f, b.x, p, e);
    two_sum(a.x, p, t, f);
    f = __fadd_rn(f, __fadd_rn(a.y, __fmaf_rn(-20.f, b.y, e)));
    fast_two_sum(t, f, h, l);
    return make_float2(h, l);
}

// A thread's matrix in shared memory, [9][kGaugeThreads]: a register matrix
// less is a block more per SM.
__device__ __forceinline__ void put_sm(float4 *s, const DM3 &U)
{
#pragma unroll
    for (int c = 0; c < 9; ++c)
        s[c * kGaugeThreads] = make_float4(U.e[c].re.x, U.e[c].re.y, U.e[c].im.x, U.e[c].im.y);
}
__device__ __forceinline__ void put_sm(double2 *s, const Mat3<double> &U)
{
#pragma unroll
    for (int c = 0; c < 9; ++c) s[c * kGaugeThreads] = make_double2(U.e[c].re, U.e[c].im);
}
__device__ __forceinline__ Cplx<float2> get_sm(const float4 *s, int c)
{
    const float4 v = s[c * kGaugeThreads];
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ Cplx<double> get_sm(const double2 *s, int c)
{
    const double2 v = s[c * kGaugeThreads];
    return {v.x, v.y};
}

__device__ __forceinline__ void put_elem(float4 *s, int c, const DC &v)
{
    s[c * kGaugeThreads] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
}
__device__ __forceinline__ void put_elem(double2 *s, int c, const Cplx<double> &v)
{
    s[c * kGaugeThreads] = make_double2(v.re, v.im);
}
// an element, conjugated if dag
__device__ __forceinline__ DC side_elem(const float4 &v, bool dag)
{
    return {make_float2(v.x, v.y), xor_sign(make_float2(v.z, v.w), dag ? 0x80000000u : 0u)};
}
__device__ __forceinline__ Cplx<double> side_elem(const double2 &v, bool dag)
{
    return {v.x, flip_sign(v.y, dag ? 0x80000000u : 0u)};
}

// M <- M^dag
template <class R>
__device__ __forceinline__ void conj_transpose(Mat3<R> &M)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
            const Cplx<R> a = M.e[i * 3 + j], b = M.e[j * 3 + i];
            M.e[i * 3 + j] = {b.re, r_neg(b.im)};
            M.e[j * 3 + i] = {a.re, r_neg(a.im)};
        }
}

// up_mn(y) or, with down, down_mn(y + n): the products of k_gauge_sides in their order,
// so the same bits as the stored ones.
template <class R>
__device__ __forceinline__ void plaquette_side(const LinkGeo &g, const typename SideT<R>::t *__restrict__ L,
                                               const int (&y)[4], bool down, int m, int n, Mat3<R> &M)
{
    const int p = down ? m : n, q = down ? n : m;
    const SiteIdx s0 = site_step(g, y, p, 0);
    Mat3<R> u;
    load_side(L, p, s0, g.Vh, false, M);
    load_side(L, q, site_step(g, y, p, 1), g.Vh, false, u);
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        mm_inplace(M, u);   // C = U_p(y) U_q(y+p); C U_p(y+q)^dag or U_q(y)^dag C
        if (k == 0 && !down) load_side(L, p, site_step(g, y, q, 1), g.Vh, true, u);
        if (k == 0 && down) {
            u = M;
            load_side(L, q, s0, g.Vh, true, M);
        }
    }
}

// Stored staples of the planes pr: thread = (ordered pair (p, q), parity, site);
// C = U_p(x) U_q(x+p) gives up_qp(x) = C U_p(x+q)^dag and
// down_pq(x+q) = U_q(x)^dag C.  One product in a loop: unrolled, the
// double-float products (about 1300 instructions each) miss the instruction cache.
template <class R>
__global__ void __launch_bounds__(kGaugeThreads, 4)
    k_gauge_sides(LinkGeo g, PlaneRange pr, const typename SideT<R>::t *__restrict__ L, typename SideT<R>::t *__restrict__ F)
{
    __shared__ typename SideT<R>::t s_c[9 * kGaugeThreads];
    const int Vh = g.Vh;
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 4L * pr.np * Vh) return;
    const int i = (int)(t % Vh), w = (int)(t / Vh);
    const int P = w & 1, pl = pr.p0 + (w >> 2), flip = (w >> 1) & 1;
    const int a = pl < 3 ? 0 : (pl < 5 ? 1 : 2), b = pl < 3 ? pl + 1 : (pl < 5 ? pl - 1 : 3);
    const int p = flip ? b : a, q = flip ? a : b;
    int x[4];
    coords_of(g, P, i, x);
    const SiteIdx s0 = {P, i}, sp = site_step(g, x, p, 1), sq = site_step(g, x, q, 1);
    typename SideT<R>::t *C = s_c + threadIdx.x;
    Mat3<R> M, u;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        // M u = U_p(x) U_q(x+p) = C; C U_p(x+q)^dag; U_q(x)^dag C
        if (k != 1) load_side(L, k == 0 ? p : q, s0, Vh, k == 2, M);
        if (k != 2) load_side(L, k == 0 ? q : p, k == 0 ? sp : sq, Vh, k == 1, u);
        if (k == 2) {
#pragma unroll
            for (int c = 0; c < 9; ++c) u.e[c] = get_sm(C, c);
        }
        mm_inplace(M, u);
        if (k == 0) put_sm(C, M);
        else store_side(F, k == 1 ? side_of(pr, q, p) : side_of(pr, p, q) + 1, k == 1 ? s0 : sq, Vh, M);
    }
}

// H_mu(x) -= eps F of the planes pr from the stored staples (F and the update in
// FP64).  A block holds the four directions of 32 sites, which share most of
// the links and staples they read through L1.  Bound by the arithmetic: 31
// products per link, about 1260 FP32 instructions each in double-float, 108 FP64
// ones natively.  A whole double-float product with its sums is 34 KB of code and
// misses the instruction cache (a quarter of the warps' time); by rows it is a
// third of that.  Left factors come by rows too and products go to shared memory,
// so one register matrix is live.  Momentum update, double-float, one GB300: 16^4
// 784 -> 645 us, 24^4 3.81 -> 3.06 ms, 32^4 15.5 -> 11.8, 8^4 102 -> 91.  Three and
// five blocks per SM: 689 and 681 at 16^4.  Native FP64, where the signs of the
// conjugates moved to the integer pipe: 16^4 2543 -> 2207 us.
// STORED = false, for a device without room for the staples: each thread forms
// the three staples of a side when it needs them, 67 products per link, with the
// same bits.  8^4 131 us (99 stored), 16^4 1059 (645), 24^4 5.69 ms (3.06); native
// 307, 3765, 18.4 ms.
template <class R, bool STORED>
__global__ void __launch_bounds__(kGaugeThreads, STORED ? 4 : 2)
    k_gauge_mom_sides(LinkGeo g, PlaneRange pr, const typename SideT<R>::t *__restrict__ L,
                      const typename SideT<R>::t *__restrict__ F, double *__restrict__ mom, double beta6, double eps)
{
    static_assert(kGaugeThreads == 128, "four directions of 32 sites");
    using T = typename SideT<R>::t;
    __shared__ T s_a[9 * kGaugeThreads], s_b[9 * kGaugeThreads];
    const int Vh = g.Vh, nt = (Vh + 31) / 32;
    const int P = (int)blockIdx.x / nt, i = ((int)blockIdx.x - P * nt) * 32 + ((int)threadIdx.x & 31);
    const int mu = (int)threadIdx.x >> 5;
    if (i >= Vh) return;
    int x[4];
    coords_of(g, P, i, x);
    const SiteIdx s0 = {P, i}, sm = site_step(g, x, mu, 1);
    T *A = s_a + threadIdx.x, *B = s_b + threadIdx.x;   // sum of the sides; the product so far
    Mat3<R> u;
    bool any = false;
    // D <- X u (+ Y): X number k of S at s (conjugate transposed if dag), or B if !S;
    // Y = D's place or B, added if add.  Rows in a loop, X's next row loaded before
    // the products of this one.
    auto product = [&](const T *S, int k, SiteIdx s, bool dag, const T *Y, bool add, T *D) {
        const T *p = S ? S + (size_t)((k * 2 + s.par) * 9) * Vh + s.idx : nullptr;
        const size_t row = (size_t)(dag ? 1 : 3) * Vh, col = (size_t)(dag ? 3 : 1) * Vh;
        T nx[3];
        auto fetch = [&](int r) {
#pragma unroll
            for (int c = 0; c < 3; ++c) nx[c] = S ? __ldg(p + r * row + c * col) : B[(r * 3 + c) * kGaugeThreads];
        };
        fetch(0);
#pragma unroll 1
        for (int r = 0; r < 3; ++r) {
            Cplx<R> xr[3], o[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) xr[c] = side_elem(nx[c], dag);
            if (r < 2) fetch(r + 1);
            mm_row(xr, u, o);
            if (add) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const Cplx<R> v = get_sm(Y, r * 3 + c);
                    o[c] = {r_add(v.re, o[c].re), r_add(v.im, o[c].im)};
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) put_elem(D, r * 3 + c, o[c]);
        }
    };
#pragma unroll 1
    for (int w = 0; w < 8; ++w) {
        const int nu = w >> 1, lower = w & 1;
        if (nu == mu) continue;
        const int pl = plane_of(mu, nu);
        if (pl < pr.p0 || pl >= pr.p0 + pr.np) continue;
        const SiteIdx sx = lower ? site_step(g, x, mu, 1, nu, -1) : sm;               // X, X'
        const SiteIdx sy = site_step(g, x, nu, lower ? -1 : 1);                       // Y, Y'
        const SiteIdx sz = lower ? sy : s0;                                           // Z, Z'
        const int kx = side_of(pr, nu, mu), ky = side_of(pr, mu, nu) + lower;
#pragma unroll 1
        for (int k = 0; k < 5; ++k) {
            // B = X Y; A += B (Z' - 20 Z); B = X' Y; B += X Y'; A += B Z
            const bool zz = k == 1 || k == 4;
            Mat3<R> z;   // Z'; X', Y' and Z' where they are not stored
            if constexpr (!STORED) {
                if (k >= 1 && k <= 3) {
                    // X' = up_{nu mu}(x+mu(-nu)), Y' = up_{mu nu}(x+nu) or down_{mu nu}(x-nu), Z' = down_{nu mu}(x(-nu))
                    const int dm = k == 2 ? 1 : (k == 3 ? 0 : -1);
                    const int dn = k == 3 ? (lower ? -2 : 1) : -lower;
                    int y[4];
#pragma unroll
                    for (int d = 0; d < 4; ++d) y[d] = wrap(x[d] + (d == mu ? dm : 0) + (d == nu ? dn : 0), g.N[d]);
                    plaquette_side(g, L, y, k == 1 || (k == 3 && lower), k == 3 ? mu : nu, k == 3 ? nu : mu, z);
                    if (k == 3 || (k == 1) == (lower == 0)) conj_transpose(z);
                    if (k == 2) {
#pragma unroll
                        for (int q = 0; q < 9; ++q) put_elem(B, q, z.e[q]);
                    }
                }
            }
            if constexpr (STORED) {
                load_side(k == 3 ? F : L, k == 3 ? ky : (zz ? nu : mu), zz ? sz : sy, Vh, zz ? lower == 0 : true, u);
                if (k == 1) load_side(F, kx + 1, sz, Vh, lower == 0, z);
            } else {
                if (k == 3) u = z;
                else load_side(L, zz ? nu : mu, zz ? sz : sy, Vh, zz ? lower == 0 : true, u);
            }
            if (k == 1) {
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    u.e[q] = {minus20(z.e[q].re, u.e[q].re), minus20(z.e[q].im, u.e[q].im)};
            }
            T *D = zz ? A : B;
            const bool left = zz || (!STORED && k == 2);   // the left factor is B
            product(left ? nullptr : (k == 2 ? F : L), k == 2 ? kx : nu, sx, !left && lower != 0, D, k == 3 || (zz && any), D);
            any |= zz;
        }
    }
    if (!any) return;
#pragma unroll
    for (int q = 0; q < 9; ++q) u.e[q] = get_sm(A, q);
    product(L, mu, s0, false, B, false, B);
    double mre[9], mim[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const Cplx<R> v = get_sm(B, q);
        mre[q] = r_double(v.re);
        mim[q] = r_double(v.im);
    }
    gauge_kick(mre, mim, mom + (size_t)((mu * 2 + P) * 8) * Vh + i, Vh, beta6 * kSymC1, eps);
}

// IEEE master -> df64 copy (the form k_convert_links writes)
__global__ void k_links_nat_to_df(const double2 *__restrict__ nat, float4 *Ldf, long n)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double2 d = nat[t];
    const float2 re = f64_to_df_slow(d.x), im = f64_to_df_slow(d.y);
    Ldf[t] = make_float4(re.x, re.y, im.x, im.y);
}

// 8 reals <-> traceless Hermitian matrix
template <class T>
__device__ __forceinline__ void herm_unpack(const T (&h)[8], Mat3<T> &H)
{
    H.e[0] = {h[0], T(0)};
    H.e[4] = {h[1], T(0)};
    H.e[8] = {-h[0] - h[1], T(0)};
    H.e[1] = {h[2], h[3]};
    H.e[3] = {h[2], -h[3]};
    H.e[2] = {h[4], h[5]};
    H.e[6] = {h[4], -h[5]};
    H.e[5] = {h[6], h[7]};
    H.e[7] = {h[6], -h[7]};
}

template <class T>
__device__ __forceinline__ const T *mom_ptr(const T *m, int mu, int P, int Vh)
{
    return m + (size_t)((mu * 2 + P) * 8) * Vh;
}

// H_mu(x) -= eps F_mu(x) for every link.  A block holds the four directions of
// 32 sites (thread = (mu, site), blocks ordered by parity and site): they share
// most of the links they read, through L1.  Read straight into registers, the
// links' way from L2 bounds it (some 75 links of 72 bytes per link in FP32, at
// eleven warps per SM); through the ring their latency is spent under the
// products, and L1's data path bounds it (81 % busy: in and out of the ring).
// FP32, one GB300: 32^4 2180 -> 1858 us, 24^4 703 -> 625, 16^4 140 -> 131, a step
// at 8^4 24.8 -> 22.8 (of which 64-bit offsets 21 and 4 us).  (One direction per block, no ring: 24^4 862.)  Rings of
// three and four slots, three and four blocks per SM: 24^4 626 / 621 and 621 /
// 636; some links through the ring and some straight: 619 to 679, slower at
// 32^4; bodies of their own for s = -1 and s = +1, without selections, outgrow the
// instruction cache: 667.
__global__ void __launch_bounds__(kGaugeThreads, 3)
    k_gauge_mom_update_f32(LinkGeo g, const float2 *__restrict__ L, float *__restrict__ mom, float beta6, float eps)
{
    using T = float;
    static_assert(kGaugeThreads == 128, "four directions of 32 sites");
    const int Vh = g.Vh, nt = (Vh + 31) / 32;
    const int P = (int)blockIdx.x / nt, i = ((int)blockIdx.x - P * nt) * 32 + ((int)threadIdx.x & 31);
    const int mu = (int)threadIdx.x >> 5, mp = mu * 2 + P;
    if (i >= Vh) return;
    int x[4];
    coords_of(g, P, i, x);
    Mat3<T> A, U, M;
    __shared__ LinkRing ring;
    staple_sum_f32(g, L, ring, x, P, i, mu, A);
    load_link_soa<T>(L, mu, P, i, Vh, U);
    mat_mul(U, A, M);
    // F = -(i beta/6)(M - M^dag): F_ij = (beta/6) * (i (conj(M_ji) - M_ij))
    //   re F_ij = (beta/6) (M_ij.im + M_ji.im),  im F_ij = (beta/6) (M_ji.re - M_ij.re)
    T f[8];
    const T d0 = beta6 * (M.e[0].im + M.e[0].im), d1 = beta6 * (M.e[4].im + M.e[4].im),
            d2 = beta6 * (M.e[8].im + M.e[8].im);
    const T tr = (d0 + d1 + d2) / T(3);
    f[0] = d0 - tr;
    f[1] = d1 - tr;
    f[2] = beta6 * (M.e[1].im + M.e[3].im);
    f[3] = beta6 * (M.e[3].re - M.e[1].re);
    f[4] = beta6 * (M.e[2].im + M.e[6].im);
    f[5] = beta6 * (M.e[6].re - M.e[2].re);
    f[6] = beta6 * (M.e[5].im + M.e[7].im);
    f[7] = beta6 * (M.e[7].re - M.e[5].re);
    T *h = mom + (size_t)(mp * 8) * Vh + i;
#pragma unroll
    for (int k = 0; k < 8; ++k) h[(size_t)k * Vh] = fma(-eps, f[k], h[(size_t)k * Vh]);
}

// E = exp(i t H) in FP32: Z = i t H scaled by 2^-k to 1-norm <= 1/4, Taylor
// series of degree 9 on the matrix, squared k times.  exp_herm rounds
// differently (2e-7 after 40 steps), and an FP32 trajectory is kept
// reproducible to the bit; the update is 8 % of an FP32 step.
__device__ __forceinline__ void exp_iH_f32(const Mat3<float> &H, float t, Mat3<float> &E)
{
    using T = float;
    T nrm = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        T c = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) c += sqrt(H.e[i * 3 + j].re * H.e[i * 3 + j].re + H.e[i * 3 + j].im * H.e[i * 3 + j].im);
        nrm = c > nrm ? c : nrm;
    }
    nrm *= fabs(t);
    int k = 0;
    while (nrm > T(0.25) && k < 60) {
        nrm *= T(0.5);
        ++k;
    }
    T sc = t;
    for (int q = 0; q < k; ++q) sc *= T(0.5);
    Mat3<T> Z;
#pragma unroll
    for (int q = 0; q < 9; ++q) Z.e[q] = {-sc * H.e[q].im, sc * H.e[q].re};
    // Horner: E = I + Z (I + Z/2 (I + Z/3 (... (I + Z/n))))
    constexpr int deg = 9;
    Mat3<T> R;
#pragma unroll
    for (int q = 0; q < 9; ++q) R.e[q] = {(q % 4 == 0) ? T(1) : T(0), T(0)};
#pragma unroll 1
    for (int n = deg; n >= 1; --n) {
        Mat3<T> ZR;
        mat_mul(Z, R, ZR);
        const T inv = T(1) / T(n);
#pragma unroll
        for (int q = 0; q < 9; ++q) R.e[q] = {((q % 4 == 0) ? T(1) : T(0)) + inv * ZR.e[q].re, inv * ZR.e[q].im};
    }
#pragma unroll 1
    for (int q = 0; q < k; ++q) {
        Mat3<T> S2;
        mat_mul(R, R, S2);
        R = S2;
    }
    E = R;
}

// U_mu(x) <- exp(i eps H_mu(x)) U_mu(x) for every link.
template <class T>
__global__ void __launch_bounds__(kGaugeThreads)
    k_gauge_link_update(int Vh, typename Vec2T<T>::t *__restrict__ L, const T *__restrict__ mom, T eps)
{
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 8L * Vh) return;
    const int i = (int)(t % Vh);
    const int mp = (int)(t / Vh);
    T h[8];
    const T *hp = mom + (size_t)(mp * 8) * Vh + i;
#pragma unroll
    for (int k = 0; k < 8; ++k) h[k] = hp[(size_t)k * Vh];
    Mat3<T> E, U, R;
    if constexpr (sizeof(T) == 4) {
        Mat3<T> H;
        herm_unpack(h, H);
        exp_iH_f32(H, eps, E);
    } else {
        exp_herm(herm_from<T>(h, eps), E);
    }
    typename Vec2T<T>::t *p = L + (size_t)(mp * 9) * Vh + i;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const typename Vec2T<T>::t v = p[(size_t)c * Vh];
        U.e[c] = {v.x, v.y};
    }
    mat_mul(E, U, R);
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        typename Vec2T<T>::t v;
        v.x = R.e[c].re;
        v.y = R.e[c].im;
        p[(size_t)c * Vh] = v;
    }
}

// U_dir(x + d)
template <class T>
__device__ __forceinline__ void link_at(const LinkGeo &g, const typename Vec2T<T>::t *L, const int (&x)[4], int d0,
                                        int d1, int d2, int d3, int dir, Mat3<T> &U)
{
    int par, idx;
    site_of(g, x, d0, d1, d2, d3, par, idx);
    load_link_soa<T>(L, dir, par, idx, g.Vh, U);
}

// Per-block partial of sum_x [c0 sum_{mu<nu} Re Tr P + c1 sum_{mu!=nu} Re Tr R]
// (FP64 accumulation); thread = site (parity, half index):
//   P = U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
//   R = U_mu(x) U_mu(x+mu) U_nu(x+2mu) U_mu(x+mu+nu)^dag U_mu(x+nu)^dag U_nu(x)^dag
template <class T>
__global__ void __launch_bounds__(kGaugeThreads)
    k_gauge_action_part(LinkGeo g, const typename Vec2T<T>::t *__restrict__ L, double *part)
{
    __shared__ double s_red[kGaugeThreads / 32];
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    double acc = 0.0;
    if (t < 2L * g.Vh) {
        const int P = (int)(t / g.Vh), i = (int)(t % g.Vh);
        int x[4];
        coords_of(g, P, i, x);
        double sp = 0.0, sr = 0.0;
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu)
#pragma unroll 1
            for (int nu = 0; nu < 4; ++nu) {
                if (nu == mu) continue;
                int em[4] = {0, 0, 0, 0}, en[4] = {0, 0, 0, 0};
                em[mu] = 1;
                en[nu] = 1;
                Mat3<T> u, b, c, d;
                link_at<T>(g, L, x, 0, 0, 0, 0, mu, u);
                if (mu < nu) {
                    link_at<T>(g, L, x, em[0], em[1], em[2], em[3], nu, b);
                    mat_mul(u, b, c);
                    link_at<T>(g, L, x, en[0], en[1], en[2], en[3], mu, b);
                    mat_mul_dag(c, b, d);
                    link_at<T>(g, L, x, 0, 0, 0, 0, nu, b);
                    mat_mul_dag(d, b, c);
                    sp += (double)c.e[0].re + (double)c.e[4].re + (double)c.e[8].re;
                }
                link_at<T>(g, L, x, em[0], em[1], em[2], em[3], mu, b);
                mat_mul(u, b, c);
                link_at<T>(g, L, x, 2 * em[0], 2 * em[1], 2 * em[2], 2 * em[3], nu, b);
                mat_mul(c, b, d);
                link_at<T>(g, L, x, em[0] + en[0], em[1] + en[1], em[2] + en[2], em[3] + en[3], mu, b);
                mat_mul_dag(d, b, c);
                link_at<T>(g, L, x, en[0], en[1], en[2], en[3], mu, b);
                mat_mul_dag(c, b, d);
                link_at<T>(g, L, x, 0, 0, 0, 0, nu, b);
                mat_mul_dag(d, b, c);
                sr += (double)c.e[0].re + (double)c.e[4].re + (double)c.e[8].re;
            }
        acc = kSymC0 * sp + kSymC1 * sr;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kGaugeThreads / 32; ++k) s += s_red[k];
        part[blockIdx.x] = s;
    }
}

// Per-block partial of (1/2) sum Tr H^2.
template <class T>
__global__ void __launch_bounds__(kGaugeThreads) k_mom_energy_part(int Vh, const T *__restrict__ mom, double *part)
{
    __shared__ double s_red[kGaugeThreads / 32];
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    double acc = 0.0;
    if (t < 8L * Vh) {
        const int i = (int)(t % Vh), mp = (int)(t / Vh);
        const T *hp = mom + (size_t)(mp * 8) * Vh + i;
        double h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) h[k] = (double)hp[(size_t)k * Vh];
        const double d2 = -h[0] - h[1];
        acc = 0.5 * (h[0] * h[0] + h[1] * h[1] + d2 * d2 +
                     2.0 * (h[2] * h[2] + h[3] * h[3] + h[4] * h[4] + h[5] * h[5] + h[6] * h[6] + h[7] * h[7]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kGaugeThreads / 32; ++k) s += s_red[k];
        part[blockIdx.x] = s;
    }
}

// One block: sum of part[0..n) in a fixed order.
__global__ void __launch_bounds__(256) k_gauge_sum_ordered(const double *__restrict__ part, int n, double *out)
{
    __shared__ double s_red[8];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += 256) s += part[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int k = 0; k < 8; ++k) tot += s_red[k];
        *out = tot;
    }
}

// ------------------------------------------------------------------ format conversions
// canonical host momenta [4][V][3][3] complex128 (staged on the device) -> 8 reals SoA (FP64 and FP32)
__global__ void k_mom_from_canonical(LinkGeo g, const double2 *__restrict__ src, double *m64, float *m32, int *bad,
                                     long V)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= 4 * V) return;
    const int mu = (int)(t / V);
    const long lex = t - (long)mu * V;
    int x[4];
    long r = lex;
    for (int m = 0; m < 4; ++m) {
        x[m] = (int)(r % g.N[m]);
        r /= g.N[m];
    }
    const int P = (x[0] + x[1] + x[2] + x[3]) & 1;
    const int idx = (int)(lex >> 1);
    const double2 *h = src + t * 9;
    // Hermitian and traceless to 1e-12 relative, else rejected
    double scale = 0.0;
    for (int c = 0; c < 9; ++c) scale = fmax(scale, fmax(fabs(h[c].x), fabs(h[c].y)));
    const double tol = 1e-12 * fmax(scale, 1e-300);
    bool ok = isfinite(scale) && fabs(h[0].y) <= tol && fabs(h[4].y) <= tol && fabs(h[8].y) <= tol &&
              fabs(h[0].x + h[4].x + h[8].x) <= 3 * tol;
    const int off[3][2] = {{1, 3}, {2, 6}, {5, 7}};
    for (int q = 0; q < 3; ++q)
        ok = ok && fabs(h[off[q][0]].x - h[off[q][1]].x) <= tol && fabs(h[off[q][0]].y + h[off[q][1]].y) <= tol;
    if (!ok) atomicOr(bad, 1);
    const double v[8] = {h[0].x, h[4].x, h[1].x, h[1].y, h[2].x, h[2].y, h[5].x, h[5].y};
    for (int k = 0; k < 8; ++k) {
        const size_t o = (size_t)((mu * 2 + P) * 8 + k) * g.Vh + idx;
        m64[o] = v[k];
        if (m32) m32[o] = (float)v[k];
    }
}

template <class T>
__global__ void k_mom_to_canonical(LinkGeo g, const T *__restrict__ m, double2 *dst, long V)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= 4 * V) return;
    const int mu = (int)(t / V);
    const long lex = t - (long)mu * V;
    int x[4];
    long r = lex;
    for (int q = 0; q < 4; ++q) {
        x[q] = (int)(r % g.N[q]);
        r /= g.N[q];
    }
    const int P = (x[0] + x[1] + x[2] + x[3]) & 1;
    const int idx = (int)(lex >> 1);
    double h[8];
    for (int k = 0; k < 8; ++k) h[k] = (double)m[(size_t)((mu * 2 + P) * 8 + k) * g.Vh + idx];
    double2 *o = dst + t * 9;
    o[0] = make_double2(h[0], 0.0);
    o[4] = make_double2(h[1], 0.0);
    o[8] = make_double2(-h[0] - h[1], 0.0);
    o[1] = make_double2(h[2], h[3]);
    o[3] = make_double2(h[2], -h[3]);
    o[2] = make_double2(h[4], h[5]);
    o[6] = make_double2(h[4], -h[5]);
    o[5] = make_double2(h[6], h[7]);
    o[7] = make_double2(h[6], -h[7]);
}

// FP64 <-> FP32 copies of links (SoA, same layout) and momenta
__global__ void k_links_f64_to_f32(const double2 *__restrict__ a, float2 *b, long n)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < n) b[t] = make_float2((float)a[t].x, (float)a[t].y);
}
__global__ void k_links_f32_to_f64(const float2 *__restrict__ a, double2 *b, long n)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < n) b[t] = make_double2((double)a[t].x, (double)a[t].y);
}
__global__ void k_mom_f64_to_f32(const double *__restrict__ a, float *b, long n)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < n) b[t] = (float)a[t];
}
__global__ void k_mom_f32_to_f64(const float *__restrict__ a, double *b, long n)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < n) b[t] = (double)a[t];
}

// ------------------------------------------------------------------ fermion force
// Force of the rational pseudofermion action S_f = phi^dag r(A) phi
// (Sec. 2.2, Eqs. rooting, shlineq), from x_i = (A + sigma_i)^{-1} phi (even
// sites) and y_i = D_oe x_i (odd sites):
//   F_mu(n) = traceless part of (i s_mu(n) / 2) c sum_i a_i (W_i - W_i^dag),
//   n even: W_i = U_mu(n) y_i(n+mu) x_i(n)^dag (c = +1); n odd: W_i = U_mu(n) x_i(n+mu) y_i(n)^dag (c = -1);
// and H -= eps F.  One thread per link, native FP64 (about 36 n + 110 FMAs).
struct FFCoef {
    double a[kMaxShifts];
    int n;
};

__global__ void __launch_bounds__(kGaugeThreads)
    k_fermion_force_update(Geom g, const double2 *__restrict__ L, const double2 *__restrict__ x,
                           const double2 *__restrict__ y, const __grid_constant__ FFCoef C, double *__restrict__ mom,
                           double eps)
{
    const int Vh = g.Vh;
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 8L * Vh) return;
    const int i = (int)(t % Vh);
    const int mp = (int)(t / Vh);
    const int mu = mp >> 1, P = mp & 1;
    Stencil S;
    make_stencil(g, i, P, S);
    int f, b;
    uint32_t nf, nb;
    hop(g, S, mu, f, b, nf, nb);
    const double sgn = nf ? -1.0 : 1.0;            // s_mu(n): staggered phase and time boundary
    const double2 *left = P == 0 ? y : x;          // field at n + mu
    const double2 *right = P == 0 ? x : y;         // field at n
    const size_t n3 = 3 * (size_t)Vh;
    double2 O[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) O[q] = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int k = 0; k < C.n; ++k) {
        double2 l[3], r[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            l[c] = __ldg(left + k * n3 + (size_t)c * Vh + f);
            r[c] = __ldg(right + k * n3 + (size_t)c * Vh + i);
        }
        const double ak = C.a[k];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                // a_k l_p conj(r_q)
                const double re = l[p].x * r[q].x + l[p].y * r[q].y;
                const double im = l[p].y * r[q].x - l[p].x * r[q].y;
                O[p * 3 + q].x = fma(ak, re, O[p * 3 + q].x);
                O[p * 3 + q].y = fma(ak, im, O[p * 3 + q].y);
            }
    }
    double2 U[9];
    const double2 *lp = L + link_base(mu, P, 9, Vh) + i;
#pragma unroll
    for (int c = 0; c < 9; ++c) U[c] = __ldg(lp + (size_t)c * Vh);
    double2 W[9];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            double re = 0.0, im = 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double2 u = U[p * 3 + k], o = O[k * 3 + q];
                re = fma(u.x, o.x, fma(-u.y, o.y, re));
                im = fma(u.x, o.y, fma(u.y, o.x, im));
            }
            W[p * 3 + q] = make_double2(re, im);
        }
    // F = (i h)(W - W^dag), h = s c / 2:  re F_pq = -h (Im W_pq + Im W_qp),  im F_pq = h (Re W_pq - Re W_qp)
    const double hsc = 0.5 * sgn * (P == 0 ? 1.0 : -1.0);
    const double d0 = -2.0 * hsc * W[0].y, d1 = -2.0 * hsc * W[4].y, d2 = -2.0 * hsc * W[8].y;
    const double tr = (d0 + d1 + d2) / 3.0;
    double fv[8];
    fv[0] = d0 - tr;
    fv[1] = d1 - tr;
    fv[2] = -hsc * (W[1].y + W[3].y);
    fv[3] = hsc * (W[1].x - W[3].x);
    fv[4] = -hsc * (W[2].y + W[6].y);
    fv[5] = hsc * (W[2].x - W[6].x);
    fv[6] = -hsc * (W[5].y + W[7].y);
    fv[7] = hsc * (W[5].x - W[7].x);
    double *h = mom + (size_t)(mp * 8) * Vh + i;
#pragma unroll
    for (int k = 0; k < 8; ++k) h[(size_t)k * Vh] = fma(-eps, fv[k], h[(size_t)k * Vh]);
}

// ------------------------------------------------------------------ stout smearing
// Stout smearing of the links (Sec. 2.1, stout-improved staggered action,
// after Morningstar and Peardon), isotropic weight rho per level:
//   C_mu(x) = rho sum_{nu != mu} [ U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
//                                 + U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu) ],
//   Omega = C U^dag, Q = (i/2)(Omega^dag - Omega) - (i/6) Tr(Omega^dag - Omega),
//   U' = exp(iQ) U.
// Native FP64, one thread per link, the SoA layout of the IEEE links.

__device__ __forceinline__ void stout_C(const LinkGeo &g, const double2 *L, const int (&x)[4], int mu, double rho,
                                        Mat3<double> &C)
{
#pragma unroll
    for (int q = 0; q < 9; ++q) C.e[q] = {0.0, 0.0};
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        int dn[4] = {0, 0, 0, 0}, dm[4] = {0, 0, 0, 0}, dmn[4] = {0, 0, 0, 0};
        dn[nu] = 1;
        dm[mu] = 1;
        dmn[mu] = 1;
        dmn[nu] = -1;
        Mat3<double> a, b, t;
        // upper: U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
        link_at<double>(g, L, x, 0, 0, 0, 0, nu, a);
        link_at<double>(g, L, x, dn[0], dn[1], dn[2], dn[3], mu, b);
        mat_mul(a, b, t);
        link_at<double>(g, L, x, dm[0], dm[1], dm[2], dm[3], nu, a);
        mat_mul_dag_add(t, a, C);
        // lower: U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
        link_at<double>(g, L, x, -dn[0], -dn[1], -dn[2], -dn[3], nu, a);
        mat_dag(a);
        link_at<double>(g, L, x, -dn[0], -dn[1], -dn[2], -dn[3], mu, b);
        mat_mul(a, b, t);
        link_at<double>(g, L, x, dmn[0], dmn[1], dmn[2], dmn[3], nu, a);
        mat_mul_add(t, a, C);
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) C.e[q] = {rho * C.e[q].re, rho * C.e[q].im};
}

// Q from C and U (Hermitian, traceless)
__device__ __forceinline__ Herm<double> stout_Q(const Mat3<double> &C, const Mat3<double> &U)
{
    Mat3<double> Om;
    mat_mul_dag(C, U, Om);
    // Q_ij = (i/2)(conj(Om_ji) - Om_ij):  re = (Om_ij.im + Om_ji.im)/2, im = (Om_ji.re - Om_ij.re)/2
    auto q = [&](int ij, int ji) -> Cplx<double> {
        return {0.5 * (Om.e[ij].im + Om.e[ji].im), 0.5 * (Om.e[ji].re - Om.e[ij].re)};
    };
    const double tr = (Om.e[0].im + Om.e[4].im + Om.e[8].im) / 3.0;
    Herm<double> Q;
    Q.d0 = Om.e[0].im - tr;
    Q.d1 = Om.e[4].im - tr;
    Q.d2 = Om.e[8].im - tr;
    Q.a = q(1, 3);
    Q.b = q(2, 6);
    Q.c = q(5, 7);
    return Q;
}

// complex helpers (FP64)
using Cd = Cplx<double>;
__device__ __forceinline__ Cd c_mul(Cd a, Cd b) { return {fma(a.re, b.re, -a.im * b.im), fma(a.re, b.im, a.im * b.re)}; }
__device__ __forceinline__ Cd c_fma(Cd a, Cd b, Cd c)
{
    return {fma(a.re, b.re, fma(-a.im, b.im, c.re)), fma(a.re, b.im, fma(a.im, b.re, c.im))};
}

__device__ __forceinline__ void herm_matrix(const Herm<double> &q, Mat3<double> &M)
{
    M.e[0] = {q.d0, 0.0};
    M.e[4] = {q.d1, 0.0};
    M.e[8] = {q.d2, 0.0};
    M.e[1] = q.a;
    M.e[3] = {q.a.re, -q.a.im};
    M.e[2] = q.b;
    M.e[6] = {q.b.re, -q.b.im};
    M.e[5] = q.c;
    M.e[7] = {q.c.re, -q.c.im};
}

// Tr(Q B) for a Hermitian Q
__device__ __forceinline__ Cd herm_trace(const Herm<double> &q, const Mat3<double> &B)
{
    Cd t = {fma(q.d0, B.e[0].re, fma(q.d1, B.e[4].re, q.d2 * B.e[8].re)),
            fma(q.d0, B.e[0].im, fma(q.d1, B.e[4].im, q.d2 * B.e[8].im))};
    auto pair = [&](const Cd &z, int ij, int ji) {  // Q_ij B_ji + conj(Q_ij) B_ij
        t = c_fma(z, B.e[ji], t);
        t = c_fma(Cd{z.re, -z.im}, B.e[ij], t);
    };
    pair(q.a, 1, 3);
    pair(q.b, 2, 6);
    pair(q.c, 5, 7);
    return t;
}

// E = exp(iQ) and D = d/dt exp(iQ + t A) at t = 0.  With A = i (B + beta 1),
// Tr B = 0: D = i beta E + df0 + df1 Q + df2 Q^2 + f1 B + f2 (Q B + B Q), where
// df_j = (df_j/dc1) Tr(Q B) + (df_j/dc0) Tr(Q^2 B) (the differentials of
// c1 = Tr Q^2 / 2 and c0 = Tr Q^3 / 3 along a traceless B).  The series and its
// two derivatives run on scalars (exp_coef's recurrence, differentiated);
// what is left of the 66 matrix products of a block-matrix series are Q B
// and B Q.  k halvings are undone by (E, D) <- (E E, E D + D E).
__device__ void exp_frechet_dev(const Herm<double> &Q, const Mat3<double> &A, Mat3<double> &E, Mat3<double> &D)
{
    const ExpArg<double> X = exp_arg(Q);
    // value (a, b, c), derivative by c1 (p, q, r) and by c0 (x, y, z)
    Cd a = {inv_factorial<double>(X.deg), 0.0}, b = {0, 0}, c = {0, 0};
    Cd p = {0, 0}, q = {0, 0}, r = {0, 0}, x = {0, 0}, y = {0, 0}, z = {0, 0};
    auto times_i = [](Cd v) -> Cd { return {-v.im, v.re}; };
    auto axpy = [](double s, Cd v, Cd w) -> Cd { return {fma(s, v.re, w.re), fma(s, v.im, w.im)}; };
#pragma unroll 1
    for (int n = X.deg - 1; n >= 0; --n) {
        const Cd a1 = times_i({c.re * X.c0, c.im * X.c0}), b1 = times_i(axpy(X.c1, c, a)), c1 = times_i(b);
        const Cd p1 = times_i({r.re * X.c0, r.im * X.c0});
        const Cd q1 = times_i(axpy(X.c1, r, {p.re + c.re, p.im + c.im})), r1 = times_i(q);
        const Cd x1 = times_i(axpy(X.c0, z, c)), y1 = times_i(axpy(X.c1, z, x)), z1 = times_i(y);
        a = {a1.re + inv_factorial<double>(n), a1.im};
        b = b1; c = c1;
        p = p1; q = q1; r = r1;
        x = x1; y = y1; z = z1;
    }
    const ExpF<double> f = {a.re, a.im, b.re, b.im, c.re, c.im};
    exp_matrix(X, f, E);
    // -i A / 2^k = B + beta 1
    const double sc = ldexp(1.0, -X.k);
    Mat3<double> B, H, T;
#pragma unroll
    for (int e = 0; e < 9; ++e) B.e[e] = {sc * A.e[e].im, -sc * A.e[e].re};
    const Cd beta = {(B.e[0].re + B.e[4].re + B.e[8].re) / 3.0, (B.e[0].im + B.e[4].im + B.e[8].im) / 3.0};
#pragma unroll
    for (int e = 0; e < 9; e += 4) B.e[e] = {B.e[e].re - beta.re, B.e[e].im - beta.im};
    const Cd t1 = herm_trace(X.Q, B), t0 = herm_trace(X.S, B);
    const Cd g0 = c_fma(p, t1, c_mul(x, t0)), g1 = c_fma(q, t1, c_mul(y, t0)), g2 = c_fma(r, t1, c_mul(z, t0));
    const Cd ib = times_i(beta);
    herm_matrix(X.Q, H);
    mat_mul(H, B, T);
    mat_mul(B, H, D);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const Cd g = {T.e[e].re + D.e[e].re, T.e[e].im + D.e[e].im};
        Cd v = c_fma(c, g, c_fma(b, B.e[e], c_mul(ib, E.e[e])));
        v = c_fma(g1, H.e[e], v);
        D.e[e] = v;
    }
    herm_matrix(X.S, H);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        D.e[e] = c_fma(g2, H.e[e], D.e[e]);
        if (e % 4 == 0) D.e[e] = {D.e[e].re + g0.re, D.e[e].im + g0.im};
    }
#pragma unroll 1
    for (int k = 0; k < X.k; ++k) {
        mat_mul(E, D, T);
        mat_mul(D, E, H);
#pragma unroll
        for (int e = 0; e < 9; ++e) D.e[e] = {T.e[e].re + H.e[e].re, T.e[e].im + H.e[e].im};
        mat_mul(E, E, T);
        E = T;
    }
}

__device__ __forceinline__ void store_link_soa(double2 *L, int mu, int P, int i, int Vh, const Mat3<double> &U)
{
    double2 *p = L + (size_t)((mu * 2 + P) * 9) * Vh + i;
#pragma unroll
    for (int c = 0; c < 9; ++c) p[(size_t)c * Vh] = make_double2(U.e[c].re, U.e[c].im);
}

// Lout = one stout level of Lin.  Thread = (mu, parity, site).
__global__ void __launch_bounds__(kGaugeThreads)
    k_stout_level(LinkGeo g, const double2 *__restrict__ Lin, double2 *__restrict__ Lout, double rho)
{
    const int Vh = g.Vh;
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 8L * Vh) return;
    const int i = (int)(t % Vh);
    const int mp = (int)(t / Vh);
    const int mu = mp >> 1, P = mp & 1;
    int x[4];
    coords_of(g, P, i, x);
    Mat3<double> C, U, E, R;
    stout_C(g, Lin, x, mu, rho, C);
    load_link_soa<double>(Lin, mu, P, i, Vh, U);
    exp_herm(stout_Q(C, U), E);
    mat_mul(E, U, R);
    store_link_soa(Lout, mu, P, i, Vh, R);
}

// First pass of the force chain of one level (the force on U' = smear(U),
// Fp as 8 reals per link, to the force on U): per link
//   Sigma' = -i U'^dag Fp,  Gamma = Dexp_{iQ}[U Sigma'],  L = traceless
//   anti-Hermitian part of Gamma,
//   Gl = Sigma' exp(iQ) - C^dag L  (the link's own terms of the gradient),
//   M = U^dag L                    (what the staples of C carry to their links).
__global__ void __launch_bounds__(kGaugeThreads)
    k_stout_local(LinkGeo g, const double2 *__restrict__ L, const double *__restrict__ Fp, double rho,
                  double2 *__restrict__ Mout, double2 *__restrict__ Gl)
{
    const int Vh = g.Vh;
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 8L * Vh) return;
    const int i = (int)(t % Vh);
    const int mp = (int)(t / Vh);
    const int mu = mp >> 1, P = mp & 1;
    int x[4];
    coords_of(g, P, i, x);
    Mat3<double> C, U, E, D, W, S, F;
    stout_C(g, L, x, mu, rho, C);
    load_link_soa<double>(L, mu, P, i, Vh, U);
    const Herm<double> Q = stout_Q(C, U);
    double h[8];
    const double *hp = Fp + (size_t)(mp * 8) * Vh + i;
#pragma unroll
    for (int k = 0; k < 8; ++k) h[k] = hp[(size_t)k * Vh];
    herm_unpack(h, F);
    exp_herm(Q, E);
    mat_mul(E, U, W);  // U'
    // S = -i U'^dag F
    mat_dag(W);
    mat_mul(W, F, S);
#pragma unroll
    for (int q = 0; q < 9; ++q) S.e[q] = {S.e[q].im, -S.e[q].re};
    Mat3<double> US;
    mat_mul(U, S, US);
    exp_frechet_dev(Q, US, E, D);
    // L = (D - D^dag)/2 - Tr(D - D^dag)/6
    Mat3<double> Lm;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            Lm.e[a * 3 + b] = {0.5 * (D.e[a * 3 + b].re - D.e[b * 3 + a].re),
                               0.5 * (D.e[a * 3 + b].im + D.e[b * 3 + a].im)};
    const double tri = (Lm.e[0].im + Lm.e[4].im + Lm.e[8].im) / 3.0;
    Lm.e[0].im -= tri;
    Lm.e[4].im -= tri;
    Lm.e[8].im -= tri;
    // Gl = S E - C^dag L
    Mat3<double> SE, CdL, Cd = C;
    mat_mul(S, E, SE);
    mat_dag(Cd);
    mat_mul(Cd, Lm, CdL);
#pragma unroll
    for (int q = 0; q < 9; ++q) SE.e[q] = {SE.e[q].re - CdL.e[q].re, SE.e[q].im - CdL.e[q].im};
    store_link_soa(Gl, mu, P, i, Vh, SE);
    // M = U^dag L
    Mat3<double> Ud = U, M;
    mat_dag(Ud);
    mat_mul(Ud, Lm, M);
    store_link_soa(Mout, mu, P, i, Vh, M);
}

// Second pass: each link (y, l) gathers the staple terms that carry M of the
// links whose C contains it (rho times, for every mu != l and nu != l):
//   U_mu(y+l) U_l(y+mu)^dag M_mu(y)            U_mu(y-mu+l)^dag U_l(y-mu)^dag M_mu(y-mu)^dag
//   M_mu(y+l)^dag U_l(y+mu)^dag U_mu(y)^dag    M_mu(y+l-mu) U_l(y-mu)^dag U_mu(y-mu)
//   U_nu(y-nu+l)^dag M_l(y-nu) U_nu(y-nu)      U_nu(y+l) M_l(y+nu) U_nu(y)^dag
// (the terms that end in the same link share its product: 10 products for the
// six terms instead of 12: 1980 -> 1692 us at 16^4, FP64 pipe; products summed
// where they are formed instead of by 18 more FMAs each: 1495), adds the link's own terms Gl and writes the force on the link,
//   F = traceless part of (i/2)(U G - G^dag U^dag), as 8 reals.
__global__ void __launch_bounds__(kGaugeThreads)
    k_stout_gather(LinkGeo g, const double2 *__restrict__ L, const double2 *__restrict__ M,
                   const double2 *__restrict__ Gl, double rho, double *__restrict__ Fout)
{
    const int Vh = g.Vh;
    const long t = blockIdx.x * (long)kGaugeThreads + threadIdx.x;
    if (t >= 8L * Vh) return;
    const int i = (int)(t % Vh);
    const int mp = (int)(t / Vh);
    const int l = mp >> 1, P = mp & 1;
    int y[4];
    coords_of(g, P, i, y);
    Mat3<double> G, acc;
    load_link_soa<double>(Gl, l, P, i, Vh, G);
#pragma unroll
    for (int q = 0; q < 9; ++q) acc.e[q] = {0.0, 0.0};
    int el[4] = {0, 0, 0, 0};
    el[l] = 1;
#pragma unroll 1
    for (int m = 0; m < 4; ++m) {
        if (m == l) continue;
        int em[4] = {0, 0, 0, 0};
        em[m] = 1;
        Mat3<double> a, b, c, t1, t2;
        // upper: U_m(y+l) U_l(y+m)^dag M_m(y)
        //        + [ U_m(y+l) M_l(y+m) + M_m(y+l)^dag U_l(y+m)^dag ] U_m(y)^dag
        link_at<double>(g, L, y, el[0], el[1], el[2], el[3], m, a);
        link_at<double>(g, M, y, em[0], em[1], em[2], em[3], l, c);
        mat_mul(a, c, t2);
        link_at<double>(g, L, y, em[0], em[1], em[2], em[3], l, b);
        mat_mul_dag(a, b, t1);
        link_at<double>(g, M, y, 0, 0, 0, 0, m, c);
        mat_mul_add(t1, c, acc);
        mat_dag(b);
        link_at<double>(g, M, y, el[0], el[1], el[2], el[3], m, c);
        mat_dag(c);
        mat_mul_add(c, b, t2);
        link_at<double>(g, L, y, 0, 0, 0, 0, m, b);
        mat_mul_dag_add(t2, b, acc);
        // lower: (M_m(y-m) U_l(y-m) U_m(y-m+l))^dag
        //        + [ M_m(y+l-m) U_l(y-m)^dag + U_m(y-m+l)^dag M_l(y-m) ] U_m(y-m)
        link_at<double>(g, L, y, el[0] - em[0], el[1] - em[1], el[2] - em[2], el[3] - em[3], m, a);
        link_at<double>(g, L, y, -em[0], -em[1], -em[2], -em[3], l, b);
        mat_mul(b, a, t1);
        link_at<double>(g, M, y, -em[0], -em[1], -em[2], -em[3], m, c);
        mat_mul_add_dag(c, t1, acc);
        mat_dag(a);
        link_at<double>(g, M, y, -em[0], -em[1], -em[2], -em[3], l, c);
        mat_mul(a, c, t2);
        link_at<double>(g, M, y, el[0] - em[0], el[1] - em[1], el[2] - em[2], el[3] - em[3], m, c);
        mat_mul_dag_add(c, b, t2);
        link_at<double>(g, L, y, -em[0], -em[1], -em[2], -em[3], m, a);
        mat_mul_add(t2, a, acc);
    }
    mat_axpy(rho, acc, G);
    Mat3<double> U, W;
    load_link_soa<double>(L, l, P, i, Vh, U);
    mat_mul(U, G, W);
    // F = (i/2)(W - W^dag): re F_pq = -(Im W_pq + Im W_qp)/2, im F_pq = (Re W_pq - Re W_qp)/2
    const double d0 = -W.e[0].im, d1 = -W.e[4].im, d2 = -W.e[8].im;
    const double tr = (d0 + d1 + d2) / 3.0;
    double f[8];
    f[0] = d0 - tr;
    f[1] = d1 - tr;
    f[2] = -0.5 * (W.e[1].im + W.e[3].im);
    f[3] = 0.5 * (W.e[1].re - W.e[3].re);
    f[4] = -0.5 * (W.e[2].im + W.e[6].im);
    f[5] = 0.5 * (W.e[2].re - W.e[6].re);
    f[6] = -0.5 * (W.e[5].im + W.e[7].im);
    f[7] = 0.5 * (W.e[5].re - W.e[7].re);
    double *fo = Fout + (size_t)(mp * 8) * Vh + i;
#pragma unroll
    for (int k = 0; k < 8; ++k) fo[(size_t)k * Vh] = f[k];
}

// y += a x over n doubles
__global__ void k_daxpy(long n, double a, const double *__restrict__ x, double *__restrict__ y)
{
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < n) y[t] = fma(a, x[t], y[t]);
}

static LinkGeo link_geo(const lqcd_ctx *c)
{
    LinkGeo g;
    for (int m = 0; m < 4; ++m) g.N[m] = c->dims[m];
    g.Vh = (int)c->Vh;
    return g;
}

static inline unsigned nblocks(long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// ------------------------------------------------------------------ copies and staleness
// links: the FP64 SoA (lnk_nat) is the master; an FP32 MD step works on lnk_f18
// and makes it the newest copy; FP64 MD steps update lnk_nat and leave every
// derived format stale until links_ready rebuilds them.
static int links_to_prec(lqcd_ctx *c, int prec)
{
    const long n = 72L * (long)c->Vh;
    if (prec == LQCD_PREC_FP32) {
        if (c->md_links_newest == LQCD_PREC_FP64 && c->links_derived_stale) {
            k_links_f64_to_f32<<<nblocks(n, 256), 256, 0, c->stream>>>(c->lnk_nat.as<double2>(), c->lnk_f18.as<float2>(), n);
            LQCD_CUDA(cudaGetLastError());
            c->launches += 1;
        }
        return LQCD_OK;
    }
    if (c->md_links_newest == LQCD_PREC_FP32) {
        k_links_f32_to_f64<<<nblocks(n, 256), 256, 0, c->stream>>>(c->lnk_f18.as<float2>(), c->lnk_nat.as<double2>(), n);
        LQCD_CUDA(cudaGetLastError());
        c->launches += 1;
        c->md_links_newest = LQCD_PREC_FP64;
        c->links_derived_stale = true;
        c->df_stale = true;
    }
    if (prec == LQCD_PREC_FP64 && c->df_stale) {  // double-float steps work on the df64 copy
        k_links_nat_to_df<<<nblocks(n, 256), 256, 0, c->stream>>>(c->lnk_nat.as<double2>(), c->lnk_df.as<float4>(), n);
        LQCD_CUDA(cudaGetLastError());
        c->launches += 1;
        c->df_stale = false;
    }
    return LQCD_OK;
}

// FP64 and native FP64 share the FP64 momenta
static inline int mom_prec(int prec) { return prec == LQCD_PREC_FP32 ? LQCD_PREC_FP32 : LQCD_PREC_FP64; }

static int mom_to_prec(lqcd_ctx *c, int prec)
{
    prec = mom_prec(prec);
    if (c->mom_newest == prec) return LQCD_OK;
    const long n = 64L * (long)c->Vh;
    if (prec == LQCD_PREC_FP32)
        k_mom_f64_to_f32<<<nblocks(n, 256), 256, 0, c->stream>>>(c->mom64.as<double>(), c->mom32.as<float>(), n);
    else
        k_mom_f32_to_f64<<<nblocks(n, 256), 256, 0, c->stream>>>(c->mom32.as<float>(), c->mom64.as<double>(), n);
    LQCD_CUDA(cudaGetLastError());
    c->launches += 1;
    c->mom_newest = prec;
    return LQCD_OK;
}

static int check_md(lqcd_ctx *c, int prec)
{
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    if (!c->links_ok) return fail(LQCD_ESTATE, "no links uploaded");
    if (!c->mom64.ptr) return fail(LQCD_ESTATE, "no momenta uploaded");
    if (prec != LQCD_PREC_FP64 && prec != LQCD_PREC_FP32 && prec != LQCD_PREC_FP64_NATIVE)
        return fail(LQCD_EINVAL, "MD precision must be FP64, FP64_NATIVE or FP32");
    return LQCD_OK;
}

// Planes of one pass of the FP64 momentum update: as many of 6, 3, 2, 1 as keep the
// stored staples within kSidesLimit (all six up to 24^4, three at 32^4, two up to
// 36^4, one beyond: 3.1 GB at 48^4).  The passes group the sum into H, so their number depends on
// the lattice alone, and the bits do not depend on how much memory is free.
constexpr size_t kSidesLimit = (size_t)2 << 30;

static size_t plane_bytes(const lqcd_ctx *c) { return (size_t)1152 * c->Vh; }

static int sides_planes(const lqcd_ctx *c)
{
    int np = 6;
    while (np > 1 && np * plane_bytes(c) > kSidesLimit) np = np == 6 ? 3 : np - 1;
    return np;
}

// Room for the stored staples; false: the kernel that forms them itself runs.
// Asked once per call, before its first launch.
static bool sides_room(lqcd_ctx *c, int prec)
{
    if (prec == LQCD_PREC_FP32) return false;
    if (c->md_sides.ensure(sides_planes(c) * plane_bytes(c)) == LQCD_OK) return true;
    set_error("");
    return false;
}

template <class R>
static void launch_mom_sides(lqcd_ctx *c, const typename SideT<R>::t *L, bool stored, double beta, double eps)
{
    const LinkGeo g = link_geo(c);
    const int np = sides_planes(c);
    typename SideT<R>::t *F = c->md_sides.as<typename SideT<R>::t>();
    double *mom = c->mom64.as<double>();
    const unsigned nt = (unsigned)(2 * ((c->Vh + 31) / 32));
    for (int p0 = 0; p0 < 6; p0 += np) {
        const PlaneRange pr = {p0, np};
        if (stored) {
            k_gauge_sides<R><<<nblocks(4L * np * (long)c->Vh, kGaugeThreads), kGaugeThreads, 0, c->stream>>>(g, pr, L, F);
            k_gauge_mom_sides<R, true><<<nt, kGaugeThreads, 0, c->stream>>>(g, pr, L, F, mom, beta / 6.0, eps);
        } else {
            k_gauge_mom_sides<R, false><<<nt, kGaugeThreads, 0, c->stream>>>(g, pr, L, nullptr, mom, beta / 6.0, eps);
        }
        c->launches += stored ? 2 : 1;
    }
}

static void launch_mom_update(lqcd_ctx *c, int prec, bool stored, double beta, double eps)
{
    if (prec == LQCD_PREC_FP64) {
        launch_mom_sides<float2>(c, c->lnk_df.as<float4>(), stored, beta, eps);
    } else if (prec == LQCD_PREC_FP64_NATIVE) {
        launch_mom_sides<double>(c, c->lnk_nat.as<double2>(), stored, beta, eps);
    } else {
        const unsigned nt = (unsigned)(2 * ((c->Vh + 31) / 32));
        k_gauge_mom_update_f32<<<nt, kGaugeThreads, 0, c->stream>>>(link_geo(c), c->lnk_f18.as<float2>(),
                                                                    c->mom32.as<float>(), (float)(beta / 6.0), (float)eps);
        c->launches += 1;
    }
}

static void launch_link_update(lqcd_ctx *c, int prec, double eps)
{
    const unsigned nb = nblocks(8L * (long)c->Vh, kGaugeThreads);
    if (prec == LQCD_PREC_FP64) {
        k_gauge_link_update_df<<<nb, kGaugeThreads, 0, c->stream>>>((int)c->Vh, c->lnk_nat.as<double2>(),
                                                                    c->lnk_df.as<float4>(), c->mom64.as<double>(), eps);
        c->md_links_newest = LQCD_PREC_FP64;
    } else if (prec == LQCD_PREC_FP64_NATIVE) {
        k_gauge_link_update<double><<<nb, kGaugeThreads, 0, c->stream>>>((int)c->Vh, c->lnk_nat.as<double2>(),
                                                                         c->mom64.as<double>(), eps);
        c->md_links_newest = LQCD_PREC_FP64;
        c->df_stale = true;
    } else {
        k_gauge_link_update<float><<<nb, kGaugeThreads, 0, c->stream>>>((int)c->Vh, c->lnk_f18.as<float2>(),
                                                                        c->mom32.as<float>(), (float)eps);
        c->md_links_newest = LQCD_PREC_FP32;
        c->df_stale = true;
    }
    c->links_derived_stale = true;
    c->launches += 1;
}

static int prepare(lqcd_ctx *c, int prec)
{
    int st;
    if ((st = links_to_prec(c, prec))) return st;
    return mom_to_prec(c, prec);
}

// MD updates move the uploaded (thin) links; they are refused while the
// links in use are stout-smeared.
static int check_thin(const lqcd_ctx *c)
{
    if (c->stout_n) return fail(LQCD_ESTATE, "links are stout-smeared: call lqcd_stout_restore first");
    return LQCD_OK;
}

// Force on the stout levels' thin links from the force F (8 reals per link,
// mom layout) on the smeared links, in place: one local and one gather
// pass per level, from level n-1 down to 0.
static int stout_chain(lqcd_ctx *c, double *F, cudaStream_t s)
{
    const LinkGeo g = link_geo(c);
    const size_t nl = 72 * c->Vh, nf = 64 * c->Vh;
    int st;
    if ((st = c->stout_M.ensure(nl * sizeof(double2))) || (st = c->stout_G.ensure(nl * sizeof(double2))) ||
        (st = c->stout_F.ensure(2 * nf * sizeof(double))))
        return st;
    double *tmp = F == c->stout_F.as<double>() ? c->stout_F.as<double>() + nf : c->stout_F.as<double>();
    double *fa = F, *fb = tmp;
    const unsigned nb = nblocks(8L * (long)c->Vh, kGaugeThreads);
    for (int k = c->stout_n - 1; k >= 0; --k) {
        const double2 *Lk = c->stout_lv.as<double2>() + (size_t)k * nl;
        k_stout_local<<<nb, kGaugeThreads, 0, s>>>(g, Lk, fa, c->stout_rho, c->stout_M.as<double2>(),
                                                    c->stout_G.as<double2>());
        k_stout_gather<<<nb, kGaugeThreads, 0, s>>>(g, Lk, c->stout_M.as<double2>(), c->stout_G.as<double2>(),
                                                     c->stout_rho, fb);
        c->launches += 2;
        std::swap(fa, fb);
    }
    LQCD_CUDA(cudaGetLastError());
    if (fa != F) LQCD_CUDA(cudaMemcpyAsync(F, fa, nf * sizeof(double), cudaMemcpyDeviceToDevice, s));
    return LQCD_OK;
}

}  // namespace lqcd

using namespace lqcd;

extern "C" {

int lqcd_mom_upload(lqcd_ctx *c, const double *H, size_t n)
{
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    const size_t want = 4 * c->V * 18;
    if (!H || n != want) return fail(LQCD_EINVAL, "momenta: expected 4*V*18 doubles");
    int st;
    if ((st = c->mom64.ensure(64 * c->Vh * sizeof(double))) || (st = c->mom32.ensure(64 * c->Vh * sizeof(float))))
        return st;
    DevBuf stage;
    if ((st = stage.ensure(want * sizeof(double) + 16))) return st;
    int *bad = (int *)((char *)stage.ptr + want * sizeof(double));
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), c->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(stage.ptr, H, want * sizeof(double), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) {
        k_mom_from_canonical<<<nblocks(4L * (long)c->V, 256), 256, 0, c->stream>>>(
            link_geo(c), stage.as<double2>(), c->mom64.as<double>(), c->mom32.as<float>(), bad, (long)c->V);
        e = cudaGetLastError();
    }
    int hbad = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    stage.release();
    if (e != cudaSuccess) return cuda_fail(e, "momenta upload");
    c->launches += 1;
    c->mom_newest = LQCD_PREC_FP64;  // both copies written; FP64 is the exact one
    if (hbad) {
        c->mom64.release();
        c->mom32.release();
        return fail(LQCD_EINVAL, "momenta must be finite, Hermitian and traceless");
    }
    return LQCD_OK;
}

int lqcd_mom_download(lqcd_ctx *c, double *H, size_t n)
{
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    const size_t want = 4 * c->V * 18;
    if (!H || n != want) return fail(LQCD_EINVAL, "momenta: expected 4*V*18 doubles");
    if (!c->mom64.ptr) return fail(LQCD_ESTATE, "no momenta uploaded");
    DevBuf stage;
    int st;
    if ((st = stage.ensure(want * sizeof(double)))) return st;
    const unsigned nb = nblocks(4L * (long)c->V, 256);
    if (c->mom_newest == LQCD_PREC_FP32)
        k_mom_to_canonical<float><<<nb, 256, 0, c->stream>>>(link_geo(c), c->mom32.as<float>(), stage.as<double2>(), (long)c->V);
    else
        k_mom_to_canonical<double><<<nb, 256, 0, c->stream>>>(link_geo(c), c->mom64.as<double>(), stage.as<double2>(), (long)c->V);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) prefault_host(H, want * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpyAsync(H, stage.ptr, want * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    stage.release();
    if (e != cudaSuccess) return cuda_fail(e, "momenta download");
    c->launches += 1;
    return LQCD_OK;
}

int lqcd_gauge_mom_update(lqcd_ctx *c, int prec, double beta, double eps)
{
    NvtxRange nvtx_("lqcd_gauge_mom_update");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    int st;
    if ((st = check_md(c, prec)) || (st = check_thin(c)) || (st = prepare(c, prec))) return st;
    launch_mom_update(c, prec, sides_room(c, prec), beta, eps);
    LQCD_CUDA(cudaGetLastError());
    LQCD_CUDA(cudaStreamSynchronize(c->stream));
    return LQCD_OK;
}

int lqcd_gauge_link_update(lqcd_ctx *c, int prec, double eps)
{
    NvtxRange nvtx_("lqcd_gauge_link_update");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    int st;
    if ((st = check_md(c, prec)) || (st = check_thin(c)) || (st = prepare(c, prec))) return st;
    launch_link_update(c, prec, eps);
    LQCD_CUDA(cudaGetLastError());
    LQCD_CUDA(cudaStreamSynchronize(c->stream));
    return LQCD_OK;
}

int lqcd_gauge_md_steps(lqcd_ctx *c, int prec, double beta, double eps, int n_steps)
{
    NvtxRange nvtx_("lqcd_gauge_md_steps");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    int st;
    if ((st = check_md(c, prec)) || (st = check_thin(c)) || (st = prepare(c, prec))) return st;
    if (n_steps < 0) return fail(LQCD_EINVAL, "n_steps must be >= 0");
    const bool stored = n_steps > 0 && sides_room(c, prec);
    for (int k = 0; k < n_steps; ++k) {
        launch_mom_update(c, prec, stored, beta, eps);
        launch_link_update(c, prec, eps);
    }
    LQCD_CUDA(cudaGetLastError());
    LQCD_CUDA(cudaStreamSynchronize(c->stream));
    return LQCD_OK;
}

int lqcd_fermion_force_update(lqcd_ctx *c, double mass, double a0, const double *a, const double *shifts, int n_shift,
                              double tol, const double *phi, double eps, double *action, lqcd_solve_info *info)
{
    NvtxRange nvtx_("lqcd_fermion_force_update");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    int st;
    if ((st = check_md(c, LQCD_PREC_FP64))) return st;
    if (!phi || !a || !shifts) return fail(LQCD_EINVAL, "NULL argument");
    if (n_shift < 1 || n_shift > kMaxShifts) return fail(LQCD_EINVAL, "n_shift must be in 1..32");
    if (!std::isfinite(eps)) return fail(LQCD_EINVAL, "eps is not finite");
    if ((st = links_to_prec(c, LQCD_PREC_FP64_NATIVE)) || (st = mom_to_prec(c, LQCD_PREC_FP64))) return st;
    const size_t n3 = 3 * c->Vh;
    DevBuf &dphi = c->host_b, &dr = c->host_x;   // kept with the context, as by the host solve
    if ((st = dphi.ensure(n3 * sizeof(double2))) || (st = dr.ensure(n3 * sizeof(double2)))) return st;
    cudaStream_t s = c->stream;
    if ((st = host_to_soa(c, phi, dphi.as<double2>(), 1, s))) return st;
    // x_i in the context's scratch (rat_x), S_f = Re <phi, r(A) phi>
    double act = 0.0;
    const int rs = rational_apply_dev(c, mass, a0, a, shifts, n_shift, tol, dphi.as<double2>(), dr.as<double2>(), &act,
                                      info, s);
    if (rs != LQCD_OK && rs != LQCD_ENOCONV) return rs;
    if ((st = c->ff_y.ensure((size_t)n_shift * n3 * sizeof(double2)))) return st;
    const double2 *x = c->rat_x.as<double2>();
    double2 *y = c->ff_y.as<double2>();
    for (int k = 0; k < n_shift; ++k)
        if ((st = deo_launch(c, 1, LQCD_PREC_FP64, 18, x + (size_t)k * n3, y + (size_t)k * n3, s))) return st;
    FFCoef C;
    C.n = n_shift;
    for (int k = 0; k < kMaxShifts; ++k) C.a[k] = k < n_shift ? a[k] : 0.0;
    const unsigned nb = nblocks(8L * (long)c->Vh, kGaugeThreads);
    if (c->stout_n) {
        // force on the smeared links (into a zeroed buffer: 0 - (-1) F), chained
        // back to the thin links, then H -= eps F
        const size_t nf = 64 * c->Vh;
        if ((st = c->stout_F.ensure(2 * nf * sizeof(double)))) return st;
        double *F = c->stout_F.as<double>();
        LQCD_CUDA(cudaMemsetAsync(F, 0, nf * sizeof(double), s));
        k_fermion_force_update<<<nb, kGaugeThreads, 0, s>>>(c->g, c->lnk_nat.as<double2>(), x, y, C, F, -1.0);
        LQCD_CUDA(cudaGetLastError());
        c->launches += 1;
        if ((st = stout_chain(c, F, s))) return st;
        k_daxpy<<<nblocks((long)nf, 256), 256, 0, s>>>((long)nf, -eps, F, c->mom64.as<double>());
    } else {
        k_fermion_force_update<<<nb, kGaugeThreads, 0, s>>>(c->g, c->lnk_nat.as<double2>(), x, y, C,
                                                             c->mom64.as<double>(), eps);
    }
    LQCD_CUDA(cudaGetLastError());
    c->launches += 1;
    c->mom_newest = LQCD_PREC_FP64;
    LQCD_CUDA(cudaStreamSynchronize(s));
    if (action) *action = act;
    if (rs == LQCD_ENOCONV) set_error("solver did not reach tol within max_iter");
    return rs;
}

int lqcd_stout_smear(lqcd_ctx *c, double rho, int n_levels)
{
    NvtxRange nvtx_("lqcd_stout_smear");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    if (!c->links_ok) return fail(LQCD_ESTATE, "no links uploaded");
    if (c->stout_n) return fail(LQCD_ESTATE, "links are already stout-smeared: call lqcd_stout_restore first");
    if (!(rho >= 0.0) || !std::isfinite(rho)) return fail(LQCD_EINVAL, "rho must be finite and >= 0");
    if (n_levels < 1 || n_levels > 8) return fail(LQCD_EINVAL, "n_levels must be in 1..8");
    int st;
    if ((st = links_to_prec(c, LQCD_PREC_FP64_NATIVE))) return st;
    const size_t nl = 72 * c->Vh;
    if ((st = c->stout_lv.ensure((size_t)n_levels * nl * sizeof(double2)))) return st;
    cudaStream_t s = c->stream;
    const unsigned nb = nblocks(8L * (long)c->Vh, kGaugeThreads);
    for (int k = 0; k < n_levels; ++k) {
        double2 *lv = c->stout_lv.as<double2>() + (size_t)k * nl;
        LQCD_CUDA(cudaMemcpyAsync(lv, c->lnk_nat.ptr, nl * sizeof(double2), cudaMemcpyDeviceToDevice, s));
        k_stout_level<<<nb, kGaugeThreads, 0, s>>>(link_geo(c), lv, c->lnk_nat.as<double2>(), rho);
        c->launches += 1;
    }
    LQCD_CUDA(cudaGetLastError());
    c->stout_n = n_levels;
    c->stout_rho = rho;
    c->md_links_newest = LQCD_PREC_FP64;
    c->links_derived_stale = true;
    c->df_stale = true;
    LQCD_CUDA(cudaStreamSynchronize(s));
    return LQCD_OK;
}

int lqcd_stout_restore(lqcd_ctx *c)
{
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    if (!c->stout_n) return LQCD_OK;
    const size_t nl = 72 * c->Vh;
    LQCD_CUDA(cudaMemcpyAsync(c->lnk_nat.ptr, c->stout_lv.ptr, nl * sizeof(double2), cudaMemcpyDeviceToDevice,
                              c->stream));
    c->stout_n = 0;
    c->md_links_newest = LQCD_PREC_FP64;
    c->links_derived_stale = true;
    c->df_stale = true;
    LQCD_CUDA(cudaStreamSynchronize(c->stream));
    return LQCD_OK;
}

int lqcd_stout_force(lqcd_ctx *c, const double *F_smeared, double *F_thin, size_t n)
{
    NvtxRange nvtx_("lqcd_stout_force");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    if (!c->stout_n) return fail(LQCD_ESTATE, "links are not stout-smeared");
    const size_t want = 4 * c->V * 18;
    if (!F_smeared || !F_thin || n != want) return fail(LQCD_EINVAL, "forces: expected 4*V*18 doubles");
    const size_t nf = 64 * c->Vh;
    int st;
    if ((st = c->stout_F.ensure(2 * nf * sizeof(double)))) return st;
    DevBuf stage;
    if ((st = stage.ensure(want * sizeof(double) + 16))) return st;
    int *bad = (int *)((char *)stage.ptr + want * sizeof(double));
    cudaStream_t s = c->stream;
    double *F = c->stout_F.as<double>();
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(stage.ptr, F_smeared, want * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "force upload");
    k_mom_from_canonical<<<nblocks(4L * (long)c->V, 256), 256, 0, s>>>(link_geo(c), stage.as<double2>(), F, nullptr,
                                                                        bad, (long)c->V);
    c->launches += 1;
    int hbad = 0;
    LQCD_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
    LQCD_CUDA(cudaStreamSynchronize(s));
    if (hbad) return fail(LQCD_EINVAL, "forces must be finite, Hermitian and traceless");
    if ((st = stout_chain(c, F, s))) return st;
    k_mom_to_canonical<double><<<nblocks(4L * (long)c->V, 256), 256, 0, s>>>(link_geo(c), F, stage.as<double2>(),
                                                                            (long)c->V);
    c->launches += 1;
    e = cudaGetLastError();
    if (e == cudaSuccess) prefault_host(F_thin, want * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpyAsync(F_thin, stage.ptr, want * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "force download");
    return LQCD_OK;
}

int lqcd_gauge_action(lqcd_ctx *c, int prec, double beta, double *S)
{
    NvtxRange nvtx_("lqcd_gauge_action");
    if (!c || !S) return fail(LQCD_EINVAL, "NULL argument");
    LQCD_ON_DEVICE(c);
    if (!c->links_ok) return fail(LQCD_ESTATE, "no links uploaded");
    if (prec != LQCD_PREC_FP64 && prec != LQCD_PREC_FP32 && prec != LQCD_PREC_FP64_NATIVE)
        return fail(LQCD_EINVAL, "precision must be FP64, FP64_NATIVE or FP32");
    if (prec == LQCD_PREC_FP64_NATIVE) prec = LQCD_PREC_FP64;  // the action is computed from the IEEE master
    int st;
    if ((st = links_to_prec(c, prec == LQCD_PREC_FP64 ? LQCD_PREC_FP64_NATIVE : prec))) return st;
    const unsigned nb = nblocks(2L * (long)c->Vh, kGaugeThreads);
    if ((st = c->md_part.ensure(((size_t)nb + 1) * sizeof(double)))) return st;
    double *part = c->md_part.as<double>();
    if (prec == LQCD_PREC_FP64)
        k_gauge_action_part<double><<<nb, kGaugeThreads, 0, c->stream>>>(link_geo(c), c->lnk_nat.as<double2>(), part);
    else
        k_gauge_action_part<float><<<nb, kGaugeThreads, 0, c->stream>>>(link_geo(c), c->lnk_f18.as<float2>(), part);
    k_gauge_sum_ordered<<<1, 256, 0, c->stream>>>(part, (int)nb, part + nb);
    LQCD_CUDA(cudaGetLastError());
    c->launches += 2;
    LQCD_CUDA(cudaMemcpyAsync(c->h_pinned_d, part + nb, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    LQCD_CUDA(cudaStreamSynchronize(c->stream));
    *S = -(beta / 3.0) * c->h_pinned_d[0];
    return LQCD_OK;
}

int lqcd_mom_energy(lqcd_ctx *c, int prec, double *K)
{
    int st;
    if (!K) return fail(LQCD_EINVAL, "NULL argument");
    if (!c) return fail(LQCD_EINVAL, "NULL context");
    LQCD_ON_DEVICE(c);
    if ((st = check_md(c, prec)) || (st = mom_to_prec(c, prec))) return st;
    const unsigned nb = nblocks(8L * (long)c->Vh, kGaugeThreads);
    if ((st = c->md_part.ensure(((size_t)nb + 1) * sizeof(double)))) return st;
    double *part = c->md_part.as<double>();
    if (mom_prec(prec) == LQCD_PREC_FP64)
        k_mom_energy_part<double><<<nb, kGaugeThreads, 0, c->stream>>>((int)c->Vh, c->mom64.as<double>(), part);
    else
        k_mom_energy_part<float><<<nb, kGaugeThreads, 0, c->stream>>>((int)c->Vh, c->mom32.as<float>(), part);
    k_gauge_sum_ordered<<<1, 256, 0, c->stream>>>(part, (int)nb, part + nb);
    LQCD_CUDA(cudaGetLastError());
    c->launches += 2;
    LQCD_CUDA(cudaMemcpyAsync(c->h_pinned_d, part + nb, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    LQCD_CUDA(cudaStreamSynchronize(c->stream));
    *K = c->h_pinned_d[0];
    return LQCD_OK;
}

}  // extern "C"
