// solver_resident.cuh -- the multi-shift CG iteration (Sec. 2.2, Eqs. lineqeo
// and shlineq) of lattices whose links stay in L2, as one cooperative kernel
// that runs many iterations per launch.
//
// What bounds it: latency.  On 8^4 an iteration moves 5 MB, under 1 us of
// HBM time, but four launches with their tile reductions and one-warp
// finalisers take 28.5 us, on 8 of 152 SMs, and 36 us on 16^4 (128 tiles).
// This kernel takes 15.8 and 31.2 us (resident.cu has the table).  So:
// - The unit of work is a sub-tile of 32 consecutive sites.  In double-float
//   three warps share it, one per colour of the result: the three rows of a
//   hop are independent sums, so the split shortens a site's serial chain by
//   three and an 8^4 lattice keeps 64 SMs busy, with the same arithmetic in
//   the same order as one thread per site.  In FP32 one warp takes it.
// - A block owns a fixed range of sub-tiles for the whole launch; r and q of
//   its sites live in shared memory when they fit.  t and p (read by
//   neighbours), x and the other directions go through L2.
// - Links never change, so every thread copies the links of its next site
//   into its own shared-memory ring (cp.async, one group per hop, half a site
//   ahead) while it works on the current one, across phases and barriers: no
//   hop waits for a link, and no two threads need to agree on a stage.
// - The two reductions need no fence: every sub-tile's warp sum is published
//   as two 64-bit words that carry the iteration's tag beside the payload, and
//   counted; when the count is full every block reads all sums (the tags tell
//   whether a sum has arrived) and forms the total itself, in the order of
//   tile_finish_block (warp sums of a tile in order, tiles strided by 256,
//   shuffle tree, warps in order).  One word is polled, by one thread of a
//   block: polling words that many blocks rewrite costs 6.7 us at 152 blocks,
//   against 1.0 us for the count (1.4 us with release and acquire).  Every block keeps the recurrence's scalars
//   in shared memory and updates them with the finalisers of the four-kernel
//   iteration, so no block waits for another one's finaliser.
// - FP64 arithmetic has a long latency on this chip; only alpha and beta are
//   on the critical path.  The shifted coefficients are computed by warp 0
//   while the other warps form r -= alpha q, and x is updated while the
//   blocks wait for ||r||^2; the p_s and x_s of that update are copied to
//   shared memory while they wait for <p, q>.
// - Two grid barriers per iteration remain (t complete, p complete).
// The results are bitwise those of the four-kernel iteration.
//
// Every wait is bounded by the global timer; a block whose wait runs out
// stops, sets the job's stall word (host memory, which no block ever clears: the
// first block writes back its own copy of the state, and would undo a mark that
// another one left there) and leaves.  The launch is cooperative, so all blocks
// are resident.  A job's blocks wait only on one another.
#pragma once

#include "bulk.cuh"
#include "solver_kernels.cuh"

namespace lqcd {

constexpr int kResSub = 32;          // sites of a sub-tile
constexpr int kResWarps = 12;        // warps of a block: 4 sub-tiles at once (double-float) or 12 (FP32)
constexpr int kResThreads = 32 * kResWarps;
constexpr int kResMaxCtas = 512;
constexpr int kResStage = 8;         // shift-update elements of a thread staged in shared memory

template <int NJ>
struct ResBatch {
    int njobs;
    int steps;                   // iterations of this launch, at most
    int in_smem;                 // 1: r and q in shared memory
    uint32_t tag0;               // tags of this launch: tag0 + it
    int cta_start[NJ + 1];       // blocks of job j
    ulonglong2 *xch[NJ];         // [2][sub-tiles] published warp sums
    unsigned *stall;             // [NJ] set to 1 by a block whose wait ran out
    unsigned *bar[NJ];           // counts at words 0 (grid barrier), 32 and 64 (sums published); zero at launch
    IterJob job[NJ];
};

struct ResShared {
    SolverState st;
    double red[kTile / 32];
    int dead;     // a bounded wait ran out
    int broke;    // <p, q> not positive or not finite
};

// Warps per sub-tile and link elements of one hop (16-byte units x lanes).
template <int VP, int LF> struct ResShape;
template <> struct ResShape<VP_DF, LF_DF18> { static constexpr int W = 3, D = 4; static constexpr size_t hop = 3 * 16; };
template <> struct ResShape<VP_F32, LF_F32_18> { static constexpr int W = 1, D = 4; static constexpr size_t hop = 9 * 8; };
template <> struct ResShape<VP_F32, LF_F32_12> { static constexpr int W = 1, D = 8; static constexpr size_t hop = 3 * 16; };
template <> struct ResShape<VP_F32, LF_F16_12> { static constexpr int W = 1, D = 8; static constexpr size_t hop = 16 + 8; };

constexpr size_t res_align(size_t n) { return (n + 127) & ~(size_t)127; }

template <int VP, int LF>
constexpr size_t res_ring_bytes()
{
    return (size_t)kResWarps * ResShape<VP, LF>::D * ResShape<VP, LF>::hop * 32;
}

// p of a sub-tile handed to the summing warp: two buffers per slot (double-float only)
template <int VP, int LF>
constexpr size_t res_pbuf_bytes()
{
    return ResShape<VP, LF>::W == 3 ? (size_t)2 * (kResWarps / 3) * 96 * sizeof(float4) : 0;
}

// p_s and x_s of the first kResStage update elements of every thread of warps 1 ..
template <int VP>
constexpr size_t res_stage_bytes()
{
    return (size_t)(kResWarps - 1) * kResStage * 2 * 32 * sizeof(typename VecT<VP>::T);
}

// A double with a tag in each of its two words: each 64-bit word is written
// and read whole, so a reader that finds both tags has the value.
__device__ __forceinline__ void xch_put(ulonglong2 *p, double v, uint32_t tag)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | (u & 0xFFFFFFFFull)),
                 "l"(t | (u >> 32))
                 : "memory");
}

__device__ __forceinline__ ulonglong2 xch_get(const ulonglong2 *p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ bool xch_ok(const ulonglong2 &v, uint32_t tag)
{
    return (uint32_t)(v.x >> 32) == tag && (uint32_t)(v.y >> 32) == tag;
}

__device__ __forceinline__ double xch_val(const ulonglong2 &v)
{
    return __longlong_as_double((long long)((v.x & 0xFFFFFFFFull) | (v.y << 32)));
}

__device__ __forceinline__ void red_add(unsigned *p, unsigned n)
{
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(n) : "memory");
}

// Until *p has reached n, or the time limit has passed (false).  The count is
// read once more after that: a block that was preempted may find it complete.
template <bool ACQ>
__device__ __forceinline__ bool poll_count(const unsigned *p, unsigned n, uint64_t limit_ns)
{
    auto reached = [=]() -> bool {
        unsigned v;
        if (ACQ) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        else asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return (int)(v - n) >= 0;
    };
    uint64_t t0 = 0;
    for (unsigned k = 1;; ++k) {
        if (reached()) return true;
        if ((k & 63u) == 0u) {
            const uint64_t t = globaltimer_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > limit_ns) return reached();
        }
    }
}

// All blocks of the job have written what they wrote before the call, and
// this block sees it.  count: barriers passed so far times ncta, plus ncta.
// Called by every thread.
__device__ __forceinline__ void res_barrier(ResShared &sh, unsigned *bar, unsigned count,
                                            uint64_t limit_ns = kStageWaitNs)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        if (!poll_count<true>(bar, count, limit_ns)) sh.dead = 1;
    }
    __syncthreads();
}

// Partial total of virtual warp vw (lanes = tiles vw * 32 + lane, strided by
// 256): the warp's shuffle-tree sum, valid in lane 0.
__device__ __noinline__ double res_warp_total(ResShared &sh, const ulonglong2 *X, int nsub, int ntiles, uint32_t tag,
                                              int vw, uint64_t limit_ns = kStageWaitNs)
{
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int tile = vw * 32 + lane; tile < ntiles; tile += kTile) {
        constexpr int K = kTile / kResSub;
        const int n = min(K, nsub - tile * K);
        const ulonglong2 *p = X + (size_t)tile * K;
        ulonglong2 v[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < n) v[k] = xch_get(p + k);
        uint64_t t0 = 0;
        unsigned tries = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (k >= n) continue;
            while (!xch_ok(v[k], tag)) {
                if ((++tries & 63u) == 0u) {
                    const uint64_t t = globaltimer_ns();
                    if (t0 == 0) t0 = t;
                    if (t - t0 > limit_ns) {
                        v[k] = xch_get(p + k);
                        if (!xch_ok(v[k], tag)) sh.dead = 1;
                        break;
                    }
                }
                __nanosleep(20);   // counted but not here yet: rare
                v[k] = xch_get(p + k);
            }
        }
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < n) t += xch_val(v[k]);
        s += t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
    return s;
}

// Waits until `count` sums of the job have been counted in *cnt (warp 0).
// The count carries no ordering: the reader of a sum checks its tags.
__device__ __forceinline__ void res_counted(ResShared &sh, const unsigned *cnt, unsigned count)
{
    if (threadIdx.x == 0 && !poll_count<false>(cnt, count, kStageWaitNs)) sh.dead = 1;
    __syncwarp();
}

// Total of the job's published warp sums for every thread; called by all.
__device__ __forceinline__ double res_total(ResShared &sh, const ulonglong2 *X, const unsigned *cnt, unsigned count,
                                            int nsub, int ntiles, uint32_t tag)
{
    const int lane = threadIdx.x & 31, w = (int)threadIdx.x >> 5;
    const int nvw = min(kTile / 32, (ntiles + 31) >> 5);
    if (w == 0) res_counted(sh, cnt, count);
    __syncthreads();
    for (int vw = w; vw < nvw; vw += kResWarps) {
        const double s = res_warp_total(sh, X, nsub, ntiles, tag, vw);
        if (lane == 0) sh.red[vw] = s;
    }
    __syncthreads();
    double tot = 0.0;
    for (int k = 0; k < nvw; ++k) tot += sh.red[k];
    return tot;
}

// ------------------------------------------------------------------ link ring
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A site a thread works on: its half index (0 beyond V/2: nothing of such a
// lane is kept), the output parity and its row of the block's table of
// neighbours: word h is the half index of hop h's neighbour (h = 2 mu +
// direction) with the hop's sign in the top bit.
struct ResItem {
    const uint32_t *tab;
    int i, P;
};

__device__ __forceinline__ void res_item(const Geom &g, const uint32_t *tab, int u0, int k, int P, ResItem &I)
{
    const int lane = threadIdx.x & 31, i = (u0 + k) * kResSub + lane;
    I.i = i < g.Vh ? i : 0;
    I.P = P;
    I.tab = tab + (size_t)(2 * k + P) * 8 * kResSub + lane;
}

// The links of one site that a thread needs for hop h (BWD: odd h), copied to
// the ring slot dst.  Each thread reads only what it copied, so the thread's
// own group count orders copy and use.
template <int VP, int LF, bool BWD>
__device__ __forceinline__ void ring_copy(unsigned char *dst, const IterJob &J, const ResItem &I, int a, int h)
{
    const int mu = h >> 1, Vh = J.g.Vh, lane = threadIdx.x & 31;
    const void *links = J.links;
    const int par = BWD ? 1 - I.P : I.P, idx = BWD ? (int)(I.tab[h * kResSub] & 0x7FFFFFFFu) : I.i;
    if constexpr (LF == LF_DF18) {
        // forward: row a (components 3 a + c); backward: column a (3 c + a)
        const int c0 = BWD ? a : 3 * a, cs = BWD ? 3 : 1;
        const float4 *p = (const float4 *)links + link_base(mu, par, 9, Vh) + (size_t)c0 * Vh + idx;
#pragma unroll
        for (int c = 0; c < 3; ++c) cp_async16(dst + (size_t)(c * 32 + lane) * 16, p + (size_t)c * cs * Vh);
    } else if constexpr (LF == LF_F32_18) {
        const float2 *p = (const float2 *)links + link_base(mu, par, 9, Vh) + idx;
#pragma unroll
        for (int c = 0; c < 9; ++c) cp_async8(dst + (size_t)(c * 32 + lane) * 8, p + (size_t)c * Vh);
    } else if constexpr (LF == LF_F32_12) {
        const float4 *p = (const float4 *)links + link_base(mu, par, 3, Vh) + idx;
#pragma unroll
        for (int c = 0; c < 3; ++c) cp_async16(dst + (size_t)(c * 32 + lane) * 16, p + (size_t)c * Vh);
    } else {
        const uint4 *pa = (const uint4 *)links;
        const uint2 *pb = (const uint2 *)(pa + (size_t)8 * Vh);
        cp_async16(dst + (size_t)lane * 16, pa + (size_t)(mu * 2 + par) * Vh + idx);
        cp_async8(dst + 512 + (size_t)lane * 8, pb + (size_t)(mu * 2 + par) * Vh + idx);
    }
    cp_commit();
}

// Neighbour spinors of hop h.  They are written by other blocks of this
// launch: plain loads, never the read-only path.
template <class T>
struct ResHop {
    T v[3];
    uint32_t neg;
};

template <class T>
__device__ __forceinline__ void gather_hop(const T *in, int Vh, const ResItem &I, int h, ResHop<T> &G)
{
    const uint32_t e = I.tab[h * kResSub];
    const int idx = (int)(e & 0x7FFFFFFFu);
    G.neg = e & 0x80000000u;
#pragma unroll
    for (int c = 0; c < 3; ++c) G.v[c] = in[(size_t)c * Vh + idx];
}

// Sums of one site: row a in double-float, the whole site in FP32.
template <int VP> struct ResAcc;
template <> struct ResAcc<VP_DF> { Acc2 re, im; float cr, ci; };
template <> struct ResAcc<VP_F32> { float2 r[3]; };

// One hop (BWD: backward) from the ring slot `src` into the sums: the order
// of products of deo_site_df (row a) or deo_site_f32.
template <int VP, int LF, bool BWD>
__device__ __forceinline__ void res_hop(const unsigned char *src, const ResHop<typename VecT<VP>::T> &G, ResAcc<VP> &A)
{
    const int lane = threadIdx.x & 31;
    const uint32_t ng = G.neg;
    if constexpr (VP == VP_DF) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 u = *(const float4 *)(src + (size_t)(c * 32 + lane) * 16), x = xor_sign4(G.v[c], ng);
            acc_prod_h(A.re, A.cr, u.x, u.y, x.x, x.y);
            if (!BWD) acc_prod_h(A.re, A.cr, -u.z, -u.w, x.z, x.w);
            else acc_prod_h(A.re, A.cr, u.z, u.w, x.z, x.w);
            acc_prod_h(A.im, A.ci, u.x, u.y, x.z, x.w);
            if (!BWD) acc_prod_h(A.im, A.ci, u.z, u.w, x.x, x.y);
            else acc_prod_h(A.im, A.ci, -u.z, -u.w, x.x, x.y);
        }
    } else {
        float2 U[9];
        if constexpr (LF == LF_F32_18) {
#pragma unroll
            for (int c = 0; c < 9; ++c) U[c] = *(const float2 *)(src + (size_t)(c * 32 + lane) * 8);
        } else if constexpr (LF == LF_F32_12) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float4 t = *(const float4 *)(src + (size_t)(k * 32 + lane) * 16);
                U[2 * k] = make_float2(t.x, t.y);
                U[2 * k + 1] = make_float2(t.z, t.w);
            }
            reconstruct_row2(U);
        } else {
            const uint4 p = *(const uint4 *)(src + (size_t)lane * 16);
            const uint2 q = *(const uint2 *)(src + 512 + (size_t)lane * 8);
            U[0] = h2f(p.x); U[1] = h2f(p.y); U[2] = h2f(p.z); U[3] = h2f(p.w);
            U[4] = h2f(q.x); U[5] = h2f(q.y);
            reconstruct_row2(U);
        }
        float2 x[3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
            x[c] = make_float2(__uint_as_float(__float_as_uint(G.v[c].x) ^ ng),
                               __uint_as_float(__float_as_uint(G.v[c].y) ^ ng));
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (!BWD) {
                    const float2 u = U[r * 3 + c];
                    A.r[r].x = __fmaf_rn(u.x, x[c].x, __fmaf_rn(-u.y, x[c].y, A.r[r].x));
                    A.r[r].y = __fmaf_rn(u.x, x[c].y, __fmaf_rn(u.y, x[c].x, A.r[r].y));
                } else {
                    const float2 u = U[c * 3 + r];
                    A.r[r].x = __fmaf_rn(u.x, x[c].x, __fmaf_rn(u.y, x[c].y, A.r[r].x));
                    A.r[r].y = __fmaf_rn(u.x, x[c].y, __fmaf_rn(-u.y, x[c].x, A.r[r].y));
                }
            }
    }
}

// D at the item's site: row a in double-float (the accumulators 2a, 2a + 1 of
// deo_site_df), the whole site in FP32.  The neighbour spinors of the next
// direction are loaded before this one's products; after a hop's products the
// ring slot takes the hop D further on, of this item or of the next one, N.
// The direction loop stays rolled: unrolled, the two stencils are 48 KB of
// code and the offsets of their 24 links spill.
template <int VP, int LF>
__device__ __forceinline__ void res_deo(unsigned char *ring, const IterJob &J, const typename VecT<VP>::T *in,
                                        const ResItem &I, const ResItem &N, int a,
                                        typename VecT<VP>::T (&out)[ResShape<VP, LF>::W == 3 ? 1 : 3])
{
    using T = typename VecT<VP>::T;
    using R = ResShape<VP, LF>;
    const int Vh = J.g.Vh;
    ResAcc<VP> A;
    if constexpr (VP == VP_DF) {
        acc_zero(A.re);
        acc_zero(A.im);
        A.cr = A.ci = 0.f;
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) A.r[c] = make_float2(0.f, 0.f);
    }
    ResHop<T> gf, gb;
    gather_hop<T>(in, Vh, I, 0, gf);
    gather_hop<T>(in, Vh, I, 1, gb);
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
        ResHop<T> nf, nb;
        const int h = 2 * mu, hn = mu < 3 ? h + 2 : h;   // the last direction loads itself again (L1)
        gather_hop<T>(in, Vh, I, hn, nf);
        gather_hop<T>(in, Vh, I, hn + 1, nb);
        unsigned char *src = ring + (size_t)(h % R::D) * R::hop * 32;
        const bool same = R::D < 8 && h + R::D < 8;      // the hop D further on is this item's
        ResItem Q = same ? I : N;
        const int hq = (h + R::D) & 7;
        cp_wait<R::D - 1>();
        res_hop<VP, LF, false>(src, gf, A);
        ring_copy<VP, LF, false>(src, J, Q, a, hq);
        cp_wait<R::D - 1>();
        res_hop<VP, LF, true>(src + R::hop * 32, gb, A);
        ring_copy<VP, LF, true>(src + R::hop * 32, J, Q, a, hq + 1);
        if constexpr (VP == VP_DF) {
            acc_flush(A.re, A.cr);
            acc_flush(A.im, A.ci);
        }
        gf = nf;
        gb = nb;
    }
    if constexpr (VP == VP_DF) {
        const float2 r = acc_result(A.re), m = acc_result(A.im);
        out[0] = make_float4(0.5f * r.x, 0.5f * r.y, 0.5f * m.x, 0.5f * m.y);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) out[c] = make_float2(0.5f * A.r[c].x, 0.5f * A.r[c].y);
    }
}

// ------------------------------------------------------------------ shift updates
// The elements of x_s += alpha_s p_s and p_s = zeta_s r + beta_s p_s of every
// active shift, spread over warps 1 .. by (active shift, sub-tile, colour).
struct ResUpd {
    unsigned mask;      // active shifts not reached yet, this one included
    int kc, m3;         // sub-tile kc / 3, colour kc % 3
    __device__ __forceinline__ bool more() const { return mask != 0u; }
    __device__ __forceinline__ int shift() const { return __ffs((int)mask) - 1; }
    __device__ __forceinline__ void skip()
    {
        while (kc >= m3 && mask) {
            kc -= m3;
            mask &= mask - 1u;
        }
    }
    __device__ __forceinline__ void next()
    {
        kc += kResWarps - 1;
        skip();
    }
};

// The shifts the coming update moves (the active list finalize_pq makes).
__device__ __forceinline__ ResUpd res_upd(const SolverState &st, int m)
{
    const int lane = threadIdx.x & 31;
    ResUpd U;
    U.mask = __ballot_sync(0xFFFFFFFFu, lane < st.n_shift && st.active_next[lane]);
    U.kc = ((int)threadIdx.x >> 5) - 1;
    U.m3 = 3 * m;
    U.skip();
    return U;
}

template <class T>
__device__ __forceinline__ void cp_async_el(T *dst, const T *src)
{
    if constexpr (sizeof(T) == 16) cp_async16(dst, src);
    else cp_async8(dst, src);
}

// Starts copying the thread's first elements of p_s and x_s to shared memory:
// they do not depend on alpha, so they arrive while the blocks wait for
// <p, q>.  stg: the thread's first slot ([element][p, x][lane] of its warp).
template <int VP>
__device__ __forceinline__ void res_stage(ResUpd U, typename VecT<VP>::T *stg, const typename VecT<VP>::T *x,
                                          const typename VecT<VP>::T *ps, int u0, int Vh)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int t = 0; t < kResStage && U.more(); ++t, U.next()) {
        const int sub = U.kc / 3, c = U.kc - 3 * sub, i = (u0 + sub) * kResSub + lane;
        if (i < Vh) {
            const size_t off = (size_t)(U.shift() * 3 + c) * Vh + i;
            cp_async_el(stg + (2 * t) * 32, ps + off);
            cp_async_el(stg + (2 * t + 1) * 32, x + off);
        }
    }
    cp_commit();
}

// DIR = false: x_s += alpha_s p_s; DIR = true: p_s = zeta_s r + beta_s p_s.
// Elements beyond the staged ones are loaded two at a time.
template <int VP, bool DIR>
__device__ __forceinline__ void res_update(const SolverState &st, ResUpd U, const typename VecT<VP>::T *stg,
                                           typename VecT<VP>::T *x, typename VecT<VP>::T *ps,
                                           const typename VecT<VP>::T *rs, size_t sk, size_t sc, int u0, int Vh)
{
    using T = typename VecT<VP>::T;
    const int lane = threadIdx.x & 31;
    auto store = [&](int s, unsigned off, const T &p, const T &y) {
        if constexpr (VP == VP_DF) {
            if constexpr (DIR) {
                const float2 zn = st.zeta_new_df[s], bs = st.beta_s_df[s];
                const float2 pr = df_mul2(zn, make_float2(y.x, y.y), bs, make_float2(p.x, p.y));
                const float2 pi = df_mul2(zn, make_float2(y.z, y.w), bs, make_float2(p.z, p.w));
                ps[off] = make_float4(pr.x, pr.y, pi.x, pi.y);
            } else {
                const float2 as = st.alpha_s_df[s];
                const float2 xr = df_fma(as, make_float2(p.x, p.y), make_float2(y.x, y.y));
                const float2 xi = df_fma(as, make_float2(p.z, p.w), make_float2(y.z, y.w));
                x[off] = make_float4(xr.x, xr.y, xi.x, xi.y);
            }
        } else if constexpr (DIR) {
            const float zn = st.zeta_new_df[s].x, bs = st.beta_s_df[s].x;
            ps[off] = make_float2(__fmaf_rn(zn, y.x, bs * p.x), __fmaf_rn(zn, y.y, bs * p.y));
        } else {
            const float as = st.alpha_s_df[s].x;
            x[off] = make_float2(__fmaf_rn(as, p.x, y.x), __fmaf_rn(as, p.y, y.y));
        }
    };
    // the sub-tile's lanes beyond V/2 have no element: off = ~0
    auto where = [&](int &s, unsigned &off, T &y) {
        const int sub = U.kc / 3, c = U.kc - 3 * sub, i = (u0 + sub) * kResSub + lane;
        s = U.shift();
        off = i < Vh ? (unsigned)(s * 3 + c) * (unsigned)Vh + (unsigned)i : ~0u;
        if (DIR && i < Vh) y = rs[(size_t)sub * sk + (size_t)c * sc + lane];
    };
#pragma unroll 1
    for (int t = 0; t < kResStage && U.more(); ++t, U.next()) {
        int s;
        unsigned off;
        T y;
        where(s, off, y);
        if (off == ~0u) continue;
        if (!DIR) y = stg[(2 * t + 1) * 32];
        store(s, off, stg[(2 * t) * 32], y);
    }
#pragma unroll 1
    while (U.more()) {
        int s0, s1 = 0;
        unsigned o0, o1 = ~0u;
        T p0, p1, y0, y1;
        where(s0, o0, y0);
        if (o0 != ~0u) {
            p0 = ps[o0];
            if (!DIR) y0 = x[o0];
        }
        U.next();
        if (U.more()) {
            where(s1, o1, y1);
            if (o1 != ~0u) {
                p1 = ps[o1];
                if (!DIR) y1 = x[o1];
            }
            U.next();
        }
        if (o0 != ~0u) store(s0, o0, p0, y0);
        if (o1 != ~0u) store(s1, o1, p1, y1);
    }
}

// ------------------------------------------------------------------ the iteration
template <int NJ, int VP, int LF>
__global__ void __launch_bounds__(kResThreads, 1) k_it_resident(const __grid_constant__ ResBatch<NJ> B)
{
    using T = typename VecT<VP>::T;
    using R = ResShape<VP, LF>;
    constexpr int W = R::W, NS = kResWarps / W;   // warps of a slot, slots
    extern __shared__ __align__(128) unsigned char smem_raw[];
    ResShared &sh = *reinterpret_cast<ResShared *>(smem_raw);
    SolverState &st = sh.st;
    const int lane = threadIdx.x & 31, w = (int)threadIdx.x >> 5;
    const int slot = w / W, a = w - W * slot;
    unsigned char *ring = smem_raw + res_align(sizeof(ResShared)) + (size_t)w * R::D * R::hop * 32;
    T *pbuf = reinterpret_cast<T *>(smem_raw + res_align(sizeof(ResShared)) + res_ring_bytes<VP, LF>());
    uint32_t *tab = reinterpret_cast<uint32_t *>(smem_raw + res_align(sizeof(ResShared)) + res_ring_bytes<VP, LF>() +
                                                 res_pbuf_bytes<VP, LF>());
    int j = 0;
    if (NJ > 1) {
#pragma unroll 1
        while (j + 1 < B.njobs && (int)blockIdx.x >= B.cta_start[j + 1]) ++j;
    }
    const IterJob &J = B.job[j];
    const int cta = (int)blockIdx.x - B.cta_start[j], ncta = B.cta_start[j + 1] - B.cta_start[j];
    const int Vh = J.g.Vh, ntiles = J.ntiles;
    const int nsub = (Vh + kResSub - 1) / kResSub;
    const int u0 = (int)((long)cta * nsub / ncta), m = (int)((long)(cta + 1) * nsub / ncta) - u0;
    ulonglong2 *X2 = B.xch[j], *X3 = X2 + nsub;
    unsigned *bar = B.bar[j];
    T *stg = reinterpret_cast<T *>(tab + (size_t)m * 16 * kResSub) + (size_t)(w - 1) * kResStage * 2 * 32 + lane;
    T *rq = reinterpret_cast<T *>(tab + (size_t)m * 16 * kResSub) + (size_t)(kResWarps - 1) * kResStage * 2 * 32;
    const bool few = ntiles <= 32;   // one warp forms the totals
    static_assert(sizeof(SolverState) % 4 == 0, "copied in words");
    for (int k = (int)threadIdx.x; k < (int)(sizeof(SolverState) / 4); k += kResThreads)
        ((uint32_t *)&st)[k] = __ldcg((const uint32_t *)J.st + k);
    if (threadIdx.x == 0) sh.dead = 0;
    T *t_g = (T *)J.t, *x_g = (T *)J.x, *ps_g = (T *)J.ps;
    // r and q of the block's sites: element (k, c, lane) at k * sk + c * sc + lane
    T *rs, *qs;
    size_t sk, sc;
    for (int k = w; k < 2 * m; k += kResWarps) {
        const int i = (u0 + (k >> 1)) * kResSub + lane;
        Stencil S;
        make_stencil(J.g, i < Vh ? i : 0, k & 1, S);
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            int f, b;
            uint32_t nf, nb;
            hop(J.g, S, mu, f, b, nf, nb);
            tab[(k * 8 + 2 * mu) * kResSub + lane] = (uint32_t)f | nf;
            tab[(k * 8 + 2 * mu + 1) * kResSub + lane] = (uint32_t)b | nb;
        }
    }
    if (B.in_smem) {
        rs = rq;
        qs = rq + (size_t)m * 96;
        sk = 96;
        sc = 32;
        for (int k = w; k < m * 3; k += kResWarps) {
            const int i = (u0 + k / 3) * kResSub + lane;
            if (i < Vh) rs[k * 32 + lane] = ((const T *)J.r)[(size_t)(k % 3) * Vh + i];
        }
    } else {
        rs = (T *)J.r + (size_t)u0 * kResSub;
        qs = (T *)J.q + (size_t)u0 * kResSub;
        sk = kResSub;
        sc = (size_t)Vh;
    }
    __syncthreads();
    if (st.halt) return;   // the same for every block of the job: written only at the end of a launch
    const T *p_g = ps_g + (size_t)st.base * 3 * Vh;
    ResItem I, N;
    if (slot < m) {
        res_item(J.g, tab, u0, slot, 1, I);
#pragma unroll 1
        for (int h = 0; h < R::D; h += 2) {
            ring_copy<VP, LF, false>(ring + (size_t)h * R::hop * 32, J, I, a, h);
            ring_copy<VP, LF, true>(ring + (size_t)(h + 1) * R::hop * 32, J, I, a, h + 1);
        }
    }
    // the item after sub-tile k of parity P in this slot's sequence
    auto next_item = [&](int k, int P) {
        if (k + NS < m) res_item(J.g, tab, u0, k + NS, P, N);
        else res_item(J.g, tab, u0, slot, 1 - P, N);
    };
    unsigned passed = 0;   // barrier arrivals of the job so far in this launch
    bool stalled = false;
#pragma unroll 1
    for (int it = 0; it < B.steps; ++it) {
        const uint32_t tag = B.tag0 + (uint32_t)it;
        // t = D_oe p
#pragma unroll 1
        for (int k = slot; k < m; k += NS) {
            next_item(k, 1);
            T o[W == 3 ? 1 : 3];
            res_deo<VP, LF>(ring, J, p_g, I, N, a, o);
            const int i = (u0 + k) * kResSub + lane;
            if (i < Vh) {
                if constexpr (W == 3) t_g[(size_t)a * Vh + i] = o[0];
                else {
#pragma unroll
                    for (int c = 0; c < 3; ++c) t_g[(size_t)c * Vh + i] = o[c];
                }
            }
            I = N;
        }
        passed += (unsigned)ncta;
        res_barrier(sh, bar, passed);
        if (sh.dead) {
            stalled = true;
            break;
        }
        // q = (m^2 + sigma) p - D_eo t, <p, q>.  In double-float the three
        // warps of a slot hand q and p to the first one, which sums the site's
        // products in colour order; p goes through one of two buffers, so a
        // warp may be one sub-tile ahead of the sum.
        int par = 0, nput = 0;
#pragma unroll 1
        for (int k = slot; k < m; k += NS) {
            next_item(k, 0);
            const int i = (u0 + k) * kResSub + lane;
            const bool live = i < Vh;
            T *qk = qs + (size_t)k * sk + lane;
            Acc2 dot;
            acc_zero(dot);
            if constexpr (W == 3) {
                T *pt = pbuf + ((size_t)par * NS + slot) * 96 + lane;
                par ^= 1;
                T pa, o[1];
                if (live) pa = p_g[(size_t)a * Vh + i];
                res_deo<VP, LF>(ring, J, t_g, I, N, a, o);
                if (live) {
                    const float2 a0 = st.a0_df;
                    const float2 qr = df_fma(a0, make_float2(pa.x, pa.y), df_neg(make_float2(o[0].x, o[0].y)));
                    const float2 qi = df_fma(a0, make_float2(pa.z, pa.w), df_neg(make_float2(o[0].z, o[0].w)));
                    pt[a * 32] = pa;
                    qk[(size_t)a * sc] = make_float4(qr.x, qr.y, qi.x, qi.y);
                }
                asm volatile("bar.sync %0, 96;" ::"r"(1 + slot) : "memory");
                if (a == 0 && live) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float4 q = qk[(size_t)c * sc], pv = pt[c * 32];
                        acc_prod(dot, pv.x, pv.y, q.x, q.y);
                        acc_prod(dot, pv.z, pv.w, q.z, q.w);
                    }
                }
            } else {
                T pv[3], o[3];
                if (live) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) pv[c] = p_g[(size_t)c * Vh + i];
                }
                res_deo<VP, LF>(ring, J, t_g, I, N, a, o);
                if (live) {
                    const float a0 = st.a0_df.x;
                    float d = 0.f;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float2 q = make_float2(__fmaf_rn(a0, pv[c].x, -o[c].x), __fmaf_rn(a0, pv[c].y, -o[c].y));
                        qk[(size_t)c * sc] = q;
                        d = __fmaf_rn(pv[c].x, q.x, __fmaf_rn(pv[c].y, q.y, d));
                    }
                    dot.s = d;
                }
            }
            if (a == 0) {
                warp_reduce_acc(dot);
                if (lane == 0) xch_put(X2 + u0 + k, (double)dot.s + (double)dot.c, tag);
                ++nput;
            }
            I = N;
        }
        // counted by the thread that published
        if (lane == 0 && nput) red_add(bar + 32, (unsigned)nput);
        ResUpd upd;
        if (w > 0) {
            upd = res_upd(st, m);
            res_stage<VP>(upd, stg, x_g, ps_g, u0, Vh);
        }
        const unsigned counted = (unsigned)nsub * (unsigned)(it + 1);
        PqCarry pc;
        if (few) {
            if (w == 0) {
                res_counted(sh, bar + 32, counted);
                const double s = res_warp_total(sh, X2, nsub, ntiles, tag, 0);
                pc = finalize_pq_alpha(&st, __shfl_sync(0xFFFFFFFFu, s, 0));
            }
        } else {
            const double pq = res_total(sh, X2, bar + 32, counted, nsub, ntiles, tag);
            if (w == 0) pc = finalize_pq_alpha(&st, pq);
        }
        if (threadIdx.x == 0) {
            st.do_k4 = 0;
            sh.broke = !pc.ok;
        }
        __syncthreads();
        if (sh.dead) {
            stalled = true;
            break;
        }
        if (sh.broke) break;
        // warp 0: the shifted coefficients; the others: r -= alpha q, ||r||^2,
        // then x_s += alpha_s p_s
        RrCarry rc;
        if (w == 0) {
            finalize_pq_shifts(&st, pc);
            __syncwarp();
            asm volatile("bar.arrive 14, %0;" ::"n"(kResThreads) : "memory");
            rc = finalize_rr_begin(&st);
            if (few) {
                res_counted(sh, bar + 64, counted);
                const double s = res_warp_total(sh, X3, nsub, ntiles, tag, 0);
                finalize_rr_end(&st, rc, __shfl_sync(0xFFFFFFFFu, s, 0));
            }
        } else {
            nput = 0;
#pragma unroll 1
            for (int k = w - 1; k < m; k += kResWarps - 1) {
                const int i = (u0 + k) * kResSub + lane;
                T *rk = rs + (size_t)k * sk + lane;
                const T *qk = qs + (size_t)k * sk + lane;
                Acc2 nrm;
                acc_zero(nrm);
                if (i < Vh) {
                    if constexpr (VP == VP_DF) {
                        const float2 na = df_neg(st.alpha_df);
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const float4 rv = rk[(size_t)c * sc], qv = qk[(size_t)c * sc];
                            const float2 x = df_fma(na, make_float2(qv.x, qv.y), make_float2(rv.x, rv.y));
                            const float2 y = df_fma(na, make_float2(qv.z, qv.w), make_float2(rv.z, rv.w));
                            rk[(size_t)c * sc] = make_float4(x.x, x.y, y.x, y.y);
                            acc_prod(nrm, x.x, x.y, x.x, x.y);
                            acc_prod(nrm, y.x, y.y, y.x, y.y);
                        }
                    } else {
                        const float na = -st.alpha_df.x;
                        float d = 0.f;
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const float2 rv = rk[(size_t)c * sc], qv = qk[(size_t)c * sc];
                            const float2 v = make_float2(__fmaf_rn(na, qv.x, rv.x), __fmaf_rn(na, qv.y, rv.y));
                            rk[(size_t)c * sc] = v;
                            d = __fmaf_rn(v.x, v.x, __fmaf_rn(v.y, v.y, d));
                        }
                        nrm.s = d;
                    }
                }
                warp_reduce_acc(nrm);
                if (lane == 0) xch_put(X3 + u0 + k, (double)nrm.s + (double)nrm.c, tag);
                ++nput;
            }
            if (lane == 0 && nput) red_add(bar + 64, (unsigned)nput);
            asm volatile("bar.sync 14, %0;" ::"n"(kResThreads) : "memory");
            cp_wait<0>();
            res_update<VP, false>(st, upd, stg, x_g, ps_g, rs, sk, sc, u0, Vh);
        }
        if (!few) {
            const double rr = res_total(sh, X3, bar + 64, counted, nsub, ntiles, tag);
            if (w == 0) finalize_rr_end(&st, rc, rr);
        }
        __syncthreads();
        if (sh.dead) {
            stalled = true;
            break;
        }
        if (!st.do_k4) break;   // NaN: the directions stay as they are
        // p_s = zeta_s r + beta_s p_s
        if (w > 0) res_update<VP, true>(st, upd, stg, x_g, ps_g, rs, sk, sc, u0, Vh);
        if (st.halt || it + 1 == B.steps) break;
        passed += (unsigned)ncta;
        res_barrier(sh, bar, passed);
        if (sh.dead) {
            stalled = true;
            break;
        }
    }
    cp_wait<0>();
    __syncthreads();
    if (B.in_smem) {
        for (int k = w; k < m * 3; k += kResWarps) {
            const int i = (u0 + k / 3) * kResSub + lane;
            if (i < Vh) ((T *)J.r)[(size_t)(k % 3) * Vh + i] = rs[k * 32 + lane];
        }
    }
    if (stalled && threadIdx.x == 0) {
        B.stall[j] = 1u;
        st.stall = 1;
        st.halt = HALT_STALL;
    }
    if (cta == 0) {
        __syncthreads();
        for (int k = (int)threadIdx.x; k < (int)(sizeof(SolverState) / 4); k += kResThreads)
            ((uint32_t *)J.st)[k] = ((const uint32_t *)&st)[k];
    }
}

// The waits with a short limit: block 0 ends at once and marks the job
// converged, as the first block of a job that missed nothing; block 1 waits for a
// barrier (which = 0) or a sum (1) that never comes.
static __global__ void __launch_bounds__(kResThreads, 1)
    k_res_wait_selftest(unsigned *bar, const ulonglong2 *X, unsigned *stall, int *halt, int which, uint64_t limit_ns)
{
    __shared__ ResShared sh;
    if (threadIdx.x == 0) sh.dead = 0;
    __syncthreads();
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) *halt = HALT_CONVERGED;
        return;
    }
    if (which == 0) {
        res_barrier(sh, bar, 2u, limit_ns);
    } else if (threadIdx.x < 32) {
        res_warp_total(sh, X, 1, 1, 1u, 0, limit_ns);
    }
    __syncthreads();
    if (sh.dead && threadIdx.x == 0) *stall = 1u;
}

}  // namespace lqcd
