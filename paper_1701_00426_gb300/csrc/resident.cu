// resident.cu -- host side of the resident iteration (solver_resident.cuh):
// which batches take it, how the blocks are shared out over the jobs, and the
// launches until every job halts.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "internal.h"
#include "solver_resident.cuh"

namespace lqcd {

// Blocks that fit at once (one per SM), 0 = the device or the kernels' shared
// memory attribute refuse: the four-kernel iteration runs.
static std::mutex g_res_mu;
static int g_res_blocks[64];
static bool g_res_done[64];
constexpr size_t kResSmemMax = 227 * 1024;
constexpr int kResWords = 96;   // three counts of a job, 128 bytes apart

template <class K>
static bool res_kernel_ok(K kern)
{
    int occ = 0;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmemMax) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kResThreads, kResSmemMax) == cudaSuccess &&
           occ >= 1;
}

template <int NJ>
static bool res_kernels_ok()
{
    return res_kernel_ok(k_it_resident<NJ, VP_DF, LF_DF18>) && res_kernel_ok(k_it_resident<NJ, VP_F32, LF_F32_18>) &&
           res_kernel_ok(k_it_resident<NJ, VP_F32, LF_F32_12>) && res_kernel_ok(k_it_resident<NJ, VP_F32, LF_F16_12>);
}

static int resident_blocks(int dev)
{
    if (dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lk(g_res_mu);
    if (!g_res_done[dev]) {
        g_res_done[dev] = true;
        int nsm = 0, coop = 0;
        if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
            res_kernels_ok<1>() && res_kernels_ok<kMaxJobs>())
            g_res_blocks[dev] = std::min(nsm, kResMaxCtas);
        cudaGetLastError();  // a refusal above only disables the path
    }
    return g_res_blocks[dev];
}

// Dynamic shared memory: state, link ring, p hand-over buffers, the table of
// neighbours of m sub-tiles and, if they fit, their r and q.
template <int VP, int LF>
static size_t res_smem_t(int m, bool in_smem)
{
    return res_align(sizeof(ResShared)) + res_ring_bytes<VP, LF>() + res_pbuf_bytes<VP, LF>() +
           (size_t)m * 16 * kResSub * sizeof(uint32_t) + res_stage_bytes<VP>() +
           (in_smem ? (size_t)2 * m * 96 * sizeof(typename VecT<VP>::T) : 0);
}

static size_t res_smem(int vp, int lf, int m, bool in_smem)
{
    if (vp == VP_DF) return res_smem_t<VP_DF, LF_DF18>(m, in_smem);
    if (lf == LF_F32_18) return res_smem_t<VP_F32, LF_F32_18>(m, in_smem);
    if (lf == LF_F32_12) return res_smem_t<VP_F32, LF_F32_12>(m, in_smem);
    return res_smem_t<VP_F32, LF_F16_12>(m, in_smem);
}

// Largest batch (sites of one parity, all jobs) that takes the resident path.
// us per iteration, four kernels -> resident, one GB300:
//            double-float, 1 / 15 shifts      FP32 12-real, 1 / 15 shifts
//   8^4      28.5 -> 15.8,  34.0 -> 17.8      28.2 -> 15.5,  37.6 -> 22.4
//   12^4     33.1 -> 20.3,  39.5 -> 24.3      29.7 -> 18.4,  39.9 -> 27.3
//   16^4     36.0 -> 31.2,  43.0 -> 37.8      32.2 -> 24.4,  43.7 -> 36.6
//   18^4     48.8 -> 44.1,  57.7 -> 59.1      39.6 -> 32.2,  55.0 -> 52.0
//   20^4     64.7 -> 68.8,  80.0 -> 99.7      47.5 -> 47.4,  69.7 -> 77.3
// (whole solves over their iterations).  Above, the staged stencils' wider
// tiles and the streaming shift update win.
constexpr long kResMaxSitesDF = 40960;
constexpr long kResMaxSitesF32 = 53248;

template <int NJ>
static void res_launch(const ResBatch<NJ> &R, int vp, int lf, int nblk, size_t smem, cudaStream_t s)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblk);
    cfg.blockDim = dim3((unsigned)kResThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (vp == VP_DF) cudaLaunchKernelEx(&cfg, k_it_resident<NJ, VP_DF, LF_DF18>, R);
    else if (lf == LF_F32_18) cudaLaunchKernelEx(&cfg, k_it_resident<NJ, VP_F32, LF_F32_18>, R);
    else if (lf == LF_F32_12) cudaLaunchKernelEx(&cfg, k_it_resident<NJ, VP_F32, LF_F32_12>, R);
    else cudaLaunchKernelEx(&cfg, k_it_resident<NJ, VP_F32, LF_F16_12>, R);
}

// Shares the blocks out: the smallest m (sub-tiles of one block) for which
// every job gets ceil(sub-tiles / m) blocks.
template <int NJ>
static int res_share(const IterBatch<NJ> &B, int nblk, int *cta_start)
{
    long most = 1;
    for (int j = 0; j < B.njobs; ++j) most = std::max(most, (long)(B.job[j].g.Vh + kResSub - 1) / kResSub);
    auto blocks = [&](long m) {
        long t = 0;
        for (int j = 0; j < B.njobs; ++j) t += ((B.job[j].g.Vh + kResSub - 1) / kResSub + m - 1) / m;
        return t;
    };
    long lo = 1, hi = most;
    if (blocks(hi) > nblk) return 0;
    while (lo < hi) {
        const long mid = (lo + hi) / 2;
        if (blocks(mid) <= nblk) hi = mid;
        else lo = mid + 1;
    }
    cta_start[0] = 0;
    for (int j = 0; j < B.njobs; ++j)
        cta_start[j + 1] = cta_start[j] + (int)(((B.job[j].g.Vh + kResSub - 1) / kResSub + lo - 1) / lo);
    return (int)lo;
}

int resident_sms(const lqcd_ctx *c)
{
    const bool df_only = c->opts.prec == LQCD_PREC_FP64;
    const int nsm = resident_blocks(c->device);
    if (c->opts.pdl || nsm <= 0 || (long)c->Vh > (df_only ? kResMaxSitesDF : kResMaxSitesF32)) return CallScope::kWhole;
    const long nsub = ((long)c->Vh + kResSub - 1) / kResSub, m = (nsub + nsm - 1) / nsm;
    return (int)((nsub + m - 1) / m);   // res_share for one job
}

// One stall word per job, in the context's pinned memory (which the kernels
// write directly); read when the stream has finished.
static unsigned *clear_stall_words(lqcd_ctx *c)
{
    unsigned *w = (unsigned *)c->h_pinned + 2 * kMaxJobs;
    std::fill(w, w + kMaxJobs, 0u);
    return w;
}

static int check_stall_words(const volatile unsigned *w, int njobs)
{
    for (int j = 0; j < njobs; ++j)
        if (w[j]) return fail(LQCD_ETIMEOUT, "a bounded device wait of the resident iteration ran out");
    return LQCD_OK;
}

int resident_wait_selftest(lqcd_ctx *c, double limit_s)
{
    if (!(limit_s > 0.0 && limit_s <= 10.0)) return fail(LQCD_EINVAL, "limit must be in (0, 10] seconds");
    DevBuf d;
    if (int st = d.ensure(512)) return st;   // [0] barrier count, [32] halt word, [64 ..] a sum, all zero
    unsigned *stall = clear_stall_words(c), *w = d.as<unsigned>();
    int status[2] = {LQCD_OK, LQCD_OK};
    cudaError_t e = cudaSuccess;
    for (int which = 0; which < 2 && e == cudaSuccess; ++which) {
        stall[0] = 0u;
        e = cudaMemsetAsync(w, 0, 512, c->stream);
        if (e != cudaSuccess) break;
        k_res_wait_selftest<<<2, kResThreads, 0, c->stream>>>(w, (const ulonglong2 *)(w + 64), stall, (int *)(w + 32),
                                                              which, (uint64_t)(limit_s * 1e9));
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e == cudaSuccess) status[which] = check_stall_words(stall, 1);
    }
    d.release();
    if (e != cudaSuccess) return cuda_fail(e, "resident wait self-test");
    for (int st : status)
        if (st != LQCD_ETIMEOUT) return fail(LQCD_ESTATE, "a wait that nothing ends did not run out");
    return check_stall_words(stall, 1);
}

template <int NJ>
int resident_run(lqcd_ctx *c, const IterBatch<NJ> &B, int vp, int lf, int max_iter, cudaStream_t s, bool &done)
{
    done = false;
    if (c->opts.pdl || persist_blocks() <= 0 || kSites != kTile) return LQCD_OK;
    long sites = 0;
    for (int j = 0; j < B.njobs; ++j) sites += B.job[j].g.Vh;
    if (sites > (vp == VP_DF ? kResMaxSitesDF : kResMaxSitesF32)) {
        CallScope::declare(c->device, CallScope::kWhole);
        return LQCD_OK;
    }
    const int nblk = resident_blocks(c->device);
    ResBatch<NJ> R;
    memset(&R, 0, sizeof R);
    const int m = nblk > 0 ? res_share(B, nblk, R.cta_start) : 0;
    if (m <= 0) return LQCD_OK;
    R.in_smem = res_smem(vp, lf, m, true) <= kResSmemMax;
    const size_t smem = res_smem(vp, lf, m, R.in_smem != 0);
    if (smem > kResSmemMax) return LQCD_OK;
    const int blocks = R.cta_start[B.njobs];
    CallScope::declare(c->device, blocks);
    if (!CallScope::fits(c->device, blocks, nblk)) return LQCD_OK;
    R.njobs = B.njobs;
    // kResWords words of counts for every job, then the published warp sums
    size_t slots = 0;
    for (int j = 0; j < B.njobs; ++j) slots += 2 * (size_t)((B.job[j].g.Vh + kResSub - 1) / kResSub);
    const size_t fbytes = (size_t)kMaxJobs * kResWords * sizeof(unsigned), bytes = fbytes + slots * sizeof(ulonglong2);
    if (c->res_xch.bytes < bytes) {
        if (c->res_xch.ensure(bytes)) {
            set_error("");
            return LQCD_OK;  // no room for the exchange buffer: the four-kernel iteration runs
        }
        LQCD_CUDA(cudaMemsetAsync(c->res_xch.ptr, 0, c->res_xch.bytes, s));
    }
    ulonglong2 *x = (ulonglong2 *)((char *)c->res_xch.ptr + fbytes);
    for (int j = 0; j < B.njobs; ++j) {
        R.job[j] = B.job[j];
        R.bar[j] = c->res_xch.as<unsigned>() + (size_t)j * kResWords;
        R.xch[j] = x;
        x += 2 * (size_t)((B.job[j].g.Vh + kResSub - 1) / kResSub);
    }
    R.steps = kResSteps;
    int *hs = c->h_pinned;
    unsigned *stall = clear_stall_words(c);
    R.stall = stall;
    cudaEvent_t ev[2];
    LQCD_CUDA(cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming));
    LQCD_CUDA(cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming));
    auto enqueue = [&](int sl) -> cudaError_t {
        // a fresh range of tags for every launch, 0 left out (the cleared buffer);
        // when they start again, no sum of the first 2^32 may be left
        const bool wrap = c->res_tag > 0xFFFF0000u;
        if (wrap) c->res_tag = 0;
        R.tag0 = c->res_tag + 1;
        c->res_tag += (uint32_t)R.steps;
        cudaError_t e = cudaMemsetAsync(c->res_xch.ptr, 0,
                                        wrap ? c->res_xch.bytes : (size_t)B.njobs * kResWords * sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
        res_launch<NJ>(R, vp, lf, blocks, smem, s);
        e = cudaGetLastError();
        c->launches += 1;
        for (int j = 0; j < B.njobs && e == cudaSuccess; ++j)
            e = cudaMemcpyAsync(hs + sl * kMaxJobs + j, &B.job[j].st->halt, sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaEventRecord(ev[sl], s);
        return e;
    };
    const int max_launches = max_iter / kResSteps + 4;
    int slot = 0;
    cudaError_t e = enqueue(0);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        // fewer SMs than the device reports (a partition): the four kernels run
        cudaGetLastError();
        cudaEventDestroy(ev[0]);
        cudaEventDestroy(ev[1]);
        return LQCD_OK;
    }
    bool shared = false;   // others need the device: the four kernels go on from the end of the last launch
    for (int k = 0; k < max_launches && e == cudaSuccess; ++k) {
        shared = !CallScope::fits(c->device, blocks, nblk);
        if (shared) break;
        const int nxt = slot ^ 1;
        e = enqueue(nxt);
        if (e != cudaSuccess) break;
        e = cudaEventSynchronize(ev[slot]);
        if (e != cudaSuccess) break;
        bool all = true;
        for (int j = 0; j < B.njobs; ++j) all &= hs[slot * kMaxJobs + j] != HALT_NONE;
        if (all) break;
        slot = nxt;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
    if (e != cudaSuccess) return cuda_fail(e, "resident iteration");
    if (int st = check_stall_words(stall, B.njobs)) return st;
    done = !shared;
    return LQCD_OK;
}

template int resident_run<1>(lqcd_ctx *, const IterBatch<1> &, int, int, int, cudaStream_t, bool &);
template int resident_run<kMaxJobs>(lqcd_ctx *, const IterBatch<kMaxJobs> &, int, int, int, cudaStream_t, bool &);

}  // namespace lqcd
