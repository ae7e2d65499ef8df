// Decoding a small problem in one cooperative launch: the iterations of a
// flooding sum-product decode (check update, variable update, syndrome check)
// run inside one kernel with grid barriers between the phases.  Included by
// small_f16.cu and small_f32.cu.
//
// A short code's iteration is a few microseconds of work in five to seven
// launches; issued one by one they cost the host ~20 us an iteration whatever
// the size.  Here a phase costs its own latency and a barrier (~1.5 us).
#pragma once

#include "kernels.cuh"
#include "wrap_count.h"

namespace {

constexpr int kSmallBlock = 512;       // one block per SM, 128 registers a thread
constexpr int kSmallMaxTerms = 6;      // core edges of a check
constexpr int kSmallMaxClasses = 12;   // check shapes of a graph
constexpr int kSmallMaxLanes = 512;    // codewords (their bookkeeping is in shared memory)
// Check or variable threads of an iteration up to which one launch is the
// faster: eight rounds of the resident threads.  50 iterations, rate 0.1, one
// launch against a launch per class and phase: n = 4096, 8 codewords, half 0.48
// against 1.07 ms; n = 65536, 16 codewords, float (236 000 threads) 1.11 / 1.42
// ms; n = 131072, 16 codewords, half (472 000) 1.29 / 1.61 ms; n = 65536, 64
// codewords, half (944 000) 2.04 / 1.95 ms; n = 131072, 64 codewords 4.17 /
// 3.44 ms.
constexpr int64_t kSmallMaxThreads = 152 * 512 * 8;
// A block takes a whole SM's registers, so a decode excludes other one-launch
// decodes from its SMs until it ends.  One whose check threads all fit half of
// the SMs takes no more than these: two such decodes run side by side.
// Microseconds a decode of 25 iterations (n = 4096, half, early termination) on
// 1 / 2 / 4 streams at once, 16 codewords: 390 / 753 / 1481 on as many SMs as
// its warps spread over, 393 / 416 / 788 on half of them; 32 codewords (29 000
// threads) 399 / 770 / 1516 and 408 / 423 / 811.  A larger decode keeps every
// SM: on half of them a single one of 64 codewords (59 000 threads) takes 440
// instead of 405, of 118 000 threads 538 instead of 446.  Several of those on
// streams of their own take turns (64 codewords: 405 / 766 / 1503; with a launch
// per phase 587 / 651 / 735); one batch or a plan serves them better.
constexpr int kSmallShareDiv = 2;
// edges in flight per thread in the variable update: the phase has few warps,
// so a VN's 20 to 34 rows are requested in two or three rounds (half) or four
// to six (float: twice the registers a row)
template <typename MsgT> constexpr int kSmallRound = IsHalf<MsgT>::value ? 12 : 6;

struct SmallArgs {
    CnArgs cn;
    VnArgs vn;
    SynArgs sy;
    ClassLaunch cls[kSmallMaxClasses];
    uint32_t first[kSmallMaxClasses + 1];  // first thread of each class (multiples of 32) and the end
    int n_cls;
    int32_t slabs, batch, iters;
    int hard1;
    size_t h1;            // bytes between the two degree-1 decision buffers
    uint32_t *fail;       // two buffers of the slabs' fail words
    int32_t *iters_dev;   // iterations used, conv: for the output kernel and the caller
    uint8_t *conv_dev;
    int32_t *iters_out;   // the caller's arrays, or null
    uint8_t *conv_out;
    uint32_t *bar;        // grid barrier: arrivals, generation, abort flag
    int32_t *status;      // may be null
    int32_t stall;        // test of the timeout path: arrivals that never come
};

// Grid barrier of a cooperative launch (every block is resident): arrivals are
// counted up (modulo 2^32), and every block polls the count itself, one L2 round
// trip after the last arrival.  Writes made before it are visible after it.  `target`:
// the count of this barrier, raised for the next one.  A wait that runs out
// (2 s) raises the abort flag, on which every block leaves (false); the flag
// stays up, and later launches with the same barrier words leave on entry.
__device__ __forceinline__ bool grid_barrier(uint32_t *bar, uint32_t &target) {
    target += gridDim.x;
    int ok = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        uint32_t now, spins = 0;
        unsigned long long t0 = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(bar) : "memory");
            if (mld::count_reached(now, target)) break;
            if ((++spins & 1023u) == 0) {
                uint32_t aborted;
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(aborted) : "l"(bar + 2) : "memory");
                if (t0 == 0) t0 = global_ns();
                if (aborted || global_ns() - t0 > kWaitLimitNs) {
                    atomicExch(bar + 2, 1u);
                    ok = 0;
                    break;
                }
            }
        }
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
    return __syncthreads_and(ok) != 0;
}

// The last block to leave resets the barrier for the next launch.
__device__ __forceinline__ void grid_leave(uint32_t *bar) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
            bar[0] = 0u;
            bar[1] = 0u;
        }
    }
}

// A check's terms read past L1 (other SMs write them between the phases).
template <typename MsgT, int W, int DC>
struct TermsCoherent {
    const float *lvb;
    const MsgT *rp;
    const float *pp;
    int32_t v[DC];
    __device__ __forceinline__ float4 lv(int i) const {
        return __ldcg(reinterpret_cast<const float4 *>(lvb + static_cast<size_t>(v[i]) * W));
    }
    __device__ __forceinline__ typename Msg<MsgT>::Raw ro(int i) const {
        return __ldcg(reinterpret_cast<const typename Msg<MsgT>::Raw *>(rp + i * W));
    }
    __device__ __forceinline__ float4 p1(int i) const { return ldf4(pp + i * W); }
};

// Check j of class cl, codewords lane0 .. lane0+3 of slab.
template <typename MsgT, int W, int DC, int DD, int PASS>
__device__ __forceinline__ void small_check(const CnArgs &a, const ClassLaunch &cl, int32_t j, int lane0, int slab) {
    constexpr int NB = W / 8;
    const int32_t e0 = cl.e0 + j * DC, s0 = cl.s0 + j * DD;
    TermsCoherent<MsgT, W, DC> t;
#pragma unroll
    for (int i = 0; i < DC; ++i) t.v[i] = __ldg(a.col + e0 + i);
    MsgT *rp = static_cast<MsgT *>(a.r) + (static_cast<size_t>(slab) * a.e_core + e0) * W + lane0;
    t.rp = rp;
    t.lvb = a.Lv + static_cast<size_t>(slab) * a.n_core * W + lane0;
    t.pp = a.phi1 + (static_cast<size_t>(slab) * a.n_deg1 + s0) * W + lane0;
    const uint32_t sb =
        static_cast<uint32_t>(a.sbits[(static_cast<size_t>(slab) * a.n_cn + cl.c0 + j) * NB + lane0 / 8]) >> (lane0 & 7);
    const uint32_t donenib = a.et ? kept_nibble<W, PASS == kPassFull>(a, slab, lane0) : 0u;
    check_terms<MsgT, W, DC, DD, PASS, false, false>(a, lane0, slab, true, rp, e0, s0, sb, donenib, t);
}

template <typename MsgT, int W, int PASS>
__device__ __forceinline__ void small_checks(const SmallArgs &s, const CnArgs &a, uint32_t t0, uint32_t step) {
    constexpr uint32_t TPC = W / kK;
    int k = 0;
    for (uint32_t t = t0; t < s.first[s.n_cls]; t += step) {
        while (t >= s.first[k + 1]) ++k;
        const ClassLaunch &cl = s.cls[k];
        const uint32_t u = t - s.first[k];  // thread of the class
        const uint32_t per_slab = static_cast<uint32_t>(cl.count) * TPC;
        const uint32_t slab = u / per_slab;
        if (slab >= static_cast<uint32_t>(s.slabs)) continue;  // padding of the class to whole warps
        if (a.et && slab_all_done<W>(a.done, slab)) continue;
        const int32_t j = static_cast<int32_t>((u - slab * per_slab) / TPC);
        const int lane0 = static_cast<int>(u % TPC) * kK;
        switch (cl.dc * 2 + (cl.deg - cl.dc)) {
#define MLD_SMALL(DCV, DDV) case (DCV) * 2 + (DDV): small_check<MsgT, W, DCV, DDV, PASS>(a, cl, j, lane0, slab); break;
            MLD_SMALL(1, 0) MLD_SMALL(2, 0) MLD_SMALL(3, 0) MLD_SMALL(4, 0) MLD_SMALL(5, 0) MLD_SMALL(6, 0)
            MLD_SMALL(1, 1) MLD_SMALL(2, 1) MLD_SMALL(3, 1) MLD_SMALL(4, 1) MLD_SMALL(5, 1) MLD_SMALL(6, 1)
#undef MLD_SMALL
            default: break;
        }
    }
}

// All iterations.  Threads are numbered warp by warp across the blocks, so that
// a phase with few items still spreads over every SM.
template <typename MsgT, int W>
__global__ void __launch_bounds__(kSmallBlock, 1) k_small_decode(SmallArgs s) {
    constexpr int DW = (W + 31) / 32;
    __shared__ uint32_t done[kSmallMaxLanes / 8], fail[kSmallMaxLanes / 8];
    __shared__ int32_t its[kSmallMaxLanes];
    __shared__ uint8_t conv[kSmallMaxLanes];
    const int words = s.slabs * DW;
    for (int i = threadIdx.x; i < words; i += blockDim.x) done[i] = padding_lanes(s.batch, W, i / DW, i % DW);
    const bool et = s.cn.et != 0;
    CnArgs cn = s.cn;
    VnArgs vn = s.vn;
    SynArgs sy = s.sy;
    cn.done = vn.done = sy.done = done;
    const uint32_t step = gridDim.x * blockDim.x;
    const uint32_t t0 = ((threadIdx.x / 32) * gridDim.x + blockIdx.x) * 32 + threadIdx.x % 32;
    const uint32_t vn_threads = static_cast<uint32_t>(vn.n_core) * (W / kVnLanes);
    const uint32_t syn_threads = (static_cast<uint32_t>(sy.n_cn) + 31) / 32 * 32;
    // The thread's place in the range of a slab: the slabs' ranges follow one
    // another around the grid, so that several slabs use all warps at once.
    // (One range over all slabs needs a division and 64-bit bases in the inner
    // loop and spills: n = 65536, 16 codewords, float 954 -> 980 us.)
    auto place = [&](int slab, uint32_t range) {
        return slab == 0 ? t0 : (t0 + step - static_cast<uint32_t>(slab) * range % step) % step;
    };
    uint32_t target = s.stall > 0 ? 1u : 0u;
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < 2 * words; i += blockDim.x) s.fail[i] = 0u;
    uint32_t aborted = 0;
    if (threadIdx.x == 0)
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(aborted) : "l"(s.bar + 2) : "memory");
    bool up = __syncthreads_or(static_cast<int>(aborted)) == 0;  // no wait has run out
    for (int32_t l = 1; up && l <= s.iters; ++l) {
        const bool last = l == s.iters;
        cn.final_pass = (last || et) ? 1 : 0;
        cn.hb1 = s.cn.hb1 + (l & 1) * s.h1;
        if (s.hard1) small_checks<MsgT, W, kPassHard>(s, cn, t0, step);
        else small_checks<MsgT, W, kPassFull>(s, cn, t0, step);
        if (!(up = grid_barrier(s.bar, target))) break;
        vn.want_bits = cn.final_pass;
        for (int slab = 0; slab < s.slabs; ++slab) {
            if (et && slab_all_done<W>(done, slab)) continue;
            for (uint32_t t = place(slab, vn_threads); t < vn_threads; t += step)
                var_body<MsgT, W, kSmallRound<MsgT>>(vn, t, slab);
        }
        // the fail words of the other parity: every block has read them
        if (blockIdx.x == 0)
            for (int i = threadIdx.x; i < words; i += blockDim.x) s.fail[(1 - (l & 1)) * words + i] = 0u;
        if (!(up = grid_barrier(s.bar, target))) break;
        if (!cn.final_pass) continue;
        uint32_t *f = s.fail + (l & 1) * words;
        sy.fail = f;
        sy.hb1 = cn.hb1;
        for (int slab = 0; slab < s.slabs; ++slab) {
            if (et && slab_all_done<W>(done, slab)) continue;
            const uint32_t t = place(slab, syn_threads);  // whole warps
            if (t < syn_threads) syndrome_body<W>(sy, t, step, slab);
        }
        if (!(up = grid_barrier(s.bar, target))) break;
        // every block forms the same lane state from the same words
        for (int i = threadIdx.x; i < words; i += blockDim.x) fail[i] = __ldcg(f + i);
        __syncthreads();
        for (int b = threadIdx.x; b < s.batch; b += blockDim.x) {
            const int word = b / W * DW + b % W / 32;
            const uint32_t bit = 1u << (b % W & 31);
            if (et && (done[word] & bit)) continue;  // stopped at an earlier iteration
            const bool ok = (fail[word] & bit) == 0u;
            its[b] = l;
            conv[b] = ok ? 1 : 0;
            if (et && (ok || last)) atomicOr(done + word, bit);
        }
        __syncthreads();
        if (et) {
            bool all = true;
            for (int slab = 0; slab < s.slabs; ++slab) all = all && slab_all_done<W>(done, slab);
            if (all) break;
        }
    }
    // given up: no codeword counts as converged, after 0 iterations, and the
    // barrier is not reset
    if (blockIdx.x == 0) {
        if (!up && threadIdx.x == 0 && s.status) atomicCAS(s.status, 0, MLD_ETIMEOUT);
        for (int b = threadIdx.x; b < s.batch; b += blockDim.x) {
            const int32_t it = up ? its[b] : 0;
            const uint8_t cv = up ? conv[b] : 0;
            s.iters_dev[b] = it;
            s.conv_dev[b] = cv;
            if (s.iters_out) s.iters_out[b] = it;
            if (s.conv_out) s.conv_out[b] = cv;
        }
    }
    if (up) grid_leave(s.bar);
}

// Runs the iterations in one launch on st; false if the problem is not small or
// not of the kernel's form, or the launch is refused (then nothing was
// enqueued).
template <typename MsgT, int W>
bool launch_small(mld_decoder *d, int32_t batch, int32_t iters, bool et, bool hard1, int32_t *iters_out,
                  uint8_t *conv_out, int sm_count, cudaStream_t st, bool soft) {
    constexpr uint32_t TPC = W / kK;
    const mld::HostGraph &h = d->g->h;
    const mld_graph *g = d->g;
    const std::vector<ClassLaunch> &launches = g->launches[W == 8 ? 0 : (W == 16 ? 1 : (W == 32 ? 2 : 3))];
    SmallArgs s{};
    s.slabs = (batch + W - 1) / W;
    s.batch = batch;
    s.iters = iters;
    s.hard1 = hard1 ? 1 : 0;
    s.h1 = static_cast<size_t>(s.slabs) * h.n_deg1 * (W / 8);
    s.fail = d->fail;
    s.iters_dev = d->iters;
    s.conv_dev = d->conv;
    s.iters_out = iters_out;
    s.conv_out = conv_out;
    s.bar = d->bar;
    s.status = d->status;
    s.stall = d->stall_test;
    s.cn = CnArgs{g->cptr, g->col, g->dptr, h.n_cn, h.n_core, h.n_deg1, h.e_core, d->r, d->Lv, d->lch1, d->phi1,
                  d->post1, d->hb1, d->sbits, nullptr, d->lmax_i, d->amin_i, 0, et ? 1 : 0};
    s.cn.batch = batch;
    if (!et && !soft) s.cn.post1 = nullptr;
    s.vn = VnArgs{g->vptr, g->vedge, h.n_core, h.e_core, d->r, d->lch, d->Lv, d->hb_core, nullptr, 0, et ? 1 : 0};
    s.sy = SynArgs{g->cptr, g->col, g->dptr, h.n_cn, h.n_core, h.n_deg1, d->sbits, d->hb_core, d->hb1, d->fail,
                   nullptr, et ? 1 : 0, batch};
    if (launches.empty() || launches.size() > kSmallMaxClasses || s.batch > kSmallMaxLanes) return false;
    uint64_t at = 0;
    s.n_cls = 0;
    for (const ClassLaunch &cl : launches) {
        const int dd = cl.deg - cl.dc;
        if (cl.dc < 1 || cl.dc > kSmallMaxTerms || (dd != 0 && dd != 1)) return false;
        s.cls[s.n_cls] = cl;
        s.first[s.n_cls++] = static_cast<uint32_t>(at);
        at += (static_cast<uint64_t>(cl.count) * TPC * s.slabs + 31) / 32 * 32;
        if (at > static_cast<uint64_t>(kSmallMaxThreads)) return false;
    }
    s.first[s.n_cls] = static_cast<uint32_t>(at);
    if (static_cast<uint64_t>(s.vn.n_core) * (W / kVnLanes) > static_cast<uint64_t>(kSmallMaxThreads)) return false;
    // at least four warps a block, one block per SM at most (kSmallShareDiv)
    const int part = std::max(1, sm_count / kSmallShareDiv);
    const bool fits = at <= static_cast<uint64_t>(part) * kSmallBlock;
    const int blocks = static_cast<int>(std::max<uint64_t>(1, std::min<uint64_t>(fits ? part : sm_count, (at + 127) / 128)));
    void *args[] = {&s};
    if (cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(&k_small_decode<MsgT, W>), dim3(blocks),
                                    dim3(kSmallBlock), args, 0, st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

}  // namespace
