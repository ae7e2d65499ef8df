// Uneven batches: many codewords over several Tanner graphs (different
// rates and lengths), each group with its own iteration cap, decoded by one
// schedule of launches that is captured once into a CUDA graph and replayed
// with a single launch.  With early termination the iterations are the bodies of
// conditional loops inside that graph, run by the device until every codeword
// has stopped.
//
// The paper decodes a batch of codewords of one code with a fixed number of
// iterations (Results, "High speed error correction with MET-LDPC codes";
// Discussion).  Here every launch of the schedule covers the work of all
// jobs that share its kernel shape: a device table of segments (job, block
// range) tells each block which job, slab and check class it serves.  With
// early termination (Methods, Step 5) each codeword stops at its first
// syndrome match or at its job's cap; its slab is skipped once all its
// codewords have stopped, and lanes past the batch count as stopped from the
// start.
#include <algorithm>
#include <map>
#include <tuple>
#include <type_traits>

#include "kernels.cuh"

namespace {

// Everything a block needs to know about one job, resident in device memory.
struct JobDev {
    CnArgs cn;
    VnArgs vn;
    SynArgs sy;
    InArgs in;
    OutArgs out;
    const uint8_t *syn;
    const int32_t *cint;
    uint8_t *sbits;
    uint32_t *done, *fail;   // fail: two buffers of slabs*DW words (iteration parity)
    int32_t *iters;
    uint8_t *conv;
    int32_t n_vn, n_cn, batch, slabs, W, max_iters;
};

// One job's share of a launch: blocks block0 .. block0 + bps*slabs - 1.
struct Seg {
    int32_t job, block0, bps, slabs, flags;
    ClassLaunch cl;
};

// The segment of this block (segments are sorted by their first block, the
// first one's is 0): every lane looks at one.
__device__ __forceinline__ int find_seg(const Seg *segs, int nseg) {
    const int lane = threadIdx.x & 31;
    int below = 0;
    for (int i0 = 0; i0 < nseg; i0 += 32) {
        const int i = i0 + lane;
        below += __popc(__ballot_sync(0xFFFFFFFFu, i < nseg && segs[i].block0 <= static_cast<int32_t>(blockIdx.x)));
    }
    return below - 1;
}

// Check arguments of job j in an iteration of the given parity (its degree-1
// decision buffer).
template <int W>
__device__ __forceinline__ CnArgs job_cn(const JobDev &j, const Seg &sg, int parity) {
    CnArgs a = j.cn;
    a.final_pass = sg.flags & 1;
    a.hb1 = j.cn.hb1 + static_cast<size_t>(parity) * j.slabs * a.n_deg1 * (W / 8);
    return a;
}

template <typename MsgT, int W, int DC, int DD, int PASS>
__global__ void __launch_bounds__(kBlock, (kCheckBlocksPerSm<DC + DD>))
    km_check(const JobDev *jobs, const Seg *segs, int nseg, int parity) {
    const Seg sg = segs[find_seg(segs, nseg)];
    const CnArgs a = job_cn<W>(jobs[sg.job], sg, parity);
    const int local = blockIdx.x - sg.block0;
    const int slab = local / sg.bps;
    if (a.et && slab_all_done<W>(a.done, slab)) return;
    // the segment's grid is capped for register classes (build_plan)
    extern __shared__ __align__(128) unsigned char smem[];
    check_class_body<MsgT, W, DC, DD, PASS>(
        a, sg.cl, static_cast<int64_t>(local % sg.bps) * blockDim.x + threadIdx.x, sg.bps, slab, smem);
}

// Shapes of up to six terms share one launch: the graph's small classes (a few
// checks to a few percent) then cost blocks instead of launches, of which a
// plan of three rates has eight per width and iteration.
#define MLD_MERGED_SHAPES(X)                                                           \
    X(1, 0) X(2, 0) X(3, 0) X(4, 0) X(5, 0) X(6, 0)                                     \
    X(0, 1) X(1, 1) X(2, 1) X(3, 1) X(4, 1) X(5, 1)
template <typename MsgT>
constexpr int kMergedSmem = RingShape<MsgT, 6, 0>::kBytes > RingShape<MsgT, 5, 1>::kBytes ? RingShape<MsgT, 6, 0>::kBytes
                                                                                         : RingShape<MsgT, 5, 1>::kBytes;

template <typename MsgT, int W, int PASS>
__global__ void __launch_bounds__(kBlock, (kCheckBlocksPerSm<6>))
    km_check_merged(const JobDev *jobs, const Seg *segs, int nseg, int parity) {
    const Seg sg = segs[find_seg(segs, nseg)];
    const CnArgs a = job_cn<W>(jobs[sg.job], sg, parity);
    const int local = blockIdx.x - sg.block0;
    const int slab = local / sg.bps;
    if (a.et && slab_all_done<W>(a.done, slab)) return;
    extern __shared__ __align__(128) unsigned char smem[];
    const int64_t t0 = static_cast<int64_t>(local % sg.bps) * blockDim.x + threadIdx.x;
    switch (sg.cl.dc * 2 + (sg.cl.deg - sg.cl.dc)) {
#define X(DC, DD) \
    case (DC) * 2 + (DD): check_class_body<MsgT, W, DC, DD, PASS>(a, sg.cl, t0, sg.bps, slab, smem); break;
        MLD_MERGED_SHAPES(X)
#undef X
        default: break;
    }
}

template <typename MsgT, int W>
__global__ void __launch_bounds__(kBlock) km_check_irregular(const JobDev *jobs, const Seg *segs, int nseg,
                                                             int parity) {
    const Seg sg = segs[find_seg(segs, nseg)];
    const CnArgs a = job_cn<W>(jobs[sg.job], sg, parity);
    const int local = blockIdx.x - sg.block0;
    const int slab = local / sg.bps;
    if (a.et && slab_all_done<W>(a.done, slab)) return;
    check_irregular<MsgT, W>(a, sg.cl, static_cast<int64_t>(local % sg.bps) * blockDim.x + threadIdx.x, slab);
}

template <typename MsgT, int W>
__global__ void __launch_bounds__(kBlock) km_var(const JobDev *jobs, const Seg *segs, int nseg) {
    const Seg sg = segs[find_seg(segs, nseg)];
    VnArgs a = jobs[sg.job].vn;
    a.want_bits = sg.flags & 1;
    const int local = blockIdx.x - sg.block0;
    const int slab = local / sg.bps;
    if (a.et && slab_all_done<W>(a.done, slab)) return;
    var_body<MsgT, W>(a, static_cast<int64_t>(local % sg.bps) * blockDim.x + threadIdx.x, slab);
}

// parity: which of the two fail buffers this iteration uses
template <int W>
__global__ void __launch_bounds__(kBlock) km_syndrome(const JobDev *jobs, const Seg *segs, int nseg, int parity) {
    constexpr int DW = (W + 31) / 32;
    const Seg sg = segs[find_seg(segs, nseg)];
    const JobDev &j = jobs[sg.job];
    SynArgs a = j.sy;
    a.fail = j.fail + parity * j.slabs * DW;
    a.hb1 = j.sy.hb1 + static_cast<size_t>(parity) * j.slabs * a.n_deg1 * (W / 8);
    const int local = blockIdx.x - sg.block0;
    const int slab = local / sg.bps;
    if (a.et && slab_all_done<W>(a.done, slab)) return;
    syndrome_body<W>(a, static_cast<int64_t>(local % sg.bps) * blockDim.x + threadIdx.x,
                     static_cast<int64_t>(sg.bps) * blockDim.x, slab);
}

// Bookkeeping of iteration l (+ lctr[0] inside the loop) after its syndrome
// check: reads this iteration's fail words and clears the other buffer for the
// next.  With early termination a codeword stops at its syndrome match or at
// its job's cap.
template <int W>
__global__ void __launch_bounds__(kBlock) km_lane(const JobDev *jobs, const Seg *segs, int nseg, int32_t l,
                                                  int parity, const int32_t *lctr) {
    constexpr int DW = (W + 31) / 32;
    const Seg sg = segs[find_seg(segs, nseg)];
    const JobDev &j = jobs[sg.job];
    const int t = (blockIdx.x - sg.block0) * blockDim.x + threadIdx.x;
    if (lctr) l += lctr[0];
    lane_body<W>(j.done, j.fail + parity * j.slabs * DW, j.iters, j.conv, j.batch, l, j.max_iters, j.cn.et, t);
    if (t < j.slabs * DW) j.fail[(1 - parity) * j.slabs * DW + t] = 0u;
}

// Lane words of every job at the start: padding lanes count as stopped, no
// failures yet; the loop's iteration counter at 0.  One block per job.
__global__ void __launch_bounds__(kBlock) km_init(const JobDev *jobs, int32_t *lctr) {
    const JobDev &j = jobs[blockIdx.x];
    const int dw = (j.W + 31) / 32;
    for (int i = threadIdx.x; i < j.slabs * dw; i += blockDim.x)
        j.done[i] = padding_lanes(j.batch, j.W, i / dw, i % dw);
    for (int i = threadIdx.x; i < 2 * j.slabs * dw; i += blockDim.x) j.fail[i] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) *lctr = 0;
}

// Whether every lane of every job has stopped (one block).
__device__ __forceinline__ bool all_stopped(const JobDev *jobs, int n_jobs) {
    bool all = true;
    for (int k = 0; k < n_jobs; ++k) {
        const JobDev &j = jobs[k];
        const uint32_t full = j.W >= 32 ? 0xFFFFFFFFu : ((1u << j.W) - 1u);
        for (int i = threadIdx.x; i < j.slabs * ((j.W + 31) / 32); i += blockDim.x) all = all && j.done[i] == full;
    }
    return __syncthreads_and(all) != 0;
}

// End of a loop's body: counts its two iterations; continue while some lane
// still iterates and fewer than `end` are done.
__global__ void __launch_bounds__(kBlock) km_loop_cond(const JobDev *jobs, int n_jobs, int32_t *lctr, int32_t end,
                                                       cudaGraphConditionalHandle h) {
    const bool all = all_stopped(jobs, n_jobs);
    if (threadIdx.x == 0) {
        const int32_t l = *lctr + (all ? 0 : 2);
        *lctr = l;
        cudaGraphSetConditional(h, !all && l < end ? 1u : 0u);
    }
}

// Before a later loop: enter it if some lane still iterates.
__global__ void __launch_bounds__(kBlock) km_loop_enter(const JobDev *jobs, int n_jobs, cudaGraphConditionalHandle h) {
    const bool all = all_stopped(jobs, n_jobs);
    if (threadIdx.x == 0) cudaGraphSetConditional(h, all ? 0u : 1u);
}

template <int W, int F>
__global__ void __launch_bounds__(kBlock) km_interleave(const JobDev *jobs, const Seg *segs, int nseg) {
    const Seg sg = segs[find_seg(segs, nseg)];
    const int local = blockIdx.x - sg.block0;
    interleave_body<W, F>(jobs[sg.job].in, local % sg.bps, local / sg.bps);
}

template <int W>
__global__ void __launch_bounds__(kBlock) km_syndrome_in(const JobDev *jobs, const Seg *segs, int nseg) {
    const Seg sg = segs[find_seg(segs, nseg)];
    const JobDev &j = jobs[sg.job];
    const int local = blockIdx.x - sg.block0;
    syndrome_in_body<W>(j.syn, j.cint, j.n_cn, j.batch, j.sbits, local % sg.bps, local / sg.bps);
}

template <int W>
__global__ void __launch_bounds__(kBlock) km_deinterleave(const JobDev *jobs, const Seg *segs, int nseg) {
    const Seg sg = segs[find_seg(segs, nseg)];
    const int local = blockIdx.x - sg.block0;
    deinterleave_body<W>(jobs[sg.job].out, local % sg.bps, local / sg.bps);
}

// ---------------------------------------------------------------------------
// schedule
// ---------------------------------------------------------------------------
enum OpKind { kOpMemset, kOpInit, kOpInterleave, kOpSynIn, kOpHard, kOpCheck, kOpVar, kOpSyn, kOpLane, kOpOut };

struct Op {
    int kind = 0, half = 0, W = 0, dc = 0, dd = 0, parity = 0;
    int pass = 0;  // check ops: kPass*
    int32_t l = 0;
    bool in_loop = false;  // l counts from the loop's iteration counter
    int seg0 = 0, nseg = 0, blocks = 0;
    // memset / hard-decision ops
    void *ptr = nullptr;
    size_t bytes = 0;
    const float *post = nullptr;
    int32_t count = 0;
    uint8_t *hb = nullptr;
    int slabs = 0;
};

}  // namespace

struct mld_plan {
    int device = 0;
    JobDev *d_jobs = nullptr;
    Seg *d_segs = nullptr;
    int32_t *d_lctr = nullptr;  // iterations before the current loop body
    int n_jobs = 0;
    // the schedule: before, the early-termination loops (none without early
    // termination), after
    struct Loop {
        std::vector<Op> body;  // two iterations
        int32_t end;           // left when so many iterations are done
    };
    std::vector<Op> before, after;
    std::vector<Loop> loops;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

namespace {

int width_index(int W) { return W == 8 ? 0 : (W == 16 ? 1 : (W == 32 ? 2 : 3)); }

template <typename MsgT, int W>
void launch_check_op(const mld_plan *p, const Op &op, cudaStream_t st) {
    const JobDev *J = p->d_jobs;
    const Seg *S = p->d_segs + op.seg0;
    auto run = [&](auto bytes, auto kernel) {
        allow_smem<decltype(bytes)::value>(kernel);
        kernel<<<op.blocks, kBlock, decltype(bytes)::value, st>>>(J, S, op.nseg, op.parity);
    };
    if (op.dc == 0) {
        const std::integral_constant<int, kMergedSmem<MsgT>> sm;
        if (op.pass == kPassHard) run(sm, km_check_merged<MsgT, W, kPassHard>);
        else if (op.pass == kPassPlain) run(sm, km_check_merged<MsgT, W, kPassPlain>);
        else run(sm, km_check_merged<MsgT, W, kPassFull>);
        return;
    }
#define MLD_CASE(DCV, DDV)                                                                          \
    if (op.dc == (DCV) && op.dd == (DDV)) {                                                         \
        const std::integral_constant<int, RingShape<MsgT, DCV, DDV>::kBytes> sm;                    \
        if (op.pass == kPassHard) run(sm, km_check<MsgT, W, DCV, DDV, kPassHard>);                  \
        else if (op.pass == kPassPlain) run(sm, km_check<MsgT, W, DCV, DDV, kPassPlain>);           \
        else run(sm, km_check<MsgT, W, DCV, DDV, kPassFull>);                                       \
        return;                                                                                     \
    }
    MLD_CASE(7, 0) MLD_CASE(8, 0) MLD_CASE(6, 1) MLD_CASE(7, 1)
#undef MLD_CASE
    km_check_irregular<MsgT, W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg, op.parity);
}

template <int W>
void launch_op_w(const mld_plan *p, const Op &op, cudaStream_t st) {
    const JobDev *J = p->d_jobs;
    const Seg *S = p->d_segs + op.seg0;
    switch (op.kind) {
        case kOpInterleave:
            if (op.half) km_interleave<W, kFitB2H><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg);
            else km_interleave<W, kFitB2><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg);
            break;
        case kOpSynIn: km_syndrome_in<W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg); break;
        case kOpHard:
            k_hard_bits<W><<<dim3(grid_x(static_cast<int64_t>(op.count) * (W / 8)), op.slabs), kBlock, 0, st>>>(
                op.post, op.count, op.hb);
            break;
        case kOpCheck:
            if (op.half) launch_check_op<__half, W>(p, op, st);
            else launch_check_op<float, W>(p, op, st);
            break;
        case kOpVar:
            if (op.half) km_var<__half, W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg);
            else km_var<float, W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg);
            break;
        case kOpSyn: km_syndrome<W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg, op.parity); break;
        case kOpLane: km_lane<W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg, op.l, op.parity, op.in_loop ? p->d_lctr : nullptr);
            break;
        case kOpOut: km_deinterleave<W><<<op.blocks, kBlock, 0, st>>>(J, S, op.nseg); break;
        default: break;
    }
}

int enqueue(const mld_plan *p, const std::vector<Op> &ops, cudaStream_t st) {
    for (const Op &op : ops) {
        if (op.kind == kOpMemset) {
            MLD_CUDA(cudaMemsetAsync(op.ptr, 0, op.bytes, st));
            continue;
        }
        if (op.kind == kOpInit) {
            km_init<<<p->n_jobs, kBlock, 0, st>>>(p->d_jobs, p->d_lctr);
            MLD_LAUNCHED("km_init");
            continue;
        }
        switch (op.W) {
            case 8: launch_op_w<8>(p, op, st); break;
            case 16: launch_op_w<16>(p, op, st); break;
            case 32: launch_op_w<32>(p, op, st); break;
            default: launch_op_w<64>(p, op, st); break;
        }
        MLD_LAUNCHED("multi-job kernel");
    }
    return MLD_OK;
}

// Captures `fill` (work enqueued on the stream it is given) into graph g.
template <typename F>
int capture_into(cudaGraph_t g, cudaStream_t cs, F &&fill) {
    MLD_CUDA(cudaStreamBeginCaptureToGraph(cs, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    const int s = fill(cs);
    cudaGraph_t got = nullptr;
    const cudaError_t e = cudaStreamEndCapture(cs, &got);
    if (s != MLD_OK) return s;
    if (e != cudaSuccess) return cuda_fail(e, "plan: capture");
    return MLD_OK;
}

// The plan's graph: the ops before the loops, the loops (conditional nodes
// whose body graphs hold two iterations), the ops after them.
int build_graph(mld_plan *p, cudaStream_t cs) {
    MLD_CUDA(cudaGraphCreate(&p->graph, 0));
    cudaGraphNode_t last = nullptr;
    auto add_ops = [&](const std::vector<Op> &ops) -> int {
        if (ops.empty()) return MLD_OK;
        cudaGraph_t part = nullptr;
        MLD_CUDA(cudaGraphCreate(&part, 0));
        int s = capture_into(part, cs, [&](cudaStream_t st) { return enqueue(p, ops, st); });
        if (s == MLD_OK) {
            cudaGraphNode_t node = nullptr;
            const cudaError_t e = cudaGraphAddChildGraphNode(&node, p->graph, last ? &last : nullptr, last ? 1 : 0, part);
            if (e != cudaSuccess) s = cuda_fail(e, "plan: child graph");
            last = node;
        }
        cudaGraphDestroy(part);
        return s;
    };
    int s = add_ops(p->before);
    if (s != MLD_OK) return s;
    for (size_t k = 0; k < p->loops.size(); ++k) {
        const mld_plan::Loop &loop = p->loops[k];
        cudaGraphConditionalHandle h;
        MLD_CUDA(cudaGraphConditionalHandleCreate(&h, p->graph, 1, cudaGraphCondAssignDefault));
        if (k > 0) {
            void *args[] = {&p->d_jobs, &p->n_jobs, &h};
            cudaKernelNodeParams kp{};
            kp.func = reinterpret_cast<void *>(&km_loop_enter);
            kp.gridDim = dim3(1);
            kp.blockDim = dim3(kBlock);
            kp.kernelParams = args;
            cudaGraphNode_t enter = nullptr;
            MLD_CUDA(cudaGraphAddKernelNode(&enter, p->graph, &last, 1, &kp));
            last = enter;
        }
        cudaGraphNodeParams np{};
        np.type = cudaGraphNodeTypeConditional;
        np.conditional.handle = h;
        np.conditional.type = cudaGraphCondTypeWhile;
        np.conditional.size = 1;
        cudaGraphNode_t node = nullptr;
        MLD_CUDA(cudaGraphAddNode(&node, p->graph, &last, nullptr, 1, &np));
        last = node;
        s = capture_into(np.conditional.phGraph_out[0], cs, [&](cudaStream_t st) -> int {
            const int q = enqueue(p, loop.body, st);
            if (q != MLD_OK) return q;
            km_loop_cond<<<1, kBlock, 0, st>>>(p->d_jobs, p->n_jobs, p->d_lctr, loop.end, h);
            MLD_LAUNCHED("km_loop_cond");
            return MLD_OK;
        });
        if (s != MLD_OK) return s;
    }
    return add_ops(p->after);
}

int64_t kernels(const std::vector<Op> &ops) {
    int64_t n = 0;
    for (const Op &op : ops) n += (op.kind == kOpMemset) ? 0 : 1;
    return n;
}

void plan_free(mld_plan *p) {
    if (!p) return;
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    dfree(p->d_jobs);
    dfree(p->d_segs);
    dfree(p->d_lctr);
    delete p;
}

// Builds the jobs' device descriptors and the launch schedule.
int build_plan(const mld_job *jobs, int32_t n_jobs, uint32_t flags, mld_plan *p,
               std::vector<JobDev> &jd, std::vector<Seg> &segs) {
    const bool et = (flags & MLD_EARLY_TERM) != 0;
    int sm_count = 152;
    cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, p->device);
    int32_t lmax_iters = 0;
    for (int32_t j = 0; j < n_jobs; ++j) {
        const mld_job &jb = jobs[j];
        mld_decoder *d = jb.decoder;
        const mld::HostGraph &h = d->g->h;
        const int W = decode_width(d, jb.batch);
        const int slabs = (jb.batch + W - 1) / W;
        JobDev x{};
        const bool y_mode = jb.sigma != nullptr;
        x.cn = CnArgs{d->g->cptr, d->g->col, d->g->dptr, h.n_cn, h.n_core, h.n_deg1, h.e_core, d->r, d->Lv,
                      d->lch1, d->phi1, d->post1, d->hb1, d->sbits, d->done, d->lmax_i, d->amin_i, 0, et ? 1 : 0};
        x.cn.batch = jb.batch;
        x.vn = VnArgs{d->g->vptr, d->g->vedge, h.n_core, h.e_core, d->r, d->lch, d->Lv, d->hb_core, d->done, 0,
                      et ? 1 : 0};
        x.sy = SynArgs{d->g->cptr, d->g->col, d->g->dptr, h.n_cn, h.n_core, h.n_deg1, d->sbits, d->hb_core,
                       d->hb1, d->fail, d->done, et ? 1 : 0, jb.batch};
        x.in = InArgs{jb.in, y_mode ? jb.sigma : nullptr, d->g->unit, h.n_vn, h.n_core, h.n_deg1, jb.batch,
                      d->lmax, d->scale_in, d->lmax_i, d->amin_i, d->lch, d->Lv, d->lch1, d->post1, d->phi1};
        x.out = OutArgs{d->g->unit, h.n_vn, h.n_core, h.n_deg1, jb.batch, d->Lv, d->post1, d->hb1, jb.iters_used,
                        static_cast<size_t>(slabs) * h.n_deg1 * (W / 8), jb.bits_out,
                        jb.post_out, d->scale_out};
        x.syn = jb.syndrome;
        x.cint = d->g->cint;
        x.sbits = d->sbits;
        x.done = d->done;
        x.fail = d->fail;
        x.iters = jb.iters_used;
        x.conv = jb.converged;
        x.n_vn = h.n_vn;
        x.n_cn = h.n_cn;
        x.batch = jb.batch;
        x.slabs = slabs;
        x.W = W;
        x.max_iters = jb.max_iters;
        // (see the prologue of a single decode)
        if (jb.max_iters > 0) {
            x.in.post1 = nullptr;
            if (et && !jb.post_out && d->g->acc_ok) x.in.lch1 = nullptr;
            if (!et && !jb.post_out) x.cn.post1 = nullptr;
        }
        jd.push_back(x);
        lmax_iters = std::max(lmax_iters, jb.max_iters);
    }

    // one op per group key; segments of the group are the jobs' shares; ops
    // are appended to the part of the schedule being built
    std::vector<Op> *ops = &p->before;
    bool in_loop = false;
    using Key = std::tuple<int, int, int, int, int, int>;  // kind, half, W, dc, dd, pass
    auto flush = [&](std::map<Key, std::vector<Seg>> &groups, int32_t l, int parity) {
        for (auto &kv : groups) {
            Op op;
            op.kind = std::get<0>(kv.first);
            op.half = std::get<1>(kv.first);
            op.W = std::get<2>(kv.first);
            op.dc = std::get<3>(kv.first);
            op.dd = std::get<4>(kv.first);
            op.pass = std::get<5>(kv.first);
            op.l = l;
            op.in_loop = in_loop;
            op.parity = parity;
            op.seg0 = static_cast<int>(segs.size());
            op.nseg = static_cast<int>(kv.second.size());
            int32_t b0 = 0;
            for (Seg s : kv.second) {
                s.block0 = b0;
                b0 += s.bps * s.slabs;
                segs.push_back(s);
            }
            op.blocks = b0;
            if (op.blocks > 0) ops->push_back(op);
            else segs.resize(op.seg0);
        }
        groups.clear();
    };
    auto seg = [](int32_t job, int32_t bps, int32_t slabs, int32_t fl) {
        Seg s{};
        s.job = job;
        s.bps = bps;
        s.slabs = slabs;
        s.flags = fl;
        return s;
    };
    std::map<Key, std::vector<Seg>> groups;

    // prologue: clear messages and per-codeword state, interleave inputs
    for (int32_t j = 0; j < n_jobs; ++j) {
        const mld_decoder *d = jobs[j].decoder;
        const size_t msz = d->msg == MLD_MSG_F16 ? 2 : 4;
        Op m;
        m.kind = kOpMemset;
        m.ptr = d->r;
        m.bytes = static_cast<size_t>(jd[j].slabs) * d->g->h.e_core * jd[j].W * msz;
        if (m.bytes) ops->push_back(m);
    }
    if (n_jobs > 0) {
        Op m;
        m.kind = kOpInit;
        ops->push_back(m);
    }
    for (int32_t j = 0; j < n_jobs; ++j) {
        const mld_decoder *d = jobs[j].decoder;
        const int half = d->msg == MLD_MSG_F16;
        if (jd[j].n_vn > 0)
            groups[Key{kOpInterleave, half, jd[j].W, 0, 0, 0}].push_back(seg(j, (jd[j].n_vn + 31) / 32, jd[j].slabs, 0));
        if (jd[j].n_cn > 0)
            groups[Key{kOpSynIn, 0, jd[j].W, 0, 0, 0}].push_back(seg(j, (jd[j].n_cn + 31) / 32, jd[j].slabs, 0));
    }
    flush(groups, 0, 0);

    auto syndrome_round = [&](const std::vector<int32_t> &js, int32_t l) {
        const int parity = l & 1;
        for (int32_t j : js) {
            const int bps = syndrome_blocks(jd[j].n_cn, sm_count);
            if (jd[j].n_cn > 0) groups[Key{kOpSyn, 0, jd[j].W, 0, 0, 0}].push_back(seg(j, bps, jd[j].slabs, 0));
        }
        flush(groups, l, parity);
        for (int32_t j : js) {
            const int lanes = std::max(jd[j].batch, jd[j].slabs * ((jd[j].W + 31) / 32));
            groups[Key{kOpLane, 0, jd[j].W, 0, 0, 0}].push_back(seg(j, (lanes + kBlock - 1) / kBlock, 1, 0));
        }
        flush(groups, l, parity);
    };

    // jobs with no iteration: decisions from the channel values
    {
        std::vector<int32_t> zero;
        for (int32_t j = 0; j < n_jobs; ++j) {
            if (jobs[j].max_iters != 0) continue;
            mld_decoder *d = jobs[j].decoder;
            const mld::HostGraph &h = d->g->h;
            Op op;
            op.kind = kOpHard;
            op.W = jd[j].W;
            op.slabs = jd[j].slabs;
            if (h.n_core > 0) {
                op.post = d->Lv;
                op.count = h.n_core;
                op.hb = d->hb_core;
                ops->push_back(op);
            }
            if (h.n_deg1 > 0) {
                op.post = d->post1;
                op.count = h.n_deg1;
                op.hb = d->hb1;
                ops->push_back(op);
            }
            zero.push_back(j);
        }
        if (!zero.empty()) syndrome_round(zero, 0);
    }

    // iteration l (counted from the loop's counter inside the loop) of the
    // given jobs; `last_of(j)`: also form decisions and check the syndrome
    auto iteration = [&](const std::vector<int32_t> &active, int32_t l, auto &&last_of) {
        const int parity = l & 1;
        std::vector<int32_t> checked;
        for (int32_t j : active) {
            const mld_decoder *d = jobs[j].decoder;
            const int half = d->msg == MLD_MSG_F16;
            const int fl = last_of(j) ? 1 : 0;
            for (const ClassLaunch &cl : d->g->launches[width_index(jd[j].W)]) {
                const int dd = cl.deg - cl.dc;
                const bool regular = cl.dc >= 0 && (dd == 0 || dd == 1);
                // early termination without soft output: degree-1 decisions only
                const int pass = !regular ? kPassFull : (et && !jobs[j].post_out) ? kPassHard : fl ? kPassFull : kPassPlain;
                Seg s = seg(j, regular ? class_blocks(cl, sm_count) : cl.blocks, jd[j].slabs, fl);
                s.cl = cl;
                const bool merged = regular && cl.deg <= 6;
                groups[Key{kOpCheck, half, jd[j].W, merged ? 0 : regular ? cl.dc : -1, merged ? 0 : regular ? dd : -1, pass}]
                    .push_back(s);
            }
        }
        flush(groups, l, parity);
        for (int32_t j : active) {
            const mld_decoder *d = jobs[j].decoder;
            const int bps = grid_x(static_cast<int64_t>(d->g->h.n_core) * (jd[j].W / kVnLanes));
            const int fl = last_of(j) ? 1 : 0;
            if (d->g->h.n_core > 0)
                groups[Key{kOpVar, d->msg == MLD_MSG_F16, jd[j].W, 0, 0, 0}].push_back(seg(j, bps, jd[j].slabs, fl));
            if (fl) checked.push_back(j);
        }
        flush(groups, l, parity);
        if (!checked.empty()) syndrome_round(checked, l);
    };
    if (et) {
        // the device repeats two iterations until every codeword has stopped.  A
        // job past its cap still launches blocks that find nothing to do, so a
        // new loop without them begins where they outnumber the blocks of the
        // jobs that go on four to one (64 codewords of n = 200000 with a cap of 2
        // beside three of n = 4096 with one of 200: 6.0 ms in one loop, 3.9 ms in
        // two); not sooner, since a further loop costs 0.15 ms and more a launch
        // (96 codewords in nine jobs of three caps, all stopped at the first:
        // 15.2 ms in one loop, 15.5 ms in two or three)
        std::vector<std::pair<int32_t, int64_t>> caps;  // rounded up to even, blocks of an iteration
        int64_t going_on = 0, past = 0;
        for (int32_t j = 0; j < n_jobs; ++j) {
            if (jobs[j].max_iters == 0) continue;
            const mld::HostGraph &h = jobs[j].decoder->g->h;
            int64_t b = grid_x(static_cast<int64_t>(h.n_core) * (jd[j].W / kVnLanes)) + syndrome_blocks(jd[j].n_cn, sm_count);
            for (const ClassLaunch &cl : jobs[j].decoder->g->launches[width_index(jd[j].W)])
                b += cl.dc >= 0 ? class_blocks(cl, sm_count) : cl.blocks;
            b *= jd[j].slabs;
            caps.push_back({static_cast<int32_t>(std::min<int64_t>((jobs[j].max_iters + 1LL) / 2 * 2, INT32_MAX)), b});
            going_on += b;
        }
        std::sort(caps.begin(), caps.end());
        int32_t begin = 0;
        for (size_t k = 0; k < caps.size(); ++k) {
            past += caps[k].second;
            going_on -= caps[k].second;
            const bool last = k + 1 == caps.size();
            if (!last && (caps[k + 1].first == caps[k].first || past <= 4 * going_on)) continue;
            std::vector<int32_t> active;
            for (int32_t j = 0; j < n_jobs; ++j)
                if (jobs[j].max_iters > begin) active.push_back(j);
            p->loops.push_back({{}, caps[k].first});
            ops = &p->loops.back().body;
            in_loop = true;
            for (int32_t l = 1; l <= 2; ++l) iteration(active, l, [](int32_t) { return true; });
            in_loop = false;
            begin = caps[k].first;
            past = 0;
        }
    } else {
        for (int32_t l = 1; l <= lmax_iters; ++l) {
            std::vector<int32_t> active;
            for (int32_t j = 0; j < n_jobs; ++j)
                if (jobs[j].max_iters >= l) active.push_back(j);
            iteration(active, l, [&](int32_t j) { return jobs[j].max_iters == l; });
        }
    }
    ops = &p->after;

    for (int32_t j = 0; j < n_jobs; ++j)
        if (jd[j].n_vn > 0)
            groups[Key{kOpOut, 0, jd[j].W, 0, 0, 0}].push_back(seg(j, (jd[j].n_vn + 31) / 32, jd[j].slabs, 0));
    flush(groups, 0, 0);
    return MLD_OK;
}

int validate_jobs(const mld_job *jobs, int32_t n_jobs, uint32_t flags, int *device) {
    if (n_jobs < 0 || (n_jobs > 0 && !jobs)) return mld::fail(MLD_EINVAL, "plan: bad job list");
    if (flags & ~(MLD_EARLY_TERM | MLD_DEVICE_PTRS)) return mld::fail(MLD_EINVAL, "plan: unknown flag");
    int dev = -1;
    MLD_CUDA(cudaGetDevice(&dev));
    *device = dev;
    for (int32_t j = 0; j < n_jobs; ++j) {
        const mld_job &jb = jobs[j];
        const std::string at = "plan: job " + std::to_string(j) + ": ";
        if (!jb.decoder) return mld::fail(MLD_EINVAL, at + "null decoder");
        if (jb.decoder->device != dev) return mld::fail(MLD_EINVAL, at + "decoder belongs to another device");
        if (jb.batch < 1 || jb.batch > jb.decoder->max_batch) return mld::fail(MLD_EINVAL, at + "batch out of range");
        if (jb.max_iters < 0) return mld::fail(MLD_EINVAL, at + "negative max_iters");
        if (jb.decoder->schedule != MLD_SCHED_FLOODING || jb.decoder->check_rule != MLD_CHECK_SUM_PRODUCT)
            return mld::fail(MLD_EINVAL, at + "plans run flooding sum-product (layered or min-sum decoder given)");
        const mld::HostGraph &h = jb.decoder->g->h;
        if ((h.n_vn > 0 && (!jb.in || !jb.bits_out)) || (h.n_cn > 0 && !jb.syndrome) || !jb.converged ||
            !jb.iters_used)
            return mld::fail(MLD_EINVAL, at + "null data pointer");
        for (int32_t k = 0; k < j; ++k)
            if (jobs[k].decoder == jb.decoder) return mld::fail(MLD_EINVAL, at + "decoder shared with job " + std::to_string(k));
    }
    return MLD_OK;
}

}  // namespace

extern "C" {

int mld_plan_create(const mld_job *jobs, int32_t n_jobs, uint32_t flags, mld_plan **out) {
    mld::clear_error();
    if (!out) return mld::fail(MLD_EINVAL, "plan_create: null out");
    int dev = 0;
    int s = validate_jobs(jobs, n_jobs, flags, &dev);
    if (s != MLD_OK) return s;
    mld_plan *p = new (std::nothrow) mld_plan();
    if (!p) return mld::fail(MLD_ENOMEM, "plan_create: host allocation");
    p->device = dev;
    p->n_jobs = n_jobs;
    std::vector<JobDev> jd;
    std::vector<Seg> segs;
    s = build_plan(jobs, n_jobs, flags, p, jd, segs);
    if (s == MLD_OK) s = upload(&p->d_jobs, jd);
    if (s == MLD_OK) s = upload(&p->d_segs, segs);
    if (s == MLD_OK) s = dalloc(&p->d_lctr, 1);
    cudaStream_t cs = nullptr;
    if (s == MLD_OK) {
        cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
        if (e != cudaSuccess) s = cuda_fail(e, "cudaStreamCreate");
    }
    if (s == MLD_OK) s = build_graph(p, cs);
    if (s == MLD_OK) {
        cudaError_t e = cudaGraphInstantiate(&p->exec, p->graph, 0);
        if (e != cudaSuccess) s = cuda_fail(e, "cudaGraphInstantiate");
    }
    if (cs) cudaStreamDestroy(cs);
    if (s != MLD_OK) {
        plan_free(p);
        return s;
    }
    *out = p;
    return MLD_OK;
}

int mld_plan_launch(mld_plan *p, void *stream) {
    mld::clear_error();
    if (!p) return mld::fail(MLD_EINVAL, "plan_launch: null plan");
    int s = check_device(p->device);
    if (s != MLD_OK) return s;
    MLD_CUDA(cudaGraphLaunch(p->exec, static_cast<cudaStream_t>(stream)));
    return MLD_OK;
}

int mld_plan_stats(const mld_plan *p, int64_t *launches) {
    mld::clear_error();
    if (!p || !launches) return mld::fail(MLD_EINVAL, "plan_stats: null pointer");
    int64_t n = 0;
    for (size_t k = 0; k < p->loops.size(); ++k) n += kernels(p->loops[k].body) + (k > 0 ? 2 : 1);  // and its conditions
    *launches = n + kernels(p->before) + kernels(p->after);
    return MLD_OK;
}

int mld_plan_launched(const mld_plan *p, int32_t iterations, int64_t *launches) {
    mld::clear_error();
    if (!p || !launches) return mld::fail(MLD_EINVAL, "plan_launched: null pointer");
    if (iterations < 0) return mld::fail(MLD_EINVAL, "plan_launched: negative iterations");
    int64_t n = kernels(p->before) + kernels(p->after), l = 0;
    for (size_t k = 0; k < p->loops.size(); ++k) {
        if (k > 0) n += 1;  // its entry condition
        for (bool first = k == 0; first || (l < iterations && l < p->loops[k].end); first = false, l += 2)
            n += kernels(p->loops[k].body) + 1;
    }
    *launches = n;
    return MLD_OK;
}

int mld_plan_destroy(mld_plan *p) {
    if (!p) return MLD_OK;
    plan_free(p);
    return MLD_OK;
}

int mld_decode_multi(const mld_job *jobs, int32_t n_jobs, uint32_t flags, void *stream) {
    mld::clear_error();
    mld_plan *p = nullptr;
    int s = mld_plan_create(jobs, n_jobs, flags, &p);
    if (s != MLD_OK) return s;
    s = mld_plan_launch(p, stream);
    if (s == MLD_OK) {
        cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
        if (e != cudaSuccess) s = cuda_fail(e, "cudaStreamSynchronize");
    }
    plan_free(p);
    return s;
}

}  // extern "C"
