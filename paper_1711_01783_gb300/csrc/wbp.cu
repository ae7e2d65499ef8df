// Differentiable weighted BP: forward over T unrolled iterations with a
// learnable scale per (iteration, edge type) on every variable-to-check
// message, and its adjoint (reverse mode), checkpointed every k iterations.
//
// Forward (LLR domain, Methods Eqs. 2-5, with weights):
//   x_e^t = L_v^{t-1} - r_e^{t-1}     (degree-1 VN: x = L_ch)
//   q_e^t = clamp(w[t][type(e)] * x_e^t)
//   r_e^t = check update of the q^t (syndrome sign, phi, clamps)
//   L_v^t = L_ch(v) + sum_e r_e^t;   output L^T.
// All weights 1 is plain BP.  The adjoint differentiates every step exactly
// (clamps: 1 strictly inside, 0 outside; sign factors: 0; phi' = -1/sinh),
// recomputing each segment of k iterations from its stored messages.
#include "kernels.cuh"

namespace {

constexpr int kMaxTerms = 16;  // check degree supported by weighted BP
constexpr int kMaxTypes = MLD_MAX_EDGE_TYPES;

struct WArgs {
    const int32_t *cptr, *col, *dptr, *vptr, *vedge;
    const uint8_t *et_core, *et_deg1;
    int32_t n_cn, n_core, n_deg1, e_core, n_types;
    const uint8_t *sbits;
    const float *lch, *lch1;   // interleaved channel LLRs (clamped)
    const float *w;            // [T][n_types] weights, device
    float lmax, amin;
};

// 1 / sinh x for 0 < x: below 0.5 the reciprocal of sinh's Taylor polynomial
// (remainder x^8 / 9!, 1e-8 relative), above 2 e / (1 - e^2) with e = exp(-x),
// formed as 2^-(x log2 e) with the product's rounding error put back.  One
// reciprocal and no branch: sinhf and a division took most of the adjoint's
// instructions.
__device__ __forceinline__ float inv_sinh(float x) {
    const float y = x * 1.44269502f;
    const float lo = fmaf(x, 1.92596303e-8f, fmaf(x, 1.44269502f, -y));
    const float e = mufu_ex2(-y) * fmaf(lo, -0.693147181f, 1.f);
    const float t = x * x;
    const float poly = fmaf(t, fmaf(t, fmaf(t, 1.f / 5040.f, 1.f / 120.f), 1.f / 6.f), 1.f);
    const bool near = x < 0.5f;
    const float den = near ? x * poly : fmaf(-e, e, 1.f);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(den));
    return near ? r : (e + e) * r;
}

// phi of two values in nats: phi_f<kFitNat> on packed pairs, same roundings.
__device__ __forceinline__ float2 phi2_nat(float2 x) {
    auto both = [](float v) { return make_float2(v, v); };
    const float kLn2 = 0.693147180559945309f;
    const float2 t = __fmul2_rn(x, x);
    float2 ps = __ffma2_rn(both(-MLD_PHI_S4), t, both(-MLD_PHI_S3));
    ps = __ffma2_rn(ps, t, both(-MLD_PHI_S2));
    ps = __ffma2_rn(ps, t, both(-MLD_PHI_S1));
    ps = __ffma2_rn(ps, t, both(-MLD_PHI_S0));
    const float2 lg = make_float2(mufu_lg2(x.x), mufu_lg2(x.y));
    const float2 small = __ffma2_rn(t, ps, __ffma2_rn(both(-kLn2), lg, both(kLn2)));
    const float2 y = __fmul2_rn(x, both(-1.442695040888963407f));
    const float2 e = make_float2(mufu_ex2(y.x), mufu_ex2(y.y));
    const float2 z = __fmul2_rn(e, e);
    float2 pl = __ffma2_rn(both(MLD_PHI_L3), z, both(MLD_PHI_L2));
    pl = __ffma2_rn(pl, z, both(MLD_PHI_L1));
    pl = __ffma2_rn(pl, z, both(MLD_PHI_L0));
    const float2 large = __fmul2_rn(e, pl);
    return make_float2(sel_lt(x.x, MLD_PHI_X0, small.x, large.x), sel_lt(x.y, MLD_PHI_X0, small.y, large.y));
}

__device__ __forceinline__ float2 clamp2(float2 x, float lo, float hi) {
    return make_float2(clampf(x.x, lo, hi), clampf(x.y, lo, hi));
}
__device__ __forceinline__ float2 pair_of(const float4 &v, int p) {
    return p == 0 ? make_float2(v.x, v.y) : make_float2(v.z, v.w);
}

// ---------------------------------------------------------------------------
// Check kernels of the register classes: one launch covers every class of the
// graph, a block finds its class in a table and runs the body of its shape
// (DC core edges, DD degree-1 VNs), with every operand of a check requested
// before any arithmetic and the arithmetic two codewords at a time.  Bound by
// latency at the few blocks their registers allow: n = 10^5, 16 codewords, T =
// 20, training step 2.38 ms at 4 / 3 blocks per SM (forward / adjoint, no
// spills), 2.22 ms at 6 / 4, 2.33 ms at 8 / 5 (4.95 ms with the runtime-degree
// kernels, one launch per class).
// ---------------------------------------------------------------------------
constexpr int kMaxTable = 16;
struct ClassTable {
    mld::ClassLaunch cls[kMaxTable];
    int32_t first[kMaxTable + 1];  // first block of each class, and the end
    int n;
};

// Operands of one check for 4 codewords.
template <int W, int DC, int DD>
struct CheckOps {
    static constexpr int D = DC + DD;
    float4 lv[DC > 0 ? DC : 1], ro[DC > 0 ? DC : 1], l1[DD > 0 ? DD : 1];
    float wt[D];
    int ty[D];
    uint32_t sb;

    // rp: the messages of the previous iteration, null for none (all zero)
    __device__ __forceinline__ void load(const WArgs &a, const mld::ClassLaunch &cl, int32_t j, int slab, int lane0,
                                         int t, const float *rp, const float *lvp) {
        constexpr int NB = W / 8;
        const int32_t c = cl.c0 + j, e0 = cl.e0 + j * DC, s0 = cl.s0 + j * DD;
#pragma unroll
        for (int i = 0; i < DC; ++i) {
            lv[i] = ldf4(lvp + (static_cast<size_t>(slab) * a.n_core + __ldg(a.col + e0 + i)) * W + lane0);
            ro[i] = rp ? *reinterpret_cast<const float4 *>(rp + (static_cast<size_t>(slab) * a.e_core + e0 + i) * W + lane0)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
            ty[i] = a.et_core[e0 + i];
        }
#pragma unroll
        for (int i = 0; i < DD; ++i) {
            l1[i] = ldf4(a.lch1 + (static_cast<size_t>(slab) * a.n_deg1 + s0 + i) * W + lane0);
            ty[DC + i] = a.et_deg1[s0 + i];
        }
        sb = static_cast<uint32_t>(a.sbits[(static_cast<size_t>(slab) * a.n_cn + c) * NB + lane0 / 8]) >> (lane0 & 7);
        const float *row = a.w + static_cast<size_t>(t - 1) * a.n_types;
#pragma unroll
        for (int i = 0; i < D; ++i) wt[i] = __ldg(row + ty[i]);
    }
    // x_e of pair p: posterior minus own message (degree-1 VN: channel LLR)
    __device__ __forceinline__ float2 x(int i, int p) const {
        return i < DC ? sub2(pair_of(lv[i], p), pair_of(ro[i], p)) : pair_of(l1[i - DC], p);
    }
};

// The forward quantities of one pair of codewords.
template <int D>
struct PairState {
    float2 q[D], f[D], pre[D];
    float2 sg;  // product of signs and syndrome sign over all terms
    template <typename Ops>
    __device__ __forceinline__ void forward(const Ops &ops, const WArgs &a, int p) {
        sg = make_float2((ops.sb >> (2 * p)) & 1u ? -1.f : 1.f, (ops.sb >> (2 * p + 1)) & 1u ? -1.f : 1.f);
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < D; ++i) {
            q[i] = clamp2(__fmul2_rn(make_float2(ops.wt[i], ops.wt[i]), ops.x(i, p)), -a.lmax, a.lmax);
            f[i] = phi2_nat(clamp2(make_float2(fabsf(q[i].x), fabsf(q[i].y)), a.amin, a.lmax));
            if (q[i].x < 0.f) sg.x = -sg.x;
            if (q[i].y < 0.f) sg.y = -sg.y;
            pre[i] = acc;
            acc = add2(acc, f[i]);
        }
    }
    // sign of the other terms' product
    __device__ __forceinline__ float2 others(int i) const {
        return make_float2(q[i].x < 0.f ? -sg.x : sg.x, q[i].y < 0.f ? -sg.y : sg.y);
    }
};

// Forward check update of iteration t, codewords lane0 .. lane0+3: messages
// r_in (null: zero) and posteriors lv of iteration t-1 to messages r_out (which
// may be r_in); degree-1 posteriors written when `last`.
template <int W, int DC, int DD>
__device__ __forceinline__ void wbp_fwd(const WArgs &a, const mld::ClassLaunch &cl, int32_t j, int slab, int lane0,
                                        const float *r_in, float *r_out, const float *lv, float *post1, int t, int last) {
    constexpr int D = DC + DD;
    CheckOps<W, DC, DD> ops;
    ops.load(a, cl, j, slab, lane0, t, r_in, lv);
    float2 out[D][kP];
#pragma unroll
    for (int p = 0; p < kP; ++p) {
        PairState<D> s;
        s.forward(ops, a, p);
        float2 suf = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = D - 1; i >= 0; --i) {
            if (i < DC || last) {
                const float2 m = phi2_nat(clamp2(add2(s.pre[i], suf), a.amin, a.lmax));
                out[i][p] = __fmul2_rn(s.others(i), make_float2(fminf(m.x, a.lmax), fminf(m.y, a.lmax)));
            }
            suf = add2(suf, s.f[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < DC; ++i)
        *reinterpret_cast<float4 *>(r_out + (static_cast<size_t>(slab) * a.e_core + cl.e0 + j * DC + i) * W + lane0) =
            make_float4(out[i][0].x, out[i][0].y, out[i][1].x, out[i][1].y);
    if (last) {
#pragma unroll
        for (int i = 0; i < DD; ++i) {
            const float4 l = ops.l1[i];
            *reinterpret_cast<float4 *>(post1 + (static_cast<size_t>(slab) * a.n_deg1 + cl.s0 + j * DD + i) * W + lane0) =
                make_float4(l.x + out[DC + i][0].x, l.y + out[DC + i][0].y, l.z + out[DC + i][1].x,
                            l.w + out[DC + i][1].y);
        }
    }
}

// Adjoint of the check update of iteration t for 4 codewords.  dloss/dr^t of
// core edge e is G_v(e) - gx_e with gx the dloss/dx^{t+1} that this pass then
// replaces by dloss/dx^t (G, gx_used: see the launches); gd1: of the degree-1
// edges (only at t = T; else null).  glch1 accumulates dloss/dL_ch of the
// degree-1 VNs, gw the weight gradients per edge type.
template <int W, int DC, int DD>
__device__ __forceinline__ void wbp_bwd(const WArgs &a, const mld::ClassLaunch &cl, int32_t j, int slab, int lane0,
                                        const float *rp, const float *lvp, const float *G, bool gx_used, float *gx,
                                        const float *gd1, float *glch1, int t, float (&gw)[kMaxTypes]) {
    constexpr int D = DC + DD;
    const int32_t e0 = cl.e0 + j * DC, s0 = cl.s0 + j * DD;
    CheckOps<W, DC, DD> ops;
    ops.load(a, cl, j, slab, lane0, t, rp, lvp);
    float *gxr = gx + (static_cast<size_t>(slab) * a.e_core + e0) * W + lane0;
    const size_t d0 = (static_cast<size_t>(slab) * a.n_deg1 + s0) * W + lane0;
    float4 g[D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
        if (i < DC) {
            g[i] = ldf4(G + (static_cast<size_t>(slab) * a.n_core + __ldg(a.col + e0 + i)) * W + lane0);
            if (gx_used) {
                const float4 o = *reinterpret_cast<const float4 *>(gxr + i * W);
                g[i] = make_float4(g[i].x - o.x, g[i].y - o.y, g[i].z - o.z, g[i].w - o.w);
            }
        } else {
            g[i] = gd1 ? ldf4(gd1 + d0 + (i - DC) * W) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    float gwi[D];
    float2 out[D][kP];
#pragma unroll
    for (int i = 0; i < D; ++i) gwi[i] = 0.f;
#pragma unroll
    for (int p = 0; p < kP; ++p) {
        PairState<D> s;
        s.forward(ops, a, p);
        // g_o_i = sign_i * g_r_i * phi'(o_i) where o_i is strictly inside the clamp
        float2 go[D], suf = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = D - 1; i >= 0; --i) {
            const float2 o = add2(s.pre[i], suf), sgn = s.others(i), gi = pair_of(g[i], p);
            go[i].x = (o.x > a.amin && o.x < a.lmax) ? -sgn.x * gi.x * inv_sinh(o.x) : 0.f;
            go[i].y = (o.y > a.amin && o.y < a.lmax) ? -sgn.y * gi.y * inv_sinh(o.y) : 0.f;
            suf = add2(suf, s.f[i]);
        }
        // g_f_j = sum_{i != j} g_o_i (prefix + suffix), then back through phi,
        // |.|, the clamps (outside them |q| is amin or below, or lmax) and the weight
        float2 gpre[D], acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < D; ++i) {
            gpre[i] = acc;
            acc = add2(acc, go[i]);
        }
        float2 gsuf = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = D - 1; i >= 0; --i) {
            const float2 gf = add2(gpre[i], gsuf), x = ops.x(i, p);
            gsuf = add2(gsuf, go[i]);
            auto through = [&](float q, float gfk) {
                const float aq = fabsf(q);
                const float ga = (aq > a.amin && aq < a.lmax) ? -gfk * inv_sinh(aq) : 0.f;
                return q < 0.f ? -ga : ga;
            };
            const float2 gp = make_float2(through(s.q[i].x, gf.x), through(s.q[i].y, gf.y));
            gwi[i] = fmaf(gp.y, x.y, fmaf(gp.x, x.x, gwi[i]));
            out[i][p] = make_float2(gp.x * ops.wt[i], gp.y * ops.wt[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
#pragma unroll
        for (int k = 0; k < kMaxTypes; ++k) gw[k] += (k == ops.ty[i]) ? gwi[i] : 0.f;
        const float4 v = make_float4(out[i][0].x, out[i][0].y, out[i][1].x, out[i][1].y);
        if (i < DC) {
            *reinterpret_cast<float4 *>(gxr + i * W) = v;
        } else {
            float4 *pp = reinterpret_cast<float4 *>(glch1 + d0 + (i - DC) * W);
            float4 o = *pp;
            o.x += v.x; o.y += v.y; o.z += v.z; o.w += v.w;
            *pp = o;
        }
    }
}

// The block's class and its thread's check; false past the class's end.
template <int W>
__device__ __forceinline__ bool table_check(const ClassTable &tb, int &k, int32_t &j, int &lane0) {
    constexpr int TPC = W / kK;
    k = 0;
    while (static_cast<int32_t>(blockIdx.x) >= tb.first[k + 1]) ++k;
    const int32_t lt = (static_cast<int32_t>(blockIdx.x) - tb.first[k]) * kBlock + static_cast<int32_t>(threadIdx.x);
    j = lt / TPC;
    lane0 = (lt % TPC) * kK;
    return j < tb.cls[k].count;
}

#define MLD_WBP_SHAPES(X)                                                              \
    X(1, 0) X(2, 0) X(3, 0) X(4, 0) X(5, 0) X(6, 0) X(7, 0) X(8, 0)                     \
    X(0, 1) X(1, 1) X(2, 1) X(3, 1) X(4, 1) X(5, 1) X(6, 1) X(7, 1)

template <int W>
__global__ void __launch_bounds__(kBlock, 6) kw_fwd(WArgs a, ClassTable tb, const float *r_in, float *r_out,
                                                    const float *lv, float *post1, int t, int last) {
    int k, lane0;
    int32_t j;
    if (!table_check<W>(tb, k, j, lane0)) return;
    const mld::ClassLaunch &cl = tb.cls[k];
    switch (cl.dc * 2 + (cl.deg - cl.dc)) {
#define X(DC, DD) \
    case (DC) * 2 + (DD): wbp_fwd<W, DC, DD>(a, cl, j, blockIdx.y, lane0, r_in, r_out, lv, post1, t, last); break;
        MLD_WBP_SHAPES(X)
#undef X
        default: break;
    }
}

// Block partial sums of the weight gradient (deterministic order) into row
// `row` of gwp.  Every thread of the block must call it.
__device__ __forceinline__ void block_weight_sums(const float (&gw)[kMaxTypes], int n_types, float *gwp, size_t row) {
    __shared__ float red[kBlock / 32][kMaxTypes];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
#pragma unroll
    for (int k = 0; k < kMaxTypes; ++k) {
        if (k < n_types) {
            float v = gw[k];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
            if (lane == 0) red[warp][k] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < n_types) {
        float v = 0.f;
        for (int i = 0; i < kBlock / 32; ++i) v += red[i][threadIdx.x];
        gwp[row * n_types + threadIdx.x] = v;
    }
}

template <int W>
__global__ void __launch_bounds__(kBlock, 4) kw_bwd(WArgs a, ClassTable tb, const float *rp, const float *lvp,
                                                    const float *G, int gx_used, float *gx, const float *gd1,
                                                    float *glch1, float *gwp, int t) {
    float gw[kMaxTypes];
#pragma unroll
    for (int k = 0; k < kMaxTypes; ++k) gw[k] = 0.f;
    int k, lane0;
    int32_t j;
    if (table_check<W>(tb, k, j, lane0)) {
        const mld::ClassLaunch &cl = tb.cls[k];
        switch (cl.dc * 2 + (cl.deg - cl.dc)) {
#define X(DC, DD)                                                                                                  \
    case (DC) * 2 + (DD):                                                                                          \
        wbp_bwd<W, DC, DD>(a, cl, j, blockIdx.y, lane0, rp, lvp, G, gx_used != 0, gx, gd1, glch1, t, gw); break;
            MLD_WBP_SHAPES(X)
#undef X
            default: break;
        }
    }
    block_weight_sums(gw, a.n_types, gwp, static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x);
}

// Recomputes the forward quantities of one check (at most DMAX terms) for 4
// codewords at iteration t from r^{t-1} (rp) and L_v^{t-1} (lvp).  Loops run
// to DMAX with the check's degree as a guard, so the arrays stay in
// registers for small DMAX.
template <int W, int DMAX>
struct CheckState {
    int nce, deg;
    int32_t e0, s0;
    float x[DMAX][kK], q[DMAX][kK], f[DMAX][kK], pre[DMAX][kK];
    float wt[DMAX];
    int ty[DMAX];
    float sg[kK];  // product of signs and syndrome sign over all terms

    __device__ __forceinline__ void load(const WArgs &a, int c, int slab, int lane0, int t, const float *rp,
                                         const float *lvp) {
        constexpr int NB = W / 8;
        e0 = a.cptr[c];
        nce = a.cptr[c + 1] - e0;
        s0 = a.dptr[c];
        deg = nce + (a.dptr[c + 1] - s0);
        const uint32_t sb =
            (static_cast<uint32_t>(a.sbits[(static_cast<size_t>(slab) * a.n_cn + c) * NB + lane0 / 8]) >> (lane0 & 7));
        const float *wt_row = a.w + static_cast<size_t>(t - 1) * a.n_types;
#pragma unroll
        for (int k = 0; k < kK; ++k) sg[k] = ((sb >> k) & 1u) ? -1.f : 1.f;
        float acc[kK] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < DMAX; ++i) {
            if (i >= deg) continue;
            float4 xv;
            if (i < nce) {
                const int32_t e = e0 + i;
                const float4 lv = ldf4(lvp + (static_cast<size_t>(slab) * a.n_core + a.col[e]) * W + lane0);
                const float4 ro = rp ? ldf4(rp + (static_cast<size_t>(slab) * a.e_core + e) * W + lane0)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                xv = make_float4(lv.x - ro.x, lv.y - ro.y, lv.z - ro.z, lv.w - ro.w);
                ty[i] = a.et_core[e];
            } else {
                const int32_t sl = s0 + i - nce;
                xv = ldf4(a.lch1 + (static_cast<size_t>(slab) * a.n_deg1 + sl) * W + lane0);
                ty[i] = a.et_deg1[sl];
            }
            wt[i] = wt_row[ty[i]];
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                x[i][k] = f4get(xv, k);
                q[i][k] = clampf(wt[i] * x[i][k], -a.lmax, a.lmax);
                f[i][k] = phi_f<kFitNat>(clampf(fabsf(q[i][k]), a.amin, a.lmax));
                if (q[i][k] < 0.f) sg[k] = -sg[k];
                pre[i][k] = acc[k];
                acc[k] += f[i][k];
            }
        }
    }
};

// Forward check update of checks of any degree up to DMAX (edges through
// cptr / dptr), for the classes without a register shape.
template <int W, int DMAX>
__global__ void __launch_bounds__(kBlock) kw_check_fwd(WArgs a, const float *r_in, float *r, const float *lv, float *post1, int t,
                                                       int last, int32_t c0, int32_t count) {
    constexpr int TPC = W / kK;
    constexpr int NB = W / 8;
    const int slab = blockIdx.y;
    const int64_t lt = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (lt / TPC >= count) return;
    const int32_t c = c0 + static_cast<int32_t>(lt / TPC);
    const int lane0 = static_cast<int>(lt % TPC) * kK;
    const int32_t e0 = a.cptr[c], nce = a.cptr[c + 1] - e0;
    const int32_t s0 = a.dptr[c], deg = nce + (a.dptr[c + 1] - s0);
    const uint32_t sb =
        (static_cast<uint32_t>(a.sbits[(static_cast<size_t>(slab) * a.n_cn + c) * NB + lane0 / 8]) >> (lane0 & 7));
    const float *wt_row = a.w + static_cast<size_t>(t - 1) * a.n_types;
    float sg[kK], q[DMAX][kK], f[DMAX][kK], pre[DMAX][kK];
#pragma unroll
    for (int k = 0; k < kK; ++k) sg[k] = ((sb >> k) & 1u) ? -1.f : 1.f;
    float acc[kK] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < DMAX; ++i) {
        if (i < deg) {
            float4 xv;
            float wt;
            if (i < nce) {
                const int32_t e = e0 + i;
                const float4 l = ldf4(lv + (static_cast<size_t>(slab) * a.n_core + a.col[e]) * W + lane0);
                const float4 ro =
                    r_in ? *reinterpret_cast<const float4 *>(r_in + (static_cast<size_t>(slab) * a.e_core + e) * W + lane0)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
                xv = make_float4(l.x - ro.x, l.y - ro.y, l.z - ro.z, l.w - ro.w);
                wt = wt_row[a.et_core[e]];
            } else {
                const int32_t sl = s0 + i - nce;
                xv = ldf4(a.lch1 + (static_cast<size_t>(slab) * a.n_deg1 + sl) * W + lane0);
                wt = wt_row[a.et_deg1[sl]];
            }
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                q[i][k] = clampf(wt * f4get(xv, k), -a.lmax, a.lmax);
                f[i][k] = phi_f<kFitNat>(clampf(fabsf(q[i][k]), a.amin, a.lmax));
                if (q[i][k] < 0.f) sg[k] = -sg[k];
                pre[i][k] = acc[k];
                acc[k] += f[i][k];
            }
        }
    }
    float suf[kK] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = DMAX - 1; i >= 0; --i) {
        if (i >= deg) continue;
        const bool core = i < nce;
        if (core || last) {
            float4 rv;
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                const float o = clampf(pre[i][k] + suf[k], a.amin, a.lmax);
                const float m = fminf(phi_f<kFitNat>(o), a.lmax);
                const float sgn = (q[i][k] < 0.f) ? -sg[k] : sg[k];  // sign of the other terms
                f4set(rv, k, sgn * m);
            }
            if (core) {
                *reinterpret_cast<float4 *>(r + (static_cast<size_t>(slab) * a.e_core + e0 + i) * W + lane0) = rv;
            } else {
                const size_t o = (static_cast<size_t>(slab) * a.n_deg1 + s0 + i - nce) * W + lane0;
                const float4 l = ldf4(a.lch1 + o);
                *reinterpret_cast<float4 *>(post1 + o) = make_float4(l.x + rv.x, l.y + rv.y, l.z + rv.z, l.w + rv.w);
            }
        }
#pragma unroll
        for (int k = 0; k < kK; ++k) suf[k] += f[i][k];
    }
}

// Launches of one check pass: the register classes together, any other class
// by itself.
struct WbpClasses {
    ClassTable table;
    std::vector<mld::ClassLaunch> other;
    int32_t parts = 0;  // blocks of an adjoint pass over one slab
};

WbpClasses wbp_classes(const std::vector<mld::ClassLaunch> &launches) {
    WbpClasses c{};
    for (const mld::ClassLaunch &cl : launches) {
        const int dd = cl.deg - cl.dc;
        const bool shaped = cl.dc >= 0 && (dd == 0 || dd == 1) && cl.deg <= mld::kMaxRegDeg;
        if (shaped && c.table.n < kMaxTable) {
            c.table.cls[c.table.n] = cl;
            c.table.first[c.table.n + 1] = c.table.first[c.table.n] + cl.blocks;
            c.table.n++;
        } else {
            c.other.push_back(cl);
        }
        c.parts += cl.blocks;
    }
    return c;
}

// Classes of at most kMaxRegDeg terms that have no shape of their own (several
// degree-1 VNs on a check, or past the table's end) run the runtime-degree
// kernels with arrays of that size: 50 000 checks of four core edges and two
// degree-1 VNs, 16 codewords, six iterations 0.92 ms with arrays of 16, 0.64 ms with
// arrays of 8.
bool in_registers(const mld::ClassLaunch &cl) { return cl.deg >= 0 && cl.deg <= mld::kMaxRegDeg; }

template <int W>
void launch_fwd(const WArgs &wa, const WbpClasses &c, const float *r_in, float *r_out, const float *lv, float *post1,
                int t, int last, int slabs, cudaStream_t st) {
    if (c.table.n)
        kw_fwd<W><<<dim3(c.table.first[c.table.n], slabs), kBlock, 0, st>>>(wa, c.table, r_in, r_out, lv, post1, t, last);
    for (const mld::ClassLaunch &cl : c.other) {
        const dim3 grid(cl.blocks, slabs);
        if (in_registers(cl)) kw_check_fwd<W, mld::kMaxRegDeg><<<grid, kBlock, 0, st>>>(wa, r_in, r_out, lv, post1, t, last, cl.c0, cl.count);
        else kw_check_fwd<W, kMaxTerms><<<grid, kBlock, 0, st>>>(wa, r_in, r_out, lv, post1, t, last, cl.c0, cl.count);
    }
}

// Adjoint check update of checks of any degree up to DMAX (see wbp_bwd), for
// the classes without a register shape; block partials from row part0 of gwp.
template <int W, int DMAX>
__global__ void __launch_bounds__(kBlock) kw_check_bwd(WArgs a, const float *rp, const float *lvp, const float *G,
                                                       int gx_used, float *gx, const float *gd1, float *glch1,
                                                       float *gwp, int t,
                                                       int32_t c0, int32_t count, int32_t part0) {
    constexpr int TPC = W / kK;
    const int slab = blockIdx.y;
    const int64_t lt = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    float gw[kMaxTypes];
#pragma unroll
    for (int k = 0; k < kMaxTypes; ++k) gw[k] = 0.f;
    if (lt / TPC < count) {
        const int32_t c = c0 + static_cast<int32_t>(lt / TPC);
        const int lane0 = static_cast<int>(lt % TPC) * kK;
        CheckState<W, DMAX> s;
        s.load(a, c, slab, lane0, t, rp, lvp);
        // g_o_i = sign_i * g_r_i * phi'(o_i) where o_i is strictly inside the clamp
        float go[DMAX][kK];
        float suf[kK] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = DMAX - 1; i >= 0; --i) {
            if (i >= s.deg) continue;
            const bool core = i < s.nce;
            float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
            if (core) {
                g = ldf4(G + (static_cast<size_t>(slab) * a.n_core + __ldg(a.col + s.e0 + i)) * W + lane0);
                if (gx_used) {
                    const float4 o = *reinterpret_cast<const float4 *>(
                        gx + (static_cast<size_t>(slab) * a.e_core + s.e0 + i) * W + lane0);
                    g = make_float4(g.x - o.x, g.y - o.y, g.z - o.z, g.w - o.w);
                }
            } else if (gd1)
                g = ldf4(gd1 + (static_cast<size_t>(slab) * a.n_deg1 + s.s0 + i - s.nce) * W + lane0);
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                const float o = s.pre[i][k] + suf[k];
                const float sgn = (s.q[i][k] < 0.f) ? -s.sg[k] : s.sg[k];
                go[i][k] = (o > a.amin && o < a.lmax) ? -sgn * f4get(g, k) * inv_sinh(o) : 0.f;
                suf[k] += s.f[i][k];
            }
        }
        // g_f_j = sum_{i != j} g_o_i (prefix + suffix), then back through phi, |.|, clamp, weight
        float gpre[DMAX][kK];
        float acc[kK] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < DMAX; ++i) {
            if (i >= s.deg) continue;
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                gpre[i][k] = acc[k];
                acc[k] += go[i][k];
            }
        }
        float gsuf[kK] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = DMAX - 1; i >= 0; --i) {
            if (i >= s.deg) continue;
            float gxd[kK];
            float gwi = 0.f;  // this term's weight gradient over the 4 codewords
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                const float gf = gpre[i][k] + gsuf[k];
                gsuf[k] += go[i][k];
                const float aq = fabsf(s.q[i][k]);
                const float ga = (aq > a.amin && aq < a.lmax) ? -gf * inv_sinh(aq) : 0.f;
                const float gq = s.q[i][k] > 0.f ? ga : (s.q[i][k] < 0.f ? -ga : 0.f);
                const float p = s.wt[i] * s.x[i][k];
                const float gp = (p > -a.lmax && p < a.lmax) ? gq : 0.f;
                gwi += gp * s.x[i][k];
                gxd[k] = gp * s.wt[i];
            }
#pragma unroll
            for (int k = 0; k < kMaxTypes; ++k) gw[k] += (k == s.ty[i]) ? gwi : 0.f;
            const float4 gxv = make_float4(gxd[0], gxd[1], gxd[2], gxd[3]);
            if (i < s.nce) {
                *reinterpret_cast<float4 *>(gx + (static_cast<size_t>(slab) * a.e_core + s.e0 + i) * W + lane0) = gxv;
            } else {
                float *pp = glch1 + (static_cast<size_t>(slab) * a.n_deg1 + s.s0 + i - s.nce) * W + lane0;
                float4 o = *reinterpret_cast<float4 *>(pp);
                o.x += gxv.x; o.y += gxv.y; o.z += gxv.z; o.w += gxv.w;
                *reinterpret_cast<float4 *>(pp) = o;
            }
        }
    }
    block_weight_sums(gw, a.n_types, gwp,
                      static_cast<size_t>(part0) + static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x);
}

template <int W>
void launch_bwd(const WArgs &wa, const WbpClasses &c, const float *rp, const float *lvp, const float *G, int gx_used,
                float *gx, const float *gd1, float *glch1, float *gwp, int t, int slabs, cudaStream_t st) {
    int32_t part0 = 0;
    if (c.table.n) {
        const int32_t blocks = c.table.first[c.table.n];
        kw_bwd<W><<<dim3(blocks, slabs), kBlock, 0, st>>>(wa, c.table, rp, lvp, G, gx_used, gx, gd1, glch1, gwp, t);
        part0 = blocks * slabs;
    }
    for (const mld::ClassLaunch &cl : c.other) {
        const dim3 grid(cl.blocks, slabs);
        if (in_registers(cl)) kw_check_bwd<W, mld::kMaxRegDeg><<<grid, kBlock, 0, st>>>(wa, rp, lvp, G, gx_used, gx, gd1, glch1, gwp, t, cl.c0, cl.count, part0);
        else kw_check_bwd<W, kMaxTerms><<<grid, kBlock, 0, st>>>(wa, rp, lvp, G, gx_used, gx, gd1, glch1, gwp, t, cl.c0, cl.count, part0);
        part0 += cl.blocks * slabs;
    }
}

// Adjoint of x_e^t = L_ch(v) + sum_{e' != e} r_{e'}^{t-1} at core VN v:
// G = sum_e gx_e; dL_ch += G.  (dr_{e'}^{t-1} = G - gx_{e'} is formed by the
// adjoint check update that reads it: the edge gradients are then gathered
// once and not scattered.)  Rows in CSC order, several in flight.
template <int W>
__global__ void __launch_bounds__(kBlock) kw_var_bwd(WArgs a, const float *gx, float *glch, float *G) {
    constexpr int TPC = W / kK;
    constexpr int kRound = 8;
    const int slab = blockIdx.y;
    const int64_t lt = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int32_t v = static_cast<int32_t>(lt / TPC);
    if (v >= a.n_core) return;
    const int lane0 = static_cast<int>(lt % TPC) * kK;
    const float *row = gx + static_cast<size_t>(slab) * a.e_core * W + lane0;
    const size_t o0 = (static_cast<size_t>(slab) * a.n_core + v) * W + lane0;
    float4 o = *reinterpret_cast<float4 *>(glch + o0);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const int32_t j1 = __ldg(a.vptr + v + 1);
    for (int32_t j = __ldg(a.vptr + v); j < j1; j += kRound) {
        float4 g[kRound];
#pragma unroll
        for (int k = 0; k < kRound; ++k)
            if (j + k < j1) g[k] = ldf4(row + static_cast<size_t>(__ldg(a.vedge + j + k)) * W);
#pragma unroll
        for (int k = 0; k < kRound; ++k)
            if (j + k < j1) { s.x += g[k].x; s.y += g[k].y; s.z += g[k].z; s.w += g[k].w; }
    }
    o.x += s.x; o.y += s.y; o.z += s.z; o.w += s.w;
    *reinterpret_cast<float4 *>(glch + o0) = o;
    *reinterpret_cast<float4 *>(G + o0) = s;
}

// Natural [B][n] -> interleaved core / degree-1 arrays (32 VNs x W codewords per block).
template <int W>
__global__ void __launch_bounds__(kBlock) kw_interleave(const float *in, const int32_t *unit, int32_t n_vn,
                                                        int32_t n_core, int32_t n_deg1, int32_t batch, float *core,
                                                        float *core_copy, float *deg1, float *deg1_copy) {
    __shared__ float tile[W][33];
    const int slab = blockIdx.y;
    const int32_t j0 = blockIdx.x * 32;
    for (int idx = threadIdx.x; idx < W * 32; idx += blockDim.x) {
        const int w = idx / 32, jj = idx % 32;
        const int b = slab * W + w;
        const int32_t j = j0 + jj;
        tile[w][jj] = (b < batch && j < n_vn) ? in[static_cast<size_t>(b) * n_vn + j] : 0.f;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < W * 32; idx += blockDim.x) {
        const int jj = idx / W, w = idx % W;
        const int32_t j = j0 + jj;
        if (j >= n_vn) continue;
        const int32_t u = unit[j];
        const float v = tile[w][jj];
        if (u < n_core) {
            const size_t o = (static_cast<size_t>(slab) * n_core + u) * W + w;
            core[o] = v;
            core_copy[o] = v;
        } else {
            const size_t o = (static_cast<size_t>(slab) * n_deg1 + (u - n_core)) * W + w;
            deg1[o] = v;
            deg1_copy[o] = v;
        }
    }
}

// Interleaved gradients -> natural [B][n], zero where the input LLR was clamped.
template <int W>
__global__ void __launch_bounds__(kBlock) kw_deinterleave(const float *core, const float *deg1, const float *lch,
                                                          const float *lch1, const int32_t *unit, int32_t n_vn,
                                                          int32_t n_core, int32_t n_deg1, int32_t batch, float lmax,
                                                          float *out) {
    __shared__ float tile[32][W + 1];
    const int slab = blockIdx.y;
    const int32_t j0 = blockIdx.x * 32;
    for (int idx = threadIdx.x; idx < W * 32; idx += blockDim.x) {
        const int jj = idx / W, w = idx % W;
        const int32_t j = j0 + jj;
        float v = 0.f;
        if (j < n_vn) {
            const int32_t u = unit[j];
            size_t o;
            float l;
            if (u < n_core) {
                o = (static_cast<size_t>(slab) * n_core + u) * W + w;
                v = core[o];
                l = lch[o];
            } else {
                o = (static_cast<size_t>(slab) * n_deg1 + (u - n_core)) * W + w;
                v = deg1[o];
                l = lch1[o];
            }
            if (!(fabsf(l) < lmax)) v = 0.f;  // L_ch = clamp(llr): no gradient when clamped
        }
        tile[jj][w] = v;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < W * 32; idx += blockDim.x) {
        const int w = idx / 32, jj = idx % 32;
        const int b = slab * W + w;
        const int32_t j = j0 + jj;
        if (b < batch && j < n_vn) out[static_cast<size_t>(b) * n_vn + j] = tile[jj][w];
    }
}

// Sum over the per-block partials of each weight type in a fixed order
// (strided over the threads, then a shared-memory tree), so the result does
// not depend on scheduling.  One block per iteration (row block y of gwp).
constexpr int kReduceThreads = 256;
__global__ void __launch_bounds__(kReduceThreads) kw_reduce_dw(const float *gwp, int blocks, int n_types,
                                                               float *dw) {
    __shared__ float part[kReduceThreads];
    gwp += static_cast<size_t>(blockIdx.x) * blocks * n_types;
    float *dw_row = dw + static_cast<size_t>(blockIdx.x) * n_types;
    for (int k = 0; k < n_types; ++k) {
        float v = 0.f;
        for (int b = threadIdx.x; b < blocks; b += kReduceThreads) v += gwp[static_cast<size_t>(b) * n_types + k];
        part[threadIdx.x] = v;
        __syncthreads();
        for (int o = kReduceThreads / 2; o > 0; o >>= 1) {
            if (static_cast<int>(threadIdx.x) < o) part[threadIdx.x] += part[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) dw_row[k] = part[0];
        __syncthreads();
    }
}

}  // namespace

struct mld_tape {
    mld_decoder *d = nullptr;
    int32_t batch = 0, T = 0, k = 1, n_types = 0, slabs = 0;
    float *w = nullptr;                 // [T][n_types]
    std::vector<float *> ckpt;          // r^{k}, r^{2k}, ... (r^0 = 0)
    float *seg_r = nullptr, *seg_lv = nullptr;  // k message / posterior arrays
    float *G = nullptr, *gx = nullptr;           // VN sums and edge gradients
    float *glch = nullptr, *glch1 = nullptr, *gd1 = nullptr;
    float *gwp = nullptr;
    int gwp_blocks = 0;
    // The iterations of the forward and the segments of the adjoint, as
    // CUDA graphs over this tape's (and its decoder's) fixed buffers:
    // captured at first use, replayed by later calls with this tape.
    cudaGraphExec_t fwd_exec = nullptr, bwd_exec = nullptr;
    float *dw = nullptr;  // [T][n_types], copied to the caller's dw
};

namespace {

void tape_free(mld_tape *t) {
    if (!t) return;
    if (t->fwd_exec) cudaGraphExecDestroy(t->fwd_exec);
    if (t->bwd_exec) cudaGraphExecDestroy(t->bwd_exec);
    dfree(t->dw);
    dfree(t->w);
    for (float *&p : t->ckpt) dfree(p);
    dfree(t->seg_r); dfree(t->seg_lv); dfree(t->G); dfree(t->gx);
    dfree(t->glch); dfree(t->glch1); dfree(t->gd1); dfree(t->gwp);
    delete t;
}

// Enqueues `enqueue(stream)` on st through the CUDA graph *exec: captured
// on the decoder's capture stream the first time (so that a few hundred
// small launches become one), replayed after.  Where capture is not
// possible (no capture stream, or another capture owns this thread) the
// work is launched directly.
template <typename F>
int run_graph(mld_decoder *d, cudaGraphExec_t *exec, cudaStream_t st, F &&enqueue) {
    if (!*exec) {
        if (!d->cap) return enqueue(st);
        cudaError_t e = cudaStreamBeginCapture(d->cap, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return enqueue(st);
        }
        const int s = enqueue(d->cap);
        cudaGraph_t gr = nullptr;
        const cudaError_t ec = cudaStreamEndCapture(d->cap, &gr);
        if (s != MLD_OK || ec != cudaSuccess) {
            if (gr) cudaGraphDestroy(gr);
            return s != MLD_OK ? s : cuda_fail(ec, "weighted BP: graph capture");
        }
        e = cudaGraphInstantiate(exec, gr, 0);
        cudaGraphDestroy(gr);
        if (e != cudaSuccess) {
            *exec = nullptr;
            return cuda_fail(e, "weighted BP: graph instantiation");
        }
    }
    MLD_CUDA(cudaGraphLaunch(*exec, st));
    return MLD_OK;
}

WArgs wargs(const mld_decoder *d, const float *w, int n_types) {
    const mld::HostGraph &h = d->g->h;
    return WArgs{d->g->cptr, d->g->col, d->g->dptr, d->g->vptr, d->g->vedge, d->g->etype_core, d->g->etype_deg1,
                 h.n_cn, h.n_core, h.n_deg1, h.e_core, n_types, d->sbits, d->lch, d->lch1, w, d->lmax, d->amin};
}

// Variable update: posteriors lv from messages r.
template <int W>
int wbp_posteriors(mld_decoder *d, const float *r, float *lv, int slabs, cudaStream_t st) {
    const mld::HostGraph &h = d->g->h;
    if (h.n_core == 0) return MLD_OK;
    VnArgs va{d->g->vptr, d->g->vedge, h.n_core, h.e_core, r, d->lch, lv, d->hb_core, d->done, 0, 0};
    k_var_update<float, W><<<dim3(grid_x(static_cast<int64_t>(h.n_core) * (W / kVnLanes)), slabs), kBlock, 0, st>>>(va);
    MLD_LAUNCHED("k_var_update");
    return MLD_OK;
}

const std::vector<mld::ClassLaunch> &width_launches(const mld_decoder *d, int W) {
    return d->g->launches[W == 8 ? 0 : (W == 16 ? 1 : (W == 32 ? 2 : 3))];
}

template <int W>
int wbp_forward_w(mld_decoder *d, const float *llr, const uint8_t *syn, int32_t batch, int32_t T, mld_tape *tape,
                  const float *w, int n_types, float *soft, cudaStream_t st) {
    const mld::HostGraph &h = d->g->h;
    const int slabs = (batch + W - 1) / W;
    // weighted BP works in nats: no scaling on entry or exit
    InArgs ia{llr, nullptr, d->g->unit, h.n_vn, h.n_core, h.n_deg1, batch, d->lmax, 1.f, d->lmax, d->amin,
              d->lch, d->Lv, d->lch1, d->post1, d->phi1};
    // (the first iteration reads no messages: nothing to clear)
    const PrologueArgs pa{ia, syn, d->g->cint, d->sbits, h.n_cn, (h.n_vn + 31) / 32, nullptr, 0};
    if (h.n_vn > 0 || h.n_cn > 0) {
        k_prologue<W, kFitNat><<<dim3(pa.in_tiles + (h.n_cn + 31) / 32, slabs), kBlock, 0, st>>>(pa);
        MLD_LAUNCHED("k_prologue");
    }
    const WArgs wa = wargs(d, w, n_types);
    auto iters = [&](cudaStream_t s2) -> int {
        // an iteration whose messages the tape keeps writes them there
        const WbpClasses classes = wbp_classes(width_launches(d, W));
        const float *r_in = nullptr;
        for (int t = 1; t <= T; ++t) {
            const bool keep = tape && t % tape->k == 0 && t < T;
            float *r_out = keep ? tape->ckpt[t / tape->k - 1] : static_cast<float *>(d->r);
            launch_fwd<W>(wa, classes, r_in, r_out, d->Lv, d->post1, t, t == T ? 1 : 0, slabs, s2);
            MLD_LAUNCHED("kw_fwd");
            const int q = wbp_posteriors<W>(d, r_out, d->Lv, slabs, s2);
            if (q != MLD_OK) return q;
            r_in = r_out;
        }
        return MLD_OK;
    };
    // with a tape every buffer the iterations touch is fixed for the tape's
    // life (the weights were copied into it), so they run as a graph
    int s = tape ? run_graph(d, &tape->fwd_exec, st, iters) : iters(st);
    if (s != MLD_OK) return s;
    OutArgs oa{d->g->unit, h.n_vn, h.n_core, h.n_deg1, batch, d->Lv, d->post1, d->hb1, nullptr, 0, d->bits_stage,
               soft, 1.f};
    if (h.n_vn > 0) {
        k_deinterleave_out<W><<<dim3((h.n_vn + 31) / 32, slabs), kBlock, 0, st>>>(oa);
        MLD_LAUNCHED("k_deinterleave_out");
    }
    return MLD_OK;
}

template <int W>
int wbp_backward_w(mld_tape *tp, const float *dsoft, float *dw, float *dllr, cudaStream_t st) {
    mld_decoder *d = tp->d;
    const mld::HostGraph &h = d->g->h;
    constexpr int TPC = W / kK;
    const int slabs = tp->slabs, T = tp->T, K = tp->k;
    const size_t rsz = static_cast<size_t>(slabs) * h.e_core * W;
    const size_t lsz = static_cast<size_t>(slabs) * h.n_core * W;
    const size_t dsz = static_cast<size_t>(slabs) * h.n_deg1 * W;
    const WArgs wa = wargs(d, tp->w, tp->n_types);
    const dim3 vgrid(grid_x(static_cast<int64_t>(h.n_core) * TPC), slabs);
    const WbpClasses classes = wbp_classes(width_launches(d, W));
    const int32_t parts = classes.parts * slabs;  // block partials of one adjoint check pass

    // dloss/dL^T: into dL_ch (the posterior is L_ch + sum r^T) and onto r^T
    if (lsz) MLD_CUDA(cudaMemsetAsync(tp->glch, 0, lsz * sizeof(float), st));
    if (dsz) MLD_CUDA(cudaMemsetAsync(tp->glch1, 0, dsz * sizeof(float), st));
    if (h.n_vn > 0) {
        kw_interleave<W><<<dim3((h.n_vn + 31) / 32, slabs), kBlock, 0, st>>>(
            dsoft, d->g->unit, h.n_vn, h.n_core, h.n_deg1, tp->batch, tp->glch, tp->G, tp->glch1, tp->gd1);
        MLD_LAUNCHED("kw_interleave");
    }
    // from dL^T on, every buffer is the tape's or the decoder's: the
    // segments run as a graph (dw into the tape, then copied out)
    auto segments = [&](cudaStream_t s2) -> int {
        // dloss/dr^T of core edge e is dloss/dL_v(e): G holds it, no gx yet
        for (int t0 = ((T - 1) / K) * K; t0 >= 0; t0 -= K) {
            const int t1 = std::min(t0 + K, T);
            // recompute r^{t0+1} .. r^{t1-1} and L^{t0} .. L^{t1-1}
            auto seg_r = [&](int t) -> const float * {
                return t == 0 ? nullptr : t == t0 ? tp->ckpt[t0 / K - 1] : tp->seg_r + static_cast<size_t>(t - t0 - 1) * rsz;
            };
            auto seg_lv = [&](int t) { return tp->seg_lv + static_cast<size_t>(t - t0) * lsz; };
            if (t0 == 0) {  // no messages: the posteriors are the channel values
                if (lsz)
                    MLD_CUDA(cudaMemcpyAsync(seg_lv(0), d->lch, lsz * sizeof(float), cudaMemcpyDeviceToDevice, s2));
            } else {
                const int q = wbp_posteriors<W>(d, seg_r(t0), seg_lv(t0), slabs, s2);
                if (q != MLD_OK) return q;
            }
            for (int t = t0 + 1; t < t1; ++t) {
                float *out = const_cast<float *>(seg_r(t));
                launch_fwd<W>(wa, classes, seg_r(t - 1), out, seg_lv(t - 1), d->post1, t, 0, slabs, s2);
                MLD_LAUNCHED("kw_fwd");
                const int q = wbp_posteriors<W>(d, out, seg_lv(t), slabs, s2);
                if (q != MLD_OK) return q;
            }
            for (int t = t1; t > t0; --t) {
                launch_bwd<W>(wa, classes, seg_r(t - 1), seg_lv(t - 1), tp->G, t < T ? 1 : 0, tp->gx,
                              t == T ? tp->gd1 : nullptr, tp->glch1,
                              tp->gwp + static_cast<size_t>(t - 1) * parts * tp->n_types, t, slabs, s2);
                MLD_LAUNCHED("kw_bwd");
                if (h.n_core > 0) {
                    kw_var_bwd<W><<<vgrid, kBlock, 0, s2>>>(wa, tp->gx, tp->glch, tp->G);
                    MLD_LAUNCHED("kw_var_bwd");
                }
            }
        }
        if (parts > 0) {
            kw_reduce_dw<<<T, kReduceThreads, 0, s2>>>(tp->gwp, parts, tp->n_types, tp->dw);
            MLD_LAUNCHED("kw_reduce_dw");
        } else {
            MLD_CUDA(cudaMemsetAsync(tp->dw, 0, sizeof(float) * T * tp->n_types, s2));
        }
        return MLD_OK;
    };
    int sg = run_graph(d, &tp->bwd_exec, st, segments);
    if (sg != MLD_OK) return sg;
    MLD_CUDA(cudaMemcpyAsync(dw, tp->dw, sizeof(float) * T * tp->n_types, cudaMemcpyDeviceToDevice, st));
    if (h.n_vn > 0) {
        kw_deinterleave<W><<<dim3((h.n_vn + 31) / 32, slabs), kBlock, 0, st>>>(
            tp->glch, tp->glch1, d->lch, d->lch1, d->g->unit, h.n_vn, h.n_core, h.n_deg1, tp->batch, d->lmax, dllr);
        MLD_LAUNCHED("kw_deinterleave");
    }
    return MLD_OK;
}

template <typename T>
int talloc(T **p, size_t n) { return dalloc(p, n); }

// A decoder keeps the buffers of its last destroyed tape and hands them to
// the next forward of the same shape, so a training loop allocates (and
// frees, which waits for the device) once instead of every step.
mld_tape *take_spare(mld_decoder *d, int32_t slabs, int32_t T, int32_t k, int32_t n_types) {
    mld_tape *tp = d->tape_spare;
    if (!tp) return nullptr;
    d->tape_spare = nullptr;
    if (tp->slabs == slabs && tp->T == T && tp->k == k && tp->n_types == n_types) return tp;
    tape_free(tp);
    return nullptr;
}

}  // namespace

namespace mld {
// Decoder teardown: frees the spare tape and detaches a tape still alive (it
// frees its own buffers when destroyed).
void tape_release(mld_decoder *d) {
    if (d->tape_spare) tape_free(d->tape_spare);
    d->tape_spare = nullptr;
    if (d->tape_live) d->tape_live->d = nullptr;
    d->tape_live = nullptr;
}
}  // namespace mld

extern "C" {

int mld_wbp_forward(mld_decoder *d, const float *llr, const uint8_t *syndrome, int32_t batch, const float *w,
                    int32_t n_types, int32_t T, int32_t ckpt_k, float *soft_out, mld_tape **tape, void *stream) {
    mld::clear_error();
    if (!d) return mld::fail(MLD_EINVAL, "wbp_forward: null decoder");
    if (d->msg != MLD_MSG_F32) return mld::fail(MLD_EINVAL, "wbp_forward: the decoder must store float messages");
    if (batch < 1 || batch > d->max_batch) return mld::fail(MLD_EINVAL, "wbp_forward: batch out of range");
    if (T < 1 || ckpt_k < 1) return mld::fail(MLD_EINVAL, "wbp_forward: T and ckpt_k must be >= 1");
    if (n_types < 1 || n_types > MLD_MAX_EDGE_TYPES) return mld::fail(MLD_EINVAL, "wbp_forward: n_types");
    const mld::HostGraph &h = d->g->h;
    if (h.max_check_deg > kMaxTerms)
        return mld::fail(MLD_EINVAL, "wbp_forward: check degree above " + std::to_string(kMaxTerms));
    for (uint8_t ty : h.etype_core)
        if (ty >= n_types) return mld::fail(MLD_EINVAL, "wbp_forward: an edge type is >= n_types");
    for (uint8_t ty : h.etype_deg1)
        if (ty >= n_types) return mld::fail(MLD_EINVAL, "wbp_forward: an edge type is >= n_types");
    if ((h.n_vn > 0 && (!llr || !soft_out)) || (h.n_cn > 0 && !syndrome) || !w)
        return mld::fail(MLD_EINVAL, "wbp_forward: null data pointer");
    int s = check_device(d->device);
    if (s != MLD_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int W = d->W;
    const int slabs = (batch + W - 1) / W;
    mld_tape *tp = nullptr;
    const float *wdev = w;
    if (tape) {
        tp = take_spare(d, slabs, T, std::min(ckpt_k, T), n_types);
        if (tp) {
            tp->batch = batch;
            cudaError_t e = cudaMemcpyAsync(tp->w, w, sizeof(float) * T * n_types, cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) {
                tape_free(tp);
                return cuda_fail(e, "wbp_forward: copy weights");
            }
        }
    }
    if (tape && !tp) {
        tp = new (std::nothrow) mld_tape();
        if (!tp) return mld::fail(MLD_ENOMEM, "wbp_forward: host allocation");
        tp->d = d;
        tp->batch = batch;
        tp->T = T;
        tp->k = std::min(ckpt_k, T);
        tp->n_types = n_types;
        tp->slabs = slabs;
        const size_t rsz = static_cast<size_t>(slabs) * h.e_core * W;
        const size_t lsz = static_cast<size_t>(slabs) * h.n_core * W;
        const size_t dsz = static_cast<size_t>(slabs) * h.n_deg1 * W;
        s = talloc(&tp->w, static_cast<size_t>(T) * n_types);
        if (s == MLD_OK) s = talloc(&tp->dw, static_cast<size_t>(T) * n_types);
        for (int c = tp->k; s == MLD_OK && c < T; c += tp->k) {
            float *p = nullptr;
            s = talloc(&p, rsz);
            tp->ckpt.push_back(p);
        }
        if (s == MLD_OK) s = talloc(&tp->seg_r, rsz * (tp->k - 1));
        if (s == MLD_OK) s = talloc(&tp->seg_lv, lsz * tp->k);
        if (s == MLD_OK) s = talloc(&tp->G, lsz);
        if (s == MLD_OK) s = talloc(&tp->gx, rsz);
        if (s == MLD_OK) s = talloc(&tp->glch, lsz);
        if (s == MLD_OK) s = talloc(&tp->glch1, dsz);
        if (s == MLD_OK) s = talloc(&tp->gd1, dsz);
        tp->gwp_blocks = 0;
        for (const mld::ClassLaunch &cl : d->g->launches[W == 8 ? 0 : (W == 16 ? 1 : (W == 32 ? 2 : 3))])
            tp->gwp_blocks += cl.blocks * slabs;
        if (s == MLD_OK) s = talloc(&tp->gwp, static_cast<size_t>(std::max(1, tp->gwp_blocks)) * T * n_types);
        if (s == MLD_OK) {
            cudaError_t e = cudaMemcpyAsync(tp->w, w, sizeof(float) * T * n_types, cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) s = cuda_fail(e, "wbp_forward: copy weights");
        }
        if (s != MLD_OK) {
            tape_free(tp);
            return s;
        }
    }
    if (tp) wdev = tp->w;
    switch (W) {
        case 8: s = wbp_forward_w<8>(d, llr, syndrome, batch, T, tp, wdev, n_types, soft_out, st); break;
        case 16: s = wbp_forward_w<16>(d, llr, syndrome, batch, T, tp, wdev, n_types, soft_out, st); break;
        case 32: s = wbp_forward_w<32>(d, llr, syndrome, batch, T, tp, wdev, n_types, soft_out, st); break;
        default: s = wbp_forward_w<64>(d, llr, syndrome, batch, T, tp, wdev, n_types, soft_out, st); break;
    }
    if (s != MLD_OK) {
        tape_free(tp);
        return s;
    }
    if (tape) {
        *tape = tp;
        d->tape_live = tp;
    }
    return MLD_OK;
}

int mld_wbp_backward(mld_tape *tp, const float *dsoft, float *dw, float *dllr, void *stream) {
    mld::clear_error();
    if (!tp || !dsoft || !dw || !dllr) return mld::fail(MLD_EINVAL, "wbp_backward: null pointer");
    int s = check_device(tp->d->device);
    if (s != MLD_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    switch (tp->d->W) {
        case 8: return wbp_backward_w<8>(tp, dsoft, dw, dllr, st);
        case 16: return wbp_backward_w<16>(tp, dsoft, dw, dllr, st);
        case 32: return wbp_backward_w<32>(tp, dsoft, dw, dllr, st);
        default: return wbp_backward_w<64>(tp, dsoft, dw, dllr, st);
    }
}

int mld_tape_destroy(mld_tape *tp) {
    if (!tp) return MLD_OK;
    mld_decoder *d = tp->d;
    if (d && d->tape_live == tp) d->tape_live = nullptr;
    if (d && !d->tape_spare) {
        d->tape_spare = tp;  // buffers kept for the next forward of this shape
        return MLD_OK;
    }
    tape_free(tp);
    return MLD_OK;
}

}  // extern "C"
