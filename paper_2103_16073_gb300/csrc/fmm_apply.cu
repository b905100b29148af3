// FMM matrix-vector product (Sec. 3.3): P2M -> M2M -> M2L -> L2L -> L2P,
// plus the stored near field.  Templated on the arithmetic type R (double
// for the plain FP64 path, float for the mixed path); input and output
// vectors are complex128 in the caller's element order.
//
// Translations use the stacked form: all box pairs of one level that share a
// translation vector share one p^2 x p^2 matrix, so each (level, offset)
// group is one complex GEMM  Y = T X  with X gathered from the source boxes
// and Y scatter-added into the target boxes.
#include <algorithm>
#include <mutex>
#include <string>

#include "common.cuh"

// ------------------------------------------------------ gather-GEMM-scatter
// Tile: 64 output rows x 32 column pairs, K chunks of 16; 256 threads, each
// 4 rows x 2 columns.  dst[dst_idx] += T * src[src_idx] (atomic adds: the
// groups of one launch may share targets).
template <class R>
__global__ void __launch_bounds__(256) k_trans(const TransTask* __restrict__ tasks,
                                               const TransTile* __restrict__ tiles,
                                               const cx<R>* __restrict__ Tbuf,
                                               const int32_t* __restrict__ src_idx,
                                               const int32_t* __restrict__ dst_idx,
                                               const cx<R>* __restrict__ src, cx<R>* __restrict__ dst) {
    constexpr int BM = 64, BN = 32, BK = 16;
    __shared__ cx<R> Ts[BK][BM];
    __shared__ cx<R> Xs[BK][BN];
    __shared__ int s_src[BN];
    __shared__ int s_dst[BN];
    TransTile tl = tiles[blockIdx.x];
    TransTask tk = tasks[tl.task];
    int tid = threadIdx.x;
    int ty = tid >> 4, tx = tid & 15;
    if (tid < BN) {
        int c = tl.col0 + tid;
        s_src[tid] = c < tk.npairs ? src_idx[tk.pair_off + c] : -1;
        s_dst[tid] = c < tk.npairs ? dst_idx[tk.pair_off + c] : -1;
    }
    __syncthreads();
    const cx<R>* T = Tbuf + tk.t_off;
    cx<R> acc[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j] = mk<R>(0, 0);
    for (int k0 = 0; k0 < tk.cols; k0 += BK) {
#pragma unroll
        for (int it = 0; it < (BM * BK) / 256; ++it) {
            int idx = tid + it * 256;
            int r = idx / BK, kk = idx % BK;
            int row = tl.row0 + r, k = k0 + kk;
            Ts[kk][r] = (row < tk.rows && k < tk.cols) ? T[(int64_t)row * tk.cols + k] : mk<R>(0, 0);
        }
#pragma unroll
        for (int it = 0; it < (BN * BK) / 256; ++it) {
            int idx = tid + it * 256;
            int c = idx / BK, kk = idx % BK;
            int k = k0 + kk;
            int sb = s_src[c];
            Xs[kk][c] = (sb >= 0 && k < tk.cols) ? src[tk.src_base + (int64_t)sb * tk.cols + k] : mk<R>(0, 0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            cx<R> a[4], b[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = Ts[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 2; ++j) b[j] = Xs[kk][tx * 2 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) cmac(acc[i][j], a[i], b[j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        int c = tx * 2 + j;
        int db = s_dst[c];
        if (db < 0) continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int row = tl.row0 + ty * 4 + i;
            if (row >= tk.rows) continue;
            cx<R>* d = dst + tk.dst_base + (int64_t)db * tk.rows + row;
            atomicAdd(&d->re, acc[i][j].re);
            atomicAdd(&d->im, acc[i][j].im);
        }
    }
}

// ----------------------------------------------------------------- P2M ----
// mp[leaf][r] = sum_{pos in leaf} W[pos][r] x[perm[pos]]
// (blockIdx.y = right-hand side: x and mp advance by xstride / mstride)
template <class R>
__global__ void k_p2m(int P, const int32_t* __restrict__ leaf_start, const int32_t* __restrict__ perm,
                      const cx<R>* __restrict__ W, const cd* __restrict__ x, cx<R>* __restrict__ mp,
                      int64_t xstride, int64_t mstride) {
    x += blockIdx.y * xstride;
    mp += blockIdx.y * mstride;
    int b = blockIdx.x;
    int s0 = leaf_start[b], s1 = leaf_start[b + 1];
    __shared__ cx<R> xs[256];
    for (int r0 = 0; r0 < P; r0 += blockDim.x) {
        int r = r0 + threadIdx.x;
        cx<R> acc = mk<R>(0, 0);
        for (int c0 = s0; c0 < s1; c0 += 256) {
            int cn = min(256, s1 - c0);
            __syncthreads();
            for (int i = threadIdx.x; i < cn; i += blockDim.x) xs[i] = from_d<R>(x[perm[c0 + i]]);
            __syncthreads();
            if (r < P)
                for (int i = 0; i < cn; ++i) cmac(acc, W[(int64_t)(c0 + i) * P + r], xs[i]);
        }
        if (r < P) mp[(int64_t)b * P + r] = acc;
    }
}

// ----------------------------------------------------- near field + L2P ----
// y[perm[pos]] = sum_c A_t[row][c] x[col c] + sum_r V[pos][r] loc[leaf][r]
// for up to NB right-hand sides per CTA (blockIdx.y selects the chunk): each
// near-field and L2P entry is read once and applied to every right-hand side
// of the chunk.  x, y advance by xstride per rhs, loc by lstride.
// A near-field entry as stored: complex FP32 / FP64, or a BF16 pair (real
// part in the low, imaginary part in the high 16 bits; BF16 is the upper
// half of an FP32 word).
__device__ __forceinline__ cf nf_entry(const cf& a) { return a; }
__device__ __forceinline__ cd nf_entry(const cd& a) { return a; }
__device__ __forceinline__ cf nf_entry(uint32_t a) {
    return mk(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u));
}

template <class R, int NB, class AS = cx<R>>
__global__ void k_near_l2p(int P, const int32_t* __restrict__ leaf_start, const int32_t* __restrict__ perm,
                           const int32_t* __restrict__ ucnt, const int32_t* __restrict__ ulist,
                           const int64_t* __restrict__ nf_off, const int32_t* __restrict__ nf_ncol,
                           const AS* __restrict__ A, const cx<R>* __restrict__ V,
                           const cx<R>* __restrict__ loc, const cd* __restrict__ x, cd* __restrict__ y,
                           int nrhs, int64_t xstride, int64_t lstride) {
    extern __shared__ unsigned char smem_raw[];
    const int r0 = blockIdx.y * NB;
    const int nr = min(NB, nrhs - r0);
    cx<R>* xs = (cx<R>*)smem_raw;       // [nr][K]
    int t = blockIdx.x;
    int K = nf_ncol[t];
    cx<R>* ls = xs + nr * K;            // [nr][P]
    // gather the x values of the U-list leaves in column order
    int nu = ucnt[t];
    int c = 0;
    for (int i = 0; i < nu; ++i) {
        int s = ulist[(int64_t)t * FB_ULIST + i];
        int a0 = leaf_start[s], a1 = leaf_start[s + 1];
        for (int q = threadIdx.x; q < a1 - a0; q += blockDim.x) {
            int e = perm[a0 + q];
            for (int j = 0; j < nr; ++j) xs[j * K + c + q] = from_d<R>(x[(r0 + j) * xstride + e]);
        }
        c += a1 - a0;
    }
    if (loc)
        for (int j = 0; j < nr; ++j)
            for (int q = threadIdx.x; q < P; q += blockDim.x)
                ls[j * P + q] = loc[(r0 + j) * lstride + (int64_t)t * P + q];
    __syncthreads();
    int rb = leaf_start[t], nrow = leaf_start[t + 1] - rb;
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const AS* At = A + nf_off[t];
    for (int r = warp; r < nrow; r += nw) {
        cx<R> acc[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j) acc[j] = mk<R>(0, 0);
        const AS* row = At + (int64_t)r * K;
        // unrolled: several independent row loads in flight per lane
#pragma unroll 4
        for (int q = lane; q < K; q += 32) {
            const cx<R> a = nf_entry(row[q]);
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (j < nr) cmac(acc[j], a, xs[j * K + q]);
        }
        if (loc) {
            const cx<R>* vr = V + (int64_t)(rb + r) * P;
            for (int q = lane; q < P; q += 32) {
                cx<R> v = vr[q];
#pragma unroll
                for (int j = 0; j < NB; ++j)
                    if (j < nr) cmac(acc[j], v, ls[j * P + q]);
            }
        }
#pragma unroll
        for (int j = 0; j < NB; ++j) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc[j].re += __shfl_xor_sync(0xffffffffu, acc[j].re, o);
                acc[j].im += __shfl_xor_sync(0xffffffffu, acc[j].im, o);
            }
        }
        if (lane == 0) {
            int e = perm[rb + r];
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (j < nr) y[(r0 + j) * xstride + e] = mk<double>((double)acc[j].re, (double)acc[j].im);
        }
    }
}


// Data of an operator for the staged RCR passes: phase tables, staging
// buffers, folded rotation tables.
template <class R>
struct RotArgs {
    const cx<R>* ph;
    int prot;
    cx<R>* U;   // staging buffers of the large-order passes
    cx<R>* V;
    const void* rf;   // folded rotation tables and their per-group stride
    int64_t fper;
    StcTabs tc;       // tables of the tensor-core staged passes (single precision)
    DfTabs dft;       // tables of the double-FP32 staged passes (FP64 operators)
};
template <class R>
static RotArgs<R> rot_args(const fb_op* op) {
    RotArgs<R> a;
    a.ph = (const cx<R>*)(sizeof(R) == 8 ? (const void*)op->rph64 : (const void*)op->rph32);
    a.prot = op->Prot;
    a.U = (cx<R>*)op->stg_u;
    a.V = (cx<R>*)op->stg_v;
    a.rf = op->rotf;
    a.fper = op->rotf_per;
    a.tc = StcTabs{op->stc_tab, op->stc_per, op->stc_err};
    a.dft = DfTabs{op->rotf_df, op->coax_df};
    return a;
}
static fb_status stg_run(void* plan, const RotArgs<float>& r, const cf* coax, const cf* src, cf* dst,
                         cudaStream_t s, int nrhs, int64_t rstride) {
    return fb_stg_run_f(plan, (const float*)r.rf, r.fper, r.ph, r.prot, coax, src, dst, r.U, r.V, s, nrhs, rstride,
                        r.tc);
}
static fb_status stg_run(void* plan, const RotArgs<double>& r, const cd* coax, const cd* src, cd* dst,
                         cudaStream_t s, int nrhs, int64_t rstride) {
    return fb_stg_run_d(plan, (const double*)r.rf, r.fper, r.ph, r.prot, coax, src, dst, r.U, r.V, s, nrhs, rstride,
                        r.dft);
}

// Device time (ms, median of 3 after one untimed run, one right-hand side)
// of each pass of every staged M2L level of an operator, on its expansion
// buffers: ms[4 l + {0..3}] = pre-pass, rotation, coaxial, back-rotation of
// level l (-1: not staged); form[l] = 1 CUDA cores, 2 rotations on the
// tensor cores, 3 double-FP32 arithmetic, 5 rotations and coaxial step on
// the tensor cores (0: not staged).
fb_status fb_stg_op_pass_times(fb_op* op, cudaStream_t s, double* ms, int* tc) {
    for (int i = 0; i < 4 * (FB_MAXLEV + 1); ++i) ms[i] = -1.0;
    for (int l = 0; l <= FB_MAXLEV; ++l) tc[l] = 0;
    const bool mixed = op->prec == FB_PREC_MIXED_FMM;
    RcrPlan& pl = (mixed && op->method == FB_TRANS_AUTO && op->tc_plan) ? op->m2l_rcr_rest : op->m2l_rcr;
    if (!pl.stg || !op->mp || !op->loc) return FB_OK;
    cudaEvent_t e0, e1;
    FB_CUDA(cudaEventCreate(&e0));
    FB_CUDA(cudaEventCreate(&e1));
    fb_status st = FB_OK;
    for (int li = 0; li < fb_stg_level_count(pl.stg) && st == FB_OK; ++li) {
        int64_t sb = 0, db = 0;
        int t = 0;
        fb_stg_level_info(pl.stg, li, &sb, &db, &t);
        int lev = -1;
        for (int l = 2; l <= op->L; ++l)
            if (op->lev_off[l] == sb) lev = l;
        if (lev < 0 || sb != db) continue;
        tc[lev] = t;
        for (int pass = 0; pass < 4 && st == FB_OK; ++pass) {
            if (pass == 0 && (t == 2 || t == 5)) continue;   // the tensor-core rotation pass folds its inputs
            auto run = [&]() {
                return mixed ? fb_stg_run_f(pl.stg, (const float*)op->rotf, op->rotf_per, (const cf*)op->rph32,
                                            op->Prot, op->coax32, (const cf*)op->mp, (cf*)op->loc, (cf*)op->stg_u,
                                            (cf*)op->stg_v, s, 1, 0, rot_args<float>(op).tc, li, 1 << pass)
                             : fb_stg_run_d(pl.stg, (const double*)op->rotf, op->rotf_per, (const cd*)op->rph64,
                                            op->Prot, op->coax64, (const cd*)op->mp, (cd*)op->loc, (cd*)op->stg_u,
                                            (cd*)op->stg_v, s, 1, 0, rot_args<double>(op).dft, li, 1 << pass);
            };
            std::vector<float> v;
            st = run();
            for (int r = 0; r < 3 && st == FB_OK; ++r) {
                cudaEventRecord(e0, s);
                st = run();
                cudaEventRecord(e1, s);
                if (cudaEventSynchronize(e1) != cudaSuccess) st = fb_fail(FB_ERR_CUDA, "staged pass timing failed");
                float x = 0.f;
                cudaEventElapsedTime(&x, e0, e1);
                v.push_back(x);
            }
            if (st == FB_OK) {
                std::sort(v.begin(), v.end());
                ms[4 * lev + pass] = v[1];
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

// The tiles of a plan in the operator's precision (FP64: also those in double-FP32).
static fb_status rcr_tiles_run(const fb_op* op, RcrPlan& pl, const cf* src, cf* dst, cudaStream_t s, int nrhs,
                               int64_t rstride) {
    return fb_rcr_tiles_run_f(op, pl, src, dst, s, nrhs, rstride);
}
static fb_status rcr_tiles_run(const fb_op* op, RcrPlan& pl, const cd* src, cd* dst, cudaStream_t s, int nrhs,
                               int64_t rstride) {
    return fb_rcr_tiles_run_d(op, pl, src, dst, s, nrhs, rstride);
}

template <class R>
static fb_status run_rcr(const fb_op* op, RcrPlan& pl, const RotArgs<R>& rot, const cx<R>* coax, const cx<R>* src,
                         cx<R>* dst, cudaStream_t s, int nrhs = 1, int64_t rstride = 0) {
    FB_CHECK(rcr_tiles_run(op, pl, src, dst, s, nrhs, rstride));
    if (pl.stg) FB_CHECK(stg_run(pl.stg, rot, coax, src, dst, s, nrhs, rstride));
    return FB_OK;
}

// Uploads an RCR plan: per-pair tiles for the tasks of moderate order and the
// staged passes of the large-order ones, whose staging buffers (shared by
// every plan of the operator: the passes of one matvec run one after the
// other) grow to the largest level's need.
fb_status fb_rcr_upload(fb_op* op, RcrPlan& pl, const int32_t* src, const int32_t* dst, size_t csize) {
    pl.src_idx = src;
    pl.dst_idx = dst;
    pl.csize = csize;
    for (const RcrTask& tk : pl.h_tasks) {
        if ((tk.staged == 2 || tk.staged == 5) && op->prec != FB_PREC_MIXED_FMM)
            return fb_fail(FB_ERR_ARG, "tensor-core staged RCR applies to mixed operators");
        if ((tk.staged == 3 || tk.staged == 4) && op->prec != FB_PREC_FP64_FMM)
            return fb_fail(FB_ERR_ARG, "double-FP32 RCR applies to FP64 operators");
    }
    // a pair whose working set does not fit one CTA can only run staged
    for (RcrTask& tk : pl.h_tasks)
        if ((tk.staged == 0 || tk.staged == 4) && !fb_rcr_tile_fits(tk.p_in, tk.p_out, csize))
            tk.staged = tk.staged == 4 ? 3 : 1;
    if (pl.h_tasks.empty()) return FB_OK;
    FB_CHECK(fb_rcr_tiles_build(op, pl, false));
    FB_CHECK(fb_rcr_tiles_build(op, pl, true));
    FB_CHECK(fb_stg_build(pl, op->theta_slot, op->per_dir, op->coax64, &pl.stg, &pl.stg_elems));
    if (fb_stg_uses_tc(pl.stg)) FB_CHECK(fb_stc_tables(op, cudaStreamLegacy));
    if (fb_stg_uses_df(pl.stg)) FB_CHECK(fb_stg_df_tables(op, cudaStreamLegacy));
    if (pl.stg_elems > op->stg_elems) {
        FB_CUDA(cudaDeviceSynchronize());
        dfree(op->stg_u);
        dfree(op->stg_v);
        op->stg_elems = 0;
        FB_CHECK(dalloc((unsigned char**)&op->stg_u, (size_t)pl.stg_elems * csize));
        FB_CHECK(dalloc((unsigned char**)&op->stg_v, (size_t)pl.stg_elems * csize));
        op->stg_elems = pl.stg_elems;
        op->buf_gen++;   // captured graphs refer to the old buffers
    }
    return FB_OK;
}

template <class R>
static fb_status run_plan(const TransPlan& pl, const cx<R>* T, const cx<R>* src, cx<R>* dst, cudaStream_t s) {
    if (pl.ntiles == 0) return FB_OK;
    k_trans<R><<<pl.ntiles, 256, 0, s>>>(pl.tasks, pl.tiles, T, pl.src_idx, pl.dst_idx, src, dst);
    FB_LAUNCH_CHECK();
    fb_count_launch();
    return FB_OK;
}

// One FMM matvec for nrhs right-hand sides (x, y: nrhs x N, rhs-major).  The
// expansions of rhs r sit at mp / loc + r * cnt; every kernel handles all
// right-hand sides in one launch, so the near-field entries, the P2M / L2P
// operators and every translation operator are read once per matvec.
template <class R>
static fb_status fmm_apply_t(fb_op* op, const cd* x, cd* y, cudaStream_t s, const cx<R>* A,
                             const cx<R>* W, const cx<R>* V, const cx<R>* T, PhaseTimer* pt,
                             void* scratch = nullptr, int nrhs = 1) {
    auto mark = [&](int i) { if (pt) cudaEventRecord(pt->ev[i], s); };
    const fb_tree* t = op->tree;
    int L = op->L;
    int pL = op->p[L], PL = pL * pL;
    int64_t cnt = op->lev_off[L + 1];
    const int64_t n = op->n;
    const bool composed = op->method == FB_TRANS_COMPOSED;
    if (composed && nrhs > 1) {   // the composed SIMT path takes one right-hand side at a time
        for (int r = 0; r < nrhs; ++r)
            FB_CHECK(fmm_apply_t<R>(op, x + r * n, y + r * n, s, A, W, V, T, r == 0 ? pt : nullptr, scratch, 1));
        return FB_OK;
    }
    // expansions: the operator's own buffers (grown to nrhs sets), or a
    // caller-provided region holding the multipoles followed by the locals
    if (!scratch && nrhs > op->exp_nrhs) {
        cudaStreamSynchronize(s);
        dfree(op->mp);
        dfree(op->loc);
        op->mp = nullptr;
        op->loc = nullptr;
        FB_CHECK(dalloc((cx<R>**)&op->mp, cnt * nrhs));
        FB_CHECK(dalloc((cx<R>**)&op->loc, cnt * nrhs));
        op->exp_nrhs = nrhs;
        op->buf_gen++;   // captured graphs of this operator refer to the old buffers
    }
    cx<R>* mp = scratch ? (cx<R>*)scratch : (cx<R>*)op->mp;
    cx<R>* loc = scratch ? (cx<R>*)scratch + cnt * nrhs : (cx<R>*)op->loc;
    mark(0);
    FB_CUDA(cudaMemsetAsync(mp, 0, sizeof(cx<R>) * cnt * nrhs, s));
    FB_CUDA(cudaMemsetAsync(loc, 0, sizeof(cx<R>) * cnt * nrhs, s));
    int nleaf = t->nbox[L];
    k_p2m<R><<<dim3(nleaf, nrhs), 128, 0, s>>>(PL, t->leaf_start, t->perm, W, x, mp + op->lev_off[L], n, cnt);
    FB_LAUNCH_CHECK();
    fb_count_launch();
    mark(1);
    const RotArgs<R> rot = rot_args<R>(op);
    const cx<R>* coax = (const cx<R>*)(sizeof(R) == 8 ? (const void*)op->coax64 : (const void*)op->coax32);
    const bool auto_tc = sizeof(R) == 4 && op->method == FB_TRANS_AUTO;
    for (int l = L; l >= 3; --l) {
        if (composed) FB_CHECK(run_plan<R>(op->m2m[l], T, mp, mp, s));
        else if (auto_tc && op->tc_m2m[l])
            FB_CHECK(fb_tc_run(op, op->tc_m2m[l], (const cf*)mp, (cf*)mp, s, nrhs, cnt));
        else FB_CHECK(run_rcr<R>(op, op->m2m_rcr[l], rot, coax, mp, mp, s, nrhs, cnt));
    }
    mark(2);
    // phase [2] is the tensor-core part of M2L: empty unless it runs below
    const bool tc_split = sizeof(R) == 4 && op->method == FB_TRANS_AUTO && op->tc_plan != nullptr;
    if (!tc_split) mark(3);
    if (composed) {
        FB_CHECK(run_plan<R>(op->m2l, T, mp, loc, s));
    } else if (op->method == FB_TRANS_RCR) {
        FB_CHECK(run_rcr<R>(op, op->m2l_rcr, rot, coax, mp, loc, s, nrhs, cnt));
    } else {
        if constexpr (sizeof(R) == 4) {
            if (op->method == FB_TRANS_TENSOR) {
                FB_CHECK(fb_tc_run(op, op->tc_plan_all, (const cf*)mp, (cf*)loc, s, nrhs, cnt));
            } else if (op->tc_plan) {
                FB_CHECK(fb_tc_run(op, op->tc_plan, (const cf*)mp, (cf*)loc, s, nrhs, cnt));
                mark(3);
                FB_CHECK(run_rcr<R>(op, op->m2l_rcr_rest, rot, coax, mp, loc, s, nrhs, cnt));
            } else {
                FB_CHECK(run_rcr<R>(op, op->m2l_rcr, rot, coax, mp, loc, s, nrhs, cnt));
            }
        } else {
            FB_CHECK(run_rcr<R>(op, op->m2l_rcr, rot, coax, mp, loc, s, nrhs, cnt));
        }
    }
    mark(4);
    for (int l = 3; l <= L; ++l) {
        if (composed) FB_CHECK(run_plan<R>(op->l2l[l], T, loc, loc, s));
        else if (auto_tc && op->tc_l2l[l])
            FB_CHECK(fb_tc_run(op, op->tc_l2l[l], (const cf*)loc, (cf*)loc, s, nrhs, cnt));
        else FB_CHECK(run_rcr<R>(op, op->l2l_rcr[l], rot, coax, loc, loc, s, nrhs, cnt));
    }
    mark(5);
    int maxK = 0;
    for (int v : op->h_nf_ncol) maxK = std::max(maxK, v);
    const cx<R>* locL = loc + op->lev_off[L];
    if (nrhs == 1) {
        size_t smem = sizeof(cx<R>) * (maxK + PL);
        bool done16 = false;
        if constexpr (sizeof(R) == 4) {
            if (op->near16 && op->nf16) {   // 16-bit near-field entries
                FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, 1, uint32_t>, smem));
                k_near_l2p<R, 1, uint32_t><<<nleaf, 256, smem, s>>>(PL, t->leaf_start, t->perm, t->ucnt,
                                                                    t->ulist, op->nf_off, op->nf_ncol, op->nf16, V,
                                                                    locL, x, y, 1, n, cnt);
                done16 = true;
            }
        }
        if (!done16) {
            FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, 1>, smem));
            k_near_l2p<R, 1><<<nleaf, 256, smem, s>>>(PL, t->leaf_start, t->perm, t->ucnt, t->ulist, op->nf_off,
                                                      op->nf_ncol, A, V, locL, x, y, 1, n, cnt);
        }
    } else {
        constexpr int NB = 4;
        int nr = std::min(nrhs, NB);
        size_t smem = sizeof(cx<R>) * (size_t)nr * (maxK + PL);
        if (smem > 227 * 1024) return fb_fail(FB_ERR_ARG, "near-field tile exceeds shared memory");
        bool done16 = false;
        if constexpr (sizeof(R) == 4) {
            if (op->near16 && op->nf16) {
                FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, NB, uint32_t>, smem));
                k_near_l2p<R, NB, uint32_t><<<dim3(nleaf, div_up(nrhs, NB)), 256, smem, s>>>(
                    PL, t->leaf_start, t->perm, t->ucnt, t->ulist, op->nf_off, op->nf_ncol, op->nf16, V, locL, x,
                    y, nrhs, n, cnt);
                done16 = true;
            }
        }
        if (!done16) {
            FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, NB>, smem));
            k_near_l2p<R, NB><<<dim3(nleaf, div_up(nrhs, NB)), 256, smem, s>>>(
                PL, t->leaf_start, t->perm, t->ucnt, t->ulist, op->nf_off, op->nf_ncol, A, V, locL, x, y, nrhs, n,
                cnt);
        }
    }
    FB_LAUNCH_CHECK();
    fb_count_launch();
    mark(6);
    return FB_OK;
}

// FP32 -> BF16 with round to nearest even (finite values)
__device__ __forceinline__ uint32_t bf16_bits(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
}
static __global__ void k_cf_to_bf16(const cf* __restrict__ in, int64_t n, uint32_t* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = bf16_bits(in[i].re) | (bf16_bits(in[i].im) << 16);
}

// Near-field entries of a mixed operator in BF16 (8-bit significand,
// relative rounding 2^-9 per entry) for low-accuracy operators, whose
// matvec then reads half the near-field bytes; enable = 0 returns to FP32.
fb_status fb_near_bf16(fb_op* op, int enable, cudaStream_t s) {
    if (op->prec != FB_PREC_MIXED_FMM || !op->nf32)
        return fb_fail(FB_ERR_ARG, "BF16 near field applies to mixed FMM operators");
    if (enable && !op->nf16) {
        FB_CHECK(dalloc(&op->nf16, (size_t)op->nf_count));
        k_cf_to_bf16<<<(unsigned)std::min<int64_t>(div_up(op->nf_count, 256), 8192), 256, 0, s>>>(
            op->nf32, op->nf_count, op->nf16);
        FB_LAUNCH_CHECK();
        FB_CUDA(cudaStreamSynchronize(s));
        fb_count_launch();
    }
    op->near16 = enable ? 1 : 0;
    op->buf_gen++;   // captured graphs read the other entries
    return FB_OK;
}

static size_t op_csize(const fb_op* op) { return op->prec == FB_PREC_MIXED_FMM ? sizeof(cf) : sizeof(cd); }

// Level whose RCR flag governs a task: M2L tasks read and write one level;
// M2M / L2L tasks are governed by their finer (child) level, whose
// expansions lie after the parent's in the level arrays.  Levels 0 and 1
// hold no expansions (their offsets equal level 2's), so the search starts
// at level 2.
static int task_level(const fb_op* op, const RcrTask& tk, bool* m2l) {
    *m2l = tk.src_base == tk.dst_base;
    const int64_t b = std::max(tk.src_base, tk.dst_base);
    for (int l = 2; l <= op->L; ++l)
        if (op->lev_off[l] == b) return l;
    return 2;
}

fb_status fb_rcr_restage(fb_op* op, const int* m2l, const int* pair) {
    const size_t csz = op_csize(op);
    for (int l = 2; l <= op->L; ++l) {
        // 1: staged on CUDA cores, 2: staged with the rotations on the tensor cores
        op->stg_m2l[l] = m2l[l] ? m2l[l] : (!fb_rcr_tile_fits(op->p[l], op->p[l], csz) ? 1 : 0);
        if (l >= 3) {
            const int pm = std::max(op->p[l], op->p[l - 1]);
            op->stg_pair[l] = pair[l] ? pair[l] : (!fb_rcr_tile_fits(pm, pm, csz) ? 1 : 0);
        }
    }
    FB_CUDA(cudaDeviceSynchronize());
    op->buf_gen++;   // captured graphs refer to the plans rebuilt here
    auto redo = [&](RcrPlan& pl) -> fb_status {
        if (pl.h_tasks.empty()) return FB_OK;
        bool changed = false;
        for (RcrTask& tk : pl.h_tasks) {
            bool is_m2l = false;
            const int l = task_level(op, tk, &is_m2l);
            const int want = is_m2l ? op->stg_m2l[l] : op->stg_pair[l];
            changed = changed || tk.staged != want;
            tk.staged = want;
        }
        if (!changed) return FB_OK;
        const int32_t* si = pl.src_idx;
        const int32_t* di = pl.dst_idx;
        fb_rcr_free(pl);
        return fb_rcr_upload(op, pl, si, di, csz);
    };
    FB_CHECK(redo(op->m2l_rcr));
    FB_CHECK(redo(op->m2l_rcr_rest));
    for (int l = 3; l <= op->L; ++l) {
        FB_CHECK(redo(op->m2m_rcr[l]));
        FB_CHECK(redo(op->l2l_rcr[l]));
    }
    return FB_OK;
}

// One RCR plan on the operator's expansion buffers (precision of the op).
fb_status fb_rcr_run_op(fb_op* op, RcrPlan& pl, void* src, void* dst, cudaStream_t s, int nrhs, int64_t rstride) {
    if (op->prec == FB_PREC_MIXED_FMM)
        return run_rcr<float>(op, pl, rot_args<float>(op), op->coax32, (const cf*)src, (cf*)dst, s, nrhs, rstride);
    return run_rcr<double>(op, pl, rot_args<double>(op), op->coax64, (const cd*)src, (cd*)dst, s, nrhs, rstride);
}

fb_status fb_fmm_apply(fb_op* op, const cd* x, cd* y, cudaStream_t s, PhaseTimer* pt, int nrhs) {
    if (op->prec == FB_PREC_MIXED_FMM)
        return fmm_apply_t<float>(op, x, y, s, op->nf32, op->w32, op->v32, op->T32, pt, nullptr, nrhs);
    return fmm_apply_t<double>(op, x, y, s, op->nf64, op->w64, op->v64, op->T64, pt, nullptr, nrhs);
}

static void free_plan(TransPlan& p) {
    dfree(p.tasks);
    dfree(p.tiles);
}
void fb_rcr_free(RcrPlan& p) {
    fb_rcr_tiles_free(p.tiles);
    fb_rcr_tiles_free(p.df_tiles);
    fb_stg_free(p.stg);
    p.stg_elems = 0;
}
static void free_plan(RcrPlan& p) { fb_rcr_free(p); }

void fb_fmm_destroy(fb_op* op) {
    dfree(op->nf_off);
    dfree(op->nf_ncol);
    dfree(op->nf64);
    dfree(op->nf32);
    dfree(op->nf16);
    dfree(op->self64);
    dfree(op->w64);
    dfree(op->w32);
    dfree(op->v64);
    dfree(op->v32);
    dfree(op->mp);
    dfree(op->loc);
    dfree(op->T64);
    dfree(op->T32);
    free_plan(op->m2l);
    free_plan(op->m2l_rcr);
    free_plan(op->m2l_rcr_rest);
    fb_tc_free(op->tc_plan);
    fb_tc_free(op->tc_plan_all);
    for (int l = 0; l <= FB_MAXLEV; ++l) {
        fb_tc_free(op->tc_m2m[l]);
        fb_tc_free(op->tc_l2l[l]);
    }
    for (int l = 0; l <= FB_MAXLEV; ++l) {
        free_plan(op->m2m[l]);
        free_plan(op->l2l[l]);
        free_plan(op->m2m_rcr[l]);
        free_plan(op->l2l_rcr[l]);
    }
    op->rot64 = nullptr;   // owned by the tree
    op->rotd64 = nullptr;
    op->rotd32 = nullptr;
    op->rph64 = nullptr;
    op->rph32 = nullptr;
    dfree(op->coax64);
    dfree(op->coax32);
    dfree(op->stg_u);
    dfree(op->stg_v);
    op->stg_elems = 0;
    if (op->rotf) cudaFree(op->rotf);
    op->rotf = nullptr;
    dfree(op->stc_tab);
    dfree(op->stc_off);
    dfree(op->stc_err);
    dfree(op->rotf_df);
    dfree(op->coax_df);
    for (RcrTables* t : {&op->rcr_tab, &op->rcr_df}) {
        dfree(t->rot);
        dfree(t->coax);
    }
    dfree(op->rcr_lut);
}

// ---------------------------------------------------------------------------
// Matvec without allocation.  Some callers cannot allocate device memory when
// they apply an operator: real-time audio callbacks that must not block in the
// driver's allocator, or hosts whose device memory is owned by a fixed arena
// that the library may not grow.  For
// them fb_operator_apply_noalloc keeps the FMM's per-call scratch (the
// multipole and local expansions of every level) in this library-wide
// static device array instead of the operator's own buffers.  Every GPU that
// loads the library holds the array until the process exits.
static __device__ __align__(256) unsigned char fb_noalloc_scratch[FB_NOALLOC_SCRATCH_BYTES];

static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[64] = {nullptr};

// Resolves the device address of the static array for the current device
// (once per device; host code only sees a stand-in for the symbol).
static fb_status noalloc_scratch_ptr(void** out) {
    int dev = 0;
    FB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fb_fail(FB_ERR_ARG, "device ordinal out of range for the static scratch");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, fb_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return fb_fail(FB_ERR_CUDA, std::string("cudaGetSymbolAddress(fb_noalloc_scratch) failed: ") +
                                            cudaGetErrorString(e));
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return FB_OK;
}

fb_status fb_fmm_apply_noalloc(fb_op* op, const cd* x, cd* y, cudaStream_t s) {
    if (op->prec == FB_PREC_FP64_DENSE)
        return fb_fail(FB_ERR_ARG, "fb_operator_apply_noalloc needs an FMM operator (dense ones use no scratch)");
    // the static array is resolved per device: the operator's data and the
    // scratch must be on the same GPU
    int cur = -1;
    FB_CUDA(cudaGetDevice(&cur));
    if (cur != op->dev)
        return fb_fail(FB_ERR_ARG, "fb_operator_apply_noalloc: current device " + std::to_string(cur) +
                                       " differs from the operator's device " + std::to_string(op->dev));
    size_t elem = op->prec == FB_PREC_MIXED_FMM ? sizeof(cf) : sizeof(cd);
    size_t need = 2 * (size_t)op->lev_off[op->L + 1] * elem;
    if (need > (size_t)FB_NOALLOC_SCRATCH_BYTES)
        return fb_fail(FB_ERR_ARG, "operator needs " + std::to_string(need) +
                                       " bytes of expansion scratch; the static buffer holds " +
                                       std::to_string((size_t)FB_NOALLOC_SCRATCH_BYTES));
    void* p = nullptr;
    FB_CHECK(noalloc_scratch_ptr(&p));
    if (op->prec == FB_PREC_MIXED_FMM)
        return fmm_apply_t<float>(op, x, y, s, op->nf32, op->w32, op->v32, op->T32, nullptr, p);
    return fmm_apply_t<double>(op, x, y, s, op->nf64, op->w64, op->v64, op->T64, nullptr, p);
}
