// FMM matrix-vector product (Sec. 3.3): P2M -> M2M -> M2L -> L2L -> L2P,
// plus the stored near field.  Templated on the arithmetic type R (double
// for the plain FP64 path, float for the mixed path); input and output
// vectors are complex128 in the caller's element order.
//
// Translations run per level in the form chosen for it: per-pair tiles
// (rcr_tiles.cu), staged passes (rcr_staged.cu, rcr_staged_tc.cu) or composed
// matrices on the tensor cores (trans_tc.cu).  k_trans below is the composed
// form on CUDA cores (FB_TRANS_COMPOSED): all box pairs of one level that share
// a translation vector share one p^2 x p^2 matrix, so each (level, offset)
// group is one complex GEMM  Y = T X  with X gathered from the source boxes and
// Y scatter-added into the target boxes.
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
// blockIdx.x = leaf, blockIdx.y = chunk of NB right-hand sides (x and mp
// advance by xstride / mstride each), blockIdx.z = chunk of coefficients.
// Bound by reading W once for the NB right-hand sides; a leaf is a chain of
// four dependent loads, so that a thread's first LU rows of W are on their way
// before the gather of x and the next LU before the current ones are used, and
// the coefficients of a large order go to a CTA per 256.  Per product (one CTA
// of 128 threads per leaf before): L-room at 2 kHz 0.25 -> 0.20 ms (all 16
// first rows at once, without the second buffer: 0.22), 240 leaves of order 66
// 0.31 -> 0.047 ms.  FP64 is bound by its pipe (85 %).
template <class R>
constexpr int LEAF_UNROLL = sizeof(R) == 4 ? 8 : 4;

template <class R, int NB>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 6) k_p2m(int P, const int32_t* __restrict__ leaf_start,
                                             const int32_t* __restrict__ perm, const cx<R>* __restrict__ W,
                                             const cd* __restrict__ x, cx<R>* __restrict__ mp, int nrhs,
                                             int64_t xstride, int64_t mstride) {
    constexpr int LU = LEAF_UNROLL<R> / (sizeof(R) / 4), CHUNK = 256;
    __shared__ cx<R> xs[NB][CHUNK];
    const int j0 = blockIdx.y * NB, nr = min(NB, nrhs - j0);
    x += j0 * xstride;
    mp += j0 * mstride;
    const int b = blockIdx.x, r = blockIdx.z * blockDim.x + threadIdx.x;
    const int s0 = leaf_start[b], s1 = leaf_start[b + 1];
    const int rc = min(r, P - 1);   // (threads past the order read its last row and store nothing)
    cx<R> w[LU], acc[NB];
#pragma unroll
    for (int u = 0; u < LU; ++u)
        if (s0 + u < s1) w[u] = W[(int64_t)(s0 + u) * P + rc];
#pragma unroll
    for (int j = 0; j < NB; ++j) acc[j] = mk<R>(0, 0);
    for (int c0 = s0; c0 < s1; c0 += CHUNK) {
        const int cn = min(CHUNK, s1 - c0);
        if (c0 > s0) __syncthreads();
        for (int i = threadIdx.x; i < cn; i += blockDim.x) {
            const int e = perm[c0 + i];
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (j < nr) xs[j][i] = from_d<R>(x[j * xstride + e]);
        }
        __syncthreads();
        for (int i = 0; i < cn; i += LU) {
            cx<R> wn[LU];
#pragma unroll
            for (int u = 0; u < LU; ++u)
                if (c0 + i + LU + u < s1) wn[u] = W[(int64_t)(c0 + i + LU + u) * P + rc];
#pragma unroll
            for (int u = 0; u < LU; ++u)
                if (i + u < cn)
#pragma unroll
                    for (int j = 0; j < NB; ++j)
                        if (j < nr) cmac(acc[j], w[u], xs[j][i + u]);
#pragma unroll
            for (int u = 0; u < LU; ++u) w[u] = wn[u];
        }
    }
    if (r < P)
#pragma unroll
        for (int j = 0; j < NB; ++j)
            if (j < nr) mp[j * mstride + (int64_t)b * P + r] = acc[j];
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

//
// Bound by reading A and V (one warp per row).  A leaf of some 18 rows is
// mostly latency: the columns are gathered by all warps at once (offsets of
// the U-list leaves from a warp scan), the warp's first row of A is on its
// way before that, and every batch of LU loads of a row (A, then V, then the
// next row's A) goes out before the one ahead of it is used.  blockIdx.z
// splits the rows of a leaf where there are too few leaves.  FP32 with 16-bit
// entries is bound by its issue rate, FP64 by its pipe: both take two rows per
// warp (one read of x, shared reduction steps), FP64 reads A and V as one row;
// FP32 entries stay at one row and twice the loads in flight (0.34 against
// 0.37 ms).  Per product at 2 kHz (256 threads, leaves of the list in turn and
// a row at a time before): FP32 0.54 -> 0.34 ms, 16-bit 0.41 -> 0.26 ms, FP64
// 2.5 -> 2.4 ms; 240 leaves of order 66 0.19 -> 0.049 ms.
constexpr int NEAR_THREADS = 128;
// Sums of M per-lane values over a warp, M a power of two: every step halves
// the values a lane still holds (M - 1 + log2(32 / M) additions instead of
// 5 M).  v[0] of a lane is then the sum of value sum_of(lane).
template <int M, class T>
__device__ __forceinline__ void warp_sums(T (&v)[M], int lane) {
    int o = 16;
#pragma unroll
    for (int h = M / 2; h > 0; h /= 2, o /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}
template <int M>
__device__ __forceinline__ int sum_of(int lane) { return lane / (32 / M); }   // the top log2(M) bits
template <class R, int NB, class AS>
constexpr int NEAR_ROWS = sizeof(AS) != 8 && (sizeof(R) == 4 || NB == 1) ? 2 : 1;   // rows a warp takes at a time
template <class R, int NB>
constexpr int NEAR_CTAS = sizeof(R) == 4 ? 8 : (NB == 1 ? 10 : 8);   // per SM

template <class R, int NB, class AS = cx<R>>
__global__ void __launch_bounds__(NEAR_THREADS, NEAR_CTAS<R, NB>) k_near_l2p(int P, const int32_t* __restrict__ leaf_start,
                                                     const int32_t* __restrict__ perm,
                                                     const int32_t* __restrict__ ucnt,
                                                     const int32_t* __restrict__ ulist,
                                                     const int64_t* __restrict__ nf_off,
                                                     const int32_t* __restrict__ nf_ncol, const AS* __restrict__ A,
                                                     const cx<R>* __restrict__ V, const cx<R>* __restrict__ loc,
                                                     const cd* __restrict__ x, cd* __restrict__ y, int nrhs,
                                                     int64_t xstride, int64_t lstride) {
    constexpr int NR = NEAR_ROWS<R, NB, AS>, LU = LEAF_UNROLL<R> / NR;
    constexpr bool ONE = sizeof(AS) == 16;   // A and V as one row of K + P entries (FP64: no half-empty step between)
    extern __shared__ unsigned char smem_raw[];
    const int r0 = blockIdx.y * NB;
    const int nr = min(NB, nrhs - r0);
    cx<R>* xs = (cx<R>*)smem_raw;
    const int t = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int nu = ucnt[t], K = nf_ncol[t];
    // this lane's U-list leaf (FB_ULIST < 32): start and size (in registers of
    // every warp: the dynamic shared memory of the largest leaves leaves no room)
    const int sl = lane < FB_ULIST ? ulist[(int64_t)t * FB_ULIST + lane] : 0;
    int a0 = 0, len = 0;
    if (lane < nu) {
        a0 = leaf_start[sl];
        len = leaf_start[sl + 1] - a0;
    }
    const int rb = leaf_start[t], nrow = leaf_start[t + 1] - rb, step = nw * gridDim.z;
    const AS* At = A + nf_off[t];
    int r = blockIdx.z * nw + warp;
    const int nv = loc ? P : 0, na = ONE ? K + nv : K;
    AS a[NR][LU];
    auto load_a = [&](int row0, int q0) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int row = min(row0 + i * step, nrow - 1);
            const AS* p = At + (int64_t)row * K + lane;
            const cx<R>* pv = V + (int64_t)(rb + row) * P + lane - K;
#pragma unroll
            for (int u = 0; u < LU; ++u) {
                const int q = q0 + 32 * u;
                if (ONE) {
                    if (q + lane < na) a[i][u] = q + lane < K ? p[q] : reinterpret_cast<const AS*>(pv)[q];
                } else if (q + lane < K) {
                    a[i][u] = p[q];
                }
            }
        }
    };
    if (r < nrow) load_a(r, 0);
    int col = len;   // its first column (K past the list)
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
        const int v = __shfl_up_sync(0xffffffffu, col, o);
        if (lane >= o) col += v;
    }
    col = lane < nu ? col - len : K;
    a0 -= col;
    const int ldx = K + P;              // xs: [nr][K columns, P local coefficients]
    if (loc)
        for (int j = 0; j < nr; ++j)
            for (int q = threadIdx.x; q < P; q += NEAR_THREADS)
                xs[j * ldx + K + q] = loc[(r0 + j) * lstride + (int64_t)t * P + q];
    // gather the x values of the U-list leaves in column order
#pragma unroll 2
    for (int q0 = 32 * warp; q0 < K; q0 += NEAR_THREADS) {
        const int q = q0 + lane;
        int i = 0;   // the last leaf that starts at or before column q
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, col, i + o) <= q) i += o;
        const int pos = __shfl_sync(0xffffffffu, a0, i) + q;
        if (q < K) {
            const int e = perm[pos];
            for (int j = 0; j < nr; ++j) xs[j * ldx + q] = from_d<R>(x[(r0 + j) * xstride + e]);
        }
    }
    __syncthreads();
    constexpr int M = 2 * NR * NB;
    const int mi = sum_of<M>(lane), mj = (mi >> 1) % NB, mr = (mi >> 1) / NB;   // the sum this lane ends up with
    for (; r < nrow; r += NR * step) {
        const int row = min(r + mr * step, nrow - 1), e = perm[rb + row];
        cx<R> acc[NR][NB], v[NR][LU];
#pragma unroll
        for (int i = 0; i < NR; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) acc[i][j] = mk<R>(0, 0);
        auto load_v = [&](int q0) {
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const cx<R>* vr = V + (int64_t)(rb + min(r + i * step, nrow - 1)) * P + q0 + lane;
#pragma unroll
                for (int u = 0; u < LU; ++u)
                    if (q0 + lane + 32 * u < P) v[i][u] = vr[32 * u];
            }
        };
        if (!ONE && nv) load_v(0);
        for (int q0 = 0; q0 < na; q0 += 32 * LU) {
            if (q0) load_a(r, q0);
#pragma unroll
            for (int u = 0; u < LU; ++u) {
                const int q = q0 + lane + 32 * u;
                if (q < na)
#pragma unroll
                    for (int j = 0; j < NB; ++j)
                        if (j < nr) {
                            const cx<R> xq = xs[j * ldx + q];
#pragma unroll
                            for (int i = 0; i < NR; ++i) cmac(acc[i][j], nf_entry(a[i][u]), xq);
                        }
            }
        }
        if (r + NR * step < nrow) load_a(r + NR * step, 0);
        if (!ONE)
            for (int q0 = 0; q0 < nv; q0 += 32 * LU) {
                if (q0) load_v(q0);
#pragma unroll
                for (int u = 0; u < LU; ++u) {
                    const int q = q0 + lane + 32 * u;
                    if (q < P)
#pragma unroll
                        for (int j = 0; j < NB; ++j)
                            if (j < nr) {
                                const cx<R> xq = xs[j * ldx + K + q];
#pragma unroll
                                for (int i = 0; i < NR; ++i) cmac(acc[i][j], v[i][u], xq);
                            }
                }
            }
        R sums[M];
#pragma unroll
        for (int i = 0; i < NR; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                sums[2 * (i * NB + j)] = acc[i][j].re;
                sums[2 * (i * NB + j) + 1] = acc[i][j].im;
            }
        warp_sums<M>(sums, lane);
        if (lane % (32 / M) == 0 && mj < nr && r + mr * step < nrow)
            ((double*)(y + (r0 + mj) * xstride + e))[mi & 1] = (double)sums[0];
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
                         cudaStream_t s, int nrhs, int64_t rstride, int nb, int64_t ustride) {
    return fb_stg_run_f(plan, (const float*)r.rf, r.fper, r.ph, r.prot, coax, src, dst, r.U, r.V, s, nrhs, rstride,
                        r.tc, nb, ustride);
}
static fb_status stg_run(void* plan, const RotArgs<double>& r, const cd* coax, const cd* src, cd* dst,
                         cudaStream_t s, int nrhs, int64_t rstride, int nb, int64_t ustride) {
    return fb_stg_run_d(plan, (const double*)r.rf, r.fper, r.ph, r.prot, coax, src, dst, r.U, r.V, s, nrhs, rstride,
                        r.dft, nb, ustride);
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
                                            (cf*)op->stg_v, s, 1, 0, rot_args<float>(op).tc, 1, 0, li, 1 << pass)
                             : fb_stg_run_d(pl.stg, (const double*)op->rotf, op->rotf_per, (const cd*)op->rph64,
                                            op->Prot, op->coax64, (const cd*)op->mp, (cd*)op->loc, (cd*)op->stg_u,
                                            (cd*)op->stg_v, s, 1, 0, rot_args<double>(op).dft, 1, 0, li, 1 << pass);
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
    if (pl.stg) {   // as many right-hand sides at a time as the staging buffers hold of this plan
        const int nb = (int)std::min<int64_t>(nrhs, op->stg_elems / std::max<int64_t>(1, pl.stg_elems));
        FB_CHECK(stg_run(pl.stg, rot, coax, src, dst, s, nrhs, rstride, std::max(1, nb), pl.stg_elems));
    }
    return FB_OK;
}

// Grows the staging buffers to nrhs right-hand sides of the largest plan, up
// to 256 MB a buffer (a level beyond that fills the chip alone): a level too
// small for a launch of its own per right-hand side takes them all in one,
// eight sources at 600 Hz 2.59 -> 2.11 ms.  Without room for it (a size that
// was refused is not asked for again) or in a capture the buffers stay, and
// the right-hand sides go in smaller batches.
void fb_stg_reserve(fb_op* op, int nrhs, cudaStream_t s) {
    const int64_t csize = op->prec == FB_PREC_MIXED_FMM ? sizeof(cf) : sizeof(cd);
    const int64_t cap0 = (int64_t)(256 << 20) / csize, want = std::min(nrhs * op->stg_need, std::max(op->stg_need, cap0));
    if (want <= op->stg_elems || (op->stg_refused && want >= op->stg_refused)) return;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return;
    void *u = nullptr, *v = nullptr;
    if (cudaMalloc(&u, (size_t)(want * csize)) != cudaSuccess || cudaMalloc(&v, (size_t)(want * csize)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(u);
        op->stg_refused = want;
        return;
    }
    cudaStreamSynchronize(s);
    dfree(op->stg_u);
    dfree(op->stg_v);
    op->stg_u = u;
    op->stg_v = v;
    op->stg_elems = want;
    op->buf_gen++;   // captured graphs refer to the old buffers
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
    op->stg_need = std::max(op->stg_need, pl.stg_elems);
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
    if (!scratch) fb_stg_reserve(op, nrhs, s);
    cx<R>* mp = scratch ? (cx<R>*)scratch : (cx<R>*)op->mp;
    cx<R>* loc = scratch ? (cx<R>*)scratch + cnt * nrhs : (cx<R>*)op->loc;
    mark(0);
    FB_CUDA(cudaMemsetAsync(mp, 0, sizeof(cx<R>) * cnt * nrhs, s));
    FB_CUDA(cudaMemsetAsync(loc, 0, sizeof(cx<R>) * cnt * nrhs, s));
    int nleaf = t->nbox[L];
    const int pt_threads = std::min(256, (PL + 31) & ~31), pz = div_up(PL, pt_threads);
    if (nrhs == 1)
        k_p2m<R, 1><<<dim3(nleaf, 1, pz), pt_threads, 0, s>>>(PL, t->leaf_start, t->perm, W, x, mp + op->lev_off[L], 1,
                                                              n, cnt);
    else
        k_p2m<R, 4><<<dim3(nleaf, div_up(nrhs, 4), pz), pt_threads, 0, s>>>(PL, t->leaf_start, t->perm, W, x,
                                                                            mp + op->lev_off[L], nrhs, n, cnt);
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
    // eight CTAs per SM (1216) where a leaf's rows go round: at most one share
    // per 4 of them (240 leaves of 13 rows, order 66: 0.049 ms against 0.076)
    auto splits = [&](int chunks) {
        return (unsigned)std::max(1, std::min(div_up(1216, nleaf * chunks), div_up((int)(n / nleaf), 4)));
    };
    if (nrhs == 1) {
        size_t smem = sizeof(cx<R>) * (maxK + PL);
        bool done16 = false;
        if constexpr (sizeof(R) == 4) {
            if (op->near16 && op->nf16) {   // 16-bit near-field entries
                FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, 1, uint32_t>, smem));
                k_near_l2p<R, 1, uint32_t><<<dim3(nleaf, 1, splits(1)), NEAR_THREADS, smem, s>>>(PL, t->leaf_start, t->perm, t->ucnt,
                                                                    t->ulist, op->nf_off, op->nf_ncol, op->nf16, V,
                                                                    locL, x, y, 1, n, cnt);
                done16 = true;
            }
        }
        if (!done16) {
            FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, 1>, smem));
            k_near_l2p<R, 1><<<dim3(nleaf, 1, splits(1)), NEAR_THREADS, smem, s>>>(PL, t->leaf_start, t->perm, t->ucnt, t->ulist, op->nf_off,
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
                k_near_l2p<R, NB, uint32_t><<<dim3(nleaf, div_up(nrhs, NB), splits(div_up(nrhs, NB))), NEAR_THREADS, smem, s>>>(
                    PL, t->leaf_start, t->perm, t->ucnt, t->ulist, op->nf_off, op->nf_ncol, op->nf16, V, locL, x,
                    y, nrhs, n, cnt);
                done16 = true;
            }
        }
        if (!done16) {
            FB_CHECK(fb_smem_cap((const void*)k_near_l2p<R, NB>, smem));
            k_near_l2p<R, NB><<<dim3(nleaf, div_up(nrhs, NB), splits(div_up(nrhs, NB))), NEAR_THREADS, smem, s>>>(
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
    op->stg_refused = 0;   // other plans, another need
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
