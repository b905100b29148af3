// Stacked translations of composed matrices on the 5th-generation tensor
// cores (tcgen05).
//
// All box pairs of one level that share a translation vector share one
// composed translation matrix T (p^2 x p^2 complex, Sec. 3.3 RCR composed in
// FP64).  The complex GEMM  Y = T X  (X: gathered source multipoles, one
// column per pair) runs as a real GEMM on interleaved (re, im) rows and
// columns,
//     [Y_re(r)]   [ T_re  -T_im ] [X_re]
//     [Y_im(r)] = [ T_im   T_re ] [X_im],
// transposed, so that the matrix rows are the MMA's N:
//     D[pair][row] = sum_k X[pair][k] T[row][k]
// in 3xTF32: every FP32 operand is split into hi (TF32) + lo, and
// D += X_hi T_hi + X_lo T_hi + X_hi T_lo with FP32 accumulation in tensor
// memory.
//
// Tile: 128 pairs x a block of rows of T (at most 224, in equal blocks padded
// to 16; or two blocks of at most 160), accumulators double-buffered (two
// blocks: a ring of three) in tensor memory.
//
// Operands:  A = gathered X rows, read as FP32 and split by the producer
// warps on the way into the canonical layout.  B = T, pre-split and stored in
// global memory already in the canonical no-swizzle K-major layout, one block
// (hi then lo) per (row tile, K chunk of 16); every CTA copies the blocks of
// its tile into its own shared memory (tiles of one matrix run side by side,
// so that all but the first read come out of L2).
//
// Persistent: every CTA walks over its share of the tiles with each role
// running ahead of the next (a tile's setup, a chain of dependent loads, and
// its scatter cost as much as its MMAs at order 12):
//   warps 0-7    A producers: warp w takes every fourth chunk (w % 4) of 64
//                pairs (w / 4), so that a chunk's fixed cost (waits, proxy
//                fence, arrival) is spread over eight pieces per lane, with
//                the loads of its next chunk in flight (two blocks: every
//                second chunk of 32 pairs, as only three stages fit);
//   warp 8       lane 0: bulk copies of T (transaction count);
//   warp 9       lane 0: MMA issuer (6 MMAs per chunk and block, commits to the
//                stage's "empty" barrier);
//   warps 10-17  epilogue: accumulator rows (lane = pair) through shared
//                memory, so that the atomic adds into the targets are
//                coalesced runs of one pair's coefficients;
//   warp 18      source offsets of the next tiles into a ring in shared
//                memory, ahead of the producers.
// L-room at 2 kHz, M2L of level 7 (order 12, 952,630 pairs): 0.78 ms (the
// MMAs alone 0.68 ms); 1.87 ms with pairs as N, one tile per CTA and hi/lo
// planes of X split in a pass of its own, 0.85 ms in clusters of four that
// shared the loads of T and so kept step with their slowest CTA.  The three
// tensor levels together 1.66 ms against 3.54 ms (1.83 in clusters); of the
// shoebox at 1 kHz 0.18 against 0.36 ms.  What is left is shared-memory
// bandwidth: the MMAs read 130 bytes per cycle of it at their peak rate, the
// copies of T, the split X and the epilogue share the rest.
// Every mbarrier wait is bounded; on timeout the kernel records an error
// flag, drains its own copies and MMAs (bounded) and releases tensor memory.
#include <algorithm>
#include <atomic>
#include <functional>

#include <map>

#include "common.cuh"
#include "tc_common.cuh"

namespace {

constexpr int TC_PAIRS = 128;     // box pairs per tile (MMA M)
constexpr int TC_RMAX = 224;      // real output rows per tile (MMA N <= 256; four stages must fit)
// ... of each of a tile's two blocks where one would not do: three accumulators
// have to fit the 512 columns of tensor memory (the third takes the next tile's
// first block while the last one's are read) and three stages shared memory
constexpr int TC_RMAX2 = 160;
constexpr int TC_ACC = 3;         // accumulators, at most
constexpr int TC_KC = 16;         // real K per stage
constexpr int TC_STAGES = 6;      // at most
constexpr int A_BLOCK = TC_PAIRS * TC_KC;   // floats per (hi or lo) block of X
constexpr int PROD_WARPS = 8;     // warps 0-7
constexpr int EPI_WARPS = 8;      // warps 10-17
constexpr int IDX_WARP = 10 + EPI_WARPS;
constexpr int TC_THREADS = 32 * (IDX_WARP + 1);
constexpr int TC_RING = 4;        // tiles of source offsets in shared memory
constexpr int TC_CS = 32;         // accumulator columns staged per epilogue pass
constexpr int TC_STAGING = EPI_WARPS * 32 * (TC_CS + 4);   // floats
// a producer warp takes every fourth chunk, with two blocks every second one
__host__ __device__ constexpr int tc_period(int nblk) { return nblk == 2 ? 2 : 4; }
using tcx::canon;
using tcx::DRAIN_LIMIT;
using tcx::LBO;
using tcx::mbar_init;
using tcx::mbar_test;
using tcx::mbar_wait;
using tcx::mma_commit;
using tcx::mma_tf32;
using tcx::smem_u32;
using tcx::tf32_hi;
using tcx::umma_desc;
static_assert(TC_KC == tcx::KC, "one canonical block width");

}  // namespace

struct TcTask {
    int64_t a_off;          // float offset of the pre-split tiles of T
    int64_t pair_off;
    int32_t npairs, nrt, nkc, p_out2;   // p_out2 = complex rows P_out
    int32_t rt_rows;                    // real rows per row tile (multiple of 16, <= TC_RMAX)
    int32_t p_in2;                      // complex columns P_in
    int64_t src_base, dst_base;         // complex offsets of the source and target levels
};
// Columns [col0, col0 + ncol) of a task, NB blocks of nrow real rows from row0
// on (their chunks of T lie t_blk floats apart).
struct alignas(16) TcTile {
    int64_t t_off, pair_off, src_base, dst_base;
    int32_t p_in2, p_out2, nkc, nrow;
    int32_t row0, col0, ncol, pad;
    int64_t t_blk;
};

// Pre-split canonical tiles of the real interleaved form of a complex matrix.
// One launch for all matrices of a plan (blockIdx.y); a launch each cost 348
// of them 1.5 ms.
struct TcPack {
    int64_t t_off, a_off;
    int32_t rows, cols, nrt, nkc, rt_rows, pad;
};
__global__ void k_tc_pack(const TcPack* __restrict__ packs, const cd* __restrict__ T64, float* __restrict__ A) {
    const TcPack pk = packs[blockIdx.y];
    const cd* T = T64 + pk.t_off;
    float* out = A + pk.a_off;
    const int rows = pk.rows, cols = pk.cols, nrt = pk.nrt, nkc = pk.nkc, rt_rows = pk.rt_rows;
    const int blk_f = rt_rows * TC_KC;
    int64_t total = (int64_t)nrt * nkc * blk_f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t blk = i / blk_f;
        int e = (int)(i % blk_f);
        int rt = (int)(blk / nkc), kc = (int)(blk % nkc);
        int ri = e / TC_KC, ki = e % TC_KC;
        int rr = rt * rt_rows + ri, kk = kc * TC_KC + ki;
        int r = rr >> 1, sr = rr & 1, k = kk >> 1, sk = kk & 1;
        double v = 0.0;
        if (r < rows && k < cols) {
            cd t = T[(int64_t)r * cols + k];
            v = sr == 0 ? (sk == 0 ? t.re : -t.im) : (sk == 0 ? t.im : t.re);
        }
        float f = (float)v;
        float hi = tf32_hi(f);
        float lo = (float)(v - (double)hi);
        float* base = out + blk * 2 * blk_f;
        int off = canon(ri, ki) >> 2;
        base[off] = hi;
        base[blk_f + off] = lo;
    }
}

struct TcArgs {
    const TcTile* tiles;
    int ntiles;
    const float* T;
    const int32_t* src_idx;
    const int32_t* dst_idx;
    const cf* src;
    cf* dst;
    int* err;
    int nrhs;
    int64_t rstride;
    long long wait_limit;
    int inject_stall;
    int nst;           // pipeline stages
    int stage_floats;  // A hi, A lo, then the largest T block (hi, lo)
    int acc_cols;      // tensor memory columns of one accumulator
    int nacc, tmem_cols;   // accumulators; columns to allocate
};

template <int NB>
__global__ void __launch_bounds__(TC_THREADS, 1) k_trans_tc(const TcArgs a) {
    constexpr int PER = tc_period(NB), NP = 2 * PER;   // a producer warp's chunks; its pieces of each per lane
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[TC_STAGES];    // A producers' stores
    __shared__ __align__(8) uint64_t b_bar[TC_STAGES];       // the bulk copies of T
    __shared__ __align__(8) uint64_t empty_bar[TC_STAGES];   // the MMAs of the stage
    __shared__ __align__(8) uint64_t acc_full[TC_ACC], acc_empty[TC_ACC];
    __shared__ __align__(8) uint64_t done_bar;
    __shared__ __align__(8) uint64_t never_bar;              // test hook: nothing arrives on it
    __shared__ __align__(8) uint64_t idx_full[TC_RING], idx_empty[TC_RING];
    __shared__ int64_t s_src[TC_RING][TC_PAIRS];   // source expansion (complex), -1: no pair
    __shared__ int s_nkc[TC_RING], s_len[TC_RING];  // chunks; floats of a source expansion
    __shared__ uint32_t tmem_holder;
    __shared__ int s_fail;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = (1024 - (raw & 1023)) & 1023;
    float* stage0 = (float*)(smem_raw + pad);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nst = a.nst;
    const int ct0 = blockIdx.x, ncta = gridDim.x;   // this CTA's tiles: ct0, ct0 + ncta, ...
    if (warp == 0) {
        tcx::tmem_alloc(&tmem_holder, a.tmem_cols);
    }
    if (tid == 0) {
        s_fail = 0;
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(&full_bar[s], PROD_WARPS / PER);   // the warps of a chunk
            mbar_init(&b_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < TC_ACC; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], EPI_WARPS);
        }
        for (int r = 0; r < TC_RING; ++r) {
            mbar_init(&idx_full[r], 1);
            mbar_init(&idx_empty[r], PROD_WARPS);
        }
        mbar_init(&done_bar, 1);
        mbar_init(&never_bar, 1);
        tcx::fence_mbar_init();
    }
    tcx::fence_before_sync();
    __syncthreads();
    tcx::fence_after_sync();
    const uint32_t tmem = tmem_holder;

    if (warp < PROD_WARPS) {
        // ---------------- A producers: NP (pair, 4 K values) pieces a lane ---
        // eight consecutive lanes store one 128-byte core matrix (no bank conflicts)
        const int quarter = lane >> 3, jb = warp / PER * (8 * NP) + (lane & 7);   // pairs jb + 8 i
        const int d0 = canon(jb, 4 * quarter) >> 2, dstep = tcx::SBO / 4;     // stage offset of piece i: d0 + i dstep
        const float* g[NP];
        int len = 0;             // floats of a source expansion from the lane's quarter on
        uint32_t has = 0;        // pieces with a pair
        bool al = true;          // every piece 16-byte aligned
        int c = warp % PER, nkc = 0, it = -1, ct = ct0 - ncta;   // load cursor: chunk of tile it
        bool fail = false;
        // moves the cursor to this warp's next chunk; false at the end
        auto seek = [&]() -> bool {
            while (c >= nkc) {
                if (it >= 0 && lane == 0)   // the tile's offsets are no longer needed
                    tcx::mbar_arrive(&idx_empty[it % TC_RING]);
                c -= nkc;
                nkc = 0;
                ++it;
                ct += ncta;
                if (ct >= a.ntiles) return false;
                const int r = it % TC_RING;
                const bool ok = mbar_wait(smem_u32(&idx_full[r]), (it / TC_RING) & 1, a.wait_limit);
                if (!__all_sync(0xffffffffu, ok)) {
                    atomicExch(&s_fail, 1);
                    fail = true;
                    return false;
                }
                nkc = s_nkc[r];
                if (c < nkc) {
                    len = s_len[r] - 4 * quarter;
                    has = 0;
                    al = true;
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        const int64_t o = s_src[r][jb + 8 * i];
                        if (o >= 0) has |= 1u << i;
                        g[i] = (const float*)(a.src + (o >= 0 ? o : 0)) + 4 * quarter;
                        al = al && ((uintptr_t)g[i] & 15) == 0;
                    }
                }
                __syncwarp();
            }
            return true;
        };
        auto fetch = [&](float4 (&v)[NP]) {
            const int n = len - c * TC_KC;   // an even count
            if (al && n >= 4) {
#pragma unroll
                for (int i = 0; i < NP; ++i)
                    v[i] = has >> i & 1 ? __ldg(reinterpret_cast<const float4*>(g[i] + c * TC_KC))
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    float2 p = make_float2(0.f, 0.f), q = p;
                    if ((has >> i & 1) && n >= 2) p = __ldg(reinterpret_cast<const float2*>(g[i] + c * TC_KC));
                    if ((has >> i & 1) && n >= 4) q = __ldg(reinterpret_cast<const float2*>(g[i] + c * TC_KC) + 1);
                    v[i] = make_float4(p.x, p.y, q.x, q.y);
                }
            }
            c += PER;
        };
        float4 cur[NP], nxt[NP];
        bool more = seek();
        if (more) fetch(cur);
        for (int s = warp % PER, u = 0; more; s += PER) {   // stage s of its u-th use
            const bool next = seek();
            if (next) fetch(nxt);
            while (s >= nst) {
                s -= nst;
                ++u;
            }
            const bool ok = u == 0 || mbar_wait(smem_u32(&empty_bar[s]), (u - 1) & 1, a.wait_limit);
            if (!__all_sync(0xffffffffu, ok)) {
                atomicExch(&s_fail, 1);
                break;
            }
            float* st = stage0 + (size_t)s * a.stage_floats + d0;
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const float4 x = cur[i];
                const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
                *reinterpret_cast<float4*>(st + i * dstep) = h;
                *reinterpret_cast<float4*>(st + A_BLOCK + i * dstep) =
                    make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
                cur[i] = nxt[i];
            }
            // generic-proxy stores become visible to the tensor core's reads
            tcx::fence_proxy_async();
            __syncwarp();
            if (lane == 0)
                tcx::mbar_arrive(&full_bar[s]);
            more = next;
        }
    } else if (warp == 8) {
        // ---------------- chunks of T: one bulk copy per block and stage ------
        if (lane == 0) {
            int64_t cc = 0;
            int s = 0;
            uint32_t ph = 1;
            bool fail = false;
            TcTile tn;
            if (ct0 < a.ntiles) tn = a.tiles[ct0];
            for (int ct = ct0; ct < a.ntiles && !fail; ct += ncta) {
                const TcTile tl = tn;
                if (ct + ncta < a.ntiles) tn = a.tiles[ct + ncta];
                const int blk = 2 * tl.nrow * TC_KC;
                const uint32_t bytes = (uint32_t)(blk * sizeof(float));
                const float* g = a.T + tl.t_off;
                for (int c = 0; c < tl.nkc; ++c, ++cc, g += blk) {
                    if (cc >= nst && !mbar_wait(smem_u32(&empty_bar[s]), ph, a.wait_limit)) {
                        atomicExch(&s_fail, 1);
                        fail = true;
                        break;
                    }
                    const uint32_t bb = smem_u32(&b_bar[s]);
                    const uint32_t dB = smem_u32(stage0 + (size_t)s * a.stage_floats + 2 * A_BLOCK);
                    tcx::mbar_expect(bb, NB * bytes);
#pragma unroll
                    for (int h = 0; h < NB; ++h) tcx::bulk_copy(dB + h * bytes, g + h * tl.t_blk, bytes, bb);
                    if (++s == nst) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            // every bulk copy this CTA issued lands before it may exit
            for (int64_t k = cc > nst ? cc - nst : 0; k < cc; ++k)
                mbar_wait(smem_u32(&b_bar[k % nst]), (uint32_t)(k / nst) & 1, DRAIN_LIMIT);
        }
        __syncwarp();
    } else if (warp == 9) {
        // ---------------- MMA issuer ----------------------------------------
        if (lane == 0) {
            // test hook: a wait on a barrier nothing arrives on runs out
            bool fail = a.inject_stall && !mbar_wait(smem_u32(&never_bar), 0, a.wait_limit);
            if (fail) atomicExch(&s_fail, 1);
            int s = 0, b = 0, unit = 0;   // unit: accumulators used so far
            uint32_t ph = 0, aph = 1;
            // Operand descriptors differ in their start address alone, a field of
            // 16-byte units that no sum below carries out of (shared memory ends
            // below its 256 KB).
            const uint64_t d0 = umma_desc(smem_u32(stage0));
            const uint32_t dlo = (uint32_t)d0, dhi = (uint32_t)(d0 >> 32), dstep = (uint32_t)(a.stage_floats * 4) >> 4;
            auto desc = [dhi](uint32_t lo) { return (uint64_t)dhi << 32 | lo; };
            uint32_t dof = dlo;
            // A wait costs this thread some 200 cycles behind the other warps'
            // shared-memory traffic: a stage's barriers are looked at while the
            // one before is issued.
            bool ready = false;
            int nkc_n = 0, nrow_n = 0;
            if (ct0 < a.ntiles) {
                nkc_n = a.tiles[ct0].nkc;
                nrow_n = a.tiles[ct0].nrow;
            }
            for (int ct = ct0; ct < a.ntiles && !fail; ct += ncta) {
                const int nkc = nkc_n, nrow = nrow_n;
                if (ct + ncta < a.ntiles) {
                    nkc_n = a.tiles[ct + ncta].nkc;
                    nrow_n = a.tiles[ct + ncta].nrow;
                }
                uint32_t acc[NB];
                uint64_t* fullb[NB];
#pragma unroll
                for (int h = 0; h < NB; ++h, ++unit) {
                    if (unit >= a.nacc && !fail && !mbar_wait(smem_u32(&acc_empty[b]), aph, a.wait_limit)) {
                        atomicExch(&s_fail, 1);
                        fail = true;
                    }
                    acc[h] = tmem + (uint32_t)(b * a.acc_cols);
                    fullb[h] = &acc_full[b];
                    if (++b == a.nacc) {
                        b = 0;
                        aph ^= 1;
                    }
                }
                if (fail) break;
                const uint32_t idesc = tcx::idesc_tf32(TC_PAIRS, nrow);
                const uint32_t blo = (uint32_t)(nrow * TC_KC * 4) >> 4;   // from T's hi block to its lo block
                for (int c = 0; c < nkc; ++c) {
                    if (!ready && (!mbar_wait(smem_u32(&full_bar[s]), ph, a.wait_limit) ||
                                   !mbar_wait(smem_u32(&b_bar[s]), ph, a.wait_limit))) {
                        atomicExch(&s_fail, 1);
                        fail = true;
                        break;
                    }
                    const int s1 = s + 1 == nst ? 0 : s + 1;
                    const uint32_t p1 = s1 == 0 ? ph ^ 1 : ph;
                    ready = mbar_test(smem_u32(&full_bar[s1]), p1) & mbar_test(smem_u32(&b_bar[s1]), p1);
                    tcx::fence_after_sync();
#pragma unroll
                    for (int h = 0; h < NB; ++h)
#pragma unroll
                        for (int ks = 0; ks < TC_KC / 8; ++ks) {
                            const uint32_t aH = dof + ((ks * 2 * LBO) >> 4),
                                           bH = aH + ((2 * A_BLOCK * 4) >> 4) + h * 2 * blo;
                            mma_tf32(acc[h], desc(aH), desc(bH), idesc, ks == 0 ? (uint32_t)c : 1u);
                            mma_tf32(acc[h], desc(aH + ((A_BLOCK * 4) >> 4)), desc(bH), idesc, 1u);
                            mma_tf32(acc[h], desc(aH), desc(bH + blo), idesc, 1u);
                        }
                    mma_commit(&empty_bar[s]);
                    dof = s1 == 0 ? dlo : dof + dstep;
                    s = s1;
                    ph = p1;
                }
                if (!fail)
#pragma unroll
                    for (int h = 0; h < NB; ++h) mma_commit(fullb[h]);
            }
            // completion of every MMA issued above (also on failure)
            mma_commit(&done_bar);
        }
        __syncwarp();
    } else if (warp == IDX_WARP) {
        // ---------------- source offsets, up to TC_RING tiles ahead -----------
        TcTile tn;
        if (ct0 < a.ntiles) tn = a.tiles[ct0];
        int it = 0;
        for (int ct = ct0; ct < a.ntiles; ct += ncta, ++it) {
            const TcTile tl = tn;
            if (ct + ncta < a.ntiles) tn = a.tiles[ct + ncta];
            int64_t o[TC_PAIRS / 32];
#pragma unroll
            for (int q = 0; q < TC_PAIRS / 32; ++q) {
                const int j = q * 32 + lane;
                o[q] = -1;
                if (j < tl.ncol) {
                    const int col = tl.col0 + j, pr = col / a.nrhs;
                    o[q] = (int64_t)(col - pr * a.nrhs) * a.rstride + tl.src_base +
                           (int64_t)a.src_idx[tl.pair_off + pr] * tl.p_in2;
                }
            }
            const int r = it % TC_RING;
            const bool ok = it < TC_RING || mbar_wait(smem_u32(&idx_empty[r]), (it / TC_RING - 1) & 1, a.wait_limit);
            if (!__all_sync(0xffffffffu, ok)) {
                atomicExch(&s_fail, 1);
                break;
            }
#pragma unroll
            for (int q = 0; q < TC_PAIRS / 32; ++q) s_src[r][q * 32 + lane] = o[q];
            if (lane == 0) {
                s_nkc[r] = tl.nkc;
                s_len[r] = 2 * tl.p_in2;
            }
            __syncwarp();
            if (lane == 0) tcx::mbar_arrive(&idx_full[r]);
        }
    } else {
        // ---------------- epilogue: accumulator lanes 32 quad .. 32 quad + 31,
        // every second group of TC_CS columns (two warps per quadrant) --------
        const int ew = warp - 10, quad = warp & 3, half = ew >> 2;
        float* sg = stage0 + (size_t)nst * a.stage_floats + ew * 32 * (TC_CS + 4);
        float* row = sg + lane * (TC_CS + 4);
        TcTile tn;
        if (ct0 < a.ntiles) tn = a.tiles[ct0];
        int b = 0;
        uint32_t aph = 0;
        bool fail = false;
        for (int ct = ct0; ct < a.ntiles && !fail; ct += ncta) {
            const TcTile tl = tn;
            const int j = quad * 32 + lane;   // this lane's pair
            int64_t dst = 0;                  // its target expansion (floats)
            if (j < tl.ncol) {
                const int col = tl.col0 + j, pr = col / a.nrhs;
                dst = 2 * ((int64_t)(col - pr * a.nrhs) * a.rstride + tl.dst_base +
                           (int64_t)a.dst_idx[tl.pair_off + pr] * tl.p_out2) + tl.row0;
            }
            if (ct + ncta < a.ntiles) tn = a.tiles[ct + ncta];
#pragma unroll 1
            for (int h = 0; h < NB; ++h, dst += tl.nrow) {
                const bool full = mbar_wait(smem_u32(&acc_full[b]), aph, a.wait_limit);
                if (!__all_sync(0xffffffffu, full)) {   // the whole warp goes on or none of it
                    atomicExch(&s_fail, 1);
                    fail = true;
                    break;
                }
                tcx::fence_after_sync();
                const int npair = min(32, tl.ncol - quad * 32), rows = min(tl.nrow, 2 * tl.p_out2 - tl.row0 - h * tl.nrow);
                const uint32_t acc = tmem + (uint32_t)(b * a.acc_cols) + ((uint32_t)(quad * 32) << 16);
                // 16-byte adds where every target of the warp is aligned to them
                const bool wide = __all_sync(0xffffffffu, (dst & 3) == 0 && (((uintptr_t)a.dst) & 15) == 0);
                int c0 = half * TC_CS;
                for (; c0 < tl.nrow; c0 += 2 * TC_CS) {
                    uint32_t v[32];   // (columns past the block lie within the accumulator's)
                    tcx::tmem_ld32(acc + (uint32_t)c0, v);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        *reinterpret_cast<uint4*>(row + 4 * q) = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                    __syncwarp();
                    float* dp = (float*)a.dst + c0;
                    const int rn = rows - c0;   // an even count
                    if (wide) {   // 8 lanes a pair, 4 pairs at a time
                        const int k = 4 * (lane & 7);
#pragma unroll 4
                        for (int t = lane >> 3; t < 32; t += 4) {
                            const int64_t dt = __shfl_sync(0xffffffffu, dst, t);
                            const float4 x = *reinterpret_cast<const float4*>(sg + t * (TC_CS + 4) + k);
                            if (t < npair) {
                                if (k + 4 <= rn) atomicAdd(reinterpret_cast<float4*>(dp + dt + k), x);
                                else if (k + 2 <= rn) atomicAdd(reinterpret_cast<float2*>(dp + dt + k), make_float2(x.x, x.y));
                            }
                        }
                    } else {      // 16 lanes a pair, 2 pairs at a time
                        const int k = 2 * (lane & 15);
#pragma unroll 4
                        for (int t = lane >> 4; t < 32; t += 2) {
                            const int64_t dt = __shfl_sync(0xffffffffu, dst, t);
                            const float2 x = *reinterpret_cast<const float2*>(sg + t * (TC_CS + 4) + k);
                            if (t < npair && k + 2 <= rn) atomicAdd(reinterpret_cast<float2*>(dp + dt + k), x);
                        }
                    }
                    __syncwarp();
                }
                // this warp's share of the accumulator is read
                tcx::fence_before_sync();
                __syncwarp();
                if (lane == 0) tcx::mbar_arrive(&acc_empty[b]);
                if (++b == a.nacc) {
                    b = 0;
                    aph ^= 1;
                }
            }
        }
    }

    const bool done = mbar_wait(smem_u32(&done_bar), 0, DRAIN_LIMIT);
    __syncthreads();
    if ((!done || s_fail) && tid == 0) atomicExch(a.err, 1);
    tcx::fence_after_sync();
    if (warp == 0)
        tcx::tmem_dealloc(tmem, a.tmem_cols);
}

// ------------------------------------------------------------- host side ----
// One launch: the tiles of the tasks with the same accumulator size.
struct TcLaunch {
    int rows_max = 0, acc_cols = 0, nblk = 1, nacc = 2, tmem_cols = 0;
    std::vector<int> tasks;
    int nst = 0;   // pipeline stages
    size_t smem = 0;
};
struct TcTiles {
    TcTile* d = nullptr;
    std::vector<int> count;   // tiles per launch, consecutive in d
};
struct TcPlanImpl {
    std::vector<TcTask> h_tasks;
    std::vector<TcLaunch> launches;
    float* A = nullptr;
    int* err = nullptr;
    const int32_t* src_idx = nullptr;
    const int32_t* dst_idx = nullptr;
    int64_t a_floats = 0;
    std::map<int, TcTiles> tiles;   // per number of right-hand sides (built on first use beyond one)
};

static size_t tc_stage_bytes(int rows) { return (size_t)(2 * A_BLOCK + 2 * rows * TC_KC) * sizeof(float); }
static const void* tc_kernel(int nblk) { return nblk == 2 ? (const void*)k_trans_tc<2> : (const void*)k_trans_tc<1>; }

// Stages and shared memory of a launch (one CTA per SM: at least a share
// such that no second CTA's allocation waits for tensor memory).  At least as
// many stages as a producer warp's period of chunks: when it waits for a
// stage's last use, all uses before that one must be known complete (its
// previous chunk's wait covers them then), or the barrier's phase parity
// would be ambiguous.
static fb_status tc_configure(TcLaunch& ln) {
    const size_t stage = tc_stage_bytes(ln.nblk * ln.rows_max), fixed = TC_STAGING * sizeof(float) + 1024;
    ln.nst = (int)std::max<size_t>(2, std::min<size_t>(TC_STAGES, (220 * 1024 - fixed) / stage));
    if (ln.nst < tc_period(ln.nblk)) return fb_fail(FB_ERR_STATE, "tensor-core translation: too few pipeline stages");
    ln.smem = std::max(ln.nst * stage + fixed, (size_t)116 * 1024);
    FB_CHECK(fb_smem_cap(tc_kernel(ln.nblk), ln.smem));
    return FB_OK;
}

// Tiles of the plan for nrhs right-hand sides: per launch the ones of most
// work first, those of one matrix side by side.
static void tc_make_tiles(const TcPlanImpl* pl, int nrhs, std::vector<TcTile>& out, std::vector<int>& count) {
    for (const TcLaunch& ln : pl->launches) {
        std::map<std::pair<int, int>, std::vector<int>, std::greater<std::pair<int, int>>> by;
        for (int ti : ln.tasks) by[{pl->h_tasks[ti].nkc, pl->h_tasks[ti].rt_rows}].push_back(ti);
        const size_t first = out.size();
        for (const auto& kv : by)
            for (int ti : kv.second) {
                const TcTask& tk = pl->h_tasks[ti];
                const int ncol = tk.npairs * nrhs;
                for (int rt = 0; rt < tk.nrt; rt += ln.nblk)
                    for (int c0 = 0; c0 < ncol; c0 += TC_PAIRS) {
                        TcTile t = {};
                        t.t_blk = (int64_t)tk.nkc * 2 * tk.rt_rows * TC_KC;
                        t.t_off = tk.a_off + rt * t.t_blk;
                        t.pair_off = tk.pair_off;
                        t.src_base = tk.src_base;
                        t.dst_base = tk.dst_base;
                        t.p_in2 = tk.p_in2;
                        t.p_out2 = tk.p_out2;
                        t.nkc = tk.nkc;
                        t.nrow = tk.rt_rows;
                        t.row0 = rt * tk.rt_rows;
                        t.col0 = c0;
                        t.ncol = std::min(TC_PAIRS, ncol - c0);
                        out.push_back(t);
                    }
            }
        count.push_back((int)(out.size() - first));
    }
}

// Bound of the pipeline's device waits (mbarrier polls) and the test hook
// that makes one of them run out; library-wide, read at each launch.
static std::atomic<long long> g_wait_limit{1LL << 26};
static std::atomic<int> g_inject_stall{0};
long long fb_tc_set_wait_limit(long long limit) { return g_wait_limit.exchange(limit); }
int fb_tc_set_inject_stall(int on) { return g_inject_stall.exchange(on ? 1 : 0); }
long long fb_tc_wait_limit() { return g_wait_limit.load(); }
int fb_tc_inject_stall() { return g_inject_stall.load(); }

static fb_status tc_tiles_for(TcPlanImpl* pl, int nrhs, const TcTiles** out) {
    auto it = pl->tiles.find(nrhs);
    if (it == pl->tiles.end()) {
        std::vector<TcTile> h;
        TcTiles t;
        tc_make_tiles(pl, nrhs, h, t.count);
        FB_CHECK(dalloc(&t.d, h.size()));
        FB_CUDA(cudaMemcpy(t.d, h.data(), sizeof(TcTile) * h.size(), cudaMemcpyHostToDevice));
        it = pl->tiles.emplace(nrhs, t).first;
    }
    if (out) *out = &it->second;
    return FB_OK;
}

// Builds a tensor-core plan for groups of box pairs; each group shares one
// composed translation matrix (job) and reads the source expansions of one
// level.
fb_status fb_tc_build_groups(fb_op* op, const std::vector<TcGroup>& groups, const int32_t* src_idx,
                             const int32_t* dst_idx, void** slot, cudaStream_t s) {
    TcPlanImpl* pl = new TcPlanImpl();
    *slot = pl;
    pl->src_idx = src_idx;
    pl->dst_idx = dst_idx;
    for (const TcGroup& g : groups) {
        const ComposeJob& jb = op->h_jobs[g.job];
        const int Pin = jb.p_in * jb.p_in, Pout = jb.p_out * jb.p_out;
        TcTask tk;
        tk.a_off = pl->a_floats;
        tk.pair_off = g.pair_off;
        tk.npairs = g.npairs;
        // Two blocks of rows in one tile where that is all rows (orders 11 and
        // 12): X is gathered and split once instead of twice, order 12 0.85
        // against 1.16 ms (level 7 above, both in clusters).  With more tiles the three stages it
        // leaves cost more than the gathers saved: order 20 in 3 x 2 blocks of
        // 144 0.59 ms, in 4 of 208 0.56 ms.
        tk.nrt = div_up(2 * Pout, TC_RMAX);
        const int nblk = tk.nrt == 2 && 2 * Pout <= 2 * TC_RMAX2 ? 2 : 1;
        tk.rt_rows = (div_up(2 * Pout, tk.nrt) + 15) & ~15;
        tk.nkc = div_up(2 * Pin, TC_KC);
        tk.p_out2 = Pout;
        tk.p_in2 = Pin;
        tk.src_base = op->lev_off[g.src_level];
        tk.dst_base = op->lev_off[g.dst_level];
        int cols = 32;
        while (cols < tk.rt_rows) cols *= 2;
        if (nblk == 2) cols = std::min(cols, TC_RMAX2);
        auto ln = std::find_if(pl->launches.begin(), pl->launches.end(),
                               [&](const TcLaunch& l) { return l.acc_cols == cols && l.nblk == nblk; });
        if (ln == pl->launches.end()) {
            TcLaunch l;
            l.acc_cols = cols;
            l.nblk = nblk;
            l.nacc = nblk == 2 ? 3 : 2;
            l.tmem_cols = nblk == 2 ? 512 : 2 * cols;
            ln = pl->launches.insert(pl->launches.end(), l);
        }
        ln->rows_max = std::max(ln->rows_max, (int)tk.rt_rows);
        ln->tasks.push_back((int)pl->h_tasks.size());
        pl->h_tasks.push_back(tk);
        pl->a_floats += (int64_t)tk.nrt * tk.nkc * 2 * tk.rt_rows * TC_KC;
    }
    if (pl->h_tasks.empty()) return FB_OK;
    FB_CHECK(dalloc(&pl->A, pl->a_floats));
    FB_CHECK(dalloc(&pl->err, 1));
    FB_CUDA(cudaMemsetAsync(pl->err, 0, sizeof(int), s));
    for (TcLaunch& ln : pl->launches) FB_CHECK(tc_configure(ln));
    FB_CHECK(tc_tiles_for(pl, 1, nullptr));
    std::vector<TcPack> packs;
    int64_t most = 0;
    for (size_t i = 0; i < groups.size(); ++i) {
        const TcTask& tk = pl->h_tasks[i];
        const ComposeJob& jb = op->h_jobs[groups[i].job];
        packs.push_back(TcPack{jb.t_off, tk.a_off, tk.p_out2, jb.p_in * jb.p_in, tk.nrt, tk.nkc, tk.rt_rows, 0});
        most = std::max(most, (int64_t)tk.nrt * tk.nkc * tk.rt_rows * TC_KC);
    }
    TcPack* d = nullptr;
    FB_CHECK(dalloc(&d, packs.size()));
    cudaError_t e = cudaMemcpyAsync(d, packs.data(), sizeof(TcPack) * packs.size(), cudaMemcpyHostToDevice, s);
    for (size_t p0 = 0; p0 < packs.size() && e == cudaSuccess; p0 += 65535) {
        k_tc_pack<<<dim3((unsigned)std::min<int64_t>(div_up(most, 256), 512),
                         (unsigned)std::min<size_t>(65535, packs.size() - p0)),
                    256, 0, s>>>(d + p0, op->T64, pl->A);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dfree(d);
    if (e != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("tensor translation tables: ") + cudaGetErrorString(e));
    return FB_OK;
}

// M2L groups (every non-empty (level, offset) group) of the given levels.
fb_status fb_tc_build(fb_op* op, const std::vector<int>& levels, void** slot, cudaStream_t s) {
    const fb_tree* t = op->tree;
    std::vector<TcGroup> groups;
    for (int l : levels)
        for (int c = 0; c < FB_NOFF; ++c) {
            int64_t g0 = t->m2l_group[(size_t)l * FB_NOFF + c], g1 = t->m2l_group[(size_t)l * FB_NOFF + c + 1];
            if (g1 == g0) continue;
            int job = op->m2l_job[(size_t)l * FB_NOFF + c];
            groups.push_back(TcGroup{job, g0, (int32_t)(g1 - g0), l, l});
        }
    return fb_tc_build_groups(op, groups, t->m2l_src, t->m2l_dst, slot, s);
}

// Runs a plan on nrhs sets of expansions (set r at src/dst + r * rstride).
// The columns of a task are its (pair, rhs) combinations, so every tile of
// the translation matrix is loaded once for all right-hand sides.
fb_status fb_tc_run(fb_op* op, void* plan, const cf* src, cf* dst, cudaStream_t s, int nrhs, int64_t rstride) {
    TcPlanImpl* pl = (TcPlanImpl*)plan;
    if (!pl || pl->h_tasks.empty()) return FB_OK;
    const TcTiles* tiles = nullptr;
    FB_CHECK(tc_tiles_for(pl, nrhs, &tiles));
    TcArgs a;
    a.tiles = tiles->d;
    a.T = pl->A;
    a.src_idx = pl->src_idx;
    a.dst_idx = pl->dst_idx;
    a.src = src;
    a.dst = dst;
    a.err = pl->err;
    a.nrhs = nrhs;
    a.rstride = rstride;
    a.wait_limit = g_wait_limit.load();
    a.inject_stall = g_inject_stall.load();
    int dev = 0, sms = 0;
    FB_CUDA(cudaGetDevice(&dev));
    FB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    for (size_t i = 0; i < pl->launches.size(); a.tiles += tiles->count[i], ++i) {
        const TcLaunch& ln = pl->launches[i];
        a.ntiles = tiles->count[i];
        a.acc_cols = ln.acc_cols;
        a.nst = ln.nst;
        a.nacc = ln.nacc;
        a.tmem_cols = ln.tmem_cols;
        a.stage_floats = (int)(tc_stage_bytes(ln.nblk * ln.rows_max) / sizeof(float));
        FB_CHECK(fb_smem_cap(tc_kernel(ln.nblk), ln.smem));
        const unsigned grid = (unsigned)std::min(sms, a.ntiles);
        if (ln.nblk == 2)
            k_trans_tc<2><<<grid, TC_THREADS, ln.smem, s>>>(a);
        else
            k_trans_tc<1><<<grid, TC_THREADS, ln.smem, s>>>(a);
        FB_LAUNCH_CHECK();
        fb_count_launch();
    }
    return FB_OK;
}

// Error flags of the tensor-core kernels of an operator (1 = a bounded wait
// ran out); read and cleared (the caller has synchronised the work).
fb_status fb_tc_check(const fb_op* op) {
    std::vector<void*> plans = {op->tc_plan, op->tc_plan_all};
    for (int l = 0; l <= FB_MAXLEV; ++l) {
        plans.push_back(op->tc_m2m[l]);
        plans.push_back(op->tc_l2l[l]);
    }
    if (op->stc_err) {   // tensor-core staged rotation passes
        int h = 0;
        FB_CUDA(cudaMemcpy(&h, op->stc_err, sizeof(int), cudaMemcpyDeviceToHost));
        if (h) {
            FB_CUDA(cudaMemset(op->stc_err, 0, sizeof(int)));
            return fb_fail(FB_ERR_TIMEOUT, "tensor-core staged rotation kernel: a bounded wait ran out");
        }
    }
    for (void* v : plans) {
        TcPlanImpl* pl = (TcPlanImpl*)v;
        if (!pl || !pl->err) continue;
        int h = 0;
        FB_CUDA(cudaMemcpy(&h, pl->err, sizeof(int), cudaMemcpyDeviceToHost));
        if (h) {
            FB_CUDA(cudaMemset(pl->err, 0, sizeof(int)));
            return fb_fail(FB_ERR_TIMEOUT, "tensor-core translation kernel: a bounded wait ran out");
        }
    }
    return FB_OK;
}

void fb_tc_free(void*& plan) {
    TcPlanImpl* pl = (TcPlanImpl*)plan;
    if (!pl) return;
    dfree(pl->A);
    dfree(pl->err);
    for (auto& kv : pl->tiles) dfree(kv.second.d);
    delete pl;
    plan = nullptr;
}
