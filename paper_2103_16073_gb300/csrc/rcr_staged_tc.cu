// The three passes of the staged RCR translation (Sec. 3.3) on the tensor
// cores (tcgen05, 3xTF32).
//
// R and B (rotation, back-rotation) of rcr_staged.cu are real-by-complex
// GEMMs per (polar-angle group, degree n, folded part): the folded real table
// block d (N x K, N = K = n + 1 or n) applied to the complex vectors of every
// slot (pair) of the group.  C (coaxial) is a complex GEMM per (|t|, order
// |m|) over the degrees.  All three run transposed, slots along M and the
// short dimension of a block as the MMA's N:
//     D[row][col] = sum_k A[row][k] T[col][k],  128 rows = 64 slots x 2,
//   R, B: row = 16 (j / 8) + 8 c + j % 8 is the real (c = 0) or imaginary
//       (c = 1) part of slot j, T the table block;
//   C: row = 64 part + j is the even or odd part of slot j (order 0: even
//       alone), K interleaved: A[row][(k, c)] = u[k].c and
//       T[(i, 0)][(k, .)] = (Re C, -Im C), T[(i, 1)][(k, .)] = (Im C, Re C),
//       so columns 2 i, 2 i + 1 are the real and imaginary part of degree i.
// T is K-major, pre-split into TF32 hi + lo and laid out canonically per K
// chunk of 16 at setup, so that one bulk copy moves a chunk; A is split by the
// producer warps.  3xTF32: D += A_hi T_hi + A_hi T_lo + A_lo T_hi.
//
// Layout of the staging buffers u and v: coefficient-major, slot innermost,
// u[e * ns + slot] with e = n^2 (+ n for the odd part) + |m|.  The rows of
// every tile are slots, so all three passes read and write whole lines along
// the lanes (8 bytes of every 32-byte sector with slots outermost, where C
// strides over the degrees and R and C store a column at a time).
//
// Persistent: one CTA per SM walks over items (one block T x 64 slots), every
// role running ahead of the next, because an item is a few microseconds of
// dependent latencies (descriptor, slots, operands, products, stores) around
// a few hundred cycles of MMAs:
//   12, 8 or 4 warps (R, C, B)  A producers: a warp takes every third, fourth
//                or second chunk of K, with the loads of its next in flight;
//   one warp     lane 0: bulk copies of the chunks of T (transaction count);
//   one warp     lane 0: MMA issuer, two to four accumulators in tensor memory;
//   4, 8 or 12 warps  epilogue: accumulator lanes 32 (w % 4) .., groups of 16
//                columns in turn; R and C store u and v, B goes through
//                shared memory so that the phased y_{+-m'} = (Y+ +- Y-)/2 are
//                added (atomics) in runs of one target's coefficients;
//   warps 18-19  items and their slots into a ring in shared memory, ahead of
//                the others.
// Room of 240 leaf boxes at 7.5 kHz (orders 116 and 66, M2L): R 0.45 ms, C
// 0.34 ms, B 0.47 ms over both levels; together 3.34 ms with one tile per
// CTA, degree-major u and v, and lanes along a row's K values.  C moves 1 GB
// per pass out of L2 at 6 TB/s; R and B are bound by their warps' issue rate
// around the waits of a chunk.
// Every mbarrier wait is bounded; on timeout the kernel records an error
// flag, drains its own bulk copies and MMAs (bounded) and frees its tensor
// memory.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "rcr_staged.cuh"
#include "tc_common.cuh"

using namespace stg;

namespace {

using tcx::canon;
using tcx::DRAIN_LIMIT;
using tcx::KC;
using tcx::mbar_arrive;
using tcx::mbar_init;
using tcx::mbar_test;
using tcx::mbar_wait;
using tcx::mma_commit;
using tcx::mma_tf32;
using tcx::smem_u32;
using tcx::tf32_hi;
using tcx::umma_desc;

enum { ST_R = 0, ST_B = 1, ST_C = 2 };   // pass

constexpr int STC_M = 2 * STC_SLOTS;     // rows of a tile
constexpr int STC_WORKW = 16;            // producer and epilogue warps
constexpr int STC_IDXW = 2;              // warps 18-19
constexpr int STC_IDX0 = STC_WORKW + 2;
constexpr int STC_THREADS = 32 * (STC_IDX0 + STC_IDXW);
constexpr int STC_STAGES = 8;            // at most
// Items in shared memory.  A producer looks up the item of the chunk two of
// its own ahead before it stores the current one, with one chunk per item 2 x
// 4 items further: the ring has to hold more than those.
constexpr int STC_RING = 12;
constexpr int STC_ACC = 4;               // accumulators, at most
constexpr int STC_SG = 20;               // floats of a staged accumulator row (16 columns, padded)
constexpr size_t STC_SMEM_MAX = 214 * 1024;   // dynamic; the ring (< 11 KB) is static
constexpr size_t STC_SMEM_MIN = 116 * 1024;   // one CTA per SM: its accumulators are always free

// Every producer warp of pass R stores single K values of 16 consecutive m
// (the order its loads coalesce in): core matrices 144 bytes apart put the
// 16 values of two slots into 32 banks.  The other passes store 16-byte rows
// and take the packed layout.
template <int PASS>
struct StcLayout {
    static constexpr int LBO = PASS == ST_R ? 144 : tcx::LBO;
    static constexpr int SBO = (KC / 4) * LBO;
    static constexpr int PLANE = STC_M / 8 * SBO / 4;   // floats of one (hi or lo) A block
    // producer and epilogue warps (R folds its inputs, B scatters with atomics);
    // a producer warp takes every PERIOD-th chunk
    static constexpr int PRODW = PASS == ST_R ? 12 : (PASS == ST_C ? 8 : 4), EPIW = STC_WORKW - PRODW;
    static constexpr int PERIOD = PASS == ST_R ? 3 : (PASS == ST_C ? 4 : 2);
    static constexpr int SHARES = EPIW / 4;             // epilogue warps per 32 accumulator lanes
    static_assert(STC_RING > 2 * PERIOD, "a producer's look-ahead fits the ring");
};

// accumulator columns N (output rows of the table block) and summed length
// K of degree n, folded part `part`, of pass R (0) or B (1)
__host__ __device__ __forceinline__ void stc_dims(int pass, int n, int part, int p_in, int& N, int& K) {
    N = n + 1 - part;
    K = pass == 0 ? N : std::min(n, p_in - 1) + 1 - part;
}

struct StcArgs {
    const StcItem* items;
    int nitems, nrhs;         // items per right-hand side
    int64_t rstride, ustride;   // expansions, u and v of the next right-hand side
    const float* tab;      // R, B: group g's R table at g * 2 tper, B table at g * 2 tper + tper; C: the coaxial blocks
    int64_t tper;
    const StgSlot* slots;
    const int32_t* cidx;   // C: slots of a |t| set
    const cf* X;           // R: source expansions; C: u; B: v
    cf* out;               // R: u; C: v; B: target expansions
    const cf* rph;         // phases e^{i m phi} per direction
    int* err;
    long long wait_limit;
    int64_t ns;            // slots: the stride of a coefficient of u and v
    int prot;
    int nst;               // pipeline stages
    int stage_floats;      // A hi, A lo, then the largest chunk of T (hi, lo)
    int acc_cols, nacc;    // tensor memory columns of an accumulator, accumulators
    int inject_stall;
};

// stores a row's 4 K values as TF32 hi and remainder
__device__ __forceinline__ void split_store(float* st, int plane, const float4& x) {
    const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
    *reinterpret_cast<float4*>(st) = h;
    *reinterpret_cast<float4*>(st + plane) = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
}

// A producer's registers for one chunk: load() issues the loads of chunk c of
// an item, take() makes them the current chunk, store() writes that one.  A
// warp's issue rate is what bounds the producers, so addresses are one
// multiply-add each and only the last chunk of an item pays for its ragged K.
// Rows past the item's slots hold copies of its last slot and are not written
// anywhere; K values past K are zero, as they are in T.
template <int PASS>
struct Producer;

__device__ __forceinline__ float2 ldg2(const char* p) { return __ldg(reinterpret_cast<const float2*>(p)); }

// R: folds and phases the source expansions on the way (m = part + k):
// s_0 = x_0, s_m = x_m e^{i m phi} + x_{-m} e^{-i m phi}, t_m = the difference.
// Lanes: 16 consecutive m of two slots 4 apart, 8 such units per warp and
// chunk.  Slots are sorted by direction, so most groups of 16 share a phase.
template <>
struct Producer<ST_R> {
    float2 xp[8], xm[8], ph[8], cur[8];
    float sg;      // sign of x_{-m} (0: m = 0)
    bool uni, in;  // one direction for all slots; k < K
    __device__ __forceinline__ void load(const StcArgs& a, const StcItem& it, const int64_t* pos, const int32_t* dir,
                                         int sub, int lane, int c) {
        const int k = c * KC + (lane & 15), n = it.n, part = it.part, m = min(part + k, n);
        sg = m == 0 ? 0.f : (part ? -1.f : 1.f);
        in = k < it.K;
        uni = it.uni >> sub & 1;
        const int j0 = 16 * sub + 4 * (lane >> 4);
        const char* xs = (const char*)(a.X + (int64_t)n * n + n);
        const char *bp = xs + 8 * m, *bm = xs - 8 * m, *bh = (const char*)(a.rph + a.prot - 1 + m);
        int64_t o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = pos[j0 + 8 * (i >> 2) + (i & 3)];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            xp[i] = ldg2(bp + 8 * o[i]);
            xm[i] = ldg2(bm + 8 * o[i]);
        }
        const int pw = 8 * (2 * a.prot - 1);
        ph[0] = ldg2(bh + (int64_t)dir[j0] * pw);
        if (!uni) {
#pragma unroll
            for (int i = 1; i < 8; ++i) ph[i] = ldg2(bh + (int64_t)dir[j0 + 8 * (i >> 2) + (i & 3)] * pw);
        }
    }
    __device__ __forceinline__ void fold(int i, float2 e) {
        const float px = xp[i].x + sg * xm[i].x, py = xp[i].y + sg * xm[i].y;
        const float qx = xp[i].x - sg * xm[i].x, qy = xp[i].y - sg * xm[i].y;
        cur[i] = make_float2(px * e.x - qy * e.y, py * e.x + qx * e.y);
    }
    __device__ __forceinline__ void take() {
        if (uni) {
            const float2 e = in ? ph[0] : make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) fold(i, e);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) fold(i, in ? ph[i] : make_float2(0.f, 0.f));
        }
    }
    __device__ __forceinline__ void store(float* st, int sub, int lane) const {
        using L = StcLayout<ST_R>;
        const int k = lane & 15;
        st += ((k >> 2) * L::LBO + 4 * (lane >> 4) * 16 + 4 * sub * L::SBO) / 4 + (k & 3);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float* d = st + (2 * (i >> 2) * L::SBO + (i & 3) * 16) / 4;   // row of the real part
            const float hr = tf32_hi(cur[i].x), hi = tf32_hi(cur[i].y);
            d[0] = hr;
            d[L::PLANE] = cur[i].x - hr;
            d[L::SBO / 4] = hi;
            d[L::PLANE + L::SBO / 4] = cur[i].y - hi;
        }
    }
};

// C: lanes along the slots, one part per warp, 2 slots x 4 pairs of degrees a
// lane.
template <>
struct Producer<ST_C> {
    float4 nxt[8], cur[8];
    __device__ __forceinline__ void load(const StcArgs& a, const StcItem& it, const int64_t* pos, const int32_t*,
                                         int sub, int lane, int c) {
        const int part = sub, am = it.n, left = it.K / 2 - c * (KC / 2);   // degrees
        const char *x0 = (const char*)(a.X + pos[lane]), *x1 = (const char*)(a.X + pos[lane + 32]);
        const int64_t es = 8 * a.ns;
        int n = am + c * (KC / 2), e = n * n + (part ? n : 0) + am;
        float2 x[2][KC / 2];
#pragma unroll
        for (int k = 0; k < KC / 2; ++k) {
            x[0][k] = x[1][k] = make_float2(0.f, 0.f);
            if (left >= KC / 2 || k < left) {
                x[0][k] = ldg2(x0 + e * es);
                x[1][k] = ldg2(x1 + e * es);
            }
            e += 2 * n + 1 + part;
            ++n;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 u = x[i & 1][i & ~1], v = x[i & 1][(i & ~1) + 1];
            nxt[i] = make_float4(u.x, u.y, v.x, v.y);
        }
    }
    __device__ __forceinline__ void take() {
#pragma unroll
        for (int i = 0; i < 8; ++i) cur[i] = nxt[i];
    }
    __device__ __forceinline__ void store(float* st, int sub, int lane) const {
        st += canon(64 * sub + lane, 0) / 4;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            split_store(st + (canon(32 * (i & 1), 4 * (i >> 1)) >> 2), StcLayout<ST_C>::PLANE, cur[i]);
    }
};

// B: E_mu / O_mu (mu = part + k) of v; lanes along the slots, 32 slots per
// warp and chunk, 4 groups of 4 consecutive mu a lane.
template <>
struct Producer<ST_B> {
    float2 nxt[16], cur[16];
    __device__ __forceinline__ void load(const StcArgs& a, const StcItem& it, const int64_t*, const int32_t*, int sub,
                                         int lane, int c) {
        const int j = min(32 * sub + lane, it.ns - 1), left = it.K - c * KC, n = it.n;
        const int64_t es = 8 * a.ns;
        const char* v = (const char*)(a.X + it.uoff + it.s0 + j) + (n * n + (it.part ? n : 0) + it.part + c * KC) * es;
        if (left >= KC) {
#pragma unroll
            for (int k = 0; k < KC; ++k) nxt[k] = ldg2(v + k * es);
        } else {
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                nxt[k] = make_float2(0.f, 0.f);
                if (k < left) nxt[k] = ldg2(v + k * es);
            }
        }
    }
    __device__ __forceinline__ void take() {
#pragma unroll
        for (int k = 0; k < KC; ++k) cur[k] = nxt[k];
    }
    __device__ __forceinline__ void store(float* st, int sub, int lane) const {
        const int j = 32 * sub + lane;
        st += canon(16 * (j >> 3) + (j & 7), 0) / 4;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2* x = cur + 4 * q;
            float* d = st + q * (tcx::LBO / 4);
            split_store(d, StcLayout<ST_B>::PLANE, make_float4(x[0].x, x[1].x, x[2].x, x[3].x));
            split_store(d + tcx::SBO / 4, StcLayout<ST_B>::PLANE, make_float4(x[0].y, x[1].y, x[2].y, x[3].y));
        }
    }
};

// The accumulator of one item to its destination (one warp's share: 32 rows,
// every SHARES-th group of 16 columns from the share-th on).  sg: 32 x STC_SG
// floats of the warp (B).
template <int PASS>
__device__ __forceinline__ void stc_epilogue(const StcArgs& a, const StcItem& it, const int64_t* pos,
                                             const int32_t* dir, uint32_t acc, int quad, int share, int lane,
                                             float* sg) {
    const int N = it.N, n = it.n, part = it.part, ns = it.ns;
    const int64_t es = 8 * a.ns;
    acc += (uint32_t)(quad * 32) << 16;
    for (int c0 = 16 * share; c0 < N; c0 += 16 * StcLayout<PASS>::SHARES) {
        uint32_t v[16];
        if (PASS == ST_R) {
            tcx::tmem_ld16(acc + (uint32_t)c0, v);
            const int j = 16 * quad + 8 * (lane >> 4) + (lane & 7);
            char* u = (char*)(a.out + it.uoff + it.s0 + j) + 4 * (lane >> 3 & 1) + (n * n + (part ? n : 0) + part + c0) * es;
            const int left = j < ns ? N - c0 : 0;
            if (left >= 16) {
#pragma unroll
                for (int i = 0; i < 16; ++i) *reinterpret_cast<uint32_t*>(u + i * es) = v[i];
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (i < left) *reinterpret_cast<uint32_t*>(u + i * es) = v[i];
            }
        } else if (PASS == ST_C) {
            tcx::tmem_ld16(acc + (uint32_t)c0, v);
            const int odd = quad >> 1, j = 32 * (quad & 1) + lane;   // (part: the block's first row)
            const int left = j < ns && (odd == 0 || n > 0) ? (N - c0) / 2 : 0;
            char* w = (char*)(a.out + pos[j]);
            int n1 = n + part + c0 / 2, e = n1 * n1 + (odd ? n1 : 0) + n;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                if (t < left) *reinterpret_cast<uint2*>(w + e * es) = make_uint2(v[2 * t], v[2 * t + 1]);
                e += 2 * n1 + 1 + odd;
                ++n1;
            }
        } else {
            // 16 lanes along m' of one slot, two slots 4 apart (their rows lie 16 banks apart)
            const int i = lane & 15, mp = part + c0 + i, j0 = 16 * quad + 4 * (lane >> 4);
            const bool in = c0 + i < N;
            const char* bh = (const char*)(a.rph + a.prot - 1 + (in ? mp : 0));
            const int pw = 8 * (2 * a.prot - 1);
            int last = dir[j0];
            float2 e = ldg2(bh + (int64_t)last * pw);   // (slots are sorted by direction)
            tcx::tmem_ld16(acc + (uint32_t)c0, v);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(sg + lane * STC_SG + 4 * q) =
                    make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            __syncwarp();
            char* d0 = (char*)(a.out + (int64_t)n * n + n);   // entry (n, 0) of a target
            char *dp = d0 + 8 * mp, *dm = d0 - 8 * mp;
            const float sgn = part ? -0.5f : 0.5f;
            const float* row = sg + 4 * (lane >> 4) * STC_SG + i;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int j = j0 + 8 * (t >> 2) + (t & 3);
                const float re = row[(16 * (t >> 2) + (t & 3)) * STC_SG], im = row[(16 * (t >> 2) + (t & 3) + 8) * STC_SG];
                if (j < ns && in) {
                    const int dj = dir[j];
                    const int64_t o = 8 * pos[j];
                    if (dj != last) {
                        last = dj;
                        e = ldg2(bh + (int64_t)dj * pw);
                    }
                    const float ex = 0.5f * e.x, ey = 0.5f * e.y, fx = sgn * e.x, fy = sgn * e.y;
                    atomicAdd(reinterpret_cast<float2*>(dp + o), make_float2(re * ex + im * ey, im * ex - re * ey));
                    if (mp > 0)
                        atomicAdd(reinterpret_cast<float2*>(dm + o), make_float2(re * fx - im * fy, re * fy + im * fx));
                }
            }
            __syncwarp();
        }
    }
}

template <int PASS>
__device__ __forceinline__ void stc_body(const StcArgs& a) {
    using L = StcLayout<PASS>;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STC_STAGES];    // A producers' stores
    __shared__ __align__(8) uint64_t b_bar[STC_STAGES];       // the bulk copy of the chunk of T
    __shared__ __align__(8) uint64_t empty_bar[STC_STAGES];   // MMAs of the stage complete
    __shared__ __align__(8) uint64_t acc_full[STC_ACC], acc_empty[STC_ACC];
    __shared__ __align__(8) uint64_t idx_full[STC_RING], idx_empty[STC_RING];
    __shared__ __align__(8) uint64_t done_bar;
    __shared__ __align__(8) uint64_t never_bar;               // test hook: nothing arrives on it
    __shared__ StcItem s_item[STC_RING];
    __shared__ int64_t s_pos[STC_RING][STC_SLOTS];   // R: source, B: target expansion, C: slot
    __shared__ int32_t s_dir[STC_RING][STC_SLOTS];   // R, B: direction (phases)
    __shared__ uint32_t tmem_holder;
    __shared__ int s_fail;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = (1024 - (raw & 1023)) & 1023;
    float* stage0 = (float*)(smem_raw + pad);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nst = a.nst;
    if (warp == 0) {
        tcx::tmem_alloc(&tmem_holder, a.nacc * a.acc_cols);
    }
    if (tid == 0) {
        s_fail = 0;
        for (int s = 0; s < STC_STAGES; ++s) {
            mbar_init(&full_bar[s], L::PRODW / L::PERIOD);   // the warps of a chunk
            mbar_init(&b_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < STC_ACC; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], L::EPIW);
        }
        for (int r = 0; r < STC_RING; ++r) {
            mbar_init(&idx_full[r], 1);
            mbar_init(&idx_empty[r], STC_WORKW + 2);
        }
        mbar_init(&done_bar, 1);
        mbar_init(&never_bar, 1);
        tcx::fence_mbar_init();
    }
    tcx::fence_before_sync();
    __syncthreads();
    tcx::fence_after_sync();
    const uint32_t tmem = tmem_holder;
    // this CTA's items: blockIdx.x, + gridDim.x, ...; the it-th is in ring entry it % STC_RING
    const int nmine = (a.nitems * a.nrhs - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    auto item_wait = [&](int it) {
        return mbar_wait(smem_u32(&idx_full[it % STC_RING]), (it / STC_RING) & 1, a.wait_limit);
    };

    if (warp < L::PRODW) {
        // ---------------- A producers ---------------------------------------
        Producer<PASS> p;
        constexpr int PER = L::PERIOD;
        const int first = PASS == ST_R ? warp >> 2 : warp % PER, sub = PASS == ST_R ? warp & 3 : warp / PER;
        int c = first, nkc = 0, it = -1;
        // moves to this warp's next chunk; false at the end
        auto seek = [&]() -> bool {
            while (c >= nkc) {
                __syncwarp();
                if (it >= 0 && lane == 0) mbar_arrive(&idx_empty[it % STC_RING]);   // the item is no longer needed
                c -= nkc;
                nkc = 0;
                if (++it >= nmine) return false;
                if (!__all_sync(0xffffffffu, item_wait(it))) {
                    atomicExch(&s_fail, 1);
                    return false;
                }
                nkc = (s_item[it % STC_RING].K + KC - 1) / KC;
            }
            return true;
        };
        auto load = [&]() {
            const int r = it % STC_RING;
            p.load(a, s_item[r], s_pos[r], s_dir[r], sub, lane, c);
            c += PER;
        };
        bool more = seek(), next = false;
        if (more) {
            load();
            next = seek();
            p.take();
        }
        for (int s = first, u = 0; more; s += PER) {   // stage s of its u-th use
            // the next chunk's loads go out before this one is stored, and its
            // successor is looked up while they are on their way
            if (next) load();
            const bool after = next && seek();
            while (s >= nst) {
                s -= nst;
                ++u;
            }
            const bool ok = u == 0 || mbar_wait(smem_u32(&empty_bar[s]), (u - 1) & 1, a.wait_limit);
            if (!__all_sync(0xffffffffu, ok)) {
                atomicExch(&s_fail, 1);
                break;
            }
            p.store(stage0 + (size_t)s * a.stage_floats, sub, lane);
            // generic-proxy stores become visible to the tensor core's reads
            tcx::fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full_bar[s]);
            if (next) p.take();
            more = next;
            next = after;
        }
    } else if (warp == L::PRODW) {
        // ---------------- chunks of T: one bulk copy per stage ---------------
        if (lane == 0) {
            int cc = 0, s = 0;
            uint32_t ph = 1;
            bool fail = false;
            for (int it = 0; it < nmine && !fail; ++it) {
                const int r = it % STC_RING;
                if (!item_wait(it)) {
                    atomicExch(&s_fail, 1);
                    break;
                }
                const StcItem tl = s_item[r];
                mbar_arrive(&idx_empty[r]);
                const int blk = 2 * stc_pad16(tl.N) * KC, nkc = (tl.K + KC - 1) / KC;
                const uint32_t bytes = (uint32_t)(blk * sizeof(float));
                const float* g = a.tab + tl.tab + (PASS == ST_C ? 0 : ((int64_t)2 * tl.g + (PASS == ST_B)) * a.tper);
                for (int c = 0; c < nkc; ++c, ++cc, g += blk) {
                    if (cc >= nst && !mbar_wait(smem_u32(&empty_bar[s]), ph, a.wait_limit)) {
                        atomicExch(&s_fail, 1);
                        fail = true;
                        break;
                    }
                    const uint32_t bb = smem_u32(&b_bar[s]);
                    const uint32_t dB = smem_u32(stage0 + (size_t)s * a.stage_floats + 2 * L::PLANE);
                    tcx::mbar_expect(bb, bytes);
                    tcx::bulk_copy(dB, g, bytes, bb);
                    if (++s == nst) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            // every bulk copy this CTA issued lands before the CTA may exit
            for (int k = cc > nst ? cc - nst : 0; k < cc; ++k)
                mbar_wait(smem_u32(&b_bar[k % nst]), (uint32_t)(k / nst) & 1, DRAIN_LIMIT);
        }
        __syncwarp();
    } else if (warp == L::PRODW + 1) {
        // ---------------- MMA issuer ----------------------------------------
        if (lane == 0) {
            // test hook: a wait on a barrier nothing arrives on runs out
            bool fail = a.inject_stall && !mbar_wait(smem_u32(&never_bar), 0, a.wait_limit);
            if (fail) atomicExch(&s_fail, 1);
            // operand descriptors: a stage's differ in their start address alone, a
            // field of 16-byte units that no sum below carries out of
            const uint32_t base = smem_u32(stage0);
            const uint64_t dA0 = ((uint64_t)1 << 46) | ((uint64_t)(L::SBO >> 4) << 32) | ((uint64_t)(L::LBO >> 4) << 16) |
                                 ((base & 0x3FFFF) >> 4);
            const uint64_t dB0 = umma_desc(base + 2 * L::PLANE * 4);
            const uint32_t a0 = (uint32_t)dA0, ahi = (uint32_t)(dA0 >> 32), b0 = (uint32_t)dB0, bhi = (uint32_t)(dB0 >> 32);
            const uint32_t dstep = (uint32_t)(a.stage_floats * 4) >> 4;
            auto desc = [](uint32_t lo, uint32_t hi) { return (uint64_t)hi << 32 | lo; };
            int s = 0, b = 0;
            uint32_t ph = 0, aph = 1, dof = 0;
            // This thread's chain of waits (some 200 cycles each behind the other
            // warps' shared-memory traffic) is longer than the MMAs: a stage's
            // barriers are looked at while the one before is issued, the next
            // item's while this one is.
            bool ready = false, iready = false, aready = false;
            int nN = 0, nK = 0;
            auto peek_stage = [&](int s1, uint32_t p1) {
                return mbar_test(smem_u32(&full_bar[s1]), p1) & mbar_test(smem_u32(&b_bar[s1]), p1);
            };
            for (int it = 0; it < nmine && !fail; ++it) {
                const int r = it % STC_RING;
                if (!iready) {
                    if (!item_wait(it)) {
                        atomicExch(&s_fail, 1);
                        break;
                    }
                    nN = s_item[r].N;
                    nK = s_item[r].K;
                }
                const int np = stc_pad16(nN), nkc = (nK + KC - 1) / KC;
                mbar_arrive(&idx_empty[r]);
                iready = false;
                const int b1 = b + 1 == a.nacc ? 0 : b + 1;
                const uint32_t ap1 = b1 == 0 ? aph ^ 1 : aph;
                const int r1 = (it + 1) % STC_RING;
                if (it + 1 < nmine) iready = mbar_test(smem_u32(&idx_full[r1]), ((it + 1) / STC_RING) & 1);
                const bool adone = aready;
                aready = it + 1 >= a.nacc && mbar_test(smem_u32(&acc_empty[b1]), ap1);
                if (it >= a.nacc && !adone && !mbar_wait(smem_u32(&acc_empty[b]), aph, a.wait_limit)) {
                    atomicExch(&s_fail, 1);
                    break;
                }
                tcx::fence_after_sync();
                const uint32_t acc = tmem + (uint32_t)(b * a.acc_cols);
                const uint32_t idesc = tcx::idesc_tf32(STC_M, np);
                const uint32_t blo = (uint32_t)(np * KC * 4) >> 4;   // from T's hi block to its lo block
                for (int c = 0; c < nkc; ++c) {
                    if (!ready && (!mbar_wait(smem_u32(&full_bar[s]), ph, a.wait_limit) ||
                                   !mbar_wait(smem_u32(&b_bar[s]), ph, a.wait_limit))) {
                        atomicExch(&s_fail, 1);
                        fail = true;
                        break;
                    }
                    const int s1 = s + 1 == nst ? 0 : s + 1;
                    const uint32_t p1 = s1 == 0 ? ph ^ 1 : ph;
                    ready = peek_stage(s1, p1);
                    tcx::fence_after_sync();
#pragma unroll
                    for (int ks = 0; ks < KC / 8; ++ks) {
                        const uint32_t aH = a0 + dof + ((ks * 2 * L::LBO) >> 4), bH = b0 + dof + ((ks * 2 * tcx::LBO) >> 4);
                        mma_tf32(acc, desc(aH, ahi), desc(bH, bhi), idesc, ks == 0 ? (uint32_t)c : 1u);
                        mma_tf32(acc, desc(aH, ahi), desc(bH + blo, bhi), idesc, 1u);
                        mma_tf32(acc, desc(aH + ((L::PLANE * 4) >> 4), ahi), desc(bH, bhi), idesc, 1u);
                    }
                    mma_commit(&empty_bar[s]);
                    dof = s1 == 0 ? 0u : dof + dstep;
                    s = s1;
                    ph = p1;
                }
                if (iready) {   // (read under the test's branch: never before its outcome is known)
                    nN = s_item[r1].N;
                    nK = s_item[r1].K;
                }
                if (!fail) mma_commit(&acc_full[b]);
                b = b1;
                aph = ap1;
            }
            // completion of every MMA issued above (also on failure)
            mma_commit(&done_bar);
        }
        __syncwarp();
    } else if (warp < STC_IDX0) {
        // ---------------- epilogue --------------------------------------------
        const int ew = warp - L::PRODW - 2, quad = warp & 3;
        float* sg = stage0 + (size_t)nst * a.stage_floats + ew * 32 * STC_SG;
        int b = 0;
        uint32_t aph = 0;
        for (int it = 0; it < nmine; ++it) {
            const int r = it % STC_RING;
            const bool known = mbar_test(smem_u32(&idx_full[r]), (it / STC_RING) & 1);
            const bool ok = mbar_wait(smem_u32(&acc_full[b]), aph, a.wait_limit) && (known || item_wait(it));
            if (!__all_sync(0xffffffffu, ok)) {   // the whole warp goes on or none of it
                atomicExch(&s_fail, 1);
                break;
            }
            tcx::fence_after_sync();
            stc_epilogue<PASS>(a, s_item[r], s_pos[r], s_dir[r], tmem + (uint32_t)(b * a.acc_cols), quad,
                               (ew / 4 + it) % L::SHARES, lane, sg);
            // this warp's share of the accumulator is read
            tcx::fence_before_sync();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&acc_empty[b]);
                mbar_arrive(&idx_empty[r]);
            }
            if (++b == a.nacc) {
                b = 0;
                aph ^= 1;
            }
        }
    } else {
        // ---------------- items, up to STC_RING ahead; two warps in turn -----
        auto slots_of = [&](const StcItem& tl, int64_t (&o)[2], int32_t (&d)[2]) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int j = tl.s0 + min(q * 32 + lane, tl.ns - 1);
                d[q] = 0;
                if (PASS == ST_C) {
                    o[q] = __ldg(a.cidx + j) + tl.uoff;
                } else {
                    o[q] = (PASS == ST_R ? __ldg(&a.slots[j].src_off) : __ldg(&a.slots[j].dst_off)) + tl.rhs * a.rstride;
                    d[q] = __ldg(&a.slots[j].dir);
                }
            }
        };
        // every CTA starts elsewhere in its share (equal weights lie together):
        // targets of different degrees at a time in B's adds
        const int rot = (int)((int64_t)blockIdx.x * nmine / gridDim.x);
        auto item_of = [&](int it) {
            it += rot;
            const int i = (int)blockIdx.x + (it < nmine ? it : it - nmine) * (int)gridDim.x;
            // the right-hand sides of an item one after the other: they share T
            StcItem tl = a.items[i / a.nrhs];
            tl.rhs = i % a.nrhs;
            tl.uoff = tl.rhs * a.ustride;
            return tl;
        };
        StcItem cur, nxt;
        int64_t o[2], on[2];
        int32_t d[2], dn[2];
        int it = warp - STC_IDX0;
        if (it < nmine) {
            cur = item_of(it);
            slots_of(cur, o, d);
        }
        if (it + STC_IDXW < nmine) nxt = item_of(it + STC_IDXW);
        for (; it < nmine; it += STC_IDXW) {
            const int r = it % STC_RING;
            if (it + STC_IDXW < nmine) slots_of(nxt, on, dn);
            const bool ok = it < STC_RING || mbar_wait(smem_u32(&idx_empty[r]), (it / STC_RING - 1) & 1, a.wait_limit);
            if (!__all_sync(0xffffffffu, ok)) {
                atomicExch(&s_fail, 1);
                break;
            }
            cur.uni = 0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (PASS == ST_R) {   // groups of 16 slots with one direction
                    const uint32_t eq = __ballot_sync(0xffffffffu, d[q] == __shfl_sync(0xffffffffu, d[q], lane & 16));
                    cur.uni |= (((eq & 0xffffu) == 0xffffu ? 1 : 0) | (eq >> 16 == 0xffffu ? 2 : 0)) << (2 * q);
                }
                s_pos[r][q * 32 + lane] = o[q];
                s_dir[r][q * 32 + lane] = d[q];
                o[q] = on[q];
                d[q] = dn[q];
            }
            if (lane == 0) s_item[r] = cur;
            __syncwarp();
            if (lane == 0) mbar_arrive(&idx_full[r]);
            cur = nxt;
            if (it + 2 * STC_IDXW < nmine) nxt = item_of(it + 2 * STC_IDXW);
        }
    }

    const bool done = mbar_wait(smem_u32(&done_bar), 0, DRAIN_LIMIT);
    __syncthreads();
    if ((!done || s_fail) && tid == 0) atomicExch(a.err, 1);
    tcx::fence_after_sync();
    if (warp == 0)
        tcx::tmem_dealloc(tmem, a.nacc * a.acc_cols);
}

// rotation (0) and back-rotation (1); coaxial pass
template <int PASS>
__global__ void __launch_bounds__(STC_THREADS, 1) k_stg_tc(const StcArgs a) {
    stc_body<PASS>(a);
}
__global__ void __launch_bounds__(STC_THREADS, 1) k_stc_coax(const StcArgs a) { stc_body<ST_C>(a); }

// Pre-split real-form coaxial blocks (grid: one CTA per block).
__global__ void k_stc_coax_tables(const StcCBlock* __restrict__ blocks, const cd* __restrict__ coax,
                                  float* __restrict__ out) {
    const StcCBlock b = blocks[blockIdx.x];
    const int np = stc_pad16(2 * b.nr), kp = ((2 * b.K + KC - 1) / KC) * KC;
    float* T = out + b.toff;
    for (int e = threadIdx.x; e < np * kp; e += blockDim.x) {
        const int j = e / kp, k2 = e % kp;   // row (i, c'), K index (k, c)
        const int i = j >> 1, cp = j & 1, k = k2 >> 1, c = k2 & 1;
        double v = 0.0;
        if (i < b.nr && k < b.K) {
            const cd C = coax[b.cs_off + ((int64_t)b.am * b.pc + b.am + b.r0 + i) * b.pc + b.am + k];
            v = cp == 0 ? (c == 0 ? C.re : -C.im) : (c == 0 ? C.im : C.re);
        }
        const int64_t o = (int64_t)(k2 / KC) * 2 * np * KC + (canon(j, k2 % KC) >> 2);
        const float h = tf32_hi((float)v);
        T[o] = h;
        T[o + (int64_t)np * KC] = (float)(v - (double)h);
    }
}

// Pre-split canonical table blocks of every group (grid: degree n, group g)
// from the FP64 real factors d^n of the group's representative direction:
// the folded R and B tables of rcr_staged.cu, zero-padded to whole
// 16 x 16 core blocks.
__global__ void k_stc_tables(const double* __restrict__ rotd, int64_t per_dir, const int* __restrict__ rep_dirs,
                             const int64_t* __restrict__ toff, int64_t tper, float* __restrict__ out) {
    const int n = blockIdx.x, g = blockIdx.y;
    const int w = 2 * n + 1;
    const double* Dc = rotd + (int64_t)rep_dirs[g] * per_dir + rot_off(n) + (int64_t)n * w + n;   // d_{0,0}
    for (int part = 0; part < 2; ++part) {
        const int nb = n + 1 - part;
        if (nb <= 0) continue;
        const int np = stc_pad16(nb);
        float* Rt = out + (int64_t)g * 2 * tper + toff[2 * n + part];
        float* Bt = Rt + tper;
        for (int e = threadIdx.x; e < np * np; e += blockDim.x) {
            const int r = e / np, k = e % np;   // block row, K index
            double rv = 0.0, bv = 0.0;
            if (r < nb && k < nb) {
                const int a = r + part, b = k + part;
                // R: row mu = a, column m = b;  B: row m' = a, column mu = b
                if (part == 0) {
                    rv = b == 0 ? 2.0 * Dc[(int64_t)a * w] : Dc[(int64_t)a * w + b] + Dc[(int64_t)a * w - b];
                    bv = b == 0 ? Dc[a] : Dc[(int64_t)b * w + a] + Dc[-(int64_t)b * w + a];
                } else {
                    rv = Dc[(int64_t)a * w + b] - Dc[(int64_t)a * w - b];
                    bv = Dc[(int64_t)b * w + a] - Dc[-(int64_t)b * w + a];
                }
            }
            const int64_t o = (int64_t)(k / KC) * 2 * np * KC + (canon(r, k % KC) >> 2);
            const float rh = tf32_hi((float)rv), bh = tf32_hi((float)bv);
            Rt[o] = rh;
            Rt[o + (int64_t)np * KC] = (float)(rv - (double)rh);
            Bt[o] = bh;
            Bt[o + (int64_t)np * KC] = (float)(bv - (double)bh);
        }
    }
}

}  // namespace

namespace stg {

int64_t fb_stc_layout(int P, std::vector<int64_t>& toff) {
    toff.assign((size_t)2 * std::max(P, 1), 0);
    int64_t off = 0;
    for (int n = 0; n < P; ++n)
        for (int part = 0; part < 2; ++part) {
            const int nb = n + 1 - part;
            toff[(size_t)2 * n + part] = off;
            if (nb <= 0) continue;
            const int64_t np = stc_pad16(nb);
            off += 2 * np * np;   // hi and lo planes of np rows x np K values
        }
    return off;
}

void fb_stc_group_items(int g, int g0, int g1, int nmax, int pass, int p_in, std::vector<StcItem>& out) {
    std::vector<int64_t> toff;
    fb_stc_layout(nmax, toff);
    for (int s0 = g0; s0 < g1; s0 += STC_SLOTS)
        for (int n = 0; n < nmax; ++n)
            for (int part = 0; part < 2; ++part) {
                int N, K;
                stc_dims(pass, n, part, p_in, N, K);
                if (N > 0 && K > 0)
                    out.push_back(StcItem{toff[2 * n + part], s0, std::min(STC_SLOTS, g1 - s0), n, part, N, K, g, 0, 0, 0});
            }
}

void fb_stc_coax_set(int c0, int ns, int64_t cs_off, int pc, int p_in, int p_out, std::vector<StcItem>& items,
                     std::vector<StcCBlock>& blocks, int64_t* tfloats) {
    for (int am = 0; am < std::min(p_in, p_out); ++am) {
        const int M = p_out - am, K = p_in - am;
        for (int r0 = 0; r0 < M; r0 += STC_CROWS) {
            const int nr = std::min(STC_CROWS, M - r0);
            const int np = stc_pad16(2 * nr), kp = ((2 * K + KC - 1) / KC) * KC;
            blocks.push_back(StcCBlock{cs_off, *tfloats, pc, am, r0, nr, K, 0});
            for (int s0 = 0; s0 < ns; s0 += STC_SLOTS)
                items.push_back(
                    StcItem{*tfloats, c0 + s0, std::min(STC_SLOTS, ns - s0), am, r0, 2 * nr, 2 * K, 0, 0, 0, 0});
            *tfloats += (int64_t)2 * np * kp;
        }
    }
}

// the heaviest items first, in equal shares of every weight to the CTAs
void fb_stc_sort(std::vector<StcItem>& items) {
    std::stable_sort(items.begin(), items.end(), [](const StcItem& x, const StcItem& y) {
        auto w = [](const StcItem& t) { return (int64_t)(stc_pad16(t.N) + 64) * ((t.K + KC - 1) / KC); };
        return w(x) > w(y);
    });
}

fb_status fb_stc_coax_tables(const StcCBlock* blocks, int nblocks, const cd* coax64, float* out, cudaStream_t s) {
    if (nblocks == 0) return FB_OK;
    k_stc_coax_tables<<<(unsigned)nblocks, 256, 0, s>>>(blocks, coax64, out);
    FB_LAUNCH_CHECK();
    fb_count_launch();
    return FB_OK;
}

fb_status fb_stc_run(int pass, const StcItem* items, int nitems, int ncol_max, const float* tab, int64_t tper,
                     const StgSlot* slots, const int32_t* cidx, const cf* X, cf* out, int64_t ns, const cf* rph,
                     int prot, int* err, cudaStream_t s, int nrhs, int64_t rstride, int64_t ustride) {
    if (nitems == 0) return FB_OK;
    const int npmax = stc_pad16(ncol_max);
    if ((int64_t)nitems * nrhs > INT32_MAX / 2) return fb_fail(FB_ERR_ARG, "tensor-core staged RCR: too many items");
    if (npmax > STC_COLS) return fb_fail(FB_ERR_ARG, "tensor-core staged RCR: order above 256");
    StcArgs a;
    a.items = items;
    a.nitems = nitems;
    a.nrhs = nrhs;
    a.rstride = rstride;
    a.ustride = ustride;
    a.tab = tab;
    a.tper = tper;
    a.slots = slots;
    a.cidx = cidx;
    a.X = X;
    a.out = out;
    a.rph = rph;
    a.err = err;
    a.wait_limit = fb_tc_wait_limit();
    a.ns = ns;
    a.prot = prot;
    const int plane = pass == ST_R ? StcLayout<ST_R>::PLANE : StcLayout<ST_B>::PLANE;
    a.stage_floats = 2 * plane + 2 * npmax * KC;
    const size_t stage = a.stage_floats * sizeof(float);
    const size_t fixed = 1024 + (pass == ST_B ? StcLayout<ST_B>::EPIW * 32 * STC_SG * sizeof(float) : 0);
    a.nst = (int)std::min<size_t>(STC_STAGES, (STC_SMEM_MAX - fixed) / stage);
    // a warp that stores every PERIOD-th chunk tells a stage's uses apart by
    // their parity: at least as many stages
    const int period = pass == ST_R   ? StcLayout<ST_R>::PERIOD
                       : pass == ST_B ? StcLayout<ST_B>::PERIOD
                                      : StcLayout<ST_C>::PERIOD;
    if (a.nst < period) return fb_fail(FB_ERR_STATE, "tensor-core staged RCR: too few pipeline stages");
    a.acc_cols = 32;
    while (a.acc_cols < npmax) a.acc_cols *= 2;
    a.nacc = std::min(STC_ACC, 2 * STC_COLS / a.acc_cols);
    a.inject_stall = fb_tc_inject_stall();
    const size_t smem = std::max(STC_SMEM_MIN, a.nst * stage + fixed);
    const void* fn = pass == ST_R   ? (const void*)k_stg_tc<ST_R>
                     : pass == ST_B ? (const void*)k_stg_tc<ST_B>
                                    : (const void*)k_stc_coax;
    FB_CHECK(fb_smem_cap(fn, smem));
    int dev = 0, sms = 0;
    FB_CUDA(cudaGetDevice(&dev));
    FB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const unsigned grid = (unsigned)std::min<int64_t>(sms, (int64_t)nitems * nrhs);
    if (pass == ST_R)
        k_stg_tc<ST_R><<<grid, STC_THREADS, smem, s>>>(a);
    else if (pass == ST_B)
        k_stg_tc<ST_B><<<grid, STC_THREADS, smem, s>>>(a);
    else
        k_stc_coax<<<grid, STC_THREADS, smem, s>>>(a);
    FB_LAUNCH_CHECK();
    fb_count_launch();
    return FB_OK;
}

}  // namespace stg

// Pre-split canonical rotation tables of the tensor-core staged passes for
// every polar-angle group of a mixed operator (built once, on first use).
fb_status fb_stc_tables(fb_op* op, cudaStream_t s) {
    if (op->stc_tab) return FB_OK;
    if (op->prec != FB_PREC_MIXED_FMM)
        return fb_fail(FB_ERR_ARG, "tensor-core staged RCR applies to mixed operators");
    const int ng = (int)op->theta_dirs.size();
    const int P = op->Prot;
    if (ng == 0 || P < 1) return fb_fail(FB_ERR_STATE, "tensor-core staged RCR: no rotation groups");
    std::vector<int64_t> toff;
    const int64_t tper = stg::fb_stc_layout(P, toff);
    if (!op->stc_err) {
        FB_CHECK(dalloc(&op->stc_err, 1));
        FB_CUDA(cudaMemsetAsync(op->stc_err, 0, sizeof(int), s));
    }
    int* d_dirs = nullptr;
    int64_t* d_off = nullptr;
    fb_status st;
    if ((st = dalloc(&d_dirs, (size_t)ng)) || (st = dalloc(&d_off, toff.size())) ||
        (st = dalloc(&op->stc_tab, (size_t)ng * 2 * tper))) {
        dfree(d_dirs);
        dfree(d_off);
        return st;
    }
    FB_CUDA(cudaMemcpyAsync(d_dirs, op->theta_dirs.data(), sizeof(int) * ng, cudaMemcpyHostToDevice, s));
    FB_CUDA(cudaMemcpyAsync(d_off, toff.data(), sizeof(int64_t) * toff.size(), cudaMemcpyHostToDevice, s));
    k_stc_tables<<<dim3(P, ng), 256, 0, s>>>(op->rotd64, op->per_dir, d_dirs, d_off, tper, op->stc_tab);
    cudaError_t e = cudaStreamSynchronize(s);
    dfree(d_dirs);
    dfree(d_off);
    if (e != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("tensor-core rotation tables: ") + cudaGetErrorString(e));
    op->stc_per = tper;
    fb_count_launch();
    return FB_OK;
}
