// Rotation - coaxial translation - back-rotation (Sec. 3.3) on CUDA cores,
// one tile of box pairs per CTA with every step in shared memory.
//
// Columns.  All box pairs of one level pass whose translation vectors share
// the polar angle theta and the length |t| are one class: they use the same
// real rotation factors d^n(theta) and the same coaxial blocks, and differ
// only in the phase e^{i m phi}, which is applied per column while loading
// and storing (up to 8 translation vectors of the 316 M2L vectors per
// class, 4 of the 8 octants of M2M / L2L).  A tile takes 2^lcw (at most 32)
// columns of one class, and the lanes of a warp are its columns: every lane
// runs the same loop with the same table entry, so a table entry is one
// broadcast load for 2^lcw columns x several rows, no lane idles on a
// shorter degree, and each shared-memory operand is read by consecutive
// lanes.  With 2^lcw < 32 the remaining lane bits split the rows.
//
// Folding (half the multiplications of u = d x): with the phased input
// x_m = e^{i m phi} src_m and s_m = x_m + x_{-m}, t_m = x_m - x_{-m} (m > 0),
// s_0 = x_0, the symmetry d^n_{-mu,-m} = d^n_{mu,m} gives
//   E_mu = u_mu + u_{-mu} = 2 d_{mu,0} s_0 + sum_{m>0} (d_{mu,m} + d_{mu,-m}) s_m   (mu = 0..n)
//   O_mu = u_mu - u_{-mu} =                  sum_{m>0} (d_{mu,m} - d_{mu,-m}) t_m   (mu = 1..n)
// the coaxial blocks, which depend on |m| only, map E to E and O to O, and
//   Y+_{m'} = y_{m'} + y_{-m'} = d_{0,m'} E_0 + sum_{mu>0} (d_{mu,m'} + d_{-mu,m'}) E_mu
//   Y-_{m'} = y_{m'} - y_{-m'} =               sum_{mu>0} (d_{mu,m'} - d_{-mu,m'}) O_mu
// and y_{+-m'} = (Y+ +- Y-)/2, e^{-+ i m' phi} applied, scatter-added into the
// target (atomic adds: tiles share targets).  Folded layout of degree n
// within a column: [n^2 + j], j = 0..n even part, j = n+1..2n odd part.
//
// In place.  Each block (degree and part of a rotation, order and part of
// the coaxial step) reads and writes its own entries only, so one warp takes
// a whole block, holds its output rows in registers and writes them back
// over the inputs: one buffer per column instead of two, which is what lets
// 32 columns of 144 complex double-FP32 values (order 12) and three CTAs
// share an SM.
//
// Bound: the FP32 pipe in double-FP32 (12 operations per multiply-add), the
// FP64 pipe in FP64 (2 multiply-adds per clock and SM), instruction issue in
// FP32 (address and load / store steps beside few FMAs).  Measured on the
// L-shaped room at 2 kHz (567,592 elements), M2L of level 7 (order 12,
// 952,630 pairs), one thread per coefficient before / this form: double-FP32
// 19.7 -> 8.1-8.6 ms (its multiply-adds alone 5.3 ms, 62 % of the FP32 pipe;
// loads 1.0 ms, the 274 M FP64 atomics 1.7 ms), FP64 44.5 -> 21.1 ms, FP32
// 3.68 -> 1.78 ms (multiply-adds 1.05 ms).
//
// Double-FP32: the load and store steps (phases, x_m +- x_-m, y_+-m') run in
// FP64 and round once, as in the staged passes; in 48 bits they added 11 % to
// the error against FP64 for 1 % of a product (L-room 29.4 against 29.8 ms).
#include <algorithm>
#include <cstdlib>
#include <map>
#include <tuple>
#include <type_traits>

#include "common.cuh"
#include "rcr_staged.cuh"

using stg::StgSlot;

// A task's pairs as slots of its class.
struct RcrSlotTask {
    int64_t pair_off, src_base, dst_base;
    int32_t npairs, slot0, pin2, pout2, dir, pad;
};

namespace {

constexpr int RT_THREADS = 768;    // resident per SM: one CTA of 24 warps, two of 12 or three of 8
// output rows a lane holds at most: 12 in FP32, 8 in the 16-byte types (more
// accumulators do not fit 24 warps' registers)
template <class R> struct RtRows { static constexpr int value = sizeof(R) == 4 ? 12 : 8; };
constexpr int RT_SLACK = 512;      // spare 16-byte vectors at the end of a table (12 rows x 32 lanes)

// padded row count of a table column: whole 16-byte vectors of E-byte entries
template <int E>
__host__ __device__ __forceinline__ int rt_pad(int s) {
    constexpr int W = E >= 16 ? 1 : 16 / E;
    return (s + W - 1) / W * W;
}
// entries of the table blocks of sizes 1..s (block of size s: s columns of
// rt_pad(s) rows)
template <int E>
__host__ __device__ __forceinline__ int rt_sum(int s) {
    if (s <= 0) return 0;
    int f = s * (s + 1) * (2 * s + 1) / 6;
    if (E == 8) f += ((s + 1) / 2) * ((s + 1) / 2);
    if (E == 4) {
        const int q = s / 4, r = s % 4;
        f += 12 * q * (q - 1) + 10 * q;
        if (r >= 1) f += 3 * (4 * q + 1);
        if (r >= 2) f += 2 * (4 * q + 2);
        if (r >= 3) f += 4 * q + 3;
    }
    return f;
}
// start of the folded block (degree n, part) in a rotation table: blocks of
// n + 1 (even) and n (odd) rows
template <int E>
__host__ __device__ __forceinline__ int rt_rot_off(int n, int part) {
    return rt_sum<E>(n + part) + rt_sum<E>(n - 1);
}

// ------------------------------------------------------ double-FP32 steps ----
// FP64 -> double-FP32 by integer steps (conversion instructions run at the
// FP64 pipe's rate, a 64th of the integer pipe's): hi is the rounded upper
// part, lo the 29 remaining bits as a signed count of 2^(E - 52).  What lies
// outside [2^-126, 2^127) and is not zero (rare) takes the instructions, which
// keep subnormals.
__device__ __forceinline__ df df_from_fast(double v) {
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const uint32_t e = (h >> 20) & 0x7ff;
    const uint32_t low = l & 0x1fffffffu, up = low >> 28, sign = h & 0x80000000u;
    uint32_t mag = (((h & 0x7fffffffu) << 3) | (l >> 29)) - 0xC0000000u + up;   // rebias 1023 -> 127 (mod 2^32)
    const int r = (int)low - (int)(up << 29);
    float lo = (__int2float_rn(r) * 2.220446049250313e-16f) * __uint_as_float((e - 896) << 23);
    if (e - 897 >= 253u) {
        if ((h & 0x7fffffffu) | l) return df_from(v);
        mag = 0;
        lo = 0.f;
    }
    return df(__uint_as_float(mag | sign), __uint_as_float(__float_as_uint(lo) ^ sign));
}
// double-FP32 -> FP64 the same way: the normalised low part is a signed
// count of ulps added to the significand of the high part (subnormal, infinite
// and NaN: the instructions).
__device__ __forceinline__ double df_to_fast(df a) {
    const float s = __fadd_rn(a.hi, a.lo);
    const float bb = __fsub_rn(s, a.hi);
    const float t = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(a.lo, bb));
    const uint32_t b = __float_as_uint(s), mag = b & 0x7fffffffu;
    const uint32_t e = mag >> 23;
    // t 2^(52 - E), E = e - 127, in two steps where the factor passes 2^127
    const bool small = e < 100;
    int q = __float2int_rn((small ? t * 1.152921504606847e18f : t) * __uint_as_float(((small ? 246u : 306u) - e) << 23));
    if (b >> 31) q = -q;
    if ((mag & 0x7fffffu) == 0 && q < 0) q *= 2;   // below a power of two the ulps are half as large
    uint32_t hi = (mag >> 3) + (896u << 20), lo = mag << 29;
    if (e - 1 >= 254u) {
        if (mag) return df_to(a);
        hi = lo = 0, q = 0;   // zero
    }
    const uint64_t w = (((uint64_t)hi << 32) | lo) + (uint64_t)(int64_t)q;
    return __longlong_as_double((long long)(w | ((uint64_t)(b & 0x80000000u) << 32)));
}

// conversions between the expansions' type O and the arithmetic type R: the
// load and store steps (phases, sums and differences) run in O
template <class R, class O>
__device__ __forceinline__ cx<R> rt_in(const cx<O>& a) { return a; }
template <>
__device__ __forceinline__ cx<df> rt_in<df, double>(const cd& a) { return mk(df_from_fast(a.re), df_from_fast(a.im)); }
template <class O, class R>
__device__ __forceinline__ cx<O> rt_out(const cx<R>& a) { return a; }
template <>
__device__ __forceinline__ cd rt_out<double, df>(const cx<df>& a) { return mk(df_to_fast(a.re), df_to_fast(a.im)); }

template <class R>
__device__ __forceinline__ cx<R> rt_conj(const cx<R>& a) { return mk(a.re, -a.im); }
__device__ __forceinline__ float rt_half(float a) { return 0.5f * a; }
__device__ __forceinline__ double rt_half(double a) { return 0.5 * a; }
__device__ __forceinline__ df rt_half(df a) { return df(0.5f * a.hi, 0.5f * a.lo); }

__device__ __forceinline__ void rt_atomic(cf* d, const cf& v) {
    atomicAdd(reinterpret_cast<float2*>(d), make_float2(v.re, v.im));
}
__device__ __forceinline__ void rt_atomic(cd* d, const cd& v) {
    atomicAdd(&d->re, v.re);
    atomicAdd(&d->im, v.im);
}

// acc += a x, a real or complex
template <class R>
__device__ __forceinline__ void rt_mac(cx<R>& acc, const R& a, const cx<R>& x) {
    acc.re = fma(a, x.re, acc.re);
    acc.im = fma(a, x.im, acc.im);
}
template <class R>
__device__ __forceinline__ void rt_mac(cx<R>& acc, const cx<R>& a, const cx<R>& x) {
    acc.re = fma(a.re, x.re, acc.re);
    acc.re = fma(-a.im, x.im, acc.re);
    acc.im = fma(a.re, x.im, acc.im);
    acc.im = fma(a.im, x.re, acc.im);
}

// ------------------------------------------------------------ one block ----
// rows r < S of  out_r = sum_{k < K} T[k][r] x_k  for this lane's column, in
// place: x_k and out_k at entry o_k, o_0 = base, o_{k+1} = o_k + step_k,
// step_{k+1} = step_k + dstep.  T: K columns of ld rows (16-byte aligned);
// the lane takes the 16-byte row chunks sub, sub + nsub, ... (NCH of them;
// ONE: nsub = 1).  Chunks past the block read the entries that follow it
// (the tables end with RT_SLACK spare vectors); their results are dropped.
template <int NCH, bool ONE, class R, class TE>
__device__ __forceinline__ void rt_block(cx<R>* col, int cwp, int base, int step, int dstep, const TE* T, int ld,
                                         int S, int K, int sub, int nsub) {
    constexpr int W = sizeof(TE) >= 16 ? 1 : 16 / sizeof(TE);
    struct alignas(16) Vec { TE v[W]; };
    cx<R> acc[NCH * W];
#pragma unroll
    for (int i = 0; i < NCH * W; ++i) acc[i] = mk<R>(R(0), R(0));
    // the block's table lines on their way to L1 before the loop asks for them
    for (int o = (threadIdx.x & 31) * 128; o < K * ld * (int)sizeof(TE); o += 32 * 128)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(T) + o));
    {
        const int rs = ONE ? W : nsub * W;
        if (!ONE) T += sub * W;
        const cx<R>* x = col + base * cwp;
        int st = step;
#pragma unroll(sizeof(R) == 4 ? 4 : 1)
        for (int k = 0; k < K; ++k) {
            const cx<R> xv = *x;
            x += st * cwp;
            st += dstep;
#pragma unroll
            for (int i = 0; i < NCH; ++i) {
                const Vec a = *reinterpret_cast<const Vec*>(T + i * rs);
#pragma unroll
                for (int q = 0; q < W; ++q) rt_mac(acc[i * W + q], a.v[q], xv);
            }
            T += ld;
        }
    }
    __syncwarp();   // every lane of the column has read its inputs
    if (ONE) {   // rows 0, 1, ...: running offset
        cx<R>* o = col + base * cwp;
        int st = step * cwp;
#pragma unroll
        for (int i = 0; i < NCH * W; ++i) {
            if (i < S) *o = acc[i];
            o += st;
            st += dstep * cwp;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
#pragma unroll
            for (int q = 0; q < W; ++q) {
                const int r = (i * nsub + sub) * W + q;
                if (r < S) col[(base + r * step + dstep * (r * (r - 1) / 2)) * cwp] = acc[i * W + q];
            }
        }
    }
}
// The rows of a block rounded up to one of a few unrolled sizes: a
// double-FP32 row of a loop body is 24 (real table) or 48 instructions, and
// with a body for every size the warps of a CTA, each in a block of its own,
// run out of the instruction cache (half of all stalls at order 12).
template <class R, class TE>
__device__ __forceinline__ void rt_block_any(cx<R>* col, int cwp, int base, int step, int dstep, const TE* T, int ld,
                                             int S, int K, int sub, int lsub) {
    constexpr int W = sizeof(TE) >= 16 ? 1 : 16 / sizeof(TE);
    const int rows = (ld + (W << lsub) - 1) / (W << lsub) * W;   // per lane
#define RT_ROWS_OF(N, ONE) rt_block<((N) + W - 1) / W, ONE>(col, cwp, base, step, dstep, T, ld, S, K, sub, 1 << lsub)
    if (lsub == 0) {
        if (rows <= 4) RT_ROWS_OF(4, true);
        else if (rows <= 8) RT_ROWS_OF(8, true);
        else if constexpr (RtRows<R>::value > 8) RT_ROWS_OF(12, true);
    } else {
        if (std::is_same<R, double>::value && rows <= 2) RT_ROWS_OF(2, false);
        else if (rows <= 4) RT_ROWS_OF(4, false);
        else if (W <= 2 && rows <= 6) RT_ROWS_OF(6, false);
        else if (rows <= 8) RT_ROWS_OF(8, false);
        else if constexpr (RtRows<R>::value > 8) RT_ROWS_OF(12, false);
    }
#undef RT_ROWS_OF
}

// dynamic shared memory of a tile with which three / two CTAs share an SM
constexpr size_t RT_SMEM3 = 76032, RT_SMEM2 = 114688;

template <class R, class O>
struct RtArgs {
    const RcrClass* cls;
    const RcrColTile* tiles;
    const StgSlot* slots;
    const uint32_t* lut;     // t = n (n + 1) / 2 + m -> n | m << 16
    const R* rot;            // group g: rotation table at g * 2 per, back-rotation table at g * 2 per + per
    const cx<R>* coax;
    int64_t per;
    const cx<O>* rph;        // phases e^{i m phi} per direction
    int prot;
    const cx<O>* src;
    cx<O>* dst;
    int nrhs;
    int64_t rstride;
};


template <class R, class O>
__global__ void __launch_bounds__(RT_THREADS, 1) k_rcr(const RtArgs<R, O> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ const cx<O>* s_src[32];
    __shared__ cx<O>* s_dst[32];
    __shared__ const cx<O>* s_ph[32];   // phase of m = 0
    cx<R>* B = reinterpret_cast<cx<R>*>(smem_raw);   // [entry][column], row stride 2^lcw + 1
    const RcrColTile tl = a.tiles[blockIdx.x];
    const RcrClass cl = a.cls[tl.cls];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    const int p_in = cl.p_in, p_out = cl.p_out;
    const int cw = 1 << tl.lcw, cwp = cw + 1;
    // column b of the tile: slot (col0 + b) / nrhs, right-hand side (col0 + b) % nrhs
    if (tid < tl.ncol) {
        const int col = tl.col0 + tid, sl = col / a.nrhs;
        const int64_t ro = (int64_t)(col - sl * a.nrhs) * a.rstride;
        const StgSlot s = a.slots[cl.slot0 + sl];
        s_src[tid] = a.src + s.src_off + ro;
        s_dst[tid] = a.dst + s.dst_off + ro;
        s_ph[tid] = a.rph + (int64_t)s.dir * (2 * a.prot - 1) + (a.prot - 1);
    }
    __syncthreads();
    // load: lanes along (n, m), columns over the warps (coalesced runs of one
    // expansion; the odd row stride keeps the stores free of bank conflicts)
    const int nt = p_in * (p_in + 1) / 2;
    for (int t = lane; t < nt; t += 32) {
        const uint32_t nm = a.lut[t];
        const int n = (int)(nm & 0xffff), m = (int)(nm >> 16);
        const int c0 = n * n + n;
#pragma unroll(sizeof(R) == 4 ? 4 : 2)
        for (int b = warp; b < tl.ncol; b += nw) {
            const cx<O>* x = s_src[b] + c0;
            cx<R>* o = B + (n * n + m) * cwp + b;
            const cx<O> xp = x[m];
            if (m == 0) {
                o[0] = rt_in<R, O>(xp);
            } else {
                const cx<O> xm = x[-m], ph = s_ph[b][m];
                const cx<O> u = xp * ph, v = xm * rt_conj(ph);
                o[0] = rt_in<R, O>(u + v);
                o[n * cwp] = rt_in<R, O>(u - v);
            }
        }
    }
    __syncthreads();
    const int lsub = 5 - tl.lcw, sub = lane >> tl.lcw;
    cx<R>* col = B + (lane & (cw - 1));
    constexpr int E = sizeof(R), EC = 2 * sizeof(R);
    const R* rot = a.rot + (int64_t)cl.g * 2 * a.per;
    // blocks in order of decreasing size, dealt to the warps back and forth:
    // the j-th block of this warp
    auto block = [&](int j) { return (j >> 1) * (2 * nw) + (j & 1 ? 2 * nw - 1 - warp : warp); };
    // rotation, degrees p_in - 1 .. 0
    for (int j = 0, i = warp; i < 2 * p_in - 1; i = block(++j)) {
        const int n = p_in - 1 - (i >> 1), part = i & 1;
        const int S = n + 1 - part;
        rt_block_any(col, cwp, n * n + (part ? n + 1 : 0), 1, 0, rot + rt_rot_off<E>(n, part), rt_pad<E>(S), S, S, sub,
                     lsub);
    }
    __syncthreads();
    // coaxial step, orders 0 .. min(p_in, p_out) - 1: v_{n'} = sum_n C^m_{n' n} u_n
    const int q = min(p_in, p_out);
    for (int j = 0, i = warp; i < 2 * q - 1; i = block(++j)) {
        const int am = (i + 1) >> 1, odd = (i && !(i & 1)) ? 1 : 0;
        const int s = cl.pc - am;
        rt_block_any(col, cwp, am * am + (odd ? am : 0) + am, 2 * am + 1 + odd, 2,
                     a.coax + cl.coax_off + rt_sum<EC>(s - 1), rt_pad<EC>(s), p_out - am, p_in - am, sub, lsub);
    }
    __syncthreads();
    // back-rotation, degrees p_out - 1 .. 0, inner orders |mu| <= min(n', p_in - 1)
    const R* back = rot + a.per;
    for (int j = 0, i = warp; i < 2 * p_out - 1; i = block(++j)) {
        const int n = p_out - 1 - (i >> 1), part = i & 1;
        const int S = n + 1 - part;
        rt_block_any(col, cwp, n * n + (part ? n + 1 : 0), 1, 0, back + rt_rot_off<E>(n, part), rt_pad<E>(S), S,
                     min(S, p_in - part), sub, lsub);
    }
    __syncthreads();
    // y_{+-m'} = (Y+ +- Y-) / 2 e^{-+ i m' phi}, scatter-added
    const int nto = p_out * (p_out + 1) / 2;
    for (int t = lane; t < nto; t += 32) {
        const uint32_t nm = a.lut[t];
        const int n = (int)(nm & 0xffff), m = (int)(nm >> 16);
        const int c0 = n * n + n;
#pragma unroll(sizeof(R) == 4 ? 2 : 1)
        for (int b = warp; b < tl.ncol; b += nw) {
            const cx<R>* o = B + (n * n + m) * cwp + b;
            cx<O>* d = s_dst[b] + c0;
            cx<R> yp = o[0];
            yp = mk(rt_half(yp.re), rt_half(yp.im));
            if (m == 0) {
                rt_atomic(d, rt_out<O, R>(yp));
            } else {
                cx<R> ym = o[n * cwp];
                ym = mk(rt_half(ym.re), rt_half(ym.im));
                const cx<O> ph = s_ph[b][m], a1 = rt_out<O, R>(yp), a2 = rt_out<O, R>(ym);
                rt_atomic(d + m, (a1 + a2) * rt_conj(ph));
                rt_atomic(d - m, (a1 - a2) * ph);
            }
        }
    }
}

// ------------------------------------------------------------------ tables ----
template <class R> __device__ __forceinline__ R rt_from(double v) { return (R)v; }
template <> __device__ __forceinline__ df rt_from<df>(double v) { return df_from(v); }

// Rotation tables of every polar-angle group, degrees < P, column by column
// (grid: degree, group): R block (n, part) column m, row mu; B block column
// mu, row m'.
template <class R>
__global__ void k_rcr_rot_tables(const double* __restrict__ rotd, int64_t per_dir, const int* __restrict__ rep_dirs,
                                 int64_t per, R* __restrict__ out) {
    const int n = blockIdx.x, g = blockIdx.y, w = 2 * n + 1;
    const double* D = rotd + (int64_t)rep_dirs[g] * per_dir + stg::rot_off(n) + (int64_t)n * w + n;   // d_{0,0}
    for (int part = 0; part < 2; ++part) {
        const int S = n + 1 - part, ld = rt_pad<sizeof(R)>(S);
        R* Rt = out + (int64_t)g * 2 * per + rt_rot_off<sizeof(R)>(n, part);
        for (int e = threadIdx.x; e < S * ld; e += blockDim.x) {
            const int k = e / ld, r = e % ld;
            double rv = 0.0, bv = 0.0;
            if (r < S) {
                const int x = r + part, y = k + part;   // row, column order
                if (part == 0) {
                    rv = y == 0 ? 2.0 * D[(int64_t)x * w] : D[(int64_t)x * w + y] + D[(int64_t)x * w - y];
                    bv = y == 0 ? D[x] : D[(int64_t)y * w + x] + D[-(int64_t)y * w + x];
                } else {
                    rv = D[(int64_t)x * w + y] - D[(int64_t)x * w - y];
                    bv = D[(int64_t)y * w + x] - D[-(int64_t)y * w + x];
                }
            }
            Rt[e] = rt_from<R>(rv);
            Rt[per + e] = rt_from<R>(bv);
        }
    }
}

struct RtSet {
    int64_t in, out;   // offset of the cube C[m][n'][n], of the table
    int32_t pc, pad;
};
// Coaxial tables (grid: order, set): block of order m, column n, row n'.
template <class R>
__global__ void k_rcr_coax_tables(const RtSet* __restrict__ sets, const cd* __restrict__ coax, cx<R>* __restrict__ out) {
    const RtSet st = sets[blockIdx.y];
    const int am = blockIdx.x, pc = st.pc;
    if (am >= pc) return;
    const int s = pc - am, ld = rt_pad<2 * sizeof(R)>(s);
    cx<R>* T = out + st.out + rt_sum<2 * sizeof(R)>(s - 1);
    for (int e = threadIdx.x; e < s * ld; e += blockDim.x) {
        const int k = e / ld, r = e % ld;
        cd v = mk(0.0, 0.0);
        if (r < s) v = coax[st.in + ((int64_t)am * pc + am + r) * pc + am + k];
        T[e] = mk(rt_from<R>(v.re), rt_from<R>(v.im));
    }
}

// Slots of the tasks of a plan (grid: task, 256 pairs each).
__global__ void k_rcr_slots(const RcrSlotTask* __restrict__ tasks, const int32_t* __restrict__ src_idx,
                            const int32_t* __restrict__ dst_idx, StgSlot* __restrict__ slots) {
    const RcrSlotTask tk = tasks[blockIdx.x];
    for (int j = blockIdx.y * blockDim.x + threadIdx.x; j < tk.npairs; j += gridDim.y * blockDim.x) {
        StgSlot s;
        s.src_off = tk.src_base + (int64_t)src_idx[tk.pair_off + j] * tk.pin2;
        s.dst_off = tk.dst_base + (int64_t)dst_idx[tk.pair_off + j] * tk.pout2;
        s.dir = tk.dir;
        s.pad = 0;
        slots[tk.slot0 + j] = s;
    }
}

template <class T>
fb_status put(T** d, const std::vector<T>& h) {
    if (h.empty()) return FB_OK;
    FB_CHECK(dalloc(d, h.size()));
    FB_CUDA(cudaMemcpy(*d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice));
    return FB_OK;
}

// log2 of the columns per tile for a class of orders up to p: at most 32, no
// more than a lane's row budget (p <= 16 rows x 32 / columns) and two CTAs'
// shared memory allow (one CTA's when four columns do not fit otherwise).
int rcr_lcw(int p, size_t csize) {
    int l = 5;
    const int rows = csize == sizeof(cf) ? RtRows<float>::value : RtRows<double>::value;
    while (l > 1 && (p << l) > 32 * rows) --l;
    auto bytes = [&](int lc) { return (size_t)p * p * ((1 << lc) + 1) * csize; };
    while (l > 2 && bytes(l) > RT_SMEM2) --l;
    while (l > 0 && bytes(l) > 226 * 1024) --l;
    return l;
}

}  // namespace

// Column tiles of the classes of `set` for nrhs right-hand sides.  A launch
// that would not give every SM two tiles takes narrower ones (down to 4
// columns, 2 in the 16-byte types, the lanes then splitting the rows): such a launch is bound by the
// latency of one tile, not by throughput.
static void rcr_make_tiles(const RcrTileSet& set, size_t csize, int nrhs, std::vector<RcrColTile> (&out)[3],
                           size_t (&smem)[3]) {
    std::vector<int> lc(set.h_cls.size());
    for (size_t c = 0; c < lc.size(); ++c)
        lc[c] = rcr_lcw(std::max(set.h_cls[c].p_in, set.h_cls[c].p_out), csize);
    const int lmin = csize == sizeof(cf) ? 2 : 1;
    auto order = [&](size_t c) { return (size_t)std::max(set.h_cls[c].p_in, set.h_cls[c].p_out); };
    auto bytes = [&](size_t c) { return order(c) * order(c) * ((1 << lc[c]) + 1) * csize; };
    auto ntiles = [&](size_t c, int l) { return (int64_t)div_up((int64_t)set.h_cls[c].nslot * nrhs, (int64_t)1 << l); };
    auto group = [&](size_t c) { return bytes(c) > RT_SMEM2 ? 0 : (bytes(c) > RT_SMEM3 ? 1 : 2); };
    int shrink = 0;
    for (;; ++shrink) {
        int64_t k = 0;
        for (size_t c = 0; c < lc.size(); ++c) k += ntiles(c, std::max(std::min(lc[c], lmin), lc[c] - shrink));
        if (shrink == 4 || k >= 152) break;
    }
    for (int& l : lc) l = std::max(std::min(l, lmin), l - shrink);
    // few tiles that need a larger share than three CTAs per SM leave: narrow
    // ones run beside the others instead of in a launch of their own
    for (int g = 0; g < 2; ++g) {
        int64_t k = 0;
        for (size_t c = 0; c < lc.size(); ++c)
            if (group(c) == g) k += ntiles(c, lc[c]);
        if (k >= 4 * 152) continue;
        for (size_t c = 0; c < lc.size(); ++c) {
            if (group(c) != g) continue;
            const int l0 = lc[c];
            while (lc[c] > lmin && group(c) != 2) --lc[c];
            if (group(c) != 2) lc[c] = l0;
        }
    }
    // tiles by the CTAs per SM their shared memory allows (a launch's tiles
    // all get the largest tile's share), heaviest first for the tail
    std::vector<std::pair<int64_t, RcrColTile>> by[3];
    for (size_t c = 0; c < lc.size(); ++c) {
        const RcrClass& k = set.h_cls[c];
        const int l = lc[c], p = (int)order(c), g = group(c);
        smem[g] = std::max(smem[g], bytes(c));
        const int64_t ncol = (int64_t)k.nslot * nrhs;
        for (int64_t c0 = 0; c0 < ncol; c0 += (int64_t)1 << l)
            by[g].emplace_back(-((int64_t)p * p * p << l),
                               RcrColTile{(int32_t)c, (int32_t)c0, (int32_t)std::min<int64_t>((int64_t)1 << l, ncol - c0), l});
    }
    for (int g = 0; g < 3; ++g) {
        std::stable_sort(by[g].begin(), by[g].end(), [](const auto& x, const auto& y) { return x.first < y.first; });
        for (const auto& t : by[g]) out[g].push_back(t.second);
    }
}

void fb_rcr_tiles_free(RcrTileSet& t) {
    dfree(t.cls);
    dfree(t.slots);
    for (auto& kv : t.tiles) dfree(kv.second.tiles);
    t.tiles.clear();
    t.h_cls.clear();
}

static fb_status rcr_tiles_for(RcrTileSet& t, size_t csize, int nrhs, RcrTileSet::Tiles* out) {
    auto it = t.tiles.find(nrhs);
    if (it == t.tiles.end()) {
        std::vector<RcrColTile> h[3];
        RcrTileSet::Tiles ts;
        rcr_make_tiles(t, csize, nrhs, h, ts.smem);
        for (int g = 0; g < 3; ++g) {
            ts.ntiles[g] = (int)h[g].size();
            if (g) h[0].insert(h[0].end(), h[g].begin(), h[g].end());
        }
        FB_CHECK(put(&ts.tiles, h[0]));
        it = t.tiles.emplace(nrhs, ts).first;
    }
    *out = it->second;
    return FB_OK;
}

// Tables of the tile kernel in the type R for orders < = P (rebuilt when a
// plan asks for a larger one): rotation factors of every polar-angle group,
// and the coaxial sets of orders up to P.  The sets lie in order of size, so
// a larger P does not move the ones plans already refer to.
template <class R>
static fb_status rcr_tables(fb_op* op, RcrTables& t, int P) {
    if (t.P >= P) return FB_OK;
    if (!op->rotd64 || P > op->Prot) return fb_fail(FB_ERR_STATE, "RCR tiles: no FP64 rotation factors");
    const int ng = (int)op->theta_dirs.size();
    int64_t off = 0;
    std::vector<RtSet> sets;
    t.coax_at.clear();
    for (const auto& s : op->coax_sets) {   // (order, offset), ascending
        if (s.first > P) break;
        sets.push_back(RtSet{s.second, off, s.first, 0});
        t.coax_at[s.second] = off;
        off += rt_sum<2 * sizeof(R)>(s.first);
    }
    if (t.rot) FB_CUDA(cudaDeviceSynchronize());   // launches in flight may read the smaller tables
    dfree(t.rot);
    dfree(t.coax);
    t.P = 0;
    t.per = rt_rot_off<sizeof(R)>(P, 0);
    int* d_dirs = nullptr;
    RtSet* d_sets = nullptr;
    fb_status st;
    const size_t nrot = (size_t)ng * 2 * t.per * sizeof(R), ncoax = (size_t)off * sizeof(cx<R>);
    if ((st = dalloc((unsigned char**)&t.rot, nrot + 16 * RT_SLACK)) ||
        (st = dalloc((unsigned char**)&t.coax, ncoax + 16 * RT_SLACK)) ||
        (st = put(&d_dirs, op->theta_dirs)) || (st = put(&d_sets, sets))) {
        dfree(d_dirs);
        dfree(d_sets);
        return st;
    }
    cudaMemsetAsync((unsigned char*)t.rot + nrot, 0, 16 * RT_SLACK, cudaStreamLegacy);
    cudaMemsetAsync((unsigned char*)t.coax + ncoax, 0, 16 * RT_SLACK, cudaStreamLegacy);
    k_rcr_rot_tables<R><<<dim3(P, ng), 128, 0, cudaStreamLegacy>>>(op->rotd64, op->per_dir, d_dirs, t.per, (R*)t.rot);
    if (!sets.empty())
        k_rcr_coax_tables<R><<<dim3(P, (unsigned)sets.size()), 128, 0, cudaStreamLegacy>>>(d_sets, op->coax64, (cx<R>*)t.coax);
    const cudaError_t e = cudaStreamSynchronize(cudaStreamLegacy);
    dfree(d_dirs);
    dfree(d_sets);
    if (e != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("RCR tile tables: ") + cudaGetErrorString(e));
    if (!op->rcr_lut) {
        std::vector<uint32_t> lut;
        for (uint32_t n = 0; n < (uint32_t)op->Prot; ++n)
            for (uint32_t m = 0; m <= n; ++m) lut.push_back(n | m << 16);
        FB_CHECK(put(&op->rcr_lut, lut));
    }
    t.P = P;
    op->buf_gen++;   // captured graphs refer to the old tables
    fb_count_launch(2);
    return FB_OK;
}

// Classes, slots and tiles of the tasks of `pl` that run as tiles (want_df:
// those in double-FP32 arithmetic).
fb_status fb_rcr_tiles_build(fb_op* op, RcrPlan& pl, bool want_df) {
    RcrTileSet& ts = want_df ? pl.df_tiles : pl.tiles;
    std::map<std::tuple<int64_t, int64_t, int64_t, int, int, int>, std::vector<int>> classes;
    int P = 0;
    for (int i = 0; i < (int)pl.h_tasks.size(); ++i) {
        const RcrTask& tk = pl.h_tasks[i];
        if (fb_stg_staged(tk) || (tk.staged == 4) != want_df || tk.npairs == 0) continue;
        const int dir = (int)(tk.rot_off / op->per_dir);
        classes[std::make_tuple(tk.src_base, tk.dst_base, tk.coax_off, tk.p_in, tk.p_out, op->theta_slot.at(dir))]
            .push_back(i);
        P = std::max(P, (int)tk.pc);
    }
    if (classes.empty()) return FB_OK;
    RcrTables& tab = want_df ? op->rcr_df : op->rcr_tab;
    if (want_df) FB_CHECK(rcr_tables<df>(op, tab, P));
    else if (pl.csize == sizeof(cf)) FB_CHECK(rcr_tables<float>(op, tab, P));
    else FB_CHECK(rcr_tables<double>(op, tab, P));
    std::vector<RcrSlotTask> st;
    int64_t nslot = 0;
    int maxpairs = 1;
    for (const auto& kv : classes) {
        const RcrTask& t0 = pl.h_tasks[kv.second[0]];
        const auto at = tab.coax_at.find(t0.coax_off);
        if (at == tab.coax_at.end()) return fb_fail(FB_ERR_STATE, "RCR tiles: unknown coaxial set");
        RcrClass c;
        c.slot0 = (int32_t)nslot;
        c.p_in = t0.p_in;
        c.p_out = t0.p_out;
        c.g = std::get<5>(kv.first);
        c.pc = t0.pc;
        c.coax_off = at->second;
        for (int i : kv.second) {
            const RcrTask& tk = pl.h_tasks[i];
            st.push_back(RcrSlotTask{tk.pair_off, tk.src_base, tk.dst_base, tk.npairs, (int32_t)nslot,
                                     tk.p_in * tk.p_in, tk.p_out * tk.p_out, (int32_t)(tk.rot_off / op->per_dir), 0});
            nslot += tk.npairs;
            maxpairs = std::max(maxpairs, (int)tk.npairs);
        }
        c.nslot = (int32_t)(nslot - c.slot0);
        ts.h_cls.push_back(c);
    }
    if (nslot > (int64_t)1 << 30) return fb_fail(FB_ERR_ARG, "RCR tiles: too many box pairs");
    RcrSlotTask* d_st = nullptr;
    fb_status s;
    if ((s = dalloc(&ts.slots, (size_t)nslot)) || (s = put(&ts.cls, ts.h_cls)) || (s = put(&d_st, st))) {
        dfree(d_st);
        return s;
    }
    k_rcr_slots<<<dim3((unsigned)st.size(), (unsigned)std::min(div_up(maxpairs, 256), 64)), 256, 0, cudaStreamLegacy>>>(
        d_st, pl.src_idx, pl.dst_idx, ts.slots);
    const cudaError_t e = cudaStreamSynchronize(cudaStreamLegacy);
    dfree(d_st);
    if (e != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("RCR tile slots: ") + cudaGetErrorString(e));
    fb_count_launch();
    RcrTileSet::Tiles one;
    return rcr_tiles_for(ts, pl.csize, 1, &one);
}

template <class R, class O>
static fb_status rcr_tiles_run(const fb_op* op, RcrTileSet& ts, const RcrTables& tab, const cx<O>* rph, const cx<O>* src,
                               cx<O>* dst, cudaStream_t s, int nrhs, int64_t rstride) {
    if (ts.h_cls.empty()) return FB_OK;
    RcrTileSet::Tiles t;
    FB_CHECK(rcr_tiles_for(ts, sizeof(cx<R>), nrhs, &t));
    if (!tab.rot || !tab.coax || !op->rcr_lut) return fb_fail(FB_ERR_STATE, "RCR tiles: tables missing");
    RtArgs<R, O> a;
    a.cls = ts.cls;
    a.slots = ts.slots;
    a.lut = op->rcr_lut;
    a.rot = (const R*)tab.rot;
    a.coax = (const cx<R>*)tab.coax;
    a.per = tab.per;
    a.rph = rph;
    a.prot = op->Prot;
    a.src = src;
    a.dst = dst;
    a.nrhs = nrhs;
    a.rstride = rstride;
    a.tiles = t.tiles;
    for (int g = 0; g < 3; a.tiles += t.ntiles[g], ++g) {
        if (!t.ntiles[g]) continue;
        FB_CHECK(fb_smem_cap((const void*)k_rcr<R, O>, t.smem[g]));
        k_rcr<R, O><<<(unsigned)t.ntiles[g], RT_THREADS / (g + 1), t.smem[g], s>>>(a);
        FB_LAUNCH_CHECK();
        fb_count_launch();
    }
    return FB_OK;
}

// The tiles of a plan on nrhs sets of expansions (precision of the operator).
fb_status fb_rcr_tiles_run_f(const fb_op* op, RcrPlan& pl, const cf* src, cf* dst, cudaStream_t s, int nrhs,
                             int64_t rstride) {
    return rcr_tiles_run<float, float>(op, pl.tiles, op->rcr_tab, op->rph32, src, dst, s, nrhs, rstride);
}
fb_status fb_rcr_tiles_run_d(const fb_op* op, RcrPlan& pl, const cd* src, cd* dst, cudaStream_t s, int nrhs,
                             int64_t rstride) {
    FB_CHECK((rcr_tiles_run<double, double>(op, pl.tiles, op->rcr_tab, op->rph64, src, dst, s, nrhs, rstride)));
    return rcr_tiles_run<df, double>(op, pl.df_tiles, op->rcr_df, op->rph64, src, dst, s, nrhs, rstride);
}
