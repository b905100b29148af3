// FMM operator setup, all in FP64 on the device (Sec. 3.3):
//   near-field entries of touching leaves (closed-form singular parts),
//   per-leaf P2M / L2P operators, coaxial coefficients by the recursions of
//   Sec. 3.3.1, rotation blocks, and the composed RCR translation matrices
//   (rotation, coaxial translation, back-rotation) for M2M, M2L and L2L.
#include <algorithm>
#include <cmath>
#include <map>
#include <numeric>

#include "sph.cuh"

int fb_order_rule(double k, double delta, double d0, int pmin) {
    double kr = k * std::sqrt(3.0) / 2.0 * delta;
    double p = std::ceil(kr + 1.8 * std::pow(d0, 2.0 / 3.0) * std::pow(kr, 1.0 / 3.0));
    return std::max(pmin, (int)p);
}

__global__ void k_d2f(const cd* a, cf* b, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = to_f(a[i]);
}

// ------------------------------------------------------------ near field ----
// One CTA per (leaf, NF_COLS columns of its block): a thread keeps one source
// element in registers and runs over the leaf's rows (coalesced stores along
// the columns).  The closed-form entries (within r_c, a tenth of the block)
// cost about ten times a far one: they are collected in shared memory and
// then shared out over all threads, instead of holding up every warp that
// has one.  FP64-pipe bound; L-room at 609 Hz (53,396 elements): 56.1 ms
// with one thread per entry and the library's sqrt, divisions and sincos,
// 12.7 ms in this form.
constexpr int NF_COLS = 128, NF_ROWS = 32;
template <int KIND>
__global__ void __launch_bounds__(NF_COLS) k_near_fill(Geom g, double k, double rc, const int32_t* __restrict__ perm,
                                                       const int32_t* __restrict__ leaf_start,
                                                       const int32_t* __restrict__ ucnt,
                                                       const int32_t* __restrict__ ulist,
                                                       const int64_t* __restrict__ nf_off,
                                                       const int32_t* __restrict__ nf_ncol, cd* __restrict__ out) {
    const int t = blockIdx.x;
    const int K = nf_ncol[t], c0 = blockIdx.y * NF_COLS;
    if (c0 >= K) return;
    __shared__ double2 s_sc[fm::SC_TAB];
    __shared__ int s_start[FB_ULIST], s_cum[FB_ULIST + 1];
    __shared__ int s_elem[NF_COLS];
    __shared__ V3 s_x[NF_ROWS], s_n[NF_ROWS];
    __shared__ int s_row[NF_ROWS];
    __shared__ uint16_t s_near[NF_ROWS * NF_COLS];
    __shared__ int s_cnt;
    const int nu = ucnt[t], tid = threadIdx.x;
    fm::sc_load(s_sc);
    if (tid == 0) {
        s_cum[0] = 0;
        for (int i = 0; i < nu; ++i) {
            const int s = ulist[(int64_t)t * FB_ULIST + i];
            s_start[i] = leaf_start[s];
            s_cum[i + 1] = s_cum[i] + (leaf_start[s + 1] - leaf_start[s]);
        }
    }
    __syncthreads();
    const int c = c0 + tid;
    const bool has = c < K;
    int64_t j = 0;
    V3 y[3], cj, nj;
    double area = 0.0;
    cd ikb = mk(0.0, 0.0);
    if (has) {
        int u = 0;
        while (s_cum[u + 1] <= c) ++u;
        j = perm[s_start[u] + (c - s_cum[u])];
        for (int q = 0; q < 3; ++q) y[q] = v3(g.gx[3 * j + q], g.gy[3 * j + q], g.gz[3 * j + q]);
        cj = v3(g.cx[j], g.cy[j], g.cz[j]);
        nj = v3(g.nx[j], g.ny[j], g.nz[j]);
        area = g.area[j];
        if (KIND == FB_OP_A) {
            const cd b = g.beta[j];
            ikb = mk(-k * b.im, k * b.re);
        }
    }
    s_elem[tid] = (int)j;
    const int r0 = leaf_start[t], nr = leaf_start[t + 1] - r0;
    cd* blk = out + nf_off[t];
    for (int rb = 0; rb < nr; rb += NF_ROWS) {
        const int rows = min(NF_ROWS, nr - rb);
        if (tid < rows) {
            const int e = perm[r0 + rb + tid];
            s_row[tid] = e;
            s_x[tid] = v3(g.cx[e], g.cy[e], g.cz[e]);
            s_n[tid] = v3(g.nx[e], g.ny[e], g.nz[e]);
        }
        if (tid == 0) s_cnt = 0;
        __syncthreads();
        if (has) {
            for (int r = 0; r < rows; ++r) {
                const V3 x = s_x[r];
                const V3 dc = x - cj;
                if (s_row[r] == (int)j || dot(dc, dc) < rc * rc) {
                    s_near[atomicAdd(&s_cnt, 1)] = (uint16_t)(r * NF_COLS + tid);
                    continue;
                }
                cd v;
                if constexpr (KIND == FB_OP_MP) {
                    v = mk(0.0, 0.0);
                    for (int q = 0; q < 3; ++q) v = v + (area / 3.0) * kernel_nn(k, y[q] - x, s_n[r], nj);
                } else {
                    v = far_entry<KIND>(s_sc, k, y, area, -dot(nj, dc), x, s_n[r], ikb);
                }
                blk[(int64_t)(rb + r) * K + c] = v;
            }
        }
        __syncthreads();
        for (int i = tid; i < s_cnt; i += NF_COLS) {
            const int r = s_near[i] / NF_COLS, cc = s_near[i] % NF_COLS;
            blk[(int64_t)(rb + r) * K + c0 + cc] = op_entry(g, KIND, s_row[r], s_elem[cc], k, rc);
        }
        __syncthreads();
    }
}

// max |z| over a complex array (non-negative doubles compare as integers)
__global__ void k_absmax(const cd* a, int64_t n, double* out) {
    double m = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double v = sqrt(abs2(a[i]));
        if (!(v <= 1e300)) v = 1e300;   // inf and NaN count as out of range
        m = fmax(m, v);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax((unsigned long long*)out, (unsigned long long)__double_as_longlong(m));
}

// ----------------------------------------------------------- P2M / L2P ----
// W[pos][nm] = ik A_j sum_q w_q [dip n_j.grad R_n^{-m}(y_q - c) + mono_j R_n^{-m}(y_q - c)]
// V[pos][nm] = R_n^m(x_i - c)  (L' : n_i . grad R_n^m(x_i - c))
//
// One CTA per group of E elements.  R_n^{-m} = conj R_n^m, so only orders
// m >= 0 are computed, and since the three Gauss points of a flat element
// share weight and normal their R are summed before the gradient:
//   A  one thread per (element, point): direction, j_n(k r), powers of
//      e^{i phi} and of sin theta;
//   B  one thread per (element, order m): the Legendre recursion up in n for
//      the points side by side, S_n^m = sum_q R_n^m into shared memory;
//   C  one thread per (element, n, m): gradient and stores of +m and -m.
// The recursion and gradient factors come from tables.  FP64-pipe bound;
// one thread per element with its arrays in global memory took 12.8 ms at
// 53,396 elements (order 12), this form 1.07 ms (and 3.3 -> 0.1 ms at 1,500
// to 6,000 elements).
struct SphTab {
    const double* leg;   // [n (n + 1) / 2 + m] (A, B) pairs of the Legendre recursion
    const double* diag;  // Q_m^m = diag[m] sin^m theta
    const double* ga;    // a_n^m at [n (M + 1) + m]
    const double* gb;    // b_n^m at [n (2 M + 1) + m + M]
    int M;
};

__global__ void k_sph_tables(int P, int M, double* __restrict__ leg, double* __restrict__ diag,
                             double* __restrict__ ga, double* __restrict__ gb) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (int i = tid; i < P * P; i += nth) {
        const int n = i / P, m = i % P;
        if (m > n) continue;
        double A = 0.0, B = 0.0;
        const double nn = (double)n * n, mm = (double)m * m;
        if (n > m) A = sqrt((4.0 * nn - 1.0) / (nn - mm));
        if (n > m + 1)
            B = sqrt(((n - 1.0) * (n - 1.0) - mm) * (2.0 * n + 1.0) / ((2.0 * n - 3.0) * (nn - mm)));
        leg[2 * (n * (n + 1) / 2 + m)] = A;
        leg[2 * (n * (n + 1) / 2 + m) + 1] = B;
    }
    for (int m = tid; m < P; m += nth) {
        double v = 0.28209479177387814347;   // 1/sqrt(4 pi)
        for (int i = 1; i <= m; ++i) v *= sqrt((2.0 * i + 1.0) / (2.0 * i));
        diag[m] = v;
    }
    const int w = 2 * M + 1;
    for (int i = tid; i < (P + 1) * w; i += nth) {
        const int n = i / w, m = i % w - M;
        gb[i] = coef_b(n, m);
        if (m >= 0) ga[n * (M + 1) + m] = coef_a(n, m);
    }
}

// bytes of shared memory per element of a group: S (unless in global memory),
// and j_n, e^{i m phi}, Q_m^m and cos theta of its four points
__host__ __device__ inline size_t p2m_elem_bytes(int Pp1, bool s_global) {
    return (s_global ? 0 : (size_t)Pp1 * (Pp1 + 1) / 2 * sizeof(cd)) + 4 * (size_t)Pp1 * 32 + 4 * 8;
}

__global__ void __launch_bounds__(128) k_p2m_l2p(Geom g, int kind, double k, int P, int64_t n, int E, SphTab tab,
                                                 const int32_t* __restrict__ perm, const int32_t* __restrict__ leaf_of,
                                                 const double* __restrict__ centers, cd* __restrict__ s_global,
                                                 cd* __restrict__ W, cd* __restrict__ V) {
    extern __shared__ __align__(16) unsigned char p2m_smem[];
    const int Pp1 = P + 1, H = Pp1 * (Pp1 + 1) / 2, tid = threadIdx.x, nth = blockDim.x, npt = 4 * E;
    cd* em = (cd*)p2m_smem;                          // [point][m]
    cd* S = s_global ? s_global + (int64_t)blockIdx.x * E * H : em + (size_t)npt * Pp1;   // [element][n (n + 1) / 2 + m]
    double* jn = (double*)(s_global ? em + (size_t)npt * Pp1 : S + (size_t)E * H);        // [point][n]
    double* dg = jn + npt * Pp1;                     // [point][m]
    double* ct = dg + npt * Pp1;                     // [point]
    const bool grad = kind != FB_OP_L && kind != FB_OP_LP;
    const bool grad_v = kind == FB_OP_LP || kind == FB_OP_MP;
    for (int64_t g0 = (int64_t)blockIdx.x * E; g0 < n; g0 += (int64_t)gridDim.x * E) {
        const int ne = (int)min((int64_t)E, n - g0);
        // ---- A: points (element, 0..2 Gauss points, 3 centroid)
        for (int pt = tid; pt < 4 * ne; pt += nth) {
            const int64_t pos = g0 + (pt >> 2), e = perm[pos];
            const int q = pt & 3, b = leaf_of[pos];
            const V3 c = v3(centers[3 * b], centers[3 * b + 1], centers[3 * b + 2]);
            const V3 y = q < 3 ? v3(g.gx[3 * e + q], g.gy[3 * e + q], g.gz[3 * e + q]) : v3(g.cx[e], g.cy[e], g.cz[e]);
            const V3 r = y - c;
            const double rho = norm(r);
            V3 u = v3(0.0, 0.0, 1.0);   // r = 0: R_0^0 = 1/sqrt(4 pi), all others vanish with j_n(0)
            if (rho > 0.0) u = v3(r.x / rho, r.y / rho, r.z / rho);
            const double st = sqrt(u.x * u.x + u.y * u.y);
            const cd e1 = st > 0.0 ? mk(u.x / st, u.y / st) : mk(1.0, 0.0);
            cd z = mk(1.0, 0.0);
            double sm = 1.0;
            for (int m = 0; m < Pp1; ++m) {
                em[pt * Pp1 + m] = z;
                dg[pt * Pp1 + m] = tab.diag[m] * sm;
                z = z * e1;
                sm *= st;
            }
            ct[pt] = u.z;
            sph_bessel_j(P, k * rho, jn + pt * Pp1);
        }
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {   // the Gauss points for W, the centroid for V
            // ---- B: S_n^m, every n of one order m
            for (int i = tid; i < ne * Pp1; i += nth) {
                const int el = i / Pp1, m = i % Pp1;
                const int p0 = 4 * el + (pass ? 3 : 0), np = pass ? 1 : 3;
                double q1[3], q2[3], x[3];
                cd z[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int pt = p0 + (q < np ? q : 0);
                    q1[q] = dg[pt * Pp1 + m];
                    q2[q] = 0.0;
                    x[q] = ct[pt];
                    z[q] = em[pt * Pp1 + m];
                }
                for (int nn = m; nn < Pp1; ++nn) {
                    const double A = tab.leg[2 * (nn * (nn + 1) / 2 + m)], B = tab.leg[2 * (nn * (nn + 1) / 2 + m) + 1];
                    cd acc = mk(0.0, 0.0);
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (q >= np) continue;
                        if (nn > m) {
                            const double t = A * x[q] * q1[q] - B * q2[q];
                            q2[q] = q1[q];
                            q1[q] = t;
                        }
                        const double v = jn[(p0 + q) * Pp1 + nn] * q1[q];
                        acc.re += v * z[q].re;
                        acc.im += v * z[q].im;
                    }
                    S[(size_t)el * H + nn * (nn + 1) / 2 + m] = acc;
                }
            }
            __syncthreads();
            // ---- C
            const int h = P * (P + 1) / 2;
            for (int i = tid; i < ne * h; i += nth) {
                const int el = i / h, t = i % h;
                int nn = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
                while (nn * (nn + 1) / 2 > t) --nn;
                while ((nn + 1) * (nn + 2) / 2 <= t) ++nn;
                const int m = t - nn * (nn + 1) / 2;
                const int64_t pos = g0 + el, e = perm[pos];
                const cd* Se = S + (size_t)el * H;
                auto get = [&](int a, int u) {   // S_a^u for u >= -1
                    if (a < 0 || abs(u) > a) return mk(0.0, 0.0);
                    const cd v = Se[a * (a + 1) / 2 + abs(u)];
                    return u < 0 ? conjg(v) : v;
                };
                const cd Sv = Se[nn * (nn + 1) / 2 + m];
                cd G = mk(0.0, 0.0);
                if (pass ? grad_v : grad) {   // n . grad S_n^m
                    const int M = tab.M;
                    auto fa = [&](int a, int u) { return a < 0 ? 0.0 : tab.ga[a * (M + 1) + u]; };
                    auto fb = [&](int a, int u) { return tab.gb[a * (2 * M + 1) + u + M]; };
                    const V3 nv = v3(g.nx[e], g.ny[e], g.nz[e]);
                    const cd dz = fa(nn - 1, m) * get(nn - 1, m) - fa(nn, m) * get(nn + 1, m);
                    const cd dp = fb(nn + 1, -m - 1) * get(nn + 1, m + 1) - fb(nn, m) * get(nn - 1, m + 1);
                    const cd dm = fb(nn + 1, m - 1) * get(nn + 1, m - 1) - fb(nn, -m) * get(nn - 1, m - 1);
                    const cd hp = mk(0.5 * nv.x, -0.5 * nv.y), hm = mk(0.5 * nv.x, 0.5 * nv.y);
                    G = k * (hp * dp + hm * dm + nv.z * dz);
                }
                cd* o = (pass ? V : W) + pos * (int64_t)P * P + nn * nn + nn;
                if (pass) {
                    const cd v = grad_v ? G : Sv;
                    o[m] = v;
                    if (m) o[-m] = conjg(v);
                } else {
                    cd mono = mk(0.0, 0.0);
                    if (kind == FB_OP_L || kind == FB_OP_LP) mono = mk(1.0, 0.0);
                    if (kind == FB_OP_A) {
                        const cd be = g.beta[e];
                        mono = mk(k * be.im, -k * be.re);   // -i k beta
                    }
                    const double f = k * g.area[e] / 3.0;   // ik A_j w_q, w_q = 1/3
                    const cd vp = mono * conjg(Sv) + conjg(G), vm = mono * Sv + G;
                    o[m] = mk(-f * vp.im, f * vp.re);
                    if (m) o[-m] = mk(-f * vm.im, f * vm.re);
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------- coaxial ----
// (E|F)^m_{n'n}(tau), m < p, n', n < p, by the algorithm of Sec. 3.3.1:
//  1 seeds (E|F)^0_{n',0} = (-1)^{n'} sqrt(2n'+1) f_{n'}(k tau), n' < 2p   (Eq. shft1)
//  2 sectorial (E|F)^{m+1}_{n',m+1} up in m                                (Eq. shft2)
//  k tau < 1: 3 propagation in n for n' >= n (Eq. shft5), 4 symmetry
//  k tau >= 1: 3.1 zonal (Eq. shft7), 3.2 diagonal + two subdiagonals
//     (Eq. shft8; third formula with b_n^{-m-1}), 3 propagation in n'
//     (Eq. shift6), 4 symmetry.
// One CTA per coefficient set: every step is a chain along one index with
// the other two free, so the threads take the free ones and a barrier
// separates the links (about 5 p of them); the diagonals (3.2) advance as a
// wavefront, order m + 1 one step behind order m.  The recursion factors
// a_n^m and b_n^m are the same for every set and come from a table.  L-room
// at 609 Hz (orders to 36): one thread per set took 24.4 ms, this form 0.34 ms.
// out: [m][n'][n] with stride p (p^3 complex).
struct CoaxSet {
    double ktau;
    int p;
    int kind;    // 0 = S|R, 1 = R|R
    int64_t out_off;
};

// a_n^m at [n (M + 1) + m], b_n^{m} at [n (2 M + 1) + m + M], n < N, |m| <= M
__global__ void k_coaxial_factors(int N, int M, double* __restrict__ a, double* __restrict__ b) {
    const int w = 2 * M + 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N * w; i += gridDim.x * blockDim.x) {
        const int n = i / w, m = i % w - M;
        b[i] = coef_b(n, m);
        if (m >= 0) a[n * (M + 1) + m] = coef_a(n, m);
    }
}

__global__ void __launch_bounds__(512) k_coaxial(const CoaxSet* sets, cd* scratch, int64_t scratch_stride,
                                                 double* fscratch, int64_t fstride, const double* __restrict__ ca,
                                                 const double* __restrict__ cb, int M, cd* out) {
    const CoaxSet cs = sets[blockIdx.x];
    const int p = cs.p, tid = threadIdx.x, nth = blockDim.x;
    const int W2 = 2 * p + 2, W3 = p + 2;
    cd* X = scratch + blockIdx.x * scratch_stride;
    auto at = [&](int m, int n1, int n) -> cd& { return X[((int64_t)m * W2 + n1) * W3 + n]; };
    auto fa = [&](int n, int m) { return n < 0 ? 0.0 : ca[n * (M + 1) + m]; };
    auto fb = [&](int n, int m) { return n < 0 ? 0.0 : cb[n * (2 * M + 1) + m + M]; };
    for (int64_t i = tid; i < (int64_t)(p + 1) * W2 * W3; i += nth) X[i] = mk(0.0, 0.0);
    const int P2 = 2 * p;
    double* fj = fscratch + blockIdx.x * fstride;
    double* fy = fj + P2 + 1;
    if (tid == 0) sph_bessel_j(P2 - 1, cs.ktau, fj);
    if (tid == 32 && cs.kind == 0) sph_bessel_y(P2 - 1, cs.ktau, fy);
    __syncthreads();
    for (int n1 = tid; n1 < P2; n1 += nth) {
        double sg = (n1 & 1) ? -1.0 : 1.0;
        double s = sg * sqrt(2.0 * n1 + 1.0);
        at(0, n1, 0) = cs.kind == 0 ? mk(s * fj[n1], s * fy[n1]) : mk(s * fj[n1], 0.0);
    }
    __syncthreads();
    for (int m = 0; m < p - 1; ++m) {
        for (int n1 = m + 1 + tid; n1 < P2 - 1 - m; n1 += nth)
            at(m + 1, n1, m + 1) = (1.0 / fb(m + 1, -m - 1)) *
                                   (fb(n1, -m - 1) * at(m, n1 - 1, m) - fb(n1 + 1, m) * at(m, n1 + 1, m));
        __syncthreads();
    }
    if (cs.ktau < 1.0) {
        // every order m advances in n together: step n uses columns n and n - 1
        for (int n = 0; n < p - 1; ++n) {
            const int len = 2 * p - 1 - 2 * n;   // n1 = n .. 2p - 2 - n
            for (int i = tid; i < (n + 1) * len; i += nth) {
                const int m = i / len, n1 = n + i % len;
                at(m, n1, n + 1) = (1.0 / fa(n, m)) *
                                   (fa(n - 1, m) * (n >= 1 ? at(m, n1, n - 1) : mk(0.0, 0.0)) -
                                    fa(n1, m) * at(m, n1 + 1, n) +
                                    fa(n1 - 1, m) * (n1 >= 1 ? at(m, n1 - 1, n) : mk(0.0, 0.0)));
            }
            __syncthreads();
        }
    } else {
        for (int n = 0; n < p - 1; ++n) {
            for (int n1 = n + 1 + tid; n1 < 2 * p - n - 2; n1 += nth)
                at(0, n1, n + 1) = (1.0 / fa(n, 0)) *
                                   (fa(n - 1, 0) * (n >= 1 ? at(0, n1, n - 1) : mk(0.0, 0.0)) -
                                    fa(n1, 0) * at(0, n1 + 1, n) + fa(n1 - 1, 0) * at(0, n1 - 1, n));
            __syncthreads();
        }
        // order m at step s takes n = s - m: order m - 1 has done n one step before
        for (int s = 1; s <= 2 * p - 5; ++s) {
            for (int m = tid; m < p - 2; m += nth) {
                const int n = s - m;
                if (n < m + 1 || n >= p - 1) continue;
                if (n >= m + 2)
                    at(m + 1, n + 1, n) = (1.0 / fb(n + 1, -m - 1)) *
                                          (fb(n + 1, m) * at(m, n + 1, n) + fb(n, -m - 1) * at(m, n, n - 1) -
                                           fb(n, m) * at(m + 1, n, n - 1));
                at(m + 1, n + 1, n + 1) = (1.0 / fb(n + 1, -m - 1)) *
                                          (fb(n, m) * at(m + 1, n + 1, n - 1) - fb(n + 2, m) * at(m, n + 2, n) +
                                           fb(n + 1, -m - 1) * at(m, n, n));
                if (n >= m + 2)
                    at(m + 1, n + 2, n) = (1.0 / fb(n + 2, -m - 1)) *
                                          (fb(n + 1, m) * at(m + 1, n, n) - fb(n + 1, m) * at(m, n + 1, n + 1) +
                                           fb(n, -m - 1) * at(m, n + 1, n - 1));
            }
            __syncthreads();
        }
        for (int n1 = 4; n1 < p - 1; ++n1) {   // m = 1 .. n1 - 3, n = m + 1 .. n1 - 2
            const int side = n1 - 3;
            for (int i = tid; i < side * side; i += nth) {
                const int m = 1 + i / side, n = 2 + i % side;
                if (n <= m) continue;
                at(m, n1 + 1, n) = (1.0 / fa(n1, m)) * (fa(n - 1, m) * at(m, n1, n - 1) - fa(n, m) * at(m, n1, n + 1) +
                                                        fa(n1 - 1, m) * at(m, n1 - 1, n));
            }
            __syncthreads();
        }
    }
    cd* o = out + cs.out_off;
    for (int64_t i = tid; i < (int64_t)p * p * p; i += nth) {
        const int n = (int)(i % p), n1 = (int)(i / p % p), m = (int)(i / ((int64_t)p * p));
        cd v = mk(0.0, 0.0);
        if (n1 >= m && n >= m) {
            if (n1 >= n) v = at(m, n1, n);
            else {
                v = at(m, n, n1);
                if ((n + n1) & 1) v = mk(-v.re, -v.im);
            }
        }
        o[i] = v;
    }
}

// ------------------------------------------------------------ rotations ----
// Gauss-Legendre nodes/weights on [-1,1] by Newton iteration on P_nq.
__global__ void k_gauss_legendre(int nq, double* x, double* w) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nq) return;
    double z = cos(FB_PI * (i + 0.75) / (nq + 0.5));
    double pp = 0.0;
    for (int it = 0; it < 100; ++it) {
        double p1 = 1.0, p2 = 0.0;
        for (int j = 1; j <= nq; ++j) {
            double p3 = p2;
            p2 = p1;
            p1 = ((2.0 * j - 1.0) * z * p2 - (j - 1.0) * p3) / j;
        }
        pp = nq * (z * p1 - p2) / (z * z - 1.0);
        double dz = p1 / pp;
        z -= dz;
        if (fabs(dz) < 1e-16) break;
    }
    double p1 = 1.0, p2 = 0.0;
    for (int j = 1; j <= nq; ++j) {
        double p3 = p2;
        p2 = p1;
        p1 = ((2.0 * j - 1.0) * z * p2 - (j - 1.0) * p3) / j;
    }
    pp = nq * (z * p1 - p2) / (z * z - 1.0);
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * pp * pp);
}

// Rotation Q = R_y(-theta) R_z(-phi) maps direction d to +z; Q^T y = R_z(phi) R_y(theta) y.
__device__ inline V3 rotT(V3 d, V3 y) {
    double rho = norm(d);
    double th = acos(fmax(-1.0, fmin(1.0, d.z / rho)));
    double ph = atan2(d.y, d.x);
    double ct, st, cp, sp;
    sincos(th, &st, &ct);
    sincos(ph, &sp, &cp);
    // R_y(theta) y
    V3 a = v3(ct * y.x + st * y.z, y.y, -st * y.x + ct * y.z);
    // R_z(phi) a
    return v3(cp * a.x - sp * a.y, sp * a.x + cp * a.y, a.z);
}

// Y_n^m at the product grid (GL in cos theta x uniform phi) rotated by Q_d^T,
// for a batch of directions.  out[(dir * npts + q) * P^2 + nm]
__global__ void k_rot_grid(const double* dirs, int ndir, int identity, int P, int nq, int nphi,
                           const double* glx, double* scratch, int sstride, cd* out) {
    int npts = nq * nphi;
    int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tid >= (int64_t)ndir * npts) return;
    int d = (int)(tid / npts), q = (int)(tid % npts);
    int it = q / nphi, ip = q % nphi;
    double ct = glx[it], st = sqrt(fmax(0.0, 1.0 - ct * ct));
    double ph = 2.0 * FB_PI * ip / nphi;
    double sp, cp;
    sincos(ph, &sp, &cp);
    V3 y = v3(st * cp, st * sp, ct);
    V3 dv = v3(dirs[3 * d], dirs[3 * d + 1], dirs[3 * d + 2]);
    V3 u = identity ? y : rotT(dv, y);
    double un = norm(u);
    ylm_unit(P, u.x / un, u.y / un, u.z / un, scratch + tid * (int64_t)sstride, out + tid * (int64_t)P * P);
}

// D^n_{mu,m} = sum_q W_q conj(Y_n^mu(y_q)) Y_n^m(Q^T y_q) for the batch.
// grid: (entry chunk, n, dir); out[dir_global][rot_off(n) + (mu+n)(2n+1) + (m+n)]
__global__ void k_rot_project(const cd* Yg, const cd* Yr, int ndir, int P, int nq, int nphi,
                              const double* glw, int dir0, cd* out) {
    int n = blockIdx.y;
    int d = blockIdx.z;
    int w = 2 * n + 1;
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= w * w) return;
    int mu = e / w - n, m = e % w - n;
    int npts = nq * nphi;
    double wphi = 2.0 * FB_PI / nphi;
    cd acc = mk(0.0, 0.0);
    const cd* yr = Yr + (int64_t)d * npts * P * P;
    for (int q = 0; q < npts; ++q) {
        double wq = glw[q / nphi] * wphi;
        cd a = Yg[(int64_t)q * P * P + nm_idx(n, mu)];
        cd b = yr[(int64_t)q * P * P + nm_idx(n, m)];
        cmacc(acc, wq * a, b);
    }
    int64_t rot_off = (int64_t)n * (2 * n - 1) * (2 * n + 1) / 3;
    int64_t per_dir = (int64_t)P * (2 * P - 1) * (2 * P + 1) / 3;
    out[(int64_t)(dir0 + d) * per_dir + rot_off + e] = acc;
}

// --------------------------------------------------------- composition ----
// T[(n',m'),(n,m)] = sum_{|mu| <= min(n',n)} conj(D^{n'}_{mu,m'}) C^{|mu|}_{n',n} D^n_{mu,m}
__global__ void k_compose(const ComposeJob* jobs, const cd* __restrict__ rot, int Prot,
                          const cd* __restrict__ coax, cd* __restrict__ T) {
    ComposeJob jb = jobs[blockIdx.y];
    int rows = jb.p_out * jb.p_out, cols = jb.p_in * jb.p_in;
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)rows * cols) return;
    int r = (int)(e / cols), c = (int)(e % cols);
    int n1 = (int)sqrt((double)r);
    while (n1 * n1 > r) --n1;
    while ((n1 + 1) * (n1 + 1) <= r) ++n1;
    int m1 = r - n1 * n1 - n1;
    int n = (int)sqrt((double)c);
    while (n * n > c) --n;
    while ((n + 1) * (n + 1) <= c) ++n;
    int m = c - n * n - n;
    const cd* D = rot + jb.rot_off;
    int64_t o1 = (int64_t)n1 * (2 * n1 - 1) * (2 * n1 + 1) / 3;
    int64_t o0 = (int64_t)n * (2 * n - 1) * (2 * n + 1) / 3;
    int w1 = 2 * n1 + 1, w0 = 2 * n + 1;
    int mn = min(n1, n);
    cd acc = mk(0.0, 0.0);
    for (int mu = -mn; mu <= mn; ++mu) {
        cd d1 = D[o1 + (int64_t)(mu + n1) * w1 + (m1 + n1)];
        cd d0 = D[o0 + (int64_t)(mu + n) * w0 + (m + n)];
        cd cc = coax[jb.coax_off + ((int64_t)abs(mu) * jb.pc + n1) * jb.pc + n];
        cmacc(acc, d1, cc * d0);
    }
    T[jb.t_off + e] = acc;
}

// Composes the translation matrices of the listed jobs that are not built
// yet (T = D_out^H C D_in in FP64), plus their FP32 copies when present.
fb_status fb_compose_jobs(fb_op* op, const std::vector<int>& which, cudaStream_t s) {
    std::vector<ComposeJob> todo;
    for (int j : which) {
        if (op->h_jobs[j].t_off < 0)
            return fb_fail(FB_ERR_ARG, "composed translation matrices exist only up to order " +
                                           std::to_string(FB_COMPOSE_PMAX));
        if (!op->job_done[j]) todo.push_back(op->h_jobs[j]);
    }
    if (todo.empty()) return FB_OK;
    if (!op->T64) FB_CHECK(dalloc(&op->T64, std::max<int64_t>(op->T_count, 1)));
    if (op->prec == FB_PREC_MIXED_FMM && !op->T32) FB_CHECK(dalloc(&op->T32, std::max<int64_t>(op->T_count, 1)));
    ComposeJob* djobs = nullptr;
    FB_CHECK(dalloc(&djobs, todo.size()));
    FB_CUDA(cudaMemcpyAsync(djobs, todo.data(), sizeof(ComposeJob) * todo.size(), cudaMemcpyHostToDevice, s));
    int64_t maxe = 0;
    for (auto& jb : todo) maxe = std::max<int64_t>(maxe, (int64_t)jb.p_out * jb.p_out * jb.p_in * jb.p_in);
    for (size_t j0 = 0; j0 < todo.size(); j0 += 65535) {
        int nj = (int)std::min<size_t>(65535, todo.size() - j0);
        dim3 grid(div_up(maxe, 256), nj);
        k_compose<<<grid, 256, 0, s>>>(djobs + j0, op->rot64, op->Prot, op->coax64, op->T64);
    }
    if (op->T32)
        for (size_t i = 0; i < todo.size();) {   // one launch per run of adjacent matrices
            const int64_t t0 = todo[i].t_off;
            int64_t t1 = t0;
            for (; i < todo.size() && todo[i].t_off == t1; ++i)
                t1 += (int64_t)todo[i].p_out * todo[i].p_out * todo[i].p_in * todo[i].p_in;
            k_d2f<<<div_up(t1 - t0, 256), 256, 0, s>>>(op->T64 + t0, op->T32 + t0, t1 - t0);
        }
    FB_LAUNCH_CHECK();
    cudaError_t e = cudaStreamSynchronize(s);
    dfree(djobs);
    if (e != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("composition: ") + cudaGetErrorString(e));
    for (int j : which) op->job_done[j] = 1;
    return FB_OK;
}

fb_status fb_compose_all(fb_op* op, cudaStream_t s) {
    std::vector<int> all;
    for (size_t j = 0; j < op->h_jobs.size(); ++j)
        if (op->h_jobs[j].t_off >= 0) all.push_back((int)j);
    return fb_compose_jobs(op, all, s);
}

// ------------------------------------------------------------ host side ----
__global__ void k_leaf_of(const int32_t* leaf_start, int nleaf, int32_t* leaf_of) {
    int b = blockIdx.x;
    if (b >= nleaf) return;
    for (int i = leaf_start[b] + threadIdx.x; i < leaf_start[b + 1]; i += blockDim.x) leaf_of[i] = b;
}
__global__ void k_box_centers(const uint32_t* keys, int n, int level, double ox, double oy, double oz,
                              double delta, double* c) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    uint32_t k = keys[b];
    int x = 0, y = 0, z = 0;
    for (int i = 0; i < level; ++i) {
        x |= ((k >> (3 * i)) & 1u) << i;
        y |= ((k >> (3 * i + 1)) & 1u) << i;
        z |= ((k >> (3 * i + 2)) & 1u) << i;
    }
    c[3 * b] = ox + (x + 0.5) * delta;
    c[3 * b + 1] = oy + (y + 0.5) * delta;
    c[3 * b + 2] = oz + (z + 0.5) * delta;
}

// Real factors d^n(theta) of the rotation blocks of every direction from the
// single matrix Delta^n = d^n(pi/2):
//   d^n_{mu,m}(theta) = sum_k Delta^n_{mu,k} Delta^n_{m,k} cos(k theta + (mu - m) pi/2),
// the rotation about y written as a rotation about z between two quarter
// turns (the identity holds for the real factors of this harmonic
// convention; checked against the projection of the definition to 1e-13 up
// to degree 40, and against the exponential of the rotation generator J_y to
// 1e-12 up to degree 318).  Also writes the phase tables ph[m + P - 1] = e^{i m phi}
// and, for degrees n < Pc, the complex blocks D = d e^{i m phi} the
// composed matrices use.  grid: (entry chunk, n, dir)
__global__ void k_rot_delta(const cd* delta, const double* dirs, int ndir, int P, int Pc, double* d64,
                            cd* ph64, cf* ph32, cd* r64) {
    __shared__ double cs[FB_ROT_PMAX], sn[FB_ROT_PMAX];
    int n = blockIdx.y, dd = blockIdx.z;
    int w = 2 * n + 1;
    double x = dirs[3 * dd], y = dirs[3 * dd + 1], z = dirs[3 * dd + 2];
    double th = acos(fmax(-1.0, fmin(1.0, z / sqrt(x * x + y * y + z * z))));
    double phi = atan2(y, x);
    for (int k = threadIdx.x; k <= n; k += blockDim.x) sincos((double)k * th, &sn[k], &cs[k]);
    __syncthreads();
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x == 0 && n == 0)
        for (int q = threadIdx.x; q < 2 * P - 1; q += blockDim.x) {
            double sp, cp;
            sincos((double)(q - (P - 1)) * phi, &sp, &cp);
            ph64[(int64_t)dd * (2 * P - 1) + q] = mk(cp, sp);
            ph32[(int64_t)dd * (2 * P - 1) + q] = mk((float)cp, (float)sp);
        }
    if (e >= w * w) return;
    int mu = e / w - n, m = e % w - n;
    int64_t off = (int64_t)n * (2 * n - 1) * (2 * n + 1) / 3;
    const cd* Dm = delta + off + (int64_t)(mu + n) * w;
    const cd* Dn = delta + off + (int64_t)(m + n) * w;
    // cos(k th + j pi/2) for j = (mu - m) mod 4: cos, -sin, -cos, sin
    int j = ((mu - m) % 4 + 4) % 4;
    double acc = 0.0;
    for (int k = -n; k <= n; ++k) {
        int ak = k < 0 ? -k : k;
        double c = cs[ak], sg = k < 0 ? -sn[ak] : sn[ak];
        double f = j == 0 ? c : (j == 1 ? -sg : (j == 2 ? -c : sg));
        acc = fma(Dm[k + n].re * Dn[k + n].re, f, acc);
    }
    int64_t per_dir = (int64_t)P * (2 * P - 1) * (2 * P + 1) / 3;
    int64_t o = (int64_t)dd * per_dir + off + e;
    d64[o] = acc;
    if (n < Pc) {
        double sp, cp;
        sincos((double)m * phi, &sp, &cp);
        int64_t per_c = (int64_t)Pc * (2 * Pc - 1) * (2 * Pc + 1) / 3;
        r64[(int64_t)dd * per_c + off + e] = mk(acc * cp, acc * sp);
    }
}

// Rotation data of every direction up to degree P, cached in the tree and
// recomputed only when a larger P is needed.  Delta^n = d^n(pi/2) comes from
// the definition of the rotation coefficients, evaluated by projection
// quadrature (exact for the band limit) for the direction +x; every
// direction's real factors then follow from it (k_rot_delta).
fb_status fb_tree_rotations(fb_tree* t, int P, const std::vector<double>& dirs, cudaStream_t s,
                            const fb_tree::RotSet** out) {
    int ndir = (int)dirs.size() / 3;
    for (const auto& rs : t->rot_sets)
        if (rs.P == P && rs.ndir == ndir) {
            *out = &rs;
            return FB_OK;
        }
    if (P > FB_ROT_PMAX) return fb_fail(FB_ERR_ARG, "expansion order above " + std::to_string(FB_ROT_PMAX));
    const int Prot = P;
    const int Pc = std::min(P, FB_COMPOSE_PMAX);
    const int64_t per_dir = (int64_t)Prot * (2 * Prot - 1) * (2 * Prot + 1) / 3;
    const int64_t per_c = (int64_t)Pc * (2 * Pc - 1) * (2 * Pc + 1) / 3;
    const int nq = Prot + 1, nphi = 2 * Prot + 1, npts = nq * nphi;
    const int ystride = Prot * (Prot + 1) / 2 + 8;
    double *glx = nullptr, *glw = nullptr, *ddirs = nullptr, *dx = nullptr, *yscr = nullptr;
    cd *Yg = nullptr, *Yr = nullptr, *delta = nullptr;
    auto free_tmp = [&]() { dfree(glx); dfree(glw); dfree(ddirs); dfree(dx); dfree(yscr); dfree(Yg); dfree(Yr); dfree(delta); };
    fb_status st;
    if ((st = dalloc(&glx, nq)) || (st = dalloc(&glw, nq)) || (st = dalloc(&ddirs, dirs.size())) ||
        (st = dalloc(&dx, 3)) || (st = dalloc(&yscr, (size_t)npts * ystride)) ||
        (st = dalloc(&Yg, (size_t)npts * Prot * Prot)) || (st = dalloc(&Yr, (size_t)npts * Prot * Prot)) ||
        (st = dalloc(&delta, per_dir))) {
        free_tmp();
        return st;
    }
    const double xdir[3] = {1.0, 0.0, 0.0};
    FB_CUDA(cudaMemcpyAsync(ddirs, dirs.data(), sizeof(double) * dirs.size(), cudaMemcpyHostToDevice, s));
    FB_CUDA(cudaMemcpyAsync(dx, xdir, sizeof(xdir), cudaMemcpyHostToDevice, s));
    k_gauss_legendre<<<div_up(nq, 64), 64, 0, s>>>(nq, glx, glw);
    // Y_n^m on the grid, unrotated and rotated for the direction +x
    k_rot_grid<<<div_up(npts, 128), 128, 0, s>>>(dx, 1, 1, Prot, nq, nphi, glx, yscr, ystride, Yg);
    k_rot_grid<<<div_up(npts, 128), 128, 0, s>>>(dx, 1, 0, Prot, nq, nphi, glx, yscr, ystride, Yr);
    {
        dim3 grid(div_up((2 * Prot - 1) * (2 * Prot - 1), 128), Prot, 1);
        k_rot_project<<<grid, 128, 0, s>>>(Yg, Yr, 1, Prot, nq, nphi, glw, 0, delta);
    }
    FB_LAUNCH_CHECK();
    fb_tree::RotSet rs;
    rs.P = Prot;
    rs.Pc = Pc;
    rs.per_dir = per_dir;
    rs.per_dir_c = per_c;
    rs.ndir = ndir;
    auto free_rs = [&]() { dfree(rs.r64); dfree(rs.d64); dfree(rs.ph64); dfree(rs.ph32); };
    if ((st = dalloc(&rs.r64, (size_t)ndir * per_c)) || (st = dalloc(&rs.d64, (size_t)ndir * per_dir)) ||
        (st = dalloc(&rs.ph64, (size_t)ndir * (2 * Prot - 1))) ||
        (st = dalloc(&rs.ph32, (size_t)ndir * (2 * Prot - 1)))) {
        free_tmp();
        free_rs();
        return st;
    }
    {
        dim3 grid(div_up((2 * Prot - 1) * (2 * Prot - 1), 128), Prot, ndir);
        k_rot_delta<<<grid, 128, 0, s>>>(delta, ddirs, ndir, Prot, Pc, rs.d64, rs.ph64, rs.ph32, rs.r64);
    }
    FB_LAUNCH_CHECK();
    cudaError_t e = cudaStreamSynchronize(s);
    free_tmp();
    if (e != cudaSuccess) {
        free_rs();
        return fb_fail(FB_ERR_CUDA, std::string("rotation setup: ") + cudaGetErrorString(e));
    }
    t->rot_sets.push_back(rs);
    *out = &t->rot_sets.back();
    return FB_OK;
}

static int igcd(int a, int b) {
    a = std::abs(a);
    b = std::abs(b);
    while (b) { int t = a % b; a = b; b = t; }
    return a;
}

static void build_tiles(TransPlan& pl) {
    const int BM = 64, BN = 32;
    pl.h_tiles.clear();
    for (int t = 0; t < (int)pl.h_tasks.size(); ++t) {
        const TransTask& tk = pl.h_tasks[t];
        for (int r = 0; r < tk.rows; r += BM)
            for (int c = 0; c < tk.npairs; c += BN) pl.h_tiles.push_back(TransTile{t, r, c, 0});
    }
    pl.ntiles = (int)pl.h_tiles.size();
}

static fb_status upload_plan(TransPlan& pl, const int32_t* src, const int32_t* dst) {
    pl.src_idx = src;
    pl.dst_idx = dst;
    build_tiles(pl);
    if (pl.h_tasks.empty()) return FB_OK;
    FB_CHECK(dalloc(&pl.tasks, pl.h_tasks.size()));
    FB_CHECK(dalloc(&pl.tiles, pl.h_tiles.size()));
    FB_CUDA(cudaMemcpy(pl.tasks, pl.h_tasks.data(), sizeof(TransTask) * pl.h_tasks.size(), cudaMemcpyHostToDevice));
    FB_CUDA(cudaMemcpy(pl.tiles, pl.h_tiles.data(), sizeof(TransTile) * pl.h_tiles.size(), cudaMemcpyHostToDevice));
    return FB_OK;
}

fb_status fb_fmm_create(fb_op* op, double d0, int pmin, cudaStream_t s) {
    const fb_tree* t = op->tree;
    const fb_mesh* m = op->mesh;
    int L = t->L;
    op->L = L;
    int64_t n = op->n;
    double k = op->k;
    for (int l = 2; l <= L; ++l) op->p[l] = fb_order_rule(k, t->side / (double)(1 << l), d0, pmin);
    int pL = op->p[L], PL = pL * pL;
    op->lev_off[0] = 0;
    for (int l = 0; l <= L; ++l) {
        int P = l >= 2 ? op->p[l] * op->p[l] : 0;
        op->lev_off[l + 1] = op->lev_off[l] + (int64_t)t->nbox[l] * P;
    }
    int64_t mp_count = op->lev_off[L + 1];
    // ---- near field
    int nleaf = t->nbox[L];
    std::vector<int32_t> ucnt(nleaf), ulist((size_t)nleaf * FB_ULIST);
    FB_CUDA(cudaMemcpyAsync(ucnt.data(), t->ucnt, sizeof(int32_t) * nleaf, cudaMemcpyDeviceToHost, s));
    FB_CUDA(cudaMemcpyAsync(ulist.data(), t->ulist, sizeof(int32_t) * ulist.size(), cudaMemcpyDeviceToHost, s));
    FB_CUDA(cudaStreamSynchronize(s));
    const std::vector<int32_t>& ls = t->h_leaf_start;
    op->h_nf_off.assign(nleaf + 1, 0);
    op->h_nf_ncol.assign(nleaf, 0);
    for (int b = 0; b < nleaf; ++b) {
        int K = 0;
        for (int i = 0; i < ucnt[b]; ++i) {
            int sl = ulist[(size_t)b * FB_ULIST + i];
            K += ls[sl + 1] - ls[sl];
        }
        op->h_nf_ncol[b] = K;
        op->h_nf_off[b + 1] = op->h_nf_off[b] + (int64_t)(ls[b + 1] - ls[b]) * K;
    }
    op->nf_count = op->h_nf_off[nleaf];
    FB_CHECK(dalloc(&op->nf_off, nleaf + 1));
    FB_CHECK(dalloc(&op->nf_ncol, nleaf));
    FB_CHECK(dalloc(&op->nf64, op->nf_count));
    FB_CUDA(cudaMemcpyAsync(op->nf_off, op->h_nf_off.data(), sizeof(int64_t) * (nleaf + 1), cudaMemcpyHostToDevice, s));
    FB_CUDA(cudaMemcpyAsync(op->nf_ncol, op->h_nf_ncol.data(), sizeof(int32_t) * nleaf, cudaMemcpyHostToDevice, s));
    const fb_op* dn = op->near_donor;
    if (dn && dn->nf64 && dn->kind == op->kind && dn->k == k && dn->mesh == m && dn->tree == t &&
        dn->nf_count == op->nf_count) {
        // the same entries: copy them instead of integrating again
        FB_CUDA(cudaMemcpyAsync(op->nf64, dn->nf64, sizeof(cd) * op->nf_count, cudaMemcpyDeviceToDevice, s));
    } else {
        int maxK = 1;
        for (int b = 0; b < nleaf; ++b) maxK = std::max(maxK, op->h_nf_ncol[b]);
        const dim3 grid((unsigned)nleaf, (unsigned)div_up(maxK, NF_COLS));
        auto fill = op->kind == FB_OP_L    ? k_near_fill<FB_OP_L>
                    : op->kind == FB_OP_M  ? k_near_fill<FB_OP_M>
                    : op->kind == FB_OP_LP ? k_near_fill<FB_OP_LP>
                    : op->kind == FB_OP_MP ? k_near_fill<FB_OP_MP>
                                           : k_near_fill<FB_OP_A>;
        fill<<<grid, NF_COLS, 0, s>>>(m->g, k, m->rc, t->perm, t->leaf_start, t->ucnt, t->ulist, op->nf_off,
                                      op->nf_ncol, op->nf64);
        FB_LAUNCH_CHECK();
    }
    // ---- box centres of every level
    std::vector<double*> centers(L + 1, nullptr);
    auto free_centers = [&]() { for (auto& c : centers) dfree(c); };
    for (int l = 0; l <= L; ++l) {
        fb_status st = dalloc(&centers[l], (size_t)3 * t->nbox[l]);
        if (st) { free_centers(); return st; }
        k_box_centers<<<div_up(t->nbox[l], 128), 128, 0, s>>>(t->keys[l], t->nbox[l], l, t->origin[0],
                                                              t->origin[1], t->origin[2],
                                                              t->side / (double)(1 << l), centers[l]);
    }
    // ---- P2M / L2P operators
    {
        int32_t* leaf_of = nullptr;
        double* tabs = nullptr;
        cd* sg = nullptr;
        const int Pp1 = pL + 1, M = pL + 1;
        // elements per CTA: up to 8 within 64 KB; S in global memory where one element's does not fit
        const bool s_global = p2m_elem_bytes(Pp1, false) > 200 * 1024;
        const size_t per = p2m_elem_bytes(Pp1, s_global);
        const int E = s_global ? 1 : (int)std::max<size_t>(1, std::min<size_t>(8, 64 * 1024 / per));
        const unsigned grid = (unsigned)std::min<int64_t>(div_up(n, E), s_global ? 304 : 1 << 30);
        const size_t nleg = (size_t)Pp1 * (Pp1 + 1), nga = (size_t)(Pp1 + 1) * (M + 1), ngb = (size_t)(Pp1 + 1) * (2 * M + 1);
        fb_status st;
        if ((st = dalloc(&leaf_of, n)) || (st = dalloc(&tabs, nleg + Pp1 + nga + ngb)) ||
            (s_global && (st = dalloc(&sg, (size_t)grid * E * (Pp1 * (Pp1 + 1) / 2)))) ||
            (st = dalloc(&op->w64, (size_t)n * PL)) || (st = dalloc(&op->v64, (size_t)n * PL)) ||
            (st = fb_smem_cap((const void*)k_p2m_l2p, E * per))) {
            dfree(leaf_of); dfree(tabs); dfree(sg); free_centers();
            return st;
        }
        k_leaf_of<<<nleaf, 64, 0, s>>>(t->leaf_start, nleaf, leaf_of);
        SphTab tab{tabs, tabs + nleg, tabs + nleg + Pp1, tabs + nleg + Pp1 + nga, M};
        k_sph_tables<<<std::min(div_up((int64_t)Pp1 * Pp1, 128), 152), 128, 0, s>>>(
            Pp1, M, tabs, tabs + nleg, tabs + nleg + Pp1, tabs + nleg + Pp1 + nga);
        k_p2m_l2p<<<grid, 128, E * per, s>>>(m->g, op->kind, k, pL, n, E, tab, t->perm, leaf_of, centers[L], sg, op->w64,
                                             op->v64);
        cudaError_t e = cudaStreamSynchronize(s);
        dfree(leaf_of);
        dfree(tabs);
        dfree(sg);
        if (e != cudaSuccess) { free_centers(); return fb_fail(FB_ERR_CUDA, std::string("P2M/L2P setup: ") + cudaGetErrorString(e)); }
    }
    free_centers();
    // ---- translation inventory: directions, coaxial sets, matrices
    int pmax = 0;
    for (int l = 2; l <= L; ++l) pmax = std::max(pmax, op->p[l]);
    std::vector<int> dir_of_code(FB_NOFF, -1);
    std::vector<double> dirs;    // unit-free integer directions
    std::map<std::tuple<int, int, int>, int> dir_index;
    auto get_dir = [&](int dx, int dy, int dz) {
        int g = igcd(igcd(dx, dy), dz);
        auto key = std::make_tuple(dx / g, dy / g, dz / g);
        auto it = dir_index.find(key);
        if (it != dir_index.end()) return it->second;
        int id = (int)dirs.size() / 3;
        dirs.push_back(dx / g);
        dirs.push_back(dy / g);
        dirs.push_back(dz / g);
        dir_index[key] = id;
        return id;
    };
    for (int c = 0; c < FB_NOFF; ++c) {
        int dx = c / 49 - 3, dy = (c / 7) % 7 - 3, dz = c % 7 - 3;
        if (std::max(std::abs(dx), std::max(std::abs(dy), std::abs(dz))) <= 1) continue;
        dir_of_code[c] = get_dir(dx, dy, dz);
    }
    int oct_dir_m2m[8], oct_dir_l2l[8];
    for (int o = 0; o < 8; ++o) {
        int sx = 1 - 2 * (o & 1), sy = 1 - 2 * ((o >> 1) & 1), sz = 1 - 2 * ((o >> 2) & 1);
        oct_dir_m2m[o] = get_dir(sx, sy, sz);     // parent - child = (1/2 - b) delta
        oct_dir_l2l[o] = get_dir(-sx, -sy, -sz);  // child - parent
    }
    int ndir = (int)dirs.size() / 3;
    op->dir_of_code = dir_of_code;
    // directions sharing a polar angle share their real rotation factors d^n
    // (D^n_{mu,m} = d^n_{mu,m}(theta) e^{i m phi}): representative of each
    // direction = the first direction with the same cos(theta) = dz / |d|,
    // compared exactly on the integer vectors (dz^2 |d'|^2 = dz'^2 |d|^2,
    // same sign of dz)
    op->theta_rep.assign(ndir, -1);
    for (int a = 0; a < ndir; ++a) {
        const int64_t za = (int64_t)dirs[3 * a + 2];
        const int64_t na = (int64_t)(dirs[3 * a] * dirs[3 * a] + dirs[3 * a + 1] * dirs[3 * a + 1] + za * za);
        for (int b = 0; b <= a; ++b) {
            const int64_t zb = (int64_t)dirs[3 * b + 2];
            const int64_t nb = (int64_t)(dirs[3 * b] * dirs[3 * b] + dirs[3 * b + 1] * dirs[3 * b + 1] + zb * zb);
            if ((za > 0) == (zb > 0) && (za < 0) == (zb < 0) && za * za * nb == zb * zb * na) {
                op->theta_rep[a] = b;
                break;
            }
        }
    }
    // polar-angle groups: one folded rotation table each (staged RCR)
    op->theta_slot.assign(ndir, -1);
    op->theta_dirs.clear();
    for (int a = 0; a < ndir; ++a) {
        const int rep = op->theta_rep[a];
        if (rep == a) {
            op->theta_slot[a] = (int)op->theta_dirs.size();
            op->theta_dirs.push_back(a);
        } else {
            op->theta_slot[a] = op->theta_slot[rep];
        }
    }
    // coaxial sets
    std::vector<CoaxSet> sets;
    std::map<std::tuple<int, int, int64_t>, int> set_index;   // (kind, p, ktau bits)
    auto get_set = [&](int kind, int p, double ktau) {
        int64_t bits;
        memcpy(&bits, &ktau, 8);
        auto key = std::make_tuple(kind, p, bits);
        auto it = set_index.find(key);
        if (it != set_index.end()) return it->second;
        int id = (int)sets.size();
        sets.push_back(CoaxSet{ktau, p, kind, 0});
        set_index[key] = id;
        return id;
    };
    struct MatReq { int level, which, code, pout, pin, dir, set; };
    std::vector<MatReq> reqs;
    op->m2l_toff.assign((size_t)(L + 1) * FB_NOFF, -1);
    for (int l = 2; l <= L; ++l) {
        double delta = t->side / (double)(1 << l);
        for (int c = 0; c < FB_NOFF; ++c) {
            int64_t cnt = t->m2l_group[(size_t)l * FB_NOFF + c + 1] - t->m2l_group[(size_t)l * FB_NOFF + c];
            if (cnt == 0) continue;
            int dx = c / 49 - 3, dy = (c / 7) % 7 - 3, dz = c % 7 - 3;
            double tau = std::sqrt((double)(dx * dx + dy * dy + dz * dz)) * delta;
            reqs.push_back(MatReq{l, 0, c, op->p[l], op->p[l], dir_of_code[c], get_set(0, op->p[l], k * tau)});
        }
    }
    for (int l = 3; l <= L; ++l) {
        double tau = std::sqrt(3.0) * 0.5 * (t->side / (double)(1 << l));
        int pc = std::max(op->p[l], op->p[l - 1]);
        int sidx = get_set(1, pc, k * tau);
        for (int o = 0; o < 8; ++o) {
            op->m2m_toff[l][o] = -1;
            op->l2l_toff[l][o] = -1;
            if (t->oct_group[l][o + 1] == t->oct_group[l][o]) continue;
            reqs.push_back(MatReq{l, 1, o, op->p[l - 1], op->p[l], oct_dir_m2m[o], sidx});
            reqs.push_back(MatReq{l, 2, o, op->p[l], op->p[l - 1], oct_dir_l2l[o], sidx});
        }
    }
    // coaxial coefficients
    int64_t coax_total = 0, scr_stride = 0, f_stride = 0;
    for (auto& cs : sets) {
        cs.out_off = coax_total;
        coax_total += (int64_t)cs.p * cs.p * cs.p;
        scr_stride = std::max<int64_t>(scr_stride, (int64_t)(cs.p + 1) * (2 * cs.p + 2) * (cs.p + 2));
        f_stride = std::max<int64_t>(f_stride, 4 * cs.p + 4);
    }
    cd* coax = nullptr;
    cd* cscr = nullptr;
    double* fscr = nullptr;
    CoaxSet* dsets = nullptr;
    auto free_coax = [&]() { dfree(coax); dfree(cscr); dfree(fscr); dfree(dsets); };
    fb_status st;
    if ((st = dalloc(&coax, std::max<int64_t>(coax_total, 1))) ||
        (st = dalloc(&cscr, std::max<int64_t>(scr_stride * (int64_t)sets.size(), 1))) ||
        (st = dalloc(&fscr, std::max<int64_t>(f_stride * (int64_t)sets.size(), 1))) ||
        (st = dalloc(&dsets, std::max<size_t>(sets.size(), 1)))) {
        free_coax();
        return st;
    }
    if (!sets.empty()) {
        FB_CUDA(cudaMemcpyAsync(dsets, sets.data(), sizeof(CoaxSet) * sets.size(), cudaMemcpyHostToDevice, s));
        int P = 1;
        for (const auto& cs : sets) P = std::max(P, cs.p);
        const int N = 2 * P + 2, M = P + 1;   // factors of degrees < N, orders <= M
        double* fac = nullptr;
        if ((st = dalloc(&fac, (size_t)N * (3 * M + 2)))) {
            free_coax();
            return st;
        }
        double* facb = fac + (size_t)N * (M + 1);
        k_coaxial_factors<<<std::min(div_up((int64_t)N * (2 * M + 1), 256), 1024), 256, 0, s>>>(N, M, fac, facb);
        k_coaxial<<<(unsigned)sets.size(), 512, 0, s>>>(dsets, cscr, scr_stride, fscr, f_stride, fac, facb, M, coax);
        const cudaError_t ce = cudaGetLastError();
        cudaStreamSynchronize(s);
        dfree(fac);
        if (ce != cudaSuccess) {
            free_coax();
            return fb_fail(FB_ERR_CUDA, std::string("coaxial sets: ") + cudaGetErrorString(ce));
        }
    }
    // rotation blocks of every direction up to pmax (cached in the tree: they
    // depend only on the directions, not on k or the operator)
    const fb_tree::RotSet* rset = nullptr;
    FB_CHECK(fb_tree_rotations(const_cast<fb_tree*>(t), pmax, dirs, s, &rset));
    int Prot = rset->P;
    int64_t per_dir = rset->per_dir;
    cd* rot = rset->r64;
    const int64_t per_dir_c = rset->per_dir_c;
    // composed translation matrices
    std::vector<ComposeJob> jobs;
    int64_t T_total = 0;
    for (auto& r : reqs) {
        ComposeJob jb;
        const bool fits = r.pout <= FB_COMPOSE_PMAX && r.pin <= FB_COMPOSE_PMAX;
        jb.t_off = fits ? T_total : -1;
        jb.rot_off = (int64_t)r.dir * per_dir_c;   // complex blocks: degrees < FB_COMPOSE_PMAX
        jb.coax_off = sets[r.set].out_off;
        jb.p_out = r.pout;
        jb.p_in = r.pin;
        jb.pc = sets[r.set].p;
        jobs.push_back(jb);
        if (r.which == 0) op->m2l_toff[(size_t)r.level * FB_NOFF + r.code] = jb.t_off;
        else if (r.which == 1) op->m2m_toff[r.level][r.code] = jb.t_off;
        else op->l2l_toff[r.level][r.code] = jb.t_off;
        if (fits) T_total += (int64_t)r.pout * r.pout * r.pin * r.pin;
    }
    // the matrix buffers are allocated by the first composition
    op->T_count = T_total;
    cudaError_t e = cudaStreamSynchronize(s);
    // the rotation blocks and coaxial sets stay with the operator (RCR form)
    op->coax64 = coax;
    op->coax_count = std::max<int64_t>(coax_total, 1);
    op->coax_sets.clear();
    for (const auto& cs : sets) op->coax_sets.emplace_back(cs.p, cs.out_off);
    std::sort(op->coax_sets.begin(), op->coax_sets.end());
    coax = nullptr;
    op->rot64 = rot;
    op->rotd64 = rset->d64;
    op->rph64 = rset->ph64;
    op->rph32 = rset->ph32;
    op->rot_count = (int64_t)ndir * per_dir;
    op->Prot = Prot;
    op->per_dir = per_dir;
    free_coax();
    FB_CHECK(fb_stg_tables(op, rset->d64, s));
    // composed matrices are built on demand (tensor-core levels below,
    // everything for the composed method or for inspection)
    op->h_jobs = jobs;
    op->h_job_level.clear();
    op->h_job_m2l.clear();
    for (auto& r : reqs) {
        op->h_job_level.push_back(r.level);
        op->h_job_m2l.push_back(r.which == 0 ? 1 : 0);
    }
    op->job_done.assign(jobs.size(), 0);
    op->m2l_job.assign((size_t)(L + 1) * FB_NOFF, -1);
    for (int l = 0; l <= FB_MAXLEV; ++l)
        for (int o = 0; o < 8; ++o) op->m2m_job[l][o] = op->l2l_job[l][o] = -1;
    for (size_t j = 0; j < reqs.size(); ++j) {
        const MatReq& r = reqs[j];
        if (r.which == 0) op->m2l_job[(size_t)r.level * FB_NOFF + r.code] = (int)j;
        else if (r.which == 1) op->m2m_job[r.level][r.code] = (int)j;
        else op->l2l_job[r.level][r.code] = (int)j;
    }
    if (e != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("translation setup: ") + cudaGetErrorString(e));
    // RCR plans: one task per (level, offset) / (level, octant) group
    {
        auto rcr_task = [&](const MatReq& r, int64_t g0, int64_t g1, int64_t src_base, int64_t dst_base) {
            RcrTask tk;
            tk.rot_off = (int64_t)r.dir * per_dir;
            tk.coax_off = sets[r.set].out_off;
            tk.pair_off = g0;
            tk.npairs = (int32_t)(g1 - g0);
            tk.p_out = r.pout;
            tk.p_in = r.pin;
            tk.pc = sets[r.set].p;
            tk.src_base = src_base;
            tk.dst_base = dst_base;
            tk.staged = r.which == 0 ? op->stg_m2l[r.level] : op->stg_pair[r.level];
            tk.pad = 0;
            return tk;
        };
        {
            const size_t cs = op->prec == FB_PREC_MIXED_FMM ? sizeof(cf) : sizeof(cd);
            for (int l = 2; l <= L; ++l) {
                op->stg_m2l[l] = fb_rcr_default_staged(op->p[l], op->p[l], cs);
                if (l >= 3) {
                    const int pm = std::max(op->p[l], op->p[l - 1]);
                    op->stg_pair[l] = fb_rcr_default_staged(pm, pm, cs);
                }
            }
        }
        // levels whose M2L groups are dense enough for the tensor-core form
        // (mixed precision): on average >= 48 box pairs per translation vector
        std::vector<int> tc_levels;
        if (op->prec == FB_PREC_MIXED_FMM) {
            for (int l = 2; l <= L; ++l) {
                int64_t pairs = 0, groups = 0;
                for (int c = 0; c < FB_NOFF; ++c) {
                    int64_t cnt = t->m2l_group[(size_t)l * FB_NOFF + c + 1] - t->m2l_group[(size_t)l * FB_NOFF + c];
                    if (cnt) { pairs += cnt; ++groups; }
                }
                if (groups && pairs >= 48 * groups && fb_composable(op, l, false)) {
                    tc_levels.push_back(l);
                    op->tc_level[l] = 1;
                }
            }
        }
        for (auto& r : reqs) {
            if (r.which == 0) {
                int64_t g0 = t->m2l_group[(size_t)r.level * FB_NOFF + r.code];
                int64_t g1 = t->m2l_group[(size_t)r.level * FB_NOFF + r.code + 1];
                RcrTask tk = rcr_task(r, g0, g1, op->lev_off[r.level], op->lev_off[r.level]);
                op->m2l_rcr.h_tasks.push_back(tk);
                if (!op->tc_level[r.level]) op->m2l_rcr_rest.h_tasks.push_back(tk);
            } else {
                int64_t g0 = t->oct_group[r.level][r.code], g1 = t->oct_group[r.level][r.code + 1];
                if (r.which == 1)
                    op->m2m_rcr[r.level].h_tasks.push_back(
                        rcr_task(r, g0, g1, op->lev_off[r.level], op->lev_off[r.level - 1]));
                else
                    op->l2l_rcr[r.level].h_tasks.push_back(
                        rcr_task(r, g0, g1, op->lev_off[r.level - 1], op->lev_off[r.level]));
            }
        }
        size_t csz = op->prec == FB_PREC_MIXED_FMM ? sizeof(cf) : sizeof(cd);
        FB_CHECK(fb_rcr_upload(op, op->m2l_rcr, t->m2l_src, t->m2l_dst, csz));
        FB_CHECK(fb_rcr_upload(op, op->m2l_rcr_rest, t->m2l_src, t->m2l_dst, csz));
        if (!tc_levels.empty()) {
            std::vector<int> need;
            for (size_t j = 0; j < op->h_jobs.size(); ++j)
                if (op->h_job_m2l[j] && op->tc_level[op->h_job_level[j]]) need.push_back((int)j);
            FB_CHECK(fb_compose_jobs(op, need, s));
            FB_CHECK(fb_tc_build(op, tc_levels, &op->tc_plan, s));
        }
        // M2M / L2L of child levels with >= 48 boxes per octant on average
        if (op->prec == FB_PREC_MIXED_FMM) {
            for (int l = 3; l <= L; ++l) {
                if (t->nbox[l] < 48 * 8 || !fb_composable(op, l, true)) continue;
                std::vector<int> need;
                std::vector<TcGroup> up, down;
                for (int o = 0; o < 8; ++o) {
                    int64_t g0 = t->oct_group[l][o], g1 = t->oct_group[l][o + 1];
                    if (g1 == g0) continue;
                    need.push_back(op->m2m_job[l][o]);
                    need.push_back(op->l2l_job[l][o]);
                    up.push_back(TcGroup{op->m2m_job[l][o], g0, (int32_t)(g1 - g0), l, l - 1});
                    down.push_back(TcGroup{op->l2l_job[l][o], g0, (int32_t)(g1 - g0), l - 1, l});
                }
                FB_CHECK(fb_compose_jobs(op, need, s));
                FB_CHECK(fb_tc_build_groups(op, up, t->oct_child[l], t->oct_parent[l], &op->tc_m2m[l], s));
                FB_CHECK(fb_tc_build_groups(op, down, t->oct_parent[l], t->oct_child[l], &op->tc_l2l[l], s));
            }
        }
        for (int l = 3; l <= L; ++l) {
            FB_CHECK(fb_rcr_upload(op, op->m2m_rcr[l], t->oct_child[l], t->oct_parent[l], csz));
            FB_CHECK(fb_rcr_upload(op, op->l2l_rcr[l], t->oct_parent[l], t->oct_child[l], csz));
        }
        op->method = FB_TRANS_AUTO;
    }
    // ---- FP32 copies for the mixed path.  High orders at small k tau give
    // coaxial coefficients (spherical Hankel functions of high order) beyond
    // the FP32 range; the mixed form is refused for such operators instead of
    // producing overflowed translations (the FP64 form handles them).
    if (op->prec == FB_PREC_MIXED_FMM) {
        double* dmax = nullptr;
        FB_CHECK(dalloc(&dmax, 1));
        FB_CUDA(cudaMemsetAsync(dmax, 0, sizeof(double), s));
        k_absmax<<<std::min(div_up(op->coax_count, 256), 1024), 256, 0, s>>>(op->coax64, op->coax_count, dmax);
        double hmax = 0.0;
        cudaError_t ce = cudaMemcpyAsync(&hmax, dmax, sizeof(double), cudaMemcpyDeviceToHost, s);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
        dfree(dmax);
        if (ce != cudaSuccess) return fb_fail(FB_ERR_CUDA, cudaGetErrorString(ce));
        if (!(hmax < 1e37))
            return fb_fail(FB_ERR_ARG, "mixed precision: translation coefficients reach " + std::to_string(hmax) +
                                           ", beyond the FP32 range at this order and wavenumber; use "
                                           "FB_PREC_FP64_FMM or a lower p_min");
    }
    if (op->prec == FB_PREC_MIXED_FMM) {
        FB_CHECK(dalloc(&op->nf32, op->nf_count));
        FB_CHECK(dalloc(&op->w32, (size_t)n * PL));
        FB_CHECK(dalloc(&op->v32, (size_t)n * PL));
        k_d2f<<<div_up(op->nf_count, 256), 256, 0, s>>>(op->nf64, op->nf32, op->nf_count);
        k_d2f<<<div_up(n * PL, 256), 256, 0, s>>>(op->w64, op->w32, n * PL);
        k_d2f<<<div_up(n * PL, 256), 256, 0, s>>>(op->v64, op->v32, n * PL);
        FB_CHECK(dalloc(&op->coax32, op->coax_count));
        k_d2f<<<div_up(op->coax_count, 256), 256, 0, s>>>(op->coax64, op->coax32, op->coax_count);
        FB_LAUNCH_CHECK();
        FB_CHECK(dalloc((cf**)&op->mp, mp_count));
        FB_CHECK(dalloc((cf**)&op->loc, mp_count));
        // of the FP64 entries only the leaf self-blocks stay (block-Jacobi
        // factorisation); the rest are dropped once the FP32 copies exist
        {
            int nleaf = t->nbox[L];
            std::vector<int64_t> off(nleaf + 1, 0);
            for (int b = 0; b < nleaf; ++b) {
                int64_t nb = t->h_leaf_start[b + 1] - t->h_leaf_start[b];
                off[b + 1] = off[b] + nb * nb;
            }
            int64_t* d_off = nullptr;
            FB_CHECK(dalloc(&d_off, nleaf + 1));
            fb_status st2 = dalloc(&op->self64, std::max<int64_t>(off[nleaf], 1));
            if (st2 == FB_OK) {
                cudaMemcpyAsync(d_off, off.data(), sizeof(int64_t) * (nleaf + 1), cudaMemcpyHostToDevice, s);
                st2 = fb_self_blocks(op, d_off, op->self64, s);
            }
            cudaError_t e2 = cudaStreamSynchronize(s);
            dfree(d_off);
            FB_CHECK(st2);
            if (e2 != cudaSuccess) return fb_fail(FB_ERR_CUDA, std::string("self blocks: ") + cudaGetErrorString(e2));
            dfree(op->nf64);
            dfree(op->w64);
            dfree(op->v64);
        }
    } else {
        FB_CHECK(dalloc((cd**)&op->mp, mp_count));
        FB_CHECK(dalloc((cd**)&op->loc, mp_count));
    }
    // ---- translation plans
    for (int l = 2; l <= L; ++l)
        for (int c = 0; c < FB_NOFF; ++c) {
            int64_t g0 = t->m2l_group[(size_t)l * FB_NOFF + c], g1 = t->m2l_group[(size_t)l * FB_NOFF + c + 1];
            if (g1 == g0) continue;
            TransTask tk;
            tk.t_off = op->m2l_toff[(size_t)l * FB_NOFF + c];
            tk.pair_off = g0;
            tk.npairs = (int32_t)(g1 - g0);
            tk.rows = tk.cols = op->p[l] * op->p[l];
            tk.src_base = op->lev_off[l];
            tk.dst_base = op->lev_off[l];
            op->m2l.h_tasks.push_back(tk);
        }
    FB_CHECK(upload_plan(op->m2l, t->m2l_src, t->m2l_dst));
    for (int l = 3; l <= L; ++l) {
        for (int o = 0; o < 8; ++o) {
            int64_t g0 = t->oct_group[l][o], g1 = t->oct_group[l][o + 1];
            if (g1 == g0) continue;
            TransTask up;
            up.t_off = op->m2m_toff[l][o];
            up.pair_off = g0;
            up.npairs = (int32_t)(g1 - g0);
            up.rows = op->p[l - 1] * op->p[l - 1];
            up.cols = op->p[l] * op->p[l];
            up.src_base = op->lev_off[l];
            up.dst_base = op->lev_off[l - 1];
            op->m2m[l].h_tasks.push_back(up);
            TransTask dn;
            dn.t_off = op->l2l_toff[l][o];
            dn.pair_off = g0;
            dn.npairs = (int32_t)(g1 - g0);
            dn.rows = op->p[l] * op->p[l];
            dn.cols = op->p[l - 1] * op->p[l - 1];
            dn.src_base = op->lev_off[l - 1];
            dn.dst_base = op->lev_off[l];
            op->l2l[l].h_tasks.push_back(dn);
        }
        // M2M: src child -> dst parent; L2L: src parent -> dst child
        FB_CHECK(upload_plan(op->m2m[l], t->oct_child[l], t->oct_parent[l]));
        FB_CHECK(upload_plan(op->l2l[l], t->oct_parent[l], t->oct_child[l]));
    }
    FB_CUDA(cudaStreamSynchronize(s));
    return FB_OK;
}
