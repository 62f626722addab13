// Cholesky-QR of complex64 state blocks: norms to FP64 accuracy, the Gram
// matrix, and the triangular update (arXiv:1501.05654, Sec. "Parallelization, optimizations
// and graphics processing units": orthogonalisation of a group of states);
// and the Gram matrices of FP64 accumulation shared with the eigensolver.
//
// What bounds them: at 128 states the Gram matrix and the update are 2 x
// 0.23 T FP32 FMAs on a 7.25 GB block, so FP32 arithmetic (about 7 ms each at
// the SIMT rate) and not memory (1.1 ms a pass) is the floor.  Both are
// register-tiled products.  FP64 instructions (two a clock per SM) are kept
// off the inner loops: runs of FP32 sums are collected in short two-float sums
// before they meet FP64.
#include <algorithm>

#include "rsg_async.cuh"
#include "rsg_internal.h"
#include "rsg_vec.cuh"

namespace rsg {

namespace {

__device__ __forceinline__ float2 f2_neg(float2 a) { return make_float2(-a.x, -a.y); }
// a - b (exact product, so one rounding)
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) { return f2_fma(b, make_float2(-1.f, -1.f), a); }

// hi += r, rounded; returns the exact rounding error (Knuth's two-sum), per
// component
__device__ __forceinline__ float2 f2_add_err(float2 &hi, float2 r) {
    const float2 s = f2_add(hi, r);
    const float2 b = f2_sub(s, hi);
    const float2 e = f2_add(f2_sub(hi, f2_sub(s, b)), f2_sub(r, b));
    hi = s;
    return e;
}
// (hi, lo) += r: hi takes the rounded sum, lo the rounding error of it
__device__ __forceinline__ void f2_two_sum(float2 &hi, float2 &lo, float2 r) {
    const float2 e = f2_add_err(hi, r);
    lo = f2_add(lo, e);
}

// ------------------------------------------------------------------ norms
// partial[blk][s] = sum over the block's points of |psi[p,s]|^2.  A thread
// owns a 16-byte vector (two states) of every by-th point.  The squares of
// eight points (each split by an FMA into its rounded value and its error) are
// summed in three floats: the second takes the exact rounding errors of the
// first, the third those of the second, so that less than 2^-60 of the sum is
// lost before it is added to FP64 once.  A group whose sum leaves the range
// where FP32 squares and their errors are exact (tails, huge values) is summed
// again in FP64.  Relative error of the norms, rms: 1e-16 to 2.5e-16 (every
// square an FP64 FMA: 1e-16 to 1e-15; two floats: 7e-16).  Bound by the issue of
// the packed additions: 192^3 x 128 states 1.85 ms (8.6 ms with FP64 FMAs).
constexpr int kNRun = 8;
constexpr float kNLow = 1e-24f, kNHigh = 1e37f;
// Adds state c's part of a group: its three-float sum, or its squares in FP64
// outside the exact range.
__device__ __forceinline__ void add_group(const float4 (&x)[kNRun], float hi, float lo, float l2, int c, double &a) {
    if (hi >= kNLow && hi <= kNHigh) {
        a += widen(hi) + (widen(lo) + widen(l2));
        return;
    }
    bool zero = true;
#pragma unroll
    for (int k = 0; k < kNRun; k++) zero = zero && (c ? x[k].z == 0.f && x[k].w == 0.f : x[k].x == 0.f && x[k].y == 0.f);
    if (zero) return;
#pragma unroll
    for (int k = 0; k < kNRun; k++) {
        const double re = c ? x[k].z : x[k].x, im = c ? x[k].w : x[k].y;
        a = fma(re, re, fma(im, im, a));
    }
}

__global__ void __launch_bounds__(256) k_norms32(const float4 *__restrict__ psi, int64_t P, int ldv, int SV, int S,
                                                 double *__restrict__ partial, int nblk) {
    __shared__ double red[256][2];
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.x * per;
    const int64_t p1 = p0 + per < P ? p0 + per : P;
    const int bx = blockDim.x, by = blockDim.y;
    for (int vb = 0; vb < SV; vb += bx) {
        const int v = vb + threadIdx.x;
        double a0 = 0.0, a1 = 0.0;
        if (v < SV) {
            for (int64_t p = p0 + threadIdx.y; p < p1; p += (int64_t)kNRun * by) {
                float4 x[kNRun];
#pragma unroll
                for (int k = 0; k < kNRun; k++) {
                    const int64_t q = p + (int64_t)k * by;
                    x[k] = q < p1 ? __ldg(psi + q * ldv + v) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                // components (state 0, state 1): re then im of each point
                float2 hi = make_float2(0.f, 0.f), lo = hi, l2 = hi;
#pragma unroll
                for (int k = 0; k < kNRun; k++) {
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        const float2 u = c ? make_float2(x[k].y, x[k].w) : make_float2(x[k].x, x[k].z);
                        const float2 sq = f2_mul(u, u);
                        const float2 er = f2_fma(u, u, f2_neg(sq));
                        const float2 e = f2_add_err(hi, sq);
                        f2_two_sum(lo, l2, e);
                        f2_two_sum(lo, l2, er);
                    }
                }
                add_group(x, hi.x, lo.x, l2.x, 0, a0);
                add_group(x, hi.y, lo.y, l2.y, 1, a1);
            }
        }
        const int tid = threadIdx.y * bx + threadIdx.x;
        red[tid][0] = a0;
        red[tid][1] = a1;
        __syncthreads();
        // the lanes of each vector in lane order, one thread per state
        for (int i = tid; i < 2 * bx; i += bx * by) {
            const int x = i >> 1, s = 2 * (vb + x) + (i & 1);
            if (s < S) {
                double t = 0.0;
                for (int l = 0; l < by; l++) t += red[l * bx + x][i & 1];
                partial[(int64_t)blockIdx.x * S + s] = t;
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------- sums over blocks
// out[i] = scale * sum_b partial[b][i], b in order: 32 outputs per block,
// whose rows are staged 32 at a time by 1024 threads while one warp adds them
// (the additions are the chain that bounds it, 29 us for 608 rows whether one
// or four groups of loads are in flight; with the loads in that chain too it
// took 100 us).
__global__ void __launch_bounds__(1024) k_sum_rows(const double *__restrict__ partial, int nblk, int64_t n,
                                                   double scale, double *__restrict__ out) {
    __shared__ double buf[2][32][33];
    const int64_t i = blockIdx.x * 32 + (int64_t)threadIdx.x;
    double s = 0.0;
    auto load = [&](int b0) {
        const int b = b0 + threadIdx.y;
        return i < n && b < nblk ? partial[(int64_t)b * n + i] : 0.0;
    };
    double v = load(0);
    for (int b0 = 0, k = 0; b0 < nblk; b0 += 32, k ^= 1) {
        buf[k][threadIdx.y][threadIdx.x] = v;
        __syncthreads();
        v = load(b0 + 32);
        if (threadIdx.y == 0) {
            const int m = min(32, nblk - b0);
#pragma unroll 8
            for (int q = 0; q < m; q++) s += buf[k][q][threadIdx.x];
        }
    }
    if (threadIdx.y == 0 && i < n) out[i] = scale * s;
}

// The same for a Hermitian S x S complex matrix of which partial holds
// s <= t: G[s][t], its mirror G[t][s] = conj, and (norms != nullptr) the
// diagonal replaced by the given FP64 norms.
__global__ void __launch_bounds__(256) k_sum_herm(const double2 *__restrict__ partial, int nblk, int S, double scale,
                                                  const double *__restrict__ norms, double2 *__restrict__ G) {
    __shared__ double2 red[16][17];
    const int s = blockIdx.y, t = blockIdx.x * 16 + threadIdx.x;
    if (blockIdx.x * 16 + 15 < s) return;
    double2 a = make_double2(0.0, 0.0);
    if (t < S && t >= s)
        for (int b = threadIdx.y; b < nblk; b += 16) {
            const double2 q = partial[((int64_t)b * S + s) * S + t];
            a.x += q.x;
            a.y += q.y;
        }
    red[threadIdx.y][threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.y != 0 || t >= S || t < s) return;
    double2 g = make_double2(0.0, 0.0);
    for (int l = 0; l < 16; l++) {
        g.x += red[l][threadIdx.x].x;
        g.y += red[l][threadIdx.x].y;
    }
    g.x *= scale;
    g.y *= scale;
    if (s == t) {
        if (norms) g.x = norms[s];
        g.y = 0.0;
        G[(int64_t)s * S + s] = g;
    } else {
        G[(int64_t)s * S + t] = g;
        G[(int64_t)t * S + s] = make_double2(g.x, -g.y);
    }
}

// ------------------------------------------------- Gram matrix, complex64
// Tile TS x TS of (s, t), tiles with s-tile <= t-tile; a thread owns 4 x 4
// entries and TS^2 / 16 threads make a group.  Below 64 columns the 256
// threads are several groups that share the staged points.  FP32 products
// are summed in FP32 over runs of 8 points; kGHeld runs are collected in a
// two-float sum (whose own rounding, below 2^-37 of its largest partial sum,
// lies under the 2^-24 of the runs), which is added to an FP64 sum.  An entry
// whose two-float sums leave the FP32 range although its runs do not (squares
// near 1e36) is summed again, every run in FP64.  The points come as
// they lie (one 16-byte asynchronous copy per two states), double-buffered;
// on the diagonal both operands are the same panel.  192^3 x 128 states: 18
// ms (108 ms when every run met two FP64 additions and conversions per value;
// kGHeld = 64 adds 0.6 ms, one two-float sum for all of a block's points, of
// less range and fewer bits, saves 0.8; a second pass of the block instead of
// the entry's own sums costs 0.6 by its code alone).
// The point blocks are `nsub` pieces of the blocks of 4096 points or more
// that gram_blocks names, cut at multiples of a run.
constexpr int kGHeld = 128;   // runs in a two-float sum
// One entry's sum again, every run added in FP64: `runs` runs of 8 points from
// p on, then those `step` points further, up to p1.
__device__ __noinline__ double2 gram_runs64(const float2 *x, const float2 *y, int64_t p, int64_t p1, int ld, int runs,
                                            int step) {
    double2 tot = make_double2(0.0, 0.0);
    for (; p < p1; p += step)
        for (int64_t r = p; r < p + 8 * runs && r < p1; r += 8) {
            float2 f = make_float2(0.f, 0.f);
            for (int64_t q = r; q < r + 8 && q < p1; q++) {
                const float2 a = x[q * ld], b = y[q * ld];
                f.x = fmaf(a.x, b.x, fmaf(a.y, b.y, f.x));
                f.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, f.y));
            }
            tot.x += (double)f.x;
            tot.y += (double)f.y;
        }
    return tot;
}
template <int TS>
struct G32Shape {
    static constexpr int NTH = TS * TS / 16, NG = 256 / NTH, RUNS = TS == 64 ? 4 : 2, KP = 8 * RUNS * NG;
    static constexpr int PANEL = KP * TS;               // complex values
    static constexpr int NL = PANEL / 2 / 256;          // 16-byte copies per thread and panel
    static constexpr int BYTES_AB = 2 * (TS == 64 ? 2 : 1) * PANEL * 8;
    static constexpr int BYTES_RED = NG > 1 ? NG * TS * TS * 16 : 0;
    static constexpr int BYTES = BYTES_AB > BYTES_RED ? BYTES_AB : BYTES_RED;
};

template <int TS>
__global__ void __launch_bounds__(256, 1) k_gram32(const float2 *__restrict__ psi, int64_t P, int ld, int S,
                                                   double2 *__restrict__ partial, int nb0, int nsub) {
    using G = G32Shape<TS>;
    constexpr int KP = G::KP;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2 *buf = (float2 *)smraw;               // [2][A, B][KP][TS] (64 columns), [2][KP][TS] else
    constexpr int BUFST = (TS == 64 ? 2 : 1) * G::PANEL;
    // tile pair (ti <= tj) of blockIdx.x
    int ti = 0, rest = blockIdx.x;
    const int nt = (S + TS - 1) / TS;
    while (rest >= nt - ti) {
        rest -= nt - ti;
        ti++;
    }
    const int tj = ti + rest;
    const bool diag = ti == tj;
    const int s0 = ti * TS, t0 = tj * TS;
    const int tid = threadIdx.x, g = tid / G::NTH, r = tid % G::NTH;
    // warp tiles of 16 rows x 32 columns; lanes 4 (rows) x 8 (columns), or
    // 4 x 4 in the 16-column tile: rows sr + {0, 1, 8, 9}, columns tc + {0, 1,
    // 2 LX, 2 LX + 1}, so that a quarter warp reads consecutive 16-byte words
    constexpr int LX = TS >= 32 ? 8 : 4, WJ = TS / (4 * LX);
    const int wt = r / (4 * LX), lr = r % (4 * LX);
    const int sr = 16 * (wt / WJ) + 2 * (lr / LX), tc = 4 * LX * (wt % WJ) + 2 * (lr % LX);
    const bool skip = diag && 4 * LX * (wt % WJ) + 4 * LX - 1 < 16 * (wt / WJ);
    const int64_t per = (P + nb0 - 1) / nb0, sub = ((per + nsub - 1) / nsub + 7) / 8 * 8;
    const int b0 = blockIdx.z / nsub, bj = blockIdx.z % nsub;
    const int64_t p0 = b0 * per + bj * sub;
    int64_t p1 = p0 + sub < (b0 + 1) * per ? p0 + sub : (b0 + 1) * per;
    if (p1 > P) p1 = P;

    const unsigned bsm = (unsigned)__cvta_generic_to_shared(buf);
    auto stage = [&](int64_t pc, int k) {
#pragma unroll
        for (int i = 0; i < G::NL; i++) {
            const int e = tid + i * 256, kk = e / (TS / 2), c = 2 * (e % (TS / 2));
            const int64_t p = pc + kk;
            const int na = p < p1 ? max(0, min(2, S - s0 - c)) * 8 : 0;   // a padding column is not reduced over
            cp_async16(bsm + (unsigned)((k * BUFST + 2 * e) * 8), psi + (na ? p * ld + s0 + c : 0), na);
            if (TS == 64 && !diag) {
                const int nb = p < p1 ? max(0, min(2, S - t0 - c)) * 8 : 0;
                cp_async16(bsm + (unsigned)((k * BUFST + G::PANEL + 2 * e) * 8), psi + (nb ? p * ld + t0 + c : 0), nb);
            }
        }
        cp_async_commit();
    };
    // sums of the 4 x 4 entries: two-float sums of up to kGHeld runs, (re, im)
    // pairs, and FP64
    double2 tot[4][4];
    float2 hi[4][4], lo[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            hi[i][j] = lo[i][j] = make_float2(0.f, 0.f);
            tot[i][j] = make_double2(0.0, 0.0);
        }
    // FP64 additions take 16 clocks a warp: the first flush has none to make
    bool first = true;
    auto flush = [&]() {
        if (first) {
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++)
                    tot[i][j] = make_double2(widen(hi[i][j].x) + widen(lo[i][j].x), widen(hi[i][j].y) + widen(lo[i][j].y));
        } else {
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    tot[i][j].x += widen(hi[i][j].x) + widen(lo[i][j].x);
                    tot[i][j].y += widen(hi[i][j].y) + widen(lo[i][j].y);
                }
        }
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) hi[i][j] = lo[i][j] = make_float2(0.f, 0.f);
        first = false;
    };
    if (p0 < p1) stage(p0, 0);
    int k = 0, held = 0;
    for (int64_t pc = p0; pc < p1; pc += KP, k ^= 1) {
        cp_async_wait<0>();
        __syncthreads();
        if (pc + KP < p1) stage(pc + KP, k ^ 1);
        if (skip) continue;
        const float2 *A = buf + k * BUFST + sr, *B = buf + k * BUFST + (TS == 64 && !diag ? G::PANEL : 0) + tc;
#pragma unroll 1
        for (int h = 0; h < G::RUNS; h++) {
            float2 f[4][4];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) f[i][j] = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int row = ((g * G::RUNS + h) * 8 + q) * TS;
                const float4 a0 = *(const float4 *)(A + row), a1 = *(const float4 *)(A + row + 8);
                const float4 b0v = *(const float4 *)(B + row), b1v = *(const float4 *)(B + row + 2 * LX);
                const float2 x[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                                     make_float2(a1.z, a1.w)};
                const float2 y[4] = {make_float2(b0v.x, b0v.y), make_float2(b0v.z, b0v.w), make_float2(b1v.x, b1v.y),
                                     make_float2(b1v.z, b1v.w)};
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        // conj(x) y
                        f[i][j].x = fmaf(x[i].x, y[j].x, fmaf(x[i].y, y[j].y, f[i][j].x));
                        f[i][j].y = fmaf(x[i].x, y[j].y, fmaf(-x[i].y, y[j].x, f[i][j].y));
                    }
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) f2_two_sum(hi[i][j], lo[i][j], f[i][j]);
        }
        if ((held += G::RUNS) >= kGHeld) {
            flush();
            held = 0;
        }
    }
    if (held) flush();
    auto row_of = [&](int i) { return sr + (i & 1) + 8 * (i >> 1); };
    auto col_of = [&](int j) { return tc + (j & 1) + 2 * LX * (j >> 1); };
    // sums that left the FP32 range: exponent of Inf and NaN
    int top = 0;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++)
            top = max(top, max(__double2hiint(tot[i][j].x) & 0x7fffffff, __double2hiint(tot[i][j].y) & 0x7fffffff));
    if (top >= 0x7ff00000) {
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int s = s0 + row_of(i), t = t0 + col_of(j);
                if ((!isfinite(tot[i][j].x) || !isfinite(tot[i][j].y)) && s < S && t < S)
                    tot[i][j] = gram_runs64(psi + s, psi + t, p0 + 8 * g * G::RUNS, p1, ld, G::RUNS, KP);
            }
    }
    if constexpr (G::NG == 1) {
        if (skip) return;
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int s = s0 + row_of(i), t = t0 + col_of(j);
                if (s < S && t < S) partial[((int64_t)blockIdx.z * S + s) * S + t] = tot[i][j];
            }
    } else {
        __syncthreads();
        double2 *red = (double2 *)smraw;   // [NG][TS][TS]
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) red[(g * TS + row_of(i)) * TS + col_of(j)] = tot[i][j];
        __syncthreads();
        for (int e = tid; e < TS * TS; e += 256) {
            const int s = s0 + e / TS, t = t0 + e % TS;
            if (s >= S || t >= S) continue;
            double2 a = red[e];
            for (int q = 1; q < G::NG; q++) {
                a.x += red[q * TS * TS + e].x;
                a.y += red[q * TS * TS + e].y;
            }
            partial[((int64_t)blockIdx.z * S + s) * S + t] = a;
        }
    }
}

// ------------------------------------- Gram matrix with FP64 accumulation
// Tile 8 x 8 of (s, t), 2 x 2 entries per thread, 16 groups of 16 threads
// that take the staged points in turn.  Bound by the FP64 pipe (two FMAs a
// clock per SM; 16 per thread and point), so the tile is small: it wastes
// little where S is small or not a multiple of it.  The values are converted
// to FP64 once, when they are staged.  phi = psi with herm: tiles s <= t.
// 61^3 x 8 complex128 states: 0.104 ms (1.87 ms with one 16 x 16 tile per 4096
// points, 56 blocks).
constexpr int kGD = 8, kGDP = 64;
template <typename R>
__global__ void __launch_bounds__(256) k_gram64(const R *__restrict__ psi, const R *__restrict__ phi, int64_t P, int ld,
                                                int S, int herm, double2 *__restrict__ partial, int nblk) {
    __shared__ double2 A[kGDP][kGD], B[kGDP][kGD + 1];
    const int nt = (S + kGD - 1) / kGD;
    int ti, tj;
    if (herm) {
        int rest = blockIdx.x;
        ti = 0;
        while (rest >= nt - ti) {
            rest -= nt - ti;
            ti++;
        }
        tj = ti + rest;
    } else {
        ti = blockIdx.x / nt;
        tj = blockIdx.x % nt;
    }
    const int s0 = ti * kGD, t0 = tj * kGD;
    const int tid = threadIdx.x, g = tid / 16, r = tid % 16;
    const int sr = r / 4, tc = r % 4;   // rows sr, sr + 4; columns tc, tc + 4
    const bool diag = herm && ti == tj;   // rows sr + 4, column tc: below the diagonal, not formed
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.z * per;
    const int64_t p1 = p0 + per < P ? p0 + per : P;
    const int lk = tid / kGD, lc = tid % kGD;   // staging: points lk, lk + 32; column lc
    double2 va[2], vb[2];
    auto load = [&](int64_t pc) {
#pragma unroll
        for (int i = 0; i < 2; i++) {
            const int64_t p = pc + lk + 32 * i;
            va[i] = vb[i] = make_double2(0.0, 0.0);
            if (p < p1) {
                if (s0 + lc < S) {
                    const R *x = psi + (p * ld + s0 + lc) * 2;
                    va[i] = make_double2((double)x[0], (double)x[1]);
                }
                if (t0 + lc < S) {
                    const R *y = phi + (p * ld + t0 + lc) * 2;
                    vb[i] = make_double2((double)y[0], (double)y[1]);
                }
            }
        }
    };
    double2 acc[2][2];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 2; j++) acc[i][j] = make_double2(0.0, 0.0);
    load(p0);
    for (int64_t pc = p0; pc < p1; pc += kGDP) {
#pragma unroll
        for (int i = 0; i < 2; i++) {
            A[lk + 32 * i][lc] = va[i];
            B[lk + 32 * i][lc] = vb[i];
        }
        __syncthreads();
        if (pc + kGDP < p1) load(pc + kGDP);
#pragma unroll
        for (int q = 0; q < kGDP / 16; q++) {
            const int k = g + 16 * q;
            const double2 x[2] = {A[k][sr], A[k][sr + 4]}, y[2] = {B[k][tc], B[k][tc + 4]};
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    if (i == 1 && j == 0 && diag) continue;
                    acc[i][j].x = fma(x[i].x, y[j].x, fma(x[i].y, y[j].y, acc[i][j].x));
                    acc[i][j].y = fma(x[i].x, y[j].y, fma(-x[i].y, y[j].x, acc[i][j].y));
                }
        }
        __syncthreads();
    }
    // the groups' sums in group order, through the staging buffers (8 KB each)
    double2 *red = &A[0][0];                    // 8 groups x 64 entries at a time
    static_assert(sizeof(A) >= 8 * 64 * sizeof(double2), "reduction buffer");
    double2 tot = make_double2(0.0, 0.0);
    for (int half = 0; half < 2; half++) {
        if (g / 8 == half)
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 2; j++) red[(g % 8) * 64 + (sr + 4 * i) * 8 + tc + 4 * j] = acc[i][j];
        __syncthreads();
        if (tid < 64)
            for (int q = 0; q < 8; q++) {
                tot.x += red[q * 64 + tid].x;
                tot.y += red[q * 64 + tid].y;
            }
        __syncthreads();
    }
    const int s = s0 + tid / 8, t = t0 + tid % 8;
    if (tid < 64 && s < S && t < S) partial[((int64_t)blockIdx.z * S + s) * S + t] = tot;
}

// ------------------------------------------- Cholesky factor and inverse
// One block factors G = L L^H (right-looking), with L's columns contiguous
// (L[j][i], i >= j) in shared memory when they fit, else in place of W's
// storage.  FP64-bound on one SM at 128 states (0.36 M complex updates): 0.96
// ms, and 0.15 ms for the inverse (4.8 ms together when one thread formed each
// pivot and each column of the inverse from global memory).
// drift (optional) records |G_ss - 1|; *status = 1 when G is not finite or
// not positive definite.
__global__ void __launch_bounds__(1024) k_chol(const double2 *__restrict__ G, double2 *__restrict__ L, int S,
                                               double *drift, int *status, int in_smem) {
    extern __shared__ double2 sm[];
    __shared__ int bad;
    const int tid = threadIdx.x, nth = blockDim.x;
    if (tid == 0) bad = 0;
    __syncthreads();
    if (drift != nullptr)
        for (int s = tid; s < S; s += nth) {
            const double e = fabs(G[(int64_t)s * S + s].x - 1.0);
            if (!(e <= drift[s])) drift[s] = e;   // NaN propagates
        }
    // column j of the lower triangle: packed in shared memory, S apart in L
    auto col = [&](int j) -> double2 * {
        return in_smem ? sm + ((int64_t)j * S - (int64_t)j * (j - 1) / 2 - j) : L + (int64_t)j * S;
    };
    for (int64_t e = tid; e < (int64_t)S * S; e += nth) {
        const double2 g = G[e];
        if (!isfinite(g.x) || !isfinite(g.y)) bad = 1;
        const int i = (int)(e / S), j = (int)(e % S);
        if (j <= i) col(j)[i] = g;
    }
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    for (int j = 0; j < S; j++) {
        double2 *cj = col(j);
        const double d = cj[j].x;
        if (bad || !(d > 0.0)) {   // the same in every thread
            __syncthreads();
            if (tid == 0) *status = 1;
            return;
        }
        const double ljj = sqrt(d);
        __syncthreads();
        for (int i = j + tid; i < S; i += nth) {
            if (i == j) cj[j] = make_double2(ljj, 0.0);
            else cj[i] = make_double2(cj[i].x / ljj, cj[i].y / ljj);
        }
        __syncthreads();
        // trailing columns k > j: L[i][k] -= L[i][j] conj(L[k][j]), a warp per column
        for (int k = j + 1 + warp; k < S; k += nw) {
            double2 *ck = col(k);
            const double2 b = cj[k];
            for (int i = k + lane; i < S; i += 32) {
                const double2 a = cj[i];
                double2 c = ck[i];
                c.x = fma(-a.x, b.x, fma(-a.y, b.y, c.x));
                c.y = fma(-a.y, b.x, fma(a.x, b.y, c.y));
                ck[i] = c;
            }
        }
        __syncthreads();
    }
    if (in_smem)
        for (int j = warp; j < S; j += nw)
            for (int i = j + lane; i < S; i += 32) L[(int64_t)j * S + i] = col(j)[i];
}

// W = L^-1 (lower), one warp per column c: forward substitution with the
// right-hand side spread over the lanes (rows c + lane, c + lane + 32, ...).
// L is column-contiguous.  NR: rows per lane held in registers.
template <int NR>
__global__ void __launch_bounds__(128) k_tri_inv(const double2 *__restrict__ L, double2 *__restrict__ W, int S) {
    const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= S) return;
    for (int i = lane; i < c; i += 32) W[(int64_t)i * S + c] = make_double2(0.0, 0.0);
    double2 r[NR];   // -(right-hand side) of rows c + lane + 32 q; unit vector at row c
#pragma unroll
    for (int q = 0; q < NR; q++) r[q] = make_double2(0.0, 0.0);
    if (lane == 0) r[0].x = 1.0;
#pragma unroll
    for (int q0 = 0; q0 < NR; q0++) {
        for (int l = 0; l < 32; l++) {
            const int i = c + 32 * q0 + l;
            if (i >= S) break;
            const double2 *li = L + (int64_t)i * S;
            const double lii = li[i].x;
            double2 w = r[q0];
            w.x = __shfl_sync(0xffffffffu, w.x, l) / lii;
            w.y = __shfl_sync(0xffffffffu, w.y, l) / lii;
            if (lane == l) r[q0] = w;
#pragma unroll
            for (int q = q0; q < NR; q++) {
                const int k = c + lane + 32 * q;
                if (k > i && k < S) {
                    const double2 a = li[k];
                    r[q].x = fma(-a.x, w.x, fma(a.y, w.y, r[q].x));
                    r[q].y = fma(-a.x, w.y, fma(-a.y, w.x, r[q].y));
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NR; q++) {
        const int k = c + lane + 32 * q;
        if (k < S) W[(int64_t)k * S + c] = r[q];
    }
}

// The same for any S, with the right-hand side in W's column.
__global__ void __launch_bounds__(128) k_tri_inv_any(const double2 *__restrict__ L, double2 *W, int S) {
    const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= S) return;
    for (int i = lane; i < S; i += 32) W[(int64_t)i * S + c] = make_double2(i == c ? 1.0 : 0.0, 0.0);
    __syncwarp();
    for (int i = c; i < S; i++) {
        const double2 *li = L + (int64_t)i * S;
        double2 w = W[(int64_t)i * S + c];
        w.x /= li[i].x;
        w.y /= li[i].x;
        __syncwarp();
        if (lane == 0) W[(int64_t)i * S + c] = w;
        for (int k = i + 1 + lane; k < S; k += 32) {
            const double2 a = li[k];
            double2 r = W[(int64_t)k * S + c];
            r.x = fma(-a.x, w.x, fma(a.y, w.y, r.x));
            r.y = fma(-a.x, w.y, fma(-a.y, w.x, r.y));
            W[(int64_t)k * S + c] = r;
        }
        __syncwarp();
    }
}

// ------------------------------------------ triangular update, complex64
// psi[p, s] <- sum_{t <= s} psi[p, t] conj(W[s][t]) in place, FP32.
// A block stages the whole rows of PT points in shared memory, transposed
// and split into re and im (X[t][p]), then forms column tiles of NT states.
// Warp w of a tile owns the 8-column groups w and NT/8 - 1 - w: the sums end
// at t = s, so a low and a high group together cost every warp the same.  A
// thread owns 8 points x (2 + 2) columns, as packed pairs of points; conj(W)
// comes from global memory, transposed and rounded, in chunks of 8 t,
// double-buffered, two columns per 16-byte shared-memory read.  Fewer states take narrower tiles and more points per
// block.  192^3 x 128 states: 12.0 ms, shared-memory reads the limit (195 ms
// with one output per thread and operands from L1; 14.1 with W staged twice
// as pairs).
constexpr int kTC = 8;   // t per staged chunk of W
template <int NT>
struct TriShape {
    static constexpr int NWS = NT / 16, NWP = 8 / NWS, PT = 64 * NWP, XS = PT + 4;
    static size_t bytes(int S) { return (size_t)((S + 7) & ~7) * 2 * XS * 4 + 2 * kTC * NT * 8; }
};

// Wt[t][s] = conj(W[s][t]) for t <= s < S, zero elsewhere
__global__ void k_wconj(const double2 *__restrict__ W, float2 *__restrict__ Wt, int S, int Sp) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)Sp * Sp) return;
    const int t = (int)(e / Sp), s = (int)(e % Sp);
    float2 v = make_float2(0.f, 0.f);
    if (s < S && t <= s) {
        const double2 w = W[(int64_t)s * S + t];
        v = make_float2((float)w.x, (float)-w.y);
    }
    Wt[e] = v;
}

template <int NT>
__global__ void __launch_bounds__(256, 2) k_tri32(float2 *psi, int64_t P, int ld, int S, const float2 *__restrict__ Wt,
                                                  int Sp) {
    using G = TriShape<NT>;
    constexpr int PT = G::PT, XS = G::XS;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int S8 = (S + 7) & ~7;
    float *Xr = (float *)smraw, *Xi = Xr + (size_t)S8 * XS;
    float2 *Wb = (float2 *)(Xi + (size_t)S8 * XS);   // [2][kTC][NT]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t p0 = (int64_t)blockIdx.x * PT;
    // stage: a warp takes 8 points x 8 states at a time (64-byte reads; the
    // transposed stores fall on 32 different banks)
    {
        const int ng = S8 / 8, tt = 2 * (lane & 3), pp = lane >> 2;
        for (int e = warp; e < ng * (PT / 8); e += 8) {
            const int t = 8 * (e % ng) + tt, pl = 8 * (e / ng) + pp;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p0 + pl < P && t < S) {
                v = *(const float4 *)(psi + (p0 + pl) * ld + t);
                if (t + 1 >= S) v.z = v.w = 0.f;
            }
            Xr[t * XS + pl] = v.x;
            Xi[t * XS + pl] = v.y;
            Xr[(t + 1) * XS + pl] = v.z;
            Xi[(t + 1) * XS + pl] = v.w;
        }
    }
    const int ws = warp % G::NWS, wp = warp / G::NWS;
    const int pl0 = 64 * wp + 4 * (lane & 7);                     // points pl0 .. +3 and pl0 + 32 .. +35
    const int cl = 8 * ws + 2 * (lane >> 3), ch = NT - 8 - 8 * ws + 2 * (lane >> 3);   // columns of the tile
    const unsigned wsm = (unsigned)__cvta_generic_to_shared(Wb);
    for (int n0 = 0; n0 < S; n0 += NT) {
        const int kend = min(n0 + NT, S8);
        auto stage_w = [&](int t0, int buf) {
            for (int e = 2 * tid; e < kTC * NT; e += 512)
                cp_async16(wsm + (unsigned)((buf * kTC * NT + e) * 8), Wt + (int64_t)(t0 + e / NT) * Sp + n0 + e % NT, 16);
            cp_async_commit();
        };
        float2 rl[2][4], il[2][4], rh[2][4], ih[2][4];   // [column][point pair]
#pragma unroll
        for (int c = 0; c < 2; c++)
#pragma unroll
            for (int q = 0; q < 4; q++) rl[c][q] = il[c][q] = rh[c][q] = ih[c][q] = make_float2(0.f, 0.f);
        stage_w(0, 0);
        for (int t0 = 0, buf = 0; t0 < kend; t0 += kTC, buf ^= 1) {
            cp_async_wait<0>();
            __syncthreads();
            if (t0 + kTC < kend) stage_w(t0 + kTC, buf ^ 1);
            const bool low = t0 < n0 + 8 * ws + 8 && n0 + 8 * ws < S;
            const bool high = t0 < n0 + NT - 8 * ws && n0 + NT - 8 - 8 * ws < S;
            if (!low && !high) continue;
            const float2 *wb = Wb + buf * kTC * NT;
// columns COL and COL + 1
#define TRI_STEP(COL, R_, I_)                                                              \
    {                                                                                      \
        const float4 w2 = *(const float4 *)(wb + q * NT + (COL));                          \
        _Pragma("unroll") for (int c = 0; c < 2; c++) {                                    \
            const float2 wr = c ? make_float2(w2.z, w2.z) : make_float2(w2.x, w2.x);       \
            const float2 wi = c ? make_float2(w2.w, w2.w) : make_float2(w2.y, w2.y);       \
            _Pragma("unroll") for (int k = 0; k < 4; k++) {                                \
                R_[c][k] = f2_fma(xr[k], wr, f2_fma(nx[k], wi, R_[c][k]));                 \
                I_[c][k] = f2_fma(xr[k], wi, f2_fma(xi[k], wr, I_[c][k]));                 \
            }                                                                              \
        }                                                                                  \
    }
#define TRI_X()                                                                                     \
    const float *xrp = Xr + (t0 + q) * XS + pl0, *xip = Xi + (t0 + q) * XS + pl0;                   \
    const float4 ra = *(const float4 *)xrp, rb = *(const float4 *)(xrp + 32);                       \
    const float4 ia = *(const float4 *)xip, ib = *(const float4 *)(xip + 32);                       \
    const float2 xr[4] = {make_float2(ra.x, ra.y), make_float2(ra.z, ra.w), make_float2(rb.x, rb.y), \
                          make_float2(rb.z, rb.w)};                                                 \
    const float2 xi[4] = {make_float2(ia.x, ia.y), make_float2(ia.z, ia.w), make_float2(ib.x, ib.y), \
                          make_float2(ib.z, ib.w)};                                                 \
    const float2 nx[4] = {f2_neg(xi[0]), f2_neg(xi[1]), f2_neg(xi[2]), f2_neg(xi[3])};
            if (low && high) {
#pragma unroll 2
                for (int q = 0; q < kTC; q++) {
                    TRI_X()
                    TRI_STEP(cl, rl, il)
                    TRI_STEP(ch, rh, ih)
                }
            } else if (high) {
#pragma unroll 2
                for (int q = 0; q < kTC; q++) {
                    TRI_X()
                    TRI_STEP(ch, rh, ih)
                }
            } else {
#pragma unroll 2
                for (int q = 0; q < kTC; q++) {
                    TRI_X()
                    TRI_STEP(cl, rl, il)
                }
            }
#undef TRI_STEP
#undef TRI_X
        }
        __syncthreads();   // the chunk buffers are free for the next tile
        auto put = [&](int s, float2 (&R_)[2][4], float2 (&I_)[2][4]) {
            if (s >= S) return;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int64_t p = p0 + pl0 + (k >> 2) * 32 + (k & 3);
                if (p >= P) continue;
                const int q = k >> 1;
                const float4 v = k & 1 ? make_float4(R_[0][q].y, I_[0][q].y, R_[1][q].y, I_[1][q].y)
                                       : make_float4(R_[0][q].x, I_[0][q].x, R_[1][q].x, I_[1][q].x);
                float2 *d = psi + p * ld + s;
                if (s + 1 < S) *(float4 *)d = v;
                else *d = make_float2(v.x, v.y);
            }
        };
        put(n0 + cl, rl, il);
        put(n0 + ch, rh, ih);
    }
}

// Fallback for blocks of more states than the staged rows hold: one output
// per thread, rows in shared memory, W from global memory.
__global__ void __launch_bounds__(256) k_tri_rows32(float2 *psi, int64_t P, int ld, int S,
                                                    const double2 *__restrict__ W, int pt) {
    extern __shared__ float2 rows[];   // pt x S
    const int64_t p0 = (int64_t)blockIdx.x * pt;
    const int n = pt * S;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int q = e / S, t = e - q * S;
        const int64_t p = p0 + q;
        rows[e] = p < P ? psi[p * ld + t] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int s = e % S, q = e / S;
        const int64_t p = p0 + q;
        if (p >= P) continue;
        const float2 *row = rows + q * S;
        float re = 0.f, im = 0.f;
        for (int t = 0; t <= s; t++) {
            const float2 a = row[t];
            const double2 w = W[(int64_t)s * S + t];
            const float bx = (float)w.x, by = (float)-w.y;
            re = fmaf(a.x, bx, fmaf(-a.y, by, re));
            im = fmaf(a.x, by, fmaf(a.y, bx, im));
        }
        psi[p * ld + s] = make_float2(re, im);
    }
}

int gram_base(int64_t P) { return (int)std::max<int64_t>(1, std::min<int64_t>(296, (P + 4095) / 4096)); }

constexpr size_t kSmemMax = 227 * 1024;
// column tile of the triangular update: the narrowest that holds S, 128 beyond
int tri_nt(int S) { return S <= 16 ? 16 : S <= 32 ? 32 : S <= 64 ? 64 : 128; }
size_t tri_bytes(int S) {
    switch (tri_nt(S)) {
    case 16: return TriShape<16>::bytes(S);
    case 32: return TriShape<32>::bytes(S);
    case 64: return TriShape<64>::bytes(S);
    default: return TriShape<128>::bytes(S);
    }
}
int tri_sp(int S) {
    const int nt = tri_nt(S);
    return (S + nt - 1) / nt * nt;
}

template <int NT>
cudaError_t tri_launch(float2 *psi, int64_t P, int ld, int S, const float2 *Wt, int Sp, cudaStream_t st) {
    const size_t smem = TriShape<NT>::bytes(S);
    cudaError_t e = cudaFuncSetAttribute(k_tri32<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t nb = (P + TriShape<NT>::PT - 1) / TriShape<NT>::PT;
    k_tri32<NT><<<(unsigned)nb, 256, smem, st>>>(psi, P, ld, S, Wt, Sp);
    return cudaGetLastError();
}

template <int TS>
cudaError_t gram32_launch(const float2 *psi, int64_t P, int ld, int S, double2 *partial, int nblk, cudaStream_t st) {
    using G = G32Shape<TS>;
    const int nb0 = gram_base(P);
    cudaError_t e = cudaFuncSetAttribute(k_gram32<TS>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::BYTES);
    if (e != cudaSuccess) return e;
    const int nt = (S + TS - 1) / TS;
    k_gram32<TS><<<dim3(nt * (nt + 1) / 2, 1, nblk), 256, G::BYTES, st>>>(psi, P, ld, S, partial, nb0, nblk / nb0);
    return cudaGetLastError();
}

}  // namespace

// Point blocks of the Gram kernels.  The complex64 kernel's runs of 8 points
// start afresh every gram_base(P)-th part of the points; each part is cut
// into pieces (at multiples of 8 points, 256 or more) until the launch has
// about four blocks per SM over all column tiles.
int gram_blocks(int64_t P, int S) {
    const int nt = (S + 63) / 64, tiles = nt * (nt + 1) / 2, nb0 = gram_base(P);
    const int64_t per = (P + nb0 - 1) / nb0;
    const int64_t nsub = std::min<int64_t>((608 + nb0 * tiles - 1) / (nb0 * tiles), (per + 255) / 256);
    return nb0 * (int)std::max<int64_t>(1, nsub);
}

int norm_blocks(int64_t P) {
    int64_t n = (P + 2047) / 2048;
    if (n > 608) n = 608;
    if (n < 1) n = 1;
    return (int)n;
}

cudaError_t launch_sum_blocks(const double *partial, int nblk, int64_t n, double scale, double *out, cudaStream_t st) {
    k_sum_rows<<<(unsigned)((n + 31) / 32), dim3(32, 32), 0, st>>>(partial, nblk, n, scale, out);
    return cudaGetLastError();
}

cudaError_t launch_norms_c64(const void *psi, int64_t P, int ld, int S, double h3, double *partial, int nblk,
                             double *out, cudaStream_t st) {
    const int SV = (S + 1) / 2;
    const int bx = SV < 32 ? SV : 32;
    k_norms32<<<nblk, dim3(bx, 256 / bx), 0, st>>>((const float4 *)psi, P, ld / 2, SV, S, partial, nblk);
    return launch_sum_blocks(partial, nblk, S, h3, out, st);
}

cudaError_t launch_gram_c64(const void *psi, int64_t P, int ld, int S, double h3, double *partial, int nblk,
                            double *G, const double *norms, cudaStream_t st) {
    double2 *pp = (double2 *)partial;
    const float2 *x = (const float2 *)psi;
    cudaError_t e = S <= 16   ? gram32_launch<16>(x, P, ld, S, pp, nblk, st)
                    : S <= 32 ? gram32_launch<32>(x, P, ld, S, pp, nblk, st)
                              : gram32_launch<64>(x, P, ld, S, pp, nblk, st);
    if (e != cudaSuccess) return e;
    k_sum_herm<<<dim3((S + 15) / 16, S), dim3(16, 16), 0, st>>>(pp, nblk, S, h3, norms, (double2 *)G);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_gram(const void *psi, int64_t P, int ld, int S, double h3, double *partial, int nblk, double *G,
                        cudaStream_t st) {
    const int nt = (S + kGD - 1) / kGD;
    k_gram64<R><<<dim3(nt * (nt + 1) / 2, 1, nblk), 256, 0, st>>>((const R *)psi, (const R *)psi, P, ld, S, 1,
                                                                 (double2 *)partial, nblk);
    k_sum_herm<<<dim3((S + 15) / 16, S), dim3(16, 16), 0, st>>>((const double2 *)partial, nblk, S, h3, nullptr,
                                                                (double2 *)G);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_cross_gram(const void *psi, const void *phi, int64_t P, int ld, int S, double h3, double *partial,
                              int nblk, double *G, cudaStream_t st) {
    const int nt = (S + kGD - 1) / kGD;
    k_gram64<R><<<dim3(nt * nt, 1, nblk), 256, 0, st>>>((const R *)psi, (const R *)phi, P, ld, S, 0, (double2 *)partial,
                                                        nblk);
    return launch_sum_blocks(partial, nblk, (int64_t)S * S * 2, h3, G, st);
}

// G (S x S complex double) = L L^H; W = L^-1.  L overwrites G (its columns
// contiguous).
cudaError_t launch_chol_inv(double *G, double *W, int S, double *drift, int *status, cudaStream_t st) {
    const size_t packed = (size_t)S * (S + 1) / 2 * sizeof(double2);
    const int in_smem = packed <= kSmemMax - 1024;
    if (in_smem) {
        cudaError_t e = cudaFuncSetAttribute(k_chol, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)packed);
        if (e != cudaSuccess) return e;
    }
    // the factor is formed in W and the inverse in G's place, then swapped by
    // the copy below; in shared memory it goes straight to G
    const int nth = S <= 16 ? 128 : S <= 48 ? 512 : 1024;
    double2 *L = (double2 *)(in_smem ? G : W);
    k_chol<<<1, nth, in_smem ? packed : 0, st>>>((const double2 *)G, L, S, drift, status, in_smem);
    double2 *inv = (double2 *)(in_smem ? W : G);
    const unsigned nb = (unsigned)((S + 3) / 4);
    if (S <= 32) k_tri_inv<1><<<nb, 128, 0, st>>>(L, inv, S);
    else if (S <= 64) k_tri_inv<2><<<nb, 128, 0, st>>>(L, inv, S);
    else if (S <= 128) k_tri_inv<4><<<nb, 128, 0, st>>>(L, inv, S);
    else if (S <= 256) k_tri_inv<8><<<nb, 128, 0, st>>>(L, inv, S);
    else k_tri_inv_any<<<nb, 128, 0, st>>>(L, inv, S);
    if (inv != (double2 *)W) {
        cudaError_t e = cudaMemcpyAsync(W, G, (size_t)S * S * sizeof(double2), cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

size_t tri_c64_bytes(int S) {
    return tri_bytes(S) <= kSmemMax ? (size_t)tri_sp(S) * tri_sp(S) * sizeof(float2) : 0;
}

cudaError_t launch_tri_apply_c64(void *psi, int64_t P, int ld, int S, const double *W, void *Wt_buf, cudaStream_t st) {
    float2 *x = (float2 *)psi;
    if (tri_bytes(S) > kSmemMax) {
        int pt = 8192 / S;
        if (pt < 1) pt = 1;
        const size_t smem = (size_t)pt * S * sizeof(float2);
        if (smem > kSmemMax) return cudaErrorInvalidValue;
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(k_tri_rows32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        k_tri_rows32<<<(unsigned)((P + pt - 1) / pt), 256, smem, st>>>(x, P, ld, S, (const double2 *)W, pt);
        return cudaGetLastError();
    }
    const int Sp = tri_sp(S);
    float2 *Wt = (float2 *)Wt_buf;
    k_wconj<<<(unsigned)(((int64_t)Sp * Sp + 255) / 256), 256, 0, st>>>((const double2 *)W, Wt, S, Sp);
    switch (tri_nt(S)) {
    case 16: return tri_launch<16>(x, P, ld, S, Wt, Sp, st);
    case 32: return tri_launch<32>(x, P, ld, S, Wt, Sp, st);
    case 64: return tri_launch<64>(x, P, ld, S, Wt, Sp, st);
    default: return tri_launch<128>(x, P, ld, S, Wt, Sp, st);
    }
}

template cudaError_t launch_gram<double>(const void *, int64_t, int, int, double, double *, int, double *, cudaStream_t);
template cudaError_t launch_cross_gram<float>(const void *, const void *, int64_t, int, int, double, double *, int,
                                              double *, cudaStream_t);
template cudaError_t launch_cross_gram<double>(const void *, const void *, int64_t, int, int, double, double *, int,
                                               double *, cudaStream_t);

}  // namespace rsg
