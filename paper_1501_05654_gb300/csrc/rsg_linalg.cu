// FP64 reductions and small dense linear algebra on state blocks.
//
// The Cholesky factor of the Gram matrix, its inverse and the sums over points
// are FP64 for both compute types; complex64 norms and Gram matrices reach
// them through short FP32 sums (rsg_qr.cu) (arXiv:1501.05654,
// Sec. "Parallelization, optimizations and graphics processing units": real-time propagation preserves orthogonality, so the
// states are re-orthonormalised only now and then; here Cholesky-QR, which
// equals Gram-Schmidt in index order; the Gram matrices, the factor and the
// complex64 update are in rsg_qr.cu).  The adjoint inner products of the
// control gradient (Sec. "Quantum optimal control", Eq. (qoctgradient)) are
// FP64 reductions as well.
#include <algorithm>

#include "rsg_chain.cuh"
#include "rsg_internal.h"
#include "rsg_vec.cuh"

namespace rsg {

namespace {

template <typename R>
__device__ __forceinline__ void ld_c(const R *p, double &re, double &im) {
    re = (double)p[0];
    im = (double)p[1];
}

}  // namespace

// psi[p, s] <- sum_t psi[p, t] M[t][s] in place, FP64 sums: the Ritz rotation
// (M = Q) or, TRI, the Cholesky-QR update (M[t][s] = conj(W[s][t]), t <= s).
// A block stages the rows of PT points and chunks of M in shared memory; a
// thread forms four neighbouring states of a point, so that 16 FP64 FMAs
// share five 16-byte reads.  Bound by the FP64 pipe (two FMAs a clock per SM).
constexpr int kRowsNT = 256, kRowsChunk = 2048;   // threads, complex values of M per chunk
template <typename R, bool TRI>
__global__ void __launch_bounds__(kRowsNT) k_rows(R *psi, int64_t P, int ld, int S, const double2 *__restrict__ M,
                                                  int pt, int nt) {
    extern __shared__ double2 rsm[];
    double2 *rows = rsm, *mc = rsm + (size_t)pt * S;   // [pt][S], [nt][S]
    const int tid = threadIdx.x, ng = (S + 3) / 4;
    const int64_t p0 = (int64_t)blockIdx.x * pt;
    for (int e = tid; e < pt * S; e += kRowsNT) {
        const int q = e / S;
        double2 v = make_double2(0.0, 0.0);
        if (p0 + q < P) ld_c(psi + ((p0 + q) * ld + (e - q * S)) * 2, v.x, v.y);
        rows[e] = v;
    }
    // items (point, group of four states): pt * ng of them, kRowsNT at a time
    for (int i0 = 0; i0 < pt * ng; i0 += kRowsNT) {
        const int i = i0 + tid, q = i / ng, s0 = 4 * (i - q * ng);
        const bool on = i < pt * ng && p0 + q < P;
        double re[4] = {0.0, 0.0, 0.0, 0.0}, im[4] = {0.0, 0.0, 0.0, 0.0};
        for (int t0 = 0; t0 < S; t0 += nt) {
            const int t1 = min(S, t0 + nt);
            if (nt < S || i0 == 0) {   // a chunk that holds all of M is staged once
                __syncthreads();
                for (int e = tid; e < (t1 - t0) * S; e += kRowsNT) {
                    const int t = t0 + e / S, s = e % S;
                    double2 m;
                    if (TRI) {
                        m = t <= s ? M[(int64_t)s * S + t] : make_double2(0.0, 0.0);
                        m.y = -m.y;
                    } else {
                        m = M[(int64_t)t * S + s];
                    }
                    mc[e] = m;
                }
                __syncthreads();
            }
            if (!on) continue;
            const int te = TRI ? min(t1, s0 + 4) : t1;
            const double2 *row = rows + (size_t)q * S;
#pragma unroll 2
            for (int t = t0; t < te; t++) {
                const double2 a = row[t], *m = mc + (size_t)(t - t0) * S + s0;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const double2 w = s0 + k < S ? m[k] : make_double2(0.0, 0.0);
                    re[k] = fma(a.x, w.x, fma(-a.y, w.y, re[k]));
                    im[k] = fma(a.x, w.y, fma(a.y, w.x, im[k]));
                }
            }
        }
        if (on)
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (s0 + k < S) {
                    R *d = psi + ((p0 + q) * ld + s0 + k) * 2;
                    d[0] = (R)re[k];
                    d[1] = (R)im[k];
                }
    }
}

// The same for blocks so wide that a row and a row of M do not fit in shared
// memory together (above 7,264 states): one point per block, M from global
// memory.
template <typename R, bool TRI>
__global__ void __launch_bounds__(kRowsNT) k_rows_wide(R *psi, int ld, int S, const double2 *__restrict__ M) {
    extern __shared__ double2 rsm[];
    R *row = psi + (int64_t)blockIdx.x * ld * 2;
    for (int t = threadIdx.x; t < S; t += kRowsNT) ld_c(row + 2 * t, rsm[t].x, rsm[t].y);
    __syncthreads();
    for (int s = threadIdx.x; s < S; s += kRowsNT) {
        double re = 0.0, im = 0.0;
        const int te = TRI ? s + 1 : S;
        for (int t = 0; t < te; t++) {
            const double2 a = rsm[t];
            double2 m = M[TRI ? (int64_t)s * S + t : (int64_t)t * S + s];
            if (TRI) m.y = -m.y;
            re = fma(a.x, m.x, fma(-a.y, m.y, re));
            im = fma(a.x, m.y, fma(a.y, m.x, im));
        }
        row[2 * s] = (R)re;
        row[2 * s + 1] = (R)im;
    }
}

template <typename R, bool TRI>
cudaError_t rows_launch(void *psi, int64_t P, int ld, int S, const double *M, cudaStream_t st) {
    // one item per thread, fewer points where the rows would not fit
    const int ng = (S + 3) / 4, pt = std::max(1, kRowsNT / ng), nt = std::min(S, std::max(1, kRowsChunk / S));
    const size_t smem = ((size_t)pt * S + (size_t)nt * S) * sizeof(double2);
    if (smem > 227 * 1024) {
        const size_t row = (size_t)S * sizeof(double2);
        if (row > 227 * 1024) return cudaErrorInvalidValue;
        cudaError_t e = cudaFuncSetAttribute(k_rows_wide<R, TRI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row);
        if (e != cudaSuccess) return e;
        k_rows_wide<R, TRI><<<(unsigned)P, kRowsNT, row, st>>>((R *)psi, ld, S, (const double2 *)M);
        return cudaGetLastError();
    }
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_rows<R, TRI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_rows<R, TRI><<<(unsigned)((P + pt - 1) / pt), kRowsNT, smem, st>>>((R *)psi, P, ld, S, (const double2 *)M, pt, nt);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_rotate(void *psi, int64_t P, int ld, int S, const double *Q, cudaStream_t st) {
    return rows_launch<R, false>(psi, P, ld, S, Q, st);
}

// partial[blk][s] = sum over the block's points of |hx[p,s] - lam[s] x[p,s]|^2
template <typename R>
__global__ void __launch_bounds__(256) k_resid(const R *__restrict__ x, const R *__restrict__ hx, int64_t P,
                                               int ld, int S, const double *__restrict__ lam,
                                               double *__restrict__ partial, int nblk) {
    __shared__ double red[256];
    const int s = blockIdx.y;
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.x * per, p1 = p0 + per < P ? p0 + per : P;
    const double l = lam[s];
    double acc = 0.0;
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        double xr, xi, yr, yi;
        ld_c(x + (p * ld + s) * 2, xr, xi);
        ld_c(hx + (p * ld + s) * 2, yr, yi);
        const double rr = yr - l * xr, ri = yi - l * xi;
        acc += rr * rr + ri * ri;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[(int64_t)blockIdx.x * S + s] = red[0];
}

// FP64 to FP32 in integer arithmetic (FP32 to FP64: widen, rsg_vec.cuh).  A conversion instruction takes two
// slots of the FP64 pipe (two a clock per SM), which bounds the complex64
// vector updates below; exponents that need denormal or special handling take
// the instruction.  R = 14 sphere x 8 states: update 293 to 91 us (with the
// unit scale of x dropped and 16-byte accesses), bilinear form 251 to 139 us.
__device__ __forceinline__ double widen(double d) { return d; }
// one complex value (8- or 16-byte aligned) in one load: the adjoint's
// gradient kernel waits for loads (9 a point instead of 17; 64^3 complex128 25.0
// to 24.0 us on one-state blocks, 26.5 to 25.0 on two-column blocks)
__device__ __forceinline__ void ld_wide(const float *q, double &re, double &im) {
    const float2 v = *reinterpret_cast<const float2 *>(q);
    re = widen(v.x);
    im = widen(v.y);
}
__device__ __forceinline__ void ld_wide(const double *q, double &re, double &im) {
    const double2 v = *reinterpret_cast<const double2 *>(q);
    re = v.x;
    im = v.y;
}
// round to nearest even
__device__ __forceinline__ float narrow(double d, float) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned e = hi & 0x7ff00000u;
    // FP32 exponents 1 .. 253: normal, and a carry stays finite
    if (e < 0x38100000u || e > 0x47d00000u) return (hi & 0x7fffffffu) == 0u && lo == 0u ? __uint_as_float(hi) : (float)d;
    const unsigned m = ((hi & 0x7fffffffu) - 0x38000000u) << 3 | lo >> 29;   // truncated
    const unsigned rest = lo & 0x1fffffffu;
    return __uint_as_float((hi & 0x80000000u) | (m + (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u)))));
}
__device__ __forceinline__ double narrow(double d, double) { return d; }

// partial[blk][s] (complex double) = sum over the block's points of
// x[p,s] y[p,s] (the bilinear form of complex symmetric systems, no
// conjugate).  A thread takes NS neighbouring states of every 256th point,
// which a 16-byte load of complex64 brings together.
template <typename R, int NS>
__global__ void __launch_bounds__(256) k_bilinear(const R *__restrict__ x, const R *__restrict__ y, int64_t P,
                                                  int ld, int S, double *__restrict__ partial, int nblk) {
    __shared__ double red[2 * NS][256];
    const int s0 = blockIdx.y * NS;
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.x * per, p1 = p0 + per < P ? p0 + per : P;
    double ar[NS], ai[NS];
#pragma unroll
    for (int k = 0; k < NS; k++) ar[k] = ai[k] = 0.0;
#pragma unroll 4
    for (int64_t p = p0 + threadIdx.x; p < p1; p += 256) {
        R xv[2 * NS], yv[2 * NS];
        const R *xp = x + (p * ld + s0) * 2, *yp = y + (p * ld + s0) * 2;
        if constexpr (NS == 2 && sizeof(R) == 4) {
            const float4 a = *(const float4 *)xp, b = *(const float4 *)yp;
            xv[0] = a.x, xv[1] = a.y, xv[2] = a.z, xv[3] = a.w;
            yv[0] = b.x, yv[1] = b.y, yv[2] = b.z, yv[3] = b.w;
        } else {
#pragma unroll
            for (int k = 0; k < 2 * NS; k++) xv[k] = xp[k], yv[k] = yp[k];
        }
#pragma unroll
        for (int k = 0; k < NS; k++) {
            const double xr = widen(xv[2 * k]), xi = widen(xv[2 * k + 1]), yr = widen(yv[2 * k]),
                         yi = widen(yv[2 * k + 1]);
            ar[k] += xr * yr - xi * yi;
            ai[k] += xr * yi + xi * yr;
        }
    }
#pragma unroll
    for (int k = 0; k < NS; k++) {
        red[2 * k][threadIdx.x] = ar[k];
        red[2 * k + 1][threadIdx.x] = ai[k];
    }
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < 2 * NS; k++) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 2 * NS && s0 + (int)threadIdx.x / 2 < S)
        partial[((int64_t)blockIdx.x * S + s0) * 2 + threadIdx.x] = red[threadIdx.x][0];
}

template <typename R>
cudaError_t launch_bilinear(const void *x, const void *y, int64_t P, int ld, int S, double h3, double *partial,
                            int nblk, double *out, cudaStream_t st) {
    constexpr int NS = sizeof(R) == 4 ? 2 : 1;   // complex64 rows are whole 16-byte vectors
    k_bilinear<R, NS><<<dim3(nblk, (S + NS - 1) / NS), 256, 0, st>>>((const R *)x, (const R *)y, P, ld, S, partial, nblk);
    return launch_sum_blocks(partial, nblk, 2 * (int64_t)S, h3, out, st);
}

// z[p,s] = x[p,s] + b[s] y[p,s] with complex per-state b (device, interleaved
// doubles), in FP64 and rounded once; z may alias x or y (each element is
// read before it is written, by the same thread).
template <typename R>
__global__ void __launch_bounds__(256) k_comb(const R *x, const R *y, R *z, int64_t P, int ld, int S,
                                              const double *__restrict__ b) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if constexpr (sizeof(R) == 4) {
        // two states per thread
        const int nv = (S + 1) / 2;
        if (i >= P * nv) return;
        const int64_t p = i / nv;
        const int s = 2 * (int)(i - p * nv);
        const int64_t o = (p * ld + s) * 2;
        const float4 xv = *(const float4 *)(x + o), yv = *(const float4 *)(y + o);
        const double2 b0 = *(const double2 *)(b + 2 * s);
        const double y0r = widen(yv.x), y0i = widen(yv.y);
        float4 r;
        r.x = narrow(fma(-b0.y, y0i, fma(b0.x, y0r, widen(xv.x))), 0.f);
        r.y = narrow(fma(b0.y, y0r, fma(b0.x, y0i, widen(xv.y))), 0.f);
        if (s + 1 < S) {
            const double2 b1 = *(const double2 *)(b + 2 * s + 2);
            const double y1r = widen(yv.z), y1i = widen(yv.w);
            r.z = narrow(fma(-b1.y, y1i, fma(b1.x, y1r, widen(xv.z))), 0.f);
            r.w = narrow(fma(b1.y, y1r, fma(b1.x, y1i, widen(xv.w))), 0.f);
            *(float4 *)(z + o) = r;
        } else {
            *(float2 *)(z + o) = make_float2(r.x, r.y);
        }
    } else {
        if (i >= P * S) return;
        const int64_t p = i / S;
        const int s = (int)(i - p * S);
        const int64_t o = (p * ld + s) * 2;
        const double2 xv = *(const double2 *)(x + o), yv = *(const double2 *)(y + o);
        const double br = b[2 * s], bi = b[2 * s + 1];
        *(double2 *)(z + o) = make_double2(fma(-bi, yv.y, fma(br, yv.x, xv.x)), fma(bi, yv.x, fma(br, yv.y, xv.y)));
    }
}

template <typename R>
cudaError_t launch_comb(const void *x, const void *y, void *z, int64_t P, int ld, int S, const double *b,
                        cudaStream_t st) {
    const int64_t n = P * (sizeof(R) == 4 ? (S + 1) / 2 : S);
    k_comb<R><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const R *)x, (const R *)y, (R *)z, P, ld, S, b);
    return cudaGetLastError();
}

// psi[p, s] *= M[p] for the first S states (mask absorber)
template <typename R>
__global__ void __launch_bounds__(256) k_mask(R *psi, int64_t P, int ld, int S, const R *__restrict__ M) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= P * S) return;
    const int64_t p = i / S;
    const int s = (int)(i - p * S);
    const R m = M[p];
    R *v = psi + (p * ld + s) * 2;
    v[0] *= m;
    v[1] *= m;
}

template <typename R>
cudaError_t launch_mask(void *psi, int64_t P, int ld, int S, const void *M, cudaStream_t st) {
    const int64_t n = P * S;
    k_mask<R><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((R *)psi, P, ld, S, (const R *)M);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_resid(const void *x, const void *hx, int64_t P, int ld, int S, const double *lam, double h3,
                         double *partial, int nblk, double *out, cudaStream_t st) {
    k_resid<R><<<dim3(nblk, S), 256, 0, st>>>((const R *)x, (const R *)hx, P, ld, S, lam, partial, nblk);
    return launch_sum_blocks(partial, nblk, S, h3, out, st);
}

template <typename R>
cudaError_t launch_tri_apply(void *psi, int64_t P, int ld, int S, const double *W, cudaStream_t st) {
    return rows_launch<R, true>(psi, P, ld, S, W, st);
}

// partial[blk][s] = sum over the block's points of |psi[p,s]|^2
template <typename R>
__global__ void __launch_bounds__(256) k_norms(const R *__restrict__ psi, int64_t P, int ld, int S,
                                               double *__restrict__ partial, int nblk) {
    __shared__ double red[256];
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.x * per;
    const int64_t p1 = p0 + per < P ? p0 + per : P;
    const int bx = blockDim.x, by = blockDim.y;
    for (int sb = 0; sb < S; sb += bx) {
        const int s = sb + threadIdx.x;
        double acc = 0.0;
        if (s < S)
            for (int64_t p = p0 + threadIdx.y; p < p1; p += by) {
                double re, im;
                ld_c(psi + (p * ld + s) * 2, re, im);
                acc += re * re + im * im;
            }
        red[threadIdx.y * bx + threadIdx.x] = acc;
        __syncthreads();
        if (threadIdx.y == 0 && s < S) {
            double t = 0.0;
            for (int l = 0; l < by; l++) t += red[l * bx + threadIdx.x];
            partial[(int64_t)blockIdx.x * S + s] = t;
        }
        __syncthreads();
    }
}

template <typename R>
cudaError_t launch_norms(const void *psi, int64_t P, int ld, int S, double h3, double *partial,
                         int nblk, double *out, cudaStream_t st) {
    if constexpr (sizeof(R) == 4) {
        return launch_norms_c64(psi, P, ld, S, h3, partial, nblk, out, st);
    } else {
        const int bx = S < 32 ? S : 32;
        k_norms<R><<<nblk, dim3(bx, 256 / bx), 0, st>>>((const R *)psi, P, ld, S, partial, nblk);
        return launch_sum_blocks(partial, nblk, S, h3, out, st);
    }
}

// Adjoint gradient of one exponential: per-block partial sums of the inner
// products M[j][i] = h^3 <b_j| X |a_i> that enter it, then the last block to
// finish (ticket counter) sums the partials in block order and adds
// 2 Re(-i tau sum_n 1/n! sum_j M[j][n-1-j]) = 2 tau Im(...) to grad_k.  The
// counter is left at zero for the next call.
template <typename R>
__global__ void __launch_bounds__(256) k_adjoint_grad(const R *b0, const R *b1, const R *b2, const R *b3,
                                                      const R *a0, const R *a1, const R *a2, const R *a3,
                                                      int64_t P, int ldb, int lda, const R *__restrict__ X,
                                                      double h3, double tau, double *__restrict__ partial, int nblk,
                                                      unsigned *counter, double *grad_k) {
    // The gradient needs only sum_{i+j<=3} Im <b_j|X|a_i> / (i+j+1)!.  With
    // c_i = sum_{j<=3-i} b_j / (i+j+1)! (real weights) it is
    // sum_p X_p sum_i Im(conj(c_i) a_i): one FP64 accumulator per thread.
    __shared__ double wsum[8];
    __shared__ bool last;
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.x * per;
    const int64_t p1 = p0 + per < P ? p0 + per : P;
    constexpr double f2 = 0.5, f3 = 1.0 / 6.0, f4 = 1.0 / 24.0;
    double acc = 0.0;
    chain_begin();
    chain_wait();
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const int64_t o = p * ldb * 2, q = p * lda * 2;
        double br0, bi0, br1, bi1, br2, bi2, br3, bi3, ar0, ai0, ar1, ai1, ar2, ai2, ar3, ai3;
        ld_wide(b0 + o, br0, bi0);
        ld_wide(b1 + o, br1, bi1);
        ld_wide(b2 + o, br2, bi2);
        ld_wide(b3 + o, br3, bi3);
        ld_wide(a0 + q, ar0, ai0);
        ld_wide(a1 + q, ar1, ai1);
        ld_wide(a2 + q, ar2, ai2);
        ld_wide(a3 + q, ar3, ai3);
        // c_0 .. c_3
        const double c0r = fma(f4, br3, fma(f3, br2, fma(f2, br1, br0)));
        const double c0i = fma(f4, bi3, fma(f3, bi2, fma(f2, bi1, bi0)));
        const double c1r = fma(f4, br2, fma(f3, br1, f2 * br0));
        const double c1i = fma(f4, bi2, fma(f3, bi1, f2 * bi0));
        const double c2r = fma(f4, br1, f3 * br0), c2i = fma(f4, bi1, f3 * bi0);
        const double c3r = f4 * br0, c3i = f4 * bi0;
        double t;
        t = fma(c0r, ai0, -c0i * ar0);
        t = fma(c1r, ai1, fma(-c1i, ar1, t));
        t = fma(c2r, ai2, fma(-c2i, ar2, t));
        t = fma(c3r, ai3, fma(-c3i, ar3, t));
        acc = fma(widen(X[p]), t, acc);
    }
    // block sum: shuffles within each warp, then the warps in order
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += wsum[w];
        partial[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(counter, 1u) == (unsigned)(nblk - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the last block sums the blocks' values: thread t takes blocks t,
    // t + 256, ..., then the same fixed shuffle and warp order
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += __ldcg(partial + b);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double tot = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) tot += wsum[w];
    *grad_k += 2.0 * tau * h3 * tot;
    *counter = 0u;
}

// Four blocks per SM: 28 FP64 instructions a point (two a clock per SM) need
// every SM; one block per 2048 points left 24 of them idle at 64^3 (28 and
// 33 us, complex128 and complex64; now 24 to 25).
int adjoint_blocks(int64_t P) { return (int)std::max<int64_t>(1, std::min<int64_t>(608, (P + 255) / 256)); }

template <typename R>
cudaError_t launch_adjoint_grad(const void *const *b, const void *const *a, int64_t P, int ldb, int lda,
                                const R *X, double h3, double tau, double *partial, int nblk, unsigned *counter,
                                double *grad_k, cudaStream_t st) {
    return launch_chained(k_adjoint_grad<R>, dim3(nblk), dim3(256), 0, st, true, (const R *)b[0], (const R *)b[1],
                          (const R *)b[2], (const R *)b[3], (const R *)a[0], (const R *)a[1], (const R *)a[2],
                          (const R *)a[3], P, ldb, lda, X, h3, tau, partial, nblk, counter, grad_k);
}

// h3 * sum_p conj(f_p) g_p for column 0 of two (P, ld) blocks.
template <typename R>
__global__ void __launch_bounds__(256) k_overlap(const R *__restrict__ f, const R *__restrict__ g,
                                                 int64_t P, int ld, double *__restrict__ partial,
                                                 int nblk) {
    __shared__ double red[2][256];
    const int64_t per = (P + nblk - 1) / nblk;
    const int64_t p0 = blockIdx.x * per;
    const int64_t p1 = p0 + per < P ? p0 + per : P;
    double sr = 0.0, si = 0.0;
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        double fr, fi, gr, gi;
        ld_c(f + p * ld * 2, fr, fi);
        ld_c(g + p * ld * 2, gr, gi);
        sr += fr * gr + fi * gi;
        si += fr * gi - fi * gr;
    }
    red[0][threadIdx.x] = sr;
    red[1][threadIdx.x] = si;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            red[0][threadIdx.x] += red[0][threadIdx.x + w];
            red[1][threadIdx.x] += red[1][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[(int64_t)blockIdx.x * 2] = red[0][0];
        partial[(int64_t)blockIdx.x * 2 + 1] = red[1][0];
    }
}

template <typename R>
cudaError_t launch_overlap(const void *f, const void *g, int64_t P, int ld, double h3,
                           double *partial, int nblk, double *out, cudaStream_t st) {
    k_overlap<R><<<nblk, 256, 0, st>>>((const R *)f, (const R *)g, P, ld, partial, nblk);
    return launch_sum_blocks(partial, nblk, 2, h3, out, st);
}

template <typename R>
__global__ void k_scale_dev(const R *__restrict__ x, R *__restrict__ y, int64_t n,
                            const double *__restrict__ a) {
    const double ar = a[0], ai = a[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double xr = x[2 * i], xi = x[2 * i + 1];
        y[2 * i] = (R)(ar * xr - ai * xi);
        y[2 * i + 1] = (R)(ar * xi + ai * xr);
    }
}

template <typename R>
cudaError_t launch_scale_dev(const void *x, void *y, int64_t n, const double *a, cudaStream_t st) {
    int64_t nb = (n + 255) / 256;
    if (nb > 152 * 16) nb = 152 * 16;
    if (nb < 1) nb = 1;
    k_scale_dev<R><<<(unsigned)nb, 256, 0, st>>>((const R *)x, (R *)y, n, a);
    return cudaGetLastError();
}

#define RSG_INST(R)                                                                               \
    template cudaError_t launch_rotate<R>(void *, int64_t, int, int, const double *, cudaStream_t);  \
    template cudaError_t launch_resid<R>(const void *, const void *, int64_t, int, int, const double *, \
                                         double, double *, int, double *, cudaStream_t);             \
    template cudaError_t launch_bilinear<R>(const void *, const void *, int64_t, int, int, double,   \
                                            double *, int, double *, cudaStream_t);                  \
    template cudaError_t launch_comb<R>(const void *, const void *, void *, int64_t, int, int,       \
                                        const double *, cudaStream_t);                               \
    template cudaError_t launch_mask<R>(void *, int64_t, int, int, const void *, cudaStream_t);      \
    template cudaError_t launch_tri_apply<R>(void *, int64_t, int, int, const double *,              \
                                             cudaStream_t);                                          \
    template cudaError_t launch_norms<R>(const void *, int64_t, int, int, double, double *, int,     \
                                         double *, cudaStream_t);                                    \
    template cudaError_t launch_adjoint_grad<R>(const void *const *, const void *const *, int64_t, int, \
                                                int, const R *, double, double, double *, int,         \
                                                unsigned *,                                            \
                                                double *, cudaStream_t);                               \
    template cudaError_t launch_overlap<R>(const void *, const void *, int64_t, int, double,         \
                                           double *, int, double *, cudaStream_t);                   \
    template cudaError_t launch_scale_dev<R>(const void *, void *, int64_t, const double *,         \
                                             cudaStream_t);
RSG_INST(float)
RSG_INST(double)

}  // namespace rsg
