// complex128 stencil with integer neighbour sums (kernel 1 of complex128).
//
// The operator is that of the other stencil kernels: the 8th-order 25-point
// star Laplacian with zero values outside the mesh, the local potential and
// dipole field on the diagonal, projector terms in the epilogue
// (arXiv:1501.05654, Sec. 1: high-order finite differences on a real-space
// grid).
//
// k_apply_sum64: the complex128 stencil with the neighbour sums in integer
// arithmetic.  The FP64 pipe does two instructions a clock per SM, and 40 of
// the 56 a value needs are the additions of the six neighbours at one
// distance.  Here the six values of a shell are added as 64-bit integers:
// each double is split once into a mantissa (53 bits, seven guard bits below)
// and an exponent, the mantissas are shifted to the largest exponent of the
// six, and the sum is rounded once when it is converted back.  A value cut off
// by the shift loses less than 2^-59 of the largest of the six, so a shell
// sum is off by less than 5 x 2^-59 of the largest before its one rounding
// (five FP64 additions round five times, by up to 2^-53 of their sums); where
// the largest cancel, that is the bound on what is left.  Negative values are
// kept as one's complements, which the arithmetic shift cuts off towards zero
// like positive ones, and every sum adds one per negative value: the sum is
// odd, H(-u) = -H(u) in every bit, and opposite values cancel.  The weights,
// the diagonal and the epilogue stay FP64.  Sums that hold Inf or NaN, or lie
// at the ends of the exponent range, take a slow path.
//
// A block owns a TX x TY tile of columns for NSC states and marches along z:
// a thread keeps its column's nine split values, the plane's tile and halo
// lie split in shared memory (two slots, one barrier a plane).  Bound by
// instruction issue at 16 warps per SM (128 registers); the FP64 pipe is
// about a third busy.  Horner stages without projectors, in a chain of steps,
// against FP64 sums: 904,089 points (R = 12 sphere) x 16 states 1.06 ms (1.65);
// 61^3 x 8 0.121 (0.209); 96^3 x 3 0.168 (0.292); 64^3 x 2 columns 39.7 us (59.2);
// 32^3 x 4 12.7 us (16.9).  Two's complements, whose shift cuts negative values
// off downwards, would save 6%, and H(-u) would differ from -H(u) in places.
// Converting the sums with the conversion instruction instead of integers costs
// 10% (two FP64 slots each).  Error against 80-bit sums on noise, packets and
// values spread over 2^+-900, of the norm: 1.35e-16, 9.8e-16, 1.1e-16 (FP64 sums
// 1.39e-16, 1.1e-15, 1.1e-16).
#include "rsg_async.cuh"
#include "rsg_chain.cuh"
#include "rsg_internal.h"
#include "rsg_point.cuh"
#include "rsg_vec.cuh"

namespace rsg {

namespace {

constexpr int kSumTX = 16, kSumNT = 256, kSumMaxZ = 32;
struct SplitC {
    long long re, im;   // mantissas, one's complement
    int e;   // exponents, re in the low half
};
__device__ __forceinline__ long long split_real(double d, int &e) {
    const int hi = __double2hiint(d);
    const unsigned eb = ((unsigned)hi >> 20) & 0x7ff;
    const unsigned mh = ((unsigned)hi & 0xfffffu) | (eb ? 0x100000u : 0u);
    long long m = (long long)(((unsigned long long)mh << 32 | (unsigned)__double2loint(d)) << 7);
    e = eb ? (int)eb : 1;
    return m ^ (long long)(hi >> 31);
}
__device__ __forceinline__ SplitC split(const double2 &d) {
    SplitC s;
    int er, ei;
    s.re = split_real(d.x, er);
    s.im = split_real(d.y, ei);
    s.e = er | (ei << 16);
    return s;
}
// S 2^(E - 1082) for sums outside the fast range; m, e: the six terms
__device__ __noinline__ double shell_slow(long long S, int E, const long long *m, const int *e) {
    if (E == 0x7ff) {
        double t = 0.0;
        for (int i = 0; i < 6; i++)
            if (e[i] == 0x7ff) {
                const unsigned long long a = (unsigned long long)(m[i] < 0 ? ~m[i] : m[i]) >> 7;
                t += __hiloint2double((m[i] < 0 ? 0xfff00000 : 0x7ff00000) | (int)((a >> 32) & 0xfffff), (int)a);
            }
        return t;
    }
    return ldexp((double)S, E - 1082);
}
// S 2^(E - 1082) rounded to nearest even.  In integers: the conversion
// instruction takes two slots of the FP64 pipe.
__device__ __forceinline__ double shell_round(long long S, int E, bool &slow) {
    slow = (unsigned)(E - 64) > 2043u - 64u && (S != 0 || E == 0x7ff);
    const unsigned long long u = (unsigned long long)(S < 0 ? -S : S);
    const int lz = __clzll((long long)u);            // 1 .. 64
    const unsigned long long n = u << (lz & 63);     // leading one in bit 63 (0 for S = 0)
    // top 53 bits, rounded: the leading one adds 1 to the exponent field, a carry another
    const unsigned long long r = (n + 0x3ff + ((n >> 11) & 1)) >> 11;
    const bool carry = n > 0xfffffffffffffbffull;    // the addition would wrap: 2^64 exactly
    const int ex = E - 1082 + 1023 + 62 - lz;        // biased exponent less one
    int hi = (int)(r >> 32) + (ex << 20);
    int lo = (int)r;
    if (carry) {
        hi = (ex + 2) << 20;
        lo = 0;
    }
    hi |= (int)((unsigned long long)S >> 32) & 0x80000000;
    return S == 0 ? 0.0 : __hiloint2double(hi, lo);
}
// m >> d, d of any size (sign fill)
__device__ __forceinline__ long long shift_down(long long m, unsigned d) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(d));
    return r;
}

template <int NSC>
__global__ void __launch_bounds__(kSumNT, 2) k_apply_sum64(const ApplyArgs<double> a, int zs, int nch) {
    using V = VT<double>;
    constexpr int TX = kSumTX, TY = kSumNT / (TX * NSC), WX = TX + 8, WY = TY + 8;
    constexpr int NH = (8 * TY + 8 * TX) * NSC, HPT = (NH + kSumNT - 1) / kSumNT;   // halo values, per thread
    __shared__ longlong2 wm[2][WY * WX * NSC];
    __shared__ int we[2][WY * WX * NSC];
    __shared__ SRow rows[(kSumMaxZ + 8) * WY];
    chain_begin();
    const int ny = a.ny, nz = a.nz, SV = a.SV;
    const int ntx = (a.nx + TX - 1) / TX;
    const int tile = blockIdx.x / nch, s0 = (blockIdx.x - tile * nch) * NSC;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY, z0 = blockIdx.y * zs;
    const int z1 = min(z0 + zs, nz);
    const int tid = threadIdx.x;
    const int sl = tid % NSC, xl = (tid / NSC) % TX, yl = tid / (NSC * TX);
    const int x = x0 + xl, y = y0 + yl, v = s0 + sl;
    bool any = false;
    for (int i = tid; i < (z1 - z0 + 8) * WY; i += kSumNT) {
        const int wy = i % WY, zz = z0 - 4 + i / WY;
        const Row r = load_row(a.rows, y0 - 4 + wy, zz, ny, nz);
        rows[i] = SRow{r.start - r.xmin, (int16_t)r.xmin, (int16_t)r.xmax};
        any = any || (wy >= 4 && wy < WY - 4 && zz >= z0 && zz < z1 && r.xmin < x0 + TX && r.xmax >= x0);
    }
    any = __syncthreads_or(any);
    chain_wait();
    if (!any) return;
    const bool vok = v < SV;
    const double2 *__restrict__ in = (const double2 *)a.in;
    auto value = [&](const SRow &r, int xx, int vv) -> double2 {
        return xx >= r.xmin && xx <= r.xmax ? V::ldg(in + (int64_t)(r.start + xx) * SV + vv) : V::zero();
    };
    // this thread's halo values: window position and state, -1 for none
    int hp[HPT], hx[HPT], hw[HPT], hv[HPT];
#pragma unroll
    for (int h = 0; h < HPT; h++) {
        const int i = tid + h * kSumNT;
        const int s = i % NSC, j = i / NSC;
        int wx, wy;
        if (j < 8 * TX) {            // rows above and below the tile
            wy = j / TX < 4 ? j / TX : TY + j / TX;
            wx = 4 + j % TX;
        } else {                     // columns left and right of it
            const int q = j - 8 * TX;
            wy = 4 + q / 8;
            wx = q % 8 < 4 ? q % 8 : TX + q % 8;
        }
        const bool ok = i < NH && s0 + s < SV;
        hp[h] = i < NH ? (wy * WX + wx) * NSC + s : -1;
        hx[h] = x0 - 4 + wx;
        hw[h] = wy;
        hv[h] = ok ? s0 + s : -1;
    }
    auto halo = [&](int z, double2 (&d)[HPT]) {
#pragma unroll
        for (int h = 0; h < HPT; h++)
            d[h] = hp[h] >= 0 && hv[h] >= 0 ? value(rows[(z - z0 + 4) * WY + hw[h]], hx[h], hv[h]) : V::zero();
    };
    const SRow *own = rows + 4 + yl;   // own row of plane z: own[(z - z0 + 4) * WY]
    auto column = [&](int z) { return vok ? value(own[(z - z0 + 4) * WY], x, v) : V::zero(); };
    SplitC q[9];
#pragma unroll
    for (int j = 0; j < 9; j++) q[j] = split(column(z0 - 4 + j));
    double2 hd[HPT], cen = column(z0);
    halo(z0, hd);
    const int wp = ((4 + yl) * WX + 4 + xl) * NSC + sl;
#pragma unroll 1
    for (int z = z0; z < z1; z++) {
        const int slot = (z - z0) & 1;
        longlong2 *M = wm[slot];
        int *Ex = we[slot];
        M[wp] = make_longlong2(q[4].re, q[4].im);
        Ex[wp] = q[4].e;
#pragma unroll
        for (int h = 0; h < HPT; h++)
            if (hp[h] >= 0) {
                const SplitC t = split(hd[h]);
                M[hp[h]] = make_longlong2(t.re, t.im);
                Ex[hp[h]] = t.e;
            }
        __syncthreads();
        const SRow rc = own[(z - z0 + 4) * WY];
        const bool ok = vok && x >= rc.xmin && x <= rc.xmax;
        const int64_t idx = ok ? (int64_t)rc.start + x : 0;
        double vloc = 0.0;
        double2 bval = V::zero();
        NlPoint nl{0, 0, 0};
        if (ok) {
            vloc = a.V[idx];
            if (a.base != nullptr) bval = ((const double2 *)a.base)[idx * SV + v];
            nl = load_projectors<double>(a, idx);
        }
        // the next plane's values, a plane ahead of their use
        double2 nxt = V::zero(), cen1 = V::zero();
        if (z + 1 < z1) {
            nxt = column(z + 5);
            cen1 = column(z + 1);
            halo(z + 1, hd);
        }
        if (ok) {
            double2 acc = V::scale(3.0 * a.w[0], cen);
#pragma unroll
            for (int k = 1; k <= 4; k++) {
                const int p[4] = {wp - k * NSC, wp + k * NSC, wp - k * WX * NSC, wp + k * WX * NSC};
                longlong2 m[6];
                int e[6];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    m[j] = M[p[j]];
                    e[j] = Ex[p[j]];
                }
                m[4] = make_longlong2(q[4 - k].re, q[4 - k].im);
                e[4] = q[4 - k].e;
                m[5] = make_longlong2(q[4 + k].re, q[4 + k].im);
                e[5] = q[4 + k].e;
                unsigned E = (unsigned)e[0];
#pragma unroll
                for (int j = 1; j < 6; j++) E = __vmaxu2(E, (unsigned)e[j]);
                // the one's complements of the negative terms are one too low each
                long long sr = 0, si = 0;
                int nr = 0, ni = 0;
#pragma unroll
                for (int j = 0; j < 6; j++) {
                    const unsigned d = E - (unsigned)e[j];   // each half >= 0: no borrow
                    sr += shift_down(m[j].x, d & 0xffff);
                    si += shift_down(m[j].y, d >> 16);
                    nr += (int)((unsigned long long)m[j].x >> 63);
                    ni += (int)((unsigned long long)m[j].y >> 63);
                }
                sr += nr;
                si += ni;
                const int er = (int)(E & 0xffff), ei = (int)(E >> 16);
                bool slr, sli;
                double2 s = make_double2(shell_round(sr, er, slr), shell_round(si, ei, sli));
                if (slr || sli) {
                    long long t[6];
                    int u[6];
                    if (slr) {
#pragma unroll
                        for (int j = 0; j < 6; j++) {
                            t[j] = m[j].x;
                            u[j] = e[j] & 0xffff;
                        }
                        s.x = shell_slow(sr, er, t, u);
                    }
                    if (sli) {
#pragma unroll
                        for (int j = 0; j < 6; j++) {
                            t[j] = m[j].y;
                            u[j] = (int)((unsigned)e[j] >> 16);
                        }
                        s.y = shell_slow(si, ei, t, u);
                    }
                }
                V::fma(acc, a.w[k], s);
            }
            finish_fp64(a, idx, x, y, z, v, cen, acc, vloc, bval, nl);
        }
#pragma unroll
        for (int j = 0; j < 8; j++) q[j] = q[j + 1];
        q[8] = split(nxt);
        cen = cen1;
    }
}

}  // namespace

int sum64_states(int SV) { return SV % 2 == 1 && SV < 16 ? 1 : 2; }
void sum64_shape(int SV, int *TX, int *TY) {
    *TX = kSumTX;
    *TY = kSumNT / (kSumTX * sum64_states(SV));
}

cudaError_t launch_apply_sum64(const ApplyArgs<double> &a, int zs, cudaStream_t st) {
    if (zs < 1 || zs > kSumMaxZ) return cudaErrorInvalidValue;
    int tx, ty;
    sum64_shape(a.SV, &tx, &ty);
    const int nsc = sum64_states(a.SV);
    const long long nch = (a.SV + nsc - 1) / nsc;
    const long long nb = (long long)((a.nx + tx - 1) / tx) * ((a.ny + ty - 1) / ty) * nch;
    if (nb > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const dim3 grid((unsigned)nb, (a.nz + zs - 1) / zs);
    return launch_chained(nsc == 1 ? k_apply_sum64<1> : k_apply_sum64<2>, grid, dim3(kSumNT), 0, st, true, a, zs,
                          (int)nch);
}

}  // namespace rsg
