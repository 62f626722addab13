// Host side of the C ABI declared in include/rsg.h: handles, mesh and
// projector tables, argument checks, workspace and the launch sequences of
// the Hamiltonian application, the Taylor-4 propagator, the Cholesky-QR
// re-orthonormalisation and the discrete adjoint of the control gradient;
// the solvers built on the application (L-BFGS control loop, Chebyshev-
// filtered eigensolver, COCG shifted solves); batches; checkpoint files;
// the failure-path and diagnostic helpers.
//
// Method passages (arXiv:1501.05654): Sec. 1 (uniform grids, finite
// differences), Sec. "Parallelization, optimizations and graphics processing units" (Hamiltonian application on groups of
// states; linear arrays plus grid tables; re-orthonormalisation only rarely
// needed in real time), Sec. "Magnetic response and gauge invariance in real-space grids" (non-local pseudopotential),
// Sec. "Quantum optimal control" (Eq. (qoctgradient), costate propagation,
// the parameters that shape the field), Sec. "The Sternheimer formulation of
// linear-response" (shifted systems), Sec. "Photoemission" (mask split),
// Sec. "Complex scaling and resonances" (H_theta).
#include <atomic>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <complex>
#include <cstdlib>
#include <cstring>
#include <unistd.h>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <tuple>
#include <type_traits>
#include <vector>

#include "rsg_internal.h"

namespace rsg {
// Bounded-wait self-test kernel (rsg_selftest.cu): one warp waits `polls`
// times on an mbarrier phase that cannot complete and records 2 in *err.
cudaError_t launch_selftest_wait(int polls, int *err, cudaStream_t st);
// Antisymmetric-image boundary (rsg_odd.cuh): the one-thread-per-value
// kernel (rsg_kernels.cu) and the complex-scaled kernel (rsg_scaled.cu).
template <typename R>
cudaError_t launch_apply_naive_odd(const ApplyArgs<R> &a, cudaStream_t st);
template <typename R>
cudaError_t launch_apply_scaled_odd(const ApplyArgs<R> &a, const R *vt, double theta, cudaStream_t st);
}  // namespace rsg

using namespace rsg;

namespace {

thread_local std::string g_err;

// Diagnostics on stderr (rsg_set_log_level): 0 silent, 1 every error
// status, 2 also stencil-kernel fallbacks.  RSG_LOG_LEVEL sets the initial
// level.
std::atomic<int> g_log_level{-1};

int log_level() {
    int l = g_log_level.load();
    if (l < 0) {
        const char *e = std::getenv("RSG_LOG_LEVEL");
        l = e ? std::max(0, std::min(2, std::atoi(e))) : 0;
        g_log_level.store(l);
    }
    return l;
}

void log_info(const char *fmt, ...) {
    if (log_level() < 2) return;
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    std::fprintf(stderr, "rsg: %s\n", buf);
}

rsg_status fail(rsg_status s, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    if (log_level() >= 1) std::fprintf(stderr, "rsg: error %d: %s\n", (int)s, buf);
    return s;
}

#define CK(call)                                                                              \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return fail(e_ == cudaErrorMemoryAllocation ? RSG_ERR_OOM : RSG_ERR_CUDA,         \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

#define CKS(expr)                    \
    do {                             \
        rsg_status s_ = (expr);      \
        if (s_ != RSG_OK) return s_; \
    } while (0)

// 8th-order central second difference weights, |k| = 0..4 (times 1/h^2).
const double kFD[5] = {-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0};

// Simulated allocation failures (rsg_debug_fail_allocations): the next
// g_fail_allocs device allocations report cudaErrorMemoryAllocation.
std::atomic<int> g_fail_allocs{0};

// Device buffer that only grows.
struct DevBuf {
    void *p = nullptr;
    size_t n = 0;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    DevBuf(DevBuf &&o) noexcept : p(o.p), n(o.n) {
        o.p = nullptr;
        o.n = 0;
    }
    ~DevBuf() { release(); }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
    cudaError_t ensure(size_t bytes) {
        if (bytes <= n && p) return cudaSuccess;
        for (int f = g_fail_allocs.load(); f > 0;)
            if (g_fail_allocs.compare_exchange_weak(f, f - 1)) return cudaErrorMemoryAllocation;
        release();
        cudaError_t e = cudaMalloc(&p, bytes ? bytes : 16);
        if (e == cudaSuccess) n = bytes ? bytes : 16;
        return e;
    }
    template <typename T>
    cudaError_t upload(const std::vector<T> &v) {
        cudaError_t e = ensure(v.size() * sizeof(T));
        if (e != cudaSuccess || v.empty()) return e;
        e = cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
        return e != cudaSuccess ? e : landed();
    }
    cudaError_t zero(size_t bytes) {
        cudaError_t e = cudaMemset(p, 0, bytes);
        return e != cudaSuccess ? e : landed();
    }
    // A copy from pageable memory may return before its last piece is on the
    // device, and a memset always may; a kernel on a non-blocking stream does
    // not wait for the legacy stream.
    static cudaError_t landed() { return cudaStreamSynchronize(cudaStreamLegacy); }
    template <typename T>
    T *as() const {
        return (T *)p;
    }
};

}  // namespace

struct rsg_mesh_s {
    int shape = 0;
    double h = 0.0;
    double origin[3] = {0, 0, 0};
    int32_t lo[3] = {0, 0, 0};     // lattice coordinate of bbox index 0
    int nx = 0, ny = 0, nz = 0;
    int64_t P = 0;
    int bc = RSG_BC_ZERO;           // boundary rule (image walls for cube/box only)
    std::vector<int32_t> ijk;       // P x 3 lattice integers
    std::vector<Row> rows;          // ny * nz
    DevBuf d_rows;
    // tables made on first use, by any Hamiltonian on this mesh: made and
    // looked up under the lock; an entry does not change or move once made
    std::mutex mu;
    // tile lists keyed by (TX, TY, zseg): device tiles and their count
    std::map<std::tuple<int, int, int>, std::pair<DevBuf, int>> tiles;
    std::map<std::tuple<int, int, int>, std::vector<Tile>> tiles_host;   // the same lists on the host
    std::map<std::pair<int, int>, std::vector<int>> col_len;   // planes of every TX x TY column of tiles
    // complex64: stencil kernel and segment length by (vectors per point,
    // complex scaling, projectors); complex128: planes per block of the integer
    // sums by vectors per point
    std::map<std::tuple<int, bool, bool>, std::pair<int, int>> choice32;
    std::map<int, int> choice64;
};

struct rsg_ham_s {
    rsg_mesh m = nullptr;
    rsg_dtype dtype = RSG_C64;
    bool has_V = false;
    DevBuf V;
    double eps = 0.0, dir[3] = {1, 0, 0};
    double vmin = 0.0, vmax = 0.0;     // range of the potential (spectral bounds of the eigensolver)
    double proj_norm = 0.0;            // bound on the non-local operator: sum over atoms of sum |h_ij|
    TileCfg cfg;
    bool force_kernel = false;   // set when the caller chose the kernel explicitly
    bool shape_set = false;      // set when the caller chose a tile shape, even the default one
    int last_kernel = -1;        // stencil kernel of the last application
    int last_zseg = 0;           // its planes per z segment (tiled kernels)
    int last_sum = 0;            // its planes per block with integer neighbour sums (complex128), 0: FP64 sums
    int sum_planes = -1;         // option "sum_planes": 0..32 as last_sum, -1 by size
    int adj_keep = -1;           // adjoint: keep segment powers (1), recompute (0), by memory (-1)
    int adj_merge = -1;          // adjoint: costate and recompute sweeps share launches (1), not (0), auto (-1)
    // projectors
    ProjDev pj;
    DevBuf q_pt, q_p, ch_atom, ch_q0, ch_q1, atom_ch0, hm, nl_ptr, u_pts, u_ptr, e_atom, e_p;
    DevBuf D, partial, pcnt;   // coefficients, their partial sums, per-atom completion counters
    // workspace
    DevBuf w0, w1, red, G, W, Wc, drift, status, dots, ov, grad, Xd, Xdir;
    DevBuf w2, cg;     // shifted solver: third work block, per-state scalars
    DevBuf mask;       // mask absorber M(r) (compute type), applied after each time step
    bool has_mask = false;
    DevBuf vtheta;     // complex scaling: v(r e^{i theta}) per point, interleaved (compute type)
    DevBuf vtheta_rot; // complex64: v(r e^{i theta}) e^{2i theta}, the register-blocked kernel's diagonal
    bool has_scaling = false;
    double theta = 0.0;
    double xdir_cached[3] = {NAN, NAN, NAN};
    std::vector<DevBuf> pool;   // control-gradient vectors
    std::vector<DevBuf> pool2;  // control-gradient two-column blocks (shared sweeps)
    // measurement
    bool prof = false;
    std::vector<cudaEvent_t> ev;   // pairs (start, stop) of stencil launches
    size_t ev_used = 0;
    int64_t n_launch = 0, n_stencil = 0;
    double stencil_bytes = 0.0;
    // option "proj_overlap": projector coefficients on a side stream,
    // concurrent with the stencil they do not feed (the scatter after the
    // stencil waits for them)
    int proj_overlap = 0;
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    ~rsg_ham_s() {
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
        if (ev_fork) cudaEventDestroy(ev_fork);
        if (ev_join) cudaEventDestroy(ev_join);
        if (side) cudaStreamDestroy(side);
    }
};

struct rsg_batch_s {
    std::vector<rsg_ham> hams;
    std::vector<int64_t> S, ld;
    std::vector<SysArgs> args;               // host copy of the device table
    DevBuf d_args, d_work, d_dot, d_red, d_sca;
    std::vector<DevBuf> w0, w1, D, partial;  // per-system work blocks and projector buffers
    int nwork = 0, ndot = 0, nred = 0, nsca = 0, npmax = 0;
    bool batched = false;                    // false: fall back to per-system propagation
    // one captured time step
    cudaStream_t cs = nullptr;
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    cudaGraphExec_t step = nullptr;
    double step_dt = NAN;
    int step_scheme = -1;
    std::vector<void *> step_psis;
    int64_t n_launch_step = 0;
    // persistent step (mode 1, the default): one k_batch_step launch per
    // time step; mode 0: one launch per Horner stage and kernel
    int mode = 1;
    int zseg = 96;                 // planes per tile segment (mode 1)
    long wait_limit = 1L << 22;    // polls of a dependency wait
    int stall = 0;                 // > 0: system 0 waits for a stencil item that never comes
    int tile_var_mask = 0;         // bit ls / 2 - 1: tile variant 1 for records of ls values (ls = 14)
    std::vector<BItem> stage_items;   // the items of one stage, stage bits 0
    int np_cap = 0, nblocks = 0, step_nst = 0;
    DevBuf d_items, d_cnt, d_ctl, d_status, d_zero;
    ~rsg_batch_s() {
        if (step) cudaGraphExecDestroy(step);
        if (ev_in) cudaEventDestroy(ev_in);
        if (ev_out) cudaEventDestroy(ev_out);
        if (cs) cudaStreamDestroy(cs);
    }
};

namespace {

size_t cbytes(rsg_dtype t) { return t == RSG_C64 ? 8 : 16; }

// ---------------------------------------------------------------- mesh ---
void build_rows(rsg_mesh m, int64_t r2max) {
    m->rows.assign((size_t)m->ny * m->nz, Row{0, 1, 0, 0});
    m->ijk.clear();
    int64_t P = 0;
    for (int z = 0; z < m->nz; z++)
        for (int y = 0; y < m->ny; y++) {
            int xmin = 0, xmax = m->nx - 1;
            if (m->shape == RSG_SHAPE_SPHERE) {
                const int64_t j = y + m->lo[1], k = z + m->lo[2];
                const int64_t rem = r2max - j * j - k * k;
                if (rem < 0) continue;
                int64_t xm = (int64_t)std::floor(std::sqrt((double)rem));
                while (xm * xm > rem) xm--;
                while ((xm + 1) * (xm + 1) <= rem) xm++;
                xmin = (int)(-xm - m->lo[0]);
                xmax = (int)(xm - m->lo[0]);
            }
            Row &r = m->rows[(size_t)z * m->ny + y];
            r.start = (int32_t)P;
            r.xmin = xmin;
            r.xmax = xmax;
            for (int x = xmin; x <= xmax; x++) {
                m->ijk.push_back(x + m->lo[0]);
                m->ijk.push_back(y + m->lo[1]);
                m->ijk.push_back(z + m->lo[2]);
            }
            P += xmax - xmin + 1;
        }
    m->P = P;
}

// Tiles of TX x TY columns; each keeps only the planes where one of its rows
// meets its x range, split into segments of zseg planes.
rsg_status get_tiles(rsg_mesh m, int TX, int TY, int zseg, const Tile **out, int *count,
                     const std::vector<Tile> **host = nullptr) {
    std::lock_guard<std::mutex> lock(m->mu);
    auto key = std::make_tuple(TX, TY, zseg);
    auto it = m->tiles.find(key);
    if (it == m->tiles.end()) {
        std::vector<Tile> tl;
        std::vector<int> seg;     // z segment index of each tile
        const int ntx = (m->nx + TX - 1) / TX, nty = (m->ny + TY - 1) / TY;
        for (int ty = 0; ty < nty; ty++)
            for (int tx = 0; tx < ntx; tx++) {
                const int xa = tx * TX, xb = std::min(m->nx - 1, xa + TX - 1);
                int zlo = m->nz, zhi = 0;
                for (int z = 0; z < m->nz; z++)
                    for (int y = ty * TY; y < std::min(m->ny, ty * TY + TY); y++) {
                        const Row &r = m->rows[(size_t)z * m->ny + y];
                        if (r.xmin <= r.xmax && r.xmax >= xa && r.xmin <= xb) {
                            zlo = std::min(zlo, z);
                            zhi = std::max(zhi, z + 1);
                        }
                    }
                for (int z0 = zlo; z0 < zhi; z0 += zseg) {
                    tl.push_back(Tile{tx, ty, z0, std::min(zhi, z0 + zseg)});
                    seg.push_back((z0 - zlo) / zseg);
                }
            }
        // launch order: longest tiles first, then by z segment and along a
        // Hilbert curve over (tx, ty), so that the blocks resident at one time
        // cover compact patches of tiles and read each other's halo rows and
        // columns from L2
        int side = 1;
        while (side < ntx || side < nty) side <<= 1;
        auto hilbert = [side](int x, int y) {
            long long d = 0;
            for (int s = side / 2; s > 0; s /= 2) {
                const int rx = (x & s) > 0, ry = (y & s) > 0;
                d += (long long)s * s * ((3 * rx) ^ ry);
                if (ry == 0) {
                    if (rx == 1) {
                        x = s - 1 - x;
                        y = s - 1 - y;
                    }
                    std::swap(x, y);
                }
            }
            return d;
        };
        // longest tiles first (8-plane buckets) so that the last blocks of a
        // launch are short ones; then the segment index and the Hilbert order
        std::vector<std::pair<long long, int>> order(tl.size());
        const long long hs = (long long)side * side;
        for (size_t i = 0; i < tl.size(); i++) {
            const long long len_bucket = 64 - std::min(63, (tl[i].zhi - tl[i].zlo) / 8);
            order[i] = {(len_bucket * 64 + seg[i]) * hs + hilbert(tl[i].tx, tl[i].ty), (int)i};
        }
        std::stable_sort(order.begin(), order.end());
        std::vector<Tile> sorted(tl.size());
        for (size_t i = 0; i < tl.size(); i++) sorted[i] = tl[order[i].second];
        tl.swap(sorted);
        m->tiles_host[key] = tl;
        auto &slot = m->tiles[key];
        cudaError_t e = slot.first.upload(tl);
        if (e != cudaSuccess) {
            m->tiles.erase(key);
            return fail(RSG_ERR_CUDA, "tile upload: %s", cudaGetErrorString(e));
        }
        slot.second = (int)tl.size();
        it = m->tiles.find(key);
    }
    *out = it->second.first.as<Tile>();
    *count = it->second.second;
    if (host) *host = &m->tiles_host[key];
    return RSG_OK;
}

int pow2_at_least(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Tile of the stencil kernel in use for SV vectors per row (must match
// launch_apply): staged kernel cv x nxr x ty threads (512), L1 z-march
// kernel 256 threads; TX = nxr * rx.
void block_shape(const TileCfg &c, int SV, int *TX, int *TY) {
    if (c.kernel == 5) {
        quad_shape(c, TX, TY);
        return;
    }
    if (c.kernel == 7) {
        wide_shape(c, TX, TY);
        return;
    }
    if (c.kernel == 3) {
        int cv, nxr, ty;
        tma_shape(c, SV, &cv, &nxr, &ty);
        *TX = nxr;
        *TY = ty;
        return;
    }
    if (c.kernel == 0 || c.kernel == 4) {
        int cv, nxr, ty;
        stage_shape(c, SV, &cv, &nxr, &ty);
        *TX = nxr;
        *TY = ty;
        return;
    }
    const int cv = std::min(8, pow2_at_least(SV));
    int ty = c.ty;
    while (cv * ty > 256) ty >>= 1;
    const int nxr = 256 / (cv * ty);
    *TX = nxr * c.rx;
    *TY = ty;
}

// Tile list of kernel configuration c (0 tiles on failure).
int tiles_for(rsg_ham H, const TileCfg &c, int SV, const Tile **tiles) {
    int TX, TY, n = 0;
    block_shape(c, SV, &TX, &TY);
    if (get_tiles(H->m, TX, TY, c.zseg, tiles, &n) != RSG_OK) return 0;
    return n;
}

// ------------------------------------------- kernel choice, complex64 ----
// Default configuration: kernel 7, 16 x 6 tiles, four producer warps,
// 190-plane segments.
TileCfg c64_config() {
    TileCfg c;
    c.kernel = 7;
    c.wty = 6;
    c.npw = 4;
    c.threads = 192;
    c.zseg = 190;
    c.stages = 3;
    return c;
}

// Planes of every TX x TY column of tiles that holds mesh points, longest
// first.
const std::vector<int> &column_lengths(rsg_mesh m, int TX, int TY) {
    std::lock_guard<std::mutex> lock(m->mu);
    auto it = m->col_len.find({TX, TY});
    if (it != m->col_len.end()) return it->second;
    const int ntx = (m->nx + TX - 1) / TX, nty = (m->ny + TY - 1) / TY;
    std::vector<int> zlo((size_t)ntx * nty, m->nz), zhi((size_t)ntx * nty, 0);
    for (int z = 0; z < m->nz; z++)
        for (int ty = 0; ty < nty; ty++) {
            // the tile's rows together (every shape is convex)
            int lo = m->nx, hi = -1;
            for (int y = ty * TY; y < std::min(m->ny, (ty + 1) * TY); y++) {
                const Row &r = m->rows[(size_t)z * m->ny + y];
                if (r.xmin > r.xmax) continue;
                lo = std::min(lo, r.xmin);
                hi = std::max(hi, r.xmax);
            }
            for (int tx = lo / TX; tx <= (hi < 0 ? -1 : hi / TX); tx++) {
                const size_t k = (size_t)ty * ntx + tx;
                zlo[k] = std::min(zlo[k], z);
                zhi[k] = z + 1;
            }
        }
    std::vector<int> len;
    for (size_t k = 0; k < zlo.size(); k++)
        if (zhi[k] > zlo[k]) len.push_back(zhi[k] - zlo[k]);
    std::sort(len.rbegin(), len.rend());
    return m->col_len[{TX, TY}] = len;
}

// Time until the last of `slots` resident blocks is done: columns cut into
// segments of zs planes, nch blocks per segment that take mul * planes + add,
// longest first to the first free slot; *blocks receives their number.  A
// schedule whose load alone takes `enough` is not worked out.
double makespan(const std::vector<int> &col, int zs, int nch, int slots, int64_t *blocks, int mul = 1, int add = 8,
                double enough = 1e300) {
    // blocks by planes, rounded up to a sixteenth of the longest
    const int longest = col.empty() ? 0 : std::min(zs, col[0]), step = longest / 16 + 1;
    std::vector<int64_t> by_len((size_t)(longest / step + 2), 0);
    int64_t n = 0;
    for (int L : col) {
        const int full = L / zs, rest = L % zs;
        if (full) by_len[(size_t)((zs + step - 1) / step)] += (int64_t)full * nch;
        if (rest) by_len[(size_t)((rest + step - 1) / step)] += nch;
        n += (int64_t)(full + (rest > 0)) * nch;
    }
    *blocks = n;
    if (n == 0) return 0.0;
    double load = 0.0;
    for (size_t k = 0; k < by_len.size(); k++)
        load += (double)by_len[k] * ((double)mul * std::min<int64_t>((int64_t)k * step, longest) + add);
    if (load / slots >= enough) return load / slots;
    // finish times of the slots and how many slots finish at each
    std::map<int64_t, int64_t> at{{0, slots}};
    for (size_t k = by_len.size(); k-- > 0;) {
        const int64_t len = (int64_t)mul * std::min<int64_t>((int64_t)k * step, longest) + add;
        int64_t left = by_len[k];
        if (left >= 4 * (int64_t)slots) {   // whole rounds keep the order of the finish times
            const int64_t rounds = left / slots - 2;
            std::map<int64_t, int64_t> moved;
            for (const auto &t : at) moved[t.first + rounds * len] = t.second;
            at.swap(moved);
            left -= rounds * slots;
        }
        while (left > 0) {
            const auto it = at.begin();
            const int64_t t = it->first, take = std::min(left, it->second);
            if ((it->second -= take) == 0) at.erase(it);
            at[t + len] += take;
            left -= take;
        }
    }
    return (double)at.rbegin()->first;
}

// Stencil kernel and segment length of the default complex64 configuration.
// The tiled kernels march whole columns, so a block takes about a microsecond
// per plane whatever its chunk holds, and a mesh of few columns leaves SMs
// idle unless the columns are cut, which costs eight halo planes a cut; the
// plain kernel has no halo and no minimum, but costs 30 ps a vector.  The
// rule takes the smallest of these times, fitted to 14 meshes from 24^3 to
// the R = 14 sphere with 2 to 64 states (us): kernel 7, one block per SM,
// 0.97 a plane; kernel 5, two blocks per SM, 1.2 a plane, 0.92 with at most
// one block per SM; the plain kernel 5 + 30e-6 per vector (a fifth more with
// projectors in its epilogue, where the tiled kernels launch a scatter, 6 us;
// the plain complex-scaled kernel 10 + 40e-6).  Measured against the plain
// kernel, which all of these ran before: R = 10 sphere, 14 values a point:
// 64 us (115); 96^3 x 16: 78 (168); 48^3 x 16: 19 (27); R = 14 sphere x 8:
// 107 (173); 64^3 x 2: the plain kernel, 12.5 (21).
// The choice is kept with the mesh.
rsg_status choose_c64(rsg_ham H, int SV, std::pair<int, int> *choice) {
    const std::tuple<int, bool, bool> key(SV, H->has_scaling, H->pj.natoms > 0);
    rsg_mesh m = H->m;
    {
        std::lock_guard<std::mutex> lock(m->mu);
        auto it = m->choice32.find(key);
        if (it != m->choice32.end()) {
            *choice = it->second;
            return RSG_OK;
        }
    }
    const TileCfg c7 = c64_config();
    TileCfg c5 = c7;
    c5.kernel = 5;
    std::pair<int, int> best(7, c7.zseg);
    auto keep = [&]() {
        std::lock_guard<std::mutex> lock(m->mu);
        *choice = m->choice32[key] = best;
        return RSG_OK;
    };
    const int nch7 = (SV + 7) / 8, nch5 = (SV + 1) / 2;
    const bool narrow = SV % 8 != 0 && SV < 20, nl = H->pj.natoms > 0;
    int tx7, ty7, tx5, ty5;
    block_shape(c7, SV, &tx7, &ty7);
    block_shape(c5, SV, &tx5, &ty5);
    if (!narrow) {
        // enough blocks without a cut: nothing to choose
        const Tile *tiles = nullptr;
        int nt = 0;
        CKS(get_tiles(m, tx7, ty7, c7.zseg, &tiles, &nt));
        if ((int64_t)nt * nch7 >= 4 * 152) return keep();
    }
    const std::vector<int> &col7 = column_lengths(m, tx7, ty7), none;
    const std::vector<int> &col5 = SV % 8 != 0 ? column_lengths(m, tx5, ty5) : none;
    int64_t n = 0;
    const double vec = (double)m->P * SV, tiled = nl ? 8.0 : 2.0;
    const double plain = H->has_scaling ? 10.0 + 40e-6 * vec : (5.0 + 30e-6 * vec) * (nl ? 1.2 : 1.0);
    auto time7 = [&](int zs, double enough = 1e300) {
        return tiled + 0.97 * makespan(col7, zs, nch7, 152, &n, 1, 8, (enough - tiled) / 0.97);
    };
    auto time5 = [&](int zs, double enough = 1e300) {
        const double mk = makespan(col5, zs, nch5, 304, &n, 1, 8, (enough - tiled) / 0.92);
        return tiled + (n <= 152 ? 0.92 : 1.2) * mk;
    };
    // without a cut: kernel 7, kernel 5 for narrow rows with a partly empty
    // chunk, the plain kernel where that leaves SMs without a block
    double cost = narrow ? time5(150) : time7(c7.zseg);
    if (narrow) best = {5, 150};
    if (n < (narrow ? 304 : 152)) {
        best.first = 1;
        cost = plain;
    }
    cost *= 0.92;   // the fit is good to a few percent: change for a clear gain only
    if (plain < cost) {
        cost = plain;
        best.first = 1;
    }
    int last = 0;
    for (int zs : {190, 150, 96, 64, 48, 32, 24, 16, 12, 8}) {
        if (!col7.empty() && zs >= col7[0] && last >= col7[0]) continue;   // no cut either way
        last = zs;
        const double t7 = time7(zs, cost);
        if (t7 < cost) {
            cost = t7;
            best = {7, zs};
        }
        const double t5 = SV % 8 != 0 && zs <= 150 ? time5(zs, cost) : cost;
        if (t5 < cost) {
            cost = t5;
            best = {5, zs};
        }
    }
    return keep();
}

// complex128: planes per block of the integer-sum kernel, or 0 for FP64 sums,
// by the smaller of two fitted times (us): FP64 sums 6 + 125e-6 per value; the
// integer kernel 3 plus its schedule over the SMs at 2.55 a plane (two blocks
// share an SM's issue slots; a block starts in a fifth of a plane), at least
// 3.2 a plane for a block by itself.  The fit is to single applications.  In a
// chain of steps (us an application, FP64 and integer sums): 16^3 x 1 3.9 and
// 5.5 (FP64 taken); 24^3 x 1 4.2 and 6.9, 24^3 x 4 8.4 and 7.5, 32^3 x 4 16.9 and
// 12.7, 61^3 x 8 209 and 121, 96^3 x 3 292 and 168 (integers taken in all five;
// at 24^3 x 1 single applications take 8.8 and 9.2).
int choose_c128(rsg_ham H, int SV) {
    rsg_mesh m = H->m;
    {
        std::lock_guard<std::mutex> lock(m->mu);
        auto it = m->choice64.find(SV);
        if (it != m->choice64.end()) return it->second;
    }
    int tx, ty;
    sum64_shape(SV, &tx, &ty);
    const std::vector<int> &col = column_lengths(m, tx, ty);
    const int ns = sum64_states(SV), nch = (SV + ns - 1) / ns;
    int best = 0;
    double cost = 0.95 * (6.0 + 125e-6 * (double)m->P * SV);
    for (int zs : {32, 24, 16, 12, 8, 6, 4, 3, 2, 1}) {
        int64_t n = 0;
        const double mk = makespan(col, zs, nch, 152, &n, 5, 1, (cost - 3.0) / (2.55 / 5));
        const double t = 3.0 + std::max(2.55 / 5 * mk, 3.2 * (col.empty() ? 0 : std::min(zs, col[0])));
        if (t < cost) {
            cost = t;
            best = zs;
        }
    }
    std::lock_guard<std::mutex> lock(m->mu);
    return m->choice64[SV] = best;
}

// ------------------------------------------------------------ checks ----
rsg_status check_block(rsg_ham H, const void *p, int64_t S, int64_t ld, const char *what) {
    if (!p) return fail(RSG_ERR_ARG, "%s is NULL", what);
    if (S < 1 || ld < S) return fail(RSG_ERR_ARG, "need 1 <= S <= ld (S=%lld ld=%lld)",
                                     (long long)S, (long long)ld);
    if (H->dtype == RSG_C64 && (ld % 2) != 0)
        return fail(RSG_ERR_ARG, "complex64 blocks need an even ld (got %lld)", (long long)ld);
    if (((uintptr_t)p) % 16 != 0) return fail(RSG_ERR_ARG, "%s must be 16-byte aligned", what);
    if ((int64_t)ld * (int64_t)cbytes(H->dtype) / 16 > (1 << 20))
        return fail(RSG_ERR_ARG, "ld too large");
    return RSG_OK;
}

bool overlaps(const void *a, const void *b, size_t n) {
    const char *x = (const char *)a, *y = (const char *)b;
    return x < y + n && y < x + n;
}

// ------------------------------------------------------ application ----
struct Epi {
    const void *base = nullptr;
    void *acc = nullptr;
    const void *acc_base = nullptr;
    double ar = 1, ai = 0, br = 1, bi = 0, gr = 0, gi = 0;
    double shift = 0;   // applies H - shift (folded into the diagonal's constant term)
    // two-column blocks (ld = 2): column 1 has field amplitude eps1 and alpha
    // (ar1, ai1); column 0 the call's eps and (ar, ai)
    bool twocol = false;
    double eps1 = 0, ar1 = 1, ai1 = 0;
    // complex64: keep the kernel that applications of this shape have always
    // run, whose sums fix every rounding (the solvers, which amplify it)
    bool fixed_kernel = false;
};

// A potential is set: the real V, or the complex v_theta of complex scaling.
bool has_potential(rsg_ham H) { return H->has_V || H->has_scaling; }

rsg_status ensure_rows(rsg_mesh m) {
    std::lock_guard<std::mutex> lock(m->mu);
    if (m->d_rows.p) return RSG_OK;
    CK(m->d_rows.upload(m->rows));
    return RSG_OK;
}

template <typename R>
rsg_status apply_t(rsg_ham H, const void *in, void *out, int SV, double eps, const double *dir,
                   const Epi &ep, cudaStream_t st) {
    rsg_mesh m = H->m;
    CKS(ensure_rows(m));
    const double h = m->h, h3 = h * h * h;
    const int ldc = SV * (int)(16 / cbytes(H->dtype));
    if (H->pj.natoms > 0) {
        const size_t need = (size_t)H->pj.nchunks * H->pj.npmax * ldc * 2 * sizeof(double);
        CK(H->partial.ensure(need));
        CK(H->D.ensure((size_t)H->pj.natoms * H->pj.npmax * ldc * cbytes(H->dtype)));
        const size_t ncnt = (size_t)H->pj.natoms * proj_slices(SV) * sizeof(unsigned);
        if (ncnt > H->pcnt.n || !H->pcnt.p) {
            CK(H->pcnt.ensure(ncnt));
            CK(cudaMemsetAsync(H->pcnt.p, 0, H->pcnt.n, st));
        }
    }
    ApplyArgs<R> a;
    a.in = in;
    a.out = out;
    a.base = ep.base;
    a.acc = ep.acc;
    a.acc_base = ep.acc_base;
    a.rows = m->d_rows.as<Row>();
    a.nx = m->nx;
    a.ny = m->ny;
    a.nz = m->nz;
    a.SV = SV;
    a.V = H->V.as<R>();
    // eps * dir.r with r = origin + h (lo + idx)
    double f0 = 0, fd[3] = {0, 0, 0};
    if (eps != 0.0 && dir) {
        for (int d = 0; d < 3; d++) {
            f0 += eps * dir[d] * (m->origin[d] + h * m->lo[d]);
            fd[d] = eps * dir[d] * h;
        }
    }
    a.f0 = (R)(f0 - ep.shift);
    a.fx = (R)fd[0];
    a.fy = (R)fd[1];
    a.fz = (R)fd[2];
    if (ep.twocol) {
        if (SV * (int)(16 / cbytes(H->dtype)) != 2 || !dir)
            return fail(RSG_ERR_ARG, "two-column applications need ld = 2 and a field direction");
        a.twocol = 1;
        const double ec[2] = {eps, ep.eps1};
        for (int c = 0; c < 2; c++) {
            double g0 = 0;
            for (int d = 0; d < 3; d++) {
                g0 += ec[c] * dir[d] * (m->origin[d] + h * m->lo[d]);
                a.cf[c][1 + d] = (R)(ec[c] * dir[d] * h);
            }
            a.cf[c][0] = (R)(g0 - ep.shift);
        }
        a.ca[0][0] = (R)ep.ar;
        a.ca[0][1] = (R)ep.ai;
        a.ca[1][0] = (R)ep.ar1;
        a.ca[1][1] = (R)ep.ai1;
    }
    for (int k = 0; k < 5; k++) a.w[k] = (R)(-0.5 * kFD[k] / (h * h));
    a.ar = (R)ep.ar;
    a.ai = (R)ep.ai;
    a.br = (R)ep.br;
    a.bi = (R)ep.bi;
    a.gr = (R)ep.gr;
    a.gi = (R)ep.gi;
    a.ef = (a.fx != 0 || a.fy != 0 || a.fz != 0 ? EF_FIELD : 0) | (a.f0 != 0 ? EF_SHIFT : 0) |
           (ep.ar == 0 && (!ep.twocol || ep.ar1 == 0) ? EF_IMAG : 0) |
           (ep.ai == 0 && (!ep.twocol || ep.ai1 == 0) ? EF_REAL : 0) | (ep.br == 1 && ep.bi == 0 ? EF_BASE1 : 0) |
           (ep.bi == 0 ? EF_BASER : 0) | (ep.gi == 0 ? EF_GAMR : 0);
    a.nl_ptr = H->pj.natoms > 0 ? H->pj.nl_ptr : nullptr;
    a.e_atom = H->pj.e_atom;
    a.e_p = (const R *)H->pj.e_p;
    a.D = H->D.p;
    a.npmax = H->pj.npmax;
    a.P = m->P;
    if (!H->status.p) {
        CK(H->status.ensure(sizeof(int)));
        CK(cudaMemsetAsync(H->status.p, 0, sizeof(int), st));
    }
    a.err = H->status.as<int>();
    int ntiles = 0;
    a.tiles = nullptr;
    TileCfg cfg = H->cfg;
    const int ldc_v = SV * (int)(16 / cbytes(H->dtype));
    const bool chosen = H->dtype == RSG_C64 && !H->force_kernel && !ep.fixed_kernel && !ep.twocol &&
                        m->bc == RSG_BC_ZERO && !H->shape_set;
    if (chosen) {
        std::pair<int, int> choice;
        CKS(choose_c64(H, SV, &choice));
        cfg.kernel = choice.first;
        cfg.zseg = choice.second;
        if (cfg.kernel == 5) {
            cfg.threads = 192;
            cfg.stages = 3;
            cfg.sync = 0;
        }
    }
    // kernel 7 moves 16-value chunks of each point row: blocks whose rows are
    // narrow or end in a mostly empty chunk take the register-blocked kernel
    // in its default shape unless kernel 7 was chosen explicitly; complex
    // scaling runs on kernel 7 in its default shape only
    if (cfg.kernel == 7 && !chosen) {
        if ((H->has_scaling && (cfg.wty != 6 || cfg.npw != 4)) ||
            (!H->force_kernel && ldc_v % 16 != 0 && ldc_v < 40)) {
            cfg.kernel = 5;
            cfg.threads = 192;
            cfg.zseg = 150;
            cfg.stages = 3;
            cfg.sync = 0;
        }
    }
    // kernels 2 and 3 keep a static row table of at most 120-plane segments
    if ((cfg.kernel == 2 || cfg.kernel == 3) && cfg.zseg > 120) cfg.zseg = 120;
    // two-column applications run on the one-thread-per-value kernel
    if (ep.twocol) cfg.kernel = 1;
    if (H->dtype == RSG_C128 && cfg.kernel == 1 && m->bc == RSG_BC_ZERO && !H->has_scaling)
        cfg.sum_zs = H->sum_planes >= 0 ? H->sum_planes : choose_c128(H, SV);
    H->last_zseg = 0;
    H->last_sum = cfg.sum_zs;
    if (cfg.kernel != 1) {
        int TX, TY;
        block_shape(cfg, SV, &TX, &TY);
        CKS(get_tiles(m, TX, TY, cfg.zseg, &a.tiles, &ntiles));
        if (cfg.kernel != 1 && cfg.kernel != 2 && !H->force_kernel && !chosen) {
            // the staged kernel runs one block per SM: small problems that
            // give fewer than two blocks per SM go to the one-thread-per-value
            // kernel instead
            int cv, nxr, ty;
            stage_shape(cfg, SV, &cv, &nxr, &ty);
            if (cfg.kernel == 7) cv = 8;   // 128-byte chunks: 8 vectors
            if ((int64_t)ntiles * ((SV + cv - 1) / cv) < (cfg.kernel == 7 ? 152 : 2 * 152)) {
                log_info("small problem (%d tiles): one-thread-per-value kernel instead of kernel %d", ntiles,
                         cfg.kernel);
                cfg.kernel = 1;
            }
        }
    }
    const bool odd = m->bc == RSG_BC_ODD;
    const bool split_nl = !odd && !H->has_scaling && cfg.kernel != 1 && cfg.kernel != 2 && H->pj.natoms > 0;
    // projector coefficients D = h_a h^3 <p|in>: read by the stencil itself
    // when it adds the projector terms (kernels 1, 2), else only by the
    // scatter after it; with "proj_overlap" they then run on a side stream
    // next to the stencil
    bool joined = true;
    if (H->pj.natoms > 0) {
        cudaStream_t cs = st;
        if (split_nl && H->proj_overlap) {
            if (!H->side) {
                CK(cudaStreamCreateWithFlags(&H->side, cudaStreamNonBlocking));
                CK(cudaEventCreateWithFlags(&H->ev_fork, cudaEventDisableTiming));
                CK(cudaEventCreateWithFlags(&H->ev_join, cudaEventDisableTiming));
            }
            CK(cudaEventRecord(H->ev_fork, st));
            CK(cudaStreamWaitEvent(H->side, H->ev_fork, 0));
            cs = H->side;
            joined = false;
        }
        CK(launch_proj_coeffs<R>(in, SV, H->pj, H->partial.as<double>(), H->pcnt.as<unsigned>(), h3, H->D.p,
                                 split_nl && joined, cs));
        if (!joined) CK(cudaEventRecord(H->ev_join, H->side));
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (H->prof) {
        if (H->ev_used + 2 > H->ev.size()) {
            for (int i = 0; i < 64; i++) {
                cudaEvent_t e;
                CK(cudaEventCreate(&e));
                H->ev.push_back(e);
            }
        }
        e0 = H->ev[H->ev_used];
        e1 = H->ev[H->ev_used + 1];
        H->ev_used += 2;
        CK(cudaEventRecord(e0, st));
    }
    if (odd) {
        // image walls: the one-thread-per-value kernels, neighbours through the image rule
        if (H->has_scaling) {
            CK(launch_apply_scaled_odd<R>(a, H->vtheta.as<R>(), H->theta, st));
            H->last_kernel = 6;
        } else {
            CK(launch_apply_naive_odd<R>(a, st));
            H->last_kernel = 1;
        }
    } else if (H->has_scaling) {
        // complex-scaled operator (no projectors, no field: refused while set)
        bool done = false;
        if constexpr (std::is_same<R, float>::value) {
            // register-blocked kernel: alpha (lap + v_theta e^{2i theta} u) with
            // alpha rotated by e^{-2i theta}, without a diagonal constant
            if ((cfg.kernel == 5 || cfg.kernel == 7) && a.f0 == 0.f && a.fx == 0.f && a.fy == 0.f && a.fz == 0.f) {
                ApplyArgs<R> b = a;
                b.Vc = H->vtheta_rot.p;
                b.nl_ptr = nullptr;
                const double kr = std::cos(2.0 * H->theta), ki = -std::sin(2.0 * H->theta);
                b.ar = (R)(ep.ar * kr - ep.ai * ki);
                b.ai = (R)(ep.ar * ki + ep.ai * kr);
                if (cfg.kernel == 7) {
                    CK(launch_apply_wide(b, cfg, ntiles, st, &done));
                    if (done) H->last_kernel = 7;
                } else {
                    CK(launch_apply_quad(b, cfg, ntiles, st, &done));
                    if (done) H->last_kernel = 5;
                }
            }
        }
        if (!done) {
            CK(launch_apply_scaled<R>(a, H->vtheta.as<R>(), H->theta, st));
            H->last_kernel = 6;
        }
    } else {
        ApplyArgs<R> b = a;
        if (split_nl) b.nl_ptr = nullptr;
        bool done = false;
        if (cfg.kernel == 3) CK(launch_apply_tma<R>(b, cfg, ntiles, st, &done));
        if (cfg.kernel == 4) CK(launch_apply_rowtma<R>(b, cfg, ntiles, st, &done));
        if constexpr (std::is_same<R, float>::value) {
            if (cfg.kernel == 5) CK(launch_apply_quad(b, cfg, ntiles, st, &done));
            if (cfg.kernel == 7) CK(launch_apply_wide(b, cfg, ntiles, st, &done));
        }
        if (done) {
            H->last_kernel = cfg.kernel;
        } else {
            TileCfg c0 = cfg;
            int n = ntiles;
            if (c0.kernel >= 3) log_info("kernel %d not available for this block shape: kernel 0 runs", c0.kernel);
            if (c0.kernel >= 3) {
                // same tiles for kernel 4 (the staged block shape)
                const bool retile = c0.kernel != 4;
                c0.kernel = 0;
                if (retile) n = tiles_for(H, c0, SV, &b.tiles);
            }
            CK(launch_apply<R>(b, c0, n, st));
            H->last_kernel = c0.kernel;
        }
    }
    if (H->prof) CK(cudaEventRecord(e1, st));
    if (!joined) CK(cudaStreamWaitEvent(st, H->ev_join, 0));
    if (split_nl) {
        CK(launch_proj_scatter<R>(a, H->pj, st));
        H->n_launch++;
    }
    if (H->last_kernel != 1 && H->last_kernel != 6) H->last_zseg = cfg.zseg;
    // algorithmic bytes: read u, write out, optional base / acc (read+write),
    // the potential, and (with projectors) the per-point entry lists,
    // entry values and the coefficient block
    const double P = (double)m->P, row = 16.0 * SV;
    double bytes = P * row * (2.0 + (ep.base ? 1.0 : 0.0) + (ep.acc ? 2.0 : 0.0)) +
                   P * sizeof(R) * (H->has_scaling ? 2.0 : 1.0);
    if (H->pj.natoms > 0 && !split_nl)
        bytes += 4.0 * (P + 1) + (double)H->pj.nq * (8.0 + H->pj.npmax * sizeof(R)) +
                 (double)H->pj.natoms * H->pj.npmax * row;
    H->n_stencil += ep.twocol ? 2 : 1;   // Hamiltonian applications (two per two-column launch)
    H->stencil_bytes += bytes;
    H->n_launch += H->pj.natoms > 0 ? 2 : 1;   // the stencil and the coefficient kernel (the scatter counts above)
    return RSG_OK;
}

rsg_status apply(rsg_ham H, const void *in, void *out, int SV, double eps, const double *dir,
                 const Epi &ep, cudaStream_t st) {
    if (H->dtype == RSG_C64) return apply_t<float>(H, in, out, SV, eps, dir, ep, st);
    return apply_t<double>(H, in, out, SV, eps, dir, ep, st);
}

int sv_of(rsg_ham H, int64_t ld) { return (int)(ld * (int64_t)cbytes(H->dtype) / 16); }

// out = T(tau) psi by Horner's rule: u <- psi; u <- psi + (-i tau / k) H u
// for k = 4..1.  out may equal psi.
rsg_status taylor(rsg_ham H, const void *psi, void *out, int64_t ld, double tau, double eps,
                  const double *dir, cudaStream_t st) {
    const size_t bytes = (size_t)H->m->P * ld * cbytes(H->dtype);
    CK(H->w0.ensure(bytes));
    CK(H->w1.ensure(bytes));
    const int SV = sv_of(H, ld);
    const void *src = psi;
    for (int k = 4; k >= 1; k--) {
        void *dst = (k == 1) ? out : ((k & 1) ? H->w1.p : H->w0.p);
        Epi ep;
        ep.ar = 0.0;
        ep.ai = -tau / k;
        ep.base = psi;
        ep.br = 1.0;
        ep.bi = 0.0;
        CKS(apply(H, src, dst, SV, eps, dir, ep, st));
        src = dst;
    }
    return RSG_OK;
}

// ------------------------------------------------------------ linalg ----
rsg_status norms_dev(rsg_ham H, const void *psi, int64_t S, int64_t ld, double *out_dev,
                     cudaStream_t st) {
    const int64_t P = H->m->P;
    const double h3 = std::pow(H->m->h, 3);
    const int nb = norm_blocks(P);
    CK(H->red.ensure((size_t)nb * S * sizeof(double)));
    if (H->dtype == RSG_C64)
        CK(launch_norms<float>(psi, P, (int)ld, (int)S, h3, H->red.as<double>(), nb, out_dev, st));
    else
        CK(launch_norms<double>(psi, P, (int)ld, (int)S, h3, H->red.as<double>(), nb, out_dev, st));
    H->n_launch += 2;
    return RSG_OK;
}

// Cholesky-QR on the device; drift (device, S) updated with |G_ss - 1|.
rsg_status orthonormalize_dev(rsg_ham H, void *psi, int64_t S, int64_t ld, double *drift_dev,
                              cudaStream_t st) {
    const int64_t P = H->m->P;
    const double h3 = std::pow(H->m->h, 3);
    const int nb = gram_blocks(P, (int)S);
    CK(H->red.ensure((size_t)nb * S * S * 2 * sizeof(double)));
    CK(H->G.ensure((size_t)S * S * 2 * sizeof(double)));
    CK(H->W.ensure((size_t)S * S * 2 * sizeof(double)));
    if (!H->status.p) {
        CK(H->status.ensure(sizeof(int)));
        CK(cudaMemsetAsync(H->status.p, 0, sizeof(int), st));
    }
    if (H->dtype == RSG_C64) {
        // FP64 norms for the diagonal, FP32 runs in two-float and FP64 sums elsewhere
        const size_t nrm_bytes = ((size_t)S * sizeof(double) + 255) / 256 * 256;
        CK(H->Wc.ensure(nrm_bytes + tri_c64_bytes((int)S)));
        double *nrm = H->Wc.as<double>();
        CKS(norms_dev(H, psi, S, ld, nrm, st));
        CK(launch_gram_c64(psi, P, (int)ld, (int)S, h3, H->red.as<double>(), nb, H->G.as<double>(), nrm, st));
        CK(launch_chol_inv(H->G.as<double>(), H->W.as<double>(), (int)S, drift_dev, H->status.as<int>(), st));
        CK(launch_tri_apply_c64(psi, P, (int)ld, (int)S, H->W.as<double>(), (char *)H->Wc.p + nrm_bytes, st));
    } else {
        CK(launch_gram<double>(psi, P, (int)ld, (int)S, h3, H->red.as<double>(), nb, H->G.as<double>(), st));
        CK(launch_chol_inv(H->G.as<double>(), H->W.as<double>(), (int)S, drift_dev, H->status.as<int>(), st));
        CK(launch_tri_apply<double>(psi, P, (int)ld, (int)S, H->W.as<double>(), st));
    }
    H->n_launch += 4;
    return RSG_OK;
}

rsg_status read_status(rsg_ham H, cudaStream_t st) {
    if (!H->status.p) return RSG_OK;
    int s = 0;
    CK(cudaMemcpyAsync(&s, H->status.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (s != 0) {
        CK(cudaMemsetAsync(H->status.p, 0, sizeof(int), st));
        CK(cudaStreamSynchronize(st));
        if (s == 2) return fail(RSG_ERR_TIMEOUT, "a bounded device wait gave up");
        if (s == 3) return fail(RSG_ERR_CUDA, "TMA destination not 128-byte aligned (copy skipped)");
        return fail(RSG_ERR_NONFINITE, "Gram matrix not finite or not positive definite");
    }
    return RSG_OK;
}

// ------------------------------------------------------- projectors ----
double solid_harmonic(int i, double x, double y, double z) {
    switch (i) {
    case 0: return 1.0;
    case 1: return x;
    case 2: return y;
    case 3: return z;
    case 4: return x * y;
    case 5: return y * z;
    case 6: return z * x;
    case 7: return x * x - y * y;
    default: return 3.0 * z * z - (x * x + y * y + z * z);
    }
}

template <typename R>
std::vector<R> cast_vec(const std::vector<double> &v) {
    return std::vector<R>(v.begin(), v.end());
}

}  // namespace

namespace rsg {
void ham_info(rsg_ham H, rsg_dtype *dtype, int64_t *P, double *spacing) {
    *dtype = H->dtype;
    *P = H->m->P;
    *spacing = H->m->h;
}
rsg_status set_error(rsg_status s, const char *msg) { return fail(s, "%s", msg); }
}  // namespace rsg

// ===================================================================== ABI

extern "C" {

const char *rsg_last_error(void) { return g_err.c_str(); }

rsg_status rsg_mesh_set_boundary(rsg_mesh m, int bc) {
    if (!m) return fail(RSG_ERR_ARG, "NULL mesh");
    if (bc != RSG_BC_ZERO && bc != RSG_BC_ODD) return fail(RSG_ERR_ARG, "unknown boundary rule %d", bc);
    if (bc == RSG_BC_ODD && m->shape == RSG_SHAPE_SPHERE)
        return fail(RSG_ERR_UNSUPPORTED, "image walls need a cube or a box");
    // the kernels reflect a neighbour once; with at least 4 points per axis
    // every neighbour up to 4 spacings away has its image inside the mesh
    if (bc == RSG_BC_ODD && (m->nx < 4 || m->ny < 4 || m->nz < 4))
        return fail(RSG_ERR_ARG, "image walls need at least 4 points along every axis (%d x %d x %d)", m->nx, m->ny,
                    m->nz);
    m->bc = bc;
    return RSG_OK;
}

rsg_status rsg_mesh_create(rsg_shape shape, const int32_t n[3], double radius, double spacing,
                           rsg_mesh *out) {
    if (!out) return fail(RSG_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!(spacing > 0.0) || !std::isfinite(spacing)) return fail(RSG_ERR_ARG, "spacing must be > 0");
    std::unique_ptr<rsg_mesh_s> m(new rsg_mesh_s());
    m->shape = shape;
    m->h = spacing;
    int64_t r2max = 0;
    if (shape == RSG_SHAPE_CUBE || shape == RSG_SHAPE_BOX) {
        if (!n) return fail(RSG_ERR_ARG, "n is NULL");
        int N[3];
        for (int d = 0; d < 3; d++) N[d] = shape == RSG_SHAPE_CUBE ? n[0] : n[d];
        for (int d = 0; d < 3; d++)
            if (N[d] < 1 || N[d] > 1024) return fail(RSG_ERR_ARG, "extent %d outside 1..1024", N[d]);
        m->nx = N[0];
        m->ny = N[1];
        m->nz = N[2];
        for (int d = 0; d < 3; d++) {
            m->lo[d] = 0;
            m->origin[d] = -0.5 * (N[d] - 1) * spacing;
        }
    } else if (shape == RSG_SHAPE_SPHERE) {
        if (!(radius > 0.0) || !std::isfinite(radius)) return fail(RSG_ERR_ARG, "radius must be > 0");
        const double q = radius / spacing;
        r2max = (int64_t)std::floor(q * q + 1e-6);
        int M = (int)std::floor(std::sqrt((double)r2max) + 1e-9);
        if (2 * M + 1 > 1024) return fail(RSG_ERR_ARG, "sphere extent %d exceeds 1024", 2 * M + 1);
        m->nx = m->ny = m->nz = 2 * M + 1;
        for (int d = 0; d < 3; d++) {
            m->lo[d] = -M;
            m->origin[d] = 0.0;
        }
    } else {
        return fail(RSG_ERR_ARG, "unknown shape %d", (int)shape);
    }
    build_rows(m.get(), r2max);
    if (m->P >= (int64_t)INT32_MAX) return fail(RSG_ERR_UNSUPPORTED, "more than 2^31 points");
    // the device copy of the row table is made on first use
    *out = m.release();
    return RSG_OK;
}

rsg_status rsg_mesh_num_points(rsg_mesh m, int64_t *P) {
    if (!m || !P) return fail(RSG_ERR_ARG, "NULL argument");
    *P = m->P;
    return RSG_OK;
}

rsg_status rsg_mesh_coords(rsg_mesh m, int32_t *ijk) {
    if (!m || !ijk) return fail(RSG_ERR_ARG, "NULL argument");
    std::memcpy(ijk, m->ijk.data(), m->ijk.size() * sizeof(int32_t));
    return RSG_OK;
}

rsg_status rsg_mesh_geometry(rsg_mesh m, double origin[3], double *spacing) {
    if (!m || !origin || !spacing) return fail(RSG_ERR_ARG, "NULL argument");
    for (int d = 0; d < 3; d++) origin[d] = m->origin[d];
    *spacing = m->h;
    return RSG_OK;
}

rsg_status rsg_mesh_destroy(rsg_mesh m) {
    delete m;
    return RSG_OK;
}

rsg_status rsg_ham_create(rsg_mesh m, rsg_dtype dtype, rsg_ham *out) {
    if (!m || !out) return fail(RSG_ERR_ARG, "NULL argument");
    if (dtype != RSG_C64 && dtype != RSG_C128) return fail(RSG_ERR_ARG, "unknown dtype");
    rsg_ham H = new rsg_ham_s();
    H->m = m;
    H->dtype = dtype;
    // complex128 is bound by FP64 arithmetic: the one-thread-per-value kernel
    // does the least of it.  complex64 runs the warp-specialised tensor-copy
    // kernel (16 x 6 tiles, four producer warps, 190-plane segments: fastest
    // on the sphere workloads measured); narrow blocks and complex scaling
    // run the register-blocked kernel (apply_t)
    if (dtype == RSG_C128)
        H->cfg.kernel = 1;
    else
        H->cfg = c64_config();
    *out = H;
    return RSG_OK;
}

rsg_status rsg_ham_destroy(rsg_ham H) {
    delete H;
    return RSG_OK;
}

rsg_status rsg_ham_profile(rsg_ham H, int enable) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    H->prof = enable != 0;
    return RSG_OK;
}

rsg_status rsg_ham_kernel_stats(rsg_ham H, double *kernel_ms, int64_t *kernel_launches,
                                double *kernel_bytes, int64_t *all_launches) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    double ms = 0.0;
    for (size_t i = 0; i + 1 < H->ev_used; i += 2) {
        CK(cudaEventSynchronize(H->ev[i + 1]));
        float t = 0.f;
        CK(cudaEventElapsedTime(&t, H->ev[i], H->ev[i + 1]));
        ms += t;
    }
    if (kernel_ms) *kernel_ms = ms;
    if (kernel_launches) *kernel_launches = H->n_stencil;
    if (kernel_bytes) *kernel_bytes = H->stencil_bytes;
    if (all_launches) *all_launches = H->n_launch;
    H->ev_used = 0;
    H->n_stencil = 0;
    H->stencil_bytes = 0.0;
    H->n_launch = 0;
    return RSG_OK;
}

rsg_status rsg_ham_autotune(rsg_ham H, const void *psi, void *work, int64_t S, int64_t ld, void *stream,
                            double *best_ms) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    CKS(check_block(H, psi, S, ld, "psi"));
    CKS(check_block(H, work, S, ld, "work"));
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    const size_t bytes = (size_t)H->m->P * ld * cbytes(H->dtype);
    if (overlaps(psi, work, bytes)) return fail(RSG_ERR_ARG, "psi and work overlap");
    cudaStream_t st = (cudaStream_t)stream;
    // candidates: the one-thread-per-value kernel and the staged kernel in
    // the block shapes that fit the SM (timed as a Horner stage)
    std::vector<TileCfg> cand;
    {
        TileCfg c;
        c.kernel = 1;
        cand.push_back(c);
    }
    const int shapes[][3] = {{256, 2, 3}, {256, 2, 4}, {256, 4, 4}, {512, 4, 4}, {512, 8, 4}, {512, 2, 4}};
    for (const auto &sh : shapes)
        for (int zs : {64, 120}) {
            TileCfg c;
            c.kernel = 0;
            c.threads = sh[0];
            c.cv = sh[1];
            c.stages = sh[2];
            c.zseg = zs;
            cand.push_back(c);
        }
    // the register-blocked staged kernel (complex64): 192 or 256 threads
    for (int th : {192, 256})
        for (int zs : {96, 120}) {
            TileCfg c;
            c.kernel = 5;
            c.threads = th;
            c.zseg = zs;
            cand.push_back(c);
        }
    // the warp-specialised tensor-copy kernel (complex64): tile rows, producer
    // warps and segment length
    const int wshapes[][3] = {{6, 4, 190}, {6, 3, 190}, {6, 2, 190}, {8, 4, 150}, {8, 2, 150}, {4, 4, 190}};
    for (const auto &sh : wshapes) {
        TileCfg c;
        c.kernel = 7;
        c.wty = sh[0];
        c.npw = sh[1];
        c.zseg = sh[2];
        c.stages = 3;
        cand.push_back(c);
    }
    // the row-TMA staged kernel: 256 threads with 4 or 5 slots, 512 with 6
    const int rshapes[][3] = {{256, 2, 4}, {256, 2, 5}, {512, 2, 4}};
    for (const auto &sh : rshapes)
        for (int zs : {96, 120}) {
            TileCfg c;
            c.kernel = 4;
            c.threads = sh[0];
            c.cv = sh[1];
            c.stages = sh[2];
            c.zseg = zs;
            cand.push_back(c);
        }
    const TileCfg saved = H->cfg;
    const bool saved_force = H->force_kernel;
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    double best = 1e30;
    TileCfg pick = saved;
    const int SV = sv_of(H, ld);
    for (const TileCfg &c : cand) {
        H->cfg = c;
        H->force_kernel = true;
        Epi ep;
        ep.ar = 0.0;
        ep.ai = -1e-3;
        ep.base = psi;
        if (apply(H, psi, work, SV, 0.0, nullptr, ep, st) != RSG_OK) continue;   // shape not usable
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; r++) apply(H, psi, work, SV, 0.0, nullptr, ep, st);
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) break;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms / 3 < best && H->last_kernel == c.kernel) {
            best = ms / 3;
            pick = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaGetLastError();
    H->cfg = best < 1e30 ? pick : saved;
    H->force_kernel = best < 1e30 ? true : saved_force;
    if (best_ms) *best_ms = best < 1e30 ? best : -1.0;
    return best < 1e30 ? read_status(H, st) : fail(RSG_ERR_CUDA, "no candidate ran");
}

rsg_status rsg_ham_get_option(rsg_ham H, const char *key, int64_t *value) {
    if (!H || !key || !value) return fail(RSG_ERR_ARG, "NULL argument");
    std::string k(key);
    if (k == "kernel") *value = H->cfg.kernel;
    else if (k == "last_kernel") *value = H->last_kernel;
    else if (k == "last_zseg") *value = H->last_zseg;
    else if (k == "last_sum_planes") *value = H->last_sum;
    else if (k == "sum_planes") *value = H->sum_planes;
    else if (k == "rx") *value = H->cfg.rx;
    else if (k == "ty") *value = H->cfg.ty;
    else if (k == "wide_ty") *value = H->cfg.wty;
    else if (k == "producers") *value = H->cfg.npw;
    else if (k == "zseg") *value = H->cfg.zseg;
    else if (k == "cv") *value = H->cfg.cv;
    else if (k == "threads") *value = H->cfg.threads;
    else if (k == "sync") *value = H->cfg.sync;
    else if (k == "stages") *value = H->cfg.stages;
    else if (k == "blocks_per_sm") *value = H->cfg.blocks_per_sm;
    else if (k == "proj_overlap") *value = H->proj_overlap;
    else return fail(RSG_ERR_ARG, "unknown option: %s", key);
    return RSG_OK;
}

rsg_status rsg_ham_set_option(rsg_ham H, const char *key, int64_t value) {
    if (!H || !key) return fail(RSG_ERR_ARG, "NULL argument");
    std::string k(key);
    if (k == "kernel" && ((value >= 0 && value <= 5) || value == 7)) {
        H->cfg.kernel = (int)value;
        H->force_kernel = true;
    }
    else if (k == "rx" && (value == 1 || value == 2 || value == 4)) H->cfg.rx = (int)value;
    else if (k == "ty" && (value == 1 || value == 2 || value == 4 || value == 8 || value == 16))
        H->cfg.ty = (int)value;
    else if (k == "zseg" && value >= 1 && value <= 256) H->cfg.zseg = (int)value;
    else if (k == "wide_ty" && (value == 4 || value == 6 || value == 8)) H->cfg.wty = (int)value;
    else if (k == "producers" && value >= 1 && value <= 4) H->cfg.npw = (int)value;
    else if (k == "cv" && (value == 1 || value == 2 || value == 4 || value == 8)) H->cfg.cv = (int)value;
    else if (k == "adjoint_keep_powers" && value >= -1 && value <= 1) H->adj_keep = (int)value;
    else if (k == "adjoint_merge" && value >= -1 && value <= 1) H->adj_merge = (int)value;
    else if (k == "proj_overlap" && (value == 0 || value == 1)) H->proj_overlap = (int)value;
    else if (k == "sum_planes" && value >= -1 && value <= 32) H->sum_planes = (int)value;
    else if (k == "threads" && (value == 160 || value == 192 || value == 256 || value == 512))
        H->cfg.threads = (int)value;
    else if (k == "sync" && value >= 0 && value <= 2) H->cfg.sync = (int)value;
    else if (k == "stages" && value >= 3 && value <= 5) H->cfg.stages = (int)value;
    else if (k == "blocks_per_sm" && (value == 2 || value == 3)) H->cfg.blocks_per_sm = (int)value;
    else return fail(RSG_ERR_ARG, "unknown option or value: %s=%lld", key, (long long)value);
    if (k == "zseg" || k == "wide_ty" || k == "producers" || k == "threads" || k == "sync" || k == "stages")
        H->shape_set = true;
    return RSG_OK;
}

rsg_status rsg_potential_set(rsg_ham H, const double *v, int v_on_device) {
    if (!H || !v) return fail(RSG_ERR_ARG, "NULL argument");
    const int64_t P = H->m->P;
    std::vector<double> hv((size_t)P);
    if (v_on_device)
        CK(cudaMemcpy(hv.data(), v, (size_t)P * sizeof(double), cudaMemcpyDeviceToHost));
    else
        std::memcpy(hv.data(), v, (size_t)P * sizeof(double));
    for (int64_t p = 0; p < P; p++)
        if (!std::isfinite(hv[p])) return fail(RSG_ERR_ARG, "potential not finite at %lld", (long long)p);
    if (H->dtype == RSG_C64)
        CK(H->V.upload(cast_vec<float>(hv)));
    else
        CK(H->V.upload(hv));
    H->has_V = true;
    H->vmin = P ? *std::min_element(hv.begin(), hv.end()) : 0.0;
    H->vmax = P ? *std::max_element(hv.begin(), hv.end()) : 0.0;
    return RSG_OK;
}

rsg_status rsg_absorber_set(rsg_ham H, const double *mask, int mask_on_device) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    if (!mask) {
        H->has_mask = false;
        return RSG_OK;
    }
    const int64_t P = H->m->P;
    std::vector<double> hm((size_t)P);
    if (mask_on_device)
        CK(cudaMemcpy(hm.data(), mask, (size_t)P * sizeof(double), cudaMemcpyDeviceToHost));
    else
        std::memcpy(hm.data(), mask, (size_t)P * sizeof(double));
    for (int64_t p = 0; p < P; p++)
        if (!(hm[(size_t)p] >= 0.0 && hm[(size_t)p] <= 1.0))
            return fail(RSG_ERR_ARG, "mask value outside [0, 1] at %lld", (long long)p);
    if (H->dtype == RSG_C64)
        CK(H->mask.upload(cast_vec<float>(hm)));
    else
        CK(H->mask.upload(hm));
    H->has_mask = true;
    return RSG_OK;
}

rsg_status rsg_complex_scaling_set(rsg_ham H, double theta, const double *v_theta, int v_on_device) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    if (!v_theta) {
        H->has_scaling = false;
        H->theta = 0.0;
        return RSG_OK;
    }
    if (!(theta >= 0.0 && theta <= 0.78539816339744830962)) return fail(RSG_ERR_ARG, "theta outside [0, pi/4]");
    if (H->pj.natoms > 0) return fail(RSG_ERR_UNSUPPORTED, "projectors are set: complex scaling takes none");
    if (H->eps != 0.0) return fail(RSG_ERR_UNSUPPORTED, "a dipole field is set: complex scaling takes none");
    const int64_t P = H->m->P;
    std::vector<double> hv((size_t)(2 * P));
    if (v_on_device)
        CK(cudaMemcpy(hv.data(), v_theta, (size_t)(2 * P) * sizeof(double), cudaMemcpyDeviceToHost));
    else
        std::memcpy(hv.data(), v_theta, (size_t)(2 * P) * sizeof(double));
    for (int64_t i = 0; i < 2 * P; i++)
        if (!std::isfinite(hv[(size_t)i])) return fail(RSG_ERR_ARG, "v_theta not finite at %lld", (long long)(i / 2));
    if (H->dtype == RSG_C64) {
        CK(H->vtheta.upload(cast_vec<float>(hv)));
        const double cr = std::cos(2.0 * theta), ci = std::sin(2.0 * theta);
        std::vector<float> rot((size_t)(2 * P));
        for (int64_t p = 0; p < P; p++) {
            const double re = hv[(size_t)(2 * p)], im = hv[(size_t)(2 * p + 1)];
            rot[(size_t)(2 * p)] = (float)(re * cr - im * ci);
            rot[(size_t)(2 * p + 1)] = (float)(re * ci + im * cr);
        }
        CK(H->vtheta_rot.upload(rot));
    } else {
        CK(H->vtheta.upload(hv));
    }
    H->theta = theta;
    H->has_scaling = true;
    return RSG_OK;
}

rsg_status rsg_field_set(rsg_ham H, double eps, const double dir[3]) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    if (eps != 0.0 && !dir) return fail(RSG_ERR_ARG, "dir is NULL");
    if (eps != 0.0 && H->has_scaling) return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: no dipole field");
    H->eps = eps;
    if (dir)
        for (int d = 0; d < 3; d++) H->dir[d] = dir[d];
    return RSG_OK;
}

// Device tables of a projector set from its entry list: entry q is point
// q_pt[q] of atom q_atom[q] with the npmax values q_p[q * npmax + i]; the
// entries of each atom are contiguous and cut into chunks of at most kProjChunk
// (ch_atom, ch_q0, ch_q1; atom_ch0 = per-atom prefix of chunks); hm holds the
// zero-padded npmax x npmax coupling matrices.
static rsg_status upload_projectors(rsg_ham H, int natoms, int npmax, const std::vector<int32_t> &q_pt,
                                    const std::vector<int32_t> &q_atom, const std::vector<double> &q_p,
                                    const std::vector<int32_t> &ch_atom, const std::vector<int32_t> &ch_q0,
                                    const std::vector<int32_t> &ch_q1, const std::vector<int32_t> &atom_ch0,
                                    const std::vector<double> &hm) {
    rsg_mesh m = H->m;
    // point-centric CSR of entries (for the fused scatter in the epilogue)
    const int64_t P = m->P;
    std::vector<int32_t> nl_ptr((size_t)P + 1, 0), nl_ent(q_pt.size());
    for (int32_t p : q_pt) nl_ptr[(size_t)p + 1]++;
    for (int64_t p = 0; p < P; p++) nl_ptr[(size_t)p + 1] += nl_ptr[(size_t)p];
    {
        std::vector<int32_t> fill(nl_ptr.begin(), nl_ptr.end() - 1);
        for (size_t q = 0; q < q_pt.size(); q++) nl_ent[(size_t)fill[(size_t)q_pt[q]]++] = (int32_t)q;
    }
    CK(H->q_pt.upload(q_pt));
    if (H->dtype == RSG_C64)
        CK(H->q_p.upload(cast_vec<float>(q_p)));
    else
        CK(H->q_p.upload(q_p));
    CK(H->ch_atom.upload(ch_atom));
    CK(H->ch_q0.upload(ch_q0));
    CK(H->ch_q1.upload(ch_q1));
    CK(H->atom_ch0.upload(atom_ch0));
    CK(H->hm.upload(hm));
    CK(H->nl_ptr.upload(nl_ptr));
    std::vector<int32_t> u_pts, u_ptr(1, 0);
    for (int64_t p = 0; p < P; p++)
        if (nl_ptr[(size_t)p + 1] > nl_ptr[(size_t)p]) {
            u_pts.push_back((int32_t)p);
            u_ptr.push_back(nl_ptr[(size_t)p + 1]);
        }
    CK(H->u_pts.upload(u_pts));
    CK(H->u_ptr.upload(u_ptr));
    // point-major copies of each entry's atom and projector values, so the
    // scatter reads them without going through the entry index
    std::vector<int32_t> e_atom(nl_ent.size());
    std::vector<double> e_p(nl_ent.size() * (size_t)std::max(npmax, 1));
    for (size_t e = 0; e < nl_ent.size(); e++) {
        const size_t q = (size_t)nl_ent[e];
        e_atom[e] = q_atom[q];
        for (int i = 0; i < npmax; i++) e_p[e * npmax + i] = q_p[q * npmax + i];
    }
    CK(H->e_atom.upload(e_atom));
    if (H->dtype == RSG_C64)
        CK(H->e_p.upload(cast_vec<float>(e_p)));
    else
        CK(H->e_p.upload(e_p));
    ProjDev &pj = H->pj;
    pj.natoms = natoms;
    pj.npmax = npmax;
    pj.nq = (int64_t)q_pt.size();
    pj.nchunks = (int)ch_q0.size();
    pj.q_pt = H->q_pt.as<int32_t>();
    pj.q_p = H->q_p.p;
    pj.chunk_atom = H->ch_atom.as<int32_t>();
    pj.chunk_q0 = H->ch_q0.as<int32_t>();
    pj.chunk_q1 = H->ch_q1.as<int32_t>();
    pj.atom_chunk0 = H->atom_ch0.as<int32_t>();
    pj.hm = H->hm.as<double>();
    pj.nl_ptr = H->nl_ptr.as<int32_t>();
    pj.nu = (int)u_pts.size();
    pj.u_pts = H->u_pts.as<int32_t>();
    pj.u_ptr = H->u_ptr.as<int32_t>();
    pj.e_atom = H->e_atom.as<int32_t>();
    pj.e_p = H->e_p.p;
    return RSG_OK;
}

rsg_status rsg_projectors_set(rsg_ham H, int natoms, const double *centres, const double *rcut,
                              const int32_t *lmax, const double *beta, const double *hmats) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    if (natoms < 0) return fail(RSG_ERR_ARG, "natoms < 0");
    if (natoms > 0 && H->has_scaling) return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: no projectors");
    H->pj = ProjDev();
    H->proj_norm = 0.0;
    if (natoms == 0) return RSG_OK;
    if (!centres || !rcut || !lmax || !beta || !hmats) return fail(RSG_ERR_ARG, "NULL array");
    rsg_mesh m = H->m;
    const double h = m->h, h3 = h * h * h;
    int npmax = 1;
    for (int a = 0; a < natoms; a++) {
        if (lmax[a] < 0 || lmax[a] > 2) return fail(RSG_ERR_UNSUPPORTED, "lmax must be 0, 1 or 2");
        if (!(rcut[a] > 0) || !(beta[a] > 0)) return fail(RSG_ERR_ARG, "rcut and beta must be > 0");
        npmax = std::max(npmax, (lmax[a] + 1) * (lmax[a] + 1));
    }
    std::vector<int32_t> q_pt, q_atom, ch_atom, ch_q0, ch_q1, atom_ch0(1, 0);
    std::vector<double> q_p, hm((size_t)natoms * npmax * npmax, 0.0);
    int64_t hoff = 0;
    for (int a = 0; a < natoms; a++) {
        const int np = (lmax[a] + 1) * (lmax[a] + 1);
        const double *c = centres + 3 * a;
        const double rc = rcut[a], b2 = 2.0 * beta[a] * beta[a];
        const size_t q_begin = q_pt.size();
        // bounding box of the sphere in bbox indices
        int lo3[3], hi3[3];
        for (int d = 0; d < 3; d++) {
            const int ext = d == 0 ? m->nx : d == 1 ? m->ny : m->nz;
            lo3[d] = std::max(0, (int)std::floor((c[d] - rc - m->origin[d]) / h) - m->lo[d] - 1);
            hi3[d] = std::min(ext - 1, (int)std::ceil((c[d] + rc - m->origin[d]) / h) - m->lo[d] + 1);
        }
        for (int z = lo3[2]; z <= hi3[2]; z++)
            for (int y = lo3[1]; y <= hi3[1]; y++) {
                const Row &rw = m->rows[(size_t)z * m->ny + y];
                for (int x = std::max(lo3[0], rw.xmin); x <= std::min(hi3[0], rw.xmax); x++) {
                    const double rx = m->origin[0] + h * (x + m->lo[0]) - c[0];
                    const double ry = m->origin[1] + h * (y + m->lo[1]) - c[1];
                    const double rz = m->origin[2] + h * (z + m->lo[2]) - c[2];
                    const double d2 = rx * rx + ry * ry + rz * rz;
                    if (d2 > rc * rc) continue;
                    q_pt.push_back(rw.start + (x - rw.xmin));
                    q_atom.push_back(a);
                    const double g = std::exp(-d2 / b2);
                    for (int i = 0; i < npmax; i++)
                        q_p.push_back(i < np ? solid_harmonic(i, rx, ry, rz) * g : 0.0);
                }
            }
        const size_t q_end = q_pt.size();
        for (int i = 0; i < np; i++) {
            double ss = 0.0;
            for (size_t q = q_begin; q < q_end; q++) ss += q_p[q * npmax + i] * q_p[q * npmax + i];
            const double nrm = std::sqrt(h3 * ss);
            if (nrm > 0)
                for (size_t q = q_begin; q < q_end; q++) q_p[q * npmax + i] /= nrm;
        }
        for (size_t q0 = q_begin; q0 < q_end; q0 += kProjChunk) {
            ch_atom.push_back(a);
            ch_q0.push_back((int32_t)q0);
            ch_q1.push_back((int32_t)std::min(q_end, q0 + kProjChunk));
        }
        atom_ch0.push_back((int32_t)ch_q0.size());
        for (int i = 0; i < np; i++)
            for (int j = 0; j < np; j++) {
                hm[((size_t)a * npmax + i) * npmax + j] = hmats[hoff + i * np + j];
                H->proj_norm += std::fabs(hmats[hoff + i * np + j]);
            }
        hoff += (int64_t)np * np;
    }
    return upload_projectors(H, natoms, npmax, q_pt, q_atom, q_p, ch_atom, ch_q0, ch_q1, atom_ch0, hm);
}

rsg_status rsg_projectors_set_raw(rsg_ham H, int natoms, const int64_t *npts, const int64_t *point_idx,
                                  const int32_t *nproj, const double *pvals, const double *hmats) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    if (natoms < 0) return fail(RSG_ERR_ARG, "natoms < 0");
    if (natoms > 0 && H->has_scaling) return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: no projectors");
    if (natoms == 0) {
        H->pj = ProjDev();
        H->proj_norm = 0.0;
        return RSG_OK;
    }
    if (!npts || !point_idx || !nproj || !pvals || !hmats) return fail(RSG_ERR_ARG, "NULL array");
    const int64_t P = H->m->P;
    int npmax = 1;
    int64_t nq = 0;
    for (int a = 0; a < natoms; a++) {
        if (nproj[a] < 1) return fail(RSG_ERR_ARG, "nproj[%d] < 1", a);
        if (nproj[a] > 9) return fail(RSG_ERR_UNSUPPORTED, "at most 9 projectors per atom");
        if (npts[a] < 0) return fail(RSG_ERR_ARG, "npts[%d] < 0", a);
        npmax = std::max(npmax, (int)nproj[a]);
        nq += npts[a];
    }
    if (nq >= (int64_t)INT32_MAX) return fail(RSG_ERR_UNSUPPORTED, "more than 2^31 projector entries");
    std::vector<int32_t> q_pt, q_atom, ch_atom, ch_q0, ch_q1, atom_ch0(1, 0);
    std::vector<double> q_p, hm((size_t)natoms * npmax * npmax, 0.0);
    q_pt.reserve((size_t)nq);
    q_atom.reserve((size_t)nq);
    q_p.reserve((size_t)nq * npmax);
    double proj_norm = 0.0;
    int64_t off = 0, voff = 0, hoff = 0;
    std::vector<int64_t> order;
    std::vector<char> seen((size_t)P, 0);
    for (int a = 0; a < natoms; a++) {
        const int np = nproj[a];
        const int64_t n = npts[a];
        // entries in ascending point order (coalesced gathers); a point may
        // appear once per atom
        order.resize((size_t)n);
        for (int64_t k = 0; k < n; k++) {
            const int64_t pt = point_idx[off + k];
            if (pt < 0 || pt >= P) return fail(RSG_ERR_ARG, "atom %d: point index %lld outside the mesh", a,
                                               (long long)pt);
            order[(size_t)k] = k;
        }
        std::sort(order.begin(), order.end(),
                  [&](int64_t x, int64_t y) { return point_idx[off + x] < point_idx[off + y]; });
        const size_t q_begin = q_pt.size();
        for (int64_t k : order) {
            const int64_t pt = point_idx[off + k];
            if (seen[(size_t)pt]) return fail(RSG_ERR_ARG, "atom %d: point %lld listed twice", a, (long long)pt);
            seen[(size_t)pt] = 1;
            q_pt.push_back((int32_t)pt);
            q_atom.push_back(a);
            for (int i = 0; i < npmax; i++) {
                const double v = i < np ? pvals[voff + k * np + i] : 0.0;
                if (!std::isfinite(v)) return fail(RSG_ERR_ARG, "atom %d: projector value not finite", a);
                q_p.push_back(v);
            }
        }
        for (size_t q = q_begin; q < q_pt.size(); q++) seen[(size_t)q_pt[q]] = 0;
        const size_t q_end = q_pt.size();
        for (size_t q0 = q_begin; q0 < q_end; q0 += kProjChunk) {
            ch_atom.push_back(a);
            ch_q0.push_back((int32_t)q0);
            ch_q1.push_back((int32_t)std::min(q_end, q0 + kProjChunk));
        }
        atom_ch0.push_back((int32_t)ch_q0.size());
        double hmax = 0.0;
        for (int i = 0; i < np * np; i++) {
            if (!std::isfinite(hmats[hoff + i])) return fail(RSG_ERR_ARG, "atom %d: h not finite", a);
            hmax = std::max(hmax, std::fabs(hmats[hoff + i]));
        }
        for (int i = 0; i < np; i++)
            for (int j = 0; j < np; j++) {
                const double hij = hmats[hoff + i * np + j];
                if (std::fabs(hij - hmats[hoff + j * np + i]) > 1e-12 * hmax)
                    return fail(RSG_ERR_ARG, "atom %d: h is not symmetric", a);
                hm[((size_t)a * npmax + i) * npmax + j] = hij;
                proj_norm += std::fabs(hij);
            }
        off += n;
        voff += n * np;
        hoff += (int64_t)np * np;
    }
    H->pj = ProjDev();
    H->proj_norm = 0.0;
    CKS(upload_projectors(H, natoms, npmax, q_pt, q_atom, q_p, ch_atom, ch_q0, ch_q1, atom_ch0, hm));
    H->proj_norm = proj_norm;
    return RSG_OK;
}

rsg_status rsg_hamiltonian_apply(rsg_ham H, const void *psi, void *hpsi, int64_t S, int64_t ld,
                                 void *stream) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    CKS(check_block(H, psi, S, ld, "psi"));
    CKS(check_block(H, hpsi, S, ld, "hpsi"));
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    const size_t bytes = (size_t)H->m->P * ld * cbytes(H->dtype);
    if (overlaps(psi, hpsi, bytes)) return fail(RSG_ERR_ARG, "psi and hpsi overlap");
    Epi ep;
    return apply(H, psi, hpsi, sv_of(H, ld), H->eps, H->dir, ep, (cudaStream_t)stream);
}

rsg_status rsg_taylor_apply(rsg_ham H, const void *psi, void *out, int64_t S, int64_t ld, double tau,
                            void *stream) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    CKS(check_block(H, psi, S, ld, "psi"));
    CKS(check_block(H, out, S, ld, "out"));
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    const size_t bytes = (size_t)H->m->P * ld * cbytes(H->dtype);
    if (out != psi && overlaps(psi, out, bytes)) return fail(RSG_ERR_ARG, "psi and out partially overlap");
    if (!std::isfinite(tau)) return fail(RSG_ERR_ARG, "tau not finite");
    return taylor(H, psi, out, ld, tau, H->eps, H->dir, (cudaStream_t)stream);
}

// ------------------------------------------------ checkpoint / resume ----
// A state block is stored as a NumPy .npy file (format 1.0: magic, version,
// little-endian header length, a Python-literal header dict padded to a
// multiple of 64 bytes) holding the live (P, S) columns in library point
// order, plus `path`.json with the step counter, time and the caller's seed.

static std::string npy_descr(rsg_dtype t) { return t == RSG_C64 ? "<c8" : "<c16"; }

rsg_status rsg_states_save(rsg_ham H, const char *path, const void *psi, int64_t S, int64_t ld,
                           int psi_on_device, int64_t step, double time, uint64_t seed) {
    if (!H || !path || !psi) return fail(RSG_ERR_ARG, "NULL argument");
    if (S < 1 || ld < S) return fail(RSG_ERR_ARG, "need 1 <= S <= ld");
    const size_t cb = cbytes(H->dtype);
    const int64_t P = H->m->P;
    std::vector<char> host;
    const char *src = (const char *)psi;
    if (psi_on_device) {
        // the block may still be written by work on any stream, including
        // non-blocking ones that the legacy stream does not wait for
        CK(cudaDeviceSynchronize());
        host.resize((size_t)P * ld * cb);
        CK(cudaMemcpy(host.data(), psi, host.size(), cudaMemcpyDeviceToHost));
        src = host.data();
    }
    char dict[256];
    std::snprintf(dict, sizeof dict, "{'descr': '%s', 'fortran_order': False, 'shape': (%lld, %lld), }",
                  npy_descr(H->dtype).c_str(), (long long)P, (long long)S);
    std::string hdr(dict);
    const size_t unpadded = 10 + hdr.size() + 1;
    hdr.append((64 - unpadded % 64) % 64, ' ');
    hdr.push_back('\n');
    // both files are written under temporary names and renamed into place,
    // so a failure part way leaves any earlier checkpoint intact
    const std::string tmp = std::string(path) + ".tmp" + std::to_string((long long)getpid());
    FILE *f = std::fopen(tmp.c_str(), "wb");
    if (!f) return fail(RSG_ERR_ARG, "cannot open %s for writing", tmp.c_str());
    const unsigned char pre[10] = {0x93, 'N', 'U', 'M', 'P', 'Y', 1, 0, (unsigned char)(hdr.size() & 0xff),
                                   (unsigned char)(hdr.size() >> 8)};
    bool ok = std::fwrite(pre, 1, 10, f) == 10 && std::fwrite(hdr.data(), 1, hdr.size(), f) == hdr.size();
    for (int64_t p = 0; ok && p < P; p++)
        ok = std::fwrite(src + (size_t)p * ld * cb, cb, (size_t)S, f) == (size_t)S;
    ok = (std::fclose(f) == 0) && ok;
    if (!ok) {
        std::remove(tmp.c_str());
        return fail(RSG_ERR_ARG, "writing %s failed", tmp.c_str());
    }
    const std::string meta = std::string(path) + ".json", mtmp = meta + ".tmp" + std::to_string((long long)getpid());
    FILE *m = std::fopen(mtmp.c_str(), "w");
    if (!m) {
        std::remove(tmp.c_str());
        return fail(RSG_ERR_ARG, "cannot open %s for writing", mtmp.c_str());
    }
    std::fprintf(m,
                 "{\"format\": \"rsg-states-1\", \"points\": %lld, \"states\": %lld, \"dtype\": \"%s\", "
                 "\"step\": %lld, \"time\": %.17g, \"seed\": %llu}\n",
                 (long long)P, (long long)S, H->dtype == RSG_C64 ? "complex64" : "complex128", (long long)step, time,
                 (unsigned long long)seed);
    if (std::fclose(m) != 0) {
        std::remove(tmp.c_str());
        std::remove(mtmp.c_str());
        return fail(RSG_ERR_ARG, "writing %s failed", mtmp.c_str());
    }
    if (std::rename(tmp.c_str(), path) != 0 || std::rename(mtmp.c_str(), meta.c_str()) != 0)
        return fail(RSG_ERR_ARG, "cannot move the checkpoint into place at %s", path);
    return RSG_OK;
}

rsg_status rsg_states_load(rsg_ham H, const char *path, void *psi, int64_t S, int64_t ld, int psi_on_device,
                           int64_t *step, double *time, uint64_t *seed) {
    if (!H || !path || !psi) return fail(RSG_ERR_ARG, "NULL argument");
    if (S < 1 || ld < S) return fail(RSG_ERR_ARG, "need 1 <= S <= ld");
    const size_t cb = cbytes(H->dtype);
    const int64_t P = H->m->P;
    FILE *f = std::fopen(path, "rb");
    if (!f) return fail(RSG_ERR_ARG, "cannot open %s", path);
    unsigned char pre[12];
    std::string hdr;
    bool ok = std::fread(pre, 1, 8, f) == 8 && std::memcmp(pre, "\x93NUMPY", 6) == 0 && (pre[6] == 1 || pre[6] == 2);
    size_t hlen = 0;
    if (ok && pre[6] == 1) {
        ok = std::fread(pre + 8, 1, 2, f) == 2;
        hlen = (size_t)pre[8] | ((size_t)pre[9] << 8);
    } else if (ok) {
        ok = std::fread(pre + 8, 1, 4, f) == 4;
        hlen = (size_t)pre[8] | ((size_t)pre[9] << 8) | ((size_t)pre[10] << 16) | ((size_t)pre[11] << 24);
    }
    if (ok && hlen < (1u << 16)) {
        hdr.resize(hlen);
        ok = std::fread(&hdr[0], 1, hlen, f) == hlen;
    } else {
        ok = false;
    }
    char want[128];
    std::snprintf(want, sizeof want, "(%lld, %lld)", (long long)P, (long long)S);
    if (ok && (hdr.find("'descr': '" + npy_descr(H->dtype) + "'") == std::string::npos ||
               hdr.find("'fortran_order': False") == std::string::npos ||
               hdr.find(std::string("'shape': ") + want) == std::string::npos)) {
        std::fclose(f);
        return fail(RSG_ERR_ARG, "%s does not hold a C-ordered %s block of shape %s", path,
                    npy_descr(H->dtype).c_str(), want);
    }
    std::vector<char> host((size_t)P * ld * cb, 0);
    for (int64_t p = 0; ok && p < P; p++)
        ok = std::fread(host.data() + (size_t)p * ld * cb, cb, (size_t)S, f) == (size_t)S;
    std::fclose(f);
    if (!ok) return fail(RSG_ERR_ARG, "%s is not a readable .npy state block", path);
    if (step || time || seed) {
        const std::string meta = std::string(path) + ".json";
        FILE *m = std::fopen(meta.c_str(), "r");
        if (!m) return fail(RSG_ERR_ARG, "metadata %s missing", meta.c_str());
        char buf[1024] = {0};
        const size_t n = std::fread(buf, 1, sizeof buf - 1, m);
        std::fclose(m);
        buf[n] = 0;
        long long st = 0, pts = -1, sts = -1;
        double t = 0.0;
        unsigned long long sd = 0;
        const char *q;
        bool mok = (q = std::strstr(buf, "\"points\":")) && std::sscanf(q + 9, "%lld", &pts) == 1 &&
                   (q = std::strstr(buf, "\"states\":")) && std::sscanf(q + 9, "%lld", &sts) == 1 &&
                   (q = std::strstr(buf, "\"step\":")) && std::sscanf(q + 7, "%lld", &st) == 1 &&
                   (q = std::strstr(buf, "\"time\":")) && std::sscanf(q + 7, "%lg", &t) == 1 &&
                   (q = std::strstr(buf, "\"seed\":")) && std::sscanf(q + 7, "%llu", &sd) == 1;
        if (!mok || pts != P || sts != S) return fail(RSG_ERR_ARG, "metadata %s does not match", meta.c_str());
        if (step) *step = st;
        if (time) *time = t;
        if (seed) *seed = sd;
    }
    if (psi_on_device) {
        // no stream may still use the block while it is overwritten, and the
        // restored values have landed before any later launch on any stream
        CK(cudaDeviceSynchronize());
        CK(cudaMemcpy(psi, host.data(), host.size(), cudaMemcpyHostToDevice));
        CK(cudaDeviceSynchronize());
    } else {
        std::memcpy(psi, host.data(), host.size());
    }
    return RSG_OK;
}

rsg_status rsg_state_norms(rsg_ham H, const void *psi, int64_t S, int64_t ld, double *norms2_out,
                           void *stream) {
    if (!H || !norms2_out) return fail(RSG_ERR_ARG, "NULL argument");
    CKS(check_block(H, psi, S, ld, "psi"));
    cudaStream_t st = (cudaStream_t)stream;
    CK(H->drift.ensure((size_t)S * sizeof(double)));
    CKS(norms_dev(H, psi, S, ld, H->drift.as<double>(), st));
    CK(cudaMemcpyAsync(norms2_out, H->drift.p, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    return read_status(H, st);
}

rsg_status rsg_selftest_bounded_wait(rsg_ham H, int polls, void *stream) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    if (polls < 1 || polls > 65536) return fail(RSG_ERR_ARG, "polls must be in 1..65536");
    cudaStream_t st = (cudaStream_t)stream;
    if (!H->status.p) {
        CK(H->status.ensure(sizeof(int)));
        CK(cudaMemsetAsync(H->status.p, 0, sizeof(int), st));
    }
    CK(launch_selftest_wait(polls, H->status.as<int>(), st));
    H->n_launch++;
    return read_status(H, st);
}

rsg_status rsg_set_log_level(int level) {
    if (level < 0 || level > 2) return fail(RSG_ERR_ARG, "log level must be 0, 1 or 2");
    g_log_level.store(level);
    return RSG_OK;
}

rsg_status rsg_debug_fail_allocations(int n) {
    if (n < 0) return fail(RSG_ERR_ARG, "n < 0");
    g_fail_allocs.store(n);
    return RSG_OK;
}

rsg_status rsg_orthonormalize(rsg_ham H, void *psi, int64_t S, int64_t ld, double *norms2_out,
                              void *stream) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    CKS(check_block(H, psi, S, ld, "psi"));
    if (S > 1024) return fail(RSG_ERR_UNSUPPORTED, "S > 1024");
    cudaStream_t st = (cudaStream_t)stream;
    if (norms2_out) {
        CK(H->drift.ensure((size_t)S * sizeof(double)));
        CKS(norms_dev(H, psi, S, ld, H->drift.as<double>(), st));
        CK(cudaMemcpyAsync(norms2_out, H->drift.p, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
    }
    CKS(orthonormalize_dev(H, psi, S, ld, nullptr, st));
    return read_status(H, st);
}

rsg_status rsg_propagate_steps(rsg_ham H, void *psi, int64_t S, int64_t ld, int64_t nsteps, double dt,
                               rsg_scheme scheme, int nsub, const double *eps, const double dir[3],
                               int gs_every, double *norm_drift_out, void *stream) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    CKS(check_block(H, psi, S, ld, "psi"));
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    if (nsteps < 0 || nsub < 1 || gs_every < 0 || !std::isfinite(dt))
        return fail(RSG_ERR_ARG, "bad nsteps/nsub/gs_every/dt");
    if (scheme != RSG_EXPMID && scheme != RSG_ETRS) return fail(RSG_ERR_ARG, "unknown scheme");
    if (S > 1024 && gs_every > 0) return fail(RSG_ERR_UNSUPPORTED, "S > 1024 with Gram-Schmidt");
    if (H->has_scaling && eps)
        for (int64_t k = 0; k < nsteps; k++)
            if (eps[k] != 0.0) return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: no dipole field");
    cudaStream_t st = (cudaStream_t)stream;
    const double xdir[3] = {1.0, 0.0, 0.0};
    const double *d = dir ? dir : xdir;
    // drift buffer: S maxima, then S scratch norms
    CK(H->drift.ensure((size_t)2 * S * sizeof(double)));
    double *drift = H->drift.as<double>();
    CK(cudaMemsetAsync(drift, 0, (size_t)S * sizeof(double), st));
    const double tsub = dt / nsub;
    for (int64_t k = 0; k < nsteps; k++) {
        const double e = eps ? eps[k] : 0.0;
        for (int u = 0; u < nsub; u++) {
            if (scheme == RSG_EXPMID) {
                CKS(taylor(H, psi, psi, ld, tsub, e, d, st));
            } else {
                // T_{H(t+dt')}(dt'/2) T_{H(t)}(dt'/2); both with the interval's eps_k
                CKS(taylor(H, psi, psi, ld, 0.5 * tsub, e, d, st));
                CKS(taylor(H, psi, psi, ld, 0.5 * tsub, e, d, st));
            }
        }
        if (H->has_mask) {
            // mask absorber: keep the bounded part M psi of every state
            if (H->dtype == RSG_C64) CK(launch_mask<float>(psi, H->m->P, (int)ld, (int)S, H->mask.p, st));
            else CK(launch_mask<double>(psi, H->m->P, (int)ld, (int)S, H->mask.p, st));
            H->n_launch++;
        }
        const bool gs_now = gs_every > 0 && (k + 1) % gs_every == 0;
        if (gs_now) {
            CKS(orthonormalize_dev(H, psi, S, ld, drift, st));
        } else if (k == nsteps - 1 && norm_drift_out) {
            // final check without re-orthonormalising: norms into scratch, then max
            CKS(norms_dev(H, psi, S, ld, drift + S, st));
            std::vector<double> a((size_t)S), b((size_t)S);
            CK(cudaMemcpyAsync(a.data(), drift, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
            CK(cudaMemcpyAsync(b.data(), drift + S, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            for (int64_t s = 0; s < S; s++) {
                const double e2 = std::fabs(b[(size_t)s] - 1.0);
                norm_drift_out[s] = (e2 > a[(size_t)s] || std::isnan(e2)) ? e2 : a[(size_t)s];
            }
            return read_status(H, st);
        }
    }
    if (norm_drift_out) {
        CK(cudaMemcpyAsync(norm_drift_out, drift, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    if (gs_every > 0 || norm_drift_out) return read_status(H, st);
    return RSG_OK;
}

// ------------------------------------------------------- eigensolver ----
// Lowest eigenpairs of H by Chebyshev-filtered subspace iteration.  Each
// filter step is one application of H - c through the stencil epilogue (the
// shift folded into the diagonal, the previous iterate added as the base);
// each iteration ends with the FP64 Cholesky-QR, a Rayleigh-Ritz step on the
// S x S FP64 matrix X^H H X (cyclic complex Jacobi on the host) and FP64
// residual norms.

}  // extern "C"

namespace {

// Cyclic Jacobi for a Hermitian n x n matrix A (row-major complex double,
// overwritten): eigenvalues ascending in w, eigenvectors in the columns of
// V (row-major, V[t][s] = component t of vector s).
void jacobi_hermitian(int n, std::vector<std::complex<double>> &A, std::vector<double> &w,
                      std::vector<std::complex<double>> &V) {
    using cd = std::complex<double>;
    V.assign((size_t)n * n, cd(0, 0));
    for (int i = 0; i < n; i++) V[(size_t)i * n + i] = 1.0;
    double scale = 0.0;
    for (const cd &x : A) scale += std::norm(x);
    scale = std::sqrt(scale);
    for (int sweep = 0; sweep < 100; sweep++) {
        double off = 0.0;
        for (int p = 0; p < n; p++)
            for (int q = 0; q < n; q++)
                if (p != q) off += std::norm(A[(size_t)p * n + q]);
        if (std::sqrt(off) <= 1e-15 * scale || off == 0.0) break;
        for (int p = 0; p < n - 1; p++)
            for (int q = p + 1; q < n; q++) {
                const cd b = A[(size_t)p * n + q];
                const double ab = std::abs(b);
                if (ab <= 1e-300) continue;
                // U = diag(1, e^{-i phi}) R(theta): zeroes A_pq, phi = arg A_pq
                const cd ph = b / ab;
                const double th = 0.5 * std::atan2(2.0 * ab, A[(size_t)p * n + p].real() - A[(size_t)q * n + q].real());
                const double c = std::cos(th), s = std::sin(th);
                const cd u00 = c, u01 = -s, u10 = s * std::conj(ph), u11 = c * std::conj(ph);
                for (int k = 0; k < n; k++) {     // A <- A U
                    const cd ap = A[(size_t)k * n + p], aq = A[(size_t)k * n + q];
                    A[(size_t)k * n + p] = ap * u00 + aq * u10;
                    A[(size_t)k * n + q] = ap * u01 + aq * u11;
                }
                for (int k = 0; k < n; k++) {     // A <- U^H A
                    const cd ap = A[(size_t)p * n + k], aq = A[(size_t)q * n + k];
                    A[(size_t)p * n + k] = std::conj(u00) * ap + std::conj(u10) * aq;
                    A[(size_t)q * n + k] = std::conj(u01) * ap + std::conj(u11) * aq;
                }
                A[(size_t)p * n + q] = A[(size_t)q * n + p] = 0.0;
                for (int k = 0; k < n; k++) {     // V <- V U
                    const cd vp = V[(size_t)k * n + p], vq = V[(size_t)k * n + q];
                    V[(size_t)k * n + p] = vp * u00 + vq * u10;
                    V[(size_t)k * n + q] = vp * u01 + vq * u11;
                }
            }
    }
    std::vector<int> order(n);
    for (int i = 0; i < n; i++) order[i] = i;
    std::stable_sort(order.begin(), order.end(),
                     [&](int x, int y) { return A[(size_t)x * n + x].real() < A[(size_t)y * n + y].real(); });
    std::vector<cd> Vs((size_t)n * n);
    w.resize(n);
    for (int j = 0; j < n; j++) {
        w[j] = A[(size_t)order[j] * n + order[j]].real();
        for (int t = 0; t < n; t++) Vs[(size_t)t * n + j] = V[(size_t)t * n + order[j]];
    }
    V.swap(Vs);
}

}  // namespace

extern "C" {

rsg_status rsg_eigensolve(rsg_ham H, void *psi, int64_t S, int64_t ld, int64_t nwant, int64_t max_iter,
                          int degree, double tol, double *evals_out, double *resid_out, int64_t *iters_out,
                          void *stream) {
    if (!H || !evals_out) return fail(RSG_ERR_ARG, "NULL argument");
    CKS(check_block(H, psi, S, ld, "psi"));
    if (nwant < 1 || nwant > S) return fail(RSG_ERR_ARG, "need 1 <= nwant <= S");
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    if (S > 256) return fail(RSG_ERR_UNSUPPORTED, "S > 256");
    if (H->has_scaling)
        return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: the eigensolver needs a Hermitian operator");
    if (degree < 1 || degree > 64) return fail(RSG_ERR_ARG, "degree must be in 1..64");
    if (max_iter < 0 || !(tol > 0)) return fail(RSG_ERR_ARG, "need max_iter >= 0 and tol > 0");
    cudaStream_t st = (cudaStream_t)stream;
    rsg_mesh m = H->m;
    const int64_t P = m->P;
    const double h = m->h, h3 = h * h * h;
    const int SV = sv_of(H, ld);
    const size_t bytes = (size_t)P * ld * cbytes(H->dtype);
    CK(H->w0.ensure(bytes));
    CK(H->w1.ensure(bytes));
    const int nbg = gram_blocks(P, (int)S), nbn = norm_blocks(P);
    CK(H->red.ensure(std::max((size_t)nbg * S * S * 2, (size_t)nbn * S) * sizeof(double)));
    CK(H->G.ensure((size_t)S * S * 2 * sizeof(double)));
    CK(H->W.ensure((size_t)S * S * 2 * sizeof(double)));
    CK(H->drift.ensure((size_t)2 * S * sizeof(double)));
    double *lam_dev = H->drift.as<double>(), *res_dev = H->drift.as<double>() + S;
    // upper bound of the spectrum: Gershgorin for the 8th-order Laplacian
    // (the row sum of |c_k| is the largest value of its symbol), the largest
    // potential, the projector bound and the field over the mesh box
    double csum = 0.0;
    for (int k = 0; k < 5; k++) csum += (k ? 2.0 : 1.0) * std::fabs(kFD[k]);
    double field = 0.0;
    for (int corner = 0; corner < 8; corner++) {
        double v = 0.0;
        for (int d = 0; d < 3; d++) {
            const int ext = d == 0 ? m->nx : d == 1 ? m->ny : m->nz;
            const int idx = (corner >> d) & 1 ? ext - 1 : 0;
            v += H->dir[d] * (m->origin[d] + h * (idx + m->lo[d]));
        }
        field = std::max(field, std::fabs(H->eps * v));
    }
    const double upper = 3.0 * csum / (2.0 * h * h) + H->vmax + H->proj_norm + field;

    std::vector<std::complex<double>> A((size_t)S * S), Q;
    std::vector<double> lam, res((size_t)S);
    // Ritz vectors of close levels amplify a change of rounding: complex64
    // results stay those of one kernel
    Epi plain;
    plain.fixed_kernel = true;
    auto rayleigh_ritz = [&]() -> rsg_status {
        Epi ep = plain;
        CKS(apply(H, psi, H->w0.p, SV, H->eps, H->dir, ep, st));
        if (H->dtype == RSG_C64)
            CK(launch_cross_gram<float>(psi, H->w0.p, P, (int)ld, (int)S, h3, H->red.as<double>(), nbg,
                                        H->G.as<double>(), st));
        else
            CK(launch_cross_gram<double>(psi, H->w0.p, P, (int)ld, (int)S, h3, H->red.as<double>(), nbg,
                                         H->G.as<double>(), st));
        CK(cudaMemcpyAsync(A.data(), H->G.p, (size_t)S * S * 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        for (int64_t i = 0; i < S; i++)
            for (int64_t j = 0; j < S; j++)
                if (!std::isfinite(A[(size_t)i * S + j].real()) || !std::isfinite(A[(size_t)i * S + j].imag()))
                    return fail(RSG_ERR_NONFINITE, "Rayleigh-Ritz matrix not finite");
        for (int64_t i = 0; i < S; i++)      // exact Hermitian part
            for (int64_t j = i; j < S; j++) {
                const std::complex<double> x = 0.5 * (A[(size_t)i * S + j] + std::conj(A[(size_t)j * S + i]));
                A[(size_t)i * S + j] = x;
                A[(size_t)j * S + i] = std::conj(x);
            }
        jacobi_hermitian((int)S, A, lam, Q);
        CK(cudaMemcpyAsync(H->W.p, Q.data(), (size_t)S * S * 2 * sizeof(double), cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(lam_dev, lam.data(), (size_t)S * sizeof(double), cudaMemcpyHostToDevice, st));
        if (H->dtype == RSG_C64) {
            CK(launch_rotate<float>(psi, P, (int)ld, (int)S, H->W.as<double>(), st));
            CK(launch_rotate<float>(H->w0.p, P, (int)ld, (int)S, H->W.as<double>(), st));
            CK(launch_resid<float>(psi, H->w0.p, P, (int)ld, (int)S, lam_dev, h3, H->red.as<double>(), nbn, res_dev,
                                   st));
        } else {
            CK(launch_rotate<double>(psi, P, (int)ld, (int)S, H->W.as<double>(), st));
            CK(launch_rotate<double>(H->w0.p, P, (int)ld, (int)S, H->W.as<double>(), st));
            CK(launch_resid<double>(psi, H->w0.p, P, (int)ld, (int)S, lam_dev, h3, H->red.as<double>(), nbn,
                                    res_dev, st));
        }
        CK(cudaMemcpyAsync(res.data(), res_dev, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        for (double &r : res) r = std::sqrt(std::max(r, 0.0));
        H->n_launch += 7;
        return RSG_OK;
    };
    auto converged = [&]() {
        for (int64_t s = 0; s < nwant; s++)
            if (!(res[(size_t)s] <= tol)) return false;
        return true;
    };

    CKS(orthonormalize_dev(H, psi, S, ld, nullptr, st));
    CKS(read_status(H, st));
    CKS(rayleigh_ritz());
    int64_t it = 0;
    while (it < max_iter && !converged()) {
        // damp [a, upper] and amplify below a = the largest Ritz value (the
        // top of the buffer states above the nwant wanted ones)
        const double a = lam[(size_t)S - 1], lo = lam[0];
        if (!(a < upper)) return fail(RSG_ERR_NONFINITE, "Ritz values above the spectral bound");
        const double e = 0.5 * (upper - a), c = 0.5 * (upper + a);
        double sigma = e / (lo - c);
        const double sigma1 = sigma, gamma = 2.0 / sigma1;
        void *X = psi, *Y = H->w0.p, *Z = H->w1.p;
        {
            Epi ep = plain;              // Y = (sigma1 / e) (H - c) X
            ep.ar = sigma1 / e;
            ep.shift = c;
            CKS(apply(H, X, Y, SV, H->eps, H->dir, ep, st));
        }
        for (int k = 2; k <= degree; k++) {
            const double sigma2 = 1.0 / (gamma - sigma);
            Epi ep = plain;              // Z = (2 sigma2 / e) (H - c) Y - sigma sigma2 X
            ep.ar = 2.0 * sigma2 / e;
            ep.shift = c;
            ep.base = X;
            ep.br = -sigma * sigma2;
            CKS(apply(H, Y, Z, SV, H->eps, H->dir, ep, st));
            void *t = X;
            X = Y;
            Y = Z;
            Z = t;
            sigma = sigma2;
        }
        if (Y != psi) CK(cudaMemcpyAsync(psi, Y, bytes, cudaMemcpyDeviceToDevice, st));
        CKS(orthonormalize_dev(H, psi, S, ld, nullptr, st));
        CKS(read_status(H, st));
        CKS(rayleigh_ritz());
        it++;
    }
    std::memcpy(evals_out, lam.data(), (size_t)S * sizeof(double));
    if (resid_out) std::memcpy(resid_out, res.data(), (size_t)S * sizeof(double));
    if (iters_out) *iters_out = it;
    return read_status(H, st);
}

// -------------------------------------------------- shifted solves ----
// (H - z) x = b for S right-hand sides at one complex shift z: the linear
// problem of the Sternheimer equation (Sec. "The Sternheimer formulation of
// linear-response"), solved by
// conjugate-orthogonal conjugate gradients for the complex symmetric matrix
// H - z (H is real symmetric here).  A x is one application with the base
// term -z x folded into the epilogue; every inner product is FP64.
rsg_status rsg_shifted_solve(rsg_ham H, const void *b, void *x, int64_t S, int64_t ld, double zr, double zi,
                             int64_t max_iter, double tol, double *resid_out, int64_t *iters_out, void *stream) {
    if (!H) return fail(RSG_ERR_ARG, "NULL handle");
    CKS(check_block(H, b, S, ld, "b"));
    CKS(check_block(H, x, S, ld, "x"));
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    if (max_iter < 0 || !(tol > 0) || !std::isfinite(zr) || !std::isfinite(zi))
        return fail(RSG_ERR_ARG, "need max_iter >= 0, tol > 0 and a finite shift");
    rsg_mesh m = H->m;
    const int64_t P = m->P;
    const size_t bytes = (size_t)P * ld * cbytes(H->dtype);
    if (overlaps(b, x, bytes)) return fail(RSG_ERR_ARG, "b and x overlap");
    cudaStream_t st = (cudaStream_t)stream;
    const double h3 = std::pow(m->h, 3);
    const int SV = sv_of(H, ld);
    CK(H->w0.ensure(bytes));
    CK(H->w1.ensure(bytes));
    CK(H->w2.ensure(bytes));
    const int nbn = norm_blocks(P);
    CK(H->red.ensure((size_t)nbn * S * 2 * sizeof(double)));
    CK(H->cg.ensure((size_t)S * 10 * sizeof(double)));
    double *cgb = H->cg.as<double>();
    double *d_dot = cgb, *d_a = cgb + 2 * S, *d_b = cgb + 4 * S, *d_nrm = cgb + 6 * S;   // complex ones 16-byte aligned
    void *r = H->w0.p, *p = H->w1.p, *q = H->w2.p;
    const bool c64 = H->dtype == RSG_C64;
    std::vector<double> coef((size_t)4 * S);
    auto Ax = [&](const void *in, void *out) -> rsg_status {     // out = (H - z) in
        Epi ep;
        ep.base = in;
        ep.br = -zr;
        ep.bi = -zi;
        // in complex64 the iterates amplify a change of rounding by orders of
        // magnitude: results stay those of one kernel
        ep.fixed_kernel = true;
        return apply(H, in, out, SV, H->eps, H->dir, ep, st);
    };
    auto comb = [&](const void *u, const void *v, void *w, const double *bb) -> rsg_status {   // w = u + bb v
        if (c64) CK(launch_comb<float>(u, v, w, P, (int)ld, (int)S, bb, st));
        else CK(launch_comb<double>(u, v, w, P, (int)ld, (int)S, bb, st));
        return RSG_OK;
    };
    std::vector<double> dot((size_t)2 * S), nrm((size_t)S), bn((size_t)S);
    auto bilinear = [&](const void *u, const void *v) -> rsg_status {    // dot = u^T v (host)
        if (c64) CK(launch_bilinear<float>(u, v, P, (int)ld, (int)S, h3, H->red.as<double>(), nbn, d_dot, st));
        else CK(launch_bilinear<double>(u, v, P, (int)ld, (int)S, h3, H->red.as<double>(), nbn, d_dot, st));
        CK(cudaMemcpyAsync(dot.data(), d_dot, (size_t)2 * S * sizeof(double), cudaMemcpyDeviceToHost, st));
        return RSG_OK;
    };
    auto norms = [&](const void *u, std::vector<double> &out) -> rsg_status {
        CKS(norms_dev(H, u, S, ld, d_nrm, st));
        CK(cudaMemcpyAsync(out.data(), d_nrm, (size_t)S * sizeof(double), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        return RSG_OK;
    };
    // dst = v and, with neg, -v behind it (d_a, d_b). The copy is not waited for:
    // coef is written again only after a stream sync, mostly that of a reduction's
    // download, which every pair of uploads has between them.
    auto upload = [&](const std::vector<std::complex<double>> &v, double *dst, bool neg) -> rsg_status {
        for (int64_t s = 0; s < S; s++) {
            coef[(size_t)2 * s] = v[(size_t)s].real();
            coef[(size_t)2 * s + 1] = v[(size_t)s].imag();
            coef[(size_t)(2 * (S + s))] = -v[(size_t)s].real();
            coef[(size_t)(2 * (S + s)) + 1] = -v[(size_t)s].imag();
        }
        CK(cudaMemcpyAsync(dst, coef.data(), (size_t)(neg ? 4 : 2) * S * sizeof(double), cudaMemcpyHostToDevice, st));
        return RSG_OK;
    };
    using cd = std::complex<double>;
    std::vector<cd> rho((size_t)S), mu((size_t)S), alpha((size_t)S), beta((size_t)S), minus((size_t)S, -1.0);
    // r = b - A x, p = r
    CKS(Ax(x, q));
    CKS(upload(minus, d_a, false));
    CKS(comb(b, q, r, d_a));
    CK(cudaMemcpyAsync(p, r, bytes, cudaMemcpyDeviceToDevice, st));
    CKS(norms(b, bn));
    CKS(bilinear(r, r));
    CKS(norms(r, nrm));
    for (int64_t s = 0; s < S; s++) rho[(size_t)s] = cd(dot[(size_t)2 * s], dot[(size_t)2 * s + 1]);
    std::vector<char> done((size_t)S, 0);
    auto check = [&]() {
        bool all = true;
        for (int64_t s = 0; s < S; s++) {
            done[(size_t)s] = std::sqrt(nrm[(size_t)s]) <= tol * std::sqrt(bn[(size_t)s]);
            all = all && done[(size_t)s];
        }
        return all;
    };
    int64_t it = 0;
    while (it < max_iter && !check()) {
        CKS(Ax(p, q));
        CKS(bilinear(p, q));
        CK(cudaStreamSynchronize(st));
        for (int64_t s = 0; s < S; s++) {
            mu[(size_t)s] = cd(dot[(size_t)2 * s], dot[(size_t)2 * s + 1]);
            if (done[(size_t)s]) {
                alpha[(size_t)s] = 0.0;
            } else {
                if (std::abs(mu[(size_t)s]) == 0.0 || !std::isfinite(std::abs(mu[(size_t)s])))
                    return fail(RSG_ERR_NONFINITE, "breakdown: p^T (H - z) p = 0 for state %lld", (long long)s);
                alpha[(size_t)s] = rho[(size_t)s] / mu[(size_t)s];
            }
        }
        CKS(upload(alpha, d_a, true));
        CKS(comb(x, p, x, d_a));          // x += alpha p
        CKS(comb(r, q, r, d_b));          // r -= alpha q
        CKS(bilinear(r, r));
        CKS(norms(r, nrm));
        for (int64_t s = 0; s < S; s++) {
            const cd rn(dot[(size_t)2 * s], dot[(size_t)2 * s + 1]);
            beta[(size_t)s] = done[(size_t)s] || std::abs(rho[(size_t)s]) == 0.0 ? cd(0.0) : rn / rho[(size_t)s];
            rho[(size_t)s] = rn;
        }
        CKS(upload(beta, d_b, false));
        CKS(comb(r, p, p, d_b));          // p = r + beta p
        it++;
    }
    // true residual |b - (H - z) x| / |b|
    CKS(Ax(x, q));
    CK(cudaStreamSynchronize(st));        // the last beta may still be in coef
    CKS(upload(minus, d_a, false));
    CKS(comb(b, q, r, d_a));
    CKS(norms(r, nrm));
    if (resid_out)
        for (int64_t s = 0; s < S; s++)
            resid_out[s] = bn[(size_t)s] > 0 ? std::sqrt(nrm[(size_t)s] / bn[(size_t)s]) : std::sqrt(nrm[(size_t)s]);
    if (iters_out) *iters_out = it;
    return read_status(H, st);
}

}  // extern "C"

// ============================================================ adjoint ====
namespace {

// One exponential by explicit powers: pw[0] = x (already there), pw[j+1] =
// A pw[j] with A = -i tau H (sgn = -1) or A^dagger = +i tau H (sgn = +1);
// next = sum_j pw[j] / j! (j = 0..4).  pw[4] is scratch.
rsg_status powers(rsg_ham H, void *const pw[5], void *next, int64_t ld, double tau, double sgn,
                  double eps, const double *dir, cudaStream_t st) {
    static const double invf[5] = {1.0, 1.0, 0.5, 1.0 / 6.0, 1.0 / 24.0};
    for (int j = 0; j < 4; j++) {
        Epi ep;
        ep.ar = 0.0;
        ep.ai = sgn * tau;
        ep.acc = next;
        if (j == 0) ep.acc_base = pw[0];   // next = pw[0] + A pw[0] + ...
        // acc += gamma * y with y = A^{j+1} x: gamma = 1/(j+1)! relative to the power
        ep.gr = invf[j + 1];
        ep.gi = 0.0;
        CKS(apply(H, pw[j], pw[j + 1], sv_of(H, ld), eps, dir, ep, st));
    }
    return RSG_OK;
}

template <typename R>
rsg_status control_gradient_t(rsg_ham H, const void *psi0, const void *target, int64_t nsteps,
                              double dt, rsg_scheme scheme, int nsub, const double *eps,
                              const double *dir, int K, double *J_out, double *grad_out,
                              cudaStream_t st) {
    rsg_mesh msh = H->m;
    const int64_t P = msh->P;
    const int64_t ld = H->dtype == RSG_C64 ? 2 : 1;   // one state, padded to 16 bytes
    const size_t cb = cbytes(H->dtype), vb = (size_t)P * ld * cb;
    const double h3 = std::pow(msh->h, 3);
    // every interval is m exponentials T(tau) of the same H_k = H0 + eps_k X
    const int m = scheme == RSG_EXPMID ? nsub : 2 * nsub;
    const double tau = scheme == RSG_EXPMID ? dt / nsub : 0.5 * dt / nsub;
    if (K <= 0 || K > nsteps) K = (int)nsteps;
    const int64_t nck = (nsteps + K - 1) / K;
    // Taylor powers A^j psi' (j = 0..3) of every exponential of one segment
    // are kept when they fit, so the backward sweep applies H only to the
    // costate (3 forward propagations in total); otherwise each interval's
    // powers are recomputed from the segment's stored states.
    size_t free_b = 0, total_b = 0;
    CK(cudaMemGetInfo(&free_b, &total_b));
    const int64_t have = (int64_t)H->pool.size();
    const int64_t seg_vecs = (int64_t)K * m * 4 + 1;
    const bool keep_powers = H->adj_keep >= 0 ? H->adj_keep == 1
                                              : (double)std::max<int64_t>(seg_vecs - have, 0) * vb < 0.6 * (double)free_b;
    int64_t at = 0;
    const int64_t ck0 = at; at += nck;
    const int64_t pw0 = at; at += keep_powers ? (int64_t)K * m * 4 + 1 : (int64_t)(K + 1) + 4 * m + 1;
    const int64_t b0 = at; at += 5;
    const int64_t sc0 = at; at += 4;
    const int64_t nvec = at;
    if ((int64_t)H->pool.size() < nvec) H->pool.resize((size_t)nvec);
    for (int64_t i = 0; i < nvec; i++) CK(H->pool[(size_t)i].ensure(vb));
    auto vec = [&](int64_t i) { return H->pool[(size_t)i].p; };
    void *chi = vec(sc0), *chi2 = vec(sc0 + 1), *phi = vec(sc0 + 2), *fa = vec(sc0 + 3);
    // column 0 of padded (P, ld) blocks
    CK(cudaMemsetAsync(vec(ck0), 0, vb, st));
    CK(cudaMemsetAsync(phi, 0, vb, st));
    CK(cudaMemcpy2DAsync(vec(ck0), ld * cb, psi0, cb, cb, (size_t)P, cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpy2DAsync(phi, ld * cb, target, cb, cb, (size_t)P, cudaMemcpyDeviceToDevice, st));
    // dipole coordinate X = dir . r in the compute type
    if (!(H->xdir_cached[0] == dir[0] && H->xdir_cached[1] == dir[1] && H->xdir_cached[2] == dir[2])) {
        std::vector<R> X((size_t)P);
        for (int64_t p = 0; p < P; p++) {
            double s = 0.0;
            for (int d = 0; d < 3; d++) s += dir[d] * (msh->origin[d] + msh->h * msh->ijk[(size_t)p * 3 + d]);
            X[(size_t)p] = (R)s;
        }
        CK(H->Xd.upload(X));
        for (int d = 0; d < 3; d++) H->xdir_cached[d] = dir[d];
    }
    const int nb = norm_blocks(P);
    const int nba = adjoint_blocks(P);
    CK(H->dots.ensure((size_t)std::max(2 * nb, nba) * sizeof(double)));
    CK(H->ov.ensure(2 * sizeof(double)));
    CK(H->grad.ensure((size_t)nsteps * sizeof(double) + 64));
    CK(cudaMemsetAsync(H->grad.p, 0, (size_t)nsteps * sizeof(double) + 64, st));
    unsigned *counter = (unsigned *)((char *)H->grad.p + (size_t)nsteps * sizeof(double));

    // forward pass by Horner stages (the same arithmetic as
    // rsg_propagate_steps), saving the state at the start of every segment
    CK(cudaMemcpyAsync(fa, vec(ck0), vb, cudaMemcpyDeviceToDevice, st));
    for (int64_t k = 0; k < nsteps; k++) {
        if (k > 0 && k % K == 0) CK(cudaMemcpyAsync(vec(ck0 + k / K), fa, vb, cudaMemcpyDeviceToDevice, st));
        for (int l = 0; l < m; l++) CKS(taylor(H, fa, fa, ld, tau, eps[k], dir, st));
    }
    // J = |<phi|psi_N>|^2 and chi_N = phi <phi|psi_N>
    CK(launch_overlap<R>(phi, fa, P, (int)ld, h3, H->dots.as<double>(), nb, H->ov.as<double>(), st));
    CK(launch_scale_dev<R>(phi, chi, P * ld, H->ov.as<double>(), st));
    double ov[2] = {0, 0};
    CK(cudaMemcpyAsync(ov, H->ov.p, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));

    // powers of exponential (k, l) of the current segment: slots j = 0..3
    auto pslot = [&](int64_t kk, int l, int j) -> void * {
        if (keep_powers) return vec(pw0 + (kk * m + l) * 4 + j);
        return j == 0 ? nullptr : vec(pw0 + (K + 1) + 4 * l + j);
    };
    const int64_t scratch = keep_powers ? pw0 + (int64_t)K * m * 4 : pw0 + (K + 1) + 4 * m;
    // x -> y through the m exponentials of interval kk (explicit powers),
    // leaving the powers of exponential l in pslot(kk, l, .)
    auto interval = [&](int64_t kk, const void *x, void *y, double e) -> rsg_status {
        const void *cur = x;
        for (int l = 0; l < m; l++) {
            void *p0 = keep_powers ? pslot(kk, l, 0) : const_cast<void *>(cur);
            if (keep_powers && p0 != cur) CK(cudaMemcpyAsync(p0, cur, vb, cudaMemcpyDeviceToDevice, st));
            void *pw[5] = {p0, pslot(kk, l, 1), pslot(kk, l, 2), pslot(kk, l, 3), vec(scratch)};
            void *next = (l == m - 1) ? y : (keep_powers ? pslot(kk, l + 1, 0) : pslot(kk, l + 1, 0));
            if (!keep_powers && l < m - 1) next = vec(pw0 + (K + 1) + 4 * (l + 1));   // holds the next input
            CKS(powers(H, pw, next, ld, tau, -1.0, e, dir, st));
            cur = next;
        }
        return RSG_OK;
    };

    // Shared sweeps: with every power of a segment kept, the costate sweep of
    // segment c (backward) and the recompute sweep of segment c - 1 (forward)
    // have the same number of exponentials and are independent, so each of
    // their Hamiltonian applications runs as one two-column launch: column 0
    // the recompute (A = -i tau H(eps_r)), column 1 the costate
    // (A^dagger = +i tau H(eps_c)).  Two banks of two-column blocks hold the
    // powers of consecutive segments.  The last segment's recompute and the
    // first segment's costate have no partner: their bank's blocks are one
    // state wide (ld = 1; complex64 rows are two values wide anyway), where a
    // complex128 application costs half of a two-column one.
    const size_t vb2 = (size_t)P * 2 * cb;
    const int64_t nper = (int64_t)K * m * 4 + 1;     // per bank: 4 powers of every step, and the segment's end
    const bool merged = keep_powers && (H->adj_merge == 1 ||
                                        (H->adj_merge < 0 && (double)(2 * nper + 1) * vb2 < 0.5 * (double)free_b));
    if (merged) {
        if ((int64_t)H->pool2.size() < 2 * nper + 1) H->pool2.resize((size_t)(2 * nper + 1));
        for (int64_t i = 0; i < 2 * nper + 1; i++) CK(H->pool2[(size_t)i].ensure(vb2));
        auto arr = [&](int b, int64_t t, int j) { return H->pool2[(size_t)(b * nper + t * 4 + j)].p; };
        void *scr = H->pool2[(size_t)(2 * nper)].p;
        int64_t width[2] = {2, 2};   // columns of each bank's blocks; the costate is the last
        // column col of a bank's block <-> a single-state vector
        auto to_col = [&](int b, void *blk, int64_t col, const void *v) {
            return cudaMemcpy2DAsync((char *)blk + col * cb, width[b] * cb, v, ld * cb, cb, (size_t)P,
                                     cudaMemcpyDeviceToDevice, st);
        };
        auto from_col = [&](void *v, int b, const void *blk, int64_t col) {
            return cudaMemcpy2DAsync(v, ld * cb, (const char *)blk + col * cb, width[b] * cb, cb, (size_t)P,
                                     cudaMemcpyDeviceToDevice, st);
        };
        static const double invf[5] = {1.0, 1.0, 0.5, 1.0 / 6.0, 1.0 / 24.0};
        // step t of bank b: the exponential from arr(b, t, 0) to arr(b, t + 1, 0)
        auto step = [&](int b, int64_t t, bool rec, double eps_r, bool cost, double eps_c) -> rsg_status {
            void *pw[5] = {arr(b, t, 0), arr(b, t, 1), arr(b, t, 2), arr(b, t, 3), scr};
            for (int j = 0; j < 4; j++) {
                Epi ep;
                ep.ar = 0.0;
                ep.acc = arr(b, t + 1, 0);
                if (j == 0) ep.acc_base = pw[0];
                ep.gr = invf[j + 1];
                ep.gi = 0.0;
                double e = eps_r;
                if (rec && cost) {
                    ep.twocol = true;
                    ep.ai = -tau;
                    ep.ar1 = 0.0;
                    ep.ai1 = tau;
                    ep.eps1 = eps_c;
                } else if (rec) {
                    ep.ai = -tau;
                } else {
                    ep.ai = tau;
                    e = eps_c;
                }
                CKS(apply(H, pw[j], pw[j + 1], sv_of(H, width[b]), e, dir, ep, st));
            }
            return RSG_OK;
        };
        // the last segment's powers first (bank of its index parity)
        {
            const int64_t c = nck - 1, k0 = c * K, L = std::min<int64_t>(k0 + K, nsteps) - k0;
            const int b = (int)(c % 2);
            width[b] = ld;
            CK(to_col(b, arr(b, 0, 0), 0, vec(ck0 + c)));
            for (int64_t t = 0; t < L * m; t++) CKS(step(b, t, true, eps[k0 + t / m], false, 0.0));
        }
        for (int64_t c = nck - 1; c >= 0; c--) {
            const int64_t k0c = c * K, k1c = std::min<int64_t>(k0c + K, nsteps), Tc = (k1c - k0c) * m;
            const int bc = (int)(c % 2), br = 1 - bc;
            const int64_t k0r = (c - 1) * K, Tr = c >= 1 ? (int64_t)K * m : 0;
            width[br] = c >= 1 ? 2 : ld;
            CK(to_col(br, arr(br, 0, 0), width[br] - 1, chi));
            if (c >= 1) CK(to_col(br, arr(br, 0, 0), 0, vec(ck0 + c - 1)));
            const int64_t T = std::max(Tc, Tr);
            for (int64_t t = 0; t < T; t++) {
                const bool rec = t < Tr, cost = t < Tc;
                const int64_t k = k1c - 1 - t / m;
                const int l = m - 1 - (int)(t % m);
                CKS(step(br, t, rec, rec ? eps[k0r + t / m] : 0.0, cost, cost ? eps[k] : 0.0));
                if (cost) {
                    const int64_t tc = (k - k0c) * m + l;   // the costate's exponential in its segment's bank
                    const void *bb[4], *aa[4];
                    for (int j = 0; j < 4; j++) {
                        bb[j] = (const char *)arr(br, t, j) + (width[br] - 1) * cb;
                        aa[j] = arr(bc, tc, j);
                    }
                    CK(launch_adjoint_grad<R>(bb, aa, P, (int)width[br], (int)width[bc], H->Xd.as<R>(), h3, tau,
                                              H->dots.as<double>(), nba,
                                              counter, H->grad.as<double>() + k, st));
                }
            }
            CK(from_col(chi, br, arr(br, Tc, 0), width[br] - 1));
        }
    }
    for (int64_t c = merged ? -1 : nck - 1; c >= 0; c--) {
        const int64_t k0 = c * K, k1 = std::min<int64_t>(k0 + K, nsteps);
        if (keep_powers) {
            // one recompute sweep over the segment keeps every power
            CK(cudaMemcpyAsync(pslot(0, 0, 0), vec(ck0 + c), vb, cudaMemcpyDeviceToDevice, st));
            for (int64_t k = k0; k < k1; k++) {
                void *y = (k + 1 < k1) ? pslot(k + 1 - k0, 0, 0) : fa;   // fa: free after the forward pass
                CKS(interval(k - k0, pslot(k - k0, 0, 0), y, eps[k]));
            }
        } else {
            CK(cudaMemcpyAsync(vec(pw0), vec(ck0 + c), vb, cudaMemcpyDeviceToDevice, st));
            for (int64_t k = k0; k < k1 - 1; k++)
                CKS(interval(0, vec(pw0 + (k - k0)), vec(pw0 + (k - k0 + 1)), eps[k]));
        }
        for (int64_t k = k1 - 1; k >= k0; k--) {
            const double e = eps[k];
            const void *first = keep_powers ? pslot(k - k0, 0, 0) : vec(pw0 + (k - k0));
            if (!keep_powers) CKS(interval(0, first, fa, e));   // powers of this interval (output unused)
            // costate: chi'_m = chi_{k+1}; chi'_l = T^dagger chi'_{l+1}
            for (int l = m - 1; l >= 0; l--) {
                void *B[5] = {chi, vec(b0 + 1), vec(b0 + 2), vec(b0 + 3), vec(b0 + 4)};
                CKS(powers(H, B, chi2, ld, tau, +1.0, e, dir, st));
                const void *bb[4] = {B[0], B[1], B[2], B[3]};
                const void *a0 = keep_powers ? pslot(k - k0, l, 0)
                                             : (l == 0 ? first : vec(pw0 + (K + 1) + 4 * l));
                const void *aa[4] = {a0, keep_powers ? pslot(k - k0, l, 1) : pslot(0, l, 1),
                                     keep_powers ? pslot(k - k0, l, 2) : pslot(0, l, 2),
                                     keep_powers ? pslot(k - k0, l, 3) : pslot(0, l, 3)};
                CK(launch_adjoint_grad<R>(bb, aa, P, (int)ld, (int)ld, H->Xd.as<R>(), h3, tau, H->dots.as<double>(), nba,
                                          counter, H->grad.as<double>() + k, st));
                std::swap(chi, chi2);
            }
        }
    }
    CK(cudaMemcpyAsync(grad_out, H->grad.p, (size_t)nsteps * sizeof(double), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    *J_out = ov[0] * ov[0] + ov[1] * ov[1];
    return read_status(H, st);
}

}  // namespace

extern "C" rsg_status rsg_control_gradient(rsg_ham H, const void *psi0, const void *target,
                                           int64_t nsteps, double dt, rsg_scheme scheme, int nsub,
                                           const double *eps, const double dir[3], int checkpoint_every,
                                           double *J_out, double *grad_out, void *stream) {
    if (!H || !psi0 || !target || !eps || !J_out || !grad_out) return fail(RSG_ERR_ARG, "NULL argument");
    if (!has_potential(H)) return fail(RSG_ERR_STATE, "potential not set");
    if (H->has_mask)
        return fail(RSG_ERR_UNSUPPORTED, "a mask absorber is set: the adjoint is that of the propagator without it");
    if (H->has_scaling)
        return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: the control field is a dipole field");
    if (nsteps < 1 || nsub < 1 || !std::isfinite(dt)) return fail(RSG_ERR_ARG, "bad nsteps/nsub/dt");
    if (scheme != RSG_EXPMID && scheme != RSG_ETRS) return fail(RSG_ERR_ARG, "unknown scheme");
    if (((uintptr_t)psi0) % 8 || ((uintptr_t)target) % 8) return fail(RSG_ERR_ARG, "misaligned state");
    const double xdir[3] = {1.0, 0.0, 0.0};
    const double *d = dir ? dir : xdir;
    cudaStream_t st = (cudaStream_t)stream;
    if (H->dtype == RSG_C64)
        return control_gradient_t<float>(H, psi0, target, nsteps, dt, scheme, nsub, eps, d,
                                         checkpoint_every, J_out, grad_out, st);
    return control_gradient_t<double>(H, psi0, target, nsteps, dt, scheme, nsub, eps, d,
                                      checkpoint_every, J_out, grad_out, st);
}

namespace {

// Limited-memory BFGS (two-loop recursion, memory 8) maximising J over x
// (n values, in/out) with an Armijo backtracking line search on f = -J.
// evaluate(at, J, grad) sets J(at) and grad = -dJ/dat and counts itself.
// J_hist (may be NULL) receives J after every accepted iteration.
template <typename Eval>
rsg_status lbfgs_maximise(size_t n, std::vector<double> &x, Eval &&evaluate, int64_t max_iter, double gtol,
                          double *J_out, double *J_hist, int64_t *iters_out) {
    constexpr int kMem = 8;
    auto dot = [n](const std::vector<double> &a, const std::vector<double> &b) {
        double s = 0.0;
        for (size_t i = 0; i < n; i++) s += a[i] * b[i];
        return s;
    };
    auto inf_norm = [n](const std::vector<double> &a) {
        double m = 0.0;
        for (size_t i = 0; i < n; i++) m = std::max(m, std::fabs(a[i]));
        return m;
    };
    std::vector<double> g(n), xt(n), gt(n), d(n);
    double J = 0.0, Jt = 0.0;
    CKS(evaluate(x, J, g));
    if (J_hist) J_hist[0] = J;
    std::vector<std::vector<double>> S, Y;
    std::vector<double> rho;
    int64_t it = 0;
    while (it < max_iter && inf_norm(g) > gtol) {
        // two-loop recursion: d = -H_k g
        d = g;
        std::vector<double> alpha(S.size());
        for (int k = (int)S.size() - 1; k >= 0; k--) {
            alpha[(size_t)k] = rho[(size_t)k] * dot(S[(size_t)k], d);
            for (size_t i = 0; i < n; i++) d[i] -= alpha[(size_t)k] * Y[(size_t)k][i];
        }
        double gamma = 1.0;
        if (!S.empty()) {
            gamma = dot(S.back(), Y.back()) / dot(Y.back(), Y.back());
        } else {
            // first step: a move of at most 1e-2 in the largest component
            gamma = 1e-2 / std::max(inf_norm(g), 1e-300);
        }
        for (size_t i = 0; i < n; i++) d[i] *= gamma;
        for (size_t k = 0; k < S.size(); k++) {
            const double beta = rho[k] * dot(Y[k], d);
            for (size_t i = 0; i < n; i++) d[i] += S[k][i] * (alpha[k] - beta);
        }
        for (size_t i = 0; i < n; i++) d[i] = -d[i];
        double slope = dot(g, d);
        if (!(slope < 0)) {       // not a descent direction: restart from steepest descent
            S.clear();
            Y.clear();
            rho.clear();
            const double sc = 1e-2 / std::max(inf_norm(g), 1e-300);
            for (size_t i = 0; i < n; i++) d[i] = -sc * g[i];
            slope = dot(g, d);
        }
        // Armijo backtracking on f = -J
        double step = 1.0;
        bool accepted = false;
        int ls = 0;
        for (; ls < 40; ls++) {
            for (size_t i = 0; i < n; i++) xt[i] = x[i] + step * d[i];
            CKS(evaluate(xt, Jt, gt));
            if (-Jt <= -J + 1e-4 * step * slope) {
                accepted = true;
                break;
            }
            step *= 0.5;
        }
        if (!accepted) break;     // no decrease along d: stationary to working precision
        // a scaled steepest-descent direction (no usable curvature pair yet,
        // e.g. while -J is concave along the path) is only a guess at the step
        // length: expand while J keeps increasing
        if (S.empty() && ls == 0) {
            std::vector<double> xe(n), ge(n);
            double Je = 0.0;
            for (int k = 0; k < 20; k++) {
                step *= 2.0;
                for (size_t i = 0; i < n; i++) xe[i] = x[i] + step * d[i];
                CKS(evaluate(xe, Je, ge));
                if (!(Je > Jt)) break;
                xt.swap(xe);
                gt.swap(ge);
                Jt = Je;
            }
        }
        std::vector<double> sv(n), yv(n);
        for (size_t i = 0; i < n; i++) {
            sv[i] = xt[i] - x[i];
            yv[i] = gt[i] - g[i];
        }
        const double sy = dot(sv, yv);
        if (sy > 1e-12 * std::sqrt(dot(sv, sv) * dot(yv, yv))) {
            if ((int)S.size() == kMem) {
                S.erase(S.begin());
                Y.erase(Y.begin());
                rho.erase(rho.begin());
            }
            S.push_back(sv);
            Y.push_back(yv);
            rho.push_back(1.0 / sy);
        }
        x.swap(xt);
        g.swap(gt);
        J = Jt;
        it++;
        if (J_hist) J_hist[it] = J;
    }
    *J_out = J;
    if (iters_out) *iters_out = it;
    return RSG_OK;
}

rsg_status check_optimize_args(rsg_ham H, int64_t nsteps, int64_t max_iter, double gtol) {
    if (H->has_scaling)
        return fail(RSG_ERR_UNSUPPORTED, "complex scaling is set: the control field is a dipole field");
    if (max_iter < 0 || !(gtol >= 0)) return fail(RSG_ERR_ARG, "need max_iter >= 0 and gtol >= 0");
    if (nsteps < 1) return fail(RSG_ERR_ARG, "nsteps < 1");
    return RSG_OK;
}

}  // namespace

// Optimal control loop (Sec. "Quantum optimal control": the gradient of
// Eq. (qoctgradient) feeds a gradient-based optimiser; the paper uses
// conjugate-gradient and BFGS schemes).  The parameters are the interval
// values of the field; every evaluation of J and its gradient is one
// rsg_control_gradient call.
extern "C" rsg_status rsg_control_optimize(rsg_ham H, const void *psi0, const void *target, int64_t nsteps,
                                           double dt, rsg_scheme scheme, int nsub, double *eps,
                                           const double dir[3], int checkpoint_every, int64_t max_iter,
                                           double gtol, double *J_out, double *J_hist, int64_t *iters_out,
                                           int64_t *evals_out, void *stream) {
    if (!H || !eps || !J_out) return fail(RSG_ERR_ARG, "NULL argument");
    CKS(check_optimize_args(H, nsteps, max_iter, gtol));
    const size_t n = (size_t)nsteps;
    std::vector<double> x(eps, eps + n);
    int64_t evals = 0;
    auto evaluate = [&](const std::vector<double> &at, double &Jv, std::vector<double> &grad) -> rsg_status {
        CKS(rsg_control_gradient(H, psi0, target, nsteps, dt, scheme, nsub, at.data(), dir, checkpoint_every, &Jv,
                                 grad.data(), stream));
        for (size_t i = 0; i < n; i++) grad[i] = -grad[i];
        evals++;
        if (!std::isfinite(Jv)) return fail(RSG_ERR_NONFINITE, "objective not finite");
        return RSG_OK;
    };
    CKS(lbfgs_maximise(n, x, evaluate, max_iter, gtol, J_out, J_hist, iters_out));
    std::memcpy(eps, x.data(), n * sizeof(double));
    if (evals_out) *evals_out = evals;
    return RSG_OK;
}

// The same loop over a linear parametrisation eps = B u of the field (the
// section's example: Fourier coefficients of the amplitude); the gradient
// in u is B^T dJ/deps.
extern "C" rsg_status rsg_control_optimize_basis(rsg_ham H, const void *psi0, const void *target, int64_t nsteps,
                                                 double dt, rsg_scheme scheme, int nsub, int64_t nparam,
                                                 const double *basis, double *u, const double dir[3],
                                                 int checkpoint_every, int64_t max_iter, double gtol, double *J_out,
                                                 double *J_hist, int64_t *iters_out, int64_t *evals_out,
                                                 void *stream) {
    if (!H || !basis || !u || !J_out) return fail(RSG_ERR_ARG, "NULL argument");
    CKS(check_optimize_args(H, nsteps, max_iter, gtol));
    if (nparam < 1) return fail(RSG_ERR_ARG, "nparam < 1");
    const size_t n = (size_t)nsteps, m = (size_t)nparam;
    for (size_t i = 0; i < n * m; i++)
        if (!std::isfinite(basis[i])) return fail(RSG_ERR_ARG, "basis not finite");
    std::vector<double> x(u, u + m), eps(n), ge(n);
    int64_t evals = 0;
    auto evaluate = [&](const std::vector<double> &at, double &Jv, std::vector<double> &grad) -> rsg_status {
        for (size_t k = 0; k < n; k++) {
            double e = 0.0;
            for (size_t j = 0; j < m; j++) e += basis[k * m + j] * at[j];
            eps[k] = e;
        }
        CKS(rsg_control_gradient(H, psi0, target, nsteps, dt, scheme, nsub, eps.data(), dir, checkpoint_every, &Jv,
                                 ge.data(), stream));
        for (size_t j = 0; j < m; j++) {
            double s = 0.0;
            for (size_t k = 0; k < n; k++) s += basis[k * m + j] * ge[k];
            grad[j] = -s;
        }
        evals++;
        if (!std::isfinite(Jv)) return fail(RSG_ERR_NONFINITE, "objective not finite");
        return RSG_OK;
    };
    CKS(lbfgs_maximise(m, x, evaluate, max_iter, gtol, J_out, J_hist, iters_out));
    std::memcpy(u, x.data(), m * sizeof(double));
    if (evals_out) *evals_out = evals;
    return RSG_OK;
}

// Sine series on [0, T], T = nsteps intervals, at the interval midpoints.
extern "C" rsg_status rsg_fourier_basis(int64_t nsteps, int64_t nparam, double *basis_out) {
    if (!basis_out || nsteps < 1 || nparam < 1) return fail(RSG_ERR_ARG, "bad basis arguments");
    const double pi = 3.14159265358979323846;
    for (int64_t k = 0; k < nsteps; k++)
        for (int64_t j = 0; j < nparam; j++)
            basis_out[k * nparam + j] = std::sin(pi * (double)(j + 1) * ((double)k + 0.5) / (double)nsteps);
    return RSG_OK;
}

// ============================================================== batch ====
namespace {

// Batched launch sequence of one exponential T(tau) on every system: four
// Horner stages, each = projector coefficients + reduction, staged stencil,
// projector scatter.  Codes: 0 = psi, 1 = w0, 2 = w1 (as in taylor()).
rsg_status batch_exponential(rsg_batch b, double tau, cudaStream_t st) {
    int src = 0;
    for (int k = 4; k >= 1; k--) {
        const int dst = (k == 1) ? 0 : ((k & 1) ? 2 : 1);
        const float ai = (float)(-tau / k);
        if (b->ndot > 0)
            CK(launch_batch_proj(b->d_args.as<SysArgs>(), b->d_dot.as<BWork>(), b->ndot, b->d_red.as<BWork>(),
                                 b->nred, src, b->npmax, st));
        CK(launch_batch_stencil(b->d_args.as<SysArgs>(), b->d_work.as<BWork>(), b->nwork, src, dst, 0.f, ai, st));
        if (b->nsca > 0)
            CK(launch_batch_scatter(b->d_args.as<SysArgs>(), b->d_sca.as<BWork>(), b->nsca, dst, 0.f, ai, st));
        src = dst;
    }
    return RSG_OK;
}

rsg_status batch_build_stages(rsg_batch b) {
    const int n = (int)b->hams.size();
    b->args.assign((size_t)n, SysArgs{});
    b->w0.resize((size_t)n);
    b->w1.resize((size_t)n);
    b->D.resize((size_t)n);
    b->partial.resize((size_t)n);
    std::vector<BWork> work, dot, red, sca;
    std::vector<int> work_len;   // planes of each stencil work item's tile
    int npmax = 0;
    bool uniform = true;
    for (int i = 0; i < n; i++) {
        rsg_ham H = b->hams[(size_t)i];
        rsg_mesh m = H->m;
        if (!H->has_V) return fail(RSG_ERR_STATE, "system %d has no potential", i);
        if (H->pj.natoms > 0) {
            if (npmax == 0) npmax = H->pj.npmax;
            else if (npmax != H->pj.npmax) uniform = false;
        }
        if ((int64_t)m->P * b->ld[(size_t)i] >= 0x7fffffffLL) uniform = false;
        if (b->ld[(size_t)i] > 16) uniform = false;   // batched kernels cover 8 vectors per point
    }
    b->batched = uniform;
    b->npmax = npmax;
    if (!uniform) return RSG_OK;
    for (int i = 0; i < n; i++) {
        rsg_ham H = b->hams[(size_t)i];
        rsg_mesh m = H->m;
        CKS(ensure_rows(m));
        const int64_t ld = b->ld[(size_t)i];
        const int SV = (int)(ld / 2);
        const size_t bytes = (size_t)m->P * ld * 8;
        CK(b->w0[(size_t)i].ensure(bytes));
        CK(b->w1[(size_t)i].ensure(bytes));
        const Tile *tiles = nullptr;
        int ntiles = 0;
        const std::vector<Tile> *host = nullptr;
        CKS(get_tiles(m, kBatchNXR, kBatchTY, kBatchZseg, &tiles, &ntiles, &host));
        SysArgs &A = b->args[(size_t)i];
        A.vec[0] = nullptr;
        A.vec[1] = b->w0[(size_t)i].p;
        A.vec[2] = b->w1[(size_t)i].p;
        A.rows = m->d_rows.as<Row>();
        A.tiles = tiles;
        A.nx = m->nx;
        A.ny = m->ny;
        A.nz = m->nz;
        A.SV = SV;
        A.P = (int)m->P;
        A.V = H->V.as<float>();
        for (int k = 0; k < 5; k++) A.w[k] = (float)(-0.5 * kFD[k] / (m->h * m->h));
        A.h3 = m->h * m->h * m->h;
        const int nch = (SV + kBatchCV - 1) / kBatchCV;
        const std::vector<Tile> &ht = *host;
        for (int t = 0; t < ntiles; t++)
            for (int c = 0; c < nch; c++) {
                work.push_back(BWork{i, t, c, 0});
                work_len.push_back(ht[(size_t)t].zhi - ht[(size_t)t].zlo);
            }
        const ProjDev &pj = H->pj;
        A.natoms = pj.natoms;
        A.npmax = pj.npmax;
        A.nu = pj.nu;
        if (pj.natoms > 0) {
            A.q_pt = pj.q_pt;
            A.chunk_q0 = pj.chunk_q0;
            A.chunk_q1 = pj.chunk_q1;
            A.atom_chunk0 = pj.atom_chunk0;
            A.u_pts = pj.u_pts;
            A.u_ptr = pj.u_ptr;
            A.e_atom = pj.e_atom;
            A.e_p = (const float *)pj.e_p;
            A.q_p = (const float *)pj.q_p;
            A.hm = pj.hm;
            CK(b->D[(size_t)i].ensure((size_t)pj.natoms * pj.npmax * ld * 8));
            CK(b->partial[(size_t)i].ensure((size_t)pj.nchunks * pj.npmax * ld * 2 * sizeof(double)));
            A.D = b->D[(size_t)i].as<float>();
            A.partial = b->partial[(size_t)i].as<double>();
            for (int c = 0; c < pj.nchunks; c++) dot.push_back(BWork{i, c, 0, 0});
            for (int at = 0; at < pj.natoms; at++) red.push_back(BWork{i, at, 0, 0});
            for (int u = 0; u < pj.nu; u += 32) sca.push_back(BWork{i, u, std::min(32, pj.nu - u), 0});
        }
    }
    {
        // longest stencil work items first, across systems, so that the last
        // blocks of a launch are short ones (stable: systems and tile order
        // are kept among equal lengths)
        std::vector<size_t> idx(work.size());
        for (size_t k = 0; k < idx.size(); k++) idx[k] = k;
        std::stable_sort(idx.begin(), idx.end(), [&](size_t x, size_t y) { return work_len[x] > work_len[y]; });
        std::vector<BWork> sorted(work.size());
        for (size_t k = 0; k < idx.size(); k++) sorted[k] = work[idx[k]];
        work.swap(sorted);
    }
    CK(b->d_work.upload(work));
    CK(b->d_dot.upload(dot));
    CK(b->d_red.upload(red));
    CK(b->d_sca.upload(sca));
    b->nwork = (int)work.size();
    b->ndot = (int)dot.size();
    b->nred = (int)red.size();
    b->nsca = (int)sca.size();
    b->n_launch_step = (b->ndot > 0 ? 2 : 0) + 1 + (b->nsca > 0 ? 1 : 0);
    return RSG_OK;
}

// Work items of one stage of the persistent step: the projector
// coefficients of every atom, the stencil items (tile segments times 16-value
// chunks, longest first across systems) and the scatter items of every
// system, in that order.
rsg_status batch_build_step(rsg_batch b) {
    const int n = (int)b->hams.size();
    b->batched = false;
    for (int i = 0; i < n; i++)
        if (b->ld[(size_t)i] > kBMaxLd) return RSG_OK;   // propagated one by one
    b->args.assign((size_t)n, SysArgs{});
    b->w0.resize((size_t)n);
    b->w1.resize((size_t)n);
    b->D.resize((size_t)n);
    b->partial.resize((size_t)n);
    std::vector<BItem> dots, sten, scat;
    std::vector<int> sten_len;
    int np_cap = 8;
    for (int i = 0; i < n; i++) {
        rsg_ham H = b->hams[(size_t)i];
        rsg_mesh m = H->m;
        if (!H->has_V) return fail(RSG_ERR_STATE, "system %d has no potential", i);
        const int64_t ld = b->ld[(size_t)i];
        if ((int64_t)m->P * ld >= 0x7fffffffLL || m->nx > 32000)
            return fail(RSG_ERR_UNSUPPORTED, "system %d: P * ld above 2^31 or nx above 32000", i);
        CKS(ensure_rows(m));
        const size_t bytes = (size_t)m->P * ld * 8;
        CK(b->w0[(size_t)i].ensure(bytes));
        CK(b->w1[(size_t)i].ensure(bytes));
        int TX = 16, TY = 6;
        const int ls = ld > 16 ? 16 : (int)ld;
        const int var = (b->tile_var_mask >> (ls / 2 - 1)) & 1;
        batch_step_tile((int)ld, var, &TX, &TY);
        const Tile *tiles = nullptr;
        int ntiles = 0;
        const std::vector<Tile> *host = nullptr;
        CKS(get_tiles(m, TX, TY, b->zseg, &tiles, &ntiles, &host));
        const std::vector<Tile> &ht = *host;
        SysArgs &A = b->args[(size_t)i];
        A.vec[0] = nullptr;
        A.vec[1] = b->w0[(size_t)i].p;
        A.vec[2] = b->w1[(size_t)i].p;
        A.rows = m->d_rows.as<Row>();
        A.tiles = tiles;
        A.nx = m->nx;
        A.ny = m->ny;
        A.nz = m->nz;
        A.SV = (int)(ld / 2);
        A.ld = (int)ld;
        A.P = (int)m->P;
        A.V = H->V.as<float>();
        for (int k = 0; k < 5; k++) A.w[k] = (float)(-0.5 * kFD[k] / (m->h * m->h));
        A.h3 = m->h * m->h * m->h;
        const int nch = ld > 16 ? (int)((ld + 15) / 16) : 1;
        for (int t = 0; t < ntiles; t++) {
            const int len = ht[(size_t)t].zhi - ht[(size_t)t].zlo;
            np_cap = std::max(np_cap, len + 8);
            for (int c = 0; c < nch; c++) {
                sten.push_back(BItem{1, i, t, c});
                sten_len.push_back(len);
            }
        }
        A.nsten = ntiles * nch;
        A.stall = (i == 0 && b->stall > 0) ? 1 : 0;
        A.var = var;
        const ProjDev &pj = H->pj;
        A.natoms = pj.natoms;
        A.npmax = pj.npmax;
        A.nu = pj.nu;
        A.ndot = 0;
        A.nsca = 0;
        if (pj.natoms > 0) {
            if (pj.npmax != 1 && pj.npmax != 4 && pj.npmax != 9)
                return fail(RSG_ERR_UNSUPPORTED, "system %d: %d projectors per atom", i, pj.npmax);
            A.q_pt = pj.q_pt;
            A.chunk_q0 = pj.chunk_q0;
            A.chunk_q1 = pj.chunk_q1;
            A.atom_chunk0 = pj.atom_chunk0;
            A.u_pts = pj.u_pts;
            A.u_ptr = pj.u_ptr;
            A.e_atom = pj.e_atom;
            A.e_p = (const float *)pj.e_p;
            A.q_p = (const float *)pj.q_p;
            A.hm = pj.hm;
            CK(b->D[(size_t)i].ensure((size_t)pj.natoms * pj.npmax * ld * 8));
            A.D = b->D[(size_t)i].as<float>();
            for (int at = 0; at < pj.natoms; at++) dots.push_back(BItem{0, i, at, 0});
            for (int u = 0; u < pj.nu; u += kBScatterPts) scat.push_back(BItem{2, i, u, std::min(kBScatterPts, pj.nu - u)});
            A.ndot = pj.natoms;
            A.nsca = (pj.nu + kBScatterPts - 1) / kBScatterPts;
        }
    }
    if (batch_step_smem(np_cap) > 227 * 1024)
        return fail(RSG_ERR_UNSUPPORTED, "tile segments of %d planes do not fit in shared memory", np_cap - 8);
    {
        std::vector<size_t> idx(sten.size());
        for (size_t k = 0; k < idx.size(); k++) idx[k] = k;
        std::stable_sort(idx.begin(), idx.end(), [&](size_t x, size_t y) { return sten_len[x] > sten_len[y]; });
        std::vector<BItem> sorted(sten.size());
        for (size_t k = 0; k < idx.size(); k++) sorted[k] = sten[idx[k]];
        sten.swap(sorted);
    }
    b->stage_items.clear();
    b->stage_items.insert(b->stage_items.end(), dots.begin(), dots.end());
    b->stage_items.insert(b->stage_items.end(), sten.begin(), sten.end());
    b->stage_items.insert(b->stage_items.end(), scat.begin(), scat.end());
    b->np_cap = np_cap;
    int dev = 0, sms = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    b->nblocks = std::max(1, std::min(sms, (int)b->stage_items.size()));
    CK(b->d_status.ensure(sizeof(int)));
    CK(b->d_status.zero(sizeof(int)));
    CK(b->d_ctl.ensure(sizeof(BCtl)));
    CK(b->d_zero.ensure(kBZeroBytes));
    CK(b->d_zero.zero(kBZeroBytes));
    b->step_nst = 0;   // items and counters follow the scheme at capture
    b->batched = true;
    b->n_launch_step = 1;
    return RSG_OK;
}

rsg_status batch_build(rsg_batch b) {
    if (b->cs) CK(cudaStreamSynchronize(b->cs));
    if (b->step) {
        CK(cudaGraphExecDestroy(b->step));
        b->step = nullptr;
    }
    return b->mode == 1 ? batch_build_step(b) : batch_build_stages(b);
}

// Stages of one step of the persistent kernel: each exponential T(tau) is
// four Horner stages k = 4..1, out = psi + (-i tau / k) H u, with the same
// buffer rotation as taylor() (0 = psi, 1 = w0, 2 = w1).
int batch_stages(rsg_scheme scheme, double dt, BStage *st) {
    const int nexp = scheme == RSG_ETRS ? 2 : 1;
    const double tau = scheme == RSG_ETRS ? 0.5 * dt : dt;
    int t = 0;
    for (int e = 0; e < nexp; e++) {
        int src = 0;
        for (int k = 4; k >= 1; k--) {
            const int dst = (k == 1) ? 0 : ((k & 1) ? 2 : 1);
            st[t++] = BStage{src, dst, (float)(-tau / k)};
            src = dst;
        }
    }
    return t;
}

// The queue of one step (every stage's items, stage bits set) and its
// counters, uploaded before the step is captured.
rsg_status batch_prepare_step(rsg_batch b, rsg_scheme scheme) {
    if (b->mode != 1) return RSG_OK;
    BStage st[8];
    const int nst = batch_stages(scheme, 1.0, st);
    if (b->step_nst == nst) return RSG_OK;
    std::vector<BItem> items;
    items.reserve(b->stage_items.size() * (size_t)nst);
    for (int t = 0; t < nst; t++)
        for (const BItem &w : b->stage_items) items.push_back(BItem{w.kind | (t << 2), w.sys, w.a, w.b});
    CK(b->d_items.upload(items));
    CK(b->d_cnt.ensure(b->hams.size() * (size_t)nst * 3 * sizeof(unsigned)));
    b->step_nst = nst;
    return RSG_OK;
}

rsg_status batch_capture_step(rsg_batch b, double dt, rsg_scheme scheme, cudaStream_t cs) {
    if (b->mode == 1) {
        BStepArgs a{};
        a.nst = batch_stages(scheme, dt, a.st);
        if (b->step_nst != a.nst) return fail(RSG_ERR_STATE, "batch queue not prepared");
        a.sys = b->d_args.as<SysArgs>();
        a.items = b->d_items.as<BItem>();
        a.nitems = (int)(b->stage_items.size() * (size_t)a.nst);
        a.cnt = b->d_cnt.as<unsigned>();
        a.ctl = b->d_ctl.as<BCtl>();
        a.status = b->d_status.as<int>();
        a.zeros = b->d_zero.p;
        a.wait_limit = b->wait_limit;
        a.np_cap = b->np_cap;
        CK(cudaMemsetAsync(b->d_cnt.p, 0, b->hams.size() * (size_t)a.nst * 3 * sizeof(unsigned), cs));
        CK(cudaMemsetAsync(b->d_ctl.p, 0, sizeof(BCtl), cs));
        CK(launch_batch_step(a, b->nblocks, cs));
        return RSG_OK;
    }
    if (scheme == RSG_EXPMID) return batch_exponential(b, dt, cs);
    CKS(batch_exponential(b, 0.5 * dt, cs));
    return batch_exponential(b, 0.5 * dt, cs);
}

}  // namespace

extern "C" {

rsg_status rsg_batch_create(const rsg_ham *hams, const int64_t *S, int nsys, rsg_batch *out) {
    if (!hams || !S || !out || nsys < 1) return fail(RSG_ERR_ARG, "bad batch arguments");
    std::unique_ptr<rsg_batch_s> b(new rsg_batch_s());
    for (int i = 0; i < nsys; i++) {
        if (!hams[i]) return fail(RSG_ERR_ARG, "NULL Hamiltonian %d", i);
        if (hams[i]->dtype != RSG_C64) return fail(RSG_ERR_UNSUPPORTED, "batches are complex64");
        if (hams[i]->has_mask) return fail(RSG_ERR_UNSUPPORTED, "batches do not apply mask absorbers");
        if (hams[i]->has_scaling) return fail(RSG_ERR_UNSUPPORTED, "batches do not apply complex scaling");
        if (hams[i]->m->bc != RSG_BC_ZERO) return fail(RSG_ERR_UNSUPPORTED, "batches use zero ghosts only");
        if (S[i] < 1) return fail(RSG_ERR_ARG, "S[%d] < 1", i);
        b->hams.push_back(hams[i]);
        b->S.push_back(S[i]);
        b->ld.push_back((S[i] + 1) / 2 * 2);
    }
    CKS(batch_build(b.get()));
    *out = b.release();
    return RSG_OK;
}

rsg_status rsg_batch_propagate(rsg_batch b, void *const *psis, int64_t nsteps, double dt,
                               rsg_scheme scheme, int gs_every, void *stream) {
    if (!b || !psis) return fail(RSG_ERR_ARG, "NULL argument");
    if (nsteps < 0 || gs_every < 0 || !std::isfinite(dt)) return fail(RSG_ERR_ARG, "bad nsteps/dt/gs_every");
    if (scheme != RSG_EXPMID && scheme != RSG_ETRS) return fail(RSG_ERR_ARG, "unknown scheme");
    const size_t n = b->hams.size();
    for (size_t i = 0; i < n; i++)
        if (!psis[i] || ((uintptr_t)psis[i]) % 16) return fail(RSG_ERR_ARG, "psis[%zu] NULL or misaligned", i);
    cudaStream_t st = (cudaStream_t)stream;
    if (!b->batched) {
        for (size_t i = 0; i < n; i++)
            CKS(rsg_propagate_steps(b->hams[i], psis[i], b->S[i], b->ld[i], nsteps, dt, scheme, 1, nullptr,
                                    nullptr, gs_every, nullptr, stream));
        return RSG_OK;
    }
    // (re)capture one time step when the step or the state blocks change
    bool same = b->step && b->step_dt == dt && b->step_scheme == (int)scheme && b->step_psis.size() == n;
    for (size_t i = 0; same && i < n; i++) same = b->step_psis[i] == psis[i];
    if (!same) {
        // the previous step graph may still read the tables being replaced
        if (b->cs) CK(cudaStreamSynchronize(b->cs));
        for (size_t i = 0; i < n; i++) b->args[i].vec[0] = psis[i];
        CK(b->d_args.upload(b->args));
        if (!b->cs) {
            CK(cudaStreamCreateWithFlags(&b->cs, cudaStreamNonBlocking));
            CK(cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming));
            CK(cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming));
        }
        if (b->step) {
            CK(cudaGraphExecDestroy(b->step));
            b->step = nullptr;
        }
        CKS(batch_prepare_step(b, scheme));
        cudaGraph_t g = nullptr;
        CK(cudaStreamBeginCapture(b->cs, cudaStreamCaptureModeThreadLocal));
        rsg_status s = batch_capture_step(b, dt, scheme, b->cs);
        cudaError_t ee = cudaStreamEndCapture(b->cs, &g);
        if (s != RSG_OK) {
            if (g) cudaGraphDestroy(g);
            return s;
        }
        CK(ee);
        cudaError_t ie = cudaGraphInstantiate(&b->step, g, 0);
        cudaGraphDestroy(g);
        CK(ie);
        b->step_dt = dt;
        b->step_scheme = (int)scheme;
        b->step_psis.assign(psis, psis + n);
    }
    CK(cudaEventRecord(b->ev_in, st));
    CK(cudaStreamWaitEvent(b->cs, b->ev_in, 0));
    for (int64_t k = 0; k < nsteps; k++) {
        CK(cudaGraphLaunch(b->step, b->cs));
        if (gs_every > 0 && (k + 1) % gs_every == 0) {
            for (size_t i = 0; i < n; i++) CKS(orthonormalize_dev(b->hams[i], psis[i], b->S[i], b->ld[i], nullptr, b->cs));
        }
    }
    CK(cudaEventRecord(b->ev_out, b->cs));
    CK(cudaStreamWaitEvent(st, b->ev_out, 0));
    if (gs_every > 0)
        for (size_t i = 0; i < n; i++) CKS(read_status(b->hams[i], st));
    if (b->mode == 1 && b->d_status.p) {
        int s = 0;
        CK(cudaMemcpyAsync(&s, b->d_status.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        if (s != 0) {
            CK(b->d_status.zero(sizeof(int)));
            return fail(RSG_ERR_TIMEOUT, "a bounded wait of the batched step gave up");
        }
    }
    return RSG_OK;
}

rsg_status rsg_batch_set_option(rsg_batch b, const char *name, int64_t value) {
    if (!b || !name) return fail(RSG_ERR_ARG, "NULL argument");
    const std::string k(name);
    if (k == "persistent" && (value == 0 || value == 1)) {
        b->mode = (int)value;
    } else if (k == "zseg" && value >= 8 && value <= 128) {
        b->zseg = (int)value;
    } else if (k == "wait_limit" && value >= 1) {
        b->wait_limit = (long)value;
        if (b->cs) CK(cudaStreamSynchronize(b->cs));
        if (b->step) {
            CK(cudaGraphExecDestroy(b->step));
            b->step = nullptr;
        }
        return RSG_OK;
    } else if (k == "debug_stall" && (value == 0 || value == 1)) {
        b->stall = (int)value;
    } else if (k == "tile_variants" && value >= 0 && value <= 255) {
        b->tile_var_mask = (int)value;

    } else {
        return fail(RSG_ERR_ARG, "unknown batch option %s = %lld", name, (long long)value);
    }
    return batch_build(b);
}

rsg_status rsg_batch_get_option(rsg_batch b, const char *name, int64_t *value) {
    if (!b || !name || !value) return fail(RSG_ERR_ARG, "NULL argument");
    const std::string k(name);
    if (k == "persistent") *value = b->mode;
    else if (k == "zseg") *value = b->zseg;
    else if (k == "wait_limit") *value = b->wait_limit;
    else if (k == "debug_stall") *value = b->stall;
    else if (k == "tile_variants") *value = b->tile_var_mask;
    else if (k == "batched") *value = b->batched ? 1 : 0;
    else if (k == "launches_per_step") *value = b->mode == 1 ? 1 : b->n_launch_step * 8;
    else if (k == "items_per_stage") *value = (int64_t)b->stage_items.size();
    else if (k == "blocks") *value = b->nblocks;
    else return fail(RSG_ERR_ARG, "unknown batch option %s", name);
    return RSG_OK;
}

rsg_status rsg_batch_autotune(rsg_batch b, void *const *psis, double dt, rsg_scheme scheme, void *stream,
                              double *best_ms) {
    if (!b || !psis) return fail(RSG_ERR_ARG, "NULL argument");
    if (!std::isfinite(dt) || (scheme != RSG_EXPMID && scheme != RSG_ETRS)) return fail(RSG_ERR_ARG, "bad dt/scheme");
    const size_t n = b->hams.size();
    for (size_t i = 0; i < n; i++)
        if (!psis[i] || ((uintptr_t)psis[i]) % 16) return fail(RSG_ERR_ARG, "psis[%zu] NULL or misaligned", i);
    cudaStream_t st = (cudaStream_t)stream;
    // trial steps run on copies of the states
    std::vector<DevBuf> sc(n);
    std::vector<void *> ptrs(n);
    for (size_t i = 0; i < n; i++) {
        const size_t bytes = (size_t)b->hams[i]->m->P * b->ld[i] * 8;
        CK(sc[i].ensure(bytes));
        CK(cudaMemcpyAsync(sc[i].p, psis[i], bytes, cudaMemcpyDeviceToDevice, st));
        ptrs[i] = sc[i].p;
    }
    CK(cudaStreamSynchronize(st));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    auto trial = [&](int mode, int zseg, int mask, double *ms) -> rsg_status {
        b->mode = mode;
        b->zseg = zseg;
        b->tile_var_mask = mask;
        CKS(batch_build(b));
        CKS(rsg_batch_propagate(b, ptrs.data(), 1, dt, scheme, 0, stream));
        CK(cudaEventRecord(e0, st));
        CKS(rsg_batch_propagate(b, ptrs.data(), 2, dt, scheme, 0, stream));
        CK(cudaEventRecord(e1, st));
        CK(cudaEventSynchronize(e1));
        float t = 0.f;
        CK(cudaEventElapsedTime(&t, e0, e1));
        *ms = 0.5 * t;
        return RSG_OK;
    };
    int bmode = b->mode, bz = b->zseg, bm = b->tile_var_mask;
    double best = 1e30, t = 0.0;
    rsg_status s = RSG_OK;
    // the per-stage launches, then the persistent step's segment length and
    // the tile variant of the record length that has two
    for (int mode : {0, 1}) {
        if (s == RSG_OK) s = trial(mode, bz, bm, &t);
        if (s == RSG_OK && t < best) {
            best = t;
            bmode = mode;
        }
    }
    if (s == RSG_OK && bmode == 1) {
        for (int z : {48, 64, 96, 128}) {
            if (z == bz) continue;
            if (trial(1, z, bm, &t) == RSG_OK && t < best) {
                best = t;
                bz = z;
            }
        }
        // the record length with two tile variants (14 values), if present
        bool has14 = false;
        for (size_t i = 0; i < n; i++) has14 = has14 || std::min<int64_t>(b->ld[i], 16) == 14;
        if (has14) {
            const int m2 = bm ^ (1 << 6);
            if (trial(1, bz, m2, &t) == RSG_OK && t < best) {
                best = t;
                bm = m2;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->mode = bmode;
    b->zseg = bz;
    b->tile_var_mask = bm;
    CKS(batch_build(b));
    if (s != RSG_OK) return s;
    if (best_ms) *best_ms = best;
    return RSG_OK;
}

rsg_status rsg_batch_destroy(rsg_batch b) {
    // the last step graph may still run on the internal stream
    if (b && b->cs) cudaStreamSynchronize(b->cs);
    delete b;
    return RSG_OK;
}

}  // extern "C"
