// Time stepping: fused leapfrog (2D, 3D, batched 2D), staggered
// pressure-velocity (2D), source injection, receiver interpolation, the exact
// discrete adjoint and checkpointed velocity gradients.
//
// Paper: p^{t+1} = 2p^t - p^{t-1} + dt^2 c^2 lap p + dt^2 f (2nd-order
// application section), first-order system with the paper's signs and a
// backward-staggered base stencil (1st-order section), modified operators near
// the boundary ("Reconciliation with the Interior Numerical Discretization"),
// zero Dirichlet outer edges (Examples section).
//
// 2D and staggered steps: column blocks for the bulk and row blocks that update the
// immersed-boundary rows whole, in one launch (ib_leap2d.cuh, and below).  3D
// second order: tiles marched along z, in FP32 through a TMA ring with the
// corrections in a pass of their own, in FP64 with the tile's corrections stored
// flattened (output slot, source offset, weight) and added by all threads of the
// block with shared-memory atomics.
//
// Arithmetic: coefficients (dt^2 c^2 / h^2, dt rho c^2 / h, dt / (rho h)) are
// formed in FP64 and rounded once; the leapfrog update is evaluated as
// p + ((p - p_prev) + Kh * lap) to keep one rounding at the field's magnitude.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>

#include "ib_common.cuh"

std::vector<double> ib_central_second(int M);
std::vector<double> ib_staggered_first(int M);

#define TRY(x)                          \
    do {                                \
        ib_status st_ = (x);            \
        if (st_ != IB_OK) return st_;   \
    } while (0)

// sampled event timing around one time-step kernel launch
#define PROF_LAUNCH(name, stream, ...)                   \
    do {                                                 \
        ProfToken tk_ = ib_prof_begin((name), (stream)); \
        __VA_ARGS__;                                     \
        ib_prof_end(tk_, (stream));                      \
    } while (0)

template <typename T>
static const char* kname(const char* f32, const char* f64) {
    return sizeof(T) == 8 ? f64 : f32;
}

// flattened corrections of one operator for one tile shape
template <typename T>
struct TileView {
    const int32_t* ptr;    // [ntiles + 1]
    const int32_t* loc;
    const int32_t* src;
    const T* w;
    int64_t ntx;
};

template <typename T>
struct PointSet {          // multilinear weights: 8 corner slots per point
    int n;
    const int64_t* idx;    // padded node
    const T* w;
};

// immersed-boundary rows of an operator: padded nodes, entry ranges, packed column offsets
template <typename T>
struct RowList {
    int64_t n;
    const int64_t* pad;
    const int64_t* ptr;
    const int32_t* code;
    const T* w;
};

// Each warp takes chunks of 32 consecutive entries, four chunks at a time so that
// four independent gathers are in flight per thread (surface tiles carry
// thousands of entries and would otherwise serialise on memory latency).
// Entries of one row are contiguous, so a segmented warp sum leaves one
// shared-memory atomic per row segment instead of one per entry.
template <typename T>
__device__ __forceinline__ void seg_add(T* acc, int32_t loc, T val, bool valid, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, val, o);
        int32_t l2 = __shfl_up_sync(0xffffffffu, loc, o);
        if (lane >= o && l2 == loc) val += y;
    }
    const int32_t next = __shfl_down_sync(0xffffffffu, loc, 1);
    if (valid && (lane == 31 || next != loc)) atomicAdd(&acc[loc], val);
}

template <typename T>
__device__ __forceinline__ void add_entries_range(const TileView<T>& v, int32_t e0, int32_t e1, const T* f,
                                                  int64_t origin, T* acc, int tid, int nthr);

template <typename T>
__device__ __forceinline__ void add_entries(const TileView<T>& v, int64_t tile, const T* f, int64_t origin, T* acc,
                                            int tid, int nthr) {
    add_entries_range(v, v.ptr[tile], v.ptr[tile + 1], f, origin, acc, tid, nthr);
}

// entries [e0, e1) of a tile (the range read ahead by the caller)
template <typename T>
__device__ __forceinline__ void add_entries_range(const TileView<T>& v, int32_t e0, int32_t e1, const T* f,
                                                  int64_t origin, T* acc, int tid, int nthr) {
    constexpr int U = 4;
    const int lane = tid & 31;
    const int32_t warp_base = (tid & ~31) * U;
    const int32_t step = nthr * U;
    for (int32_t base = e0 + warp_base; base < e1; base += step) {
        int32_t loc[U];
        T val[U];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int32_t e = base + u * 32 + lane;
            ok[u] = e < e1;
            loc[u] = ok[u] ? v.loc[e] : -1 - lane;
            val[u] = ok[u] ? v.w[e] * f[origin + v.src[e]] : (T)0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) seg_add(acc, loc[u], val[u], ok[u], lane);
    }
}

// source terms landing in a 2D tile (or one plane of a 3D tile): sadd[local] += w * wavelet
template <typename T, int TXA, int TYA>
__device__ __forceinline__ void tile_sources(const PointSet<T>& src, T wv, int64_t origin, int64_t px, T* sadd,
                                             int tid) {
    if (tid < 8 * src.n) {
        const int64_t rel = src.idx[tid] - origin;
        if (rel >= 0) {
            const int64_t ly = rel / px, lx = rel - ly * px;
            if (ly < TYA && lx < TXA && src.w[tid] != (T)0) atomicAdd(&sadd[ly * TXA + lx], src.w[tid] * wv);
        }
    }
}

// Receivers gid, gid + stride, ... of this launch (stride = the threads that
// record for this shot), so that every receiver is recorded whatever the grid.
template <typename T>
__device__ __forceinline__ void record_receivers(const PointSet<T>& rec, const T* p, T* traces, int nt, int col,
                                                 int64_t gid, int64_t stride) {
    if (col < 0) return;
    for (int64_t r = gid; r < rec.n; r += stride) {
        T s = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) s += rec.w[8 * r + c] * p[rec.idx[8 * r + c]];
        traces[r * nt + col] = s;
    }
}

__device__ __forceinline__ int64_t launch_threads() {
    return (int64_t)gridDim.x * gridDim.y * gridDim.z * blockDim.x * blockDim.y * blockDim.z;
}

// ---------------------------------------------------------------------------
// second-order leapfrog
// ---------------------------------------------------------------------------
template <typename T>
struct StepArgs {
    Layout L;
    T w2[5];             // central 2nd-derivative weights w[0..H]
    const T* p;          // p^n
    const T* pm;         // p^{n-1}
    T* out;              // p^{n+1} (may alias pm)
    const T* Kh;         // dt^2 c^2 / h^2 (0 outside the domain)
    TileView<T> op;
    PointSet<T> src;     // weights include dt^2 / h^d
    const T* wavelet;
    int step;
    PointSet<T> rec;     // receivers sampled from p (the previous step's output)
    T* traces;
    int nt;
    int rec_step;        // trace column written from p (-1: none)
    // batched runs: the two wavefield buffers (p^n is buf[step & 1])
    T* buf0;
    T* buf1;
    RowList<T> rows;     // 2D: the immersed-boundary rows (ib_leap2d.cuh) ...
    int64_t nrb, ntx;    // ... their blocks, and column blocks along x
    const T* damp;       // 2D: g of each node (dw > 0)
    int dw;              // absorbing layer width in nodes (0: none)
    T da;                // its largest a = eta_max dt / 2
};

// Absorbing layer along the side edges and the bottom (not the top, where the
// immersed boundary is): a = a_max min(1, d^2 / W^2) with d the node's distance
// into the layer of W nodes, d^2 = dx^2 (+ dy^2) + dz^2, dz counted from the
// bottom only.  The damped leapfrog step of p_tt + 2 a / dt p_t = c^2 lap p + f,
//   p^{n+1} = (2 p^n - (1 - a) p^{n-1} + dt^2 c^2 L p^n + dt^2 f) / (1 + a),
// is the undamped update u followed by u - g (u - p^{n-1}) with g = a / (1 + a).
template <typename T>
__device__ __forceinline__ T damp_a(const Layout& L, int dw, T da, int64_t x, int64_t y, int64_t z) {
    const int64_t w = dw;
    const int64_t dx = max(max(w - x, x - (L.nx - 1 - w)), (int64_t)0);
    const int64_t dy = L.ndim == 3 ? max(max(w - y, y - (L.ny - 1 - w)), (int64_t)0) : 0;
    const int64_t dz = max(z - (L.nz - 1 - w), (int64_t)0);
    const int64_t d2 = dx * dx + dy * dy + dz * dz;
    if (d2 == 0) return (T)0;
    const T r = (T)d2 / (T)(w * w);
    return da * (r < (T)1 ? r : (T)1);
}
// does the box [x0, x1] x [y0, y1] x [.., z1] reach into the layer (dw > 0)?
__device__ __forceinline__ bool damp_box(const Layout& L, int dw, int64_t x0, int64_t x1, int64_t y0, int64_t y1,
                                         int64_t z1) {
    return dw > 0 && (x0 < dw || x1 > L.nx - 1 - dw || z1 > L.nz - 1 - dw ||
                      (L.ndim == 3 && (y0 < dw || y1 > L.ny - 1 - dw)));
}
template <typename T>
__device__ __forceinline__ T damp_g(const Layout& L, int dw, T da, int64_t x, int64_t y, int64_t z) {
    const T av = damp_a<T>(L, dw, da, x, y, z);
    return av / ((T)1 + av);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// rounded arithmetic that the compiler may not contract into FMAs
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// asynchronous global -> shared copy of B bytes (zero fill when !valid)
template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(smem_u32(dst)), "l"(src), "n"(B),
                 "r"(valid ? B : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

#include "ib_leap2d.cuh"

// Per-shot field copies between wavefield buffers, checkpoints and segment buffers
template <typename T>
struct ShotCopy {
    const T* a;           // batched forward: the shot's buf0 (steps n even: p^n) ...
    const T* b;           // ... and buf1; adjoint restore: the checkpoint slot base
    T* dst;               // checkpoint base (forward) or segment buffer (restore)
    int64_t total;        // padded field size
};

// forward, before step n: checkpoint k = [p^n, p^{n-1}] of every shot
template <typename T>
__global__ void k_ckpt_batch(const ShotCopy<T>* __restrict__ items, int n, int k) {
    const ShotCopy<T> it = items[blockIdx.y];
    const T* cur = (n & 1) ? it.b : it.a;
    const T* prev = (n & 1) ? it.a : it.b;
    T* slot = it.dst + (int64_t)k * 2 * it.total;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < it.total; i += (int64_t)gridDim.x * blockDim.x) {
        slot[i] = cur[i];
        slot[it.total + i] = prev[i];
    }
}

// adjoint, start of segment k: segment slots 0, 1 = p^{c-1}, p^c from checkpoint k
template <typename T>
__global__ void k_seg_restore_batch(const ShotCopy<T>* __restrict__ items, int k) {
    const ShotCopy<T> it = items[blockIdx.y];
    const T* slot = it.a + (int64_t)k * 2 * it.total;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < it.total; i += (int64_t)gridDim.x * blockDim.x) {
        it.dst[i] = slot[it.total + i];
        it.dst[it.total + i] = slot[i];
    }
}

// receivers only (after the last step)
template <typename T>
__global__ void k_receivers(PointSet<T> rec, const T* p, T* traces, int nt, int col) {
    record_receivers(rec, p, traces, nt, col, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, launch_threads());
}

// 3D: (x, y) tile of 32 x 8 columns marching in z with a register queue of the
// 2H + 1 values of its own column; x/y neighbours from a shared-memory copy of
// the current plane with its halo.
template <typename T, int H>
__global__ void __launch_bounds__(256) k_leap3d(StepArgs<T> a, int zchunk, int64_t nty) {
    constexpr int TX = 32, TY = 8;
    __shared__ T tile[TY + 2 * H][TX + 2 * H];
    __shared__ T acc[TY * TX];
    __shared__ T sadd[TY * TX];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int tid = ty * TX + tx;
    const int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    record_receivers(a.rec, a.p, a.traces, a.nt, a.rec_step, blk * 256 + tid, launch_threads());
    const Layout& L = a.L;
    const int64_t x0 = (int64_t)blockIdx.x * TX, y0 = (int64_t)blockIdx.y * TY;
    const int64_t x = x0 + tx, y = y0 + ty;
    const int64_t zb = (int64_t)blockIdx.z * zchunk;
    const int64_t ze = min(zb + zchunk, L.nz);
    const bool col_ok = x < L.nx + H && y < L.ny + H;
    const bool valid = x < L.nx && y < L.ny;
    T q[2 * H + 1];
#pragma unroll
    for (int k = 0; k <= 2 * H; ++k) q[k] = col_ok ? a.p[L.idx(x, y, zb - H + k)] : (T)0;
    const T wv = a.src.n ? a.wavelet[a.step] : (T)0;
    for (int64_t z = zb; z < ze; ++z) {
        for (int i = tid; i < (TY + 2 * H) * (TX + 2 * H); i += TX * TY) {
            int ly = i / (TX + 2 * H), lx = i - ly * (TX + 2 * H);
            int64_t gx = x0 + lx - H, gy = y0 + ly - H;
            T v = 0;
            if (gx < L.nx + H && gy < L.ny + H) v = a.p[L.idx(gx, gy, z)];
            tile[ly][lx] = v;
        }
        sadd[tid] = (T)0;
        __syncthreads();
        {
            // the grouping of the TMA kernel (see there): exact zero on constants
            const T c = q[H];
            const T c6 = mul_rn((T)6, c);
            T s = 0;
#pragma unroll
            for (int k = 1; k <= H; ++k) {
                const T g = add_rn(add_rn(add_rn(tile[ty + H][tx + H + k], tile[ty + H][tx + H - k]),
                                          add_rn(tile[ty + H + k][tx + H], tile[ty + H - k][tx + H])),
                                   add_rn(q[H + k], q[H - k]));
                s = fma_(a.w2[k], sub_rn(g, c6), s);
            }
            acc[tid] = s;
        }
        const int64_t origin = L.idx(x0, y0, z);
        tile_sources<T, TX, TY>(a.src, wv, origin, L.px, sadd, tid);
        __syncthreads();
        if (a.op.ptr) add_entries(a.op, (z * nty + blockIdx.y) * a.op.ntx + blockIdx.x, a.p, origin, acc, tid, 256);
        __syncthreads();
        if (valid) {
            int64_t qi = L.idx(x, y, z);
            T c = q[H];
            const T pmq = a.pm[qi];
            T u = c + ((c - pmq) + a.Kh[qi] * acc[tid]) + sadd[tid];
            if (a.dw && damp_box(L, a.dw, x, x, y, y, z)) u -= damp_g<T>(L, a.dw, a.da, x, y, z) * (u - pmq);
            a.out[qi] = u;
        }
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) q[k] = q[k + 1];
        // plane z + 1 + H exists only while z + 1 < ze (the last allocated plane is nz + H - 1)
        q[2 * H] = (col_ok && z + 1 < ze) ? a.p[L.idx(x, y, z + 1 + H)] : (T)0;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// 3D leapfrog, FP32, with the plane tiles staged by TMA.  Each block marches a
// 32 x 8 column tile through its z chunk.  Plane z (with an x halo of 4 -- the
// 16-byte alignment of the box -- and a y halo of H) is fetched by one
// cp.async.bulk.tensor into a ring of NS shared-memory slots, NS - H - 1 planes
// ahead of use, each slot tracked by an mbarrier.  The z neighbours come from a
// register queue fed by the centre of plane z + H.  Every wait is bounded: on
// timeout the block records an error and leaves.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(tm), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// bounded wait; returns false once about one second has passed (or after 2^22
// polls, should the global timer not advance)
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (int it = 0; it < (1 << 22); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > 1000000000ull) break;
    }
    return false;
}

// Self-test of the bounded wait: one thread arms an mbarrier for bytes that no
// copy will ever deliver and waits with the same bound as the TMA kernels; the
// wait gives up and the kernel reports it through the error word.
__global__ void k_wait_selftest(int* err) {
    __shared__ alignas(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&bar, 16);
    if (!mbar_wait_bounded(&bar, 0)) atomicExch(err, 1);
}

// compact corrections of the 3D tile planes (TileBins compact form): entries of
// tile plane t are [ptr[t], ptr[t + 1]), each an output slot (one byte), a 16-bit
// footprint code and an FP32 weight
struct Rows3 {
    const int32_t* ptr;
    const uint8_t* slot;
    const uint16_t* code;
    const float* w;
};

// Entries [e0, e1) of a tile plane: each warp takes chunks of 32 consecutive
// entries, four chunks at a time (four independent gathers in flight per
// thread); entries of one row are contiguous, so a segmented warp sum leaves one
// shared-memory atomic per row segment.  Values are read from p^n (L2).
__device__ __forceinline__ void add_entries3(const Rows3& r, int32_t e0, int32_t e1, const float* prow0,
                                             int64_t px, int64_t plane, float* acc, int tid) {
    constexpr int U = 4;
    const int lane = tid & 31;
    const int32_t warp_base = (tid & ~31) * U;
    for (int32_t base = e0 + warp_base; base < e1; base += 256 * U) {
        int32_t loc[U];
        float val[U];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int32_t e = base + u * 32 + lane;
            ok[u] = e < e1;
            float v = 0.f;
            loc[u] = -1 - lane;
            if (ok[u]) {
                const int sl = r.slot[e];
                const int c = r.code[e];
                const int dx = (c & 31) - 16, dy = ((c >> 5) & 31) - 16, dz = (c >> 10) - 16;
                loc[u] = sl;
                v = r.w[e] * prow0[(int64_t)dz * plane + ((sl >> 5) + dy) * px + (sl & 31) + dx];
            }
            val[u] = v;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) seg_add(acc, loc[u], val[u], ok[u], lane);
    }
}

template <int H, int D>
struct Tma3D {
    static constexpr int TX = 32, TY = 8;
    static constexpr int BW = TX + 8;         // x halo 4 on each side (16-byte aligned box)
    static constexpr int BH = TY + 2 * H;
    static constexpr int NS = H + 1 + D;      // ring slots: planes z .. z + H + D (D planes in flight)
    static constexpr int PF = BW * BH;        // p plane with halo (floats)
    static constexpr int TF = TX * TY;        // p_prev or K tile (floats)
    static constexpr int SLOT = (PF + 2 * TF + 31) / 32 * 32;   // slot stride in floats (128-byte multiple)
    static constexpr uint32_t BYTES = (PF + 2 * TF) * 4;
};

// Laplacian (difference form) at the centre r0 of a staged plane, z neighbours from
// the register queue q (centre q[H + O]): sum_k w_k (((a + b) + (d + e)) + (f + g)
// - 6 c) over the six neighbours at distance k.  For a constant field each group
// is exactly zero in floating point (6 c rounds like the sum of the pairs), so the
// discrete operator annihilates constants.
template <int H, int O>
__device__ __forceinline__ float lap3_tma(const float* r0, const float (&q)[2 * H + 2], const float* w2) {
    constexpr int BW = 40;
    const float c = q[H + O];
    const float c6 = __fmul_rn(6.f, c);
    float sum = 0.f;
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        const float g = __fadd_rn(__fadd_rn(__fadd_rn(r0[k], r0[-k]), __fadd_rn(r0[k * BW], r0[-k * BW])),
                                  __fadd_rn(q[H + O + k], q[H + O - k]));
        sum = fmaf(w2[k], __fsub_rn(g, c6), sum);
    }
    return sum;
}

// Each block marches a 32 x 8 column tile through its z chunk, two planes per
// iteration.  Ring slot k holds plane z (with an x halo of 4 and a y halo of H) of
// p^n, and the tiles of p^{n-1} and of K = dt^2 c^2 / h^2 at plane z: three
// cp.async.bulk.tensor copies on one mbarrier, issued when the slot's previous
// plane is done.  The z neighbours come from a register queue fed by the centres of
// planes z + H and z + H + 1.  The corrections of each tile plane are gathered by
// all threads (add_entries3): per entry a one-byte output slot, a 16-bit footprint
// code and an FP32 weight (7 bytes), the value read from p^n in global memory
// (L2).  Every wait is bounded: on timeout the block records an error, waits
// (bounded) for the planes already requested, and leaves.
template <int H, int D>
__global__ void __launch_bounds__(256, D <= 2 ? 6 : 5) k_leap3d_tma(StepArgs<float> a, const __grid_constant__ CUtensorMap tm,
                                                    const __grid_constant__ CUtensorMap tmm,
                                                    const __grid_constant__ CUtensorMap tmk, Rows3 rw, int zchunk,
                                                    int64_t nty, int* err) {
    using C = Tma3D<H, D>;
    constexpr int TX = C::TX, TY = C::TY, BW = C::BW, NS = C::NS, SLOT = C::SLOT, PF = C::PF, TF = C::TF;
    static_assert(NS >= H + 2, "planes z .. z + H + 1 are resident together");
    static_assert(BW == 40, "lap3_tma reads rows of 40 floats");
    extern __shared__ __align__(128) float dsm[];
    float* ring = dsm;                                  // NS * SLOT
    float* acc = ring + NS * SLOT;                      // [2][TY * TX]
    float* sadd = acc + 2 * TY * TX;                    // [2][TY * TX]
    uint64_t* bar = (uint64_t*)(sadd + 2 * TY * TX);    // NS
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int tid = ty * TX + tx;
    const int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    record_receivers(a.rec, a.p, a.traces, a.nt, a.rec_step, blk * 256 + tid, launch_threads());
    const Layout& L = a.L;
    const int64_t x0 = (int64_t)blockIdx.x * TX, y0 = (int64_t)blockIdx.y * TY;
    const int64_t x = x0 + tx, y = y0 + ty;
    const int64_t zb = (int64_t)blockIdx.z * zchunk;
    const int64_t ze = min(zb + zchunk, L.nz);
    const int64_t zlast = ze - 1 + H;                 // last p plane fetched
    const bool col_ok = x < L.nx + H && y < L.ny + H;
    const bool valid = x < L.nx && y < L.ny;
    const bool damped_xy = damp_box(L, a.dw, x0, x0 + TX - 1, y0, y0 + TY - 1, 0);
    // tensor rows: p plane z, tile row y0 - H at (H + 1 + z) py + y0; tile row y0 at + H
    auto prow = [&](int64_t z) { return (int)((H + 1 + z) * L.py + y0); };
    // slot for plane zz: p box always; the p_prev / K tiles only for planes the block updates
    auto issue = [&](int slot, int64_t zz) {
        const bool upd = zz < ze;
        mbar_expect_tx(&bar[slot], (uint32_t)(PF * 4 + (upd ? 2 * TF * 4 : 0)));
        float* dst = ring + slot * SLOT;
        tma_load_2d(dst, &tm, (int)(x0 - 4), prow(zz), &bar[slot]);
        if (upd) {
            tma_load_2d(dst + PF, &tmm, (int)x0, prow(zz) + H, &bar[slot]);
            tma_load_2d(dst + PF + TF, &tmk, (int)x0, prow(zz) + H, &bar[slot]);
        }
    };
    // bounded wait for plane zz of this chunk
    auto wait_plane = [&](int64_t zz) {
        const int ip = (int)(zz - zb);
        return mbar_wait_bounded(&bar[ip % NS], (uint32_t)((ip / NS) & 1));
    };
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) mbar_init(&bar[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (tid == 0)
        for (int i = 0; i < NS && zb + i <= zlast; ++i) issue(i, zb + i);
    float q[2 * H + 2];
#pragma unroll
    for (int k = 0; k < 2 * H; ++k) q[k] = col_ok ? a.p[L.idx(x, y, zb - H + k)] : 0.f;
    const float wv = a.src.n ? a.wavelet[a.step] : 0.f;
    const int64_t tile_z = nty * a.op.ntx;              // tiles per plane
    const int64_t tile0 = (int64_t)blockIdx.y * a.op.ntx + blockIdx.x;
    const bool src_me = tid < 8 * a.src.n;
    const int64_t s_idx = src_me ? a.src.idx[tid] : 0;
    const float s_w = src_me ? a.src.w[tid] : 0.f;
    int64_t qi = L.idx(x, y, zb);
    for (int64_t z = zb; z < ze; z += 2) {
        const bool two = z + 1 < ze;
        const int ia = (int)(z - zb);
        // entry ranges of the two tile planes (read while the planes are waited for)
        int32_t ea0 = 0, ea1 = 0, eb0 = 0, eb1 = 0;
        if (rw.ptr) {
            const int32_t* pp = rw.ptr + z * tile_z + tile0;
            ea0 = pp[0];
            ea1 = pp[1];
            if (two) {
                eb0 = pp[tile_z];
                eb1 = pp[tile_z + 1];
            }
        }
        bool ok = wait_plane(z) && wait_plane(z + H);
        if (two) ok = ok && wait_plane(z + 1) && wait_plane(z + 1 + H);
        // (after a failed wait the reads below see stale shared memory; the barrier
        // that follows them tells every thread, and the block leaves)
        const float* ra = ring + (ia % NS) * SLOT;           // plane z, row j <-> y0 - H + j
        const float* rb = ring + ((ia + 1) % NS) * SLOT;     // plane z + 1
        const int ci = (H + ty) * BW + 4 + tx;
        q[2 * H] = ring[((ia + H) % NS) * SLOT + ci];
        q[2 * H + 1] = two ? ring[((ia + H + 1) % NS) * SLOT + ci] : 0.f;
        const float pma = ra[PF + tid], kha = ra[PF + TF + tid];
        const float pmb = rb[PF + tid], khb = rb[PF + TF + tid];
        acc[tid] = lap3_tma<H, 0>(ra + ci, q, a.w2);
        acc[TX * TY + tid] = lap3_tma<H, 1>(rb + ci, q, a.w2);
        sadd[tid] = 0.f;
        sadd[TX * TY + tid] = 0.f;
        const int64_t origin = L.idx(x0, y0, z);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicExch(err, 1);
                // issue nothing more, and wait (bounded) for every plane already issued
                // (planes z .. z + NS - 1), so that no copy is still landing in this
                // block's shared memory when it leaves
                const int64_t ziss = min(z + NS - 1, zlast);
                for (int64_t zp = z; zp <= ziss; ++zp) wait_plane(zp);
            }
            return;
        }
        if (src_me && s_w != 0.f) {
            const int64_t rel = s_idx - origin;
            if (rel >= 0) {
                const int64_t lz = rel / L.plane, r2 = rel - lz * L.plane;
                const int64_t ly = r2 / L.px, lx = r2 - ly * L.px;
                if (lz < (two ? 2 : 1) && ly < TY && lx < TX) atomicAdd(&sadd[lz * TX * TY + ly * TX + lx], s_w * wv);
            }
        }
        if (ea1 > ea0) add_entries3(rw, ea0, ea1, a.p + origin, L.px, L.plane, acc, tid);
        if (eb1 > eb0) add_entries3(rw, eb0, eb1, a.p + origin + L.plane, L.px, L.plane, acc + TX * TY, tid);
        __syncthreads();
        // the two slots are free (p_prev and K read above, the stencils done): the
        // planes NS further into them
        if (tid == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (z + NS <= zlast) issue(ia % NS, z + NS);
            if (two && z + 1 + NS <= zlast) issue((ia + 1) % NS, z + 1 + NS);
        }
        if (valid) {
            float u = q[H] + ((q[H] - pma) + kha * acc[tid]) + sadd[tid];
            if (damped_xy || (a.dw && z > L.nz - 1 - a.dw)) u -= damp_g<float>(L, a.dw, a.da, x, y, z) * (u - pma);
            a.out[qi] = u;
            if (two) {
                float ub = q[H + 1] + ((q[H + 1] - pmb) + khb * acc[TX * TY + tid]) + sadd[TX * TY + tid];
                if (damped_xy || (a.dw && z + 1 > L.nz - 1 - a.dw))
                    ub -= damp_g<float>(L, a.dw, a.da, x, y, z + 1) * (ub - pmb);
                a.out[qi + L.plane] = ub;
            }
        }
        qi += 2 * L.plane;
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) q[k] = q[k + 2];
    }
    // planes fetched past the chunk that no iteration waited for (chunks shorter than H):
    // complete them before the block leaves
    bool ok = true;
    for (int64_t zz = ze; zz <= zlast; ++zz) ok = ok && wait_plane(zz);
    if (!ok && tid == 0) atomicExch(err, 1);
}

// Corrections of the modified Laplacian for a 3D step whose kernel applied the
// standard stencil only, over all IB rows of the grid at once:
//   out[q] += (1 - g(q)) K[q] sum_j w_j p[q + off_j]
// (g the absorbing-layer factor of the step, 0 outside the layer), entries as a
// 16-bit footprint code and an FP32 weight in row order.  A group of 8 lanes takes
// one row (a warp four rows), each lane up to U entries per round with their
// gathers in flight together, and the sum is added with a reduction that returns
// nothing (rows are distinct nodes), so no lane waits on it.
template <int U>
__global__ void __launch_bounds__(256) k_ib_add3(int64_t nrows, const int64_t* __restrict__ row_pad,
                                                 const int64_t* __restrict__ row_ptr,
                                                 const uint16_t* __restrict__ code, const float* __restrict__ w,
                                                 const float* __restrict__ p, const float* __restrict__ Kh,
                                                 float* out, Layout L, int dw, float da) {
    const int lane = threadIdx.x & 31, gl = lane & 7;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    auto gather = [&](int64_t q, int c) {
        return p[q + (int64_t)((c >> 10) - 16) * L.plane + (int64_t)(((c >> 5) & 31) - 16) * L.px + ((c & 31) - 16)];
    };
    for (int64_t rb = warp * 4; rb < nrows; rb += nwarp * 4) {
        const int64_t r = rb + (lane >> 3);
        const bool act = r < nrows;
        const int64_t q = act ? row_pad[r] : 0;
        const int64_t j0 = act ? row_ptr[r] : 0, j1 = act ? row_ptr[r + 1] : 0;
        float v = 0.f;
        for (int64_t j = j0 + gl; j < j1; j += 8 * U) {
            float wv[U], pv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t e = j + 8 * u;
                const bool ok = e < j1;
                const int c = ok ? code[e] : 16 | (16 << 5) | (16 << 10);
                wv[u] = ok ? w[e] : 0.f;
                pv[u] = gather(q, c);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) v += wv[u] * pv[u];
        }
        v += __shfl_xor_sync(0xffffffffu, v, 4, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 2, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 1, 8);
        if (act && gl == 0) {
            float add = Kh[q] * v;
            if (dw) {
                const int64_t rel = q - L.base, z = rel / L.plane, rem = rel - z * L.plane;
                const int64_t y = rem / L.px, x = rem - y * L.px;
                add *= 1.f - damp_g<float>(L, dw, da, x, y, z);
            }
            atomicAdd(&out[q], add);
        }
    }
}

template <int H, int D>
static size_t tma3d_smem() {
    using C = Tma3D<H, D>;
    return sizeof(float) * ((size_t)C::NS * C::SLOT + 4 * C::TX * C::TY) + sizeof(uint64_t) * C::NS;
}

// planes in flight per block: 3 by default (IB_RING=2 or 5 selects 2 or 5, for tuning)
template <int H>
static void launch_leap3d_tma(const StepArgs<float>& a, const CUtensorMap& tm, const CUtensorMap& tmm,
                              const CUtensorMap& tmk, const Rows3& rw, int zchunk, int64_t nty, int* err, dim3 grid,
                              cudaStream_t s) {
    static const int ring = [] {
        const char* e = getenv("IB_RING");
        const int r = e ? atoi(e) : 3;
        return r == 5 || r == 2 ? r : 3;
    }();
    const dim3 blk(32, 8);
    if (ring == 2) {
        k_leap3d_tma<H, 2><<<grid, blk, tma3d_smem<H, 2>(), s>>>(a, tm, tmm, tmk, rw, zchunk, nty, err);
    } else if (ring == 5) {
        const size_t sm = tma3d_smem<H, 5>();
        cudaFuncSetAttribute(k_leap3d_tma<H, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_leap3d_tma<H, 5><<<grid, blk, sm, s>>>(a, tm, tmm, tmk, rw, zchunk, nty, err);
    } else {
        k_leap3d_tma<H, 3><<<grid, blk, tma3d_smem<H, 3>(), s>>>(a, tm, tmm, tmk, rw, zchunk, nty, err);
    }
}

// ---------------------------------------------------------------------------
// 3D step on x-pairs: the 64 x 8 column tile of a block is marched in z two
// planes per iteration like k_leap3d_tma, with each thread computing two
// x-adjacent points.  The x and y neighbours of the pair come in as 8-byte
// shared-memory loads (the x row -4 .. +5 in five, each y neighbour pair in one)
// and the waits, barriers and address arithmetic of an iteration are shared by
// four points instead of two.  The corrections are added by k_ib_add3 after the
// launch; sources touch shared memory only in the blocks that hold one.
// ---------------------------------------------------------------------------
template <int H, int D>
struct Tma3P {
    static constexpr int TX = 64, TY = 8;
    static constexpr int BW = TX + 8;         // x halo 4 on each side (16-byte aligned box)
    static constexpr int BH = TY + 2 * H;
    static constexpr int NS = H + 1 + D;      // ring slots: planes z .. z + H + D
    static constexpr int PF = (BW * BH + 31) / 32 * 32;   // p plane, padded to 128 bytes
    static constexpr int TF = TX * TY;
    static constexpr int SLOT = PF + 2 * TF;
};

// Laplacians of the pair centred at r0[0], r0[1] (r0 8-byte aligned, rows of 72
// floats), z neighbours from the register queue q (centre q[H + O]); the grouping
// and rounding of lap3_tma for each point
template <int H, int O>
__device__ __forceinline__ float2 lap3_pair(const float* r0, const float2 (&q)[2 * H + 2], const float* w2) {
    constexpr int BW = 72;
    float2 xv[5];   // r0[-4 .. 5]
#pragma unroll
    for (int j = 0; j < 5; ++j) xv[j] = *reinterpret_cast<const float2*>(r0 + 2 * j - 4);
    auto X = [&](int o) -> float {
        const int j = o + 4;
        return (j & 1) ? xv[j >> 1].y : xv[j >> 1].x;
    };
    const float2 c = q[H + O];
    const float c6a = __fmul_rn(6.f, c.x), c6b = __fmul_rn(6.f, c.y);
    float sa = 0.f, sb = 0.f;
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        const float2 yp = *reinterpret_cast<const float2*>(r0 + k * BW);
        const float2 ym = *reinterpret_cast<const float2*>(r0 - k * BW);
        const float ga = __fadd_rn(__fadd_rn(__fadd_rn(X(k), X(-k)), __fadd_rn(yp.x, ym.x)),
                                   __fadd_rn(q[H + O + k].x, q[H + O - k].x));
        const float gb = __fadd_rn(__fadd_rn(__fadd_rn(X(1 + k), X(1 - k)), __fadd_rn(yp.y, ym.y)),
                                   __fadd_rn(q[H + O + k].y, q[H + O - k].y));
        sa = fmaf(w2[k], __fsub_rn(ga, c6a), sa);
        sb = fmaf(w2[k], __fsub_rn(gb, c6b), sb);
    }
    return make_float2(sa, sb);
}

template <int H, int D>
__global__ void __launch_bounds__(256, 3) k_leap3d_tma2(StepArgs<float> a, const __grid_constant__ CUtensorMap tm,
                                                        const __grid_constant__ CUtensorMap tmm,
                                                        const __grid_constant__ CUtensorMap tmk, int zchunk,
                                                        int* err) {
    using C = Tma3P<H, D>;
    constexpr int TX = C::TX, TY = C::TY, BW = C::BW, NS = C::NS, SLOT = C::SLOT, PF = C::PF, TF = C::TF;
    static_assert(NS >= H + 2, "planes z .. z + H + 1 are resident together");
    static_assert(BW == 72 && H <= 4, "lap3_pair reads rows of 72 floats, x halo 4");
    extern __shared__ __align__(128) float dsm[];
    float* ring = dsm;                                  // NS * SLOT
    float* sadd = ring + NS * SLOT;                     // [2][TY * TX]
    uint64_t* bar = (uint64_t*)(sadd + 2 * TY * TX);    // NS
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int tid = ty * 32 + tx;
    const int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    record_receivers(a.rec, a.p, a.traces, a.nt, a.rec_step, blk * 256 + tid, launch_threads());
    const Layout& L = a.L;
    const int64_t x0 = (int64_t)blockIdx.x * TX, y0 = (int64_t)blockIdx.y * TY;
    const int64_t xa = x0 + 2 * tx, y = y0 + ty;        // this thread's points: (xa, y), (xa + 1, y)
    const int64_t zb = (int64_t)blockIdx.z * zchunk;
    const int64_t ze = min(zb + zchunk, L.nz);
    const int64_t zlast = ze - 1 + H;
    const bool va = xa < L.nx && y < L.ny, vb = xa + 1 < L.nx && y < L.ny;
    const bool damped_xy = damp_box(L, a.dw, x0, x0 + TX - 1, y0, y0 + TY - 1, 0);
    auto prow = [&](int64_t z) { return (int)((H + 1 + z) * L.py + y0); };
    auto issue = [&](int slot, int64_t zz) {
        const bool upd = zz < ze;
        mbar_expect_tx(&bar[slot], (uint32_t)(BW * C::BH * 4 + (upd ? 2 * TF * 4 : 0)));
        float* dst = ring + slot * SLOT;
        tma_load_2d(dst, &tm, (int)(x0 - 4), prow(zz), &bar[slot]);
        if (upd) {
            tma_load_2d(dst + PF, &tmm, (int)x0, prow(zz) + H, &bar[slot]);
            tma_load_2d(dst + PF + TF, &tmk, (int)x0, prow(zz) + H, &bar[slot]);
        }
    };
    auto wait_plane = [&](int64_t zz) {
        const int ip = (int)(zz - zb);
        return mbar_wait_bounded(&bar[ip % NS], (uint32_t)((ip / NS) & 1));
    };
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) mbar_init(&bar[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // does a source corner fall in this block's columns and z chunk? (block-uniform)
    int src_here = 0;
    const float wv = a.src.n ? a.wavelet[a.step] : 0.f;
    const bool src_me = tid < 8 * a.src.n;
    int64_t s_rel = -1;   // this thread's corner, relative to node (x0, y0, zb)
    float s_val = 0.f;
    if (src_me && a.src.w[tid] != 0.f) {
        const int64_t rel = a.src.idx[tid] - L.idx(x0, y0, zb);
        if (rel >= 0) {
            const int64_t lz = rel / L.plane, r2 = rel - lz * L.plane;
            const int64_t ly = r2 / L.px, lx = r2 - ly * L.px;
            if (lz < ze - zb && ly < TY && lx < TX) {
                s_rel = rel;
                s_val = a.src.w[tid] * wv;
            }
        }
    }
    src_here = __syncthreads_or(s_rel >= 0);
    if (tid == 0)
        for (int i = 0; i < NS && zb + i <= zlast; ++i) issue(i, zb + i);
    float2 q[2 * H + 2];
    {
        const bool ca = xa < L.nx + H && y < L.ny + H, cb = xa + 1 < L.nx + H && y < L.ny + H;
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) {
            const int64_t i = L.idx(xa, y, zb - H + k);
            q[k] = make_float2(ca ? a.p[i] : 0.f, cb ? a.p[i + 1] : 0.f);
        }
    }
    int64_t qi = L.idx(xa, y, zb);
    const int ci = (H + ty) * BW + 4 + 2 * tx;   // pair centre in a slot's p plane
    const int ti = ty * TX + 2 * tx;             // pair in a slot's p_prev / K tile
    for (int64_t z = zb; z < ze; z += 2) {
        const bool two = z + 1 < ze;
        const int ia = (int)(z - zb);
        bool ok = wait_plane(z) && wait_plane(z + H);
        if (two) ok = ok && wait_plane(z + 1) && wait_plane(z + 1 + H);
        // (after a failed wait the reads below see stale shared memory; the barrier
        // that follows them tells every thread, and the block leaves)
        const float* ra = ring + (ia % NS) * SLOT;
        const float* rb = ring + ((ia + 1) % NS) * SLOT;
        q[2 * H] = *reinterpret_cast<const float2*>(ring + ((ia + H) % NS) * SLOT + ci);
        q[2 * H + 1] = two ? *reinterpret_cast<const float2*>(ring + ((ia + H + 1) % NS) * SLOT + ci)
                           : make_float2(0.f, 0.f);
        const float2 pma = *reinterpret_cast<const float2*>(ra + PF + ti);
        const float2 kha = *reinterpret_cast<const float2*>(ra + PF + TF + ti);
        const float2 pmb = *reinterpret_cast<const float2*>(rb + PF + ti);
        const float2 khb = *reinterpret_cast<const float2*>(rb + PF + TF + ti);
        const float2 la = lap3_pair<H, 0>(ra + ci, q, a.w2);
        const float2 lb = lap3_pair<H, 1>(rb + ci, q, a.w2);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicExch(err, 1);
                const int64_t ziss = min(z + NS - 1, zlast);
                for (int64_t zp = z; zp <= ziss; ++zp) wait_plane(zp);
            }
            return;
        }
        // the two slots are free: the planes NS further into them
        if (tid == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (z + NS <= zlast) issue(ia % NS, z + NS);
            if (two && z + 1 + NS <= zlast) issue((ia + 1) % NS, z + 1 + NS);
        }
        float2 ua, ub;
        ua.x = q[H].x + ((q[H].x - pma.x) + kha.x * la.x);
        ua.y = q[H].y + ((q[H].y - pma.y) + kha.y * la.y);
        ub.x = q[H + 1].x + ((q[H + 1].x - pmb.x) + khb.x * lb.x);
        ub.y = q[H + 1].y + ((q[H + 1].y - pmb.y) + khb.y * lb.y);
        if (src_here) {   // block-uniform
            float2* s2 = reinterpret_cast<float2*>(sadd);
            s2[tid] = make_float2(0.f, 0.f);
            s2[TX * TY / 2 + tid] = make_float2(0.f, 0.f);
            __syncthreads();
            if (s_rel >= 0) {
                const int64_t r = s_rel - (z - zb) * L.plane;
                if (r >= 0) {
                    const int64_t lz = r / L.plane, r2 = r - lz * L.plane;
                    const int64_t ly = r2 / L.px, lx = r2 - ly * L.px;
                    if (lz < (two ? 2 : 1)) atomicAdd(&sadd[lz * TX * TY + ly * TX + lx], s_val);
                }
            }
            __syncthreads();
            const float2 sa = s2[ti / 2], sb = s2[TX * TY / 2 + ti / 2];
            ua.x += sa.x;
            ua.y += sa.y;
            ub.x += sb.x;
            ub.y += sb.y;
        }
        if (damped_xy || (a.dw && z + 1 > L.nz - 1 - a.dw)) {
            ua.x -= damp_g<float>(L, a.dw, a.da, xa, y, z) * (ua.x - pma.x);
            ua.y -= damp_g<float>(L, a.dw, a.da, xa + 1, y, z) * (ua.y - pma.y);
            if (two) {
                ub.x -= damp_g<float>(L, a.dw, a.da, xa, y, z + 1) * (ub.x - pmb.x);
                ub.y -= damp_g<float>(L, a.dw, a.da, xa + 1, y, z + 1) * (ub.y - pmb.y);
            }
        }
        if (va && vb) {
            *reinterpret_cast<float2*>(a.out + qi) = ua;
            if (two) *reinterpret_cast<float2*>(a.out + qi + L.plane) = ub;
        } else if (va) {
            a.out[qi] = ua.x;
            if (two) a.out[qi + L.plane] = ub.x;
        }
        qi += 2 * L.plane;
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) q[k] = q[k + 2];
    }
    bool ok = true;
    for (int64_t zz = ze; zz <= zlast; ++zz) ok = ok && wait_plane(zz);
    if (!ok && tid == 0) atomicExch(err, 1);
}

template <int H, int D>
static size_t tma3p_smem() {
    using C = Tma3P<H, D>;
    return sizeof(float) * ((size_t)C::NS * C::SLOT + 2 * C::TX * C::TY) + sizeof(uint64_t) * C::NS;
}

// x-pair kernel: 3 planes in flight beyond the ones read (IB_RING=2: 2).  At
// 512^2 x 384, order 8: 325 us per launch with 3, 383 us with 2 (three blocks of
// 74 KB or 65 KB per SM either way).
template <int H>
static void launch_leap3d_tma2(const StepArgs<float>& a, const CUtensorMap& tm, const CUtensorMap& tmm,
                               const CUtensorMap& tmk, int zchunk, int* err, dim3 grid, cudaStream_t s) {
    static const int ring = [] {
        const char* e = getenv("IB_RING");
        return e && atoi(e) == 2 ? 2 : 3;
    }();
    const dim3 blk(32, 8);
    if (ring == 3) {
        static const size_t sm = tma3p_smem<H, 3>();
        static const bool attr = (cudaFuncSetAttribute(k_leap3d_tma2<H, 3>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                                  true);
        (void)attr;
        k_leap3d_tma2<H, 3><<<grid, blk, sm, s>>>(a, tm, tmm, tmk, zchunk, err);
    } else {
        static const size_t sm = tma3p_smem<H, 2>();
        static const bool attr = (cudaFuncSetAttribute(k_leap3d_tma2<H, 2>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                                  true);
        (void)attr;
        k_leap3d_tma2<H, 2><<<grid, blk, sm, s>>>(a, tm, tmm, tmk, zchunk, err);
    }
}

// ---------------------------------------------------------------------------
// setup kernels (coefficients formed in FP64, rounded once)
// ---------------------------------------------------------------------------
// a square without the sign bit that a NaN may carry (the mark of a row node); integer operations,
// since the conversions keep the FP64 pipe busy as it is
__device__ __forceinline__ float no_sign(float k) { return __uint_as_float(__float_as_uint(k) & 0x7fffffffu); }
__device__ __forceinline__ double no_sign(double k) {
    return __hiloint2double(__double2hiint(k) & 0x7fffffff, __double2loint(k));
}
template <typename T>
__global__ void k_leap_coef(Layout L, const T* vel, const uint8_t* mask, double dt_over_h, T* Kh) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < L.N; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t x = i % L.nx, r = i / L.nx, y = r % L.ny, z = r / L.ny;
        int64_t q = L.idx(x, y, z);
        double c = (double)vel[i] * dt_over_h;
        Kh[q] = mask[q] ? no_sign((T)(c * c)) : (T)0;
    }
}

// The mark of a row node in a staggered coefficient field: a NaN of a bit pattern of its own
// (coefficients have either sign, a negative density's are negative).
static const uint32_t MARK3_32 = 0x7fc5a3c1u;
static const uint64_t MARK3_64 = 0x7ffd5a3c00000000ull;
__device__ __forceinline__ bool marked3(float k) { return __float_as_uint(k) == MARK3_32; }
__device__ __forceinline__ bool marked3(double k) { return __double2hiint(k) == (int)(MARK3_64 >> 32); }
__device__ __forceinline__ void set_mark3(float& k) { k = __uint_as_float(MARK3_32); }
__device__ __forceinline__ void set_mark3(double& k) { k = __longlong_as_double((long long)MARK3_64); }
// a coefficient, whose own NaN is not that one (a conversion to FP32 gives the canonical NaN)
template <typename T>
__device__ __forceinline__ T stag_coef(double v) {
    if (sizeof(T) == 8 && marked3(v)) v = __longlong_as_double(0x7ff8000000000000ll);
    return (T)v;
}
template <typename T>
__global__ void k_stag_coef(Layout L, const T* vel, const T* rho, const uint8_t* mp, const uint8_t* mvx,
                            const uint8_t* mvz, double dt, double inv_h, T* kp, T* bx, T* bz) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < L.N; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t x = i % L.nx, z = i / L.nx;
        int64_t q = L.idx(x, 0, z);
        double r0 = rho ? (double)rho[i] : 1.0;
        double c = (double)vel[i];
        kp[q] = mp[q] ? stag_coef<T>(dt * r0 * c * c * inv_h) : (T)0;
        double rx = (rho && x + 1 < L.nx) ? (double)rho[i + 1] : r0;
        double rz = (rho && z + 1 < L.nz) ? (double)rho[i + L.nx] : r0;
        bx[q] = mvx[q] ? stag_coef<T>(dt * 0.5 * (1.0 / r0 + 1.0 / rx) * inv_h) : (T)0;
        bz[q] = mvz[q] ? stag_coef<T>(dt * 0.5 * (1.0 / r0 + 1.0 / rz) * inv_h) : (T)0;
    }
}

template <typename T>
__global__ void k_interp_setup(int n, const double* xyz, int ndim, double inv_h, Layout L, const uint8_t* mask,
                               double scale, int64_t* idx, T* w) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int64_t b[3] = {0, 0, 0};
        double fr[3] = {0, 0, 0};
        int64_t nn[3] = {L.nx, ndim == 3 ? L.ny : L.nz, L.nz};
        for (int a = 0; a < ndim; ++a) {
            double xi = xyz[(int64_t)i * ndim + a] * inv_h;
            b[a] = (int64_t)floor(xi);
            fr[a] = xi - (double)b[a];
        }
        for (int c = 0; c < 8; ++c) {
            double wt = 0.0;
            int64_t q = L.base;
            if (c < (1 << ndim)) {
                wt = 1.0;
                int64_t node[3] = {0, 0, 0};
                bool in = true;
                for (int a = 0; a < ndim; ++a) {
                    int bit = (c >> a) & 1;
                    node[a] = b[a] + bit;
                    wt *= bit ? fr[a] : 1.0 - fr[a];
                    if (node[a] < 0 || node[a] >= nn[a]) in = false;
                }
                if (in) {
                    q = ndim == 3 ? L.idx(node[0], node[1], node[2]) : L.idx(node[0], 0, node[1]);
                    if (mask && !mask[q]) wt = 0.0;
                } else {
                    wt = 0.0;
                }
                if (wt == 0.0) q = L.base;
            }
            idx[8 * (int64_t)i + c] = q;
            w[8 * (int64_t)i + c] = (T)(wt * scale);
        }
    }
}

// ---------------------------------------------------------------------------
// stability checks
//   - every forward / adjoint run ends with a pass over its final fields; a
//     NaN or Inf sets bit 0 of a per-device status word that ib_sync_status
//     reports as IB_ERR_UNSTABLE (a non-finite value never leaves the leapfrog
//     or staggered recursion once it appears, so the final fields suffice);
//   - ib_stability runs the step kernels source-free from a random state and
//     renormalises every STAB_BLOCK steps: a power iteration on the one-step
//     map whose per-step growth estimates its spectral radius.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_check_finite(int64_t n, const T* __restrict__ a, const T* __restrict__ b,
                               const T* __restrict__ c) {
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        bad |= !isfinite(a[i]);
        if (b) bad |= !isfinite(b[i]);
        if (c) bad |= !isfinite(c[i]);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&g_dev_status, STATUS_UNSTABLE);
}

// SplitMix64 output function (Steele, Lea & Flood, "Fast splittable
// pseudorandom number generators", 2014) as a counter-based generator
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// f[i] = f2[i] = uniform(-1, 1) where coef[i] != 0 (interior nodes), else 0
template <typename T>
__global__ void k_rand_fill(int64_t n, const T* __restrict__ coef, uint64_t seed, T* f, T* f2) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T v = (T)0;
        if (coef[i] != (T)0) v = (T)((double)(splitmix64(seed * 0x632be59bd9b4e019ull + (uint64_t)i) >> 11) *
                                         (2.0 / 9007199254740992.0) - 1.0);
        f[i] = v;
        if (f2) f2[i] = v;
    }
}

// *out += sum of squares of a, b, c (nullable)
template <typename T>
__global__ void k_sumsq(int64_t n, const T* __restrict__ a, const T* __restrict__ b, const T* __restrict__ c,
                        double* out) {
    __shared__ double part[32];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double x = (double)a[i];
        s += x * x;
        if (b) {
            x = (double)b[i];
            s += x * x;
        }
        if (c) {
            x = (double)c[i];
            s += x * x;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        atomicAdd(out, t);
    }
}

// divide a, b, c by sqrt(*sumsq); *logn = log sqrt(*sumsq)
template <typename T>
__global__ void k_rescale(int64_t n, T* a, T* b, T* c, const double* sumsq, double* logn) {
    const double nrm = sqrt(*sumsq);
    const T inv = (T)(nrm > 0.0 ? 1.0 / nrm : 0.0);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        a[i] *= inv;
        if (b) b[i] *= inv;
        if (c) c[i] *= inv;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *logn = log(nrm);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int grid1(int64_t n, int bs) {
    int64_t g = (n + bs - 1) / bs;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 32));
}

struct Scratch {
    cudaStream_t s;
    std::vector<void*> ptrs;
    explicit Scratch(cudaStream_t st) : s(st) {}
    ~Scratch() {
        for (void* p : ptrs) cudaFreeAsync(p, s);
    }
    template <class T>
    ib_status alloc(T** p, int64_t n, bool zero = false) {
        *p = nullptr;
        if (n <= 0) n = 1;
        IB_CUDA(cudaMallocAsync((void**)p, sizeof(T) * (size_t)n, s));
        ptrs.push_back(*p);
        if (zero) IB_CUDA(cudaMemsetAsync(*p, 0, sizeof(T) * (size_t)n, s));
        return IB_OK;
    }
};

// Zeroed fields: parts of one allocation that was sized for all of them, or (at = null)
// allocations of their own.
struct Fields {
    Scratch& S;
    unsigned char* at = nullptr;
    explicit Fields(Scratch& s) : S(s) {}
    static int64_t bytes(int64_t n, size_t es) { return (n * (int64_t)es + 255) & ~(int64_t)255; }
    ib_status reserve(int64_t b) { return S.alloc(&at, b, true); }
    template <class T>
    ib_status alloc(T** p, int64_t n) {
        if (!at) return S.alloc(p, n, true);
        *p = reinterpret_cast<T*>(at);
        at += bytes(n, sizeof(T));
        return IB_OK;
    }
};

// power-iteration probe of ib_stability: random start, renormalisation every
// STAB_BLOCK steps into slot k of the device arrays sums / logs
static const int STAB_BLOCK = 50;
struct Probe {
    uint64_t seed;
    int nslot;          // nt / STAB_BLOCK + 1 (slot 0: the initial norm)
    double* sums;       // [nslot], zeroed
    double* logs;       // [nslot]
};

// renormalise the state (a, b, c) by its norm
template <typename T>
static ib_status probe_rescale(const Probe* pr, int slot, int64_t n, T* a, T* b, T* c, cudaStream_t s) {
    k_sumsq<T><<<grid1(n, 256), 256, 0, s>>>(n, a, b, c, pr->sums + slot);
    k_rescale<T><<<grid1(n, 256), 256, 0, s>>>(n, a, b, c, pr->sums + slot, pr->logs + slot);
    ib_count_launch("setup");
    ib_count_launch("setup");
    IB_CHECK_LAUNCH("stability probe");
    return IB_OK;
}

template <typename T>
static ib_status check_finite(int64_t n, const T* a, const T* b, const T* c, cudaStream_t s) {
    k_check_finite<T><<<grid1(n, 256), 256, 0, s>>>(n, a, b, c);
    IB_CHECK_LAUNCH("k_check_finite");
    ib_count_launch("setup");
    return IB_OK;
}

template <typename T>
static void stencil_weights(int M, T w2o[5], T c1o[4]) {
    std::vector<double> w2 = ib_central_second(M);
    std::vector<double> c1 = ib_staggered_first(M);
    int H = M / 2;
    for (int k = 0; k < 5; ++k) w2o[k] = k <= H ? (T)w2[H + k] : (T)0;
    for (int k = 0; k < 4; ++k) c1o[k] = k < H ? (T)c1[H + k] : (T)0;   // offset +(k + 1/2)
}

template <typename T>
static TileView<T> tview(const TileBins* b) {
    TileView<T> v;
    memset(&v, 0, sizeof v);
    if (!b || b->nent == 0) return v;
    v.ptr = b->ent_ptr;
    v.loc = b->ent_loc;
    v.src = b->ent_src;
    v.w = (const T*)(sizeof(T) == 8 ? (const void*)b->ent_w64 : (const void*)b->ent_w32);
    v.ntx = b->ntx;
    return v;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no libcuda link)
static PFN_cuTensorMapEncodeTiled_v12000 tma_encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        cudaDriverEntryPointQueryResult q;
        void* f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)f;
    }
    return fn;
}

static bool tma_enabled() {
    const char* e = getenv("IB_NO_TMA");
    return tma_encode_fn() != nullptr && !(e && e[0] == '1');
}

// 2D view of a padded FP32 3D field: rows of px elements; box (tw + 8) x (8 + 2H)
// (a plane of a tile tw wide with its halo) or, with tile_only, tw x 8 (a tile
// without halo)
static ib_status make_plane_map(CUtensorMap& tm, void* base, const Layout& L, bool tile_only = false,
                                uint32_t tw = 32) {
    cuuint64_t dims[2] = {(cuuint64_t)L.px, (cuuint64_t)(L.total / L.px)};
    cuuint64_t strides[1] = {(cuuint64_t)L.px * 4};
    cuuint32_t box[2] = {tile_only ? tw : tw + 8u, tile_only ? 8u : (cuuint32_t)(8 + 2 * L.H)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = tma_encode_fn()(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr,
                                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        ib_set_error("cuTensorMapEncodeTiled failed");
        return IB_ERR_CUDA;
    }
    return IB_OK;
}

static bool shot_damped(const ib_shot* sh) { return sh->damp_width > 0 && sh->damp_eta > 0.0; }

static ib_status check_shot(const ib_table* t, const ib_shot* sh, int precision, double dt, int nt,
                            bool need_traces = true) {
    if (!t || !sh) {
        ib_set_error("null table or shot");
        return IB_ERR_ARG;
    }
    if (precision != 32 && precision != 64) {
        ib_set_error("precision must be 32 or 64");
        return IB_ERR_ARG;
    }
    if (!(dt > 0.0) || nt < 1) {
        ib_set_error("dt must be positive and nt >= 1");
        return IB_ERR_ARG;
    }
    if (!sh->vel_dev || sh->nsrc < 0 || sh->nrec < 0 || (sh->nsrc && (!sh->src_dev || !sh->wavelet_dev)) ||
        (sh->nrec && (!sh->rec_dev || (need_traces && !sh->traces_dev)))) {
        ib_set_error("missing shot arrays");
        return IB_ERR_ARG;
    }
    if (!(sh->damp_eta >= 0.0) || sh->damp_width < 0 ||
        (shot_damped(sh) && 2 * (int64_t)sh->damp_width >= t->grid.n[0])) {
        ib_set_error("absorbing layer: damp_eta >= 0 and 0 <= damp_width < nx / 2 required");
        return IB_ERR_ARG;
    }
    if (sh->nsrc > 32) {
        // the 3D second-order and the two-step kernels spread each source over its 8
        // interpolation corners with one thread per corner of a 256-thread block
        ib_set_error("at most 32 sources per shot");
        return IB_ERR_ARG;
    }
    return IB_OK;
}

template <typename T>
struct Geom {
    PointSet<T> src, rec;
};

// absorbing layer of a shot: width and a_max = eta_max dt / 2 (formed in FP64)
template <typename T>
static void set_damping(const ib_shot* sh, double dt, int& dw, T& da) {
    dw = shot_damped(sh) ? sh->damp_width : 0;
    da = dw ? (T)(0.5 * sh->damp_eta * dt) : (T)0;
}

template <typename T>
static ib_status setup_points(const ib_table* t, const ib_shot* sh, double scale, Scratch& S, Geom<T>& g) {
    const Layout& L = t->L;
    int d = t->grid.ndim;
    int64_t* si;
    T* sw;
    int64_t* ri;
    T* rw;
    TRY(S.alloc(&si, 8 * std::max(sh->nsrc, 1)));
    TRY(S.alloc(&sw, 8 * std::max(sh->nsrc, 1)));
    TRY(S.alloc(&ri, 8 * std::max(sh->nrec, 1)));
    TRY(S.alloc(&rw, 8 * std::max(sh->nrec, 1)));
    if (sh->nsrc) {
        k_interp_setup<T><<<grid1(sh->nsrc, 64), 64, 0, S.s>>>(sh->nsrc, sh->src_dev, d, 1.0 / t->grid.h, L,
                                                                t->mask_pad[0], scale, si, sw);
        ib_count_launch("setup");
    }
    if (sh->nrec) {
        k_interp_setup<T><<<grid1(sh->nrec, 64), 64, 0, S.s>>>(sh->nrec, sh->rec_dev, d, 1.0 / t->grid.h, L,
                                                                t->mask_pad[0], 1.0, ri, rw);
        ib_count_launch("setup");
    }
    IB_CHECK_LAUNCH("k_interp_setup");
    g.src = {sh->nsrc, si, sw};
    g.rec = {sh->nrec, ri, rw};
    return IB_OK;
}

// checkpoint slot k holds (p^{c_k}, p^{c_k - 1}), c_k = k * seg
static int64_t ckpt_seg(int nt, int n_ckpt) { return (nt + n_ckpt - 1) / n_ckpt; }

extern "C" int64_t ib_checkpoint_bytes(const ib_table* t, int32_t precision, int32_t nt, int32_t n_ckpt) {
    if (!t || n_ckpt < 1 || nt < 1) return 0;
    int64_t es = precision == 64 ? 8 : 4;
    return (int64_t)n_ckpt * 2 * t->L.total * es;
}

// Shapes of the 2D steps: vx columns a thread; rz rows (burst) or a march of zc rows.  The rules
// below take 0, 1, 3 and marches of 4-16 rows; the others are there for IB_BATCH_SHAPE.
struct LeapShape {
    int vx, rz, zc;
};
static const int kNumShapes = 10;
static const LeapShape kShapes[kNumShapes] = {{1, 1, 0},  {2, 2, 0},  {2, 4, 0},  {4, 2, 0},  {4, 0, 16},
                                              {4, 0, 24}, {4, 0, 32}, {4, 0, 48}, {4, 0, 64}, {4, 0, 128}};
static int64_t shape_ntx(const LeapShape& p, const Layout& L) { return (L.nx + 32 * p.vx - 1) / (32 * p.vx); }
static int64_t shape_blocks(const LeapShape& p, const Layout& L) {
    const int64_t rows = (int64_t)LEAP_WARPS * (p.rz ? p.rz : p.zc);
    return shape_ntx(p, L) * ((L.nz + rows - 1) / rows);
}

static int64_t row_blocks(int64_t rows, int rz) {
    const int64_t per = rz ? RowsPer<1>::N : RowsPer<0>::N;
    return (rows + per - 1) / per;
}

// IB_STRIP=0 / 1 forces bursts / marches (one FP32 shot and both adjoints); -1: not set
static int strip_switch() {
    const char* e = getenv("IB_STRIP");
    return e && *e ? e[0] != '0' : -1;
}
// Rows a warp marches, for `points` grid points in one launch: few rows make many short marches,
// which fill the SMs and end together; a march's first step reads its 2H halo rows again, so long
// ones move less.  The even count next to 3.2 sqrt(points / 10^6), 4 to 16; us per step, order 8:
//   10^6 points, one shot  4.2   6.0   7.5  10.5  12.0  18.0  33.6   batch  3.0   5.5   8.3  13.3  28.9
//   4 rows                                                                 21.5  33.4  53.7  80.7   162
//   6 rows                16.4  20.5  26.5  36.9  41.3  57.6  98.5         22.2  32.8  52.2  74.4   147
//   8 rows                18.3  20.8  24.4  35.0  39.0  54.1  92.5         24.0  33.2  51.4  71.9   140
//   12 rows               22.3  22.9  26.6  33.1  37.3  51.2  88.3         27.5  36.7  53.0  73.4   136
//   16 rows               26.9  28.8  30.5  35.0  37.4  51.9  88.0         31.8  39.9  55.7  77.3   138
//   24 rows               35.7  37.8  38.8  43.1  44.4  53.4  88.6         42.5  48.1  63.9  83.2   142
static int march_rows(int64_t points) {
    const int r = 2 * (int)lrint(1.6 * sqrt(1e-6 * (double)points));
    return std::min(std::max(r, 4), 16);
}
// Shape of a step over `points` grid points in one launch, for half-order H.  A small grid needs many threads
// with little to do, a large one few instructions a point.  us per step, order 8, damped, set-up
// included (a launch takes the host about 7):
//   10^6 points        0.16   0.42   0.79   2.1    4.2    7.5   16.8   33.6
//   burst 1 x 1         7.2    9.3   12.3   23.9   43.6   79.3   178    358
//   burst 2 x 2         7.1    7.2    9.2   15.7   25.2   48.5   109    219
//   burst 4 x 2         7.2    9.0    9.2   13.6   21.0   40.3    91    182
// The march, at the rows above, passes the burst of 4 x 2 the earlier the wider the stencil, whose
// rows a burst reads again for every two it writes (us per step, burst and march; the
// strips and tiles before them took 31 at 6.0 x 10^6 points of order 2 and 42 at 5.5 x 10^6 of order 8):
//   order 8   2.2: 12.5, 14.3   3.0: 24.9, 21.5 (batch)   4.2: 18.4, 16.4   5.5: 43.7, 32.8 (batch)
//   order 4   3.0: 17.4, 18.6   4.1: 23.0, 22.5   5.5: 28.8, 27.1   6.6: 39.2, 32.2 (batches)
//   order 2   4.2: 12.1, 14.2   6.0: 14.9, 16.5   6.8: 17.9, 16.6   10.5: 32.9, 29.9
static LeapShape leap_shape(int64_t points, int H) {
    static const int64_t march_from[4] = {6600000, 4500000, 3600000, 3000000};
    if (points >= march_from[H - 1]) return {4, 0, march_rows(points)};
    return kShapes[points >= 1200000 ? 3 : points >= 150000 ? 1 : 0];
}
static LeapShape leap_shape_shot(const Layout& L, int H) {
    const int f = strip_switch();
    if (f < 0) return leap_shape(L.nx * L.nz, H);
    return f ? LeapShape{4, 0, march_rows(L.nx * L.nz)} : kShapes[1];
}

template <typename T>
static RowList<T> row_list(const IbOp& op) {
    return {op.nrows, op.row_pad, op.row_ptr, op.col_code,
            (const T*)(sizeof(T) == 8 ? (const void*)op.w64 : (const void*)op.w32)};
}

// calls f(H as a constant, shape's VX and RZ as constants)
template <int VX, int RZ, class F>
static void with_h(int H, F f) {
    std::integral_constant<int, VX> vx;
    std::integral_constant<int, RZ> rz;
    if (H == 1) f(std::integral_constant<int, 1>(), vx, rz);
    else if (H == 2) f(std::integral_constant<int, 2>(), vx, rz);
    else if (H == 3) f(std::integral_constant<int, 3>(), vx, rz);
    else f(std::integral_constant<int, 4>(), vx, rz);
}
template <class F>
static void with_shape(const LeapShape& p, int H, F f) {
    if (p.rz == 1) with_h<1, 1>(H, f);
    else if (p.vx == 2 && p.rz == 2) with_h<2, 2>(H, f);
    else if (p.vx == 2 && p.rz == 4) with_h<2, 4>(H, f);
    else if (p.rz == 2) with_h<4, 2>(H, f);
    else with_h<4, 0>(H, f);
}

// one step of one shot; a.nrb and a.ntx are set here
static void launch_leap2d(StepArgs<float>& a, const LeapShape& p, int H, cudaStream_t s) {
    a.nrb = row_blocks(a.rows.n, p.rz);
    a.ntx = shape_ntx(p, a.L);
    const unsigned grid = (unsigned)(a.nrb + shape_blocks(p, a.L));
    PROF_LAUNCH(p.rz ? "leap2d_f32" : "leap2d_strip_f32", s, {
        with_shape(p, H, [&](auto h, auto vx, auto rz) {
            constexpr size_t sm = leap_smem<h.value, rz.value>();
            if (sm > 48 * 1024)
                cudaFuncSetAttribute(k_leap2d<float, h.value, vx.value, rz.value>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sm);
            k_leap2d<float, h.value, vx.value, rz.value><<<grid, LEAP_THREADS, sm, s>>>(a, p.zc);
        });
    });
}
static void launch_leap2d(StepArgs<double>& a, const LeapShape&, int H, cudaStream_t s) {
    const LeapShape& p = kShapes[0];
    a.nrb = row_blocks(a.rows.n, p.rz);
    a.ntx = shape_ntx(p, a.L);
    const unsigned grid = (unsigned)(a.nrb + shape_blocks(p, a.L));
    PROF_LAUNCH("leap2d_f64", s, {
        with_h<1, 1>(H, [&](auto h, auto, auto) { k_leap2d<double, h.value, 1, 1><<<grid, LEAP_THREADS, 0, s>>>(a, 0); });
    });
}
// the absorbing layer's factor at every node (null without a layer)
template <typename T>
static ib_status damp_field(const Layout& L, int dw, T da, bool adjoint, Fields& F, const T** out) {
    *out = nullptr;
    if (!dw) return IB_OK;
    T* f;
    TRY(F.alloc(&f, L.total));
    k_damp_field<T><<<grid1(L.N, 256), 256, 0, F.S.s>>>(L, dw, da, adjoint, f);
    IB_CHECK_LAUNCH("k_damp_field");
    ib_count_launch("setup");
    *out = f;
    return IB_OK;
}
// Small grids: all steps between two checkpoints in one cooperative launch (k_leap2d_run), if
// one block per SM can hold the grid with 1 or 4 points a thread (about 430 000 points;
// with 16, for twice that, a step took 13.9 us at 1013 x 777 against 9.2 us launch by launch).
// us per step in one launch and launch by launch, FP32 order 8: 201 x 201 3.5 and 7.2, 400 x 400
// 4.4 and 7.1, 700 x 600 5.4 and 7.2; FP64 order 4, 201 x 201: 3.9, and 12.4 on the tiles before.
struct RunPlan {
    int vx, rz, cw;
    int64_t blocks;          // 0: the grid does not fit
};
template <typename T>
static RunPlan run_plan(const Layout& L, int H) {
    int dev = 0, sms = 0, coop = 0;
    RunPlan none = {0, 0, 0, 0};
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
        return none;
    const int shapes[2][2] = {{1, 1}, {2, 2}};
    const int threads[2] = {sizeof(T) == 8 ? (H <= 2 ? 1024 : 512) : 1024, 768};
    for (int i = 0; i < (sizeof(T) == 8 ? 1 : 2); ++i) {
        const int vx = shapes[i][0], rz = shapes[i][1], most = threads[i] / 32 - RUN_RW;
        const int64_t ntx = (L.nx + 32 * vx - 1) / (32 * vx);
        if (ntx > sms) continue;
        const int64_t cw = (L.nz + (sms / ntx) * rz - 1) / ((sms / ntx) * rz);
        if (cw <= most) return {vx, rz, (int)cw, ntx * ((L.nz + cw * rz - 1) / (cw * rz))};
    }
    return none;
}
// the plan of a forward or of a recomputation (IB_STRIP asks for launch by launch)
template <typename T>
static RunPlan run_plan_unless_forced(const Layout& L, int H) {
    return strip_switch() < 0 ? run_plan<T>(L, H) : RunPlan{0, 0, 0, 0};
}
template <typename T, int H, int VX, int RZ>
static cudaError_t launch_run_shape(RunArgs<T>& r, const RunPlan& p, cudaStream_t s) {
    const int threads = 32 * (p.cw + RUN_RW);
    const size_t sm = sizeof(RunRow<T>) * RUN_ROWS + (sizeof(T) + sizeof(int)) * RUN_ENT + sizeof(T) * 2 * VX * RZ * threads;
    cudaError_t e = cudaFuncSetAttribute(k_leap2d_run<T, H, VX, RZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    r.cw = p.cw;
    r.a.ntx = (r.a.L.nx + 32 * VX - 1) / (32 * VX);
    void* args[] = {&r};
    const char* coop = getenv("IB_COOP");   // IB_COOP=0: the answer where too few SMs are usable
    if (coop && coop[0] == '0') return cudaErrorCooperativeLaunchTooLarge;
    return cudaLaunchCooperativeKernel((const void*)k_leap2d_run<T, H, VX, RZ>, dim3((unsigned)p.blocks), dim3(threads), args,
                                       sm, s);
}
template <typename T, int H>
static cudaError_t launch_run_h(RunArgs<T>& r, const RunPlan& p, cudaStream_t s) {
    if (p.vx == 1) return launch_run_shape<T, H, 1, 1>(r, p, s);
    if constexpr (sizeof(T) == 4) {
        if (p.vx == 2) return launch_run_shape<T, H, 2, 2>(r, p, s);
    }
    return cudaErrorInvalidValue;
}
// Steps n0 .. n1 - 1; bar: a zeroed word of this launch; err: a zeroed word of the call, or null.  *refused: the device (or the part of
// it that this context may use) cannot hold all blocks at once, nothing was launched, and the
// caller takes the steps launch by launch.
template <typename T>
static ib_status launch_run(const StepArgs<T>& a, const RunPlan& p, int H, T* buf0, T* buf1, int64_t stride, int n0, int n1,
                            unsigned* bar, int* err, bool* refused, cudaStream_t s) {
    RunArgs<T> r;
    memset(&r, 0, sizeof r);
    r.a = a;
    r.buf0 = buf0;
    r.buf1 = buf1;
    r.stride = stride;
    r.n0 = n0;
    r.n1 = n1;
    r.bar = bar;
    r.err = err;
    cudaError_t e = cudaSuccess;
    PROF_LAUNCH(kname<T>("leap2d_run_f32", "leap2d_run_f64"), s, {
        if (H == 1) e = launch_run_h<T, 1>(r, p, s);
        else if (H == 2) e = launch_run_h<T, 2>(r, p, s);
        else if (H == 3) e = launch_run_h<T, 3>(r, p, s);
        else e = launch_run_h<T, 4>(r, p, s);
    });
    *refused = e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported || e == cudaErrorLaunchOutOfResources;
    if (*refused) {
        cudaGetLastError();
        return IB_OK;
    }
    if (e != cudaSuccess) return ib_cuda_fail(e, "k_leap2d_run", __FILE__, __LINE__);
    return IB_OK;
}

template <typename T>
static ib_status mark_rows(const RowList<T>& r, T* Kh, cudaStream_t s) {
    if (r.n == 0) return IB_OK;
    k_mark_rows<T><<<grid1(r.n, 256), 256, 0, s>>>(r.n, r.pad, Kh);
    IB_CHECK_LAUNCH("k_mark_rows");
    ib_count_launch("setup");
    return IB_OK;
}

// ---------------------------------------------------------------------------
// Temporal blocking: two leapfrog steps per launch (2D, second order, FP32).
//
// A block owns a TX x TZ output tile.  It stages p^n on the tile grown by 2R
// ("region 2"), computes p^{n+1} on the tile grown by R ("region 1": standard
// stencil, the immersed-boundary rows that lie there, source, absorbing
// layer) and keeps it in shared memory, then computes p^{n+2} on the tile from
// it.  R >= M/2 and R >= the reach of every correction row, so both steps read
// shared memory only.  The ring of region 1 outside the tile is computed by the
// neighbouring blocks as well: 2 x (1 + 2R/TX)(1 + 2R/TZ)/2 stencils per point
// and step instead of 1, for DRAM traffic of p^n, p^{n-1}, K read and p^{n+1},
// p^{n+2} written per two steps (20 bytes per point, 10 per point and step,
// against 16 for one step per launch).  Outputs go to two further buffers:
// the neighbours still read p^n and p^{n-1} in their halos.
//
// Correction entries of a tile: every row in region 1, those inside the tile
// first (used by both steps), one int32 code per entry -- the row's position
// in region 1 (x, z: 8 bits each) and the column offset (dx, dz: int8 each) --
// and the FP32 weight.
// ---------------------------------------------------------------------------
struct TbArgs {
    Layout L;
    float w2[5];
    const float* pn;         // p^n
    const float* pm;         // p^{n-1}
    const float* Kh;
    float* out1;             // p^{n+1}
    float* out2;             // p^{n+2}
    const int32_t* ent_ptr;  // [2 ntiles + 1]: tile t has rows [2t, 2t+1) in the tile, [2t+1, 2t+2) in its ring
    const int32_t* ent_code;
    const float* ent_w;
    PointSet<float> src;
    const float* wavelet;
    int step;                // n (the launch advances n -> n + 2)
    PointSet<float> rec;
    float* traces;
    int nt;
    int dw;
    float da;
};

__device__ __forceinline__ void tb_decode(int32_t c, int& lx, int& lz, int& dx, int& dz) {
    lx = c & 0xff;
    lz = (c >> 8) & 0xff;
    dx = (int)(int8_t)((c >> 16) & 0xff);
    dz = (int)(int8_t)((c >> 24) & 0xff);
}

// dst[loc(e)] += w[e] * f[col(e)] for the entries [e0, e1): four chunks of 32
// entries in flight per warp, segmented warp sums (entries of a row are
// contiguous), one shared-memory atomic per row segment
template <class LocCol>
__device__ __forceinline__ void tb_entries(const TbArgs& a, int32_t e0, int32_t e1, LocCol lc, const float* f,
                                           float* dst, int tid) {
    constexpr int U = 4;
    const int lane = tid & 31;
    for (int32_t base = e0 + (tid & ~31) * U; base < e1; base += 256 * U) {
        int32_t loc[U];
        float val[U];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int32_t e = base + u * 32 + lane;
            ok[u] = e < e1;
            int l = -1 - lane, col = 0;
            if (ok[u]) lc(a.ent_code[e], l, col);
            loc[u] = l;
            val[u] = ok[u] ? a.ent_w[e] * f[col] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) seg_add(dst, loc[u], val[u], ok[u], lane);
    }
}

// dst[(z - zr) W + (x - xr)] += w wv for the source corners in the W x Z box at
// (xr, zr) that are nodes of the model (corners in the zero padding are dropped,
// as the one-step kernels drop them)
__device__ __forceinline__ void tb_sources(const PointSet<float>& src, float wv, const Layout& L, int64_t xr,
                                           int64_t zr, int W, int Z, float* dst, int tid) {
    if (tid >= 8 * src.n) return;
    const float w = src.w[tid];
    if (w == 0.f) return;
    const int64_t rel = src.idx[tid] - L.base;
    const int64_t z = rel >= 0 ? rel / L.px : -((-rel + L.px - 1) / L.px);
    const int64_t x = rel - z * L.px;
    if (x >= L.nx || z < 0 || z >= L.nz) return;
    const int64_t lx = x - xr, lz = z - zr;
    if (lx >= 0 && lx < W && lz >= 0 && lz < Z) atomicAdd(&dst[lz * W + lx], w * wv);
}

template <int R, int TX, int TZ>
struct TbShape {
    static constexpr int W1 = TX + 2 * R, Z1 = TZ + 2 * R, W2 = TX + 4 * R, Z2 = TZ + 4 * R;
    static constexpr size_t smem = sizeof(float) * ((size_t)W2 * Z2 + 2 * (size_t)W1 * Z1);
    static_assert(W1 <= 256 && Z1 <= 256, "region-1 positions take 8 bits per axis");
    static_assert((TX * TZ) % 256 == 0, "whole tile points per thread");
};

template <int H, int R, int TX, int TZ>
__global__ void __launch_bounds__(256) k_leap2d_tb2(TbArgs a) {
    using S = TbShape<R, TX, TZ>;
    constexpr int W1 = S::W1, Z1 = S::Z1, W2 = S::W2, Z2 = S::Z2;
    extern __shared__ float tb_sm[];
    float* P0 = tb_sm;             // p^n on region 2
    float* P1 = P0 + W2 * Z2;      // p^{n+1} on region 1
    float* A = P1 + W1 * Z1;       // accumulator (region 1, then the tile)
    const int tid = threadIdx.x;
    const Layout& L = a.L;
    const int64_t x0 = (int64_t)blockIdx.x * TX, z0 = (int64_t)blockIdx.y * TZ;
    const int64_t tile = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
    // trace columns n - 1 (p^n) and n - 2 (p^{n-1}): both inputs of this launch
    {
        const int64_t gid = tile * 256 + tid, stride = launch_threads();
        record_receivers(a.rec, a.pn, a.traces, a.nt, a.step - 1, gid, stride);
        record_receivers(a.rec, a.pm, a.traces, a.nt, a.step - 2, gid, stride);
    }
    for (int i = tid; i < W2 * Z2; i += 256) {
        const int lz = i / W2, lx = i - lz * W2;
        const int64_t x = x0 + lx - 2 * R, z = z0 + lz - 2 * R;
        const bool ok = x >= 0 && x < L.nx && z >= 0 && z < L.nz;
        cp_async<4>(&P0[i], ok ? a.pn + L.base + z * L.px + x : a.pn, ok);
    }
    cp_async_commit();
    const int32_t e0 = a.ent_ptr[2 * tile], em = a.ent_ptr[2 * tile + 1], e1 = a.ent_ptr[2 * tile + 2];
    cp_async_wait_all();
    __syncthreads();
    // ---- step n -> n + 1 on region 1
    for (int i = tid; i < W1 * Z1; i += 256) {
        const int lz = i / W1, lx = i - lz * W1;
        const float* q = P0 + (lz + R) * W2 + lx + R;
        const float c = q[0];
        float s = 0.f;
#pragma unroll
        for (int k = 1; k <= H; ++k)
            s += a.w2[k] * (((q[k] - c) + (q[-k] - c)) + ((q[k * W2] - c) + (q[-k * W2] - c)));
        A[i] = s;
    }
    __syncthreads();
    if (e1 > e0)
        tb_entries(
            a, e0, e1,
            [](int32_t code, int& loc, int& col) {
                int lx, lz, dx, dz;
                tb_decode(code, lx, lz, dx, dz);
                loc = lz * W1 + lx;
                col = (lz + R + dz) * W2 + lx + R + dx;
            },
            P0, A, tid);
    __syncthreads();
    // update (A keeps p^{n-1} for the absorbing layer), then the source
    for (int i = tid; i < W1 * Z1; i += 256) {
        const int lz = i / W1, lx = i - lz * W1;
        const int64_t x = x0 + lx - R, z = z0 + lz - R;
        float u = 0.f, pmv = 0.f;
        if (x >= 0 && x < L.nx && z >= 0 && z < L.nz) {
            const int64_t q = L.base + z * L.px + x;
            const float c = P0[(lz + R) * W2 + lx + R];
            pmv = a.pm[q];
            u = c + ((c - pmv) + a.Kh[q] * A[i]);
        }
        P1[i] = u;
        A[i] = pmv;
    }
    __syncthreads();
    if (a.src.n) {
        tb_sources(a.src, a.wavelet[a.step], L, x0 - R, z0 - R, W1, Z1, P1, tid);
        __syncthreads();
    }
    if (damp_box(L, a.dw, x0 - R, x0 + TX - 1 + R, 0, 0, z0 + TZ - 1 + R)) {
        for (int i = tid; i < W1 * Z1; i += 256) {
            const int lz = i / W1, lx = i - lz * W1;
            const int64_t x = x0 + lx - R, z = z0 + lz - R;
            if (x >= 0 && x < L.nx && z >= 0 && z < L.nz)
                P1[i] -= damp_g<float>(L, a.dw, a.da, x, 0, z) * (P1[i] - A[i]);
        }
    }
    __syncthreads();
    // ---- step n + 1 -> n + 2 on the tile
    constexpr int PT = TX * TZ / 256;
#pragma unroll
    for (int j = 0; j < PT; ++j) {
        const int i = tid + 256 * j, lz = i / TX, lx = i - lz * TX;
        const float* q = P1 + (lz + R) * W1 + lx + R;
        const float c = q[0];
        float s = 0.f;
#pragma unroll
        for (int k = 1; k <= H; ++k)
            s += a.w2[k] * (((q[k] - c) + (q[-k] - c)) + ((q[k * W1] - c) + (q[-k * W1] - c)));
        A[i] = s;
    }
    __syncthreads();
    if (em > e0)
        tb_entries(
            a, e0, em,
            [](int32_t code, int& loc, int& col) {
                int lx, lz, dx, dz;
                tb_decode(code, lx, lz, dx, dz);
                loc = (lz - R) * TX + lx - R;
                col = (lz + dz) * W1 + lx + dx;
            },
            P1, A, tid);
    __syncthreads();
    float uv[PT];
#pragma unroll
    for (int j = 0; j < PT; ++j) {
        const int i = tid + 256 * j, lz = i / TX, lx = i - lz * TX;
        const int64_t x = x0 + lx, z = z0 + lz;
        uv[j] = 0.f;
        if (x < L.nx && z < L.nz) {
            const int64_t q = L.base + z * L.px + x;
            const float c = P1[(lz + R) * W1 + lx + R];
            const float pmv = P0[(lz + 2 * R) * W2 + lx + 2 * R];
            uv[j] = c + ((c - pmv) + a.Kh[q] * A[i]);
            a.out1[q] = c;
        }
    }
    if (a.src.n) {
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PT; ++j) A[tid + 256 * j] = uv[j];
        __syncthreads();
        tb_sources(a.src, a.wavelet[a.step + 1], L, x0, z0, TX, TZ, A, tid);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PT; ++j) uv[j] = A[tid + 256 * j];
    }
    const bool damped = damp_box(L, a.dw, x0, x0 + TX - 1, 0, 0, z0 + TZ - 1);
#pragma unroll
    for (int j = 0; j < PT; ++j) {
        const int i = tid + 256 * j, lz = i / TX, lx = i - lz * TX;
        const int64_t x = x0 + lx, z = z0 + lz;
        if (x >= L.nx || z >= L.nz) continue;
        float u = uv[j];
        if (damped) {
            const float pmv = P0[(lz + 2 * R) * W2 + lx + 2 * R];
            u -= damp_g<float>(L, a.dw, a.da, x, 0, z) * (u - pmv);
        }
        a.out2[L.base + z * L.px + x] = u;
    }
}

static const int TBX = 64, TBZ = 32;

// Correction entries of the two-step kernel for region margin R, cached in the
// table's bins of operator 0 (key tx = TBX, ty = -R, tz = TBZ).  *ok = false
// when a correction reaches further than R (the one-step kernels run then).
static ib_status tb_bins(ib_table* t, int R, TileBins* out, bool* ok) {
    IbOp& op = t->ops[0];
    for (const TileBins& b : op.bins)
        if (b.tx == TBX && b.ty == -R && b.tz == TBZ) {
            *out = b;
            *ok = b.nent >= 0;
            return IB_OK;
        }
    const Layout& L = t->L;
    const int64_t nr = op.nrows, nnz = op.nnz;
    std::vector<int64_t> lin(nr), rp(nr + 1, 0);
    std::vector<int32_t> code(nnz);
    std::vector<float> w(nnz);
    if (nr) {
        IB_CUDA(cudaMemcpy(lin.data(), op.row_lin, 8 * nr, cudaMemcpyDeviceToHost));
        IB_CUDA(cudaMemcpy(rp.data(), op.row_ptr, 8 * (nr + 1), cudaMemcpyDeviceToHost));
    }
    if (nnz) {
        IB_CUDA(cudaMemcpy(code.data(), op.col_code, 4 * nnz, cudaMemcpyDeviceToHost));
        IB_CUDA(cudaMemcpy(w.data(), op.w32, 4 * nnz, cudaMemcpyDeviceToHost));
    }
    TileBins b;
    b.tx = TBX;
    b.ty = -R;
    b.tz = TBZ;
    b.ntx = (L.nx + TBX - 1) / TBX;
    b.nty = 1;
    const int64_t ntz = (L.nz + TBZ - 1) / TBZ;
    b.ntiles = b.ntx * ntz;
    bool fits = true;
    for (int64_t e = 0; e < nnz && fits; ++e) {
        int dx, dy, dz;
        unpack_off(code[e], dx, dy, dz);
        fits = std::abs(dx) <= R && std::abs(dy) <= R;
    }
    if (!fits) {   // remembered, so that the check runs once per table
        b.nent = -1;
        op.bins.push_back(b);
        *out = b;
        *ok = false;
        return IB_OK;
    }
    // visit (row, tile, in-tile?) for every tile whose region 1 holds the row
    auto each = [&](auto&& f) {
        for (int64_t r = 0; r < nr; ++r) {
            const int64_t x = lin[r] % L.nx, z = lin[r] / L.nx;
            for (int64_t bz = std::max<int64_t>(0, (z - R) / TBZ - 1); bz <= std::min(ntz - 1, (z + R) / TBZ); ++bz) {
                if (z < bz * TBZ - R || z > bz * TBZ + TBZ - 1 + R) continue;
                for (int64_t bx = std::max<int64_t>(0, (x - R) / TBX - 1); bx <= std::min(b.ntx - 1, (x + R) / TBX);
                     ++bx) {
                    if (x < bx * TBX - R || x > bx * TBX + TBX - 1 + R) continue;
                    const bool in = x >= bx * TBX && x < bx * TBX + TBX && z >= bz * TBZ && z < bz * TBZ + TBZ;
                    f(r, x, z, bx, bz, in);
                }
            }
        }
    };
    std::vector<int64_t> cnt(2 * b.ntiles, 0);
    each([&](int64_t r, int64_t, int64_t, int64_t bx, int64_t bz, bool in) {
        cnt[2 * (bz * b.ntx + bx) + (in ? 0 : 1)] += rp[r + 1] - rp[r];
    });
    std::vector<int32_t> ptr(2 * b.ntiles + 1, 0);
    int64_t tot = 0;
    for (int64_t i = 0; i < 2 * b.ntiles; ++i) {
        ptr[i] = (int32_t)tot;
        tot += cnt[i];
    }
    if (tot >= INT32_MAX) {
        ib_set_error("two-step correction list exceeds 2^31 entries");
        return IB_ERR_ARG;
    }
    ptr[2 * b.ntiles] = (int32_t)tot;
    std::vector<int32_t> ecode(std::max<int64_t>(tot, 1));
    std::vector<float> ew(std::max<int64_t>(tot, 1));
    std::vector<int64_t> cur(ptr.begin(), ptr.end() - 1);
    each([&](int64_t r, int64_t x, int64_t z, int64_t bx, int64_t bz, bool in) {
        const uint32_t lx = (uint32_t)(x - (bx * TBX - R)), lz = (uint32_t)(z - (bz * TBZ - R));
        int64_t& c = cur[2 * (bz * b.ntx + bx) + (in ? 0 : 1)];
        for (int64_t e = rp[r]; e < rp[r + 1]; ++e, ++c) {
            int dx, dy, dz;
            unpack_off(code[e], dx, dy, dz);
            ecode[c] = (int32_t)(lx | lz << 8 | (uint32_t)(dx & 0xff) << 16 | (uint32_t)(dy & 0xff) << 24);
            ew[c] = w[e];
        }
    });
    b.nent = tot;
    auto up = [](auto** d, const auto& v) -> ib_status {
        IB_CUDA(cudaMalloc((void**)d, sizeof(v[0]) * v.size()));
        IB_CUDA(cudaMemcpy(*d, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice));
        return IB_OK;
    };
    ib_status st = up(&b.ent_ptr, ptr);
    if (st == IB_OK) st = up(&b.ent_loc, ecode);
    if (st == IB_OK) st = up(&b.ent_w32, ew);
    // (legacy-stream copies, which a non-blocking stream's steps are not ordered after)
    if (st == IB_OK && cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) st = IB_ERR_CUDA;
    if (st != IB_OK) {
        ib_free_bins(b);
        return st;
    }
    op.bins.push_back(b);
    *out = b;
    *ok = true;
    return IB_OK;
}

// IB_TEMPORAL_BLOCK=0 / 1 turns the two-step kernel off / on
static bool tb_enabled() {
    const char* e = getenv("IB_TEMPORAL_BLOCK");
    return e && e[0] == '1';
}

template <int H, int R>
static void launch_tb2_hr(const TbArgs& a, dim3 grid, cudaStream_t s) {
    using Sh = TbShape<R, TBX, TBZ>;
    static const bool attr = (cudaFuncSetAttribute(k_leap2d_tb2<H, R, TBX, TBZ>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem),
                              true);
    (void)attr;
    k_leap2d_tb2<H, R, TBX, TBZ><<<grid, 256, Sh::smem, s>>>(a);
}
template <int R>
static void launch_tb2_r(const TbArgs& a, int H, dim3 grid, cudaStream_t s) {
    if (H == 1) launch_tb2_hr<1, R>(a, grid, s);
    else if (H == 2) launch_tb2_hr<2, R>(a, grid, s);
    else if (H == 3) launch_tb2_hr<3, R>(a, grid, s);
    else launch_tb2_hr<4, R>(a, grid, s);
}
// region margins the two-step kernel is built for (R >= M/2 and >= the reach)
static const int TB_MARGINS[2] = {4, 6};
static void launch_tb2(const TbArgs& a, int H, int R, dim3 grid, cudaStream_t s) {
    PROF_LAUNCH("leap2d_tb2_f32", s, {
        if (R == 4) launch_tb2_r<4>(a, H, grid, s);
        else launch_tb2_r<6>(a, H, grid, s);
    });
}

// Planes per block of the FP32 3D step on 64 x 8 column tiles.  A block costs its planes and
// about 10 more (the 2H planes read before the first, the ring's start, the tail); three run on
// an SM, so the launch takes ceil(blocks / (3 SMs)) such times, and half a one for the blocks
// that hold a source and take longer.  The even count that minimises it: 48 at 512^2 x 384 (us per
// step with its corrections: 32 planes 465, 48 planes 457, 64 planes 461), 10 at 131 x 97 x 110,
// where 32 planes left two thirds of the block slots empty and the others marching (51 us; 4
// planes 25, 10 planes 24, 16 planes 31); 30 at 500 x 73 x 300, whose 400 blocks of 60 planes
// waited for the two sources' blocks (86 us; 32 planes 80).
//   With the absorbing layer the blocks that reach it take about twice as long (a division a
// point), so the slots free up at different times instead of in rounds: blocks / (3 SMs) times
// the planes and 3.5 more (the fixed part is mostly hidden behind the other blocks of the SM), and
// half a block's whole time as the tail.  us per step with its corrections, order 8, layer of 20
// nodes, by this rule | by the rule without a layer | at 32 planes:
//   200 x 180 x 160   94 | 107 |  96      401 x 478 x 182  334 | 400 | 339
//   300 x 260 x 200  170 | 186 | 172      384 x 384 x 256  310 | 354 | 310
//   500 x  73 x 300  124 | 142 | 132      512 x 512 x 384  650 | 664 | 644
static int z_planes(const Layout& L, bool layer) {
    const int64_t tiles = ((L.nx + 63) / 64) * ((L.ny + 7) / 8), slots = 3 * (int64_t)ib_sm_count();
    int best = 32;
    double cost = INFINITY;
    for (int zc = 4; zc <= 96; zc += 2) {
        const int64_t blocks = tiles * ((L.nz + zc - 1) / zc);
        const double c = layer ? (double)blocks / (double)slots * (zc + 3.5) + 0.5 * (zc + 10)
                               : ((double)((blocks + slots - 1) / slots) + 0.5) * (zc + 10);
        if (c < cost) {
            cost = c;
            best = zc;
        }
    }
    return best;
}

template <typename T>
static ib_status forward_2nd(ib_table* t, const ib_shot* sh, double dt, int nt, void* ckpt, int n_ckpt,
                             cudaStream_t s, const Probe* probe = nullptr) {
    const Layout& L = t->L;
    const int d = t->grid.ndim;
    const int M = t->opts.space_order;
    const int H = M / 2;
    Scratch S(s);
    T *p0, *p1, *Kh;
    TRY(S.alloc(&p0, L.total, true));
    TRY(S.alloc(&p1, L.total, true));
    TRY(S.alloc(&Kh, L.total, true));
    k_leap_coef<T><<<grid1(L.N, 256), 256, 0, s>>>(L, (const T*)sh->vel_dev, t->mask_pad[0], dt / t->grid.h, Kh);
    IB_CHECK_LAUNCH("k_leap_coef");
    ib_count_launch("setup");
    if (probe) {   // p^0 = p^{-1} = random on interior nodes, normalised
        k_rand_fill<T><<<grid1(L.total, 256), 256, 0, s>>>(L.total, Kh, probe->seed, p0, p1);
        IB_CHECK_LAUNCH("k_rand_fill");
        TRY(probe_rescale<T>(probe, 0, L.total, p0, p1, (T*)nullptr, s));
    }
    Geom<T> g;
    TRY(setup_points<T>(t, sh, dt * dt / pow(t->grid.h, d), S, g));
    const TileBins* bins = nullptr;
    if (d == 3) TRY(ib_table_bins(t, 0, 32, 8, 1, &bins, s));
    StepArgs<T> a;
    memset(&a, 0, sizeof a);
    a.L = L;
    {
        T c1u[4];
        stencil_weights<T>(M, a.w2, c1u);
    }
    a.Kh = Kh;
    a.op = tview<T>(bins);
    a.rows = row_list<T>(t->ops[0]);
    a.src = g.src;
    a.wavelet = (const T*)sh->wavelet_dev;
    a.rec = g.rec;
    a.traces = (T*)sh->traces_dev;
    a.nt = nt;
    set_damping<T>(sh, dt, a.dw, a.da);
    const int64_t seg = ckpt ? ckpt_seg(nt, n_ckpt) : 0;
    T* cur = p0;   // p^n
    T* prev = p1;  // p^{n-1}
    const LeapShape shape = d == 2 ? leap_shape_shot(L, H) : kShapes[0];
    if (d == 2) {
        Fields F(S);
        TRY(damp_field<T>(L, a.dw, a.da, false, F, &a.damp));
    }
    // two steps per launch (FP32 2D; not with checkpoints or the stability probe)
    int tbR = 0;
    TileBins tbb;
    float *tb_o1 = nullptr, *tb_o2 = nullptr;
    if (d == 2 && sizeof(T) == 4 && !ckpt && !probe && nt >= 2 && tb_enabled()) {
        for (int R : TB_MARGINS) {
            if (R < H) continue;
            bool ok = false;
            TRY(tb_bins(t, R, &tbb, &ok));
            if (ok) {
                tbR = R;
                break;
            }
        }
        if (tbR) {
            TRY(S.alloc(&tb_o1, L.total, true));
            TRY(S.alloc(&tb_o2, L.total, true));
        }
    }
    // FP32 3D: TMA, where the table's entries have 16-bit codes
    const bool use_tma = d == 3 && sizeof(T) == 4 && tma_enabled() && (t->ops[0].nnz == 0 || t->ops[0].code16);
    // planes per 3D block (IB_ZCHUNK overrides it for tuning)
    int zchunk = use_tma ? z_planes(L, a.dw > 0) : 32;
    if (const char* e = getenv("IB_ZCHUNK")) zchunk = std::max(1, atoi(e));
    dim3 grid3((unsigned)((L.nx + 31) / 32), (unsigned)((L.ny + 7) / 8), (unsigned)((L.nz + zchunk - 1) / zchunk));
    const int64_t nty3 = (L.ny + 7) / 8;
    // FP32 3D: TMA-staged planes of p (with halo) and tiles of p_prev and K (one
    // tensor map of each kind per buffer), compact correction rows
    CUtensorMap tmap[2], tmtile[2], tmK;
    Rows3 rows3;
    memset(&rows3, 0, sizeof rows3);
    const uint16_t* code16 = nullptr;
    int* err = nullptr;
    // x-pair kernel (64 x 8 tiles; IB_TMA3_PAIRS=0 selects the 32 x 8 kernel)
    bool pairs = false;
    // correction pass: entries in flight per lane, 4 (IB_ADD3_U=8 selects 8: at
    // 512^2 x 384, order 8, 150 us per launch against 141 us with 4)
    int add3_u = 4;
    if (const char* e = getenv("IB_ADD3_U")) add3_u = atoi(e) == 8 ? 8 : 4;
    if (use_tma) {
        const char* fe = getenv("IB_FUSED3");
        const char* pe = getenv("IB_TMA3_PAIRS");
        pairs = !(fe && fe[0] == '1') && !(pe && pe[0] == '0');
        const uint32_t tw = pairs ? 64 : 32;
        TRY(make_plane_map(tmap[0], (void*)p0, L, false, tw));
        TRY(make_plane_map(tmap[1], (void*)p1, L, false, tw));
        TRY(make_plane_map(tmtile[0], (void*)p0, L, true, tw));
        TRY(make_plane_map(tmtile[1], (void*)p1, L, true, tw));
        TRY(make_plane_map(tmK, (void*)Kh, L, true, tw));
        TRY(S.alloc(&err, 1, true));
        // corrections: fused into the step kernel (IB_FUSED3=1) or added by k_ib_add3
        if (fe && fe[0] == '1') {
            if (bins && bins->nent > 0) {
                rows3.ptr = bins->ent_ptr;
                rows3.slot = bins->ent_slot;
                rows3.code = bins->ent_code;
                rows3.w = bins->ent_w32;
            }
        } else {
            code16 = t->ops[0].code16;
        }
    }
    int n0 = 0;
    if (tbR) {
        TbArgs ta;
        memset(&ta, 0, sizeof ta);
        ta.L = L;
        for (int k = 0; k < 5; ++k) ta.w2[k] = (float)a.w2[k];
        ta.Kh = (const float*)Kh;
        ta.ent_ptr = tbb.ent_ptr;
        ta.ent_code = tbb.ent_loc;
        ta.ent_w = tbb.ent_w32;
        ta.src = *reinterpret_cast<const PointSet<float>*>(&g.src);
        ta.wavelet = (const float*)sh->wavelet_dev;
        ta.rec = *reinterpret_cast<const PointSet<float>*>(&g.rec);
        ta.traces = (float*)sh->traces_dev;
        ta.nt = nt;
        ta.dw = a.dw;
        ta.da = (float)a.da;
        dim3 gtb((unsigned)((L.nx + TBX - 1) / TBX), (unsigned)((L.nz + TBZ - 1) / TBZ));
        float *pc = (float*)cur, *pp = (float*)prev;
        for (; n0 + 2 <= nt; n0 += 2) {
            ta.pn = pc;
            ta.pm = pp;
            ta.out1 = tb_o1;
            ta.out2 = tb_o2;
            ta.step = n0;
            launch_tb2(ta, H, tbR, gtb, s);
            IB_CHECK_LAUNCH("two-step leapfrog");
            // p^{n+1}, p^{n+2} become (prev, cur); the old pair takes the next outputs
            tb_o1 = pp;
            tb_o2 = pc;
            pp = ta.out1;
            pc = ta.out2;
        }
        cur = (T*)pc;
        prev = (T*)pp;
        if (g.rec.n) {   // trace column n - 2 (p^{n-1}): the launches recorded columns up to n - 3
            k_receivers<T><<<grid1(g.rec.n, 256), 256, 0, s>>>(g.rec, prev, (T*)sh->traces_dev, nt, n0 - 2);
            IB_CHECK_LAUNCH("k_receivers");
            ib_count_launch("setup");
        }
    }
    // (the two-step kernel reads the coefficients unmarked)
    if (d == 2) TRY(mark_rows<T>(a.rows, Kh, s));
    const RunPlan plan = d == 2 && !tb_enabled() ? run_plan_unless_forced<T>(L, H) : RunPlan{0, 0, 0, 0};
    if (plan.blocks) {
        // up to the next checkpoint (or renormalisation of the probe) in one launch
        const int64_t part = ckpt ? seg : probe ? STAB_BLOCK : nt;
        unsigned* bars;
        TRY(S.alloc(&bars, (nt + part - 1) / part, true));
        while (n0 < nt) {
            if (ckpt) {
                T* slot = (T*)ckpt + (n0 / seg) * 2 * L.total;
                IB_CUDA(cudaMemcpyAsync(slot, cur, sizeof(T) * L.total, cudaMemcpyDeviceToDevice, s));
                IB_CUDA(cudaMemcpyAsync(slot + L.total, prev, sizeof(T) * L.total, cudaMemcpyDeviceToDevice, s));
            }
            const int n1 = (int)std::min<int64_t>(n0 + part, nt);
            bool refused;
            TRY(launch_run<T>(a, plan, H, cur, prev, 0, n0, n1, bars + n0 / part, nullptr, &refused, s));
            if (refused) break;   // the loop below
            if ((n1 - n0) & 1) std::swap(cur, prev);
            if (probe && n1 % STAB_BLOCK == 0)
                TRY(probe_rescale<T>(probe, n1 / STAB_BLOCK, L.total, cur, prev, (T*)nullptr, s));
            n0 = n1;
        }
    }
    for (int n = n0; n < nt; ++n) {
        if (ckpt && n % seg == 0) {
            T* slot = (T*)ckpt + (int64_t)(n / seg) * 2 * L.total;
            IB_CUDA(cudaMemcpyAsync(slot, cur, sizeof(T) * L.total, cudaMemcpyDeviceToDevice, s));
            IB_CUDA(cudaMemcpyAsync(slot + L.total, prev, sizeof(T) * L.total, cudaMemcpyDeviceToDevice, s));
        }
        a.p = cur;
        a.pm = prev;
        a.out = prev;
        a.step = n;
        a.rec_step = n - 1;
        if (d == 2) {
            launch_leap2d(a, shape, H, s);
        } else if (use_tma) {
            dim3 blk(32, 8);
            const CUtensorMap& tmc = (cur == p0) ? tmap[0] : tmap[1];
            const CUtensorMap& tmm = (cur == p0) ? tmtile[1] : tmtile[0];   // p_prev: the other buffer
            PROF_LAUNCH("leap3d_tma_f32", s, {
                const StepArgs<float>& af = *reinterpret_cast<const StepArgs<float>*>(&a);
                if (pairs) {
                    dim3 gp((unsigned)((L.nx + 63) / 64), grid3.y, grid3.z);
                    if (H == 1) launch_leap3d_tma2<1>(af, tmc, tmm, tmK, zchunk, err, gp, s);
                    else if (H == 2) launch_leap3d_tma2<2>(af, tmc, tmm, tmK, zchunk, err, gp, s);
                    else if (H == 3) launch_leap3d_tma2<3>(af, tmc, tmm, tmK, zchunk, err, gp, s);
                    else launch_leap3d_tma2<4>(af, tmc, tmm, tmK, zchunk, err, gp, s);
                } else if (H == 1) launch_leap3d_tma<1>(af, tmc, tmm, tmK, rows3, zchunk, nty3, err, grid3, s);
                else if (H == 2) launch_leap3d_tma<2>(af, tmc, tmm, tmK, rows3, zchunk, nty3, err, grid3, s);
                else if (H == 3) launch_leap3d_tma<3>(af, tmc, tmm, tmK, rows3, zchunk, nty3, err, grid3, s);
                else launch_leap3d_tma<4>(af, tmc, tmm, tmK, rows3, zchunk, nty3, err, grid3, s);
            });
            if (code16) {
                const IbOp& op = t->ops[0];
                PROF_LAUNCH("ib_add3_f32", s, {
                    if (add3_u == 4)
                        k_ib_add3<4><<<grid1(op.nrows * 32, 256), 256, 0, s>>>(
                            op.nrows, op.row_pad, op.row_ptr, code16, op.w32, (const float*)a.p, (const float*)Kh,
                            (float*)a.out, L, a.dw, (float)a.da);
                    else
                        k_ib_add3<8><<<grid1(op.nrows * 32, 256), 256, 0, s>>>(
                            op.nrows, op.row_pad, op.row_ptr, code16, op.w32, (const float*)a.p, (const float*)Kh,
                            (float*)a.out, L, a.dw, (float)a.da);
                });
            }
        } else {
            dim3 blk(32, 8);
            PROF_LAUNCH(kname<T>("leap3d_f32", "leap3d_f64"), s, {
                if (H == 1) k_leap3d<T, 1><<<grid3, blk, 0, s>>>(a, zchunk, nty3);
                else if (H == 2) k_leap3d<T, 2><<<grid3, blk, 0, s>>>(a, zchunk, nty3);
                else if (H == 3) k_leap3d<T, 3><<<grid3, blk, 0, s>>>(a, zchunk, nty3);
                else k_leap3d<T, 4><<<grid3, blk, 0, s>>>(a, zchunk, nty3);
            });
        }
        IB_CHECK_LAUNCH("leapfrog step");
        std::swap(cur, prev);
        if (probe && (n + 1) % STAB_BLOCK == 0)
            TRY(probe_rescale<T>(probe, (n + 1) / STAB_BLOCK, L.total, cur, prev, (T*)nullptr, s));
    }
    if (g.rec.n) {
        k_receivers<T><<<grid1(g.rec.n, 256), 256, 0, s>>>(g.rec, cur, (T*)sh->traces_dev, nt, nt - 1);
        IB_CHECK_LAUNCH("k_receivers");
        ib_count_launch("setup");
    }
    if (!probe) TRY(check_finite<T>(L.total, cur, prev, (const T*)nullptr, s));
    if (use_tma) {
        int herr = 0;
        IB_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
        IB_CUDA(cudaStreamSynchronize(s));
        if (herr) {
            ib_set_error("a bounded TMA wait in the 3D step timed out");
            return IB_ERR_TIMEOUT;
        }
    }
    return IB_OK;
}

// ---------------------------------------------------------------------------
// 3D staggered pressure-velocity (1st-order section: the paper's signs and the
// backward-staggered base stencil; 3D first-order example):
//   v_a[j] (at j + e_a/2) += b_a[j] (sum_k c_k (p[j + k e_a] - p[j - (k-1) e_a]) + G_a corrections)
//   p[j] += kp[j] (sum_a sum_k c_k (v_a[j + (k-1) e_a] - v_a[j - k e_a]) + D corrections) + src
// with b_a = dt / (rho h) (mean of 1/rho at the two nodes) and kp = dt rho c^2 / h.
// The updated field is not read by its own update, so the modified rows are updated beside
// the others in the same launch.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_stag_coef3(Layout L, const T* vel, const T* rho, const uint8_t* mp, const uint8_t* mv0,
                             const uint8_t* mv1, const uint8_t* mv2, double dt, double inv_h, T* kp, T* b0, T* b1,
                             T* b2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < L.N; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = i % L.nx, r = i / L.nx, y = r % L.ny, z = r / L.ny;
        const int64_t q = L.idx(x, y, z);
        const double r0 = rho ? (double)rho[i] : 1.0;
        const double c = (double)vel[i];
        kp[q] = mp[q] ? stag_coef<T>(dt * r0 * c * c * inv_h) : (T)0;
        const double rx = (rho && x + 1 < L.nx) ? (double)rho[i + 1] : r0;
        const double ry = (rho && y + 1 < L.ny) ? (double)rho[i + L.nx] : r0;
        const double rz = (rho && z + 1 < L.nz) ? (double)rho[i + L.nx * L.ny] : r0;
        b0[q] = mv0[q] ? stag_coef<T>(dt * 0.5 * (1.0 / r0 + 1.0 / rx) * inv_h) : (T)0;
        b1[q] = mv1[q] ? stag_coef<T>(dt * 0.5 * (1.0 / r0 + 1.0 / ry) * inv_h) : (T)0;
        b2[q] = mv2[q] ? stag_coef<T>(dt * 0.5 * (1.0 / r0 + 1.0 / rz) * inv_h) : (T)0;
    }
}

// Lane gl of 8's share of sum_j w_j f[q + off_j] over the entries [j0, j1) of a 3D row: pairs
// of adjacent entries (their columns and weights as one vector load each; a pair that straddles
// the row's ends has the foreign weight dropped), U pairs in flight.  Columns are 16-bit footprint
// codes, decoded mostly in 32-bit arithmetic against a base moved by the code's offset of 16 nodes
// per axis, or, for a table that has none, padded offsets of 64 bits.  32-bit offsets, which need no
// decoding but two more bytes an entry, took 5 % longer.  In FP64 the rounds past the end of the warp's
// longest row are left out whole: an operation takes the pipe of an SM for 16 cycles whatever its
// lanes do.
template <typename T>
struct PairOf;
template <> struct PairOf<float> { typedef float2 type; };
template <> struct PairOf<double> { typedef double2 type; };
template <typename T, typename O, int U>
__device__ __forceinline__ T row_gather3(const O* __restrict__ col, const T* __restrict__ w, int64_t j0, int64_t j1,
                                         const T* __restrict__ f, int64_t q, int px, int plane, int gl) {
    constexpr bool CODES = sizeof(O) == 2;
    const int64_t centre = CODES ? 16 * ((int64_t)plane + px + 1) : 0;
    const T* base = f + (q - centre);
    const int64_t js = j0 & ~(int64_t)1;
    const int most = sizeof(T) == 8 ? __reduce_max_sync(0xffffffffu, (int)(j1 - js)) : (int)(j1 - js);
    T v = 0;
    for (int k = sizeof(T) == 8 ? 0 : 2 * gl; k < most; k += 16 * U) {
        T w0[U], w1[U], p0[U], p1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (sizeof(T) == 8 && k + 16 * u >= most) continue;   // warp-uniform
            const int64_t e = js + k + 16 * u + (sizeof(T) == 8 ? 2 * gl : 0);
            int64_t o0 = centre, o1 = centre;
            w0[u] = w1[u] = (T)0;
            if (e < j1) {
                const typename PairOf<T>::type ww = *reinterpret_cast<const typename PairOf<T>::type*>(w + e);
                int64_t c0, c1;
                if constexpr (CODES) {
                    const uint32_t c = *reinterpret_cast<const uint32_t*>(col + e);
                    c0 = (int64_t)(int)((c >> 10) & 63) * plane + ((int)(c & 31) + (int)((c >> 5) & 31) * px);
                    c1 = (int64_t)(int)(c >> 26) * plane + ((int)((c >> 16) & 31) + (int)((c >> 21) & 31) * px);
                } else {
                    const longlong2 c = *reinterpret_cast<const longlong2*>(col + e);
                    c0 = c.x;
                    c1 = c.y;
                }
                if (e >= j0) {
                    w0[u] = ww.x;
                    o0 = c0;
                }
                if (e + 1 < j1) {
                    w1[u] = ww.y;
                    o1 = c1;
                }
            }
            p0[u] = base[o0];
            p1[u] = base[o1];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (sizeof(T) == 8 && k + 16 * u >= most) continue;
            v += w0[u] * p0[u];
            v += w1[u] * p1[u];
        }
    }
    return v;
}
// c[k - 1] for a k that differs between lanes, without indexing the arguments
template <int H, typename T>
__device__ __forceinline__ T coef_at(const T* c, int k) {
    T r = c[0];
#pragma unroll
    for (int j = 2; j <= H; ++j) r = j == k ? c[j - 1] : r;
    return r;
}
template <typename T>
__device__ __forceinline__ T sum8(T v) {
    v += __shfl_xor_sync(0xffffffffu, v, 4, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 2, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 1, 8);
    return v;
}

// rows of one or several operators on the same row nodes
template <typename T>
struct Rows3D {
    int64_t n;
    const int64_t* pad;
    const T* k;          // the row nodes' coefficients
    const int64_t* ptr[3];
    const void* col[3];  // the entries' columns: 16-bit codes or 64-bit offsets
    const T* w[3];
};

template <typename T, int H>
struct Stag3Args {
    Layout L;
    T c[4];              // c[k - 1]: weight of the pair at offsets +(k - 1/2), -(k - 1/2)
    T* p;
    T* v[3];
    const T* kp;         // in kp and b, a mark (marked3) stands at the nodes of the modified rows
    const T* b[3];
    Rows3D<T> g[3];      // gradient rows of v_a (columns p: operator 0 of each)
    Rows3D<T> d;         // divergence rows (columns v_0, v_1, v_2)
    int nrb[4];          // row blocks: v_0, v_1, v_2; p
    int nbx, nby;        // column blocks along x and y
    PointSet<T> src;     // weights include dt / h^3
    const T* wavelet;
    int step;
    PointSet<T> rec;     // receivers, sampled from p before the v update
    T* traces;
    int nt;
    int rec_step;
};

// Both kernels: column blocks of 256 threads own VX x-adjacent nodes per thread (16-byte
// vectors) in a 32 VX x 8 x 1 box; row blocks update the nodes of the modified rows whole,
// which the column blocks leave out (a mark in place of their coefficient).  Two
// launches per step: with one thread per node, a pass per operator over its rows, and
// separate source and receiver launches a step had ten, and 64-bit divisions for every node.
// 160 x 144 x 122, order 4, FP32: 172 -> 108 us a step (v 31, p 74; a whole warp per divergence
// row: p 104).  The p rows, 3 gathers of about 60 entries each, bound it by instruction issue.
//   From 24 000 divergence rows on, orders 6 and 8 launch the two kinds of blocks one after the
// other: in one kernel with columns of 100-127 registers a thread the rows' gathers have 16 warps on
// an SM, alone 40 (FP32).  30 steps of order 8, ms, in one launch | apart | with ten launches:
//   180 x 170 x 140   FP32 11.4 |  7.8 | 10.0    FP64 26.2 | 21.0 | 20.9
//    60 x  60 x  80   FP32  1.6 |  1.8 |  2.6    FP64  2.7 |  3.4 |  5.1
// In FP64 its pipe bounds the step, so vectors of nodes above the surface and idle rounds of the
// gathers are left out.
static const int S3_ROWS = 32;   // rows per row block, 8 lanes each
static const int64_t S3_SPLIT_ROWS = 24000;   // divergence rows from which orders 6 and 8 take launches of their own

// is any of a thread's coefficients not zero (integer operations)
__device__ __forceinline__ bool nonzero(float k) { return (__float_as_uint(k) << 1) != 0u; }
__device__ __forceinline__ bool nonzero(double k) { return ((__double2hiint(k) << 1) | __double2loint(k)) != 0; }
template <typename T, int VX>
__device__ __forceinline__ void load3(T (&d)[VX], const T* p) {
    typedef typename std::conditional<sizeof(T) == 4, float4, double2>::type V;
    static_assert(sizeof(V) == sizeof(T) * VX, "16-byte vectors");
    *reinterpret_cast<V*>(&d[0]) = *reinterpret_cast<const V*>(p);
}
template <typename T, int VX>
__device__ __forceinline__ void store3(T* p, const T (&d)[VX], const T (&k)[VX], int64_t x, int64_t nx) {
    typedef typename std::conditional<sizeof(T) == 4, float4, double2>::type V;
    bool all = x + VX <= nx;
#pragma unroll
    for (int j = 0; j < VX; ++j) all = all && !marked3(k[j]);
    if (all) {
        *reinterpret_cast<V*>(p) = *reinterpret_cast<const V*>(&d[0]);
    } else {
#pragma unroll
        for (int j = 0; j < VX; ++j)
            if (x + j < nx && !marked3(k[j])) p[j] = d[j];
    }
}

// PART of a launch: row blocks and column blocks (S3_BOTH), or only the ones or the others; O: the
// type of the entries' columns
enum { S3_BOTH = 0, S3_ROWS_ONLY = 1, S3_COLUMNS = 2 };

// v_a += b_a (forward-staggered d/dx_a p) at every interior v_a node
template <typename T, int H, int PART, typename O>
__global__ void __launch_bounds__(256) k_stag_v3d(const __grid_constant__ Stag3Args<T, H> a) {
    constexpr int VX = 16 / (int)sizeof(T), HV = (H + VX - 1) / VX, HX = HV * VX;
    const Layout& L = a.L;
    int64_t blk = blockIdx.x;
    if (PART != S3_ROWS_ONLY)
        record_receivers(a.rec, (const T*)a.p, a.traces, a.nt, a.rec_step, blk * 256 + threadIdx.x, (int64_t)gridDim.x * 256);
    const int64_t st[3] = {1, L.px, L.plane};
#pragma unroll
    for (int ax = 0; ax < 3 && PART != S3_COLUMNS; ++ax) {
        if (blk < a.nrb[ax]) {
            const Rows3D<T>& R = a.g[ax];
            const int gl = threadIdx.x & 7;
            const int64_t r = blk * S3_ROWS + (threadIdx.x >> 3);
            const bool act = r < R.n;
            const int64_t q = act ? R.pad[r] : L.base;
            const T bq = act && gl == 0 ? R.k[r] : (T)0, vq = gl == 0 ? a.v[ax][q] : (T)0;
            T s = row_gather3<T, O, 4>((const O*)R.col[0], R.w[0], act ? R.ptr[0][r] : 0, act ? R.ptr[0][r + 1] : 0, a.p, q,
                                       (int)L.px, (int)L.plane, gl);
            // lane k takes the stencil's pair k; in FP64 all lanes in one operation
            if constexpr (sizeof(T) == 8) {
                T up = 0, dn = 0;
                if (gl >= 1 && gl <= H) {
                    up = a.p[q + gl * st[ax]];
                    dn = a.p[q - (gl - 1) * st[ax]];
                }
                s += coef_at<H>(a.c, gl) * (up - dn);
            } else {
#pragma unroll
                for (int k = 1; k <= H; ++k)
                    if (gl == k) s += a.c[k - 1] * (a.p[q + k * st[ax]] - a.p[q - (k - 1) * st[ax]]);
            }
            s = sum8(s);
            if (act && gl == 0) a.v[ax][q] = vq + bq * s;
            return;
        }
        blk -= a.nrb[ax];
    }
    if (PART == S3_ROWS_ONLY) return;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int bx = (int)(blk % a.nbx), by = (int)(blk / a.nbx % a.nby);
    const int64_t z = blk / a.nbx / a.nby, x = ((int64_t)bx * 32 + lane) * VX, y = by * 8 + wy;
    if (x >= L.nx || y >= L.ny) return;
    const int64_t q = L.idx(x, y, z);
    T w[VX + 2 * HX], y2[2 * H][VX], z2[2 * H][VX], vv[3][VX], bb[3][VX];
#pragma unroll
    for (int m = 0; m < 2 * HV + 1; ++m) load3<T, VX>(*reinterpret_cast<T(*)[VX]>(&w[m * VX]), a.p + q + (m - HV) * VX);
#pragma unroll
    for (int k = 0; k < 2 * H; ++k) {   // offsets 1 - H .. H
        if (k == H - 1) continue;
        load3<T, VX>(y2[k], a.p + q + (k + 1 - H) * L.px);
        load3<T, VX>(z2[k], a.p + q + (k + 1 - H) * L.plane);
    }
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        load3<T, VX>(vv[ax], a.v[ax] + q);
        load3<T, VX>(bb[ax], a.b[ax] + q);
    }
    if (sizeof(T) == 8) {   // the FP64 pipe bounds the step: leave out the nodes above the surface
        bool any = false;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
#pragma unroll
            for (int j = 0; j < VX; ++j) any = any || nonzero(bb[ax][j]);
        if (!any) return;
    }
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        const T c = w[HX + j];
        T sx = 0, sy = 0, sz = 0;
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            sx += a.c[k - 1] * (w[HX + j + k] - w[HX + j - k + 1]);
            sy += a.c[k - 1] * (y2[H - 1 + k][j] - (k == 1 ? c : y2[H - k][j]));
            sz += a.c[k - 1] * (z2[H - 1 + k][j] - (k == 1 ? c : z2[H - k][j]));
        }
        vv[0][j] += bb[0][j] * sx;
        vv[1][j] += bb[1][j] * sy;
        vv[2][j] += bb[2][j] * sz;
    }
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) store3<T, VX>(a.v[ax] + q, vv[ax], bb[ax], x, L.nx);
}

// p += kp (backward-staggered divergence of v) + sources at every interior p node
template <typename T, int H, int PART, typename O>
__global__ void __launch_bounds__(256) k_stag_p3d(const __grid_constant__ Stag3Args<T, H> a) {
    constexpr int VX = 16 / (int)sizeof(T), HV = (H + VX - 1) / VX, HX = HV * VX;
    const Layout& L = a.L;
    int64_t blk = blockIdx.x;
    if (PART == S3_ROWS_ONLY || (PART == S3_BOTH && blk < a.nrb[3])) {
        const int gl = threadIdx.x & 7;
        const int64_t r = blk * S3_ROWS + (threadIdx.x >> 3);
        const bool act = r < a.d.n;
        const int64_t q = act ? a.d.pad[r] : L.base;
        const T kq = act && gl == 0 ? a.d.k[r] : (T)0, pq = gl == 0 ? a.p[q] : (T)0;
        T s = 0, sv = 0;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
            s += row_gather3<T, O, 4>((const O*)a.d.col[ax], a.d.w[ax], act ? a.d.ptr[ax][r] : 0, act ? a.d.ptr[ax][r + 1] : 0,
                                      a.v[ax], q, (int)L.px, (int)L.plane, gl);
        if constexpr (sizeof(T) == 4) {
            const int64_t st[3] = {1, L.px, L.plane};
#pragma unroll
            for (int ax = 0; ax < 3; ++ax)
#pragma unroll
                for (int k = 1; k <= H; ++k)
                    if (gl == ((ax * H + k) & 7))
                        s += a.c[k - 1] * (a.v[ax][q + (k - 1) * st[ax]] - a.v[ax][q - k * st[ax]]);
        }
#pragma unroll
        for (int i0 = 0; i0 < (sizeof(T) == 8 ? 3 * H : 0); i0 += 8) {   // the 3 H pairs of the stencil, one a lane
            const int i = i0 + gl, ax = i / H, k = i - ax * H + 1;
            T up = 0, dn = 0;
            if (i < 3 * H) {
                const T* f = (ax == 0 ? a.v[0] : ax == 1 ? a.v[1] : a.v[2]) + q;
                const int64_t d = ax == 0 ? 1 : ax == 1 ? L.px : L.plane;
                up = f[(k - 1) * d];
                dn = f[-k * d];
            }
            s += coef_at<H>(a.c, k) * (up - dn);
        }
        for (int i = gl; i < 8 * a.src.n; i += 8)
            if (a.src.idx[i] == q) sv += a.src.w[i];
        s = sum8(s);
        sv = sum8(sv);
        if (act && gl == 0) a.p[q] = pq + kq * s + (sv != (T)0 ? sv * a.wavelet[a.step] : (T)0);
        return;
    }
    if (PART == S3_BOTH) blk -= a.nrb[3];
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int bx = (int)(blk % a.nbx), by = (int)(blk / a.nbx % a.nby);
    const int64_t z = blk / a.nbx / a.nby, x = ((int64_t)bx * 32 + lane) * VX, y = by * 8 + wy;
    const bool in = x < L.nx && y < L.ny;
    const int64_t q = L.idx(x, y, z);
    T w[VX + 2 * HX], y2[2 * H][VX], z2[2 * H][VX], pp[VX], kk[VX];
    if (in) {
#pragma unroll
        for (int m = 0; m < 2 * HV + 1; ++m) load3<T, VX>(*reinterpret_cast<T(*)[VX]>(&w[m * VX]), a.v[0] + q + (m - HV) * VX);
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) {   // offsets -H .. H - 1
            load3<T, VX>(y2[k], a.v[1] + q + (k - H) * L.px);
            load3<T, VX>(z2[k], a.v[2] + q + (k - H) * L.plane);
        }
        load3<T, VX>(pp, a.p + q);
        load3<T, VX>(kk, a.kp + q);
    }
    // does a source corner fall in this block's box? (block-uniform)
    int here = 0;
    if (a.src.n) {
        for (int i = threadIdx.x; i < 8 * a.src.n; i += 256) {
            if (a.src.w[i] == (T)0) continue;
            const int64_t rel = a.src.idx[i] - L.base, sz = rel / L.plane, r2 = rel - sz * L.plane, sy = r2 / L.px,
                          sx = r2 - sy * L.px;
            here |= sz == z && sy / 8 == by && sx / (32 * VX) == bx;
        }
        here = __syncthreads_or(here);
    }
    if (!in) return;
    if (sizeof(T) == 8) {
        bool any = false;
#pragma unroll
        for (int j = 0; j < VX; ++j) any = any || nonzero(kk[j]);
        if (!any) return;
    }
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        T s = 0;
#pragma unroll
        for (int k = 1; k <= H; ++k) s += a.c[k - 1] * (w[HX + j + k - 1] - w[HX + j - k]);
#pragma unroll
        for (int k = 1; k <= H; ++k) s += a.c[k - 1] * (y2[H + k - 1][j] - y2[H - k][j]);
#pragma unroll
        for (int k = 1; k <= H; ++k) s += a.c[k - 1] * (z2[H + k - 1][j] - z2[H - k][j]);
        pp[j] += kk[j] * s;
        if (here) {
            T sv = 0;
            for (int i = 0; i < 8 * a.src.n; ++i)
                if (a.src.idx[i] == q + j) sv += a.src.w[i];
            if (sv != (T)0) pp[j] += sv * a.wavelet[a.step];
        }
    }
    store3<T, VX>(a.p + q, pp, kk, x, L.nx);
}

// the row nodes' coefficients in row order, and marks in their places
template <typename T>
__global__ void k_mark_rows3(int64_t n, const int64_t* __restrict__ pad, T* k, T* rk) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        rk[i] = k[pad[i]];
        set_mark3(k[pad[i]]);
    }
}
template <typename T>
static ib_status mark_rows3(const IbOp& op, T* k, const T** rk, Scratch& S) {
    *rk = nullptr;
    if (!op.nrows) return IB_OK;
    T* r;
    TRY(S.alloc(&r, op.nrows));
    k_mark_rows3<T><<<grid1(op.nrows, 256), 256, 0, S.s>>>(op.nrows, op.row_pad, k, r);
    IB_CHECK_LAUNCH("k_mark_rows3");
    ib_count_launch("setup");
    *rk = r;
    return IB_OK;
}

template <typename T>
static ib_status forward_stag3(ib_table* t, const ib_shot* sh, double dt, int nt, cudaStream_t s) {
    const Layout& L = t->L;
    if (shot_damped(sh)) {
        ib_set_error("the absorbing layer is implemented for the second-order form");
        return IB_ERR_STATE;
    }
    const int M = t->opts.space_order;
    const int H = M / 2;
    Scratch S(s);
    T *p, *v0, *v1, *v2, *kp, *b0, *b1, *b2;
    TRY(S.alloc(&p, L.total, true));
    TRY(S.alloc(&v0, L.total, true));
    TRY(S.alloc(&v1, L.total, true));
    TRY(S.alloc(&v2, L.total, true));
    TRY(S.alloc(&kp, L.total, true));
    TRY(S.alloc(&b0, L.total, true));
    TRY(S.alloc(&b1, L.total, true));
    TRY(S.alloc(&b2, L.total, true));
    k_stag_coef3<T><<<grid1(L.N, 256), 256, 0, s>>>(L, (const T*)sh->vel_dev, (const T*)sh->rho_dev, t->mask_pad[0],
                                                    t->mask_pad[1], t->mask_pad[2], t->mask_pad[3], dt,
                                                    1.0 / t->grid.h, kp, b0, b1, b2);
    IB_CHECK_LAUNCH("k_stag_coef3");
    ib_count_launch("setup");
    Geom<T> g;
    TRY(setup_points<T>(t, sh, dt / pow(t->grid.h, 3), S, g));
    T w2u[5], c1[4];
    stencil_weights<T>(M, w2u, c1);
    T* coef[4] = {b0, b1, b2, kp};
    auto run = [&](auto hc) -> ib_status {
        constexpr int HH = decltype(hc)::value, VX = 16 / (int)sizeof(T);
        Stag3Args<T, HH> a;
        memset(&a, 0, sizeof a);
        a.L = L;
        for (int k = 0; k < 4; ++k) a.c[k] = c1[k];
        a.p = p;
        a.v[0] = v0;
        a.v[1] = v1;
        a.v[2] = v2;
        a.kp = kp;
        a.b[0] = b0;
        a.b[1] = b1;
        a.b[2] = b2;
        // IB_ROW_OFF64=1: 64-bit offsets, as where some operator's columns have no codes
        const char* e64 = getenv("IB_ROW_OFF64");
        bool wide = e64 && e64[0] == '1';
        for (int o = 0; o < 6; ++o) wide = wide || (t->ops[o].nnz && !t->ops[o].code16);
        // operators 0-2: gradients; 3-5: the divergence's parts, on one set of rows
        for (int o = 0; o < 6; ++o) {
            const IbOp& op = t->ops[o];
            Rows3D<T>& R = o < 3 ? a.g[o] : a.d;
            const int i = o < 3 ? 0 : o - 3;
            R.n = op.nrows;
            R.pad = op.row_pad;
            R.ptr[i] = op.row_ptr;
            R.w[i] = sizeof(T) == 8 ? (const T*)op.w64 : (const T*)op.w32;
            R.col[i] = wide ? (const void*)op.col_pad : (const void*)op.code16;
            if (o < 4) TRY(mark_rows3<T>(op, coef[o], &R.k, S));
        }
        for (int o = 0; o < 4; ++o) a.nrb[o] = (int)((t->ops[o].nrows + S3_ROWS - 1) / S3_ROWS);
        a.nbx = (int)((L.nx + 32 * VX - 1) / (32 * VX));
        a.nby = (int)((L.ny + 7) / 8);
        a.src = g.src;
        a.wavelet = (const T*)sh->wavelet_dev;
        a.rec = g.rec;
        a.traces = (T*)sh->traces_dev;
        a.nt = nt;
        const int64_t cols = (int64_t)a.nbx * a.nby * L.nz;
        const unsigned rv = (unsigned)(a.nrb[0] + a.nrb[1] + a.nrb[2]), rp = (unsigned)a.nrb[3];
        const bool split = wide || (HH > 2 && a.d.n >= S3_SPLIT_ROWS);
        for (int n = 0; n < nt; ++n) {
            a.step = n;
            a.rec_step = n - 1;
            PROF_LAUNCH(kname<T>("stag_v3d_f32", "stag_v3d_f64"), s, {
                if (!split) {
                    k_stag_v3d<T, HH, S3_BOTH, uint16_t><<<(unsigned)cols + rv, 256, 0, s>>>(a);
                } else {
                    if (rv && wide) k_stag_v3d<T, HH, S3_ROWS_ONLY, int64_t><<<rv, 256, 0, s>>>(a);
                    else if (rv) k_stag_v3d<T, HH, S3_ROWS_ONLY, uint16_t><<<rv, 256, 0, s>>>(a);
                    k_stag_v3d<T, HH, S3_COLUMNS, uint16_t><<<(unsigned)cols, 256, 0, s>>>(a);
                }
            });
            PROF_LAUNCH(kname<T>("stag_p3d_f32", "stag_p3d_f64"), s, {
                if (!split) {
                    k_stag_p3d<T, HH, S3_BOTH, uint16_t><<<(unsigned)cols + rp, 256, 0, s>>>(a);
                } else {
                    if (rp && wide) k_stag_p3d<T, HH, S3_ROWS_ONLY, int64_t><<<rp, 256, 0, s>>>(a);
                    else if (rp) k_stag_p3d<T, HH, S3_ROWS_ONLY, uint16_t><<<rp, 256, 0, s>>>(a);
                    k_stag_p3d<T, HH, S3_COLUMNS, uint16_t><<<(unsigned)cols, 256, 0, s>>>(a);
                }
            });
            IB_CHECK_LAUNCH("3D staggered step");
        }
        if (g.rec.n) {
            k_receivers<T><<<grid1(g.rec.n, 256), 256, 0, s>>>(g.rec, p, (T*)sh->traces_dev, nt, nt - 1);
            IB_CHECK_LAUNCH("k_receivers");
            ib_count_launch("setup");
        }
        return IB_OK;
    };
    if (H == 1) TRY(run(std::integral_constant<int, 1>()));
    else if (H == 2) TRY(run(std::integral_constant<int, 2>()));
    else if (H == 3) TRY(run(std::integral_constant<int, 3>()));
    else TRY(run(std::integral_constant<int, 4>()));
    TRY(check_finite<T>(L.total, p, v0, v1, s));
    TRY(check_finite<T>(L.total, v2, (const T*)nullptr, (const T*)nullptr, s));
    return IB_OK;
}

// ---------------------------------------------------------------------------
// 2D staggered pressure-velocity
//   v_a[j] (at j + e_a/2) += bh_a[j] (sum_k c_k (p[j + k e_a] - p[j - (k-1) e_a]) + IB)
//   p[j] += kh[j] (sum_a sum_k c_k (v_a[j + (k-1) e_a] - v_a[j - k e_a]) + IB) + src
// with bh_a = dt / (rho h) and kh = dt rho c^2 / h.  Column and row blocks as in 3D: a thread
// owns 16 bytes of adjacent nodes of one row, the modified rows are updated whole by 8 lanes
// each.  The state of a 1001 x 1001 shot stays in the L2 and a kernel is a few microseconds
// of latency; correction sums formed by the producing tiles in shared memory, which this
// replaces, took 22 us per step and 7 ms of host plans per shot; 50 steps are now 683 us (749
// with 16 lanes per divergence row).
// ---------------------------------------------------------------------------
template <typename T>
struct Rows2D {
    int64_t n;
    const int64_t* pad;
    const T* k;          // the row nodes' coefficients
    const int64_t* ptr[2];
    const int32_t* code[2];
    const T* w[2];
};
template <typename T>
struct Stag2Args {
    Layout L;
    T c[4];              // c[k - 1]: weight of the pair at offsets +(k - 1/2), -(k - 1/2)
    T* p;
    T* v[2];
    const T* kp;         // in kp and b, a mark (marked3) stands at the nodes of the modified rows
    const T* b[2];
    Rows2D<T> g[2];      // gradient rows of v_x, v_z
    Rows2D<T> d;         // divergence rows (columns v_x, v_z)
    int nrb[3];          // row blocks: v_x, v_z; p
    int nbx;             // column blocks along x
    PointSet<T> src;     // weights include dt / h^2
    const T* wavelet;
    const int* step_base; // device step offset added to step / rec_step (graph replays)
    int step;
    PointSet<T> rec;     // receivers, sampled from p before the v update
    T* traces;
    int nt;
    int rec_step;
};

// lane gl of 8's share of sum_j w_j f[q + off_j] over the entries [j0, j1) of a 2D row
template <typename T>
__device__ __forceinline__ T row_gather2(const int32_t* __restrict__ code, const T* __restrict__ w, int64_t j0, int64_t j1,
                                         const T* f, int64_t q, int64_t px, int gl) {
    T v = 0;
    for (int64_t e = j0 + gl; e < j1; e += 8) {
        int dx, dz, dy;
        unpack_off(code[e], dx, dz, dy);   // 2D codes: (x, z, 0)
        v += w[e] * f[q + dz * px + dx];
    }
    return v;
}

// v^{n+1/2} = v^{n-1/2} + (dt / rho) G_mod p^n
template <typename T, int H>
__global__ void __launch_bounds__(256) k_stag_v2d(const __grid_constant__ Stag2Args<T> a) {
    constexpr int VX = 16 / (int)sizeof(T), HV = (H + VX - 1) / VX, HX = HV * VX;
    const Layout& L = a.L;
    int64_t blk = blockIdx.x;
    const int rs = a.rec_step + (a.step_base ? *a.step_base : 0);
    record_receivers(a.rec, (const T*)a.p, a.traces, a.nt, rs, blk * 256 + threadIdx.x, (int64_t)gridDim.x * 256);
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
        if (blk < a.nrb[ax]) {
            const Rows2D<T>& R = a.g[ax];
            const int gl = threadIdx.x & 7;
            const int64_t r = blk * S3_ROWS + (threadIdx.x >> 3), st = ax ? L.px : 1;
            const bool act = r < R.n;
            const int64_t q = act ? R.pad[r] : L.base;
            const T bq = act && gl == 0 ? R.k[r] : (T)0, vq = gl == 0 ? a.v[ax][q] : (T)0;
            T s = 0;
            if (act) s = row_gather2(R.code[0], R.w[0], R.ptr[0][r], R.ptr[0][r + 1], (const T*)a.p, q, L.px, gl);
#pragma unroll
            for (int k = 1; k <= H; ++k)
                if (gl == k) s += a.c[k - 1] * (a.p[q + k * st] - a.p[q - (k - 1) * st]);
            s = sum8(s);
            if (act && gl == 0) a.v[ax][q] = vq + bq * s;
            return;
        }
        blk -= a.nrb[ax];
    }
    const int lane = threadIdx.x & 31, wz = threadIdx.x >> 5;
    const int64_t x = ((blk % a.nbx) * 32 + lane) * VX, z = blk / a.nbx * 8 + wz;
    if (x >= L.nx || z >= L.nz) return;
    const int64_t q = L.base + z * L.px + x;
    T w[VX + 2 * HX], z2[2 * H][VX], vv[2][VX], bb[2][VX];
#pragma unroll
    for (int m = 0; m < 2 * HV + 1; ++m) load3<T, VX>(*reinterpret_cast<T(*)[VX]>(&w[m * VX]), a.p + q + (m - HV) * VX);
#pragma unroll
    for (int k = 0; k < 2 * H; ++k)   // offsets 1 - H .. H
        if (k != H - 1) load3<T, VX>(z2[k], a.p + q + (k + 1 - H) * L.px);
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
        load3<T, VX>(vv[ax], a.v[ax] + q);
        load3<T, VX>(bb[ax], a.b[ax] + q);
    }
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        T sx = 0, sz = 0;
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            sx += a.c[k - 1] * (w[HX + j + k] - w[HX + j - k + 1]);
            sz += a.c[k - 1] * (z2[H - 1 + k][j] - (k == 1 ? w[HX + j] : z2[H - k][j]));
        }
        vv[0][j] += bb[0][j] * sx;
        vv[1][j] += bb[1][j] * sz;
    }
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) store3<T, VX>(a.v[ax] + q, vv[ax], bb[ax], x, L.nx);
}

// p^{n+1} = p^n + dt rho c^2 D_mod v^{n+1/2} (+ source)
template <typename T, int H>
__global__ void __launch_bounds__(256) k_stag_p2d(const __grid_constant__ Stag2Args<T> a) {
    constexpr int VX = 16 / (int)sizeof(T), HV = (H + VX - 1) / VX, HX = HV * VX;
    const Layout& L = a.L;
    int64_t blk = blockIdx.x;
    const int n = a.step + (a.step_base ? *a.step_base : 0);
    if (blk < a.nrb[2]) {
        const int gl = threadIdx.x & 7;
        const int64_t r = blk * S3_ROWS + (threadIdx.x >> 3);
        const bool act = r < a.d.n;
        const int64_t q = act ? a.d.pad[r] : L.base;
        const T kq = act && gl == 0 ? a.d.k[r] : (T)0, pq = gl == 0 ? a.p[q] : (T)0;
        T s = 0, sv = 0;
#pragma unroll
        for (int ax = 0; ax < 2; ++ax) {
            const int64_t st = ax ? L.px : 1;
            if (act)
                s += row_gather2(a.d.code[ax], a.d.w[ax], a.d.ptr[ax][r], a.d.ptr[ax][r + 1], (const T*)a.v[ax], q, L.px, gl);
#pragma unroll
            for (int k = 1; k <= H; ++k)
                if (gl == ax * H + k - 1) s += a.c[k - 1] * (a.v[ax][q + (k - 1) * st] - a.v[ax][q - k * st]);
        }
        for (int i = gl; i < 8 * a.src.n; i += 8)
            if (a.src.idx[i] == q) sv += a.src.w[i];
        s = sum8(s);
        sv = sum8(sv);
        if (act && gl == 0) a.p[q] = pq + kq * s + (sv != (T)0 ? sv * a.wavelet[n] : (T)0);
        return;
    }
    blk -= a.nrb[2];
    const int lane = threadIdx.x & 31, wz = threadIdx.x >> 5;
    const int64_t bx = blk % a.nbx, bz = blk / a.nbx, x = (bx * 32 + lane) * VX, z = bz * 8 + wz;
    const bool in = x < L.nx && z < L.nz;
    const int64_t q = L.base + z * L.px + x;
    T w[VX + 2 * HX], z2[2 * H][VX], pp[VX], kk[VX];
    if (in) {
#pragma unroll
        for (int m = 0; m < 2 * HV + 1; ++m) load3<T, VX>(*reinterpret_cast<T(*)[VX]>(&w[m * VX]), a.v[0] + q + (m - HV) * VX);
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) load3<T, VX>(z2[k], a.v[1] + q + (k - H) * L.px);   // offsets -H .. H - 1
        load3<T, VX>(pp, a.p + q);
        load3<T, VX>(kk, a.kp + q);
    }
    // does a source corner fall in this block's box? (block-uniform)
    int here = 0;
    if (a.src.n) {
        for (int i = threadIdx.x; i < 8 * a.src.n; i += 256) {
            if (a.src.w[i] == (T)0) continue;
            const int64_t rel = a.src.idx[i] - L.base, sz = rel / L.px, sx = rel - sz * L.px;
            here |= sz / 8 == bz && sx / (32 * VX) == bx;
        }
        here = __syncthreads_or(here);
    }
    if (!in) return;
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        T s = 0;
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            s += a.c[k - 1] * (w[HX + j + k - 1] - w[HX + j - k]);
            s += a.c[k - 1] * (z2[H + k - 1][j] - z2[H - k][j]);
        }
        pp[j] += kk[j] * s;
        if (here) {
            T sv = 0;
            for (int i = 0; i < 8 * a.src.n; ++i)
                if (a.src.idx[i] == q + j) sv += a.src.w[i];
            if (sv != (T)0) pp[j] += sv * a.wavelet[n];
        }
    }
    store3<T, VX>(a.p + q, pp, kk, x, L.nx);
}

__global__ void k_add_step(int* base, int k) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *base += k;
}

// time steps per captured graph of the staggered loop (the graph is replayed nt / STAG_GRAPH_STEPS times)
static const int STAG_GRAPH_STEPS = 50;
static_assert(STAG_GRAPH_STEPS == STAB_BLOCK, "the stability probe renormalises between graph replays");

template <typename T>
static ib_status forward_stag(ib_table* t, const ib_shot* sh, double dt, int nt, cudaStream_t s,
                              const Probe* probe = nullptr) {
    const Layout& L = t->L;
    const int d = t->grid.ndim;
    if (shot_damped(sh)) {
        ib_set_error("the absorbing layer is implemented for the second-order form");
        return IB_ERR_STATE;
    }
    if (d != 2) {
        ib_set_error("the staggered form is implemented in 2D");
        return IB_ERR_STATE;
    }
    const int M = t->opts.space_order;
    const int H = M / 2;
    Scratch S(s);
    T *p, *vx, *vz, *kp, *bx, *bz;
    TRY(S.alloc(&p, L.total, true));
    TRY(S.alloc(&vx, L.total, true));
    TRY(S.alloc(&vz, L.total, true));
    TRY(S.alloc(&kp, L.total, true));
    TRY(S.alloc(&bx, L.total, true));
    TRY(S.alloc(&bz, L.total, true));
    k_stag_coef<T><<<grid1(L.N, 256), 256, 0, s>>>(L, (const T*)sh->vel_dev, (const T*)sh->rho_dev, t->mask_pad[0],
                                                   t->mask_pad[1], t->mask_pad[2], dt, 1.0 / t->grid.h, kp, bx, bz);
    IB_CHECK_LAUNCH("k_stag_coef");
    ib_count_launch("setup");
    if (probe) {   // random p, v_x, v_z on their interior nodes, normalised together
        k_rand_fill<T><<<grid1(L.total, 256), 256, 0, s>>>(L.total, kp, probe->seed, p, (T*)nullptr);
        k_rand_fill<T><<<grid1(L.total, 256), 256, 0, s>>>(L.total, bx, probe->seed + 1, vx, (T*)nullptr);
        k_rand_fill<T><<<grid1(L.total, 256), 256, 0, s>>>(L.total, bz, probe->seed + 2, vz, (T*)nullptr);
        IB_CHECK_LAUNCH("k_rand_fill");
        TRY(probe_rescale<T>(probe, 0, L.total, p, vx, vz, s));
    }
    Geom<T> g;
    TRY(setup_points<T>(t, sh, dt / pow(t->grid.h, d), S, g));
    Stag2Args<T> a;
    memset(&a, 0, sizeof a);
    a.L = L;
    {
        T w2u[5];
        stencil_weights<T>(M, w2u, a.c);
    }
    a.p = p;
    a.v[0] = vx;
    a.v[1] = vz;
    a.b[0] = bx;
    a.b[1] = bz;
    a.kp = kp;
    // operators 0, 1: gradients; 2, 3: the divergence's parts, on one set of rows
    T* coef[3] = {bx, bz, kp};
    for (int o = 0; o < 4; ++o) {
        const IbOp& op = t->ops[o];
        Rows2D<T>& R = o < 2 ? a.g[o] : a.d;
        const int i = o < 2 ? 0 : o - 2;
        R.n = op.nrows;
        R.pad = op.row_pad;
        R.ptr[i] = op.row_ptr;
        R.code[i] = op.col_code;
        R.w[i] = sizeof(T) == 8 ? (const T*)op.w64 : (const T*)op.w32;
        if (o < 3) TRY(mark_rows3<T>(op, coef[o], &R.k, S));
        if (o < 3) a.nrb[o] = (int)((op.nrows + S3_ROWS - 1) / S3_ROWS);
    }
    constexpr int VX = 16 / (int)sizeof(T);
    a.nbx = (int)((L.nx + 32 * VX - 1) / (32 * VX));
    a.src = g.src;
    a.wavelet = (const T*)sh->wavelet_dev;
    a.rec = g.rec;
    a.traces = (T*)sh->traces_dev;
    a.nt = nt;
    const int64_t cols = (int64_t)a.nbx * ((L.nz + 7) / 8);
    const unsigned gv = (unsigned)(cols + a.nrb[0] + a.nrb[1]), gp = (unsigned)(cols + a.nrb[2]);
    auto launch_step = [&](cudaStream_t st, bool prof) -> ib_status {
        auto v = [&]() {
            if (H == 1) k_stag_v2d<T, 1><<<gv, 256, 0, st>>>(a);
            else if (H == 2) k_stag_v2d<T, 2><<<gv, 256, 0, st>>>(a);
            else if (H == 3) k_stag_v2d<T, 3><<<gv, 256, 0, st>>>(a);
            else k_stag_v2d<T, 4><<<gv, 256, 0, st>>>(a);
        };
        auto pk = [&]() {
            if (H == 1) k_stag_p2d<T, 1><<<gp, 256, 0, st>>>(a);
            else if (H == 2) k_stag_p2d<T, 2><<<gp, 256, 0, st>>>(a);
            else if (H == 3) k_stag_p2d<T, 3><<<gp, 256, 0, st>>>(a);
            else k_stag_p2d<T, 4><<<gp, 256, 0, st>>>(a);
        };
        if (prof) {
            PROF_LAUNCH(kname<T>("stag_v2d_f32", "stag_v2d_f64"), st, { v(); });
            PROF_LAUNCH(kname<T>("stag_p2d_f32", "stag_p2d_f64"), st, { pk(); });
        } else {
            v();
            pk();
            ib_count_launch(kname<T>("stag_v2d_f32", "stag_v2d_f64"));
            ib_count_launch(kname<T>("stag_p2d_f32", "stag_p2d_f64"));
        }
        IB_CHECK_LAUNCH("staggered step");
        return IB_OK;
    };
    int* d_base;
    TRY(S.alloc(&d_base, 1, true));
    a.step_base = d_base;
    const int K = STAG_GRAPH_STEPS;
    const int nrep = (nt >= 2 * K && !getenv("IB_NO_GRAPH")) ? nt / K : 0;
    cudaStream_t cs = s;
    cudaEvent_t ready = nullptr;
    if (nrep) {
        // K steps (and the step-offset bump) as one graph, replayed nrep times on a side stream
        IB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        IB_CUDA(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
        IB_CUDA(cudaEventRecord(ready, s));
        IB_CUDA(cudaStreamWaitEvent(cs, ready, 0));
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        IB_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        ib_status st = IB_OK;
        for (int k = 0; k < K && st == IB_OK; ++k) {
            a.step = k;
            a.rec_step = k - 1;
            st = launch_step(cs, false);
        }
        k_add_step<<<1, 32, 0, cs>>>(d_base, K);
        cudaError_t ce = cudaStreamEndCapture(cs, &graph);
        if (st != IB_OK) return st;
        if (ce != cudaSuccess) return ib_cuda_fail(ce, "graph capture", __FILE__, __LINE__);
        IB_CUDA(cudaGraphInstantiate(&exec, graph, 0));
        for (int r = 0; r < nrep; ++r) {
            ProfToken tk = ib_prof_begin(kname<T>("stag_graph50_f32", "stag_graph50_f64"), cs);
            IB_CUDA(cudaGraphLaunch(exec, cs));
            ib_prof_end(tk, cs);
            if (probe)
                TRY(probe_rescale<T>(probe, r + 1, L.total, p, vx, vz, cs));
            for (int k = 0; k < K; ++k) {
                ib_count_launch(kname<T>("stag_v2d_f32", "stag_v2d_f64"));
                ib_count_launch(kname<T>("stag_p2d_f32", "stag_p2d_f64"));
            }
        }
        IB_CUDA(cudaStreamSynchronize(cs));
        cudaGraphExecDestroy(exec);
        cudaGraphDestroy(graph);
    }
    for (int k = 0; k < nt - nrep * K; ++k) {     // the remaining steps, offset by the graphs' bumps
        a.step = k;
        a.rec_step = k - 1;
        TRY(launch_step(cs, true));
        if (probe && (nrep * K + k + 1) % STAB_BLOCK == 0)
            TRY(probe_rescale<T>(probe, (nrep * K + k + 1) / STAB_BLOCK, L.total, p, vx, vz, cs));
    }
    if (g.rec.n) {
        k_receivers<T><<<grid1(g.rec.n, 256), 256, 0, cs>>>(g.rec, p, (T*)sh->traces_dev, nt, nt - 1);
        IB_CHECK_LAUNCH("k_receivers");
        ib_count_launch("setup");
    }
    if (!probe) TRY(check_finite<T>(L.total, p, vx, vz, cs));
    if (nrep) {
        IB_CUDA(cudaEventRecord(ready, cs));
        IB_CUDA(cudaStreamWaitEvent(s, ready, 0));
        IB_CUDA(cudaStreamSynchronize(cs));
        cudaEventDestroy(ready);
        cudaStreamDestroy(cs);
    }
    return IB_OK;
}

extern "C" ib_status ib_forward(const ib_table* tc, const ib_shot* sh, int32_t precision, double dt, int32_t nt,
                                void* ckpt, int32_t n_ckpt, void* stream) {
    ib_set_error("");
    TRY(check_shot(tc, sh, precision, dt, nt));
    ib_table* t = const_cast<ib_table*>(tc);
    cudaStream_t s = (cudaStream_t)stream;
    if (t->form == IB_SECOND_ORDER) {
        if (ckpt && n_ckpt < 1) {
            ib_set_error("n_ckpt must be >= 1");
            return IB_ERR_ARG;
        }
        return precision == 64 ? forward_2nd<double>(t, sh, dt, nt, ckpt, n_ckpt, s)
                               : forward_2nd<float>(t, sh, dt, nt, ckpt, n_ckpt, s);
    }
    if (ckpt) {
        ib_set_error("checkpoints are supported for the second-order form");
        return IB_ERR_STATE;
    }
    if (t->grid.ndim == 3)
        return precision == 64 ? forward_stag3<double>(t, sh, dt, nt, s) : forward_stag3<float>(t, sh, dt, nt, s);
    return precision == 64 ? forward_stag<double>(t, sh, dt, nt, s) : forward_stag<float>(t, sh, dt, nt, s);
}

// receiver injection rows: node -> (receiver, weight), regrouped on the host
template <typename T>
static ib_status build_injection(const PointSet<T>& rec, Scratch& S, AdjArgs<T>& a) {
    a.n_inj = 0;
    if (rec.n == 0) return IB_OK;
    std::vector<int64_t> idx(8 * (size_t)rec.n);
    std::vector<T> w(8 * (size_t)rec.n);
    IB_CUDA(cudaMemcpyAsync(idx.data(), rec.idx, 8 * idx.size(), cudaMemcpyDeviceToHost, S.s));
    IB_CUDA(cudaMemcpyAsync(w.data(), rec.w, sizeof(T) * w.size(), cudaMemcpyDeviceToHost, S.s));
    IB_CUDA(cudaStreamSynchronize(S.s));
    struct E {
        int64_t q;
        int64_t r;
        T w;
    };
    std::vector<E> es;
    for (int r = 0; r < rec.n; ++r)
        for (int c = 0; c < 8; ++c)
            if (w[8 * r + c] != (T)0) es.push_back({idx[8 * r + c], r, w[8 * r + c]});
    std::sort(es.begin(), es.end(), [](const E& a, const E& b) { return a.q != b.q ? a.q < b.q : a.r < b.r; });
    std::vector<int64_t> rows, ptr, col;
    std::vector<T> ww;
    for (size_t i = 0; i < es.size(); ++i) {
        if (i == 0 || es[i].q != es[i - 1].q) {
            rows.push_back(es[i].q);
            ptr.push_back((int64_t)i);
        }
        col.push_back(es[i].r);
        ww.push_back(es[i].w);
    }
    ptr.push_back((int64_t)es.size());
    if (rows.empty()) return IB_OK;
    int64_t *drows, *dptr, *dcol;
    T* dw;
    TRY(S.alloc(&drows, (int64_t)rows.size()));
    TRY(S.alloc(&dptr, (int64_t)ptr.size()));
    TRY(S.alloc(&dcol, (int64_t)col.size()));
    TRY(S.alloc(&dw, (int64_t)ww.size()));
    IB_CUDA(cudaMemcpyAsync(drows, rows.data(), 8 * rows.size(), cudaMemcpyHostToDevice, S.s));
    IB_CUDA(cudaMemcpyAsync(dptr, ptr.data(), 8 * ptr.size(), cudaMemcpyHostToDevice, S.s));
    IB_CUDA(cudaMemcpyAsync(dcol, col.data(), 8 * col.size(), cudaMemcpyHostToDevice, S.s));
    IB_CUDA(cudaMemcpyAsync(dw, ww.data(), sizeof(T) * ww.size(), cudaMemcpyHostToDevice, S.s));
    a.n_inj = (int64_t)rows.size();
    a.i_pad = drows;
    a.i_ptr = dptr;
    a.i_rec = dcol;
    a.i_w = dw;
    IB_CUDA(cudaStreamSynchronize(S.s));
    return IB_OK;
}

// Adjoint step arguments of one shot: coefficients marked at the nodes of the transposed rows
// and of the receiver injection, their lists and the map between them.
template <typename T>
static ib_status adj_setup(ib_table* t, const ib_shot* sh, double dt, int nt, const PointSet<T>& rec,
                           const PointSet<T>& src, const T* res, Fields& F, AdjArgs<T>& a) {
    Scratch& S = F.S;
    const Layout& L = t->L;
    IbOp& op = t->ops[0];
    TRY(ib_table_transpose(t, 0, S.s));
    memset(&a, 0, sizeof a);
    a.L = L;
    T c1u[4];
    stencil_weights<T>(t->opts.space_order, a.w2, c1u);
    T* Kh;
    int32_t* map;
    TRY(F.alloc(&Kh, L.total));
    TRY(F.alloc(&map, L.total));
    TRY(F.alloc(&a.grad, L.total));
    k_leap_coef<T><<<grid1(L.N, 256), 256, 0, S.s>>>(L, (const T*)sh->vel_dev, t->mask_pad[0], dt / t->grid.h, Kh);
    IB_CHECK_LAUNCH("k_leap_coef");
    ib_count_launch("setup");
    a.nt_rows = op.t_nrows;
    a.t_pad = op.t_row_pad;
    a.t_ptr = op.t_ptr;
    a.t_off = op.t_src_off;
    a.t_w = (const T*)(sizeof(T) == 8 ? (const void*)op.t_w64 : (const void*)op.t_w32);
    TRY(build_injection<T>(rec, S, a));
    if (a.nt_rows) k_map_nodes<T><<<grid1(a.nt_rows, 256), 256, 0, S.s>>>(a.nt_rows, a.t_pad, false, map, Kh);
    if (a.n_inj) k_map_nodes<T><<<grid1(a.n_inj, 256), 256, 0, S.s>>>(a.n_inj, a.i_pad, true, map, Kh);
    IB_CHECK_LAUNCH("k_map_nodes");
    ib_count_launch("setup");
    a.Kh = Kh;
    a.nodemap = map;
    a.res = res;
    a.nt = nt;
    a.src = src;
    a.wavelet = (const T*)sh->wavelet_dev;
    set_damping<T>(sh, dt, a.dw, a.da);
    return damp_field<T>(L, a.dw, a.da, true, F, &a.damp);
}

// Shape of an adjoint step over `points` grid points: one point a thread (zc = 0) or a march of
// 128 columns and zc rows a warp.  A march's block holds three quarters of the warps that an SM
// could and walks its rows one pair after the other, so few rows a warp (whose halo rows come
// from the L2) keep the SMs full and end together: marches of 32 rows took 232 us where the
// 64 x 8 tiles before them took about 170.  us per recompute and adjoint step of a batch, order 8
// (order 4 has the same best rows):
//   10^6 points          0.90   1.42   2.2    2.9    3.8    5.1    6.5    9.0   12.8   15.3
//   one point a thread     41     58     90    126    171    234    284    380    530    627
//   4 rows                 40     49     68     92    117    158    179    231    311    371
//   6 rows                 42     52     71     94    116    162    180    228    308    364
//   8 rows                 46     55     73     98    123    165    178    229    307    366
//   12 rows                57     62     83    105    131    174    189    235    315    373
//   32 rows               104    120    129    160    187    232    246    290    362    431
struct AdjShape {
    int zc;
};
static AdjShape adj_shape(int64_t points) {
    const int f = strip_switch();
    if (f == 0 || (f < 0 && points < 1200000)) return {0};
    return {points < 8000000 ? 6 : 8};
}
static int64_t adj_ntx(AdjShape p, const Layout& L) { return (L.nx + (p.zc ? 128 : 32) - 1) / (p.zc ? 128 : 32); }
static int64_t adj_blocks(AdjShape p, const Layout& L) {
    const int64_t rows = (int64_t)LEAP_WARPS * (p.zc ? p.zc : 1);
    return adj_ntx(p, L) * ((L.nz + rows - 1) / rows);
}
template <class F>
static void with_adj_shape(AdjShape p, int H, F f) {
    if (p.zc == 0) with_h<1, 1>(H, f);
    else with_h<4, 0>(H, f);
}

static void launch_adj2d(const AdjArgs<float>& a, AdjShape p, int H, unsigned grid, cudaStream_t s) {
    with_adj_shape(p, H, [&](auto h, auto vx, auto rz) {
        constexpr size_t sm = adj_smem<h.value, rz.value>();
        if (sm)
            cudaFuncSetAttribute(k_adj2d<float, h.value, vx.value, rz.value>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm);
        k_adj2d<float, h.value, vx.value, rz.value><<<grid, LEAP_THREADS, sm, s>>>(a, p.zc);
    });
}
static void launch_adj2d(const AdjArgs<double>& a, AdjShape, int H, unsigned grid, cudaStream_t s) {
    with_h<1, 1>(H, [&](auto h, auto, auto) { k_adj2d<double, h.value, 1, 1><<<grid, LEAP_THREADS, 0, s>>>(a, 0); });
}

template <typename T>
static ib_status adjoint_2nd(ib_table* t, const ib_shot* sh, double dt, int nt, const void* ckpt, int n_ckpt,
                             const T* res, T* grad_out, T* gw, cudaStream_t s) {
    const Layout& L = t->L;
    const int d = t->grid.ndim;
    if (d != 2) {
        ib_set_error("the adjoint is implemented in 2D");
        return IB_ERR_STATE;
    }
    const int M = t->opts.space_order;
    const int H = M / 2;
    Scratch S(s);
    T *Kh, *mu1, *mu2;
    TRY(S.alloc(&Kh, L.total, true));
    TRY(S.alloc(&mu1, L.total, true));
    TRY(S.alloc(&mu2, L.total, true));
    k_leap_coef<T><<<grid1(L.N, 256), 256, 0, s>>>(L, (const T*)sh->vel_dev, t->mask_pad[0], dt / t->grid.h, Kh);
    IB_CHECK_LAUNCH("k_leap_coef");
    ib_count_launch("setup");
    Geom<T> g;
    TRY(setup_points<T>(t, sh, dt * dt / pow(t->grid.h, d), S, g));
    AdjArgs<T> aa;
    Fields F(S);
    TRY(adj_setup<T>(t, sh, dt, nt, g.rec, g.src, res, F, aa));
    const int64_t seg = ckpt_seg(nt, n_ckpt);
    T* segbuf;
    TRY(S.alloc(&segbuf, (seg + 2) * L.total, true));
    if (gw) IB_CUDA(cudaMemsetAsync(gw, 0, sizeof(T) * nt, s));
    StepArgs<T> fa;
    memset(&fa, 0, sizeof fa);
    fa.L = L;
    {
        T c1u[4];
        stencil_weights<T>(M, fa.w2, c1u);
    }
    fa.Kh = Kh;
    fa.rows = row_list<T>(t->ops[0]);
    TRY(mark_rows<T>(fa.rows, Kh, s));
    fa.src = g.src;
    fa.wavelet = (const T*)sh->wavelet_dev;
    fa.rec.n = 0;
    fa.rec_step = -1;
    fa.nt = nt;
    set_damping<T>(sh, dt, fa.dw, fa.da);
    TRY(damp_field<T>(L, fa.dw, fa.da, false, F, &fa.damp));
    aa.gw = gw;
    const LeapShape fshape = leap_shape_shot(L, H);
    const AdjShape ashape = sizeof(T) == 8 ? AdjShape{0} : adj_shape(L.nx * L.nz);
    aa.ntx = adj_ntx(ashape, L);
    aa.nrb = row_blocks(aa.nt_rows + aa.n_inj, ashape.zc ? 0 : 1);
    const unsigned agrid = (unsigned)(aa.nrb + adj_blocks(ashape, L));
    const RunPlan plan = run_plan_unless_forced<T>(L, H);
    unsigned* bars;
    TRY(S.alloc(&bars, (int64_t)n_ckpt + 1, true));   // one per segment, then the error word
    T* mu_a = mu1;   // mu^{m+1}
    T* mu_b = mu2;   // mu^{m+2}
    for (int k = n_ckpt - 1; k >= 0; --k) {
        const int64_t c = (int64_t)k * seg;
        if (c >= nt) continue;
        const int64_t e = std::min<int64_t>(c + seg, nt);
        const T* slot = (const T*)ckpt + (int64_t)k * 2 * L.total;
        // segment slots j hold p^{c - 1 + j}
        IB_CUDA(cudaMemcpyAsync(segbuf, slot + L.total, sizeof(T) * L.total, cudaMemcpyDeviceToDevice, s));
        IB_CUDA(cudaMemcpyAsync(segbuf + L.total, slot, sizeof(T) * L.total, cudaMemcpyDeviceToDevice, s));
        bool refused = !plan.blocks;
        if (!refused) TRY(launch_run<T>(fa, plan, H, segbuf, segbuf, L.total, (int)c, (int)e, bars + k, (int*)(bars + n_ckpt), &refused, s));
        if (refused) for (int64_t n = c; n < e; ++n) {
            fa.p = segbuf + (n - c + 1) * L.total;
            fa.pm = segbuf + (n - c) * L.total;
            fa.out = segbuf + (n - c + 2) * L.total;
            fa.step = (int)n;
            launch_leap2d(fa, fshape, H, s);
            IB_CHECK_LAUNCH("recompute step");
        }
        for (int64_t m = e; m >= c + 1; --m) {
            aa.mu = mu_a;
            aa.mum = mu_b;
            aa.out = mu_b;
            aa.m = (int)m;
            aa.pm0 = segbuf + (m - c + 1) * L.total;
            aa.pm1 = segbuf + (m - c) * L.total;
            aa.pm2 = segbuf + (m - c - 1) * L.total;
            PROF_LAUNCH(kname<T>("adj2d_f32", "adj2d_f64"), s, { launch_adj2d(aa, ashape, H, agrid, s); });
            IB_CHECK_LAUNCH("adjoint step");
            std::swap(mu_a, mu_b);
        }
    }
    k_unpad_grad<T><<<grid1(L.N, 256), 256, 0, s>>>(L, aa.grad, aa.Kh, (T)(2.0 * dt / t->grid.h), grad_out);
    IB_CHECK_LAUNCH("k_unpad");
    ib_count_launch("setup");
    TRY(check_finite<T>(L.N, grad_out, (const T*)nullptr, (const T*)nullptr, s));
    int herr = 0;
    IB_CUDA(cudaMemcpyAsync(&herr, bars + n_ckpt, sizeof(int), cudaMemcpyDeviceToHost, s));
    IB_CUDA(cudaStreamSynchronize(s));
    if (herr) {
        ib_set_error("a bounded wait between the steps of a 2D run timed out");
        return IB_ERR_TIMEOUT;
    }
    return IB_OK;
}

extern "C" ib_status ib_adjoint(const ib_table* tc, const ib_shot* sh, int32_t precision, double dt, int32_t nt,
                                const void* ckpt, int32_t n_ckpt, const void* residual, void* grad_vel,
                                void* grad_wavelet, void* stream) {
    ib_set_error("");
    TRY(check_shot(tc, sh, precision, dt, nt, false));
    if (!ckpt || n_ckpt < 1 || !residual || !grad_vel) {
        ib_set_error("adjoint needs checkpoints, residual and gradient buffers");
        return IB_ERR_ARG;
    }
    ib_table* t = const_cast<ib_table*>(tc);
    if (t->form != IB_SECOND_ORDER) {
        ib_set_error("the adjoint is implemented for the second-order form");
        return IB_ERR_STATE;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (precision == 64)
        return adjoint_2nd<double>(t, sh, dt, nt, ckpt, n_ckpt, (const double*)residual, (double*)grad_vel,
                                   (double*)grad_wavelet, s);
    return adjoint_2nd<float>(t, sh, dt, nt, ckpt, n_ckpt, (const float*)residual, (float*)grad_vel,
                              (float*)grad_wavelet, s);
}

// ---------------------------------------------------------------------------
// batched shots: one launch per time step over the blocks of every shot, captured with all
// nt steps into one CUDA graph
// ---------------------------------------------------------------------------
static void launch_batch(const LeapShape& p, int H, const StepArgs<float>* args, const int64_t* tile0, const int32_t* shot_of,
                         int step, int seg, int64_t nblk, cudaStream_t s) {
    with_shape(p, H, [&](auto h, auto vx, auto rz) {
        constexpr size_t sm = leap_smem<h.value, rz.value>();
        if (sm > 48 * 1024)
            cudaFuncSetAttribute(k_leap2d_batch<h.value, vx.value, rz.value>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm);
        k_leap2d_batch<h.value, vx.value, rz.value>
            <<<(unsigned)nblk, LEAP_THREADS, sm, s>>>(args, tile0, shot_of, step, seg, p.zc);
    });
}

// the shape by the batch's size; IB_BATCH_SHAPE=<index into kShapes> fixes it instead
static ib_status batch_shape(int64_t points, int H, LeapShape* p) {
    *p = leap_shape(points, H);
    const char* forced = getenv("IB_BATCH_SHAPE");
    if (!forced || !*forced) return IB_OK;
    const int si = atoi(forced);
    if (si < 0 || si >= kNumShapes) {
        ib_set_error("IB_BATCH_SHAPE must name a shape index in [0, 10)");
        return IB_ERR_ARG;
    }
    *p = kShapes[si];
    return IB_OK;
}

struct BatchSetup {
    std::vector<StepArgs<float>> args;
    std::vector<int64_t> tile0;
    StepArgs<float>* d_args = nullptr;
    int64_t* d_tile0 = nullptr;
    int32_t* d_shot_of = nullptr;   // shot of each block
    int64_t nblk = 0;
};

static ib_status batch_prepare(ib_table* const* ts, const ib_shot* shots, int nshot, const LeapShape& p, double dt, int nt,
                               const std::vector<float*>& buf0, const std::vector<float*>& buf1,
                               const std::vector<float*>& Kh, const std::vector<Geom<float>>& geo, Fields& F,
                               BatchSetup& B) {
    Scratch& S = F.S;
    B.args.assign(nshot, StepArgs<float>());
    B.tile0.assign(nshot + 1, 0);
    for (int i = 0; i < nshot; ++i) {
        ib_table* t = ts[i];
        const Layout& L = t->L;
        StepArgs<float>& a = B.args[i];
        memset(&a, 0, sizeof a);
        a.L = L;
        float c1u[4];
        stencil_weights<float>(t->opts.space_order, a.w2, c1u);
        a.Kh = Kh[i];
        a.rows = row_list<float>(t->ops[0]);
        a.src = geo[i].src;
        a.wavelet = (const float*)shots[i].wavelet_dev;
        a.rec = geo[i].rec;
        a.traces = (float*)shots[i].traces_dev;
        a.nt = nt;
        a.buf0 = buf0[i];
        a.buf1 = buf1[i];
        set_damping<float>(&shots[i], dt, a.dw, a.da);
        TRY(damp_field<float>(L, a.dw, a.da, false, F, &a.damp));
        a.ntx = shape_ntx(p, L);
        a.nrb = row_blocks(a.rows.n, p.rz);
        B.tile0[i + 1] = B.tile0[i] + a.nrb + shape_blocks(p, L);
    }
    B.nblk = B.tile0[nshot];
    TRY(S.alloc(&B.d_args, nshot));
    TRY(S.alloc(&B.d_tile0, nshot + 1));
    IB_CUDA(cudaMemcpyAsync(B.d_args, B.args.data(), sizeof(StepArgs<float>) * nshot, cudaMemcpyHostToDevice, S.s));
    IB_CUDA(cudaMemcpyAsync(B.d_tile0, B.tile0.data(), 8 * (nshot + 1), cudaMemcpyHostToDevice, S.s));
    std::vector<int32_t> shot_of(B.nblk);
    for (int i = 0; i < nshot; ++i)
        for (int64_t b = B.tile0[i]; b < B.tile0[i + 1]; ++b) shot_of[b] = i;
    TRY(S.alloc(&B.d_shot_of, std::max<int64_t>(B.nblk, 1)));
    IB_CUDA(cudaMemcpyAsync(B.d_shot_of, shot_of.data(), 4 * B.nblk, cudaMemcpyHostToDevice, S.s));
    IB_CUDA(cudaStreamSynchronize(S.s));   // the host table goes out of scope
    return IB_OK;
}

static ib_status forward_batch_impl(const ib_table* const* tables, const ib_shot* shots, int32_t nshot,
                                    int32_t precision, double dt, int32_t nt, void* const* ckpts, int32_t n_ckpt,
                                    void* stream) {
    ib_set_error("");
    if (ckpts && n_ckpt < 1) {
        ib_set_error("n_ckpt must be >= 1");
        return IB_ERR_ARG;
    }
    if (!tables || !shots || nshot < 1) {
        ib_set_error("empty batch");
        return IB_ERR_ARG;
    }
    if (precision != 32) {
        ib_set_error("batched shots run in FP32");
        return IB_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<ib_table*> ts(nshot);
    int H = -1;
    for (int i = 0; i < nshot; ++i) {
        TRY(check_shot(tables[i], &shots[i], precision, dt, nt));
        ts[i] = const_cast<ib_table*>(tables[i]);
        if (ts[i]->form != IB_SECOND_ORDER || ts[i]->grid.ndim != 2) {
            ib_set_error("batched shots: 2D second-order tables only");
            return IB_ERR_STATE;
        }
        int h = ts[i]->opts.space_order / 2;
        if (H >= 0 && h != H) {
            ib_set_error("batched shots must share the space order");
            return IB_ERR_ARG;
        }
        H = h;
    }
    Scratch S(s);
    std::vector<float*> b0(nshot), b1(nshot), Kh(nshot);
    std::vector<Geom<float>> geo(nshot);
    int64_t total = 0;
    // all shots' fields in one allocation, zeroed at once (48 damped shots of 400-1200 squared, 6
    // steps, set-up included: 9.7 ms with four allocations a shot, 8.7 with one for all)
    Fields F(S);
    int64_t need = 0;
    for (int i = 0; i < nshot; ++i) need += (shot_damped(&shots[i]) ? 4 : 3) * Fields::bytes(ts[i]->L.total, 4);
    TRY(F.reserve(need));
    for (int i = 0; i < nshot; ++i) {
        const Layout& L = ts[i]->L;
        TRY(F.alloc(&b0[i], L.total));
        TRY(F.alloc(&b1[i], L.total));
        TRY(F.alloc(&Kh[i], L.total));
        k_leap_coef<float><<<grid1(L.N, 256), 256, 0, s>>>(L, (const float*)shots[i].vel_dev, ts[i]->mask_pad[0],
                                                           dt / ts[i]->grid.h, Kh[i]);
        IB_CHECK_LAUNCH("k_leap_coef");
        ib_count_launch("setup");
        TRY(mark_rows<float>(row_list<float>(ts[i]->ops[0]), Kh[i], s));
        TRY(setup_points<float>(ts[i], &shots[i], dt * dt / pow(ts[i]->grid.h, 2), S, geo[i]));
        total += L.N;
    }
    LeapShape best;
    TRY(batch_shape(total, H, &best));
    BatchSetup B;
    TRY(batch_prepare(ts.data(), shots, nshot, best, dt, nt, b0, b1, Kh, geo, F, B));
    // checkpoint copies (ib_forward's layout: slot k = [p^{k seg}, p^{k seg - 1}])
    ShotCopy<float>* d_items = nullptr;
    int64_t seg = 0, maxtot = 0;
    if (ckpts) {
        std::vector<ShotCopy<float>> items(nshot);
        for (int i = 0; i < nshot; ++i) {
            if (!ckpts[i]) {
                ib_set_error("null checkpoint buffer");
                return IB_ERR_ARG;
            }
            items[i] = {b0[i], b1[i], (float*)ckpts[i], ts[i]->L.total};
            maxtot = std::max(maxtot, ts[i]->L.total);
        }
        TRY(S.alloc(&d_items, nshot));
        IB_CUDA(cudaMemcpyAsync(d_items, items.data(), sizeof(ShotCopy<float>) * nshot, cudaMemcpyHostToDevice, s));
        IB_CUDA(cudaStreamSynchronize(s));
        seg = ckpt_seg(nt, n_ckpt);
    }
    const dim3 cgrid((unsigned)std::min<int64_t>((maxtot + 255) / 256, 256), (unsigned)nshot);
    // ---- all nt steps as one captured graph
    cudaStream_t cs;
    IB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaEvent_t ready;
    IB_CUDA(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    IB_CUDA(cudaEventRecord(ready, s));
    IB_CUDA(cudaStreamWaitEvent(cs, ready, 0));
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    IB_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    for (int n = 0; n < nt; ++n) {
        if (d_items && n % seg == 0) k_ckpt_batch<float><<<cgrid, 256, 0, cs>>>(d_items, n, (int)(n / seg));
        launch_batch(best, H, B.d_args, B.d_tile0, B.d_shot_of, n, -1, B.nblk, cs);
    }
    cudaError_t ce = cudaStreamEndCapture(cs, &graph);
    if (ce != cudaSuccess) return ib_cuda_fail(ce, "graph capture", __FILE__, __LINE__);
    IB_CUDA(cudaGraphInstantiate(&exec, graph, 0));
    {
        ProfToken tk = ib_prof_begin("leap2d_batch_graph_f32", cs);
        IB_CUDA(cudaGraphLaunch(exec, cs));
        ib_prof_end(tk, cs);
        for (int n = 0; n < nt; ++n) ib_count_launch("leap2d_batch_f32");
    }
    // final receivers per shot
    for (int i = 0; i < nshot; ++i) {
        if (!geo[i].rec.n) continue;
        float* cur = (nt & 1) ? b1[i] : b0[i];
        k_receivers<float><<<grid1(geo[i].rec.n, 256), 256, 0, cs>>>(geo[i].rec, cur, (float*)shots[i].traces_dev,
                                                                      nt, nt - 1);
        ib_count_launch("setup");
    }
    IB_CHECK_LAUNCH("k_receivers");
    for (int i = 0; i < nshot; ++i) TRY(check_finite<float>(ts[i]->L.total, b0[i], b1[i], (const float*)nullptr, cs));
    IB_CUDA(cudaEventRecord(ready, cs));
    IB_CUDA(cudaStreamWaitEvent(s, ready, 0));
    IB_CUDA(cudaStreamSynchronize(cs));
    cudaGraphExecDestroy(exec);
    cudaGraphDestroy(graph);
    cudaEventDestroy(ready);
    cudaStreamDestroy(cs);
    return IB_OK;
}

extern "C" ib_status ib_forward_batch(const ib_table* const* tables, const ib_shot* shots, int32_t nshot,
                                      int32_t precision, double dt, int32_t nt, void* stream) {
    return forward_batch_impl(tables, shots, nshot, precision, dt, nt, nullptr, 0, stream);
}

extern "C" ib_status ib_forward_batch_ckpt(const ib_table* const* tables, const ib_shot* shots, int32_t nshot,
                                           int32_t precision, double dt, int32_t nt, void* const* ckpts,
                                           int32_t n_ckpt, void* stream) {
    if (!ckpts) {
        ib_set_error("null checkpoint array");
        return IB_ERR_ARG;
    }
    return forward_batch_impl(tables, shots, nshot, precision, dt, nt, ckpts, n_ckpt, stream);
}

// ---------------------------------------------------------------------------
// batched adjoint: every shot's segments in lockstep, one graph for the whole
// backward pass (segment restore, batched recompute steps, batched adjoint steps)
// ---------------------------------------------------------------------------
// block maps: tile0 / shot_of of the adjoint steps, stile0 / sshot_of of the recompute steps
static void launch_adj_batch(int H, const LeapShape& fshape, AdjShape ashape, const StepArgs<float>* fargs, const AdjBatch<float>* aargs,
                             const ShotCopy<float>* rst, const int64_t* tile0, const int32_t* shot_of, int64_t nblk,
                             const int64_t* stile0, const int32_t* sshot_of, int64_t nsblk, dim3 cgrid, int nt, int64_t c,
                             int64_t e, int k, cudaStream_t s) {
    k_seg_restore_batch<float><<<cgrid, 256, 0, s>>>(rst, k);
    for (int64_t n = c; n < e; ++n) launch_batch(fshape, H, fargs, stile0, sshot_of, (int)n, (int)(n - c), nsblk, s);
    for (int64_t m = e; m >= c + 1; --m)
        with_adj_shape(ashape, H, [&](auto h, auto vx, auto rz) {
            constexpr size_t sm = adj_smem<h.value, rz.value>();
            if (sm)
                cudaFuncSetAttribute(k_adj2d_batch<h.value, vx.value, rz.value>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sm);
            k_adj2d_batch<h.value, vx.value, rz.value><<<(unsigned)nblk, LEAP_THREADS, sm, s>>>(
                aargs, tile0, shot_of, (int)m, (int)(m - c), nt, ashape.zc);
        });
}

extern "C" ib_status ib_adjoint_batch(const ib_table* const* tables, const ib_shot* shots, int32_t nshot,
                                      int32_t precision, double dt, int32_t nt, const void* const* ckpts,
                                      int32_t n_ckpt, const void* const* residuals, void* const* grads,
                                      void* stream) {
    ib_set_error("");
    if (!tables || !shots || nshot < 1 || !ckpts || !residuals || !grads || n_ckpt < 1) {
        ib_set_error("batched adjoint needs tables, shots, checkpoints, residuals and gradients");
        return IB_ERR_ARG;
    }
    if (precision != 32) {
        ib_set_error("batched shots run in FP32");
        return IB_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<ib_table*> ts(nshot);
    int H = -1;
    for (int i = 0; i < nshot; ++i) {
        TRY(check_shot(tables[i], &shots[i], precision, dt, nt, false));
        ts[i] = const_cast<ib_table*>(tables[i]);
        if (ts[i]->form != IB_SECOND_ORDER || ts[i]->grid.ndim != 2) {
            ib_set_error("batched adjoint: 2D second-order tables only");
            return IB_ERR_STATE;
        }
        if (!ckpts[i] || !residuals[i] || !grads[i]) {
            ib_set_error("null checkpoint, residual or gradient buffer");
            return IB_ERR_ARG;
        }
        const int h = ts[i]->opts.space_order / 2;
        if (H >= 0 && h != H) {
            ib_set_error("batched shots must share the space order");
            return IB_ERR_ARG;
        }
        H = h;
    }
    const int64_t seg = ckpt_seg(nt, n_ckpt);
    Scratch S(s);
    std::vector<StepArgs<float>> fargs(nshot);
    std::vector<AdjBatch<float>> aargs(nshot);
    std::vector<ShotCopy<float>> rst(nshot);
    std::vector<int64_t> tile0(nshot + 1, 0), stile0(nshot + 1, 0);
    int64_t points = 0;
    for (int i = 0; i < nshot; ++i) points += ts[i]->L.N;
    LeapShape fshape;
    TRY(batch_shape(points, H, &fshape));
    const AdjShape ashape = adj_shape(points);
    int64_t maxtot = 0;
    // all shots' fields in one allocation: coefficients, multipliers, gradient and node map, the
    // absorbing layer's two fields, and the segment
    Fields F(S);
    int64_t need = 0;
    for (int i = 0; i < nshot; ++i)
        need += (shot_damped(&shots[i]) ? 8 : 6) * Fields::bytes(ts[i]->L.total, 4) +
                Fields::bytes((seg + 2) * ts[i]->L.total, 4);
    TRY(F.reserve(need));
    for (int i = 0; i < nshot; ++i) {
        ib_table* t = ts[i];
        const Layout& L = t->L;
        float *Kh, *mu1, *mu2, *segbuf;
        TRY(F.alloc(&Kh, L.total));
        TRY(F.alloc(&mu1, L.total));
        TRY(F.alloc(&mu2, L.total));
        TRY(F.alloc(&segbuf, (seg + 2) * L.total));
        k_leap_coef<float><<<grid1(L.N, 256), 256, 0, s>>>(L, (const float*)shots[i].vel_dev, t->mask_pad[0],
                                                           dt / t->grid.h, Kh);
        IB_CHECK_LAUNCH("k_leap_coef");
        ib_count_launch("setup");
        Geom<float> g;
        TRY(setup_points<float>(t, &shots[i], dt * dt / pow(t->grid.h, 2), S, g));
        StepArgs<float>& fa = fargs[i];
        memset(&fa, 0, sizeof fa);
        fa.L = L;
        float c1u[4];
        stencil_weights<float>(t->opts.space_order, fa.w2, c1u);
        fa.Kh = Kh;
        fa.rows = row_list<float>(t->ops[0]);
        TRY(mark_rows<float>(fa.rows, Kh, s));
        fa.src = g.src;
        fa.wavelet = (const float*)shots[i].wavelet_dev;
        fa.rec.n = 0;
        fa.rec_step = -1;
        fa.nt = nt;
        set_damping<float>(&shots[i], dt, fa.dw, fa.da);
        TRY(damp_field<float>(L, fa.dw, fa.da, false, F, &fa.damp));
        fa.buf0 = segbuf;
        fa.ntx = shape_ntx(fshape, L);
        fa.nrb = row_blocks(fa.rows.n, fshape.rz);
        AdjArgs<float>& aa = aargs[i].a;
        TRY(adj_setup<float>(t, &shots[i], dt, nt, g.rec, g.src, (const float*)residuals[i], F, aa));
        aa.ntx = adj_ntx(ashape, L);
        aa.nrb = row_blocks(aa.nt_rows + aa.n_inj, ashape.zc ? 0 : 1);
        aargs[i].mu1 = mu1;
        aargs[i].mu2 = mu2;
        aargs[i].seg = segbuf;
        rst[i] = {(const float*)ckpts[i], nullptr, segbuf, L.total};
        tile0[i + 1] = tile0[i] + aa.nrb + adj_blocks(ashape, L);
        stile0[i + 1] = stile0[i] + fa.nrb + shape_blocks(fshape, L);
        maxtot = std::max(maxtot, L.total);
    }
    const int64_t nblk = tile0[nshot], nsblk = stile0[nshot];
    std::vector<int32_t> shot_of(nblk), sshot_of(nsblk);
    for (int i = 0; i < nshot; ++i) {
        for (int64_t b = tile0[i]; b < tile0[i + 1]; ++b) shot_of[b] = i;
        for (int64_t b = stile0[i]; b < stile0[i + 1]; ++b) sshot_of[b] = i;
    }
    StepArgs<float>* d_f;
    AdjBatch<float>* d_a;
    ShotCopy<float>* d_r;
    int64_t *d_t0, *d_st0;
    int32_t *d_so, *d_sso;
    TRY(S.alloc(&d_f, nshot));
    TRY(S.alloc(&d_a, nshot));
    TRY(S.alloc(&d_r, nshot));
    TRY(S.alloc(&d_t0, nshot + 1));
    TRY(S.alloc(&d_so, std::max<int64_t>(nblk, 1)));
    TRY(S.alloc(&d_st0, nshot + 1));
    TRY(S.alloc(&d_sso, std::max<int64_t>(nsblk, 1)));
    IB_CUDA(cudaMemcpyAsync(d_st0, stile0.data(), 8 * (nshot + 1), cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaMemcpyAsync(d_sso, sshot_of.data(), 4 * nsblk, cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaMemcpyAsync(d_f, fargs.data(), sizeof(StepArgs<float>) * nshot, cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaMemcpyAsync(d_a, aargs.data(), sizeof(AdjBatch<float>) * nshot, cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaMemcpyAsync(d_r, rst.data(), sizeof(ShotCopy<float>) * nshot, cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaMemcpyAsync(d_t0, tile0.data(), 8 * (nshot + 1), cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaMemcpyAsync(d_so, shot_of.data(), 4 * nblk, cudaMemcpyHostToDevice, s));
    IB_CUDA(cudaStreamSynchronize(s));   // the host tables go out of scope
    const dim3 cgrid((unsigned)std::min<int64_t>((maxtot + 255) / 256, 256), (unsigned)nshot);
    // ---- the whole backward pass as one captured graph
    cudaStream_t cs;
    IB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaEvent_t ready;
    IB_CUDA(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    IB_CUDA(cudaEventRecord(ready, s));
    IB_CUDA(cudaStreamWaitEvent(cs, ready, 0));
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    IB_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    int64_t nadj = 0;
    for (int k = n_ckpt - 1; k >= 0; --k) {
        const int64_t c = (int64_t)k * seg;
        if (c >= nt) continue;
        const int64_t e = std::min<int64_t>(c + seg, nt);
        launch_adj_batch(H, fshape, ashape, d_f, d_a, d_r, d_t0, d_so, nblk, d_st0, d_sso, nsblk, cgrid, nt, c, e, k, cs);
        nadj += e - c;
    }
    cudaError_t ce = cudaStreamEndCapture(cs, &graph);
    if (ce != cudaSuccess) return ib_cuda_fail(ce, "graph capture", __FILE__, __LINE__);
    ce = cudaGraphInstantiate(&exec, graph, 0);
    if (ce != cudaSuccess) {
        cudaGraphDestroy(graph);
        return ib_cuda_fail(ce, "graph instantiate", __FILE__, __LINE__);
    }
    {
        ProfToken tk = ib_prof_begin("adj2d_batch_graph_f32", cs);
        IB_CUDA(cudaGraphLaunch(exec, cs));
        ib_prof_end(tk, cs);
        for (int64_t q = 0; q < nadj; ++q) {
            ib_count_launch("adj2d_batch_f32");
            ib_count_launch("leap2d_batch_seg_f32");
        }
    }
    for (int i = 0; i < nshot; ++i) {
        const Layout& L = ts[i]->L;
        k_unpad_grad<float><<<grid1(L.N, 256), 256, 0, cs>>>(L, aargs[i].a.grad, aargs[i].a.Kh,
                                                             (float)(2.0 * dt / ts[i]->grid.h), (float*)grads[i]);
        ib_count_launch("setup");
        TRY(check_finite<float>(L.N, (const float*)grads[i], (const float*)nullptr, (const float*)nullptr, cs));
    }
    IB_CHECK_LAUNCH("k_unpad");
    IB_CUDA(cudaEventRecord(ready, cs));
    IB_CUDA(cudaStreamWaitEvent(s, ready, 0));
    IB_CUDA(cudaStreamSynchronize(cs));
    cudaGraphExecDestroy(exec);
    cudaGraphDestroy(graph);
    cudaEventDestroy(ready);
    cudaStreamDestroy(cs);
    return IB_OK;
}

// the grid barrier with a target one arrival too high (every block gives up), and with the right one
static ib_status selftest_barrier(Scratch& S, bool* ok) {
    unsigned* w;
    TRY(S.alloc(&w, 4, true));
    for (int i = 0; i < 2; ++i) {
        unsigned* bar = w + i;
        unsigned target = i ? 4 : 5;
        uint64_t limit = 20000000ull;
        int* gave_up = (int*)(w + 2 + i);
        void* args[] = {&bar, &target, &limit, &gave_up};
        IB_CUDA(cudaLaunchCooperativeKernel((const void*)k_barrier_selftest, dim3(4), dim3(64), args, 0, S.s));
    }
    int h[2] = {0, 0};
    IB_CUDA(cudaMemcpyAsync(h, w + 2, sizeof h, cudaMemcpyDeviceToHost, S.s));
    IB_CUDA(cudaStreamSynchronize(S.s));
    *ok = h[0] == 4 && h[1] == 0;
    return IB_OK;
}

extern "C" ib_status ib_selftest_bounded_wait(void* stream) {
    ib_set_error("");
    cudaStream_t s = (cudaStream_t)stream;
    Scratch S(s);
    int* err;
    TRY(S.alloc(&err, 1, true));
    k_wait_selftest<<<1, 32, 0, s>>>(err);
    IB_CHECK_LAUNCH("k_wait_selftest");
    int h = 0;
    IB_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    IB_CUDA(cudaStreamSynchronize(s));
    bool barrier = false;
    TRY(selftest_barrier(S, &barrier));
    if (h && barrier) {
        ib_set_error("bounded device waits gave up (self-test: expected): copy wait, grid barrier");
        return IB_ERR_TIMEOUT;
    }
    ib_set_error(h ? "the grid barrier's bound did not work" : "the copy wait's bound did not work");
    return IB_OK;
}

extern "C" ib_status ib_sync_status(void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return ib_cuda_fail(e, "stream", __FILE__, __LINE__);
    e = cudaGetLastError();
    if (e != cudaSuccess) return ib_cuda_fail(e, "device", __FILE__, __LINE__);
    int word = 0;
    IB_CUDA(cudaMemcpyFromSymbolAsync(&word, g_dev_status, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
    IB_CUDA(cudaStreamSynchronize(s));
    if (word) {
        const int zero = 0;
        IB_CUDA(cudaMemcpyToSymbolAsync(g_dev_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s));
        IB_CUDA(cudaStreamSynchronize(s));
        if (word & STATUS_TIMEOUT) {
            ib_set_error("a bounded wait between the steps of a 2D run timed out");
            return IB_ERR_TIMEOUT;
        }
        ib_set_error("non-finite values (NaN/Inf) in the final wavefield or gradient of a run on this device: "
                     "the scheme is unstable for that model and time step");
        return IB_ERR_UNSTABLE;
    }
    return IB_OK;
}

extern "C" ib_status ib_stability(const ib_table* tc, const ib_shot* shot, int32_t precision, double dt,
                                  int32_t n_steps, uint64_t seed, double max_gain, double* growth, void* stream) {
    ib_set_error("");
    if (!tc || !shot || !shot->vel_dev || !growth || (precision != 32 && precision != 64) || !(dt > 0.0) ||
        n_steps < 1 || !(max_gain > 1.0)) {
        ib_set_error("ib_stability: table, shot with velocity and output required; precision 32 or 64, dt > 0, "
                     "n_steps >= 1, max_gain > 1");
        return IB_ERR_ARG;
    }
    ib_table* t = const_cast<ib_table*>(tc);
    if (t->form != IB_SECOND_ORDER && t->grid.ndim != 2) {
        ib_set_error("ib_stability: the staggered form is implemented in 2D");
        return IB_ERR_STATE;
    }
    cudaStream_t s = (cudaStream_t)stream;
    // whole renormalisation blocks, an even number of them
    const int nblk = std::max(2, ((n_steps + STAB_BLOCK - 1) / STAB_BLOCK + 1) / 2 * 2);
    const int nt = nblk * STAB_BLOCK;
    Scratch S(s);
    Probe pr;
    pr.seed = seed;
    pr.nslot = nblk + 1;
    TRY(S.alloc(&pr.sums, pr.nslot, true));
    TRY(S.alloc(&pr.logs, pr.nslot, true));
    ib_shot sh;
    memset(&sh, 0, sizeof sh);
    sh.vel_dev = shot->vel_dev;
    sh.rho_dev = shot->rho_dev;
    sh.damp_eta = shot->damp_eta;
    sh.damp_width = shot->damp_width;
    TRY(check_shot(tc, &sh, precision, dt, n_steps));
    if (t->form == IB_SECOND_ORDER)
        TRY(precision == 64 ? forward_2nd<double>(t, &sh, dt, nt, nullptr, 0, s, &pr)
                            : forward_2nd<float>(t, &sh, dt, nt, nullptr, 0, s, &pr));
    else
        TRY(precision == 64 ? forward_stag<double>(t, &sh, dt, nt, s, &pr)
                            : forward_stag<float>(t, &sh, dt, nt, s, &pr));
    std::vector<double> logs(pr.nslot);
    IB_CUDA(cudaMemcpyAsync(logs.data(), pr.logs, sizeof(double) * pr.nslot, cudaMemcpyDeviceToHost, s));
    IB_CUDA(cudaStreamSynchronize(s));
    // per-step growth over the second half of the blocks (the first half lets the
    // dominant mode emerge from the random start)
    double acc = 0.0;
    for (int k = nblk / 2 + 1; k <= nblk; ++k) acc += logs[k];
    const double rate = acc / (double)((nblk - nblk / 2) * STAB_BLOCK);
    *growth = std::isfinite(rate) ? exp(rate) : INFINITY;
    if (!std::isfinite(rate) || rate * (double)n_steps > log(max_gain)) {
        char buf[256];
        snprintf(buf, sizeof buf,
                 "ib_stability: per-step growth %.6f amplifies an unstable mode by %.3g over %d steps "
                 "(limit %.3g)", *growth, std::isfinite(rate) ? exp(rate * (double)n_steps) : INFINITY, n_steps,
                 max_gain);
        ib_set_error(buf);
        return IB_ERR_UNSTABLE;
    }
    return IB_OK;
}

// ---------------------------------------------------------------------------
// ib_forward_noalloc: the 2D second-order FP32 forward with its scratch in a
// file-scope device array instead of stream-ordered allocations, for callers
// that may not allocate device memory (see include/ib.h).
// ---------------------------------------------------------------------------
#define IB_NOALLOC_SCRATCH_BYTES (64ll << 20)

static __device__ __align__(256) unsigned char g_noalloc_scratch[IB_NOALLOC_SCRATCH_BYTES + 256];   // + the run's barrier word

static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[64] = {nullptr};

// Device address of the static scratch for the current device.  Outside stream
// capture it is looked up on every call (a device reset or a new primary
// context reloads the module and can move the array); while `s` is capturing,
// the address remembered from the last uncaptured call on this device is used,
// so the first call on a device must come before any capture.
static ib_status noalloc_scratch(cudaStream_t s, unsigned char** out) {
    int dev = 0;
    IB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        ib_set_error("device index out of range for the static scratch");
        return IB_ERR_ARG;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    IB_CUDA(cudaStreamIsCapturing(s, &cap));
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (cap == cudaStreamCaptureStatusNone) {
        void* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess) return ib_cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)", __FILE__, __LINE__);
        g_noalloc_ptr[dev] = ptr;
    } else if (!g_noalloc_ptr[dev]) {
        ib_set_error("ib_forward_noalloc: the first call on a device must not be captured");
        return IB_ERR_STATE;
    }
    *out = (unsigned char*)g_noalloc_ptr[dev];
    return IB_OK;
}

static int64_t align256(int64_t b) { return (b + 255) & ~(int64_t)255; }

extern "C" ib_status ib_forward_noalloc(const ib_table* tc, const ib_shot* sh, double dt, int32_t nt, void* stream) {
    ib_set_error("");
    TRY(check_shot(tc, sh, 32, dt, nt));
    ib_table* t = const_cast<ib_table*>(tc);
    if (t->form != IB_SECOND_ORDER || t->grid.ndim != 2) {
        ib_set_error("ib_forward_noalloc: 2D second-order tables only");
        return IB_ERR_STATE;
    }
    if (shot_damped(sh)) {
        ib_set_error("ib_forward_noalloc: no absorbing layer");
        return IB_ERR_STATE;
    }
    const Layout& L = t->L;
    const int64_t field = align256(sizeof(float) * L.total);
    const int64_t srcb = align256(8 * (int64_t)sh->nsrc * (8 + 4));
    const int64_t recb = align256(8 * (int64_t)sh->nrec * (8 + 4));
    const int64_t need = 3 * field + 2 * srcb + 2 * recb + 4 * 256;
    if (need > IB_NOALLOC_SCRATCH_BYTES) {
        char buf[200];
        snprintf(buf, sizeof buf, "ib_forward_noalloc: needs %lld bytes of scratch, the static limit is %lld",
                 (long long)need, (long long)IB_NOALLOC_SCRATCH_BYTES);
        ib_set_error(buf);
        return IB_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    unsigned char* base = nullptr;
    TRY(noalloc_scratch(s, &base));
    int64_t off = 0;
    auto carve = [&](int64_t bytes) {
        unsigned char* p = base + off;
        off += align256(bytes);
        return p;
    };
    float* p0 = (float*)carve(sizeof(float) * L.total);
    float* p1 = (float*)carve(sizeof(float) * L.total);
    float* Kh = (float*)carve(sizeof(float) * L.total);
    int64_t* si = (int64_t*)carve(8 * 8 * (int64_t)std::max(sh->nsrc, 1));
    float* sw = (float*)carve(4 * 8 * (int64_t)std::max(sh->nsrc, 1));
    int64_t* ri = (int64_t*)carve(8 * 8 * (int64_t)std::max(sh->nrec, 1));
    float* rw = (float*)carve(4 * 8 * (int64_t)std::max(sh->nrec, 1));
    unsigned* bar = (unsigned*)(base + IB_NOALLOC_SCRATCH_BYTES);
    IB_CUDA(cudaMemsetAsync(bar, 0, 256, s));
    // every call starts from zero wavefields and a zero padding ring
    IB_CUDA(cudaMemsetAsync(p0, 0, sizeof(float) * L.total, s));
    IB_CUDA(cudaMemsetAsync(p1, 0, sizeof(float) * L.total, s));
    IB_CUDA(cudaMemsetAsync(Kh, 0, sizeof(float) * L.total, s));
    k_leap_coef<float><<<grid1(L.N, 256), 256, 0, s>>>(L, (const float*)sh->vel_dev, t->mask_pad[0], dt / t->grid.h,
                                                       Kh);
    if (sh->nsrc)
        k_interp_setup<float><<<grid1(sh->nsrc, 64), 64, 0, s>>>(sh->nsrc, sh->src_dev, 2, 1.0 / t->grid.h, L,
                                                                  t->mask_pad[0], dt * dt / (t->grid.h * t->grid.h),
                                                                  si, sw);
    if (sh->nrec)
        k_interp_setup<float><<<grid1(sh->nrec, 64), 64, 0, s>>>(sh->nrec, sh->rec_dev, 2, 1.0 / t->grid.h, L,
                                                                  t->mask_pad[0], 1.0, ri, rw);
    IB_CHECK_LAUNCH("ib_forward_noalloc setup");
    const int M = t->opts.space_order;
    const int H = M / 2;
    StepArgs<float> a;
    memset(&a, 0, sizeof a);
    a.L = L;
    {
        float c1u[4];
        stencil_weights<float>(M, a.w2, c1u);
    }
    a.Kh = Kh;
    a.src = {sh->nsrc, si, sw};
    a.wavelet = (const float*)sh->wavelet_dev;
    a.rec = {sh->nrec, ri, rw};
    a.traces = (float*)sh->traces_dev;
    a.nt = nt;
    a.rows = row_list<float>(t->ops[0]);
    TRY(mark_rows<float>(a.rows, Kh, s));
    const LeapShape shape = leap_shape(L.nx * L.nz, H);
    float* cur = p0;
    float* prev = p1;
    const RunPlan plan = run_plan<float>(L, H);
    bool refused = !plan.blocks;
    if (!refused) TRY(launch_run<float>(a, plan, H, cur, prev, 0, 0, nt, bar, nullptr, &refused, s));
    if (!refused && (nt & 1)) std::swap(cur, prev);
    for (int n = refused ? 0 : nt; n < nt; ++n) {
        a.p = cur;
        a.pm = prev;
        a.out = prev;
        a.step = n;
        a.rec_step = n - 1;
        launch_leap2d(a, shape, H, s);
        IB_CHECK_LAUNCH("ib_forward_noalloc step");
        std::swap(cur, prev);
    }
    if (sh->nrec)
        k_receivers<float><<<grid1(sh->nrec, 256), 256, 0, s>>>(a.rec, cur, (float*)sh->traces_dev, nt, nt - 1);
    IB_CHECK_LAUNCH("ib_forward_noalloc receivers");
    return IB_OK;
}
