// 2D second-order steps: the leapfrog step (one shot, many shots, checkpoint segments) and
// the adjoint step.
//
// A launch has two kinds of blocks.
//   Column blocks.  Burst: a thread owns VX adjacent columns of RZ rows and loads everything
// with VX-wide vectors straight from memory (its rows, the vectors left and right of them for
// the x neighbours, p_prev and K), one memory latency per step.  March: a warp owns 128 columns
// and walks down zc rows, two at a time, over a ring of rows of its own in shared memory that
// cp.async fills ahead (no barrier between warps), four columns a lane in 16-byte vectors and
// packed pairs.  The staged tiles and strips that these replace spent 120 thread instructions
// a point and were bound by their issue; the march spends about 45 and is bound by memory:
// 8192 x 4096, order 8: 134 -> 95 us a step, 0.83 of copy bandwidth.
//   Row blocks: the immersed-boundary rows, 8 lanes each: a lane takes one of the 2H stencil
// pairs (H <= 4) and every 8th correction entry, and the row's whole update is done there.
// Column blocks leave those nodes out; they carry the sign bit of K as a mark.  So a row's
// corrections need no atomics, and run beside the bulk of the step instead of between two
// barriers of its surface tiles.
//
// 48 damped shots of 400-1200 squared, order 8: 171 -> 135 us a step; 24 gradients of such
// shots: 99 -> 75 ms; one of 613 x 487, order 4: 8.4 -> 4.7 ms.
#pragma once

__device__ __forceinline__ uint64_t global_ns();

template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

template <typename T, int VX>
struct Vec;
template <> struct Vec<float, 1> { typedef float type; };
template <> struct Vec<float, 2> { typedef float2 type; };
template <> struct Vec<float, 4> { typedef float4 type; };
template <> struct Vec<double, 1> { typedef double type; };
template <> struct Vec<double, 2> { typedef double2 type; };

template <typename T, int VX>
__device__ __forceinline__ void ldv(T (&d)[VX], const T* p) {
    typedef typename Vec<T, VX>::type V;
    *reinterpret_cast<V*>(&d[0]) = *reinterpret_cast<const V*>(p);
}
template <typename T, int VX>
__device__ __forceinline__ void stv(T* p, const T (&d)[VX]) {
    typedef typename Vec<T, VX>::type V;
    *reinterpret_cast<V*>(p) = *reinterpret_cast<const V*>(&d[0]);
}

// a node that a row block updates: the sign bit of its coefficient
__device__ __forceinline__ bool marked(float k) { return __float_as_int(k) < 0; }
__device__ __forceinline__ bool marked(double k) { return __double2hiint(k) < 0; }

// absorbing-layer coefficient of a 2D node (damp_a in 32-bit indices)
template <typename T>
__device__ __forceinline__ T damp_a2(int nx, int nz, int dw, T da, int x, int z) {
    const int dx = max(max(dw - x, x - (nx - 1 - dw)), 0), dz = max(z - (nz - 1 - dw), 0);
    const int64_t d2 = (int64_t)dx * dx + (int64_t)dz * dz;
    if (d2 == 0) return (T)0;
    const T r = (T)d2 / (T)((int64_t)dw * dw);
    return da * (r < (T)1 ? r : (T)1);
}

// Laplacian at window element i (HX = centre of the window): in FP32 the difference form
// sum_k w_k sum_axes (p_{+k} - p_0 + p_{-k} - p_0); in FP64, whose pipe bounds the step, the
// grouping of the 3D kernels, sum_k w_k (((l + r) + (u + d)) - 4 p_0), 5 instead of 8
// operations per k.  Both annihilate constants exactly.
template <int H, typename T, class X, class Z>
__device__ __forceinline__ T lap2(const T* w2, T c, X xk, Z zk) {
    T s = 0;
    if (sizeof(T) == 8) {
        const T c4 = (T)4 * c;
#pragma unroll
        for (int k = 1; k <= H; ++k)
            s = fma_(w2[k], sub_rn(add_rn(add_rn(xk(k), xk(-k)), add_rn(zk(k), zk(-k))), c4), s);
    } else {
#pragma unroll
        for (int k = 1; k <= H; ++k) s += w2[k] * (((xk(k) - c) + (xk(-k) - c)) + ((zk(k) - c) + (zk(-k) - c)));
    }
    return s;
}

// does a source corner lie in columns [x0, x1) and rows [z0, z1)?  (block-uniform; barrier)
template <typename T>
__device__ __forceinline__ bool sources_here(const PointSet<T>& src, const Layout& L, int x0, int x1, int z0, int z1) {
    if (src.n == 0) return false;
    int hit = 0;
    for (int i = threadIdx.x; i < 8 * src.n; i += blockDim.x) {
        if (src.w[i] == (T)0) continue;
        const int64_t rel = src.idx[i] - L.base;
        const int z = (int)(rel / L.px), x = (int)(rel - (int64_t)z * L.px);
        hit |= x >= x0 && x < x1 && z >= z0 && z < z1;
    }
    return __syncthreads_or(hit) != 0;
}
// sum of the source weights at padded node q
template <typename T>
__device__ __forceinline__ T source_at(const PointSet<T>& src, int64_t q) {
    T s = 0;
    for (int i = 0; i < 8 * src.n; ++i)
        if (src.idx[i] == q) s += src.w[i];
    return s;
}

static const int LEAP_THREADS = 128, LEAP_WARPS = LEAP_THREADS / 32, LEAP_ROWS = LEAP_THREADS / 8;

// Two FP32 values in one 64-bit register: one packed instruction does both points' operation
// with the rounding of the scalar one.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float x, float y) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void f2_get(F2 a, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// a - b, rounded once
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) { return f2_fma(b, f2(-1.f, -1.f), a); }

// undamped values of VX points: win[0 .. VX + 2 HX) is the row from x - HX, zk(k, j) element j
// of the row z + k
template <typename T, int H, int VX, int HX, class Z>
__device__ __forceinline__ void leap_points(const StepArgs<T>& a, const T (&win)[VX + 2 * HX], Z zk, const T (&pm)[VX],
                                            const T (&kh)[VX], T (&u)[VX]) {
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        const T c = win[HX + j];
        const T s = lap2<H>(a.w2, c, [&](int k) { return win[HX + j + k]; }, [&](int k) { return zk(k, j); });
        u[j] = c + ((c - pm[j]) + kh[j] * s);
    }
}
// Laplacians of elements j and j + 1 of a window, as lap2 forms them
template <int H, int HX, int N, class Z>
__device__ __forceinline__ F2 lap2_pair(const float* w2, const float (&win)[N], Z zk, int j, F2 c) {
    F2 s = f2(0.f, 0.f);
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        const F2 x = f2_add(f2_sub(f2(win[HX + j + k], win[HX + j + k + 1]), c),
                            f2_sub(f2(win[HX + j - k], win[HX + j - k + 1]), c));
        const F2 z = f2_add(f2_sub(f2(zk(k, j), zk(k, j + 1)), c), f2_sub(f2(zk(-k, j), zk(-k, j + 1)), c));
        s = f2_fma(f2(w2[k], w2[k]), f2_add(x, z), s);
    }
    return s;
}
template <int H, int HX, class Z>
__device__ __forceinline__ void leap_points4(const float* w2, const float (&win)[4 + 2 * HX], Z zk, const float (&pm)[4],
                                             const float (&kh)[4], float (&u)[4]) {
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
        const F2 c = f2(win[HX + j], win[HX + j + 1]);
        const F2 s = lap2_pair<H, HX>(w2, win, zk, j, c);
        f2_get(f2_add(c, f2_fma(f2(kh[j], kh[j + 1]), s, f2_sub(c, f2(pm[j], pm[j + 1])))), u[j], u[j + 1]);
    }
}

// sources and partial stores of VX points (and their absorbing layer): a call, off the path of
// the others
template <typename T>
struct Finish {
    int nx;
    T wv;                // the wavelet's sample where a source is near, else src.n = 0
    PointSet<T> src;
    const T* damp;       // g of each node, or null
    T* out;
};
template <typename T, int VX>
struct Points {
    T u[VX], pm[VX], kh[VX];
};
template <typename T, int VX>
__device__ __noinline__ void leap_finish(Finish<T> a, Points<T, VX> v, int x, int64_t q) {
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        if (x + j >= a.nx || marked(v.kh[j])) continue;
        T u = v.u[j];
        if (a.src.n) {   // the source term rounded by itself; a wavelet that is not finite stays at its nodes
            const T sw = source_at(a.src, q + j);
            if (sw != (T)0) u = add_rn(u, mul_rn(sw, a.wv));
        }
        if (a.damp) u -= a.damp[q + j] * (u - v.pm[j]);
        a.out[q + j] = u;
    }
}
// whole vectors of unmarked nodes without sources are stored at once; layer: inside the
// absorbing layer
template <typename T, int VX>
__device__ __forceinline__ void leap_put(const StepArgs<T>& a, T (&u)[VX], const T (&pm)[VX], const T (&kh)[VX], int x,
                                         int64_t q, bool layer, bool slow, bool srcs, T wv) {
#pragma unroll
    for (int j = 0; j < VX; ++j) slow = slow || marked(kh[j]);
    if (!slow) {
        if (layer) {
            T g[VX];
            ldv<T, VX>(g, a.damp + q);
#pragma unroll
            for (int j = 0; j < VX; ++j) u[j] -= g[j] * (u[j] - pm[j]);
        }
        stv<T, VX>(a.out + q, u);
    } else {
        Points<T, VX> v;
#pragma unroll
        for (int j = 0; j < VX; ++j) {
            v.u[j] = u[j];
            v.pm[j] = pm[j];
            v.kh[j] = kh[j];
        }
        Finish<T> f = {(int)a.L.nx, wv, a.src, layer ? a.damp : nullptr, a.out};
        if (!srcs) f.src.n = 0;
        leap_finish<T, VX>(f, v, x, q);
    }
}

// absorbing-layer factors of a 2D shot's nodes: g = a / (1 + a), or a itself for the adjoint
// (formed once; a division per point and step cost the layer's columns more than the stencil)
template <typename T>
__global__ void k_damp_field(Layout L, int dw, T da, bool adjoint, T* f) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < L.N; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % L.nx), z = (int)(i / L.nx);
        const T av = damp_a2<T>((int)L.nx, (int)L.nz, dw, da, x, z);
        f[L.idx(x, 0, z)] = adjoint ? av : av / ((T)1 + av);
    }
}

// HX: window half-width, H rounded up to whole vectors
template <int H, int VX>
struct Win {
    static constexpr int HX = (H + VX - 1) / VX * VX, NV = HX / VX;
};

// columns x .. x + VX - 1 of rows z0 .. z0 + RZ - 1, every load issued before the first use
template <typename T, int H, int VX, int RZ>
__device__ __forceinline__ void leap_burst(const StepArgs<T>& a, int64_t bx, int64_t bz) {
    constexpr int HX = Win<H, VX>::HX, NV = Win<H, VX>::NV;
    const Layout& L = a.L;
    const int nx = (int)L.nx, nz = (int)L.nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int xb = (int)(bx * 32) * VX, zb = (int)(bz * LEAP_WARPS) * RZ;
    const int x = xb + lane * VX, z0 = zb + warp * RZ;
    const bool in = x < nx && z0 < nz;
    const int64_t q = L.base + (int64_t)z0 * L.px + x;
    const T wv = a.src.n ? a.wavelet[a.step] : (T)0;
    T row[RZ + 2 * H][VX], sl[RZ][NV][VX], sr[RZ][NV][VX], pm[RZ][VX], kh[RZ][VX];
    if (in) {
#pragma unroll
        for (int k = 0; k < RZ + 2 * H; ++k) {
            // rows past nz + H - 1 are not allocated; they feed no stored point
            if (z0 + k - H < nz + H) ldv<T, VX>(row[k], a.p + q + (k - H) * L.px);
            else
#pragma unroll
                for (int j = 0; j < VX; ++j) row[k][j] = (T)0;
        }
#pragma unroll
        for (int r = 0; r < RZ; ++r)
            if (z0 + r < nz) {
                const int64_t qr = q + r * L.px;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    ldv<T, VX>(sl[r][v], a.p + qr - HX + v * VX);
                    ldv<T, VX>(sr[r][v], a.p + qr + VX + v * VX);
                }
                ldv<T, VX>(pm[r], a.pm + qr);
                ldv<T, VX>(kh[r], a.Kh + qr);
            }
    }
    const bool srcs = sources_here(a.src, L, xb, xb + 32 * VX, zb, zb + LEAP_WARPS * RZ);
    if (!in) return;
    const bool slow = srcs || x + VX > nx, layer_x = a.dw && (x < a.dw || x + VX > nx - a.dw);
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
        if (z0 + r >= nz) break;
        T win[VX + 2 * HX];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int j = 0; j < VX; ++j) {
                win[v * VX + j] = sl[r][v][j];
                win[HX + VX + v * VX + j] = sr[r][v][j];
            }
#pragma unroll
        for (int j = 0; j < VX; ++j) win[HX + j] = row[r + H][j];
        T u[VX];
        leap_points<T, H, VX, HX>(a, win, [&](int k, int j) { return row[r + H + k][j]; }, pm[r], kh[r], u);
        leap_put<T, VX>(a, u, pm[r], kh[r], x, q + r * L.px, layer_x || (a.dw && z0 + r > nz - 1 - a.dw), slow, srcs, wv);
    }
}

// A warp marches 128 columns (4 per lane) down zc rows, two rows a step, from its own ring in
// shared memory: 2H + 2 + 2 RD rows of p (136 floats: a halo of 4 on either side) and RD + 1
// steps of p_prev and K.  Copies are 16-byte cp.async, RD steps ahead of use; a warp waits for
// its own copies only, so there is no block barrier.  The z neighbours of a lane's columns are
// read from the ring (2H + 2 vectors for 8 points), the arithmetic runs on packed pairs.
static const int RD = 2;
template <int H>
struct Ring {
    static constexpr int NP = H + 1 + RD;            // row pairs of p
    static constexpr int W = 136, PF = NP * 2 * W;   // floats
    static constexpr int FLOATS = PF + (RD + 1) * 2 * 256;
};
template <int H>
__device__ __forceinline__ void leap_ring(const StepArgs<float>& a, int64_t bx, int64_t bz, int zc, float* sm) {
    using R = Ring<H>;
    constexpr int W = R::W, NP = R::NP;
    const Layout& L = a.L;
    const int nx = (int)L.nx, nz = (int)L.nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int xb = (int)bx * 128, zb = (int)(bz * LEAP_WARPS) * zc;
    const int x = xb + lane * 4, z0 = zb + warp * zc, z1 = min(z0 + zc, nz);
    float* ring = sm + warp * R::FLOATS;
    float* st = ring + R::PF;
    const uint32_t ring_s = smem_u32(ring) + 16u * lane, st_s = smem_u32(st) + 16u * lane;
    const int64_t qlim = L.total - 4;
    // this lane's chunk of the next row to copy: element offset of p (from x - 4) and of p_prev, K
    int64_t cq = (int64_t)(z0 + 1) * L.px + xb - 4 + 4 * lane;   // row z0 - H
    int64_t sq = (int64_t)(z0 + H + 1) * L.px + xb + 4 * lane;   // row z0
    int cz = z0 - H, sz = z0, cp = 0, ss = 0;
    auto copy_pair = [&]() {   // the next two rows of p
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const bool rok = cz + e < nz + H;
            const int64_t q = cq + e * L.px;
            const bool ok = rok && q <= qlim;
            cp_async16(ring_s + 4u * (uint32_t)((cp * 2 + e) * W), ok ? a.p + q : a.p, ok);
            if (lane < 2) {
                const bool ok2 = rok && q + 128 <= qlim;
                cp_async16(ring_s + 4u * (uint32_t)((cp * 2 + e) * W + 128), ok2 ? a.p + q + 128 : a.p, ok2);
            }
        }
        cq += 2 * L.px;
        cz += 2;
        cp = cp == NP - 1 ? 0 : cp + 1;
    };
    auto issue = [&]() {   // the next step: its new pair of rows of p, its p_prev and K
        if (sz < z1) {
            copy_pair();
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t q = sq + e * L.px;
                const bool ok = sz + e < nz && q <= qlim;
                const uint32_t d = st_s + 4u * (uint32_t)((ss * 2 + e) * 256);
                cp_async16(d, ok ? a.pm + q : a.pm, ok);
                cp_async16(d + 512u, ok ? a.Kh + q : a.Kh, ok);
            }
            sq += 2 * L.px;
            sz += 2;
            ss = ss == RD ? 0 : ss + 1;
        }
        cp_async_commit();   // empty groups keep the count uniform
    };
    if (z0 < nz) {
#pragma unroll
        for (int k = 0; k < H; ++k) copy_pair();   // the first step's other rows: its group
#pragma unroll
        for (int k = 0; k < RD; ++k) issue();
    }
    const bool srcs = sources_here(a.src, L, xb, xb + 128, zb, zb + LEAP_WARPS * zc);
    if (z0 >= nz) return;
    const float wv = srcs ? a.wavelet[a.step] : 0.f;
    const bool in = x < nx;
    const bool slow_x = srcs || x + 4 > nx, layer_x = a.dw && (x < a.dw || x + 4 > nx - a.dw);
    const int zlow = a.dw ? nz - a.dw : nz;   // rows from here on lie in the layer
    int64_t q = L.base + (int64_t)z0 * L.px + x;
    int sp = 0, sc = 0;
#pragma unroll 1
    for (int z = z0; z < z1; z += 2) {
        cp_async_wait_group<RD - 1>();
        __syncwarp();   // the step's rows have landed; every lane is done with the step before
        issue();
        float C[2 * H + 2][4], pm[2][4], kh[2][4], win[2][12];
#pragma unroll
        for (int kk = 0; kk <= H; ++kk) {
            int t = sp + kk;
            t = t >= NP ? t - NP : t;
            const float* rp = ring + t * 2 * W + 4 * lane;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                ldv<float, 4>(C[2 * kk + e], rp + e * W + 4);
                const int r = 2 * kk + e - H;   // row z + r
                if (r == 0 || r == 1) {
                    ldv<float, 4>(*reinterpret_cast<float(*)[4]>(&win[r][0]), rp + e * W);
                    ldv<float, 4>(*reinterpret_cast<float(*)[4]>(&win[r][8]), rp + e * W + 8);
                }
            }
        }
        const float* sr = st + sc * 512 + 4 * lane;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            ldv<float, 4>(pm[r], sr + r * 256);
            ldv<float, 4>(kh[r], sr + r * 256 + 128);
#pragma unroll
            for (int j = 0; j < 4; ++j) win[r][4 + j] = C[H + r][j];
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float u[4];
            leap_points4<H, 4>(a.w2, win[r], [&](int k, int j) { return C[H + r + k][j]; }, pm[r], kh[r], u);
            if (in && z + r < z1)
                leap_put<float, 4>(a, u, pm[r], kh[r], x, q + r * L.px, layer_x || z + r >= zlow, slow_x, srcs, wv);
        }
        q += 2 * L.px;
        sp = sp == NP - 1 ? 0 : sp + 1;
        sc = sc == RD ? 0 : sc + 1;
    }
    cp_async_wait_group<0>();   // the empty groups past the chunk's end
}

// w2[k] for a k that differs between lanes, without indexing the arguments
template <int H, typename T>
__device__ __forceinline__ T weight_at(const T* w2, int k) {
    T w = w2[1];
#pragma unroll
    for (int j = 2; j <= H; ++j) w = j == k ? w2[j] : w;
    return w;
}

// The updates of U immersed-boundary rows r, r + step, ... by lane gl of 8, their loads asked for
// together: a row is a chain of four dependent loads (node, entry range, entry, value), so the
// march's blocks, whose 128 registers a thread leave 16 warps on an SM, take 4 rows a lane
// group (48 damped shots of 400-1200 squared: 151 -> 135 us a step).
template <typename T, int H, int U>
__device__ __forceinline__ void leap_row(const StepArgs<T>& a, int64_t r, int64_t step, const T* p, const T* pm, T* out, T wv,
                                         int gl) {
    static_assert(H <= 4, "one stencil pair per lane");
    const Layout& L = a.L;
    int64_t q[U], j0[U];
    int n[U], most = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const bool act = r + u * step < a.rows.n;
        q[u] = act ? a.rows.pad[r + u * step] : -1;
        j0[u] = act ? a.rows.ptr[r + u * step] : 0;
        n[u] = act ? (int)(a.rows.ptr[r + u * step + 1] - j0[u]) : 0;
    }
    T c[U], pmv[U], kh[U], v[U], sv[U];
    const int k1 = (gl >> 1) + 1;
    const int64_t st = (gl & 1) ? k1 * L.px : k1;
    const T wk = gl < 2 * H ? weight_at<H>(a.w2, k1) : (T)0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        most = max(most, n[u]);
        const int64_t qq = q[u] < 0 ? L.base : q[u];
        const T* f = p + qq;
        c[u] = f[0];
        pmv[u] = kh[u] = v[u] = sv[u] = (T)0;
        if (gl == 0) {
            pmv[u] = pm[qq];
            kh[u] = a.Kh[qq];
        }
        if (gl < 2 * H) v[u] = wk * ((f[st] - c[u]) + (f[-st] - c[u]));
    }
    for (int k = gl; k < most; k += 8) {
        T w[U], f[U];
        int64_t at[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            w[u] = (T)0;
            at[u] = L.base;
            if (k < n[u]) {
                int dx, dz, dy;
                unpack_off(a.rows.code[j0[u] + k], dx, dz, dy);   // 2D codes: (x, z, 0)
                w[u] = a.rows.w[j0[u] + k];
                at[u] = q[u] + (int64_t)dz * L.px + dx;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) f[u] = p[at[u]];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (k < n[u]) v[u] += w[u] * f[u];
    }
    for (int i = gl; i < 8 * a.src.n; i += 8) {
        const int64_t si = a.src.idx[i];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (si == q[u]) sv[u] += a.src.w[i];
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
            if (a.src.n) sv[u] += __shfl_xor_sync(0xffffffffu, sv[u], o);
        }
    if (gl == 0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (q[u] < 0) continue;
            T x = c[u] + ((c[u] - pmv[u]) + (kh[u] < (T)0 ? -kh[u] : kh[u]) * v[u]);
            if (sv[u] != (T)0) x = add_rn(x, mul_rn(sv[u], wv));
            if (a.dw) x -= a.damp[q[u]] * (x - pmv[u]);
            out[q[u]] = x;
        }
    }
}
template <int RZ>
struct RowsPer {
    static constexpr int U = RZ ? 1 : 4, N = U * LEAP_ROWS;   // a lane group's rows, a block's
};

// Shapes: VX columns a thread; RZ rows (burst), or a march (RZ = 0) of the launch's zc rows.
template <typename T, int H, int VX, int RZ>
__device__ __forceinline__ void leap_block(const StepArgs<T>& a, int64_t local, int zc, float* sm) {
    if (local < a.nrb) {
        constexpr int U = RowsPer<RZ>::U;
        leap_row<T, H, U>(a, local * RowsPer<RZ>::N + (threadIdx.x >> 3), LEAP_ROWS, a.p, a.pm, a.out,
                          a.src.n ? a.wavelet[a.step] : (T)0, threadIdx.x & 7);
        return;
    }
    const int64_t c = local - a.nrb;
    if constexpr (RZ > 0) leap_burst<T, H, VX, RZ>(a, c % a.ntx, c / a.ntx);
    else leap_ring<H>(a, c % a.ntx, c / a.ntx, zc, sm);
}
template <int H, int RZ>
static constexpr size_t leap_smem() {
    return RZ ? 0 : sizeof(float) * LEAP_WARPS * Ring<H>::FLOATS;
}

template <typename T, int H, int VX, int RZ>
__global__ void __launch_bounds__(LEAP_THREADS, RZ ? 1 : 4) k_leap2d(const __grid_constant__ StepArgs<T> a, int zc) {
    extern __shared__ __align__(16) float leap_sm[];
    record_receivers(a.rec, a.p, a.traces, a.nt, a.rec_step, (int64_t)blockIdx.x * LEAP_THREADS + threadIdx.x,
                     (int64_t)gridDim.x * LEAP_THREADS);
    leap_block<T, H, VX, RZ>(a, blockIdx.x, zc, leap_sm);
}

// many shots in one launch: block -> shot by table.  seg < 0: step of a run, p^n = buf[step & 1];
// seg = j >= 0: recompute step `step` of a checkpoint segment, whose buffer (buf0) holds
// p^{c-1+j} in slot j and takes the result in slot j + 2.
template <int H, int VX, int RZ>
__global__ void __launch_bounds__(LEAP_THREADS, RZ ? 1 : 4) k_leap2d_batch(const StepArgs<float>* __restrict__ shots,
                                                               const int64_t* __restrict__ tile0,
                                                               const int32_t* __restrict__ shot_of, int step, int seg,
                                                               int zc) {
    extern __shared__ __align__(16) float leap_sm[];
    const int64_t b = blockIdx.x;
    const int sh = shot_of[b];
    StepArgs<float> a = shots[sh];
    if (seg < 0) {
        a.p = (step & 1) ? a.buf1 : a.buf0;
        a.pm = (step & 1) ? a.buf0 : a.buf1;
        a.out = const_cast<float*>(a.pm);
    } else {
        a.p = a.buf0 + (int64_t)(seg + 1) * a.L.total;
        a.pm = a.buf0 + (int64_t)seg * a.L.total;
        a.out = a.buf0 + (int64_t)(seg + 2) * a.L.total;
    }
    a.step = step;
    a.rec_step = seg < 0 ? step - 1 : -1;
    const int64_t local = b - tile0[sh];
    record_receivers(a.rec, a.p, a.traces, a.nt, a.rec_step, local * LEAP_THREADS + threadIdx.x,
                     (tile0[sh + 1] - tile0[sh]) * LEAP_THREADS);
    leap_block<float, H, VX, RZ>(a, local, zc, leap_sm);
}

// mark the row nodes of an operator in a coefficient field (sign bit)
template <typename T>
__global__ void k_mark_rows(int64_t n, const int64_t* __restrict__ pad, T* Kh) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T k = Kh[pad[i]];
        if (!marked(k)) Kh[pad[i]] = -k;
    }
}

// ---------------------------------------------------------------------------
// 2D adjoint of the leapfrog map and the velocity gradient
//   mu^m = 2 mu^{m+1} - mu^{m+2} + mask (L^T (K mu^{m+1})) + R^T res^{m-1}
//   g   += mu^m (p^m - 2 p^{m-1} + p^{m-2} - s^{m-1})      (scaled by 2 / c at the end)
//   gw[m-1] = S . mu^m
// With an absorbing layer the buffers hold nu = mu / (1 + a): the transpose of
// p^{n+1} = ((2 + K L) p^n - (1 - a) p^{n-1} + s) / (1 + a) is
// mu^m = 2 nu^{m+1} - (1 - a) nu^{m+2} + L^T (K nu^{m+1}) + R^T res^{m-1}, and
// dt^2 c^2 (L p^{m-1}) = (1 + a) p^m - 2 p^{m-1} + (1 - a) p^{m-2} - s^{m-1}.
// The same block kinds as the leapfrog step: column blocks (the queue holds K mu), and row
// blocks for the nodes that the transposed corrections or the receivers add to.
// ---------------------------------------------------------------------------
template <typename T>
struct AdjArgs {
    Layout L;
    T w2[5];
    const T* mu;         // mu^{m+1}
    const T* mum;        // mu^{m+2}
    T* out;              // mu^m (may alias mum)
    const T* Kh;         // dt^2 c^2 / h^2, sign bit: a row block's node; 0 outside the domain
    // transposed corrections, keyed by column node, and the receiver injection
    int64_t nt_rows;
    const int64_t* t_pad;
    const int64_t* t_ptr;
    const int64_t* t_off;
    const T* t_w;
    int64_t n_inj;
    const int64_t* i_pad;
    const int64_t* i_ptr;
    const int64_t* i_rec;
    const T* i_w;
    const int32_t* nodemap;  // bit 31: a transposed row; low bits: injection row + 1
    int64_t nrb, ntx;        // row blocks, column blocks along x
    const T* res;        // [nrec][nt]
    int nt;
    int m;
    const T* pm0;        // p^m
    const T* pm1;        // p^{m-1}
    const T* pm2;        // p^{m-2}
    T* grad;             // padded accumulator
    PointSet<T> src;
    const T* wavelet;
    T* gw;               // [nt] or null
    int dw;              // absorbing layer (as StepArgs); the stored multiplier is
    T da;                // nu^m = mu^m / (1 + a)
    const T* damp;       // a of each node (dw > 0)
};

template <typename T>
__device__ __forceinline__ T abs_(T v) { return v < (T)0 ? -v : v; }

// mu^m and the gradient's addend of one node (acc = mask L^T (K mu) + R^T res)
template <typename T>
__device__ __forceinline__ void adj_point(T* gw, bool damped, T av, bool inside, T acc, T mu, T mum, T p0, T p1, T p2,
                                          T srcw, T wv, T& mu_new, T& add) {
    mu_new = (T)2 * mu - ((T)1 - av) * mum + acc;
    if (damped) mu_new = mu_new / ((T)1 + av);
    add = 0;
    if (inside) {
        T d2 = (p0 - p1) - (p1 - p2);
        if (damped) d2 += av * (p0 - p2);
        d2 -= srcw * wv;
        add = mu_new * d2;
        if (gw && srcw != (T)0) atomicAdd(gw, srcw * mu_new);
    }
}

template <typename T, int H, int VX, int HX, class Z>
__device__ __forceinline__ void adj_store(const AdjArgs<T>& a, const T (&win)[VX + 2 * HX], Z zk, const T (&mu)[VX],
                                          const T (&kh)[VX], const T (&mum)[VX], const T (&p0)[VX], const T (&p1)[VX],
                                          const T (&p2)[VX], const T (&gr)[VX], int x, int z, int64_t q, bool srcs, T wv) {
    const int nx = (int)a.L.nx, nz = (int)a.L.nz;
    const bool damped = a.dw && (x < a.dw || x + VX > nx - a.dw || z > nz - 1 - a.dw);
    T u[VX], g[VX];
#pragma unroll
    for (int j = 0; j < VX; ++j) {
        const bool inside = kh[j] != (T)0;
        T s = 0;
        if (inside) s = lap2<H>(a.w2, win[HX + j], [&](int k) { return win[HX + j + k]; }, [&](int k) { return zk(k, j); });
        T add = 0;
        if (!marked(kh[j]) && x + j < nx)
            adj_point(a.gw ? a.gw + a.m - 1 : nullptr, damped, damped ? a.damp[q + j] : (T)0, inside, s, mu[j], mum[j], p0[j],
                      p1[j], p2[j], srcs ? source_at(a.src, q + j) : (T)0, wv, u[j], add);
        g[j] = gr[j] + add;
    }
    bool all = x + VX <= nx;
#pragma unroll
    for (int j = 0; j < VX; ++j) all = all && !marked(kh[j]);
    if (all) {
        stv<T, VX>(a.out + q, u);
        stv<T, VX>(a.grad + q, g);
    } else {
#pragma unroll
        for (int j = 0; j < VX; ++j)
            if (x + j < nx && !marked(kh[j])) {
                a.out[q + j] = u[j];
                a.grad[q + j] = g[j];
            }
    }
}

template <typename T, int H, int VX, int RZ>
__device__ __forceinline__ void adj_burst(const AdjArgs<T>& a, int64_t bx, int64_t bz) {
    constexpr int HX = Win<H, VX>::HX, NV = Win<H, VX>::NV;
    const Layout& L = a.L;
    const int nx = (int)L.nx, nz = (int)L.nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int xb = (int)(bx * 32) * VX, zb = (int)(bz * LEAP_WARPS) * RZ;
    const int x = xb + lane * VX, z0 = zb + warp * RZ;
    const bool in = x < nx && z0 < nz;
    const int64_t q = L.base + (int64_t)z0 * L.px + x;
    T mr[RZ + 2 * H][VX], kr[RZ + 2 * H][VX], ml[RZ][2 * NV][VX], kl[RZ][2 * NV][VX];
    T mum[RZ][VX], p0[RZ][VX], p1[RZ][VX], p2[RZ][VX], gr[RZ][VX];
    if (in) {
#pragma unroll
        for (int k = 0; k < RZ + 2 * H; ++k) {
            if (z0 + k - H < nz + H) {
                ldv<T, VX>(mr[k], a.mu + q + (k - H) * L.px);
                ldv<T, VX>(kr[k], a.Kh + q + (k - H) * L.px);
            } else {
#pragma unroll
                for (int j = 0; j < VX; ++j) mr[k][j] = kr[k][j] = (T)0;
            }
        }
#pragma unroll
        for (int r = 0; r < RZ; ++r)
            if (z0 + r < nz) {
                const int64_t qr = q + r * L.px;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    ldv<T, VX>(ml[r][v], a.mu + qr - HX + v * VX);
                    ldv<T, VX>(kl[r][v], a.Kh + qr - HX + v * VX);
                    ldv<T, VX>(ml[r][NV + v], a.mu + qr + VX + v * VX);
                    ldv<T, VX>(kl[r][NV + v], a.Kh + qr + VX + v * VX);
                }
                ldv<T, VX>(mum[r], a.mum + qr);
                ldv<T, VX>(p0[r], a.pm0 + qr);
                ldv<T, VX>(p1[r], a.pm1 + qr);
                ldv<T, VX>(p2[r], a.pm2 + qr);
                ldv<T, VX>(gr[r], a.grad + qr);
            }
    }
    const bool srcs = sources_here(a.src, L, xb, xb + 32 * VX, zb, zb + LEAP_WARPS * RZ);
    if (!in) return;
    const T wv = srcs ? a.wavelet[a.m - 1] : (T)0;
    T f[RZ + 2 * H][VX];
#pragma unroll
    for (int k = 0; k < RZ + 2 * H; ++k)
#pragma unroll
        for (int j = 0; j < VX; ++j) f[k][j] = abs_(kr[k][j]) * mr[k][j];
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
        if (z0 + r >= nz) break;
        T win[VX + 2 * HX];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int j = 0; j < VX; ++j) {
                win[v * VX + j] = abs_(kl[r][v][j]) * ml[r][v][j];
                win[HX + VX + v * VX + j] = abs_(kl[r][NV + v][j]) * ml[r][NV + v][j];
            }
#pragma unroll
        for (int j = 0; j < VX; ++j) win[HX + j] = f[r + H][j];
        adj_store<T, H, VX, HX>(a, win, [&](int k, int j) { return f[r + H + k][j]; }, mr[r + H], kr[r + H], mum[r], p0[r],
                                p1[r], p2[r], gr[r], x, z0 + r, q + r * L.px, srcs, wv);
    }
}

// everything but the plain interior vectors: a call
struct AdjVec {
    float s[4], mu[4], kh[4], mum[4], p0[4], p1[4], p2[4], gr[4];
};
struct AdjFinish {
    int nx;
    float wv;
    PointSet<float> src;      // n = 0 where no source is near
    const float* damp;        // null outside the layer
    float *gw, *out, *grad;   // gw: the step's element, or null
};
__device__ __noinline__ void adj_finish(const AdjFinish f, const AdjVec& v, int x, int64_t q) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (x + j >= f.nx || marked(v.kh[j])) continue;
        float u, add;
        const bool inside = v.kh[j] != 0.f;
        adj_point(f.gw, f.damp != nullptr, f.damp ? f.damp[q + j] : 0.f, inside, inside ? v.s[j] : 0.f, v.mu[j], v.mum[j],
                  v.p0[j], v.p1[j], v.p2[j], f.src.n ? source_at(f.src, q + j) : 0.f, f.wv, u, add);
        f.out[q + j] = u;
        f.grad[q + j] = v.gr[j] + add;
    }
}

// The adjoint's march: leap_ring's geometry with rings of mu and K (15 KB a warp at H = 4), the
// products formed on reading; the five operands of a step's rows come straight from memory,
// asked for before the wait for the rings.
template <int H>
struct AdjRing {
    static constexpr int NP = H + 1 + RD, W = 136, PF = NP * 2 * W, FLOATS = 2 * PF;
};
template <int H>
__device__ __forceinline__ void adj_ring(const AdjArgs<float>& a, int64_t bx, int64_t bz, int zc, float* sm) {
    using R = AdjRing<H>;
    constexpr int W = R::W, NP = R::NP;
    const Layout& L = a.L;
    const int nx = (int)L.nx, nz = (int)L.nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int xb = (int)bx * 128, zb = (int)(bz * LEAP_WARPS) * zc;
    const int x = xb + lane * 4, z0 = zb + warp * zc, z1 = min(z0 + zc, nz);
    float* ring = sm + warp * R::FLOATS;
    const uint32_t ring_s = smem_u32(ring) + 16u * lane;
    const int64_t qlim = L.total - 4;
    int64_t cq = (int64_t)(z0 + 1) * L.px + xb - 4 + 4 * lane;   // row z0 - H
    int cz = z0 - H, cp = 0, left = (z1 - z0 + 1) / 2;
    auto copy_pair = [&]() {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const bool rok = cz + e < nz + H;
            const int64_t q = cq + e * L.px;
            const bool ok = rok && q <= qlim;
            const uint32_t d = ring_s + 4u * (uint32_t)((cp * 2 + e) * W);
            cp_async16(d, ok ? a.mu + q : a.mu, ok);
            cp_async16(d + 4u * R::PF, ok ? a.Kh + q : a.Kh, ok);
            if (lane < 2) {
                const bool ok2 = rok && q + 128 <= qlim;
                cp_async16(d + 512u, ok2 ? a.mu + q + 128 : a.mu, ok2);
                cp_async16(d + 4u * R::PF + 512u, ok2 ? a.Kh + q + 128 : a.Kh, ok2);
            }
        }
        cq += 2 * L.px;
        cz += 2;
        cp = cp == NP - 1 ? 0 : cp + 1;
    };
    auto issue = [&]() {
        if (left > 0) {
            copy_pair();
            --left;
        }
        cp_async_commit();
    };
    if (z0 < nz) {
#pragma unroll
        for (int k = 0; k < H; ++k) copy_pair();
#pragma unroll
        for (int k = 0; k < RD; ++k) issue();
    }
    const bool srcs = sources_here(a.src, L, xb, xb + 128, zb, zb + LEAP_WARPS * zc);
    if (z0 >= nz) return;
    const float wv = srcs ? a.wavelet[a.m - 1] : 0.f;
    const bool in = x < nx;
    const bool slow_x = srcs || x + 4 > nx, layer_x = a.dw && (x < a.dw || x + 4 > nx - a.dw);
    const int zlow = a.dw ? nz - a.dw : nz;
    int64_t q = L.base + (int64_t)z0 * L.px + x;
    int sp = 0;
#pragma unroll 1
    for (int z = z0; z < z1; z += 2) {
        AdjVec v[2];
        if (in) {
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (z + r < z1) {
                    const int64_t qr = q + r * L.px;
                    ldv<float, 4>(v[r].mum, a.mum + qr);
                    ldv<float, 4>(v[r].p0, a.pm0 + qr);
                    ldv<float, 4>(v[r].p1, a.pm1 + qr);
                    ldv<float, 4>(v[r].p2, a.pm2 + qr);
                    ldv<float, 4>(v[r].gr, a.grad + qr);
                }
        }
        cp_async_wait_group<RD - 1>();
        __syncwarp();
        issue();
        float C[2 * H + 2][4], win[2][12];
#pragma unroll
        for (int kk = 0; kk <= H; ++kk) {
            int t = sp + kk;
            t = t >= NP ? t - NP : t;
            const float* rp = ring + t * 2 * W + 4 * lane;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float m4[4], k4[4];
                ldv<float, 4>(m4, rp + e * W + 4);
                ldv<float, 4>(k4, rp + e * W + 4 + R::PF);
                const int r = 2 * kk + e - H;
#pragma unroll
                for (int j = 0; j < 4; ++j) C[2 * kk + e][j] = fabsf(k4[j]) * m4[j];
                if (r == 0 || r == 1) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        v[r].mu[j] = m4[j];
                        v[r].kh[j] = k4[j];
                        win[r][4 + j] = C[2 * kk + e][j];
                    }
                    ldv<float, 4>(m4, rp + e * W);
                    ldv<float, 4>(k4, rp + e * W + R::PF);
#pragma unroll
                    for (int j = 0; j < 4; ++j) win[r][j] = fabsf(k4[j]) * m4[j];
                    ldv<float, 4>(m4, rp + e * W + 8);
                    ldv<float, 4>(k4, rp + e * W + 8 + R::PF);
#pragma unroll
                    for (int j = 0; j < 4; ++j) win[r][8 + j] = fabsf(k4[j]) * m4[j];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            AdjVec& w = v[r];
#pragma unroll
            for (int j = 0; j < 4; j += 2)
                f2_get(lap2_pair<H, 4>(a.w2, win[r], [&](int k, int i) { return C[H + r + k][i]; }, j,
                                       f2(win[r][4 + j], win[r][5 + j])),
                       w.s[j], w.s[j + 1]);
            if (!in || z + r >= z1) continue;
            const bool layer = layer_x || z + r >= zlow;
            bool slow = slow_x;
#pragma unroll
            for (int j = 0; j < 4; ++j) slow = slow || marked(w.kh[j]);
            const int64_t qr = q + r * L.px;
            if (!slow) {
                float u[4], g[4], av[4] = {0.f, 0.f, 0.f, 0.f};
                if (layer) ldv<float, 4>(av, a.damp + qr);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool inside = w.kh[j] != 0.f;
                    float add;
                    adj_point((float*)nullptr, layer, av[j], inside, inside ? w.s[j] : 0.f, w.mu[j], w.mum[j], w.p0[j],
                              w.p1[j], w.p2[j], 0.f, 0.f, u[j], add);
                    g[j] = w.gr[j] + add;
                }
                stv<float, 4>(a.out + qr, u);
                stv<float, 4>(a.grad + qr, g);
            } else {
                AdjFinish f = {nx, wv, a.src, layer ? a.damp : nullptr, a.gw ? a.gw + a.m - 1 : nullptr, a.out, a.grad};
                if (!srcs) f.src.n = 0;
                const AdjVec copy = w;
                adj_finish(f, copy, x, qr);
            }
        }
        q += 2 * L.px;
        sp = sp == NP - 1 ? 0 : sp + 1;
    }
    cp_async_wait_group<0>();
}

// nodes r, r + LEAP_ROWS, ... (U of them) of the transposed rows and then of the receiver
// injection, 8 lanes each, their loads asked for together as in leap_row
template <typename T, int H, int U>
__device__ __forceinline__ void adj_rows(const AdjArgs<T>& a, int64_t r) {
    const Layout& L = a.L;
    const int gl = threadIdx.x & 7;
    int64_t q[U], j0[U];
    int n[U], inj[U], most = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t i = r + u * LEAP_ROWS;
        const bool trow = i < a.nt_rows;
        q[u] = trow ? a.t_pad[i] : i < a.nt_rows + a.n_inj ? a.i_pad[i - a.nt_rows] : -1;
        j0[u] = trow ? a.t_ptr[i] : 0;
        n[u] = trow ? (int)(a.t_ptr[i + 1] - j0[u]) : 0;
    }
    T kq[U], mu[U], mum[U], p0[U], p1[U], p2[U], gr[U], v[U], rs[U], sv[U];
    const int k1 = (gl >> 1) + 1;
    const int64_t st = (gl & 1) ? k1 * L.px : k1;
    const T wk = gl < 2 * H ? weight_at<H>(a.w2, k1) : (T)0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        most = max(most, n[u]);
        const int64_t qq = q[u] < 0 ? L.base : q[u];
        const int32_t map = q[u] < 0 ? 0 : a.nodemap[qq];
        kq[u] = a.Kh[qq];
        mu[u] = a.mu[qq];
        mum[u] = p0[u] = p1[u] = p2[u] = gr[u] = v[u] = rs[u] = sv[u] = (T)0;
        if (gl == 0) {
            mum[u] = a.mum[qq];
            p0[u] = a.pm0[qq];
            p1[u] = a.pm1[qq];
            p2[u] = a.pm2[qq];
            gr[u] = a.grad[qq];
        }
        if (gl < 2 * H) {
            const T c = abs_(kq[u]) * mu[u];
            v[u] = wk * ((abs_(a.Kh[qq + st]) * a.mu[qq + st] - c) + (abs_(a.Kh[qq - st]) * a.mu[qq - st] - c));
        }
        if (r + u * LEAP_ROWS >= a.nt_rows && map < 0) q[u] = -1;   // its transposed row injects it
        inj[u] = (map & 0x7fffffff) - 1;
    }
    for (int k = gl; k < most; k += 8) {
        T w[U], f[U], g[U];
        int64_t at[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            w[u] = (T)0;
            at[u] = L.base;
            if (k < n[u]) {
                at[u] = q[u] + a.t_off[j0[u] + k];
                w[u] = a.t_w[j0[u] + k];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            f[u] = a.Kh[at[u]];
            g[u] = a.mu[at[u]];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (k < n[u]) v[u] += w[u] * (abs_(f[u]) * g[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (q[u] >= 0 && inj[u] >= 0)
            for (int64_t e = a.i_ptr[inj[u]] + gl; e < a.i_ptr[inj[u] + 1]; e += 8)
                rs[u] += a.i_w[e] * a.res[a.i_rec[e] * (int64_t)a.nt + (a.m - 1)];
    for (int i = gl; i < 8 * a.src.n; i += 8) {
        const int64_t si = a.src.idx[i];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (si == q[u]) sv[u] += a.src.w[i];
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
            rs[u] += __shfl_xor_sync(0xffffffffu, rs[u], o);
            sv[u] += __shfl_xor_sync(0xffffffffu, sv[u], o);
        }
    if (gl == 0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (q[u] < 0) continue;
            const bool inside = kq[u] != (T)0;
            T x, add;
            adj_point(a.gw ? a.gw + a.m - 1 : nullptr, a.dw > 0, a.dw ? a.damp[q[u]] : (T)0, inside,
                      (inside ? v[u] : (T)0) + rs[u], mu[u], mum[u], p0[u], p1[u], p2[u], sv[u],
                      a.src.n ? a.wavelet[a.m - 1] : (T)0, x, add);
            a.out[q[u]] = x;
            a.grad[q[u]] = gr[u] + add;
        }
    }
}

// RZ = 1: burst of VX columns; 0: march of zc rows
template <typename T, int H, int VX, int RZ>
__device__ __forceinline__ void adj_block(const AdjArgs<T>& a, int64_t local, int zc, float* sm) {
    if (local < a.nrb) {
        adj_rows<T, H, RowsPer<RZ>::U>(a, local * RowsPer<RZ>::N + (threadIdx.x >> 3));
        return;
    }
    const int64_t c = local - a.nrb;
    if constexpr (RZ > 0) adj_burst<T, H, VX, RZ>(a, c % a.ntx, c / a.ntx);
    else adj_ring<H>(a, c % a.ntx, c / a.ntx, zc, sm);
}
template <int H, int RZ>
static constexpr size_t adj_smem() {
    return RZ ? 0 : sizeof(float) * LEAP_WARPS * AdjRing<H>::FLOATS;
}

template <typename T, int H, int VX, int RZ>
__global__ void __launch_bounds__(LEAP_THREADS, RZ ? 1 : 3) k_adj2d(const __grid_constant__ AdjArgs<T> a, int zc) {
    extern __shared__ __align__(16) float adj_sm[];
    adj_block<T, H, VX, RZ>(a, blockIdx.x, zc, adj_sm);
}

// Batched adjoint step m of segment [c, e) over many shots: block -> shot by table.
// mu^{m+1} / mu^{m+2} alternate between the shot's two buffers with the number of steps
// taken (nt - m); the segment buffer holds p^{c-1+j} in slot j.
template <typename T>
struct AdjBatch {
    AdjArgs<T> a;
    T* mu1;
    T* mu2;
    T* seg;               // segment buffer: (seg_len + 2) padded fields
};

template <int H, int VX, int RZ>
__global__ void __launch_bounds__(LEAP_THREADS, RZ ? 1 : 3) k_adj2d_batch(const AdjBatch<float>* __restrict__ shots,
                                                              const int64_t* __restrict__ tile0,
                                                              const int32_t* __restrict__ shot_of, int m, int j, int nt,
                                                              int zc) {
    extern __shared__ __align__(16) float adj_sm[];
    const int64_t b = blockIdx.x;
    const int sh = shot_of[b];
    const AdjBatch<float>& B = shots[sh];
    AdjArgs<float> a = B.a;
    const bool even = ((nt - m) & 1) == 0;
    a.mu = even ? B.mu1 : B.mu2;
    a.mum = even ? B.mu2 : B.mu1;
    a.out = const_cast<float*>(a.mum);
    a.m = m;
    const int64_t tot = a.L.total;
    a.pm0 = B.seg + (int64_t)(j + 1) * tot;
    a.pm1 = B.seg + (int64_t)j * tot;
    a.pm2 = B.seg + (int64_t)(j - 1) * tot;
    adj_block<float, H, VX, RZ>(a, b - tile0[sh], zc, adj_sm);
}

// nodemap and marks of the adjoint's row-block nodes
template <typename T>
__global__ void k_map_nodes(int64_t n, const int64_t* __restrict__ pad, bool inj, int32_t* nodemap, T* Kh) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = pad[i];
        nodemap[q] |= inj ? (int32_t)(i + 1) : (int32_t)0x80000000;
        const T k = Kh[q];
        if (!marked(k)) Kh[q] = -k;
    }
}

// unpadded gradient: the accumulated mu^m (p_tt) times 2 / c = (2 dt / h) / sqrt(K)
template <typename T>
__global__ void k_unpad_grad(Layout L, const T* pad, const T* Kh, T two_dt_over_h, T* out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < L.N; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = i % L.nx, z = i / L.nx, q = L.idx(x, 0, z);
        const T k = abs_(Kh[q]);
        out[i] = k > (T)0 ? pad[q] * (two_dt_over_h / sqrt(k)) : (T)0;
    }
}

// ---------------------------------------------------------------------------
// Many steps of one small grid in one launch.  A step of some 10^5 points takes a couple of
// microseconds of memory latency, less than the gap between two launches, so all the steps
// of a run (or of the part between two checkpoints) run in one cooperative launch with a
// grid barrier after each: at most one block per SM, every block resident.  A thread keeps
// its VX x RZ points, p_prev and K in registers and reads only their halo, from L1/L2 (the
// barrier's release and acquire order the other blocks' stores before these reads).  The last
// two warps of a block do what the row blocks do: the immersed-boundary rows (their entries held
// in shared memory, since the barrier empties L1) and the receivers, beside the column warps.
// The absorbing-layer factor and the source weight of each point sit in shared memory.
//   FP64, 201 x 201, order 4, 500 steps: 6.2 -> 1.97 ms.  A step is the barrier (about 1.5 us),
// the halo's latency and, in FP64, 1.3 us of a pipe that issues a warp every 16 cycles.
//   The barrier's wait is bounded (about a second): a block that gives up sets the device's
// status word (ib_sync_status) and the call's word (the adjoint, which waits for its result,
// returns IB_ERR_TIMEOUT) and leaves, and so do the others.
// ---------------------------------------------------------------------------
template <typename T>
struct RunArgs {
    StepArgs<T> a;       // p, pm, out unused
    T* buf0;             // step n reads p^n from field(n) and writes p^{n+1} to field(n + 1) ..
    T* buf1;             // .. which are buf0 / buf1 by the parity of n - n0,
    int64_t stride;      // or, with a stride, buf0 + (n - n0 + 1) stride (p^{n0-1} at buf0)
    int n0, n1;
    int cw;              // column warps per block
    unsigned* bar;       // barrier count, zero at launch
    int* err;            // this call's word, set with the device's status word; or null
};
static const int STATUS_UNSTABLE = 1, STATUS_TIMEOUT = 2;
static __device__ int g_dev_status;

template <typename T>
__device__ __forceinline__ T* run_field(const RunArgs<T>& r, int n) {
    if (r.stride) return r.buf0 + (int64_t)(n - r.n0 + 1) * r.stride;
    return ((n - r.n0) & 1) ? r.buf1 : r.buf0;
}

static const uint64_t BARRIER_LIMIT_NS = 1000000000ull;
// all blocks of the launch; false when the wait gave up (after limit_ns)
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned target, uint64_t limit_ns, int* dead) {
    __syncthreads();
    if (threadIdx.x == 0) {
        // the block's stores (ordered before by the barrier) are released with the arrival, and the
        // acquiring load orders the block's reads after the other blocks' arrivals
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(1u) : "memory");
        bool ok = false;
        const uint64_t t0 = global_ns();
        for (int it = 0; it < (1 << 26); ++it) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (v >= target) {
                ok = true;
                break;
            }
            if ((it & 1023) == 1023 && global_ns() - t0 > limit_ns) break;
        }
        if (!ok) *dead = 1;
    }
    __syncthreads();
    return *dead == 0;
}
// Self-test: every block arrives once and waits for target arrivals.
__global__ void k_barrier_selftest(unsigned* bar, unsigned target, uint64_t limit_ns, int* gave_up) {
    __shared__ int dead;
    if (threadIdx.x == 0) dead = 0;
    if (!grid_barrier(bar, target, limit_ns, &dead) && threadIdx.x == 0) atomicAdd(gave_up, 1);
}

// the shape's largest block: registers for VX x RZ points (c, p_prev, K, halo)
template <typename T, int H, int VX, int RZ>
struct RunShape {
    static constexpr int THREADS = sizeof(T) == 8 ? (H <= 2 ? 1024 : 512) : (VX * RZ == 1 ? 1024 : 768);
};
static const int RUN_RW = 2;        // row warps
static const int RUN_ROWS = 64, RUN_ENT = 1536;   // rows and entries of a block held in shared memory
template <typename T>
struct RunRow {
    int64_t q;
    T kh, g, sw;
    int e0, e1;          // entries; e1 < 0: not held
};

template <typename T, int H, int VX, int RZ>
__global__ void __launch_bounds__(RunShape<T, H, VX, RZ>::THREADS) k_leap2d_run(const __grid_constant__ RunArgs<T> r) {
    constexpr int HX = Win<H, VX>::HX, NV = Win<H, VX>::NV;
    extern __shared__ __align__(16) unsigned char run_sm[];
    __shared__ int dead;
    const StepArgs<T>& a = r.a;
    const Layout& L = a.L;
    const int nx = (int)L.nx, nz = (int)L.nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // this block's rows (a contiguous part of the list), their entries, then per thread the damping
    // factors and source weights of its points
    RunRow<T>* srow = reinterpret_cast<RunRow<T>*>(run_sm);
    T* ew = reinterpret_cast<T*>(srow + RUN_ROWS);
    int* eo = reinterpret_cast<int*>(ew + RUN_ENT);
    T* gd = reinterpret_cast<T*>(eo + RUN_ENT) + threadIdx.x * (2 * VX * RZ);
    T* gs = gd + VX * RZ;
    const int64_t rpb = (a.rows.n + gridDim.x - 1) / gridDim.x, rfirst = rpb * blockIdx.x;
    const int nrow = (int)(rfirst < a.rows.n ? (rpb < a.rows.n - rfirst ? rpb : a.rows.n - rfirst) : 0);
    const int64_t ebase = nrow ? a.rows.ptr[rfirst] : 0;
    for (int i = threadIdx.x; i < nrow && i < RUN_ROWS; i += blockDim.x) {
        RunRow<T> w;
        w.q = a.rows.pad[rfirst + i];
        const T k = a.Kh[w.q];
        w.kh = k < (T)0 ? -k : k;
        w.g = a.dw ? a.damp[w.q] : (T)0;
        w.sw = source_at(a.src, w.q);
        const int64_t e0 = a.rows.ptr[rfirst + i] - ebase, e1 = a.rows.ptr[rfirst + i + 1] - ebase;
        w.e0 = (int)e0;
        w.e1 = e1 <= RUN_ENT ? (int)e1 : -1;
        srow[i] = w;
    }
    {
        const int64_t ne = nrow ? a.rows.ptr[rfirst + nrow] - ebase : 0;
        for (int i = threadIdx.x; i < ne && i < RUN_ENT; i += blockDim.x) {
            int dx, dz, dy;
            unpack_off(a.rows.code[ebase + i], dx, dz, dy);   // 2D codes: (x, z, 0)
            eo[i] = (int)(dz * L.px) + dx;
            ew[i] = a.rows.w[ebase + i];
        }
    }
    if (threadIdx.x == 0) dead = 0;
    const bool column = warp < r.cw;
    const int bx = (int)(blockIdx.x % a.ntx), bz = (int)(blockIdx.x / a.ntx);
    const int x = (bx * 32 + lane) * VX, z0 = (bz * r.cw + warp) * RZ;
    const bool in = column && x < nx && z0 < nz;
    const int64_t q = L.base + (int64_t)z0 * L.px + x;
    T c[RZ][VX], pm[RZ][VX], kh[RZ][VX];
    bool slow = false, mark = false;
    if (in) {
        const T* p0 = run_field(r, r.n0);
        const T* q0 = r.stride ? r.buf0 : r.buf1;
#pragma unroll
        for (int k = 0; k < RZ; ++k) {
            if (z0 + k < nz) {
                ldv<T, VX>(c[k], p0 + q + k * L.px);
                ldv<T, VX>(pm[k], q0 + q + k * L.px);
                ldv<T, VX>(kh[k], a.Kh + q + k * L.px);
            } else {
#pragma unroll
                for (int j = 0; j < VX; ++j) c[k][j] = pm[k][j] = kh[k][j] = (T)0;
            }
#pragma unroll
            for (int j = 0; j < VX; ++j) {
                const int i = k * VX + j;
                T g = 0, sw = 0;
                if (x + j < nx && z0 + k < nz) {
                    if (a.dw) g = a.damp[q + k * L.px + j];
                    sw = source_at(a.src, q + k * L.px + j);
                }
                gd[i] = g;
                gs[i] = sw;
                slow = slow || g != (T)0 || sw != (T)0;
                mark = mark || marked(kh[k][j]);
            }
        }
    }
    const bool edge = x + VX > nx;   // partial vectors
    // row warps: 8 lanes a row
    const int gl = lane & 7, grp = (warp - r.cw) * 4 + (lane >> 3);
    __syncthreads();
    unsigned target = 0;
    for (int n = r.n0; n < r.n1; ++n) {
        const T* p = run_field(r, n);
        T* out = run_field(r, n + 1);
        const T wv = a.src.n ? a.wavelet[n] : (T)0;
        if (in) {
            T up[H][VX], dn[H][VX], sl[RZ][NV][VX], sr[RZ][NV][VX];
#pragma unroll
            for (int k = 0; k < H; ++k) {
                ldv<T, VX>(up[k], p + q + (k - H) * L.px);
                // rows past nz + H - 1 are not allocated; they feed no stored point
                if (z0 + RZ + k < nz + H) ldv<T, VX>(dn[k], p + q + (RZ + k) * L.px);
                else
#pragma unroll
                    for (int j = 0; j < VX; ++j) dn[k][j] = (T)0;
            }
#pragma unroll
            for (int k = 0; k < RZ; ++k)
                if (z0 + k < nz) {
                    const int64_t qr = q + k * L.px;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        ldv<T, VX>(sl[k][v], p + qr - HX + v * VX);
                        ldv<T, VX>(sr[k][v], p + qr + VX + v * VX);
                    }
                    if (mark || edge) ldv<T, VX>(c[k], p + qr);   // nodes that the row warps, or nobody, wrote
                } else {
                    // a row of the padding: zero
#pragma unroll
                    for (int j = 0; j < VX; ++j) c[k][j] = (T)0;
                }
            T u[RZ][VX];
#pragma unroll
            for (int k = 0; k < RZ; ++k) {
                T win[VX + 2 * HX];
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int j = 0; j < VX; ++j) {
                        win[v * VX + j] = sl[k][v][j];
                        win[HX + VX + v * VX + j] = sr[k][v][j];
                    }
#pragma unroll
                for (int j = 0; j < VX; ++j) win[HX + j] = c[k][j];
                leap_points<T, H, VX, HX>(a, win, [&](int o, int j) {
                    const int m = k + o;   // compile-time after unrolling
                    return m < 0 ? up[m < 0 ? H + m : 0][j] : m >= RZ ? dn[m >= RZ ? m - RZ : 0][j] : c[m < 0 || m >= RZ ? 0 : m][j];
                }, pm[k], kh[k], u[k]);
            }
#pragma unroll
            for (int k = 0; k < RZ; ++k) {
                if (slow) {
#pragma unroll
                    for (int j = 0; j < VX; ++j) {
                        const T sw = gs[k * VX + j];
                        if (sw != (T)0) u[k][j] = add_rn(u[k][j], mul_rn(sw, wv));
                        u[k][j] -= gd[k * VX + j] * (u[k][j] - pm[k][j]);
                    }
                }
                if (z0 + k < nz) {
                    T* o = out + q + k * L.px;
                    if (mark || edge) {
#pragma unroll
                        for (int j = 0; j < VX; ++j)
                            if (x + j < nx && !marked(kh[k][j])) o[j] = u[k][j];
                    } else {
                        stv<T, VX>(o, u[k]);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < RZ; ++k)
#pragma unroll
                for (int j = 0; j < VX; ++j) {
                    pm[k][j] = c[k][j];
                    c[k][j] = u[k][j];
                }
        } else if (!column) {
            const T* pmf = r.stride ? p - r.stride : out;
            for (int i0 = 0; i0 < nrow; i0 += 4 * RUN_RW) {   // warp-uniform
                const int i = i0 + grp;
                const bool held = i < RUN_ROWS && i < nrow && srow[i].e1 >= 0;
                if (__any_sync(0xffffffffu, i < nrow && !held)) {
                    leap_row<T, H, 1>(a, i < nrow ? rfirst + i : a.rows.n, 0, p, pmf, out, wv, gl);
                    continue;
                }
                const RunRow<T> w = srow[held ? i : 0];
                const T cc = p[w.q];
                T pmv = 0, v = 0;
                if (gl == 0) pmv = pmf[w.q];
                if (gl < 2 * H) {
                    const int k = (gl >> 1) + 1;
                    const int64_t st = (gl & 1) ? k * L.px : k;
                    v = weight_at<H>(a.w2, k) * ((p[w.q + st] - cc) + (p[w.q - st] - cc));
                }
                for (int e = w.e0 + gl; e < w.e1; e += 8) v += ew[e] * p[w.q + eo[e]];
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (held && gl == 0) {
                    T u = cc + ((cc - pmv) + w.kh * v);
                    if (w.sw != (T)0) u = add_rn(u, mul_rn(w.sw, wv));
                    if (a.dw) u -= w.g * (u - pmv);
                    out[w.q] = u;
                }
            }
            record_receivers(a.rec, p, a.traces, a.nt, a.rec_step < 0 ? -1 : n - 1,
                             (int64_t)blockIdx.x * (32 * RUN_RW) + (warp - r.cw) * 32 + lane,
                             (int64_t)gridDim.x * (32 * RUN_RW));
        }
        if (n + 1 < r.n1) {
            target += gridDim.x;
            if (!grid_barrier(r.bar, target, BARRIER_LIMIT_NS, &dead)) {
                if (threadIdx.x == 0) {
                    atomicOr(&g_dev_status, STATUS_TIMEOUT);
                    if (r.err) atomicExch(r.err, 1);
                }
                return;
            }
        }
    }
}
