// Learned modified stencils: input features, a bfloat16 tensor-core MLP
// (mma.sync m16n8k16, FP32 accumulation), its training step (mean squared
// error, Adam) and the row predictions that the constructor checks.
//
// The paper fits every modified row by constrained least squares; the network
// only proposes rows, and ib_build_stencils_learned keeps a proposal when it
// passes the exactness test of the fit (see k_fit's learned_residual).
#include <cuda_bf16.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "ib_common.cuh"

#define TRY(x)                                  \
    do {                                        \
        ib_status st_ = (x);                    \
        if (st_ != IB_OK) return st_;           \
    } while (0)

#define MLP_MAX_LINEAR 9
typedef __nv_bfloat16 bf16;

struct ib_mlp {
    int device = 0;
    ib_mlp_config cfg;
    int nl = 0;                         // linear layers
    int dims[MLP_MAX_LINEAR + 1];       // dims[0] = n_in, dims[nl] = n_out
    int64_t w_off[MLP_MAX_LINEAR], b_off[MLP_MAX_LINEAR], wb_off[MLP_MAX_LINEAR];
    int64_t n_params = 0, n_wb = 0;
    int n_in_off = 0, n_in = 0, n_out = 0, out_R = 0;
    float* params = nullptr;
    float* grads = nullptr;
    float* adam_m = nullptr;
    float* adam_v = nullptr;
    bf16* wb = nullptr;                 // bfloat16 copies of the weight matrices
    int8_t* in_off = nullptr;           // [n_in_off][3]
    int32_t* out_lut = nullptr;         // [(2R+1)^3] footprint index or -1
    int64_t step = 0;
    // training scratch (rows <= cap)
    int64_t cap = 0;
    bf16* act = nullptr;                // hidden activations, [nl - 1][cap][n_hidden]
    bf16* g16 = nullptr;                // gradients of the layers' outputs, [nl][cap][max(n_hidden, n_out rounded up to 8)]
    bf16* xg = nullptr;                 // gathered inputs, [cap][n_in rounded up to 8]
    float* bpart = nullptr;             // [row tiles of cap][sum of layer widths], then the loss partials
    // inference scratch (rows per chunk)
    int64_t icap = 0;
    bf16* ia = nullptr;
    bf16* ib = nullptr;
    bf16* ix = nullptr;                 // features of one chunk
};

// ---------------------------------------------------------------------------
// offsets |o| <= r in support order: distance, then array order (z, y, x)
// ---------------------------------------------------------------------------
static std::vector<std::array<int, 3>> ball_offsets(int d, double r) {
    const int R = (int)std::ceil(r) + 1;
    const int64_t q_lim = (int64_t)std::floor(4.0 * r * r + 1e-9);
    struct E {
        int64_t q;
        int z, y, x;
    };
    std::vector<E> e;
    for (int z = (d == 3 ? -R : 0); z <= (d == 3 ? R : 0); ++z)
        for (int y = -R; y <= R; ++y)
            for (int x = -R; x <= R; ++x) {
                int64_t q = 4LL * (x * x + y * y + z * z);
                if (q <= q_lim) e.push_back({q, z, y, x});
            }
    std::sort(e.begin(), e.end(), [](const E& a, const E& b) {
        if (a.q != b.q) return a.q < b.q;
        if (a.z != b.z) return a.z < b.z;
        if (a.y != b.y) return a.y < b.y;
        return a.x < b.x;
    });
    std::vector<std::array<int, 3>> out;
    // in 2D the second coordinate is the array's second axis: (x, y) with z = 0
    for (auto& v : e) out.push_back({v.x, v.y, v.z});
    return out;
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
__global__ void k_features(int ndim, int64_t n0, int64_t n1, int64_t n2, double h, const double* sdf,
                           const int64_t* nodes, int64_t n, const int8_t* off, int noff, int n_in,
                           float f_free, float f_rigid, float f_order, bf16* X) {
    const int64_t total = n * n_in;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / n_in;
        const int j = (int)(e - i * n_in);
        float v;
        if (j < noff) {
            const int64_t lin = nodes[i];
            int64_t x = lin % n0, r = lin / n0, y, z;
            if (ndim == 3) {
                y = r % n1;
                z = r / n1;
            } else {
                y = r;
                z = 0;
            }
            int64_t qx = x + off[3 * j], qy = y + off[3 * j + 1], qz = z + off[3 * j + 2];
            qx = qx < 0 ? 0 : (qx >= n0 ? n0 - 1 : qx);
            qy = qy < 0 ? 0 : (qy >= n1 ? n1 - 1 : qy);
            qz = qz < 0 ? 0 : (qz >= n2 ? n2 - 1 : qz);
            v = (float)(sdf[(qz * n1 + qy) * n0 + qx] / h);
        } else if (j == noff) {
            v = f_free;
        } else if (j == noff + 1) {
            v = f_rigid;
        } else {
            v = f_order;
        }
        X[e] = __float2bfloat16(v);
    }
}

// C = A B with bfloat16 operands and FP32 accumulation on the tensor cores
// (mma.sync m16n8k16 over ascending k, so that a sum does not depend on the tiling).
// A is [m][k]; B is [n][k] (forward: the weights) or [k][n] (input gradients).
//   128 x 128 x 32 tiles of 8 warps (64 x 32 each), four cp.async stages (82 KB, two
// blocks per SM), fragments by ldmatrix (.trans for the [k][*] layouts).  Copies are 16
// bytes where the operand's rows allow it, 8 bytes for rows of 4 j elements (260 network
// inputs), single elements otherwise.
//   What bounds the training step is the number of blocks, passes and launches, not the
// tensor pipe: the epilogues form the loss and its gradient, the ReLU mask and the column
// sums of the bias gradients, so no FP32 gradient is stored, and the weight gradients of
// all layers are one launch (k_weight_grad).
enum { EPI_BIAS_F32 = 0, EPI_BIAS_RELU_BF16 = 1, EPI_RELU_GRAD = 2, EPI_MSE = 3 };
struct Operand {
    const bf16* p;
    int64_t ld;              // elements between rows
    int rows, ext;           // valid rows; valid elements of a row (copies stay inside)
};
struct Gemm {
    int M, N, K;
    Operand a, b;
    const float* bias;       // [N]
    const bf16* act;         // EPI_RELU_GRAD: forward activation [m][n] (ld ldc); gradient kept where > 0
    float* c32;              // EPI_BIAS_F32: [m][ldc]
    bf16* c16;               // [m][ldc]
    int64_t ldc;
    float* colpart;          // [gridDim.y][N] column sums of the tile's gradient
    const float* T;          // EPI_MSE: targets [*][N], rows t_idx
    const int64_t* t_idx;
    float scale;             // EPI_MSE: 2 / (rows N)
    float* losspart;         // EPI_MSE: [gridDim.y][gridDim.x] sums of (Y - T)^2
};

#define GBM 128
#define GBN 128
#define GBK 32
#define GST 4
#define GLDK (GBK + 8)    // [m][k] tile row (80 bytes: ldmatrix rows fall in distinct banks)
#define GLDM (GBN + 8)    // [k][n] tile row (272 bytes)

__device__ __forceinline__ void mma_16816(float* d, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t* r, const bf16* p) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// rows r0 .. r0 + R - 1, elements c0 .. c0 + C - 1 of an operand into a tile of row pitch LD,
// zero beyond its rows and row extent; VEC elements per copy (8 or 4: cp.async, 1: plain)
template <int VEC, int R, int C, int LD>
__device__ __forceinline__ void load_tile(bf16* dst, const Operand& o, int r0, int c0, int tid) {
    constexpr int CH = C / VEC;
#pragma unroll
    for (int i = 0; i < R * CH / 256; ++i) {
        const int e = tid + 256 * i, r = e / CH, c = (e - r * CH) * VEC;
        const bool ok = r0 + r < o.rows && c0 + c < o.ext;
        const bf16* src = o.p;
        if (ok) src += (int64_t)(r0 + r) * o.ld + c0 + c;
        bf16* d = dst + r * LD + c;
        if (VEC == 1) {
            *d = ok ? *src : __float2bfloat16(0.f);
        } else {
            const uint32_t s = (uint32_t)__cvta_generic_to_shared(d);
            if (VEC == 8)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(src), "r"(ok ? 16 : 0) : "memory");
            else
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(src), "r"(ok ? 8 : 0) : "memory");
        }
    }
}

template <bool BK, int MODE, int VA, int VB>
__global__ void __launch_bounds__(256, 2) k_gemm(Gemm g) {
    constexpr int SA = GBM * GLDK, SB = BK ? GBN * GLDK : GBK * GLDM;
    extern __shared__ __align__(16) unsigned char gemm_sm[];
    bf16* As = reinterpret_cast<bf16*>(gemm_sm);
    bf16* Bs = As + GST * SA;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.y * GBM, n0 = blockIdx.x * GBN;
    const int wm = (warp >> 2) * 64, wn = (warp & 3) * 32;
    const int nk = (g.K + GBK - 1) / GBK;
    float acc[4][4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    auto fetch = [&](int t) {
        if (t < nk) {
            const int k0 = t * GBK;
            bf16* a = As + (t % GST) * SA;
            bf16* b = Bs + (t % GST) * SB;
            load_tile<VA, GBM, GBK, GLDK>(a, g.a, m0, k0, tid);
            if (BK) load_tile<VB, GBN, GBK, GLDK>(b, g.b, n0, k0, tid);
            else load_tile<VB, GBK, GBN, GLDM>(b, g.b, k0, n0, tid);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
#pragma unroll
    for (int t = 0; t < GST - 1; ++t) fetch(t);
    for (int t = 0; t < nk; ++t) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(GST - 2) : "memory");
        __syncthreads();   // tile t has landed, tile t - 1 is consumed
        fetch(t + GST - 1);
        const bf16* a = As + (t % GST) * SA;
        const bf16* b = Bs + (t % GST) * SB;
#pragma unroll
        for (int ks = 0; ks < GBK; ks += 16) {
            uint32_t af[4][4], bfr[2][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                ldsm4<false>(af[i], a + (wm + i * 16 + (lane & 15)) * GLDK + ks + 8 * (lane >> 4));
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {   // two n8 blocks each: (n, k), (n, k + 8), (n + 8, k), (n + 8, k + 8)
                const int n = wn + j * 16;
                if (BK) ldsm4<false>(bfr[j], b + (n + (lane & 7) + 8 * (lane >> 4)) * GLDK + ks + 8 * ((lane >> 3) & 1));
                else ldsm4<true>(bfr[j], b + (ks + (lane & 15)) * GLDM + n + 8 * (lane >> 4));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_16816(acc[i][j], af[i], bfr[j >> 1] + 2 * (j & 1));
        }
    }
    // thread's elements: rows m0 + wm + 16 i + (lane >> 2) + 8 h, columns n0 + wn + 8 j + 2 (lane & 3) + {0, 1}
    const int gr = lane >> 2, tc = (lane & 3) * 2;
    float loss = 0.f, col[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) col[j][0] = col[j][1] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int n = n0 + wn + j * 8 + tc;
        float bias[2] = {0.f, 0.f};
        if (MODE == EPI_BIAS_F32 || MODE == EPI_BIAS_RELU_BF16 || MODE == EPI_MSE) {
            if (n < g.N) bias[0] = g.bias[n];
            if (n + 1 < g.N) bias[1] = g.bias[n + 1];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = m0 + wm + i * 16 + gr + 8 * h;
                if (m >= g.M) continue;
                const float x0 = acc[i][j][2 * h], x1 = acc[i][j][2 * h + 1];
                if (MODE == EPI_BIAS_F32) {
                    float* c = g.c32 + (int64_t)m * g.ldc + n;
                    if (n < g.N) c[0] = x0 + bias[0];
                    if (n + 1 < g.N) c[1] = x1 + bias[1];
                } else if (MODE == EPI_BIAS_RELU_BF16) {   // N is even: n < N covers the pair
                    if (n < g.N)
                        *reinterpret_cast<__nv_bfloat162*>(g.c16 + (int64_t)m * g.ldc + n) =
                            __floats2bfloat162_rn(fmaxf(x0 + bias[0], 0.f), fmaxf(x1 + bias[1], 0.f));
                } else if (MODE == EPI_RELU_GRAD) {
                    if (n < g.N) {
                        const __nv_bfloat162 f = *reinterpret_cast<const __nv_bfloat162*>(g.act + (int64_t)m * g.ldc + n);
                        const float k0 = __low2float(f) > 0.f ? x0 : 0.f, k1 = __high2float(f) > 0.f ? x1 : 0.f;
                        col[j][0] += k0;
                        col[j][1] += k1;
                        *reinterpret_cast<__nv_bfloat162*>(g.c16 + (int64_t)m * g.ldc + n) = __floats2bfloat162_rn(k0, k1);
                    }
                } else {   // EPI_MSE: d = Y - T, gradient scale * d; the row's padding up to ldc is zero
                    const float* t = g.T + g.t_idx[m] * g.N;
                    float g0 = 0.f, g1 = 0.f;
                    if (n < g.N) {
                        const float d = (x0 + bias[0]) - t[n];
                        loss += d * d;
                        g0 = g.scale * d;
                    }
                    if (n + 1 < g.N) {
                        const float d = (x1 + bias[1]) - t[n + 1];
                        loss += d * d;
                        g1 = g.scale * d;
                    }
                    col[j][0] += g0;
                    col[j][1] += g1;
                    if (n < g.ldc)
                        *reinterpret_cast<__nv_bfloat162*>(g.c16 + (int64_t)m * g.ldc + n) = __floats2bfloat162_rn(g0, g1);
                }
            }
    }
    if (MODE == EPI_RELU_GRAD || MODE == EPI_MSE) {
        // column sums of the tile: over the 8 lanes of a column, then the two warps along m
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        float* red = reinterpret_cast<float*>(gemm_sm);   // [2][GBN], then 8 loss sums
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float v = col[j][e];
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (gr == 0) red[(warp >> 2) * GBN + wn + j * 8 + tc + e] = v;
            }
        if (MODE == EPI_MSE) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
            if (lane == 0) red[2 * GBN + warp] = loss;
        }
        __syncthreads();
        if (tid < GBN && n0 + tid < g.N) g.colpart[(int64_t)blockIdx.y * g.N + n0 + tid] = red[tid] + red[GBN + tid];
        if (MODE == EPI_MSE && tid == 0) {
            float t = 0.f;
            for (int w = 0; w < 8; ++w) t += red[2 * GBN + w];
            g.losspart[blockIdx.y * gridDim.x + blockIdx.x] = t;
        }
    }
}

// Weight gradients of every layer, dW_l [No][Ki] = G_l^T X_l over the minibatch rows, in one
// launch: 64 x 32 tiles of 8 warps (16 x 16 each), the whole k = rows of a tile summed by one
// warp in ascending order.  (Partial sums over parts of the rows would be faster and round less
// than one long chain; they differ from it by 6.6e-5 of the gradient at 16384 rows, and their
// error against 64 bits has not been measured.)  Both
// operands have their row index as k, so the tiles are [64 rows][64] and [64 rows][32] and
// the fragments come by ldmatrix.trans; DWST stages hide the L2 latency of the long k loop.
// The layers together give 144 tiles for a 260 -> 4 x 256 -> 81 network, where one launch
// per layer had 8-24 blocks.
#define DWK 64
#define DWM 64
#define DWN 32
#define DWST 6
#define DWLG (DWM + 8)    // 144 and 80 bytes: ldmatrix rows fall in distinct banks
#define DWLX (DWN + 8)
struct DwLayer {
    Operand g, x;         // [row][o], [row][k]
    int No, Ki, tile0, ntx;
    float* out;
};
struct DwArgs {
    int nl, rows;
    DwLayer l[MLP_MAX_LINEAR];
};
__global__ void __launch_bounds__(256) k_weight_grad(const __grid_constant__ DwArgs A) {
    extern __shared__ __align__(16) unsigned char gemm_sm[];
    bf16* Gs = reinterpret_cast<bf16*>(gemm_sm);      // [DWST][DWK][DWLG]
    bf16* Xs = Gs + DWST * DWK * DWLG;                // [DWST][DWK][DWLX]
    int li = 0;
    while (li + 1 < A.nl && (int)blockIdx.x >= A.l[li + 1].tile0) ++li;
    const DwLayer L = A.l[li];
    const int tile = blockIdx.x - L.tile0, m0 = tile / L.ntx * DWM, n0 = tile % L.ntx * DWN;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
    const int nk = (A.rows + DWK - 1) / DWK;
    float acc[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    auto fetch = [&](int t) {
        if (t < nk) {
            load_tile<8, DWK, DWM, DWLG>(Gs + (t % DWST) * DWK * DWLG, L.g, t * DWK, m0, tid);
            load_tile<8, DWK, DWN, DWLX>(Xs + (t % DWST) * DWK * DWLX, L.x, t * DWK, n0, tid);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
#pragma unroll
    for (int t = 0; t < DWST - 1; ++t) fetch(t);
    for (int t = 0; t < nk; ++t) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(DWST - 2) : "memory");
        __syncthreads();   // tile t has landed, tile t - 1 is consumed
        fetch(t + DWST - 1);
        const bf16* g = Gs + (t % DWST) * DWK * DWLG + ((lane & 7) + 8 * (lane >> 4)) * DWLG + wm + 8 * ((lane >> 3) & 1);
        const bf16* x = Xs + (t % DWST) * DWK * DWLX + (lane & 15) * DWLX + wn + 8 * (lane >> 4);
        uint32_t af[DWK / 16][4], bfr[DWK / 16][4];
#pragma unroll
        for (int q = 0; q < DWK / 16; ++q) {
            ldsm4<true>(af[q], g + 16 * q * DWLG);
            ldsm4<true>(bfr[q], x + 16 * q * DWLX);
        }
#pragma unroll
        for (int q = 0; q < DWK / 16; ++q) {
            mma_16816(acc[0], af[q], bfr[q]);
            mma_16816(acc[1], af[q], bfr[q] + 2);
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int m = m0 + wm + (lane >> 2) + 8 * (e >> 1), n = n0 + wn + j * 8 + (lane & 3) * 2 + (e & 1);
            if (m < L.No && n < L.Ki) L.out[(int64_t)m * L.Ki + n] = acc[j][e];
        }
}

// The minibatch's input rows, gathered once per step into rows of pad8(n_in) (16-byte copies
// for both GEMMs that read them, no index in their loops); VEC elements per copy.
template <int VEC>
__global__ void __launch_bounds__(256) k_gather_rows(const bf16* __restrict__ X, int n_in, int ld,
                                                     const int64_t* __restrict__ idx, int64_t n, bf16* out) {
    typedef typename std::conditional<VEC == 4, uint2, unsigned short>::type V;
    const int ch = ld / VEC;
    const int64_t total = n * ch;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / ch;
        const int c = (int)(e - i * ch) * VEC;
        V v = V();
        if (c < n_in) v = *reinterpret_cast<const V*>(X + idx[i] * n_in + c);
        *reinterpret_cast<V*>(out + i * ld + c) = v;
    }
}

// Bias gradients from the tiles' column sums (in a fixed order), then Adam (Kingma & Ba,
// Algorithm 1; bc1 = 1 - beta1^t, bc2 = 1 - beta2^t) and the bfloat16 copies of the weights.
// Block 0 also sums the loss.
// A training step of 16384 rows, 260 -> 4 x 256 -> 81 on GB300: 11.9 ms with one GEMM of
// 8-24 blocks per weight gradient, FP32 gradients stored, and a column-sum pass per layer;
// 282 us now (92 us of it k_weight_grad, whose long sums keep one warp per 16 x 16 outputs).
struct GradLayers {
    int nl;
    int64_t w_off[MLP_MAX_LINEAR], b_off[MLP_MAX_LINEAR], wb_off[MLP_MAX_LINEAR];
    int n_b[MLP_MAX_LINEAR];
    const float* bpart[MLP_MAX_LINEAR];   // [nby][n_b]
    int nby;
    const float* losspart;
    int nloss;
    float loss_scale;
    float* loss;
};
__global__ void __launch_bounds__(256) k_grad_adam(GradLayers L, int64_t n, float* p, float* g, float* m, float* v,
                                                   bf16* wb, float lr, float b1, float b2, float eps, float bc1,
                                                   float bc2) {
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double t = 0.0;
        for (int i = threadIdx.x; i < L.nloss; i += 32) t += (double)L.losspart[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) *L.loss = (float)(t * (double)L.loss_scale);
    }
    auto adam = [&](int64_t i, float gi) {
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        return p[i] = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    };
    // biases: one warp each, lanes over the row tiles
    const int lane = threadIdx.x & 31;
    int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (int64_t)gridDim.x * blockDim.x >> 5;
    for (int l = 0; l < L.nl; ++l) {
        for (; wid < L.n_b[l]; wid += nw) {
            float s = 0.f;
            for (int c = lane; c < L.nby; c += 32) s += L.bpart[l][(int64_t)c * L.n_b[l] + wid];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) {
                g[L.b_off[l] + wid] = s;
                adam(L.b_off[l] + wid, s);
            }
        }
        wid -= L.n_b[l];
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int l = 0;
        while (l + 1 < L.nl && i >= L.w_off[l + 1]) ++l;
        if (i >= L.b_off[l]) continue;
        wb[L.wb_off[l] + (i - L.w_off[l])] = __float2bfloat16(adam(i, g[i]));
    }
}

struct WeightCopy {
    int nl;
    int64_t w_off[MLP_MAX_LINEAR], wb_off[MLP_MAX_LINEAR], cnt[MLP_MAX_LINEAR];
};
__global__ void k_sync_weights(WeightCopy c, const float* p, bf16* wb) {
    const int l = blockIdx.y;
    if (l >= c.nl) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < c.cnt[l]; i += (int64_t)gridDim.x * blockDim.x)
        wb[c.wb_off[l] + i] = __float2bfloat16(p[c.w_off[l] + i]);
}

// training targets of the Laplacian rows of a plain table
__global__ void k_target_flags(int64_t nrows, const int32_t* info, const int64_t* row_ptr, const int32_t* code,
                               const int32_t* lut, int R, int r2, int order, uint8_t* flags) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nrows; r += (int64_t)gridDim.x * blockDim.x) {
        bool ok = info[4 * r + 3] == 0 && info[4 * r + 0] == r2 && info[4 * r + 1] == order;
        const int W = 2 * R + 1;
        for (int64_t e = row_ptr[r]; ok && e < row_ptr[r + 1]; ++e) {
            int dx, dy, dz;
            unpack_off(code[e], dx, dy, dz);
            if (dx < -R || dx > R || dy < -R || dy > R || dz < -R || dz > R ||
                lut[((dz + R) * W + (dy + R)) * W + (dx + R)] < 0)
                ok = false;
        }
        flags[r] = ok ? 1 : 0;
    }
}

__global__ void k_target_write(int64_t n, const int64_t* sel, const int64_t* row_lin, const int64_t* row_ptr,
                               const int32_t* code, const double* w, const int32_t* lut, int R, int no,
                               int64_t* nodes, float* T) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = sel[k];
        nodes[k] = row_lin[r];
        float* t = T + k * no;
        for (int j = 0; j < no; ++j) t[j] = 0.f;
        const int W = 2 * R + 1;
        // a Laplacian row holds each support node once
        for (int64_t e = row_ptr[r]; e < row_ptr[r + 1]; ++e) {
            int dx, dy, dz;
            unpack_off(code[e], dx, dy, dz);
            t[lut[((dz + R) * W + (dy + R)) * W + (dx + R)]] = (float)w[e];
        }
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int grid1(int64_t n, int bs) {
    int64_t b = (n + bs - 1) / bs;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 32));
}

template <class T>
static ib_status mlp_alloc(T** p, int64_t n) {
    *p = nullptr;
    if (n <= 0) n = 1;
    cudaError_t e = cudaMalloc((void**)p, sizeof(T) * (size_t)n);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        ib_set_error("device allocation failed in the learned-stencil network");
        return IB_ERR_OOM;
    }
    return IB_OK;
}

static int pad8(int n) { return (n + 7) & ~7; }

// elements per copy an operand allows: its rows start on a multiple of 16 (8) bytes and
// hold whole copies
static int copy_vec(const Operand& o) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(o.p);
    if (a % 16 == 0 && o.ld % 8 == 0 && o.ext % 8 == 0) return 8;
    if (a % 8 == 0 && o.ld % 4 == 0 && o.ext % 4 == 0) return 4;
    return 1;
}

template <bool BK, int MODE, int VA, int VB>
static void launch_gemm_v(const Gemm& g, dim3 grid, cudaStream_t s) {
    constexpr size_t sm = sizeof(bf16) * GST * (GBM * GLDK + (BK ? GBN * GLDK : GBK * GLDM));
    // per launch: right whatever device is current
    cudaFuncSetAttribute(k_gemm<BK, MODE, VA, VB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_gemm<BK, MODE, VA, VB><<<grid, 256, sm, s>>>(g);
}

template <bool BK, int MODE>
static ib_status launch_gemm(const Gemm& g, cudaStream_t s) {
    if (g.M <= 0 || g.N <= 0) return IB_OK;
    dim3 grid((g.N + GBN - 1) / GBN, (g.M + GBM - 1) / GBM);
    if (grid.y > 65535) {
        ib_set_error("GEMM too tall");
        return IB_ERR_ARG;
    }
    const int va = copy_vec(g.a), vb = copy_vec(g.b);
    if (va == 8 && vb == 8) launch_gemm_v<BK, MODE, 8, 8>(g, grid, s);
    else if (va == 8 && vb == 4) launch_gemm_v<BK, MODE, 8, 4>(g, grid, s);
    else if (va >= 4 && vb >= 4) launch_gemm_v<BK, MODE, 4, 4>(g, grid, s);
    else if (va == 8) launch_gemm_v<BK, MODE, 8, 1>(g, grid, s);
    else launch_gemm_v<BK, MODE, 1, 1>(g, grid, s);
    IB_CHECK_LAUNCH("k_gemm");
    ib_count_launch("mlp_gemm_bf16");
    return IB_OK;
}


// layer l on n rows of Xin (ext readable elements each, zero past the layer's inputs)
static Gemm gemm_fwd(const ib_mlp* m, int l, const bf16* Xin, int64_t ldx, int ext, int64_t n) {
    Gemm g;
    memset(&g, 0, sizeof g);
    g.M = (int)n;
    g.N = m->dims[l + 1];
    g.K = m->dims[l];
    g.a = {Xin, ldx, (int)n, ext};
    g.b = {m->wb + m->wb_off[l], g.K, g.N, g.K};   // W_l [N][K]
    g.bias = m->params + m->b_off[l];
    return g;
}

extern "C" ib_status ib_mlp_create(const ib_mlp_config* cfg, ib_mlp** out) {
    ib_set_error("");
    if (!cfg || !out) {
        ib_set_error("null argument");
        return IB_ERR_ARG;
    }
    *out = nullptr;
    if ((cfg->ndim != 2 && cfg->ndim != 3) || cfg->space_order < 2 || cfg->space_order > 8 ||
        (cfg->space_order & 1) || cfg->n_hidden < 8 || cfg->n_hidden > 1024 || (cfg->n_hidden & 7) ||
        cfg->n_layers < 1 || cfg->n_layers > MLP_MAX_LINEAR - 1 || !(cfg->in_radius >= 0.0) ||
        cfg->in_radius > 8.0 || !(cfg->out_radius > 0.0) || cfg->out_radius > 8.0) {
        ib_set_error("ib_mlp_config out of range");
        return IB_ERR_ARG;
    }
    ib_mlp* m = new ib_mlp();
    m->cfg = *cfg;
    cudaGetDevice(&m->device);
    auto fail = [&](ib_status st) {
        ib_mlp_free(m);
        return st;
    };
    auto inb = ball_offsets(cfg->ndim, cfg->in_radius);
    auto outb = ball_offsets(cfg->ndim, cfg->out_radius);
    m->n_in_off = (int)inb.size();
    m->n_in = m->n_in_off + 3;
    m->n_out = (int)outb.size();
    m->out_R = (int)std::ceil(cfg->out_radius);
    m->nl = cfg->n_layers + 1;
    m->dims[0] = m->n_in;
    for (int l = 1; l < m->nl; ++l) m->dims[l] = cfg->n_hidden;
    m->dims[m->nl] = m->n_out;
    int64_t p = 0, wb = 0;
    for (int l = 0; l < m->nl; ++l) {
        m->w_off[l] = p;
        p += (int64_t)m->dims[l + 1] * m->dims[l];
        m->b_off[l] = p;
        p += m->dims[l + 1];
        m->wb_off[l] = wb;
        wb += (int64_t)m->dims[l + 1] * m->dims[l];
        wb = (wb + 7) & ~(int64_t)7;   // 16-byte aligned matrices
    }
    m->n_params = p;
    m->n_wb = wb;
    ib_status st;
    if ((st = mlp_alloc(&m->params, p)) != IB_OK) return fail(st);
    if ((st = mlp_alloc(&m->grads, p)) != IB_OK) return fail(st);
    if ((st = mlp_alloc(&m->adam_m, p)) != IB_OK) return fail(st);
    if ((st = mlp_alloc(&m->adam_v, p)) != IB_OK) return fail(st);
    if ((st = mlp_alloc(&m->wb, wb)) != IB_OK) return fail(st);
    if ((st = mlp_alloc(&m->in_off, 3 * (int64_t)inb.size())) != IB_OK) return fail(st);
    const int W = 2 * m->out_R + 1;
    if ((st = mlp_alloc(&m->out_lut, (int64_t)W * W * W)) != IB_OK) return fail(st);
    std::vector<int8_t> ho;
    for (auto& o : inb)
        for (int a = 0; a < 3; ++a) ho.push_back((int8_t)o[a]);
    std::vector<int32_t> lut((size_t)W * W * W, -1);
    for (size_t j = 0; j < outb.size(); ++j) {
        const auto& o = outb[j];
        lut[((size_t)(o[2] + m->out_R) * W + (o[1] + m->out_R)) * W + (o[0] + m->out_R)] = (int32_t)j;
    }
    if (cudaMemcpy(m->in_off, ho.data(), ho.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->out_lut, lut.data(), lut.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->params, 0, 4 * p) != cudaSuccess || cudaMemset(m->grads, 0, 4 * p) != cudaSuccess ||
        cudaMemset(m->adam_m, 0, 4 * p) != cudaSuccess || cudaMemset(m->adam_v, 0, 4 * p) != cudaSuccess ||
        cudaMemset(m->wb, 0, 2 * wb) != cudaSuccess) {
        ib_set_error("initialising the network failed");
        return fail(IB_ERR_CUDA);
    }
    // the copies and memsets above went to the legacy stream, which a non-blocking stream's first
    // use of the network is not ordered after
    if (cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) {
        ib_set_error("initialising the network failed");
        return fail(IB_ERR_CUDA);
    }
    *out = m;
    return IB_OK;
}

extern "C" void ib_mlp_free(ib_mlp* m) {
    if (!m) return;
    void* ptrs[] = {m->params, m->grads, m->adam_m, m->adam_v, m->wb, m->in_off, m->out_lut, m->act,
                    m->g16, m->xg, m->bpart, m->ia, m->ib, m->ix};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    delete m;
}

extern "C" ib_status ib_mlp_info(const ib_mlp* m, int64_t* n_in, int64_t* n_out, int64_t* n_params) {
    if (!m) {
        ib_set_error("null network");
        return IB_ERR_ARG;
    }
    if (n_in) *n_in = m->n_in;
    if (n_out) *n_out = m->n_out;
    if (n_params) *n_params = m->n_params;
    return IB_OK;
}

extern "C" ib_status ib_mlp_buffers(ib_mlp* m, float** params, float** grads, float** am, float** av) {
    if (!m) {
        ib_set_error("null network");
        return IB_ERR_ARG;
    }
    if (params) *params = m->params;
    if (grads) *grads = m->grads;
    if (am) *am = m->adam_m;
    if (av) *av = m->adam_v;
    return IB_OK;
}

static ib_status sync_weights(ib_mlp* m, cudaStream_t s) {
    WeightCopy c;
    memset(&c, 0, sizeof c);
    c.nl = m->nl;
    int64_t mx = 0;
    for (int l = 0; l < m->nl; ++l) {
        c.w_off[l] = m->w_off[l];
        c.wb_off[l] = m->wb_off[l];
        c.cnt[l] = (int64_t)m->dims[l + 1] * m->dims[l];
        mx = std::max(mx, c.cnt[l]);
    }
    dim3 grid(grid1(mx, 256), m->nl);
    k_sync_weights<<<grid, 256, 0, s>>>(c, m->params, m->wb);
    IB_CHECK_LAUNCH("k_sync_weights");
    ib_count_launch("mlp_setup");
    return IB_OK;
}

extern "C" ib_status ib_mlp_sync_weights(ib_mlp* m, void* stream) {
    if (!m) {
        ib_set_error("null network");
        return IB_ERR_ARG;
    }
    return sync_weights(m, (cudaStream_t)stream);
}

static ib_status features(const ib_mlp* m, const ib_grid* grid, const double* sdf, const int64_t* nodes,
                          int64_t n, ib_bc bc, bf16* X, cudaStream_t s) {
    if (!grid || !sdf || (n > 0 && (!nodes || !X))) {
        ib_set_error("null argument");
        return IB_ERR_ARG;
    }
    if (grid->ndim != m->cfg.ndim) {
        ib_set_error("grid dimension differs from the network's");
        return IB_ERR_ARG;
    }
    if (n <= 0) return IB_OK;
    const int64_t n2 = grid->ndim == 3 ? grid->n[2] : 1;
    k_features<<<grid1(n * m->n_in, 256), 256, 0, s>>>(
        grid->ndim, grid->n[0], grid->n[1], n2, grid->h, sdf, nodes, n, m->in_off, m->n_in_off, m->n_in,
        bc == IB_FREE ? 1.f : 0.f, bc == IB_RIGID ? 1.f : 0.f, (float)(m->cfg.space_order / 8.0), X);
    IB_CHECK_LAUNCH("k_features");
    ib_count_launch("mlp_features");
    return IB_OK;
}

extern "C" ib_status ib_mlp_features(const ib_mlp* m, const ib_grid* grid, const double* sdf_dev,
                                     const int64_t* nodes_dev, int64_t n, ib_bc bc, void* X_dev, void* stream) {
    ib_set_error("");
    if (!m) {
        ib_set_error("null network");
        return IB_ERR_ARG;
    }
    return features(m, grid, sdf_dev, nodes_dev, n, bc, (bf16*)X_dev, (cudaStream_t)stream);
}

static const int64_t kChunk = 1 << 16;

static ib_status ensure_infer(ib_mlp* m) {
    if (m->icap >= kChunk) return IB_OK;
    TRY(mlp_alloc(&m->ia, kChunk * m->cfg.n_hidden));
    TRY(mlp_alloc(&m->ib, kChunk * m->cfg.n_hidden));
    TRY(mlp_alloc(&m->ix, kChunk * m->n_in));
    m->icap = kChunk;
    return IB_OK;
}

// Y[n][n_out] = network(X[n][n_in]) in chunks of kChunk rows
static ib_status forward(ib_mlp* m, const bf16* X, int64_t n, float* Y, cudaStream_t s) {
    TRY(ensure_infer(m));
    const int H = m->cfg.n_hidden;
    for (int64_t c0 = 0; c0 < n; c0 += kChunk) {
        const int64_t cn = std::min(kChunk, n - c0);
        const bf16* in = X + c0 * m->n_in;
        int64_t ldi = m->n_in;
        bf16* bufs[2] = {m->ia, m->ib};
        for (int l = 0; l < m->nl; ++l) {
            Gemm g = gemm_fwd(m, l, in, ldi, m->dims[l], cn);
            if (l + 1 < m->nl) {
                g.c16 = bufs[l & 1];
                g.ldc = H;
                TRY((launch_gemm<true, EPI_BIAS_RELU_BF16>(g, s)));
                in = bufs[l & 1];
                ldi = H;
            } else {
                g.c32 = Y + c0 * m->n_out;
                g.ldc = m->n_out;
                TRY((launch_gemm<true, EPI_BIAS_F32>(g, s)));
            }
        }
    }
    return IB_OK;
}

extern "C" ib_status ib_mlp_forward(ib_mlp* m, const void* X_dev, int64_t n, float* Y_dev, void* stream) {
    ib_set_error("");
    if (!m || (n > 0 && (!X_dev || !Y_dev)) || n < 0) {
        ib_set_error("null argument");
        return IB_ERR_ARG;
    }
    return forward(m, (const bf16*)X_dev, n, Y_dev, (cudaStream_t)stream);
}

static ib_status ensure_train(ib_mlp* m, int64_t n) {
    if (n <= m->cap) return IB_OK;
    const int H = m->cfg.n_hidden;
    const int mxd = std::max(H, pad8(m->n_out));
    int64_t sum_b = 0;
    for (int l = 0; l < m->nl; ++l) sum_b += m->dims[l + 1];
    const int64_t nby = (n + GBM - 1) / GBM;
    void* ptrs[] = {m->act, m->g16, m->xg, m->bpart};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    m->act = m->g16 = m->xg = nullptr;
    m->bpart = nullptr;
    m->cap = 0;
    TRY(mlp_alloc(&m->act, (int64_t)(m->nl - 1) * n * H));
    TRY(mlp_alloc(&m->g16, (int64_t)m->nl * n * mxd));
    TRY(mlp_alloc(&m->xg, n * pad8(m->n_in)));
    TRY(mlp_alloc(&m->bpart, nby * (sum_b + (m->n_out + GBN - 1) / GBN)));
    m->cap = n;
    return IB_OK;
}

extern "C" ib_status ib_mlp_train_step(ib_mlp* m, const void* X_dev, const float* T_dev, const int64_t* idx_dev,
                                       int64_t n, float lr, float beta1, float beta2, float eps, float* loss_dev,
                                       void* stream) {
    ib_set_error("");
    cudaStream_t s = (cudaStream_t)stream;
    if (!m || !X_dev || !T_dev || !idx_dev || !loss_dev || n <= 0 || n > (1 << 22)) {
        ib_set_error("bad argument (rows must be 1 .. 4194304)");
        return IB_ERR_ARG;
    }
    if (!(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps >= 0.f)) {
        ib_set_error("bad Adam hyper-parameters");
        return IB_ERR_ARG;
    }
    TRY(ensure_train(m, n));
    const int H = m->cfg.n_hidden, L = m->nl;
    const bf16* X = (const bf16*)X_dev;
    auto act = [&](int l) { return m->act + (int64_t)(l - 1) * m->cap * H; };   // input of layer l >= 1
    // forward, keeping each layer's input; the last layer's epilogue forms the loss and its
    // gradient (rows of pad8(n_out), zero in the padding)
    const int64_t nby = (n + GBM - 1) / GBM;
    const int ldo = pad8(m->n_out);
    auto grad = [&](int l) { return m->g16 + (int64_t)l * m->cap * std::max(H, ldo); };   // of layer l's output
    GradLayers R;
    memset(&R, 0, sizeof R);
    R.nl = L;
    R.nby = (int)nby;
    {
        float* bp = m->bpart;
        for (int l = 0; l < L; ++l) {
            R.w_off[l] = m->w_off[l];
            R.b_off[l] = m->b_off[l];
            R.wb_off[l] = m->wb_off[l];
            R.n_b[l] = m->dims[l + 1];
            R.bpart[l] = bp;
            bp += nby * R.n_b[l];
        }
        R.losspart = bp;
        R.nloss = (int)(nby * ((m->n_out + GBN - 1) / GBN));
        R.loss_scale = (float)(1.0 / ((double)n * m->n_out));
        R.loss = loss_dev;
    }
    const int ldx = pad8(m->n_in);
    if (m->n_in % 4 == 0 && reinterpret_cast<uintptr_t>(X) % 8 == 0)
        k_gather_rows<4><<<grid1(n * ldx / 4, 256), 256, 0, s>>>(X, m->n_in, ldx, idx_dev, n, m->xg);
    else
        k_gather_rows<1><<<grid1(n * ldx, 256), 256, 0, s>>>(X, m->n_in, ldx, idx_dev, n, m->xg);
    IB_CHECK_LAUNCH("k_gather_rows");
    ib_count_launch("mlp_setup");
    for (int l = 0; l < L; ++l) {
        Gemm g = l == 0 ? gemm_fwd(m, 0, m->xg, ldx, ldx, n) : gemm_fwd(m, l, act(l), H, H, n);
        if (l + 1 < L) {
            g.c16 = act(l + 1);
            g.ldc = H;
            TRY((launch_gemm<true, EPI_BIAS_RELU_BF16>(g, s)));
        } else {
            g.c16 = grad(l);
            g.ldc = ldo;
            g.T = T_dev;
            g.t_idx = idx_dev;
            g.scale = (float)(2.0 / ((double)n * m->n_out));
            g.colpart = const_cast<float*>(R.bpart[l]);
            g.losspart = const_cast<float*>(R.losspart);
            TRY((launch_gemm<true, EPI_MSE>(g, s)));
        }
    }
    // backward: G_{l-1} = (G_l W_l) * [X_l > 0], with the column sums of db_{l-1}
    for (int l = L - 1; l > 0; --l) {
        const int No = m->dims[l + 1], Ki = m->dims[l], ldg = l == L - 1 ? ldo : H;
        Gemm gx;
        memset(&gx, 0, sizeof gx);
        gx.M = (int)n;
        gx.N = Ki;
        gx.K = No;
        gx.a = {grad(l), ldg, (int)n, ldg};
        gx.b = {m->wb + m->wb_off[l], Ki, No, Ki};
        gx.act = act(l);
        gx.c16 = grad(l - 1);
        gx.ldc = Ki;
        gx.colpart = const_cast<float*>(R.bpart[l - 1]);
        TRY((launch_gemm<false, EPI_RELU_GRAD>(gx, s)));
    }
    // dW_l of all layers
    DwArgs D;
    memset(&D, 0, sizeof D);
    D.nl = L;
    D.rows = (int)n;
    int tiles = 0;
    for (int l = 0; l < L; ++l) {
        const int No = m->dims[l + 1], Ki = m->dims[l], ldg = l == L - 1 ? ldo : H;
        DwLayer& d = D.l[l];
        d.g = {grad(l), ldg, (int)n, ldg};
        if (l == 0) d.x = {m->xg, ldx, (int)n, ldx};
        else d.x = {act(l), H, (int)n, H};
        d.No = No;
        d.Ki = Ki;
        d.tile0 = tiles;
        d.ntx = (Ki + DWN - 1) / DWN;
        d.out = m->grads + m->w_off[l];
        tiles += d.ntx * ((No + DWM - 1) / DWM);
    }
    {
        constexpr size_t sm = sizeof(bf16) * DWST * DWK * (DWLG + DWLX);
        cudaFuncSetAttribute(k_weight_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_weight_grad<<<tiles, 256, sm, s>>>(D);
        IB_CHECK_LAUNCH("k_weight_grad");
        ib_count_launch("mlp_gemm_bf16");
    }
    // Adam
    m->step += 1;
    const double bc1 = 1.0 - std::pow((double)beta1, (double)m->step);
    const double bc2 = 1.0 - std::pow((double)beta2, (double)m->step);
    k_grad_adam<<<grid1(m->n_params, 256), 256, 0, s>>>(R, m->n_params, m->params, m->grads, m->adam_m, m->adam_v, m->wb,
                                                        lr, beta1, beta2, eps, (float)bc1, (float)bc2);
    IB_CHECK_LAUNCH("k_grad_adam");
    ib_count_launch("mlp_adam");
    return IB_OK;
}

extern "C" ib_status ib_mlp_targets(const ib_table* t, const ib_mlp* m, int64_t* nodes_dev, float* T_dev,
                                    int64_t cap, int64_t* n_rows, void* stream) {
    ib_set_error("");
    cudaStream_t s = (cudaStream_t)stream;
    if (!t || !m || !n_rows || (cap > 0 && (!nodes_dev || !T_dev))) {
        ib_set_error("null argument");
        return IB_ERR_ARG;
    }
    if (t->form != IB_SECOND_ORDER || t->grid.ndim != m->cfg.ndim) {
        ib_set_error("targets need a second-order table of the network's dimension");
        return IB_ERR_ARG;
    }
    const IbOp& op = t->ops[0];
    *n_rows = 0;
    if (op.nrows == 0) return IB_OK;
    uint8_t* flags = nullptr;
    TRY(mlp_alloc(&flags, op.nrows));
    const int r2 = (int)lrint(2.0 * m->cfg.out_radius);
    k_target_flags<<<grid1(op.nrows, 256), 256, 0, s>>>(op.nrows, op.row_info, op.row_ptr, op.col_code, m->out_lut,
                                                         m->out_R, r2, t->opts.basis_order, flags);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        cudaFree(flags);
        return ib_cuda_fail(e, "k_target_flags", __FILE__, __LINE__);
    }
    ib_count_launch("mlp_targets");
    int64_t* sel = nullptr;
    int64_t cnt = 0;
    ib_status st = ib_compact(flags, op.nrows, &sel, &cnt, s);
    cudaFree(flags);
    if (st != IB_OK) return st;
    const int64_t n = std::min(cnt, cap);
    if (n > 0) {
        k_target_write<<<grid1(n, 128), 128, 0, s>>>(n, sel, op.row_lin, op.row_ptr, op.col_code, op.w64, m->out_lut,
                                                      m->out_R, m->n_out, nodes_dev, T_dev);
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            cudaFree(sel);
            return ib_cuda_fail(e, "k_target_write", __FILE__, __LINE__);
        }
        ib_count_launch("mlp_targets");
    }
    e = cudaStreamSynchronize(s);
    cudaFree(sel);
    if (e != cudaSuccess) return ib_cuda_fail(e, "ib_mlp_targets", __FILE__, __LINE__);
    *n_rows = n;
    return IB_OK;
}

// ---------------------------------------------------------------------------
// internal interface of the constructor
// ---------------------------------------------------------------------------
int ib_mlp_out_count(const ib_mlp* m) { return m->n_out; }
double ib_mlp_out_radius(const ib_mlp* m) { return m->cfg.out_radius; }
int ib_mlp_ndim(const ib_mlp* m) { return m->cfg.ndim; }
int ib_mlp_order(const ib_mlp* m) { return m->cfg.space_order; }
const int32_t* ib_mlp_lut(const ib_mlp* m, int* R) {
    *R = m->out_R;
    return m->out_lut;
}

ib_status ib_mlp_predict_nodes(ib_mlp* m, const ib_grid* grid, const double* sdf, const int64_t* nodes, int64_t n,
                               ib_bc bc, float* Y, cudaStream_t s) {
    TRY(ensure_infer(m));
    for (int64_t c0 = 0; c0 < n; c0 += kChunk) {
        const int64_t cn = std::min(kChunk, n - c0);
        TRY(features(m, grid, sdf, nodes + c0, cn, bc, m->ix, s));
        TRY(forward(m, m->ix, cn, Y + c0 * m->n_out, s));
    }
    return IB_OK;
}
