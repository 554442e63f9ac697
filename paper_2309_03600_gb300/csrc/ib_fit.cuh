// The constrained fit of an immersed-boundary row by one warp (basis order <= 4, at most 35
// unknowns: 2D, 2D staggered and 3D scalar rows).  The steps, decisions and row contents are
// those of k_fit, which keeps the larger fits and the rows that outgrow a warp's buffers.
//
// What bounds it is the FP64 pipe, which issues a warp instruction every 16 cycles per SM
// whatever the number of active lanes; k_fit spent 11 k of them on a 3D order-8 row (35
// unknowns, ~120 rows of A), about half with idle lanes.  Here a row takes about 2.5 k:
//   - The interior rows of A are monomials of lattice offsets, the same for every IB row, so
//     their values are tables, and their share of the Gram matrix follows from the moments
//     sum x^gamma (|gamma| <= 2P) of the support: integers in doubled coordinates, summed
//     exactly in 64-bit integers over the chosen or over the missing offsets, whichever are
//     fewer.
//   - Boundary-condition rows are linear combinations of the monomials of their boundary
//     point (8 points at a time in shared memory); constant rows enter in closed form.
//   - The Gram matrix is factored as U^T D U and U inverted in the same sweep, over packed
//     element lists that keep all lanes busy; V = U^{-1} serves the solves and the rank test.
//   - The rank test iterates in FP32 on A^T A and (R R^T)^{-1} held in registers, the
//     iterations of k_fit on the same starting vectors.
//   - y = A z is refined by the corrected seminormal equations: rho = u - A^T y, y += A
//     (A^T A)^{-1} rho.
// One warp per block: rows are independent and a warp never waits for another.  Warps at
// different phases share the instruction cache, so the code is kept small (loops over the
// triangle instead of unrolled register tiles, calls for what appears twice): with the tiles
// unrolled and everything inlined an SM waited for instructions most of the time and the FP64
// pipe was 34-36 % busy at 8 and at 11 warps alike.
//
// Measured on GB300, 65,536 rows of a 128 x 128 x 96 hills surface at order 8: 54 ms in k_fit,
// 12.7 ms here (FP64 pipe 57 % busy); ib_build_stencils of 256 x 256 x 192 (262,144 rows) with the training rows
// taken from the table 410 ms -> 56.5 ms, of which a factor of two is the room for the
// entries (see run_fit), whose overflow had every 3D table fitted twice.
#pragma once

#define RF_CAP 320      // support nodes of a row
#define RF_BP 64        // boundary points of a row
#define RF_CB 8         // boundary points per chunk
#define RF_NG (32 / RF_CB)
#define RF_PITCH 10     // doubles per column of a chunk (16-byte reads of 8 columns fall in distinct banks)
#define RF_MAXCOL 35    // unknowns: the FP32 triangle of V fits the RF_CAP doubles of y
#define RF_GROW 17

struct RowOrder {
    int order, T, n, np, nbc;
    double r0;
    int gpad;                    // moments per field, padded to whole warps
    const int32_t* mom;          // [field][candidate][gpad] moments of doubled offsets
    const long long* full;       // [field][growth][gpad] their sums over the whole ball
    const double* phi;           // [field][candidate][T]
    const double* phiT;          // [field][T][candidates]
    const uint16_t* pair;        // [np] i | j << 8, row by row of the upper triangle
    const int16_t* pgam;         // [np] moment index (field * gpad + ..) or -1
    const double* pcoef;         // [np] 2^-|gamma| / (alpha_i! alpha_j!)
    const double* pconst;        // [np] sum over the constant rows of c_i c_j
    const double* uE;            // [stencil point][n] weighted basis row of an exterior point
    int nrow, nconst;            // non-constant and constant boundary-condition rows
    int ident;                   // the non-constant row that is the monomials themselves, or -1
    const int32_t* prog_ptr;     // [nrow][n + 1]
    const uint32_t* prog;        // monomial | (axis + 1) << 8
    const double* prog_c;
    const double* crow;          // [nconst][n]
    const uint32_t* mono;        // [T] parent | axis << 8 | exponent << 16 | degree << 24
    int nb[3][RF_GROW];          // candidates per field within the radius
    int lo[3][RF_GROW], hi[3][RF_GROW];   // owners of boundary points in reach, from the row node
};

struct RowFit {
    RowOrder ord[FIT_MAX_ORDERS];
    const uint8_t* kept[3];      // [N] interior and outside every eta box
    int ncand[3];
    int bc_doubles;              // shared doubles of a chunk (monomials and rows)
    unsigned long long* next;    // row queue
    int32_t* redo;               // rows left to k_fit
    unsigned int* nredo;
};

// interior nodes of a field, then without those that have a boundary point strictly inside
// their 2 eta box
__global__ void k_kept(Geo g, int kind, uint8_t* kept) {
    const int64_t N = g.n[0] * g.n[1] * (g.ndim == 3 ? g.n[2] : 1);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t p[3];
        p[0] = i % g.n[0];
        const int64_t r = i / g.n[0];
        p[1] = g.ndim == 3 ? r % g.n[1] : r;
        p[2] = g.ndim == 3 ? r / g.n[1] : 0;
        kept[i] = field_interior(g, kind, p) ? 1 : 0;
    }
}
struct EtaBox {
    int reach;
    int shift2[3];
    double eta;
};
__global__ void k_eta_drop(Geo g, int64_t nbp, const int64_t* __restrict__ owner, const double* __restrict__ xb, EtaBox b,
                           uint8_t* kept) {
    const int R = b.reach, W = 2 * R + 1, cells = g.ndim == 3 ? W * W * W : W * W;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nbp * cells;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = i / cells, lin = owner[k];
        int c = (int)(i - k * cells);
        int64_t q[3];
        q[0] = lin % g.n[0];
        const int64_t r = lin / g.n[0];
        q[1] = g.ndim == 3 ? r % g.n[1] : r;
        q[2] = g.ndim == 3 ? r / g.n[1] : 0;
        double mx = 0.0;
        for (int a = 0; a < g.ndim; ++a) {
            q[a] += c % W - R;
            c /= W;
            mx = fmax(mx, fabs(xb[3 * k + a] - ((double)q[a] + 0.5 * b.shift2[a])));
        }
        if (mx < b.eta && in_arr(g, q)) kept[lin_p(g, q)] = 0;
    }
}

__device__ __forceinline__ double rf_shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

// 1 / x by Newton's method from the FP32 reciprocal (x > 0, within the FP32 range)
__device__ __forceinline__ double rf_rcp(double x) {
    double r = (double)(1.0f / (float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}
__device__ __forceinline__ int rf_off(int i, int n) { return i * (2 * n - 1 - i) / 2; }   // + j: element (i, j), j >= i

// Square root of the largest eigenvalue of the symmetric F (FP32, columns of pitch NMAX, zero
// past n) by power iteration: k_fit's block_sigma_max on M with M^T M = F.  A lane keeps its
// rows of F in registers.
template <int NMAX>
__device__ __noinline__ float rf_sigma(const float* F, int n, float* v, int iters) {
    constexpr int NS = (NMAX + 31) / 32, NV = NMAX / 4;
    const int lane = threadIdx.x;
    float a[NS][NMAX];
    __syncwarp();
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int c = 0; c < NMAX; ++c) a[s][c] = lane + 32 * s < NMAX ? F[c * NMAX + lane + 32 * s] : 0.f;
    float t0 = 0.f;
    for (int i = lane; i < NMAX; i += 32) {
        v[i] = i < n ? 1.f + 0.01f * (float)(i % 5) : 0.f;
        t0 += v[i] * v[i];
    }
    for (int o = 16; o > 0; o >>= 1) t0 += __shfl_xor_sync(0xffffffffu, t0, o);
    const float nrm = sqrtf(t0);
    for (int i = lane; i < n; i += 32) v[i] /= nrm;
    __syncwarp();
    float lam = 0.f;
    for (int it = 0; it < iters; ++it) {
        float t[NS][4];
#pragma unroll
        for (int s = 0; s < NS; ++s) t[s][0] = t[s][1] = t[s][2] = t[s][3] = 0.f;
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            const float4 x = *reinterpret_cast<const float4*>(v + 4 * c);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                t[s][0] += a[s][4 * c] * x.x;
                t[s][1] += a[s][4 * c + 1] * x.y;
                t[s][2] += a[s][4 * c + 2] * x.z;
                t[s][3] += a[s][4 * c + 3] * x.w;
            }
        }
        float w[NS], t2 = 0.f;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            w[s] = (t[s][0] + t[s][1]) + (t[s][2] + t[s][3]);
            t2 += w[s] * w[s];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, o);
        lam = sqrtf(t2);
        if (!(lam > 0.f) || !(lam < 3e38f)) return lam;
        __syncwarp();
#pragma unroll
        for (int s = 0; s < NS; ++s)
            if (lane + 32 * s < n) v[lane + 32 * s] = w[s] / lam;
        __syncwarp();
    }
    return sqrtf(lam);
}

// shared memory of one warp (carved by k_fit_rows)
struct RfSmem {
    double *M, *bc, *vec, *y, *sb, *dinv;
    float *GF, *fv;
    uint32_t* words;
    uint16_t* sup;
    int32_t* bps;
};

// monomials and boundary-condition rows of the boundary points b0 .. of a row's list
__device__ __noinline__ void rf_chunk(const FitParams& P, const RowOrder& o, const RfSmem& S, const double x0[3], int b0,
                                         int nbp) {
    const int lane = threadIdx.x, b = lane % RF_CB, h = lane / RF_CB;
    const bool act = b0 + b < nbp;
    double x[3] = {0.0, 0.0, 0.0}, nn[3] = {0.0, 0.0, 0.0};
    if (act) {
        const int id = S.bps[b0 + b];
        for (int a = 0; a < 3; ++a) {
            if (a < P.g.ndim) x[a] = P.bp_xb[3 * id + a] - x0[a];
            nn[a] = P.bp_n[3 * id + a];
        }
    }
    double* phi = S.bc;
    __syncwarp();
    if (h == 0) phi[b] = act ? 1.0 : 0.0;
    int k0 = 1;
    for (int deg = 1; deg <= o.order; ++deg) {
        __syncwarp();
        int k = k0 + h;
        for (; k < o.T; k += RF_NG) {
            const uint32_t m = o.mono[k];
            if ((int)(m >> 24) != deg) break;
            const int ax = (m >> 8) & 0xff;
            const double xa = ax == 0 ? x[0] : ax == 1 ? x[1] : x[2];
            phi[k * RF_PITCH + b] = phi[(m & 0xff) * RF_PITCH + b] * (xa * c_inv_int[(m >> 16) & 0xff]);
        }
        while (k0 < o.T && (int)(o.mono[k0] >> 24) == deg) ++k0;
    }
    __syncwarp();
    double* row = phi + o.T * RF_PITCH;
    for (int r = 0; r < o.nrow; ++r) {
        if (r == o.ident) continue;
        const int32_t* pp = o.prog_ptr + r * (o.n + 1);
        for (int c = h; c < o.n; c += RF_NG) {
            double v = 0.0;
            for (int t = pp[c]; t < pp[c + 1]; ++t) {
                const uint32_t w = o.prog[t];
                const int ax = (int)(w >> 8) - 1;
                double f = o.prog_c[t] * phi[(w & 0xff) * RF_PITCH + b];
                if (ax >= 0) f *= ax == 0 ? nn[0] : ax == 1 ? nn[1] : nn[2];
                v += f;
            }
            row[c * RF_PITCH + b] = v;
        }
        row += o.n * RF_PITCH;
    }
    __syncwarp();
}

// out = (A^T A)^{-1} in = V D^{-1} V^T in, V unit upper in S.M
__device__ __noinline__ void rf_solve(const RfSmem& S, int n, const double* in, double* tmp, double* out) {
    const int lane = threadIdx.x;
    __syncwarp();
    for (int j = lane; j < n; j += 32) {
        double s = in[j];
        for (int i = 0; i < j; ++i) s = fma(S.M[rf_off(i, n) + j], in[i], s);
        tmp[j] = s * S.dinv[j];
    }
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
        const double* row = S.M + rf_off(i, n);
        double s = tmp[i];
        for (int j = n - 1; j > i; --j) s = fma(row[j], tmp[j], s);
        out[i] = s;
    }
    __syncwarp();
}

template <int NMAX>
__global__ void __launch_bounds__(32) k_fit_rows(const __grid_constant__ FitParams P, const __grid_constant__ RowFit R) {
    constexpr int NPP = NMAX * (NMAX + 1) / 2;
    extern __shared__ __align__(16) double rf_sm[];
    RfSmem S;
    S.M = rf_sm;
    S.bc = S.M + NPP;
    S.vec = S.bc + R.bc_doubles;                 // 6 x NMAX: u, z, rho, tmp, g, t
    S.dinv = S.vec + 6 * NMAX;
    S.y = S.dinv + NMAX;                         // RF_CAP (moments before the Gram matrix)
    S.sb = S.y + RF_CAP;                         // 8 x RF_CB
    S.GF = (float*)(S.sb + 8 * RF_CB);           // NMAX x NMAX
    S.fv = S.GF + NMAX * NMAX;                   // 40
    S.words = (uint32_t*)(S.fv + 40);            // 3 x 24
    S.bps = (int32_t*)(S.words + 72);
    S.sup = (uint16_t*)(S.bps + RF_BP);
    const int lane = threadIdx.x;
    double* u = S.vec;
    double* z = S.vec + NMAX;
    double* rho = S.vec + 2 * NMAX;
    double* tmp = S.vec + 3 * NMAX;
    double* gb = S.vec + 4 * NMAX;
    double* tb = S.vec + 5 * NMAX;
    for (;;) {
        unsigned long long rq = 0;
        if (lane == 0) rq = atomicAdd(R.next, 1ull);
        const int64_t row = (int64_t)__shfl_sync(0xffffffffu, rq, 0);
        if (row >= P.nrows) break;
        if (P.accepted && P.accepted[row]) continue;
        const int64_t lin = P.rows[row];
        int64_t node[3];
        node[0] = lin % P.g.n[0];
        const int64_t rr = lin / P.g.n[0];
        node[1] = P.g.ndim == 3 ? rr % P.g.n[1] : rr;
        node[2] = P.g.ndim == 3 ? rr / P.g.n[1] : 0;
        double x0[3];
        for (int a = 0; a < 3; ++a) x0[a] = (double)node[a] + 0.5 * P.x0shift2[a];
        bool ext = false;
        if (lane < P.rule.nE) {
            const int64_t q[3] = {node[0] + P.rule.Eoff[lane][0], node[1] + P.rule.Eoff[lane][1],
                                  node[2] + P.rule.Eoff[lane][2]};
            ext = in_arr(P.g, q) && !field_interior(P.g, P.rule.Efield[lane], q);
        }
        const unsigned emask = __ballot_sync(0xffffffffu, ext);
        int status = 1, used_order = 0, used_r2 = 0, used_nbp = 0, nsup_final = 0;
        bool done = false, redo = false;
        for (int oi = 0; oi < P.norders && !done; ++oi) {
            const RowOrder& o = R.ord[oi];
            const int n = o.n, T = o.T, np = o.np;
            for (int g = 0; g <= P.ngrow && !done; ++g) {
                const double r = o.r0 + 0.5 * g;
                // ---- interior support, in the order of the balls
                int nsup = 0, nsf[3] = {0, 0, 0};
                __syncwarp();
                for (int f = 0; f < P.nf; ++f) {
                    const int nb = o.nb[f][g];
                    for (int c0 = 0; c0 < nb; c0 += 32) {
                        const int c = c0 + lane;
                        bool ok = false;
                        if (c < nb) {
                            const int8_t* bo = P.ball_off[f] + 3 * c;
                            const int64_t q[3] = {node[0] + bo[0], node[1] + bo[1], node[2] + bo[2]};
                            ok = in_arr(P.g, q) && R.kept[f][lin_p(P.g, q)] != 0;
                        }
                        const unsigned w = __ballot_sync(0xffffffffu, ok);
                        const int at = nsup + __popc(w & ((1u << lane) - 1u));
                        if (ok && at < RF_CAP) S.sup[at] = (uint16_t)c;
                        if (lane == 0) S.words[f * 24 + (c0 >> 5)] = w;
                        nsup += __popc(w);
                        nsf[f] += __popc(w);
                    }
                }
                // ---- boundary points within r of x0, in owner order
                int nbp = 0;
                {
                    const int wx = o.hi[0][g] - o.lo[0][g] + 1, wy = o.hi[1][g] - o.lo[1][g] + 1;
                    const int span = wx * wy * (o.hi[2][g] - o.lo[2][g] + 1);
                    for (int c0 = 0; c0 < span; c0 += 32) {
                        const int c = c0 + lane;
                        int32_t b = -1;
                        if (c < span) {
                            const int cy = c / wx;
                            const int64_t w[3] = {node[0] + o.lo[0][g] + c - cy * wx, node[1] + o.lo[1][g] + cy % wy,
                                                  node[2] + o.lo[2][g] + cy / wy};
                            if (in_arr(P.g, w)) b = P.bp_index[lin_p(P.g, w)];
                        }
                        bool ok = b >= 0;
                        if (!__any_sync(0xffffffffu, ok)) continue;
                        if (ok) {
                            double d2 = 0.0;
                            for (int a = 0; a < P.g.ndim; ++a) {
                                const double dd = P.bp_xb[3 * b + a] - x0[a];
                                d2 += dd * dd;
                            }
                            ok = d2 <= r * r + 1e-9;
                        }
                        const unsigned w = __ballot_sync(0xffffffffu, ok);
                        const int at = nbp + __popc(w & ((1u << lane) - 1u));
                        if (ok && at < RF_BP) S.bps[at] = b;
                        nbp += __popc(w);
                    }
                }
                if (nsup > RF_CAP || nbp > RF_BP) {
                    redo = done = true;
                    break;
                }
                const int m = nsup + nbp * o.nbc;
                if (m < n) continue;
                __syncwarp();
                // ---- moments of the support
                for (int f = 0; f < P.nf; ++f) {
                    const int nb = o.nb[f][g];
                    const bool comp = 2 * nsf[f] > nb;
                    const int32_t* tab = o.mom + (int64_t)f * R.ncand[f] * o.gpad + lane;
                    long long acc[6] = {0, 0, 0, 0, 0, 0};
                    for (int c0 = 0; c0 < nb; c0 += 32) {
                        uint32_t w = S.words[f * 24 + (c0 >> 5)];
                        if (comp) w = ~w & (nb - c0 >= 32 ? 0xffffffffu : (1u << (nb - c0)) - 1u);
                        while (w) {
                            const int32_t* t0 = tab + (int64_t)(c0 + __ffs(w) - 1) * o.gpad;
                            w &= w - 1;
                            const int32_t* t1 = t0;
                            const bool two = w != 0;
                            if (two) {
                                t1 = tab + (int64_t)(c0 + __ffs(w) - 1) * o.gpad;
                                w &= w - 1;
                            }
#pragma unroll
                            for (int s = 0; s < 6; ++s)
                                if (32 * s < o.gpad) {
                                    const int32_t a0 = t0[32 * s], a1 = t1[32 * s];
                                    acc[s] += (long long)a0 + (two ? a1 : 0);
                                }
                        }
                    }
                    const long long* full = o.full + ((int64_t)f * RF_GROW + g) * o.gpad + lane;
#pragma unroll
                    for (int s = 0; s < 6; ++s)
                        if (32 * s < o.gpad) S.y[f * o.gpad + lane + 32 * s] = (double)(comp ? full[32 * s] - acc[s] : acc[s]);
                }
                __syncwarp();
                // ---- Gram matrix, upper triangle row by row
                for (int p = lane; p < np; p += 32) {
                    const int gm = o.pgam[p];
                    double v = gm >= 0 ? S.y[gm] * o.pcoef[p] : 0.0;
                    if (o.nconst && nbp) v = fma((double)nbp, o.pconst[p], v);
                    S.M[p] = v;
                }
                for (int b0 = 0; b0 < nbp; b0 += RF_CB) {
                    rf_chunk(P, o, S, x0, b0, nbp);
                    const int nb4 = (min(nbp - b0, RF_CB) + 1) & ~1;
#pragma unroll 1
                    for (int p = lane; p < np; p += 32) {
                        const int ij = o.pair[p];
                        const int oi2 = (ij & 0xff) * RF_PITCH, oj2 = (ij >> 8) * RF_PITCH;
                        const double* A = S.bc + T * RF_PITCH;
                        double s = S.M[p];
                        for (int q = 0; q < o.nrow; ++q) {
                            const double* base = q == o.ident ? S.bc : A;
                            if (q != o.ident) A += n * RF_PITCH;
                            for (int b = 0; b < nb4; b += 2) {
                                const double2 xi = *reinterpret_cast<const double2*>(base + oi2 + b);
                                const double2 xj = *reinterpret_cast<const double2*>(base + oj2 + b);
                                s = fma(xi.x, xj.x, s);
                                s = fma(xi.y, xj.y, s);
                            }
                        }
                        S.M[p] = s;
                    }
                    __syncwarp();
                }
                for (int p = lane; p < NMAX * NMAX; p += 32) S.GF[p] = 0.f;
                __syncwarp();
                for (int p = lane; p < np; p += 32) {
                    const int ij = o.pair[p], i = ij & 0xff, j = ij >> 8;
                    const float v = (float)S.M[p];
                    S.GF[i * NMAX + j] = v;
                    S.GF[j * NMAX + i] = v;
                }
                __syncwarp();
                // ---- U^T D U and V = U^{-1} in one sweep: after step k row k of the triangle holds
                // V's partial sums, rows above it are updated like the trailing block
                bool singular = false;
                for (int k = 0; k < n; ++k) {
                    double* Mk = S.M + rf_off(k, n);
                    const double piv = Mk[k];
                    if (!(piv > 0.0)) {
                        singular = true;
                        break;
                    }
                    const double inv = rf_rcp(piv);
                    if (lane == 0) S.dinv[k] = inv;
                    const int w = n - 1 - k;
                    for (int j = k + 1 + lane; j < n; j += 32) {
                        const double gv = Mk[j], tv = gv * inv;
                        gb[j] = gv;
                        tb[j] = tv;
                        Mk[j] = -tv;
                    }
                    __syncwarp();
                    const int kw = k * w, tot = kw + w * (w + 1) / 2;
                    const float rw = 1.f / (float)w;
                    for (int q = lane; q < tot; q += 32) {
                        int i, j;
                        double f;
                        if (q < kw) {
                            i = (int)(((float)q + 0.5f) * rw);
                            j = k + 1 + q - i * w;
                            f = S.M[rf_off(i, n) + k];
                        } else {
                            const int t = q - kw;
                            int bb = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
                            int aa = t - bb * (bb + 1) / 2;
                            if (aa < 0) {
                                aa += bb;
                                --bb;
                            } else if (aa > bb) {
                                ++bb;
                                aa -= bb;
                            }
                            i = n - 1 - bb;
                            j = n - 1 - aa;
                            f = gb[i];
                        }
                        double* e = S.M + rf_off(i, n) + j;
                        *e = fma(-f, tb[j], *e);
                    }
                    __syncwarp();
                }
                if (singular) continue;
                // ---- rank test (FP32, as k_fit): sigma_max of R from A^T A, of R^{-1} from P = (R R^T)^{-1}
                double ratio;
                {
                    float* VF = (float*)S.y;     // the moments are done with
                    float* PF = (float*)S.bc;
                    for (int p = lane; p < np; p += 32) {
                        const int ij = o.pair[p];
                        VF[p] = (ij & 0xff) == (ij >> 8) ? 1.f : (float)S.M[p];
                    }
                    for (int p = lane; p < NMAX * NMAX; p += 32) PF[p] = 0.f;
                    __syncwarp();
#pragma unroll 1
                    for (int p = lane; p < np; p += 32) {
                        const int ij = o.pair[p], i = ij & 0xff, j = ij >> 8;
                        float s = 0.f;
                        int off = 0;
                        for (int c = 0; c <= i; ++c) {
                            s = fmaf(VF[off + i], VF[off + j], s);
                            off += n - 1 - c;
                        }
                        s = s * sqrtf((float)S.dinv[i]) * sqrtf((float)S.dinv[j]);
                        PF[i * NMAX + j] = s;
                        PF[j * NMAX + i] = s;
                    }
                    __syncwarp();
                    ratio = 0.0;
                    for (int pass = 0; pass < 2; ++pass) {
                        const int iters = pass ? RANK_ITERS_FINE : 30;
                        const float smax = rf_sigma<NMAX>(S.GF, n, S.fv, iters);
                        const float sinv = rf_sigma<NMAX>(PF, n, S.fv, iters);
                        ratio = (smax > 0.f && sinv > 0.f && sinv < 3e38f) ? 1.0 / ((double)smax * (double)sinv) : 0.0;
                        if (!(ratio > P.rank_tol && ratio < RANK_RECHECK * P.rank_tol)) break;
                    }
                }
                if (!(ratio > P.rank_tol)) continue;
                // ---- u, z = (A^T A)^{-1} u
                for (int c = lane; c < n; c += 32) {
                    double s = 0.0;
                    for (unsigned e = emask; e; e &= e - 1) s += o.uE[(__ffs(e) - 1) * n + c];
                    u[c] = s;
                }
                rf_solve(S, n, u, tmp, z);
                // ---- y = A z on the interior rows; rho = u - A^T (A z)
                {
                    int i0 = 0;
                    for (int f = 0; f < P.nf; ++f) {
                        const double* ph = o.phiT + (int64_t)f * T * R.ncand[f];
                        for (int i = i0 + lane; i < i0 + nsf[f]; i += 32) {
                            const double* pc = ph + S.sup[i];
                            double s = 0.0;
                            for (int k = 0; k < T; ++k) s = fma(pc[(int64_t)k * R.ncand[f]], z[f * T + k], s);
                            S.y[i] = s;
                        }
                        i0 += nsf[f];
                    }
                }
                __syncwarp();
                double tc[2] = {0.0, 0.0};   // constant rows: their value of A z times the boundary points
                for (int q = 0; q < o.nconst; ++q) {
                    double t = 0.0;
                    for (int c = lane; c < n; c += 32) t = fma(o.crow[q * n + c], z[c], t);
#pragma unroll
                    for (int sh = 16; sh > 0; sh >>= 1) t += rf_shfl(t, sh);
                    tc[q] = (double)nbp * t;
                }
                for (int c = lane; c < n; c += 32) {
                    const int f = c / T;
                    int i0 = 0;
                    for (int ff = 0; ff < f; ++ff) i0 += nsf[ff];
                    const double* ph = o.phi + (int64_t)f * R.ncand[f] * T + (c - f * T);
                    double s = u[c];
                    for (int i = i0; i < i0 + nsf[f]; ++i) s = fma(-ph[(int)S.sup[i] * T], S.y[i], s);
                    for (int q = 0; q < o.nconst; ++q) s = fma(-tc[q], o.crow[q * n + c], s);
                    rho[c] = s;
                }
                for (int b0 = 0; b0 < nbp; b0 += RF_CB) {
                    rf_chunk(P, o, S, x0, b0, nbp);
                    const int b = lane % RF_CB, h = lane / RF_CB;
                    const double* A = S.bc + T * RF_PITCH;
                    for (int q = 0; q < o.nrow; ++q) {
                        const double* base = q == o.ident ? S.bc : A;
                        if (q != o.ident) A += n * RF_PITCH;
                        double s = 0.0;
                        for (int c = h; c < n; c += RF_NG) s = fma(base[c * RF_PITCH + b], z[c], s);
#pragma unroll
                        for (int sh = 16; sh >= RF_CB; sh >>= 1) s += rf_shfl(s, sh);
                        if (h == 0) S.sb[q * RF_CB + b] = s;
                    }
                    __syncwarp();
                    const int cnt = min(nbp - b0, RF_CB);
                    for (int c = lane; c < n; c += 32) {
                        A = S.bc + T * RF_PITCH;
                        double s = rho[c];
                        for (int q = 0; q < o.nrow; ++q) {
                            const double* base = q == o.ident ? S.bc : A;
                            if (q != o.ident) A += n * RF_PITCH;
                            for (int i = 0; i < cnt; ++i) s = fma(-base[c * RF_PITCH + i], S.sb[q * RF_CB + i], s);
                        }
                        rho[c] = s;
                    }
                    __syncwarp();
                }
                rf_solve(S, n, rho, tmp, gb);
                // ---- output: y + A (A^T A)^{-1} rho
                unsigned long long st = 0;
                if (lane == 0) st = atomicAdd(P.pool_top, (unsigned long long)nsup);
                const int64_t start = (int64_t)__shfl_sync(0xffffffffu, st, 0);
                if (start + nsup > P.pool_cap) {
                    status = 3;   // pool overflow: re-run with a larger pool
                    done = true;
                    break;
                }
                {
                    int i0 = 0;
                    for (int f = 0; f < P.nf; ++f) {
                        const double* ph = o.phiT + (int64_t)f * T * R.ncand[f];
                        for (int i = i0 + lane; i < i0 + nsf[f]; i += 32) {
                            const int c = S.sup[i];
                            double s = S.y[i];
                            for (int k = 0; k < T; ++k) s = fma(ph[(int64_t)k * R.ncand[f] + c], gb[f * T + k], s);
                            const int8_t* bo = P.ball_off[f] + 3 * c;
                            P.pool_code[start + i] = pack_off(bo[0], bo[1], bo[2]);
                            P.pool_field[start + i] = (int8_t)f;
                            P.pool_w[start + i] = s;
                        }
                        i0 += nsf[f];
                    }
                }
                if (lane == 0) P.start[row] = start;
                status = 0;
                used_order = o.order;
                used_r2 = (int)lrint(2.0 * r);
                used_nbp = nbp;
                nsup_final = nsup;
                done = true;
            }
        }
        if (lane == 0) {
            if (redo) {
                R.redo[atomicAdd(R.nredo, 1u)] = (int32_t)row;
            } else {
                P.info[4 * row + 0] = used_r2;
                P.info[4 * row + 1] = used_order;
                P.info[4 * row + 2] = used_nbp;
                P.info[4 * row + 3] = status;
                P.cnt[row] = status == 0 ? nsup_final : 0;
            }
        }
        __syncwarp();
    }
}
