// TensorNet energy and forces (Sec. 2.1.1; Sec. 2 Fig. 1): forward pass and a
// hand-written reverse pass for the forces, on the compact I/A/S coordinates
// of internal.cuh.  FP32 arithmetic, FP64 per-system energy reduction.
//
// Pass structure (one call of tnet_energy_forces):
//   graph prep   reverse-edge index; undirected active-edge list (i < j,
//                d < cutoff) so the radial MLP runs once per pair (its output
//                depends only on d, hence g_ij = g_ji)
//   embedding    edge kernel (pair embedding x radial projections x edge
//                basis, segmented over CSR rows) -> per-atom norm/LayerNorm,
//                scalar MLP and channel mixing
//   L layers     normalise, mix, radial MLP per pair, message gather, tensor
//                products Y M + M Y, normalise, mix, residual X + dX + dX^2
//   output       I/A/S norms, LayerNorm, MLP head, FP64 sum per system
//   reverse      the adjoint of every step in reverse order, ending in one
//                3-vector dE/dr_ij per directed edge; forces are assembled
//                per atom from its row and the reverse edges (no atomics).
#include <type_traits>

#include "gemm.cuh"
#include "internal.cuh"
#include "tc_gemm.cuh"

namespace tnet {

constexpr int kMU = 4;  // edges whose loads are in flight together in the row kernels
constexpr int kChunk = 128;  // row edges whose indices are staged in shared memory at a time

// ----------------------------------------------------------- weights ---
struct LayerW {
    const float *mlp1_w, *mlp1_b, *mlp2_w, *mlp2_b, *mlp3_w, *mlp3_b, *mix1_w, *mix2_w;
};
struct Weights {
    const float *emb, *emb2_w, *emb2_b, *dproj_w, *dproj_b, *emb_ln_g, *emb_ln_b, *emb_mlp1_w,
        *emb_mlp1_b, *emb_mlp2_w, *emb_mlp2_b, *emb_mix_w;
    LayerW layer[8];
    const float *out_ln_g, *out_ln_b, *out_w, *out_b, *head1_w, *head1_b, *head2_w, *head2_b;
};

// Offsets of the blob layout documented in tnet.h.  Returns the total.
int64_t weight_offsets(const tnet_model_desc *d, const float *base, Weights *w) {
    const int64_t F = d->F, K = d->K, Z = d->max_z;
    int64_t o = 0;
    auto take = [&](int64_t n) { const float *p = base ? base + o : nullptr; o += n; return p; };
    Weights t{};
    t.emb = take(Z * F);
    t.emb2_w = take(F * 2 * F); t.emb2_b = take(F);
    t.dproj_w = take(3 * F * K); t.dproj_b = take(3 * F);
    t.emb_ln_g = take(F); t.emb_ln_b = take(F);
    t.emb_mlp1_w = take(2 * F * F); t.emb_mlp1_b = take(2 * F);
    t.emb_mlp2_w = take(3 * F * 2 * F); t.emb_mlp2_b = take(3 * F);
    t.emb_mix_w = take(3 * F * F);
    for (int l = 0; l < d->L; ++l) {
        LayerW &L = t.layer[l];
        L.mlp1_w = take(F * K); L.mlp1_b = take(F);
        L.mlp2_w = take(2 * F * F); L.mlp2_b = take(2 * F);
        L.mlp3_w = take(3 * F * 2 * F); L.mlp3_b = take(3 * F);
        L.mix1_w = take(3 * F * F);
        L.mix2_w = take(3 * F * F);
    }
    t.out_ln_g = take(3 * F); t.out_ln_b = take(3 * F);
    t.out_w = take(F * 3 * F); t.out_b = take(F);
    t.head1_w = take(F / 2 * F); t.head1_b = take(F / 2);
    t.head2_w = take(F / 2); t.head2_b = take(1);
    if (w) *w = t;
    return o;
}

// --------------------------------------------------------- utilities ---
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// sum over the block (blockDim.x a multiple of 32, <= 1024); all threads get it
__device__ __forceinline__ float block_sum(float v, float *sm) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) sm[wid] = v;
    __syncthreads();
    float t = 0.f;
    for (int k = 0; k < nw; ++k) t += sm[k];
    return t;
}

// pair vector r_ij = mic(r_i - r_j) for rectangular or triclinic
// (lower-triangular) boxes, with fixed rounding (see mic_lower)
__device__ __forceinline__ void pair_vec(const float *__restrict__ pos, const float *__restrict__ box,
                                         const int32_t *__restrict__ batch, int i, int j, float &x,
                                         float &y, float &zz) {
    x = __fsub_rn(pos[3LL * i], pos[3LL * j]);
    y = __fsub_rn(pos[3LL * i + 1], pos[3LL * j + 1]);
    zz = __fsub_rn(pos[3LL * i + 2], pos[3LL * j + 2]);
    if (box) mic_box(x, y, zz, box + 9LL * (batch ? batch[i] : 0));
}

// ------------------------------------------------------- graph prep ---
// Row offsets are read clamped to [0, cap] (cap = the context's pair capacity,
// which sizes every per-edge buffer), so a caller's CSR never sends a kernel
// outside those buffers.
__device__ __forceinline__ int32_t row_offset(const int32_t *__restrict__ row_ptr, int64_t t, int64_t cap) {
    const int32_t v = row_ptr[t];
    return v < 0 ? 0 : (v > cap ? (int32_t)cap : v);
}

// One warp per row: the clamped copy of the row offsets that every later
// kernel reads (offsets out of range or decreasing are reported as ARG, or
// CAPACITY when they pass the capacity), the system bounds, the reverse edges
// rev[e] = position of (j, i) in row j (e itself: none, reported as ARG), and
// the count of the row's upper (j > i) edges with d < rc that have a reverse:
// those become pairs, so a list that lacks half of its edges (a half list, a
// truncated one) never has more pairs than half of its edges, which is what
// the pair buffers hold.  Every edge starts inactive.  Decreasing offsets make
// rows overlap, and rows that share edges would write each other's rev and be
// walked once per row; a row of more than N edges repeats columns: either
// raises rows_bad (reported as ARG), and the list is then taken as empty.  One
// launch in the place of four (launches and their gaps were most of the time of
// small systems' graph preparation).
__global__ void k_graph_rows(const float *__restrict__ pos, const float *__restrict__ box,
                             const int32_t *__restrict__ batch, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, int N, int S, int64_t cap, float rc,
                             int32_t *__restrict__ safe, int32_t *__restrict__ sys_start,
                             int32_t *__restrict__ sys_end, int32_t *__restrict__ rows_bad,
                             int32_t *__restrict__ rev, int32_t *__restrict__ pair_of, int32_t *__restrict__ ucnt,
                             int32_t *status) {
    pdl_entry();
    const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (i >= N) return;
    const int lane = threadIdx.x & 31;
    const int e0 = row_offset(row_ptr, i, cap), e1 = row_offset(row_ptr, (int64_t)i + 1, cap);
    if (lane == 0) {
        mark_bounds(batch, i, N, S, sys_start, sys_end, status);
        const int32_t v0 = row_ptr[i], v1 = row_ptr[i + 1];
        if (v0 < 0 || (i == 0 && v0 != 0) || v1 < 0 || v0 > v1) set_status(status, TNET_ERR_ARG);
        if (v0 > cap || v1 > cap) set_status(status, TNET_ERR_CAPACITY);
        if (e0 > e1 || e1 - e0 > N) {
            set_status(status, TNET_ERR_ARG);
            *rows_bad = 1;
        }
        safe[i] = e0;
        if (i == N - 1) safe[N] = e1;
    }
    if (e1 - e0 > N) return;  // (see rows_bad)
    int cnt = 0;
    for (int eb = e0; eb < e1; eb += 32) {
        const int e = eb + lane;
        bool up = false;
        if (e < e1) {
            const int j = col[e];
            int r = e;  // e itself: no reverse edge
            if (j < 0 || j >= N || (e > e0 && col[e - 1] >= j)) {  // rows must ascend strictly
                set_status(status, TNET_ERR_ARG);
            } else {
                int lo = row_offset(row_ptr, j, cap);
                const int end = row_offset(row_ptr, (int64_t)j + 1, cap);
                int hi = end;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (col[mid] < i) lo = mid + 1;
                    else hi = mid;
                }
                if (lo < end && col[lo] == i) r = lo;
                else set_status(status, TNET_ERR_ARG);  // pair list not symmetric
            }
            rev[e] = r;
            pair_of[e] = -1;
            if (r != e && j > i) {
                float x, y, zz;
                pair_vec(pos, box, batch, i, j, x, y, zz);
                up = sqrtf(norm2_rn(x, y, zz)) < rc;
            }
        }
        cnt += __popc(__ballot_sync(0xffffffffu, up));
    }
    if (lane == 0) ucnt[i] = cnt;
}

// Numbers the active undirected pairs by their upper edges and tells both
// directed edges (an edge without a reverse stays inactive).  Columns that
// ascend strictly give at most E / 2 pairs; repeated columns (reported) can
// give more, and those past maxU, the size of the pair buffers, stay inactive.
// nu, the scan's total, is brought in line: the kernels after this one take
// their pairs from it.  rows_bad: no pairs, and every row empty.
__global__ void k_upper_assign(const float *__restrict__ pos, const float *__restrict__ box,
                               const int32_t *__restrict__ batch, int32_t *__restrict__ row_ptr,
                               const int32_t *__restrict__ col, const int32_t *__restrict__ rev, int N, float rc,
                               const int32_t *__restrict__ uoff, const int32_t *__restrict__ rows_bad, int maxU,
                               int32_t *__restrict__ nu, int32_t *__restrict__ pair_of, int2 *__restrict__ uij,
                               int32_t *__restrict__ ue) {
    pdl_entry();
    const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (i >= N) return;
    const int lane = threadIdx.x & 31;
    // one round of loads: the flag does not hold up what follows
    const bool bad = *rows_bad != 0;
    const int total = *nu, r0 = row_ptr[i], r1 = row_ptr[i + 1];
    int base = uoff[i];
    if (i == 0 && lane == 0 && (bad || total > maxU)) *nu = bad ? 0 : maxU;
    if (bad) {
        if (lane == 0) {
            row_ptr[i] = 0;
            if (i == N - 1) row_ptr[N] = 0;
        }
        return;
    }
    for (int e0 = r0; e0 < r1; e0 += 32) {
        const int e = e0 + lane;
        bool up = false;
        int j = -1, r = -1;
        if (e < r1) {
            j = col[e];
            r = rev[e];
            if (r != e && j > i) {
                float x, y, zz;
                pair_vec(pos, box, batch, i, j, x, y, zz);
                up = sqrtf(norm2_rn(x, y, zz)) < rc;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, up);
        const int u = base + __popc(m & ((1u << lane) - 1u));
        if (up && u < maxU) {
            pair_of[e] = u;
            uij[u] = make_int2(i, j);
            ue[u] = e;
            pair_of[r] = u;
        }
        base += __popc(m);
    }
}

// Radial basis and cutoff of each undirected active edge, and its geometry
// (unit vector u_ij for i < j, and phi) for the embedding kernels.
__global__ void k_edge_rbf(const float *__restrict__ pos, const float *__restrict__ box,
                           const int32_t *__restrict__ batch, const int2 *__restrict__ uij,
                           const int32_t *__restrict__ nu, int maxU, RadialParams rp,
                           float *__restrict__ eu, float *__restrict__ phiu, float4 *__restrict__ geo,
                           OpCopy eu_cp) {
    pdl_entry();
    // a block takes groups of P = blockDim.x (<= 256) pairs: one thread per
    // pair computes its geometry, then all threads evaluate the P x K basis
    // values from it (coalesced writes of eu)
    __shared__ float s_ex[256], s_phi[256];
    const int U = *nu, K = rp.K;
    const int P = blockDim.x < 256 ? blockDim.x : 256;
    for (int64_t u0 = (int64_t)blockIdx.x * P; u0 < U; u0 += (int64_t)gridDim.x * P) {
        const int np = U - u0 < P ? (int)(U - u0) : P;
        if (threadIdx.x < np) {
            const int u = (int)u0 + threadIdx.x;
            const int2 p = uij[u];
            float x, y, zz;
            pair_vec(pos, box, batch, p.x, p.y, x, y, zz);
            const float d = sqrtf(norm2_rn(x, y, zz));
            const float phi = cutoff_phi(d, rp);
            s_ex[threadIdx.x] = expf(rp.alpha * (rp.rl - d));
            s_phi[threadIdx.x] = phi;
            phiu[u] = phi;
            const float inv = 1.0f / d;
            geo[u] = make_float4(x * inv, y * inv, zz * inv, phi);  // u_ij for i < j, and phi
        }
        __syncthreads();
        for (int idx = threadIdx.x; idx < np * K; idx += blockDim.x) {
            const int q = idx / K, k = idx % K;
            const float e = expnorm_value(s_ex[q], k, rp, s_phi[q]);
            const int64_t t = (u0 + q) * K + k;
            eu[t] = e;
            opcopy_store(eu_cp, t, e);
        }
        __syncthreads();
    }
}

// ------------------------------------------------ tabulated radial functions ---
// The radial projections f(d) and every layer's filter g(d) depend on the pair
// distance alone.  In table mode they are evaluated in FP64, with their
// d-derivatives (forward mode through the same layers), at the grid d_k = k h
// (k < n, h = rc/(n - 1)).  Each interval [d_k, d_k+1] stores the cubic
// Hermite polynomial p(s) = c0 + c1 s + c2 s^2 + c3 s^3, s = (d - d_k)/h, whose
// coefficients are formed in FP64 before rounding to FP32: the derivative
// p'(s)/h then carries no cancellation between neighbouring table values, and
// the forces are the derivatives of the interpolated energy.

struct RadialParams64 {
    double rc, rl, alpha, beta, mu0, dmu;
    int K;
};

__device__ __forceinline__ void silu64(double a, double &v, double &g) {
    const double sg = 1.0 / (1.0 + exp(-a));
    v = a * sg;
    g = sg * (1.0 + a * (1.0 - sg));
}

// basis e_q(d_k) (the cosine cutoff included), de_q/dd, phi(d_k), dphi/dd
__global__ void k_tab_rbf(int n, double h, RadialParams64 rp, double *__restrict__ e, double *__restrict__ de,
                          double *__restrict__ phi, double *__restrict__ dphi) {
    pdl_entry();
    const int K = rp.K;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)n * K;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(t / K), q = (int)(t % K);
        const double d = k * h;
        const double ph = d < rp.rc ? 0.5 * (cospi(d / rp.rc) + 1.0) : 0.0;
        const double dph = d < rp.rc ? -0.5 * 3.141592653589793 / rp.rc * sinpi(d / rp.rc) : 0.0;
        const double ex = exp(rp.alpha * (rp.rl - d));
        const double u = ex - (rp.mu0 + q * rp.dmu);
        const double rho = exp(-rp.beta * u * u);
        e[t] = ph * rho;
        de[t] = dph * rho + ph * rho * (2.0 * rp.beta * u * rp.alpha * ex);
        if (q == 0) {
            phi[k] = ph;
            dphi[k] = dph;
        }
    }
}

// One dense layer of the radial chain at the grid points, FP64, with its
// tangent: a = x W^T + b, ta = tx W^T, and
//   mode 0 (hidden layers): y = silu(a),       ty = silu'(a) ta
//   mode 1 (projections f): y = a,             ty = ta
//   mode 2 (filters g):     y = phi silu(a),   ty = dphi silu(a) + phi silu'(a) ta
// 64 x 64 output tiles, 256 threads with 4 x 4 outputs (and tangents) each.
__global__ void __launch_bounds__(256)
    k_tab_layer(int n, int Nout, int Kin, const double *__restrict__ x, const double *__restrict__ tx,
                const float *__restrict__ Wt, const float *__restrict__ b, int mode, const double *__restrict__ phi,
                const double *__restrict__ dphi, double *__restrict__ y, double *__restrict__ ty) {
    pdl_entry();
    constexpr int T = 64, BK = 16;
    __shared__ double xs[BK][T], ts[BK][T], ws[BK][T];
    const int tid = threadIdx.x, tr = tid / 16, tc = tid % 16;
    const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
    double acc[4][4], tac[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = tac[i][j] = 0.0;
    for (int k0 = 0; k0 < Kin; k0 += BK) {
        for (int i = tid; i < BK * T; i += blockDim.x) {
            const int r = i / BK, kk = i % BK, gk = k0 + kk;
            const int gm = m0 + r, gn = n0 + r;
            const bool okx = gm < n && gk < Kin, okw = gn < Nout && gk < Kin;
            xs[kk][r] = okx ? x[(int64_t)gm * Kin + gk] : 0.0;
            ts[kk][r] = okx ? tx[(int64_t)gm * Kin + gk] : 0.0;
            ws[kk][r] = okw ? (double)Wt[(int64_t)gn * Kin + gk] : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            double xv[4], tv[4], wv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                xv[i] = xs[kk][tr * 4 + i];
                tv[i] = ts[kk][tr * 4 + i];
                wv[i] = ws[kk][tc * 4 + i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fma(xv[i], wv[j], acc[i][j]);
                    tac[i][j] = fma(tv[i], wv[j], tac[i][j]);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + tr * 4 + i;
        if (gm >= n) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + tc * 4 + j;
            if (gn >= Nout) continue;
            const double a = acc[i][j] + (double)b[gn], ta = tac[i][j];
            double v, g, out, tout;
            if (mode == 1) {
                out = a;
                tout = ta;
            } else {
                silu64(a, v, g);
                if (mode == 0) {
                    out = v;
                    tout = g * ta;
                } else {
                    out = phi[gm] * v;
                    tout = dphi[gm] * v + phi[gm] * g * ta;
                }
            }
            y[(int64_t)gm * Nout + gn] = out;
            ty[(int64_t)gm * Nout + gn] = tout;
        }
    }
}

// Hermite coefficients of each interval, [n-1][W] float4 (c0, c1, c2, c3):
//   c0 = v0, c1 = h v0', c2 = 3 (v1 - v0) - 2 h v0' - h v1', c3 = 2 (v0 - v1) + h v0' + h v1'
__global__ void k_tab_coef(int n, int W, double h, const double *__restrict__ v, const double *__restrict__ dv,
                           float4 *__restrict__ coef) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)(n - 1) * W;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / W;
        const int w = (int)(t % W);
        const double v0 = v[k * W + w], v1 = v[(k + 1) * W + w];
        const double d0 = h * dv[k * W + w], d1 = h * dv[(k + 1) * W + w];
        coef[k * W + w] = make_float4((float)v0, (float)d0, (float)(3.0 * (v1 - v0) - 2.0 * d0 - d1),
                                      (float)(2.0 * (v0 - v1) + d0 + d1));
    }
}

// A table-mode view of one radial function: the consumers (embedding,
// messages and their adjoints) evaluate p(s) and p'(s)/h of the pair's
// interval themselves, reading one float4 per channel (L2-resident tables).
struct TabFn {
    const float4 *coef;  // [n-1][3F]
    const float *dist;   // [U] pair distances
    int n;
    float inv_h;
};
__device__ __forceinline__ void tab_locate(const TabFn &T, int u, int &k, float &s) {
    const float x = T.dist[u] * T.inv_h;
    int kk = (int)floorf(x);
    kk = kk < 0 ? 0 : (kk > T.n - 2 ? T.n - 2 : kk);
    k = kk;
    s = x - (float)kk;
}
__device__ __forceinline__ float tab_value(const float4 &c, float s) {
    return fmaf(s, fmaf(s, fmaf(s, c.w, c.z), c.y), c.x);
}
__device__ __forceinline__ float tab_slope(const float4 &c, float s, float inv_h) {
    return fmaf(s, fmaf(s, 3.f * c.w, 2.f * c.z), c.y) * inv_h;
}

// per undirected pair: u_ij, phi (geo), phi alone (phiu) and d (dist)
__global__ void k_pair_geo(const float *__restrict__ pos, const float *__restrict__ box,
                           const int32_t *__restrict__ batch, const int2 *__restrict__ uij,
                           const int32_t *__restrict__ nu, RadialParams rp, float *__restrict__ phiu,
                           float4 *__restrict__ geo, float *__restrict__ dist) {
    pdl_entry();
    const int U = *nu;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < U; u += gridDim.x * blockDim.x) {
        const int2 p = uij[u];
        float x, y, zz;
        pair_vec(pos, box, batch, p.x, p.y, x, y, zz);
        const float d = sqrtf(norm2_rn(x, y, zz));
        const float phi = cutoff_phi(d, rp);
        const float inv = 1.0f / d;
        phiu[u] = phi;
        dist[u] = d;
        geo[u] = make_float4(x * inv, y * inv, zz * inv, phi);
    }
}

// Per-element pair-embedding tables: Ta[z] = W_e[:, :F] emb[z],
// Tb[z] = W_e[:, F:] emb[z] + b_e, so that Z_ij = Ta[z_i] + Tb[z_j].  One warp
// per output row of W (lanes along the row, so the reads of W are coalesced),
// a fixed-order warp reduction; part of `parts` of element z's rows.
__device__ __forceinline__ void elem_tables(int z, int part, int parts, const float *__restrict__ emb,
                                            const float *__restrict__ W, const float *__restrict__ b, int F,
                                            float *__restrict__ Ta, float *__restrict__ Tb) {
    const int lane = threadIdx.x & 31, nw = (blockDim.x >> 5) * parts;
    const float *e = emb + (int64_t)z * F;
#pragma unroll 4
    for (int r = part * (blockDim.x >> 5) + (threadIdx.x >> 5); r < 2 * F; r += nw) {  // rows c (Ta) and F + c (Tb)
        const int c = r % F, half = r / F;
        const float *w = W + (int64_t)c * 2 * F + half * F;
        float s = 0.f;
        for (int k = lane; k < F; k += 32) s = fmaf(w[k], e[k], s);
        s = warp_sum(s);
        if (lane == 0) {
            if (half == 0) Ta[(int64_t)z * F + c] = s;
            else Tb[(int64_t)z * F + c] = s + b[c];
        }
    }
}

// ------------------------------------------------------- embedding ---

struct EdgeGeo {
    int j, active;
    float d, u[3], phi, dphi;
};

__device__ __forceinline__ EdgeGeo edge_geo(const float *__restrict__ pos, const float *__restrict__ box,
                                            const int32_t *__restrict__ batch, int i, int j,
                                            const RadialParams &rp) {
    EdgeGeo g;
    g.j = j;
    float x, y, zz;
    pair_vec(pos, box, batch, i, j, x, y, zz);
    g.d = sqrtf(norm2_rn(x, y, zz));
    g.active = (g.d < rp.rc) && (g.d > 0.f);
    const float inv = g.d > 0.f ? 1.0f / g.d : 0.f;
    g.u[0] = x * inv; g.u[1] = y * inv; g.u[2] = zz * inv;
    g.phi = g.active ? cutoff_phi(g.d, rp) : 0.f;
    g.dphi = g.active ? cutoff_dphi(g.d, rp) : 0.f;
    return g;
}

// X_raw_i = sum_j phi Z_ij (f^I I0 + f^A A0(u) + f^S S0(u)) over the active
// edges of row i, in row order.  f^p = W^p e(d) + b^p depends only on d, so
// it is computed once per undirected pair by a GEMM (fu, columns p*F + c),
// or, with TAB, evaluated here from the Hermite table; u and phi come once
// per pair from geo (k_edge_rbf or k_pair_geo).
// Block = F threads (thread = channel), persistent over atoms; loads for kMU
// edges are in flight together.
template <int F, bool TAB>
__global__ void __launch_bounds__(F) k_emb_edges(const float4 *__restrict__ geo, const int32_t *__restrict__ z,
                                                 const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                                 const int32_t *__restrict__ pair_of, int N, int max_z,
                                                 const float *__restrict__ fu, TabFn tf, const float *__restrict__ Ta,
                                                 const float *__restrict__ Tb, float *__restrict__ Xraw,
                                                 const float *__restrict__ ln_g, const float *__restrict__ ln_b,
                                                 float *__restrict__ n0, float2 *__restrict__ ln,
                                                 float *__restrict__ q0, int32_t *status, OpCopy Xraw_cp) {
    pdl_entry();
    __shared__ int32_t s_u[kChunk], s_zs[kChunk];  // pair index; element of the column atom, signed by direction
    __shared__ int32_t s_kt[TAB ? kChunk : 1];      // table mode: interval and offset of the pair distance
    __shared__ float s_st[TAB ? kChunk : 1];
    __shared__ float s_red[32];
    const int c = threadIdx.x;
    for (int i = blockIdx.x; i < N; i += gridDim.x) {
        int zi = z[i];
        if (zi < 0 || zi >= max_z) {
            set_status(status, TNET_ERR_Z);
            zi = 0;
        }
        const float ta = Ta[(int64_t)zi * F + c];
        float v[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const int e0 = row_ptr[i], e1 = row_ptr[i + 1];
        for (int cb = e0; cb < e1; cb += kChunk) {
            const int n = e1 - cb < kChunk ? e1 - cb : kChunk;
            __syncthreads();
            for (int t = c; t < n; t += F) {
                const int u = pair_of[cb + t];
                s_u[t] = u;
                int zj = 0, j = i;
                if (u >= 0) {
                    j = col[cb + t];
                    zj = z[j];
                    zj = (zj < 0 || zj >= max_z) ? 0 : zj;
                }
                s_zs[t] = j > i ? zj : -1 - zj;   // u_ij = +u of the pair when i is its first atom
                if constexpr (TAB) {
                    int kt = 0;
                    float st = 0.f;
                    if (u >= 0) tab_locate(tf, u, kt, st);
                    s_kt[t] = kt;
                    s_st[t] = st;
                }
            }
            __syncthreads();
            for (int k0 = 0; k0 < n; k0 += kMU) {
                int uu[kMU], zz[kMU];
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    uu[k] = k0 + k < n ? s_u[k0 + k] : -1;
                    zz[k] = k0 + k < n ? s_zs[k0 + k] : 0;
                }
                float f[kMU][3], tb[kMU];
                float4 gk[kMU];
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    if (uu[k] < 0) continue;
                    if constexpr (TAB) {
                        const float4 *cp = tf.coef + (int64_t)s_kt[k0 + k] * 3 * F + c;
                        const float st = s_st[k0 + k];
                        f[k][0] = tab_value(cp[0], st); f[k][1] = tab_value(cp[F], st); f[k][2] = tab_value(cp[2 * F], st);
                    } else {
                        const float *fp = fu + (int64_t)uu[k] * 3 * F + c;
                        f[k][0] = fp[0]; f[k][1] = fp[F]; f[k][2] = fp[2 * F];
                    }
                    tb[k] = Tb[(int64_t)(zz[k] >= 0 ? zz[k] : -1 - zz[k]) * F + c];
                    gk[k] = geo[uu[k]];
                }
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    if (uu[k] < 0) continue;
                    const float sg = zz[k] >= 0 ? 1.0f : -1.0f;
                    const float ux = sg * gk[k].x, uy = sg * gk[k].y, uz = sg * gk[k].z;
                    const float pz = gk[k].w * (ta + tb[k]);
                    const float cI = pz * f[k][0], cA = pz * f[k][1], cS = pz * f[k][2];
                    v[0] += cI;
                    v[1] += cA * ux; v[2] += cA * uy; v[3] += cA * uz;
                    v[4] += cS * (ux * ux - (1.0f / 3.0f));
                    v[5] += cS * (uy * uy - (1.0f / 3.0f));
                    v[6] += cS * ux * uy; v[7] += cS * ux * uz; v[8] += cS * uy * uz;
                }
            }
        }
        store_coords(Xraw, i, c, N, F, v);
        store_coords_cp(Xraw_cp, i, c, N, F, v);
        // q0 = ||X_raw|| per channel, LayerNorm over channels -> n0 (the block
        // holds the atom's channels); caches (mean, rstd)
        const float q = cnorm(v);
        const float mean = block_sum(q, s_red) / F;
        const float dv = q - mean;
        const float var = block_sum(dv * dv, s_red) / F;
        const float rstd = rsqrtf(var + 1e-5f);
        n0[(int64_t)i * F + c] = dv * rstd * ln_g[c] + ln_b[c];
        q0[(int64_t)i * F + c] = q;
        if (c == 0) ln[i] = make_float2(mean, rstd);
    }
}

// The layer input's normalisation Xn = X / (||X|| + 1), from registers: X itself
// is not stored (the adjoint forms it again).
__device__ __forceinline__ void store_normed(float v[9], int64_t t, int i, int c, int N, int F, float *__restrict__ qn,
                                             float *__restrict__ Xn, const OpCopy &Xn_cp) {
    const float q = cnorm(v);
    qn[t] = q;
    const float r = 1.0f / (q + 1.0f);
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] *= r;
    store_coords(Xn, i, c, N, F, v);
    store_coords_cp(Xn_cp, i, c, N, F, v);
}

// X0 = s_p * U (p = class of the coordinate), s channel-major [N][F][3], and
// the first layer's normalisation of it; without layers (qn NULL) X0 itself is
// stored.  The elementwise kernels are bound by HBM: fused with their neighbour
// where one's output is the other's input, they read and write 5 of the 8
// node tensors they did (96,000 atoms: the call 38.1 -> 37.7 ms).
__global__ void k_emb_scale(const float *__restrict__ U, const float *__restrict__ s, int N, int F,
                            float *__restrict__ X0, float *__restrict__ qn, float *__restrict__ Xn, OpCopy Xn_cp) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * F;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / F), c = (int)(t % F);
        float v[9];
        load_coords(U, i, c, N, F, v);
        const float *si = s + ((int64_t)i * F + c) * 3;
        v[0] = __fmul_rn(v[0], si[0]);
#pragma unroll
        for (int k = 1; k < 4; ++k) v[k] = __fmul_rn(v[k], si[1]);
#pragma unroll
        for (int k = 4; k < 9; ++k) v[k] = __fmul_rn(v[k], si[2]);
        if (qn) store_normed(v, t, i, c, N, F, qn, Xn, Xn_cp);
        else store_coords(X0, i, c, N, F, v);
    }
}

// ----------------------------------------------------- interaction ---
// M_i = sum_j g^p_ij Y^p_j over the row (block = F threads, thread = channel).
// The filter is never stored: g = phi(d) SiLU(a3) is formed here from the last
// radial layer's pre-activation a3 of pair u, stored plane-major, a3[u][p][c],
// so each of its three loads is one coalesced F-channel row, and phi of the
// pair (the same expression as the GEMM epilogue would evaluate).  The row's pair and column indices are staged in
// shared memory (one coalesced load per chunk of kChunk edges), so each group of
// kMU edges waits for one round of gathers, not for its indices first; the
// sums still run in row order.  F is a template parameter so the coordinate
// offsets are immediates.
//
// RB consecutive rows per block, one group of F threads per row (named
// barrier 1 + group): consecutive atoms share most of their neighbours (the
// three atoms of a water, the next molecule of the lattice), so the groups of
// a block gather mostly the same rows of Y at about the same time (columns
// ascend in every row) and the repeats hit the SM's L1 instead of L2.
template <int F, bool TAB, int RB>
__global__ void __launch_bounds__(F * RB, (768 / (F * RB)) > 0 ? 768 / (F * RB) : 1)
    k_message(const int32_t *__restrict__ row_ptr,
                                                    const int32_t *__restrict__ col,
                                                    const int32_t *__restrict__ pair_of, const float *__restrict__ a3,
                                                    const float *__restrict__ phiu, TabFn tg,
                                                    const float *__restrict__ Y, int N, float *__restrict__ M) {
    pdl_entry();
    __shared__ int32_t s_u_all[RB][kChunk], s_j_all[RB][kChunk];
    __shared__ int32_t s_kt_all[RB][TAB ? kChunk : 1];
    __shared__ float s_st_all[RB][TAB ? kChunk : 1];
    const int grp = RB > 1 ? (int)threadIdx.x / F : 0, c = RB > 1 ? (int)threadIdx.x % F : (int)threadIdx.x;
    int32_t *s_u = s_u_all[grp], *s_j = s_j_all[grp], *s_kt = s_kt_all[grp];
    float *s_st = s_st_all[grp];
    for (int i = blockIdx.x * RB + grp; i < N; i += gridDim.x * RB) {
        float m[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const int e0 = row_ptr[i], e1 = row_ptr[i + 1];
        for (int cb = e0; cb < e1; cb += kChunk) {
            const int n = e1 - cb < kChunk ? e1 - cb : kChunk;
            group_sync<F, RB>(grp);  // the previous chunk is consumed
            for (int t = c; t < n; t += F) {
                const int u = pair_of[cb + t];
                s_u[t] = u;
                s_j[t] = col[cb + t];
                if constexpr (TAB) {
                    int kt = 0;
                    float st = 0.f;
                    if (u >= 0) tab_locate(tg, u, kt, st);
                    s_kt[t] = kt;
                    s_st[t] = st;
                }
            }
            group_sync<F, RB>(grp);
            for (int k0 = 0; k0 < n; k0 += kMU) {
                int uu[kMU], jj[kMU];
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    uu[k] = k0 + k < n ? s_u[k0 + k] : -1;
                    jj[k] = k0 + k < n ? s_j[k0 + k] : 0;
                }
                float g[kMU][3], y[kMU][9], ph[kMU];
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    if (uu[k] < 0) continue;
                    if constexpr (TAB) {
                        const float4 *cp = tg.coef + (int64_t)s_kt[k0 + k] * 3 * F + c;
                        const float st = s_st[k0 + k];
                        g[k][0] = tab_value(cp[0], st); g[k][1] = tab_value(cp[F], st); g[k][2] = tab_value(cp[2 * F], st);
                    } else {
                        const float *ap = a3 + (int64_t)uu[k] * 3 * F + c;
                        g[k][0] = ap[0]; g[k][1] = ap[F]; g[k][2] = ap[2 * F];
                        ph[k] = phiu[uu[k]];
                    }
                    load_coords(Y, jj[k], c, N, F, y[k]);
                }
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    if (uu[k] < 0) continue;
                    if constexpr (!TAB) {
#pragma unroll
                        for (int p = 0; p < 3; ++p) g[k][p] = silu_f(g[k][p]) * ph[k];
                    }
                    m[0] = fmaf(g[k][0], y[k][0], m[0]);
#pragma unroll
                    for (int q = 1; q < 4; ++q) m[q] = fmaf(g[k][1], y[k][q], m[q]);
#pragma unroll
                    for (int q = 4; q < 9; ++q) m[q] = fmaf(g[k][2], y[k][q], m[q]);
                }
            }
        }
        store_coords(M, i, c, N, F, m);
    }
}

// T = Y M + M Y; Tn = decomp(T) / (||T|| + 1)
__global__ void k_node_update(const float *__restrict__ Y, const float *__restrict__ M, int N, int F,
                              float *__restrict__ Tn, OpCopy Tn_cp) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * F;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / F), c = (int)(t % F);
        float yv[9], mv[9], Yf[9], Mf[9], A[9], B[9], T[9], tc[9];
        load_coords(Y, i, c, N, F, yv);
        load_coords(M, i, c, N, F, mv);
        expand(yv, Yf);
        expand(mv, Mf);
        mm3(Yf, Mf, A);
        mm3(Mf, Yf, B);
#pragma unroll
        for (int k = 0; k < 9; ++k) T[k] = A[k] + B[k];
        decomp(T, tc);
        const float r = 1.0f / (cnorm(tc) + 1.0f);
#pragma unroll
        for (int k = 0; k < 9; ++k) tc[k] *= r;
        store_coords(Tn, i, c, N, F, tc);
        store_coords_cp(Tn_cp, i, c, N, F, tc);
    }
}

// X_out = Xn + dX + dX dX
__device__ __forceinline__ void residual(const float *__restrict__ Xn, const float *__restrict__ dX, int i, int c, int N,
                                         int F, float xv[9]) {
    float dv[9], Q[9], Q2[9], q2[9];
    load_coords(Xn, i, c, N, F, xv);
    load_coords(dX, i, c, N, F, dv);
    expand(dv, Q);
    mm3(Q, Q, Q2);
    decomp(Q2, q2);
#pragma unroll
    for (int k = 0; k < 9; ++k) xv[k] += dv[k] + q2[k];
}

// a layer's residual and the next layer's normalisation of it
__global__ void k_residual(const float *__restrict__ Xn, const float *__restrict__ dX, int N, int F,
                           float *__restrict__ qn, float *__restrict__ Xn_out, OpCopy Xn_cp) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * F;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / F), c = (int)(t % F);
        float xv[9];
        residual(Xn, dX, i, c, N, F, xv);
        store_normed(xv, t, i, c, N, F, qn, Xn_out, Xn_cp);
    }
}

// ---------------------------------------------------------- output ---
// h = (||I||, ||A||, ||S||) in blocks of F, LayerNorm over 3F.  Block per
// atom, thread per channel.  dX given: X is the last layer's residual, formed
// here from X (its Xn) and dX and stored to Xout.
__global__ void k_out_norms(const float *__restrict__ X, const float *__restrict__ dX, int N, int F,
                            const float *__restrict__ g, const float *__restrict__ b, float *__restrict__ Xout,
                            float *__restrict__ h, float *__restrict__ hn, float2 *__restrict__ ln) {
    pdl_entry();
    __shared__ float sm[32];
    const int i = blockIdx.x, c = threadIdx.x;
    float v[9];
    if (dX) {
        residual(X, dX, i, c, N, F, v);
        store_coords(Xout, i, c, N, F, v);
    } else {
        load_coords(X, i, c, N, F, v);
    }
    const float sxx = v[4], syy = v[5], szz = -(v[4] + v[5]);
    const float hv[3] = {3.0f * v[0] * v[0], 2.0f * (v[1] * v[1] + v[2] * v[2] + v[3] * v[3]),
                         sxx * sxx + syy * syy + szz * szz + 2.0f * (v[6] * v[6] + v[7] * v[7] + v[8] * v[8])};
    const float mean = block_sum(hv[0] + hv[1] + hv[2], sm) / (3 * F);
    const float d0 = hv[0] - mean, d1 = hv[1] - mean, d2 = hv[2] - mean;
    const float var = block_sum(d0 * d0 + d1 * d1 + d2 * d2, sm) / (3 * F);
    const float rstd = rsqrtf(var + 1e-5f);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int64_t o = (int64_t)i * 3 * F + p * F + c;
        h[o] = hv[p];
        hn[o] = (hv[p] - mean) * rstd * g[p * F + c] + b[p * F + c];
    }
    if (c == 0) ln[i] = make_float2(mean, rstd);
}

// E_i = w2 . t_i + b2 (one warp per atom)
__global__ void k_head(const float *__restrict__ t, int N, int H, const float *__restrict__ w2,
                       const float *__restrict__ b2, float *__restrict__ Ei) {
    pdl_entry();
    const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (i >= N) return;
    const int lane = threadIdx.x & 31;
    float s = 0.f;
    for (int k = lane; k < H; k += 32) s = fmaf(t[(int64_t)i * H + k], w2[k], s);
    s = warp_sum(s);
    if (lane == 0) Ei[i] = s + b2[0];
}

// E_s = sum of E_i over the system, in FP64 (one block per system; eight loads
// in flight per thread)
__global__ void k_energy(const float *__restrict__ Ei, const int32_t *__restrict__ sys_start,
                         const int32_t *__restrict__ sys_end, double *__restrict__ energy) {
    pdl_entry();
    __shared__ double sm[32];
    const int s = blockIdx.x;
    double acc = 0.0;
#pragma unroll 8
    for (int n = sys_start[s] + threadIdx.x; n < sys_end[s]; n += blockDim.x) acc += (double)Ei[n];
#pragma unroll
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sm[w];
        energy[s] = t;
    }
}

// ========================================================= reverse ===
__global__ void k_head_bwd(const float *__restrict__ at, int N, int H, const float *__restrict__ w2,
                           const float *__restrict__ seed, const int32_t *__restrict__ batch,
                           float *__restrict__ gat) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * H;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / H), k = (int)(t % H);
        const float gE = seed ? seed[batch ? batch[i] : 0] : 1.0f;
        gat[t] = gE * w2[k] * silu_grad_f(at[t]);
    }
}

// X_out = Xn + dX + dX dX:  g_dX = g + expand^T(G Q^T + Q^T G), G = decomp^T(g)
__device__ __forceinline__ void store_residual_adj(float g[9], const float *__restrict__ dX, int i, int c, int N, int F,
                                                   float *__restrict__ gdX, const OpCopy &gdX_cp) {
    float dv[9], G[9], Q[9], A[9], B[9], GQ[9], gq[9];
    load_coords(dX, i, c, N, F, dv);
    decomp_T(g, G);
    expand(dv, Q);
    mm3_nt(G, Q, A);
    mm3_tn(Q, G, B);
#pragma unroll
    for (int k = 0; k < 9; ++k) GQ[k] = A[k] + B[k];
    expand_T(GQ, gq);
#pragma unroll
    for (int k = 0; k < 9; ++k) g[k] += gq[k];
    store_coords(gdX, i, c, N, F, g);
    store_coords_cp(gdX_cp, i, c, N, F, g);
}

// LayerNorm backward over 3F, then d(norms)/d(coordinates) -> gX, and (dX
// given) the last layer's residual adjoint of it -> gdX
__global__ void k_out_norms_bwd(const float *__restrict__ X, const float *__restrict__ h,
                                const float *__restrict__ ghn, const float2 *__restrict__ ln,
                                const float *__restrict__ g, int N, int F, float *__restrict__ gX,
                                const float *__restrict__ dX, float *__restrict__ gdX, OpCopy gdX_cp) {
    pdl_entry();
    __shared__ float sm[32];
    const int i = blockIdx.x, c = threadIdx.x;
    const float2 mr = ln[i];
    float xh[3], gx[3];
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int64_t o = (int64_t)i * 3 * F + p * F + c;
        xh[p] = (h[o] - mr.x) * mr.y;
        gx[p] = ghn[o] * g[p * F + c];
        s1 += gx[p];
        s2 += gx[p] * xh[p];
    }
    const float m1 = block_sum(s1, sm) / (3 * F);
    const float m2 = block_sum(s2, sm) / (3 * F);
    float gh[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) gh[p] = mr.y * (gx[p] - m1 - xh[p] * m2);
    float v[9], gv[9];
    load_coords(X, i, c, N, F, v);
    gv[0] = __fmul_rn(6.0f * v[0], gh[0]);
#pragma unroll
    for (int k = 1; k < 4; ++k) gv[k] = __fmul_rn(4.0f * v[k], gh[1]);
    gv[4] = __fmul_rn(4.0f * v[4] + 2.0f * v[5], gh[2]);
    gv[5] = __fmul_rn(4.0f * v[5] + 2.0f * v[4], gh[2]);
#pragma unroll
    for (int k = 6; k < 9; ++k) gv[k] = __fmul_rn(4.0f * v[k], gh[2]);
    store_coords(gX, i, c, N, F, gv);
    if (dX) store_residual_adj(gv, dX, i, c, N, F, gdX, gdX_cp);
}

// Tn = decomp(Y M + M Y) / (p + 1): gradients to Y (written) and M (written)
__global__ void k_T_bwd(const float *__restrict__ Y, const float *__restrict__ M,
                        const float *__restrict__ gTn, int N, int F, float *__restrict__ gY,
                        float *__restrict__ gM) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * F;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / F), c = (int)(t % F);
        float yv[9], mv[9], Yf[9], Mf[9], A[9], B[9], T[9], tc[9], g[9], ng[9], GT[9];
        load_coords(Y, i, c, N, F, yv);
        load_coords(M, i, c, N, F, mv);
        load_coords(gTn, i, c, N, F, g);
        expand(yv, Yf);
        expand(mv, Mf);
        mm3(Yf, Mf, A);
        mm3(Mf, Yf, B);
#pragma unroll
        for (int k = 0; k < 9; ++k) T[k] = A[k] + B[k];
        decomp(T, tc);
        const float den = cnorm(tc) + 1.0f;
        float dot = 0.f;
#pragma unroll
        for (int k = 0; k < 9; ++k) dot = fmaf(g[k], tc[k], dot);
        cnorm_grad(tc, ng);
        const float a = 1.0f / den, bcoef = dot / (den * den);
#pragma unroll
        for (int k = 0; k < 9; ++k) g[k] = g[k] * a - bcoef * ng[k];
        decomp_T(g, GT);
        // dY = G M^T + M^T G ; dM = Y^T G + G Y^T
        float gYf[9], gMf[9], out[9];
        mm3_nt(GT, Mf, A);
        mm3_tn(Mf, GT, B);
#pragma unroll
        for (int k = 0; k < 9; ++k) gYf[k] = A[k] + B[k];
        mm3_tn(Yf, GT, A);
        mm3_nt(GT, Yf, B);
#pragma unroll
        for (int k = 0; k < 9; ++k) gMf[k] = A[k] + B[k];
        expand_T(gYf, out);
        store_coords(gY, i, c, N, F, out);
        expand_T(gMf, out);
        store_coords(gM, i, c, N, F, out);
    }
}

// Message adjoint and the last radial layer's elementwise adjoint.  For atom
// i (block, thread per channel):
//   gY_i += sum_j g^p_ij gM_j                          (g_ij = g_ji)
//   gg^p[u(i,j)] = <gM_i, Y^p_j> + <gM_j, Y^p_i>        for upper edges j > i
// with g = phi silu(a3) formed here from the pair's stored a3 and phi (the
// filter itself is never stored), and, for the same upper edge:
//   ga3 = gg phi silu'(a3)       (fp32 if ga3 != NULL, plus its operand copy)
//   gphi[u] += sum over the 3F entries of gg silu(a3)
// Each undirected pair is handled once, by its upper edge: no atomics.  The
// gphi sum is reduced per warp, then over the warps in a fixed order at the end
// of each chunk.  Rows ascend, so the upper edges are the row's suffix: the
// lower part gathers gM_j alone (kMU edges in flight), the upper part gM_j,
// Y_j and a3 together (kMUU edges).  Indices are staged in shared memory as in
// k_message; the gY sums run in row order.
// With TAB (tabulated radial functions) g and dg/dd come from the table: the
// kernel adds sum dE/dg dg/dd to gphi (then dE/dd of the pair) and writes no
// dE/da3.
// RB consecutive rows per block, one group of F threads per row, as in
// k_message (the groups' repeated gathers of gM_j and Y_j hit L1).
constexpr int kMUU = 2;
template <int F, bool TAB, int RB>
__global__ void __launch_bounds__(F * RB, (512 / (F * RB)) > 0 ? 512 / (F * RB) : 1)
    k_message_bwd(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                  const int32_t *__restrict__ pair_of, const float *__restrict__ Y,
                  const float *__restrict__ gM, const float *__restrict__ a3, const float *__restrict__ phiu,
                  TabFn tg, int N, float *__restrict__ gY, OpCopy gY_cp, float *__restrict__ ga3, OpCopy ga3_cp,
                  float *__restrict__ gphi) {
    pdl_entry();
    constexpr int NW = F / 32;
    constexpr int CH = RB >= 4 ? kChunk / 2 : kChunk;  // staged edges per chunk (static smem stays below 48 KB)
    __shared__ int32_t s_u_all[RB][CH], s_j_all[RB][CH];
    __shared__ int32_t s_kt_all[RB][TAB ? CH : 1];
    __shared__ float s_st_all[RB][TAB ? CH : 1];
    __shared__ float s_red_all[RB][CH][NW];
    __shared__ float s_yi_all[RB][9][F], s_gmi_all[RB][9][F];  // row i's Y and gM (per thread's channel)
    const int grp = RB > 1 ? (int)threadIdx.x / F : 0, c = RB > 1 ? (int)threadIdx.x % F : (int)threadIdx.x;
    const int lane = c & 31, warp = c >> 5;
    int32_t *s_u = s_u_all[grp], *s_j = s_j_all[grp], *s_kt = s_kt_all[grp];
    float *s_st = s_st_all[grp];
    float(*s_red)[NW] = s_red_all[grp];
    float(*s_yi)[F] = s_yi_all[grp];
    float(*s_gmi)[F] = s_gmi_all[grp];
    for (int i = blockIdx.x * RB + grp; i < N; i += gridDim.x * RB) {
        float acc[9];
        {
            float t[9];
            load_coords(Y, i, c, N, F, t);
#pragma unroll
            for (int q = 0; q < 9; ++q) s_yi[q][c] = t[q];
            load_coords(gM, i, c, N, F, t);
#pragma unroll
            for (int q = 0; q < 9; ++q) s_gmi[q][c] = t[q];
        }
        load_coords(gY, i, c, N, F, acc);
        const int e0 = row_ptr[i], e1 = row_ptr[i + 1];
        int eu = e0, hi = e1;  // eu = first edge with col > i
        while (eu < hi) {
            const int mid = (eu + hi) >> 1;
            if (col[mid] <= i) eu = mid + 1;
            else hi = mid;
        }
        for (int cb = e0; cb < e1; cb += CH) {
            const int n = e1 - cb < CH ? e1 - cb : CH;
            group_sync<F, RB>(grp);
            for (int t = c; t < n; t += F) {
                const int u = pair_of[cb + t];
                s_u[t] = u;
                s_j[t] = col[cb + t];
                if constexpr (TAB) {
                    int kt = 0;
                    float st = 0.f;
                    if (u >= 0) tab_locate(tg, u, kt, st);
                    s_kt[t] = kt;
                    s_st[t] = st;
                }
            }
            group_sync<F, RB>(grp);
            const int nl = eu - cb < 0 ? 0 : (eu - cb < n ? eu - cb : n);  // lower edges of the chunk
            for (int k0 = 0; k0 < nl; k0 += kMU) {
                int uu[kMU], jj[kMU];
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    uu[k] = k0 + k < nl ? s_u[k0 + k] : -1;
                    jj[k] = k0 + k < nl ? s_j[k0 + k] : 0;
                }
                float g[kMU][3], gmj[kMU][9], ph[kMU];
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    if (uu[k] < 0) continue;
                    if constexpr (TAB) {
                        const float4 *cp = tg.coef + (int64_t)s_kt[k0 + k] * 3 * F + c;
                        const float st = s_st[k0 + k];
                        g[k][0] = tab_value(cp[0], st); g[k][1] = tab_value(cp[F], st); g[k][2] = tab_value(cp[2 * F], st);
                    } else {
                        const float *ap = a3 + (int64_t)uu[k] * 3 * F + c;
                        g[k][0] = ap[0]; g[k][1] = ap[F]; g[k][2] = ap[2 * F];
                        ph[k] = phiu[uu[k]];
                    }
                    load_coords(gM, jj[k], c, N, F, gmj[k]);
                }
#pragma unroll
                for (int k = 0; k < kMU; ++k) {
                    if (uu[k] < 0) continue;
                    if constexpr (!TAB) {
#pragma unroll
                        for (int p = 0; p < 3; ++p) g[k][p] = silu_f(g[k][p]) * ph[k];
                    }
                    acc[0] = fmaf(g[k][0], gmj[k][0], acc[0]);
#pragma unroll
                    for (int q = 1; q < 4; ++q) acc[q] = fmaf(g[k][1], gmj[k][q], acc[q]);
#pragma unroll
                    for (int q = 4; q < 9; ++q) acc[q] = fmaf(g[k][2], gmj[k][q], acc[q]);
                }
            }
            for (int k0 = nl; k0 < n; k0 += kMUU) {
                int uu[kMUU], jj[kMUU];
#pragma unroll
                for (int k = 0; k < kMUU; ++k) {
                    uu[k] = k0 + k < n ? s_u[k0 + k] : -1;
                    jj[k] = k0 + k < n ? s_j[k0 + k] : 0;
                }
                float g[kMUU][3], gmj[kMUU][9], yj[kMUU][9], a[kMUU][3], phi[kMUU];
#pragma unroll
                for (int k = 0; k < kMUU; ++k) {
                    if (uu[k] < 0) continue;
                    if constexpr (TAB) {   // g and dg/dd (in a) from the pair's interval
                        const float4 *cp = tg.coef + (int64_t)s_kt[k0 + k] * 3 * F + c;
                        const float st = s_st[k0 + k];
#pragma unroll
                        for (int p = 0; p < 3; ++p) {
                            const float4 cq = cp[p * F];
                            g[k][p] = tab_value(cq, st);
                            a[k][p] = tab_slope(cq, st, tg.inv_h);
                        }
                        phi[k] = 0.f;
                    } else {
                        const int64_t o = (int64_t)uu[k] * 3 * F + c;
                        a[k][0] = a3[o]; a[k][1] = a3[o + F]; a[k][2] = a3[o + 2 * F];
                        phi[k] = phiu[uu[k]];
#pragma unroll
                        for (int p = 0; p < 3; ++p) g[k][p] = silu_f(a[k][p]) * phi[k];
                    }
                    load_coords(gM, jj[k], c, N, F, gmj[k]);
                    load_coords(Y, jj[k], c, N, F, yj[k]);
                }
#pragma unroll
                for (int k = 0; k < kMUU; ++k) {
                    if (uu[k] < 0) continue;
                    acc[0] = fmaf(g[k][0], gmj[k][0], acc[0]);
#pragma unroll
                    for (int q = 1; q < 4; ++q) acc[q] = fmaf(g[k][1], gmj[k][q], acc[q]);
#pragma unroll
                    for (int q = 4; q < 9; ++q) acc[q] = fmaf(g[k][2], gmj[k][q], acc[q]);
                    float sp[3];
                    sp[0] = s_gmi[0][c] * yj[k][0] + gmj[k][0] * s_yi[0][c];
                    sp[1] = 0.f; sp[2] = 0.f;
#pragma unroll
                    for (int q = 1; q < 4; ++q) sp[1] += s_gmi[q][c] * yj[k][q] + gmj[k][q] * s_yi[q][c];
#pragma unroll
                    for (int q = 4; q < 9; ++q) sp[2] += s_gmi[q][c] * yj[k][q] + gmj[k][q] * s_yi[q][c];
                    const int64_t o = (int64_t)uu[k] * 3 * F + c;
                    float r = 0.f;
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        if constexpr (TAB) {
                            r = fmaf(sp[p], a[k][p], r);
                        } else {
                            float sv, sd;
                            silu_and_grad_f(a[k][p], sv, sd);
                            r = fmaf(sp[p], sv, r);
                            const float ga = sp[p] * phi[k] * sd;
                            if (ga3) ga3[o + p * F] = ga;
                            opcopy_store(ga3_cp, o + p * F, ga);
                        }
                    }
                    r = warp_sum(r);
                    if (lane == 0) s_red[k0 + k - nl][warp] = r;
                }
            }
            group_sync<F, RB>(grp);
            for (int t = c; t < n - nl; t += F) {
                const int u = s_u[nl + t];
                if (u < 0) continue;
                float r = 0.f;
#pragma unroll
                for (int w = 0; w < NW; ++w) r += s_red[t][w];
                gphi[u] += r;
            }
        }
        store_coords(gY, i, c, N, F, acc);
        store_coords_cp(gY_cp, i, c, N, F, acc);
    }
}

// ------------------------------------------------ staged message kernels ---
// The same sums as k_message and k_message_bwd (exact mode, F = 64 or 128), with the
// gathered node rows shared by a group of rows.  A block takes up to G
// consecutive rows at a time.  One warp merges the rows' column lists (they
// ascend), three copy each distinct column's node rows into a ring of
// shared-memory slots, once for the whole group: consecutive atoms share most
// of their neighbours (in a water box 12 rows use a column 4.4 times, 6 rows
// 3.2 times).  Consumer warps, one per row with four channels a lane (the
// adjoint: two per row with two, so that row i's own Y and gM stay in
// registers), take the slots their row needs in column order, the same order
// of additions as the gathers.  The pair's a3 rows, which nothing else in the
// group uses, come through a ring per warp, a few edges ahead.
// What bounded the gathers was not bandwidth but latency (long-scoreboard
// stalls, 12 warps with 24 row loads each in flight, 115 SM cycles an edge with
// every pipe below half); both rings keep their loads ahead of the warps.  Now
// the consumers' own work bounds both, with four warps a scheduler to hide it:
// at 24,000 atoms a consumer waits for a stage a quarter of the time in the
// messages and 13% in the adjoint, the merge (213 cycles a column) 44% and 62%
// for a free one; half of the issue slots and 60-66% of the shared-memory
// wavefronts are used (ncu).  Per launch, 96,000 atoms (5.2 M edges): messages 2.00 -> 1.46
// ms, adjoint 4.16 -> 3.46; 3,000 atoms 76 -> 55 us and 148 -> 140.
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// first element (in floats) of coordinate row q (0..8) of atom n in a node
// tensor laid out as I rows [0, N), A rows [N, 4N), S rows [4N, 9N)
__device__ __forceinline__ uint32_t coord_row(int q, uint32_t n, uint32_t N, uint32_t F) {
    return (q == 0 ? n : (q < 4 ? N + 3u * n + (uint32_t)(q - 1) : 4u * N + 5u * n + (uint32_t)(q - 4))) * F;
}
// plane p (I, A, S) of coordinate q
__device__ __forceinline__ constexpr int plane_of(int q) { return q == 0 ? 0 : (q < 4 ? 1 : 2); }

// 2 NP consecutive channels of a lane as NP packed pairs
template <int NP>
struct Ch {
    uint64_t v[NP];
};
template <int NP>
__device__ __forceinline__ Ch<NP> ldc(const float *__restrict__ p) {
    Ch<NP> r;
    if constexpr (NP == 2) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
        r.v[0] = t.x; r.v[1] = t.y;
    } else {
        r.v[0] = *reinterpret_cast<const unsigned long long *>(p);
    }
    return r;
}
template <int NP>
__device__ __forceinline__ void stc(float *__restrict__ p, const Ch<NP> &c) {
    if constexpr (NP == 2) *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(c.v[0], c.v[1]);
    else *reinterpret_cast<unsigned long long *>(p) = c.v[0];
}
template <int NP>
__device__ __forceinline__ void opcopy_store_c(const OpCopy &o, int64_t idx, const Ch<NP> &c) {
    if (o.mode != 1) return;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const float2 t = f2_unpack(c.v[k]);
        *reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(o.p) + idx + 2 * k) =
            __floats2bfloat162_rn(t.x, t.y);
    }
}
// asynchronous copy of a lane's 16 or 8 bytes, in the thread's copy groups
template <int BYTES>
__device__ __forceinline__ void cp_lane(void *dst, const void *src) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}
// one arrival of this thread on a barrier once its copies so far have landed
__device__ __forceinline__ void cp_arrive(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

// Shape of the staged kernels: warps per row, rows per group, slots per stage
// and stages of the node ring, depth of the a3 rings, copying warps, and the
// edges of a row listed at a time (longer rows take several passes over the
// group).  Sixteen warps leave 128 registers to each, which the adjoint needs
// (row i's Y, gM and sum, 54 of them): with twenty and 96 it spills, and with
// nearly all of L1 given to shared memory a spill goes to L2 (15.3 ms against
// 6.9).  Measured at 96,000 atoms, both launches of a call: messages with 16
// rows (twenty warps) 3.00 ms, 13 rows 3.06, 12 rows 2.91; adjoint with 7 rows
// and one copying warp 7.50, 6 and three 6.91, 5 and two 8.27.
template <int N>
using Channels = std::integral_constant<int, N>;
template <int F, bool BWD>
struct MsgTile {
    static constexpr int HW = BWD && F > 64 ? 2 : 1, G = 12 / HW, NS = BWD ? 4 : 8, ST = BWD ? 4 : 3, D = BWD ? 4 : 3;
    static constexpr int CAP = 100, C = G * HW, CW = 3, THREADS = 32 * (C + 1 + CW), FH = F / HW, NP = FH / 64;
    static constexpr int NODE = 9 * F * 4, SLOT = (BWD ? 2 : 1) * NODE, A3 = 3 * FH * 4;
    static constexpr int o_ring = ST * NS * SLOT, o_col = o_ring + C * D * A3, o_u = o_col + 2 * G * CAP * 4;
    static constexpr int o_ph = o_u + 2 * G * CAP * 4, o_cnt = o_ph + 2 * G * CAP * 4, o_more = o_cnt + 2 * G * 4;
    static constexpr int o_mask = o_more + 2 * G * 4, o_j = o_mask + ST * NS * 4, o_meta = o_j + ST * NS * 4, o_bar = (o_meta + ST * 4 + 15) & ~15;
    static constexpr int BARS = 3 * ST + 4, SMEM = o_bar + 8 * BARS;
    static_assert(NP >= 1 && FH == 64 * NP && SMEM <= 232448 - 256, "shared memory above 227 KB");
};

// F = 64 runs both at one warp per row, two channels a lane (12,003 atoms, 612,000
// edges, per launch against a thread per channel: messages 205 -> 147 us, adjoint
// 377 -> 264 us).
// BWD false: V = Y, out = M, M_i = sum_j g_ij Y_j.
// BWD true: V = gM, V2 = Y, out = gY (added to), and per upper edge (j > i)
// dE/dg = <gM_i, Y_j> + <gM_j, Y_i>, ga3 = dE/dg phi SiLU'(a3) and gphi[half][u]
// += sum dE/dg SiLU(a3) over the warp's channels.
// Every wait is bounded and its verdict is the warp's: on expiry the block
// records TIMEOUT, each warp stops as a whole and waits for its own copies.
// Testing only (zero in every library call): spin_limit, a smaller bound on
// each wait, and hold_copies, copying warps that copy nothing and arrive
// nowhere, so that the consumers' waits run out.
template <int F, bool BWD>
__global__ void __launch_bounds__(MsgTile<F, BWD>::THREADS, 1)
    k_message_tile(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                   const int32_t *__restrict__ pair_of, const float *__restrict__ a3, const float *__restrict__ phiu,
                   const float *__restrict__ V, const float *__restrict__ V2, int N, int R, float *__restrict__ out,
                   OpCopy out_cp, float *__restrict__ ga3, OpCopy ga3_cp, float *__restrict__ gphi,
                   int64_t gphi_stride, int32_t *status, uint32_t spin_limit, int hold_copies) {
    pdl_entry();
    using T = MsgTile<F, BWD>;
    constexpr int NP = T::NP, FH = T::FH, G = T::G, HW = T::HW, NS = T::NS, ST = T::ST, D = T::D, C = T::C, CAP = T::CAP;
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ int s_abort;
    int *l_col = reinterpret_cast<int *>(sm + T::o_col);          // [2][G][CAP] columns of the active edges
    int *l_u = reinterpret_cast<int *>(sm + T::o_u);              // their pairs
    float *l_ph = reinterpret_cast<float *>(sm + T::o_ph);        // and cutoff factors
    int *l_cnt = reinterpret_cast<int *>(sm + T::o_cnt);          // [2][G] edges listed
    int *l_more = reinterpret_cast<int *>(sm + T::o_more);        // [2][G] the row has edges beyond this pass
    uint32_t *s_mask = reinterpret_cast<uint32_t *>(sm + T::o_mask);  // [ST][NS] rows that use the slot
    int *s_j = reinterpret_cast<int *>(sm + T::o_j);              // [ST][NS] the slot's atom; ~j: its V2 rows too
    int *s_meta = reinterpret_cast<int *>(sm + T::o_meta);        // [ST] slots filled, + 256 on a pass's last stage
                                                                  // (+ 512 on the block's last)
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + T::o_bar), *empty = full + ST, *l_full = empty + ST, *l_empty = l_full + 2, *named = l_empty + 2;
    volatile int *abort_flag = &s_abort;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            tc::mbar_init(&full[s], 32 * T::CW + 1);
            tc::mbar_init(&empty[s], C);
            tc::mbar_init(&named[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&l_full[b], G);
            tc::mbar_init(&l_empty[b], C + 1);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int groups = (N + R - 1) / R;
    bool ok = true;
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        if (!tc::mbar_wait_warp(bar, parity, abort_flag, spin_limit)) {
            if (!*abort_flag) set_status(status, TNET_ERR_TIMEOUT);
            *abort_flag = 1;
            ok = false;
        }
        return ok;
    };
    // whether any row of list buffer b goes on beyond its pass
    auto any_more = [&](int b) { return __any_sync(0xffffffffu, lane < G && l_more[b * G + lane] != 0); };

    if (w == C) {  // ------------------------------------- merges the rows' columns
        int n_stage = 0;
        int g = blockIdx.x;
        for (int t = 0; ok && g < groups; ++t) {
            const int b = t & 1;
            if (!wait(&l_full[b], (t >> 1) & 1)) break;
            const bool more = any_more(b);
            const int g_next = more ? g : g + gridDim.x;
            // this lane's row: its next two columns, the one after them loaded
            // ahead of each step (two entries of INT_MAX end a list)
            const int *mine = l_col + (b * G + (lane < G ? lane : 0)) * CAP;
            int cur = lane < G ? mine[0] : 0x7fffffff, nxt = lane < G ? mine[1] : 0x7fffffff, k = 2, slot = 0;
            if (cur == 0x7fffffff) nxt = cur;
            for (;;) {
                const int s = n_stage % ST;
                if (slot == 0 && n_stage >= ST && !wait(&empty[s], ((n_stage / ST) - 1) & 1)) break;
                const int after = mine[k < CAP ? k : CAP - 1];
                const int j = __reduce_min_sync(0xffffffffu, cur);
                const bool end = j == 0x7fffffff;
                if (!end) {
                    // no branches on the lane: every lane writes the same words
                    const bool use = cur == j;
                    const unsigned rows = __ballot_sync(0xffffffffu, use);
                    cur = use ? nxt : cur;
                    nxt = use ? (nxt == 0x7fffffff ? nxt : after) : nxt;
                    k += use;
                    s_mask[s * NS + slot] = rows;
                    // Y_j serves upper edges alone
                    s_j[s * NS + slot] = BWD && j > g * R + __ffs(rows) - 1 ? ~j : j;
                    ++slot;
                }
                if (end || slot == NS) {
                    __syncwarp();
                    if (lane == 0) {
                        s_meta[s] = slot | (end ? 256 : 0) | (end && g_next >= groups ? 512 : 0);
                        tc::mbar_arrive(&named[s]);
                        tc::mbar_arrive(&full[s]);
                    }
                    ++n_stage;
                    slot = 0;
                    if (end) break;
                }
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&l_empty[b]);
            g = g_next;
        }
    } else if (w > C) {  // -------------------------------- copy the node rows in
        for (int n_stage = 0; !hold_copies; ++n_stage) {
            const int s = n_stage % ST;
            if (!wait(&named[s], (n_stage / ST) & 1)) break;
            const int meta = s_meta[s];
            for (int slot = w - C - 1; slot < (meta & 255); slot += T::CW) {
                int j = s_j[s * NS + slot];
                const bool both = j < 0;
                if (both) j = ~j;
                uint8_t *dst = sm + (s * NS + slot) * T::SLOT + 16 * lane;
                const float *rI = V + (int64_t)j * F + 4 * lane, *rA = V + ((int64_t)N + 3LL * j) * F + 4 * lane,
                            *rS = V + (4LL * N + 5LL * j) * F + 4 * lane;
                if (4 * lane < F) {
#pragma unroll
                    for (int q = 0; q < 9; ++q)
                        cp_lane<16>(dst + q * F * 4, q == 0 ? rI : (q < 4 ? rA + (q - 1) * F : rS + (q - 4) * F));
                    if (both) {
                        const int64_t d = V2 - V;
#pragma unroll
                        for (int q = 0; q < 9; ++q)
                            cp_lane<16>(dst + T::NODE + q * F * 4,
                                        d + (q == 0 ? rI : (q < 4 ? rA + (q - 1) * F : rS + (q - 4) * F)));
                    }
                }
            }
            cp_arrive(&full[s]);  // each lane, once its copies have landed
            if (meta & 512) break;
        }
        // own copies, which are in no copy group, land before the warp exits
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else {  // ----------------------------------------------------- consumers
        const int r = w / HW, half = w % HW;
        const uint32_t c0 = half * FH + 2 * NP * lane;
        // the lane's own a3 values: D edges of three planes
        uint8_t *ring = sm + T::o_ring + w * D * T::A3 + 8 * NP * lane;
        if (BWD) gphi += half * gphi_stride;
        int e_next = 0, e_end = 0;  // edges of the row not listed yet
        auto row_of = [&](int g) {
            const int64_t i = (int64_t)g * R + r;
            return r < R && g < groups && i < N ? (int)i : -1;
        };
        auto open_row = [&](int g) {
            const int i = row_of(g);
            e_next = i >= 0 ? row_ptr[i] : 0;
            e_end = i >= 0 ? row_ptr[i + 1] : 0;
        };
        // the row's next active edges into list buffer b (both halves keep
        // count, the first writes)
        auto list_row = [&](int b) {
            int n = 0;
            const int at = (b * G + r) * CAP;
            while (e_next < e_end && n <= CAP - 34) {
                const int e = e_next + lane;
                const int u = e < e_end ? pair_of[e] : -1;
                const int j = e < e_end ? col[e] : 0;
                const unsigned m = __ballot_sync(0xffffffffu, u >= 0);
                if (half == 0 && u >= 0) {
                    const int q = at + n + __popc(m & ((1u << lane) - 1u));
                    l_col[q] = j;
                    l_u[q] = u;
                    l_ph[q] = phiu[u];
                }
                n += __popc(m);
                e_next += 32;
            }
            if (half == 0) {
                if (lane < 2) l_col[at + n + lane] = 0x7fffffff;  // two past the end, for the merge
                if (lane == 0) {
                    l_cnt[b * G + r] = n;
                    l_more[b * G + r] = e_next < e_end;
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&l_full[b]);
            }
        };
        // edge u's a3 into ring place d, one copy group per edge
        auto fetch = [&](int u, int d) {
            const float *src = a3 + (int64_t)u * 3 * F + c0;
#pragma unroll
            for (int p = 0; p < 3; ++p) cp_lane<8 * NP>(ring + d * T::A3 + p * FH * 4, src + p * F);
        };
        int g = blockIdx.x, n_stage = 0;
        open_row(g);
        if (g < groups) list_row(0);
        Ch<NP> acc[9], yi[9], gi[9];
        bool fresh = true;  // the group's first pass
        for (int t = 0; ok && g < groups; ++t) {
            const int b = t & 1;
            if (!wait(&l_full[b], (t >> 1) & 1)) break;
            const bool more = any_more(b);
            const int i = row_of(g), n = l_cnt[b * G + r], at = (b * G + r) * CAP;
            int k = 0, place = 0;  // edges done; ring place of the next one
#pragma unroll
            for (int d = 0; d < D; ++d) {
                if (d < n) fetch(l_u[at + d], d);
                cp_commit();
            }
            if (fresh) {
#pragma unroll
                for (int q = 0; q < 9; ++q) {
#pragma unroll
                    for (int x = 0; x < NP; ++x) acc[q].v[x] = 0;
                    if (BWD && i >= 0) {
                        const uint32_t o = coord_row(q, (uint32_t)i, (uint32_t)N, F) + c0;
                        yi[q] = ldc<NP>(V2 + o);
                        gi[q] = ldc<NP>(V + o);
                        acc[q] = ldc<NP>(out + o);
                    }
                }
            }
            const int g_next = more ? g : g + gridDim.x;
            for (bool first = true;; first = false) {
                const int s = n_stage % ST;
                if (!wait(&full[s], (n_stage / ST) & 1)) break;
                const int meta = s_meta[s];
                unsigned slots = __ballot_sync(0xffffffffu, lane < (meta & 255) && ((s_mask[s * NS + (lane < NS ? lane : 0)] >> r) & 1u));
                while (slots && ok) {
                    const int sl = __ffs(slots) - 1;
                    slots &= slots - 1;
                    const float *node = reinterpret_cast<const float *>(sm + (s * NS + sl) * T::SLOT) + c0;
                    const int u = l_u[at + k], j = l_col[at + k];
                    const float ph = l_ph[at + k];
                    cp_wait<D - 1>();  // one group per edge: the oldest has landed
                    const float *sa = reinterpret_cast<const float *>(ring + place * T::A3);
                    Ch<NP> a[3], sg[3], gv[3];
#pragma unroll
                    for (int p = 0; p < 3; ++p) a[p] = ldc<NP>(sa + p * FH);
                    const bool upper = BWD && j > i;  // the same in every lane
                    Ch<NP> v[9], sp[3];
                    const uint64_t ph2 = f2_pack(ph, ph);
#pragma unroll
                    for (int p = 0; p < 3; ++p)
#pragma unroll
                        for (int x = 0; x < NP; ++x) {
                            const float2 t = f2_unpack(a[p].v[x]);
                            if constexpr (BWD) {  // the sigmoid, kept for SiLU'
                                sg[p].v[x] = f2_pack(sigmoid_f(t.x), sigmoid_f(t.y));
                                gv[p].v[x] = f2_mul(f2_mul(a[p].v[x], sg[p].v[x]), ph2);
                            } else {
                                gv[p].v[x] = f2_mul(f2_pack(silu_f(t.x), silu_f(t.y)), ph2);
                            }
                        }
                    // the place is read: the edge D further on takes it
                    if (k + D < n) fetch(l_u[at + k + D], place);
                    cp_commit();
                    ++k;
                    place = place + 1 == D ? 0 : place + 1;
#pragma unroll
                    for (int q = 0; q < 9; ++q) v[q] = ldc<NP>(node + q * F);
#pragma unroll
                    for (int q = 0; q < 9; ++q)
#pragma unroll
                        for (int x = 0; x < NP; ++x)
                            acc[q].v[x] = f2_fma(gv[plane_of(q)].v[x], v[q].v[x], acc[q].v[x]);
                    if constexpr (BWD) {
                        if (!upper) continue;
#pragma unroll
                        for (int q = 0; q < 9; ++q)
#pragma unroll
                            for (int x = 0; x < NP; ++x)
                                sp[plane_of(q)].v[x] = f2_fma(v[q].v[x], yi[q].v[x],
                                                              (q == 0 || q == 1 || q == 4) ? 0 : sp[plane_of(q)].v[x]);
#pragma unroll
                        for (int q = 0; q < 9; ++q) {
                            const Ch<NP> yj = ldc<NP>(node + (9 + q) * F);
#pragma unroll
                            for (int x = 0; x < NP; ++x)
                                sp[plane_of(q)].v[x] = f2_fma(gi[q].v[x], yj.v[x], sp[plane_of(q)].v[x]);
                        }
                        const uint32_t ab = (uint32_t)u * 3u * F + c0;
                        uint64_t r2 = 0;
                        const uint64_t one = f2_pack(1.f, 1.f), neg = f2_pack(-1.f, -1.f);
#pragma unroll
                        for (int p = 0; p < 3; ++p) {
                            Ch<NP> ga;
#pragma unroll
                            for (int x = 0; x < NP; ++x) {
                                const uint64_t v = a[p].v[x], sv = sg[p].v[x], d = sp[p].v[x];
                                r2 = f2_fma(d, f2_mul(v, sv), r2);
                                // SiLU' = s (1 + x (1 - s))
                                const uint64_t sd = f2_mul(sv, f2_fma(v, f2_fma(sv, neg, one), one));
                                ga.v[x] = f2_mul(f2_mul(d, ph2), sd);
                            }
                            if (ga3) stc<NP>(ga3 + ab + p * F, ga);
                            opcopy_store_c<NP>(ga3_cp, ab + p * F, ga);
                        }
                        const float2 rr = f2_unpack(r2);
                        float rsum = rr.x + rr.y;
                        rsum = warp_sum(rsum);
                        if (lane == 0) gphi[u] += rsum;
                    }
                }
                if (!ok) break;
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&empty[s]);
                ++n_stage;
                if (first && g_next < groups) {
                    // the next pass's list, while this one's copies run: its
                    // buffer is free once every warp is through with pass t - 1
                    if (t >= 1 && !wait(&l_empty[b ^ 1], ((t - 1) >> 1) & 1)) break;
                    if (!more) open_row(g_next);
                    list_row(b ^ 1);
                }
                if (meta & 256) break;
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&l_empty[b]);
            fresh = !more;
            if (!more && i >= 0) {
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    const uint32_t o = coord_row(q, (uint32_t)i, (uint32_t)N, F) + c0;
                    stc<NP>(out + o, acc[q]);
                    if (BWD) opcopy_store_c<NP>(out_cp, o, acc[q]);
                }
            }
            g = g_next;
        }
        cp_wait<0>();
    }
}

// Rows per group of the staged message kernels: at most `most`, and as few as
// let every SM have the same number of groups.
static void msg_shape(int N, int sms, int most, int &run, int &grid) {
    const int64_t rounds = (N + (int64_t)most * sms - 1) / ((int64_t)most * sms);
    run = (int)((N + rounds * sms - 1) / (rounds * sms));
    const int groups = (N + run - 1) / run;
    grid = groups < sms ? groups : sms;
}
template <int F, bool BWD>
static int message_tile(int sms, cudaStream_t st, const int32_t *row_ptr, const int32_t *col, const int32_t *pair_of,
                        const float *a3, const float *phiu, const float *V, const float *V2, int N, float *out,
                        OpCopy out_cp, float *ga3, OpCopy ga3_cp, float *gphi, int64_t gphi_stride, int32_t *status,
                        uint32_t spin_limit = 0, int hold_copies = 0) {
    using T = MsgTile<F, BWD>;
    const int rc = ensure_smem_attr((const void *)k_message_tile<F, BWD>, T::SMEM);
    if (rc) return rc;
    int run, grid;
    msg_shape(N, sms, T::G, run, grid);
    launch(k_message_tile<F, BWD>, grid, T::THREADS, T::SMEM, st, row_ptr, col, pair_of, a3, phiu, V, V2, N, run, out,
           out_cp, ga3, ga3_cp, gphi, gphi_stride, status, spin_limit, hold_copies);
    return TNET_OK;
}

// Xn = X / (q + 1), q = ||X||:  gX = gXn / (q + 1) - <gXn, X> / (q + 1)^2 * dq/dX
__device__ __forceinline__ void norm_adj(const float xv[9], float q, float g[9]) {
    float ng[9];
    const float den = q + 1.0f;
    float dot = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) dot = fmaf(g[k], xv[k], dot);
    cnorm_grad(xv, ng);
    const float a = 1.0f / den, b = dot / (den * den);
#pragma unroll
    for (int k = 0; k < 9; ++k) g[k] = g[k] * a - b * ng[k];
}

// The normalisation adjoint of a layer's input X, in place on gX, and the
// residual adjoint of the layer before, whose output X is: X is formed again
// from that layer's Xn and dX, as the forward pass formed it.
__global__ void k_node_norm_bwd(const float *__restrict__ Xn, const float *__restrict__ dX,
                                const float *__restrict__ qn, int N, int F, float *__restrict__ gX,
                                float *__restrict__ gdX, OpCopy gdX_cp) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * F;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / F), c = (int)(t % F);
        float xv[9], g[9];
        residual(Xn, dX, i, c, N, F, xv);
        load_coords(gX, i, c, N, F, g);
        norm_adj(xv, qn[t], g);
        store_coords(gX, i, c, N, F, g);
        store_residual_adj(g, dX, i, c, N, F, gdX, gdX_cp);
    }
}

// X0 = s_p * U:  gU = s_p gX0; gas2 = <gX0, U>_p * silu'(as2).  gX0 comes from
// the first layer's normalisation adjoint (qn given; X0 is formed again) or,
// without layers, as it lies in gX.
__global__ void k_emb_scale_bwd(const float *__restrict__ gX, const float *__restrict__ qn,
                                const float *__restrict__ U, const float *__restrict__ s, const float *__restrict__ as2,
                                int N, int F, float *__restrict__ gU, float *__restrict__ gas2, OpCopy gU_cp) {
    pdl_entry();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)N * F;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / F), c = (int)(t % F);
        float g[9], uv[9];
        load_coords(gX, i, c, N, F, g);
        load_coords(U, i, c, N, F, uv);
        const float *si = s + t * 3;
        if (qn) {
            float xv[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) xv[k] = __fmul_rn(uv[k], si[plane_of(k)]);
            norm_adj(xv, qn[t], g);
        }
        float gs[3] = {g[0] * uv[0], 0.f, 0.f};
#pragma unroll
        for (int k = 1; k < 4; ++k) gs[1] += g[k] * uv[k];
#pragma unroll
        for (int k = 4; k < 9; ++k) gs[2] += g[k] * uv[k];
        g[0] *= si[0];
#pragma unroll
        for (int k = 1; k < 4; ++k) g[k] *= si[1];
#pragma unroll
        for (int k = 4; k < 9; ++k) g[k] *= si[2];
        store_coords(gU, i, c, N, F, g);
        store_coords_cp(gU_cp, i, c, N, F, g);
#pragma unroll
        for (int p = 0; p < 3; ++p) gas2[t * 3 + p] = gs[p] * silu_grad_f(as2[t * 3 + p]);
    }
}

// LayerNorm of q0 = ||X_raw||: adds gq0 * dq0/dX_raw to gXraw (which holds the
// channel-mixing adjoint)
__global__ void k_ln0_bwd(const float *__restrict__ Xraw, const float *__restrict__ gn0,
                          const float2 *__restrict__ ln, const float *__restrict__ g, int N, int F,
                          float *__restrict__ gXraw) {
    pdl_entry();
    __shared__ float sm[32];
    const int i = blockIdx.x, c = threadIdx.x;
    float v[9], gv[9], ng[9];
    load_coords(Xraw, i, c, N, F, v);
    const float2 mr = ln[i];
    const float xh = (cnorm(v) - mr.x) * mr.y;
    const float gx = gn0[(int64_t)i * F + c] * g[c];
    const float m1 = block_sum(gx, sm) / F;
    const float m2 = block_sum(gx * xh, sm) / F;
    const float gq = mr.y * (gx - m1 - xh * m2);
    load_coords(gXraw, i, c, N, F, gv);
    cnorm_grad(v, ng);
#pragma unroll
    for (int k = 0; k < 9; ++k) gv[k] = fmaf(gq, ng[k], gv[k]);
    store_coords(gXraw, i, c, N, F, gv);
}

// Embedding edge adjoint, one warp per atom i (lane = channels lane + 32k).
// For each active directed edge e = (i, j) of the row it writes
//   edge_g[e] = (dE/dphi, dE/du) of that directed use of the pair (u = r_ij/d),
// and for upper edges (j > i) the pair's projection adjoint summed over both
// directions, gfu[u] = dE/df^p (columns p*F + c), which needs gXraw_j.
// With want_z it also sums the pair-embedding adjoints dE/dZ per atom as
// receiver (gA_atom) and as sender (gB_atom) for the embedding-table gradients.
template <int CPL>
__global__ void k_emb_bwd(const float *__restrict__ pos, const float *__restrict__ box,
                          const int32_t *__restrict__ batch, const int32_t *__restrict__ z,
                          const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                          const int32_t *__restrict__ pair_of, int N, int max_z, RadialParams rp,
                          const float *__restrict__ fu, const float *__restrict__ Ta,
                          const float *__restrict__ Tb, const float *__restrict__ gXraw, int want_z,
                          float *__restrict__ gfu, float4 *__restrict__ edge_g, float *__restrict__ gA_atom,
                          float *__restrict__ gB_atom, OpCopy gfu_cp) {
    pdl_entry();
    constexpr int F = CPL * 32;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t ii = warp0; ii < N; ii += nwarps) {
        const int i = (int)ii;
        int zi = z[i];
        zi = (zi < 0 || zi >= max_z) ? 0 : zi;
        float gi[CPL][9], ta[CPL], tbi[CPL], accA[CPL], accB[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int c = lane + 32 * k;
            load_coords(gXraw, i, c, N, F, gi[k]);
            ta[k] = Ta[(int64_t)zi * F + c];
            tbi[k] = Tb[(int64_t)zi * F + c];
            accA[k] = accB[k] = 0.f;
        }
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            const int u = pair_of[e];
            if (u < 0) {
                if (lane == 0) edge_g[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                continue;
            }
            const int j = col[e];
            float x, y, zz;
            pair_vec(pos, box, batch, i, j, x, y, zz);
            const float d = sqrtf(norm2_rn(x, y, zz));
            const float inv = 1.0f / d;
            const float ux = x * inv, uy = y * inv, uz = zz * inv;
            const float phi = cutoff_phi(d, rp);
            const float bxx = ux * ux - (1.0f / 3.0f), byy = uy * uy - (1.0f / 3.0f);
            const float bxy = ux * uy, bxz = ux * uz, byz = uy * uz;
            int zj = z[j];
            zj = (zj < 0 || zj >= max_z) ? 0 : zj;
            const bool upper = j > i;
            const bool need_j = upper || want_z;
            float gphi = 0.f, gux = 0.f, guy = 0.f, guz = 0.f;
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                const int c = lane + 32 * k;
                const float *fp = fu + (int64_t)u * 3 * F + c;
                const float f0 = fp[0], f1 = fp[F], f2 = fp[2 * F];
                const float Zij = ta[k] + Tb[(int64_t)zj * F + c];
                const float *g = gi[k];
                const float gc0 = g[0];
                const float gcA = g[1] * ux + g[2] * uy + g[3] * uz;
                const float gcS = g[4] * bxx + g[5] * byy + g[6] * bxy + g[7] * bxz + g[8] * byz;
                const float dot = gc0 * f0 + gcA * f1 + gcS * f2;
                gphi = fmaf(Zij, dot, gphi);
                const float cA = phi * Zij * f1, cS = phi * Zij * f2;
                gux += cA * g[1] + cS * (2.f * ux * g[4] + uy * g[6] + uz * g[7]);
                guy += cA * g[2] + cS * (2.f * uy * g[5] + ux * g[6] + uz * g[8]);
                guz += cA * g[3] + cS * (ux * g[7] + uy * g[8]);
                accA[k] = fmaf(phi, dot, accA[k]);
                if (need_j) {
                    float gj[9];
                    load_coords(gXraw, j, c, N, F, gj);
                    // the reverse use (j, i): u_ji = -u, the S basis is even in u
                    const float hc0 = gj[0];
                    const float hcA = -(gj[1] * ux + gj[2] * uy + gj[3] * uz);
                    const float hcS = gj[4] * bxx + gj[5] * byy + gj[6] * bxy + gj[7] * bxz + gj[8] * byz;
                    const float Zji = Ta[(int64_t)zj * F + c] + tbi[k];
                    if (upper) {
                        float *o = gfu + (int64_t)u * 3 * F + c;
                        const float o0 = phi * (Zij * gc0 + Zji * hc0);
                        const float o1 = phi * (Zij * gcA + Zji * hcA);
                        const float o2 = phi * (Zij * gcS + Zji * hcS);
                        o[0] = o0;
                        o[F] = o1;
                        o[2 * F] = o2;
                        const int64_t ob = (int64_t)u * 3 * F + c;
                        opcopy_store(gfu_cp, ob, o0);
                        opcopy_store(gfu_cp, ob + F, o1);
                        opcopy_store(gfu_cp, ob + 2 * F, o2);
                    }
                    accB[k] = fmaf(phi, hc0 * f0 + hcA * f1 + hcS * f2, accB[k]);
                }
            }
            gphi = warp_sum(gphi);
            gux = warp_sum(gux);
            guy = warp_sum(guy);
            guz = warp_sum(guz);
            if (lane == 0) edge_g[e] = make_float4(gphi, gux, guy, guz);
        }
        if (want_z) {
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                gA_atom[(int64_t)i * F + lane + 32 * k] = accA[k];
                gB_atom[(int64_t)i * F + lane + 32 * k] = accB[k];
            }
        }
    }
}

// Embedding edge adjoint for forces only, one warp per undirected pair
// (lane = channels lane + 32k): both directed uses of the pair at once,
//   edge_g[e]      = (dE/dphi, dE/du) of the use (i, j), u = r_ij / d
//   edge_g[rev e]  = the same for (j, i), u_ji = -u
//   gfu[u]         = dE/df^p summed over both uses (columns p*F + c).
// Pair-parallel, so small systems still fill the GPU.
template <int CPL, bool TAB>
__global__ void k_emb_bwd_pairs(const float4 *__restrict__ geo, const int32_t *__restrict__ z,
                                const int2 *__restrict__ uij, const int32_t *__restrict__ ue,
                                const int32_t *__restrict__ rev, const int32_t *__restrict__ nu, int N, int max_z,
                                const float *__restrict__ fu, TabFn tf, const float *__restrict__ Ta,
                                const float *__restrict__ Tb, const float *__restrict__ gXraw,
                                float *__restrict__ gfu, float4 *__restrict__ edge_g,
                                OpCopy gfu_cp, float *__restrict__ dEdd) {
    pdl_entry();
    constexpr int F = CPL * 32;
    const int lane = threadIdx.x & 31;
    const int U = *nu;
    for (int64_t uu = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; uu < U;
         uu += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int u = (int)uu;
        const int2 p = uij[u];
        const int i = p.x, j = p.y;
        const float4 gu = geo[u];  // u_ij and phi of the pair (k_edge_rbf or k_pair_geo)
        const float ux = gu.x, uy = gu.y, uz = gu.z, phi = gu.w;
        const float bxx = ux * ux - (1.0f / 3.0f), byy = uy * uy - (1.0f / 3.0f);
        const float bxy = ux * uy, bxz = ux * uz, byz = uy * uz;
        int zi = z[i], zj = z[j];
        zi = (zi < 0 || zi >= max_z) ? 0 : zi;
        zj = (zj < 0 || zj >= max_z) ? 0 : zj;
        float a_phi = 0.f, ax = 0.f, ay = 0.f, az = 0.f;   // use (i, j)
        float b_phi = 0.f, bx = 0.f, by = 0.f, bz = 0.f;   // use (j, i), gradient w.r.t. u_ji
        float gd = 0.f;                                    // sum dE/df df/dd (table mode)
        int kt = 0;
        float st = 0.f;
        if constexpr (TAB) tab_locate(tf, u, kt, st);
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int c = lane + 32 * k;
            float f0, f1, f2, df0 = 0.f, df1 = 0.f, df2 = 0.f;
            if constexpr (TAB) {
                const float4 *cp = tf.coef + (int64_t)kt * 3 * F + c;
                const float4 q0 = cp[0], q1 = cp[F], q2 = cp[2 * F];
                f0 = tab_value(q0, st); f1 = tab_value(q1, st); f2 = tab_value(q2, st);
                df0 = tab_slope(q0, st, tf.inv_h); df1 = tab_slope(q1, st, tf.inv_h); df2 = tab_slope(q2, st, tf.inv_h);
            } else {
                const float *fp = fu + (int64_t)u * 3 * F + c;
                f0 = fp[0]; f1 = fp[F]; f2 = fp[2 * F];
            }
            float gi[9], gj[9];
            load_coords(gXraw, i, c, N, F, gi);
            load_coords(gXraw, j, c, N, F, gj);
            const float Zij = Ta[(int64_t)zi * F + c] + Tb[(int64_t)zj * F + c];
            const float Zji = Ta[(int64_t)zj * F + c] + Tb[(int64_t)zi * F + c];
            // use (i, j)
            const float gc0 = gi[0];
            const float gcA = gi[1] * ux + gi[2] * uy + gi[3] * uz;
            const float gcS = gi[4] * bxx + gi[5] * byy + gi[6] * bxy + gi[7] * bxz + gi[8] * byz;
            a_phi = fmaf(Zij, gc0 * f0 + gcA * f1 + gcS * f2, a_phi);
            {
                const float cA = phi * Zij * f1, cS = phi * Zij * f2;
                ax += cA * gi[1] + cS * (2.f * ux * gi[4] + uy * gi[6] + uz * gi[7]);
                ay += cA * gi[2] + cS * (2.f * uy * gi[5] + ux * gi[6] + uz * gi[8]);
                az += cA * gi[3] + cS * (ux * gi[7] + uy * gi[8]);
            }
            // use (j, i): v = -u, the S basis is even in u
            const float vx = -ux, vy = -uy, vz = -uz;
            const float hc0 = gj[0];
            const float hcA = gj[1] * vx + gj[2] * vy + gj[3] * vz;
            const float hcS = gj[4] * bxx + gj[5] * byy + gj[6] * bxy + gj[7] * bxz + gj[8] * byz;
            b_phi = fmaf(Zji, hc0 * f0 + hcA * f1 + hcS * f2, b_phi);
            {
                const float cA = phi * Zji * f1, cS = phi * Zji * f2;
                bx += cA * gj[1] + cS * (2.f * vx * gj[4] + vy * gj[6] + vz * gj[7]);
                by += cA * gj[2] + cS * (2.f * vy * gj[5] + vx * gj[6] + vz * gj[8]);
                bz += cA * gj[3] + cS * (vx * gj[7] + vy * gj[8]);
            }
            const float o0 = phi * (Zij * gc0 + Zji * hc0);
            const float o1 = phi * (Zij * gcA + Zji * hcA);
            const float o2 = phi * (Zij * gcS + Zji * hcS);
            const int64_t ob = (int64_t)u * 3 * F + c;
            if constexpr (TAB) {   // no projection weights to go back through
                gd += o0 * df0 + o1 * df1 + o2 * df2;
            } else {
                gfu[ob] = o0;
                gfu[ob + F] = o1;
                gfu[ob + 2 * F] = o2;
                opcopy_store(gfu_cp, ob, o0);
                opcopy_store(gfu_cp, ob + F, o1);
                opcopy_store(gfu_cp, ob + 2 * F, o2);
            }
        }
        a_phi = warp_sum(a_phi); ax = warp_sum(ax); ay = warp_sum(ay); az = warp_sum(az);
        b_phi = warp_sum(b_phi); bx = warp_sum(bx); by = warp_sum(by); bz = warp_sum(bz);
        if constexpr (TAB) gd = warp_sum(gd);
        if (lane == 0) {
            if constexpr (TAB) dEdd[u] += gd;
            const int e = ue[u];
            edge_g[e] = make_float4(a_phi, ax, ay, az);
            edge_g[rev[e]] = make_float4(b_phi, bx, by, bz);
        }
    }
}

// The same adjoint with four consecutive channels per lane (F = 128, exact
// mode, forces only), and both uses of the pair taken together: with
// q = Z_ij g_i +- Z_ji g_j per coordinate (minus for the skew part, which is
// odd in u), dE/df = phi (q basis), and one sum per pair serves dE/dphi and
// dE/du of the two uses, which enter the forces only as their sum and their
// difference:
//   pair_g[u] = (dE/dphi(i,j) + dE/dphi(j,i), dE/du(i,j) - dE/du(j,i)).
// 48 operations per channel instead of 110, two channels per instruction.
// Warps take runs of consecutive pairs, which share their first atom: row i of
// gX_raw and its table rows stay in registers until i changes, so a pair
// gathers only row j.  The runs go round the warps, so the pairs in flight
// sweep the atoms together and the gathered rows stay in L2 (one long run per
// warp: 2.77 ms against 2.06).  Row j and f come through a ring in shared
// memory, two pairs ahead (in registers, without the ring: 2.06 against 1.52;
// three pairs ahead at three blocks: 1.66): what bounds it is the latency of
// the gathers against the bytes under way (6.1 KB a pair through L2), then f
// and dE/df in HBM.  96,000-atom water (2.58 M pairs): 3.04 -> 1.52 ms; 3,000
// atoms 105 -> 50 us.  Offsets are 32-bit (the host checks the sizes).
constexpr int kPairRun = 32;       // consecutive pairs a warp takes at a time
constexpr int kPairBlocks = 4;     // resident blocks per SM, and the grid: one wave
constexpr int kPairDepth = 2;      // pairs under way per warp
constexpr int kPairBytes = 12 * 128 * 4;
struct F4 {  // four FP32 values as two packed pairs
    uint64_t v[2];
};
__device__ __forceinline__ F4 ld4p(const float *__restrict__ p) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
    return F4{{t.x, t.y}};
}
template <int F>
__global__ void __launch_bounds__(128, kPairBlocks) k_emb_bwd_pairs_v4(const float4 *__restrict__ geo,
                                                          const int32_t *__restrict__ z,
                                                          const int2 *__restrict__ uij,
                                                          const int32_t *__restrict__ nu, int N, int max_z,
                                                          const float *__restrict__ fu, const float *__restrict__ Ta,
                                                          const float *__restrict__ Tb,
                                                          const float *__restrict__ gXraw, float *__restrict__ gfu,
                                                          float4 *__restrict__ pair_g) {
    pdl_entry();
    static_assert(F == 128, "one float4 per lane and row");
    extern __shared__ __align__(128) uint8_t pair_ring[];
    const int lane = threadIdx.x & 31;
    const int U = *nu;
    const uint32_t c4 = 4u * lane;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t share = (U + warps - 1) / warps;
    // equal runs of at most kPairRun pairs
    const int64_t rounds = (share + kPairRun - 1) / kPairRun;
    const int per = (int)(rounds > 0 ? (share + rounds - 1) / rounds : 1);
    int cur = -1;
    F4 gi[9], tai, tbi;
    auto elem = [&](int a) {
        const int q = z[a];
        return (q < 0 || q >= max_z) ? 0 : q;
    };
    // gX_raw_j and f of a pair through the lane's own places of a ring, kPairDepth
    // pairs ahead (each lane copies what it will read: no barrier)
    uint8_t *ring = pair_ring + (threadIdx.x >> 5) * kPairDepth * kPairBytes + 16 * lane;
    auto fetch = [&](int64_t u, int j, int place) {
        uint8_t *d = ring + place * kPairBytes;
        const float *f = fu + u * 3 * F + c4, *h = gXraw + (int64_t)j * F + c4;
        const float *hA = gXraw + ((int64_t)N + 3LL * j) * F + c4, *hS = gXraw + (4LL * N + 5LL * j) * F + c4;
        cp_lane<16>(d, h);
#pragma unroll
        for (int q = 0; q < 3; ++q) cp_lane<16>(d + (1 + q) * F * 4, hA + q * F);
#pragma unroll
        for (int q = 0; q < 5; ++q) cp_lane<16>(d + (4 + q) * F * 4, hS + q * F);
#pragma unroll
        for (int q = 0; q < 3; ++q) cp_lane<16>(d + (9 + q) * F * 4, f + q * F);
    };
    auto use = [&](int u, int i, int zj_, const float4 gu, int place) {
        F4 h[9], f[3];
#pragma unroll
        for (int q = 0; q < 9; ++q) h[q] = ld4p(reinterpret_cast<const float *>(ring + place * kPairBytes + q * F * 4));
#pragma unroll
        for (int q = 0; q < 3; ++q) f[q] = ld4p(reinterpret_cast<const float *>(ring + place * kPairBytes + (9 + q) * F * 4));
        if (i != cur) {  // the same in every lane
            cur = i;
            const uint32_t zi = (uint32_t)elem(cur) * F + c4;
            tai = ld4p(Ta + zi);
            tbi = ld4p(Tb + zi);
#pragma unroll
            for (int q = 0; q < 9; ++q) gi[q] = ld4p(gXraw + coord_row(q, (uint32_t)cur, (uint32_t)N, F) + c4);
        }
        const uint32_t zj = (uint32_t)zj_ * F + c4;
        const uint32_t fb = (uint32_t)u * 3u * F + c4;
        const F4 taj = ld4p(Ta + zj), tbj = ld4p(Tb + zj);
        const float ux = gu.x, uy = gu.y, uz = gu.z;
        auto dup = [](float x) { return f2_pack(x, x); };
        const uint64_t x2 = dup(ux), y2 = dup(uy), z2 = dup(uz), xx2 = dup(2.f * ux), yy2 = dup(2.f * uy);
        const uint64_t bxx = dup(ux * ux - (1.0f / 3.0f)), byy = dup(uy * uy - (1.0f / 3.0f));
        const uint64_t bxy = dup(ux * uy), bxz = dup(ux * uz), byz = dup(uy * uz);
        const uint64_t ph2 = dup(gu.w), neg = dup(-1.f);
        uint64_t sp = 0, sx = 0, sy = 0, sz = 0;
        F4 o[3];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint64_t zij = f2_add(tai.v[k], tbj.v[k]), zji = f2_add(taj.v[k], tbi.v[k]);
            const uint64_t nji = f2_mul(zji, neg);
            uint64_t q[9];
#pragma unroll
            for (int c = 0; c < 9; ++c)
                q[c] = f2_fma((c >= 1 && c < 4) ? nji : zji, h[c].v[k], f2_mul(zij, gi[c].v[k]));
            const uint64_t q1 = f2_fma(z2, q[3], f2_fma(y2, q[2], f2_mul(x2, q[1])));
            const uint64_t q2 = f2_fma(byz, q[8], f2_fma(bxz, q[7], f2_fma(bxy, q[6], f2_fma(byy, q[5], f2_mul(bxx, q[4])))));
            sp = f2_fma(f[2].v[k], q2, f2_fma(f[1].v[k], q1, f2_fma(f[0].v[k], q[0], sp)));
            const uint64_t dx = f2_fma(z2, q[7], f2_fma(y2, q[6], f2_mul(xx2, q[4])));
            const uint64_t dy = f2_fma(z2, q[8], f2_fma(x2, q[6], f2_mul(yy2, q[5])));
            const uint64_t dz = f2_fma(y2, q[8], f2_mul(x2, q[7]));
            sx = f2_fma(f[2].v[k], dx, f2_fma(f[1].v[k], q[1], sx));
            sy = f2_fma(f[2].v[k], dy, f2_fma(f[1].v[k], q[2], sy));
            sz = f2_fma(f[2].v[k], dz, f2_fma(f[1].v[k], q[3], sz));
            o[0].v[k] = f2_mul(ph2, q[0]);
            o[1].v[k] = f2_mul(ph2, q1);
            o[2].v[k] = f2_mul(ph2, q2);
        }
#pragma unroll
        for (int pl = 0; pl < 3; ++pl)
            *reinterpret_cast<ulonglong2 *>(gfu + fb + pl * F) = make_ulonglong2(o[pl].v[0], o[pl].v[1]);
        // four warp sums in six exchanges: each step halves the values a lane
        // carries, so lanes 0, 8, 16, 24 end with one sum each
        auto fold = [](uint64_t v) {
            const float2 t = f2_unpack(v);
            return t.x + t.y;
        };
        float a0 = fold(sp), a1 = fold(sx), a2 = fold(sy), a3 = fold(sz);
        const bool hi = lane & 16, hj = lane & 8;
        const float r0 = __shfl_xor_sync(0xffffffffu, hi ? a0 : a2, 16), r1 = __shfl_xor_sync(0xffffffffu, hi ? a1 : a3, 16);
        a0 = (hi ? a2 : a0) + r0;
        a1 = (hi ? a3 : a1) + r1;
        const float r2 = __shfl_xor_sync(0xffffffffu, hj ? a0 : a1, 8);
        a0 = (hj ? a1 : a0) + r2;
        a0 += __shfl_xor_sync(0xffffffffu, a0, 4);
        a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
        a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
        if ((lane & 7) == 0)
            reinterpret_cast<float *>(pair_g)[4LL * u + (lane >> 3)] = lane == 0 ? a0 : gu.w * a0;
    };
    for (int64_t u0 = wid * per; u0 < U; u0 += warps * per) {
        const int u_end = (int)(u0 + per < U ? u0 + per : U);
        // the run's pairs, one per lane
        const int n = u_end - (int)u0;
        int2 p = make_int2(0, 0);
        float4 gl = make_float4(0.f, 0.f, 0.f, 0.f);
        int zl = 0;
        if (lane < n) {
            p = uij[u0 + lane];
            gl = geo[u0 + lane];
            zl = elem(p.y);
        }
#pragma unroll
        for (int d = 0; d < kPairDepth; ++d) {
            if (d < n) fetch(u0 + d, __shfl_sync(0xffffffffu, p.y, d), d);
            cp_commit();
        }
        int place = 0;
        for (int k = 0; k < n; ++k) {
            const float4 gu = make_float4(__shfl_sync(0xffffffffu, gl.x, k), __shfl_sync(0xffffffffu, gl.y, k),
                                          __shfl_sync(0xffffffffu, gl.z, k), __shfl_sync(0xffffffffu, gl.w, k));
            const int i = __shfl_sync(0xffffffffu, p.x, k), zj = __shfl_sync(0xffffffffu, zl, k);
            const int jn = __shfl_sync(0xffffffffu, p.y, k + kPairDepth < n ? k + kPairDepth : 0);
            cp_wait<kPairDepth - 1>();  // one copy group per pair: the oldest has landed
            use((int)u0 + k, i, zj, gu, place);
            if (k + kPairDepth < n) fetch(u0 + k + kPairDepth, jn, place);
            cp_commit();
            place = place + 1 == kPairDepth ? 0 : place + 1;
        }
        cp_wait<0>();
    }
}

// dE/dr_ij of each undirected pair (i < j): one warp per pair, lane k < K.
//   dE/dd   = sum_k ge[u][k] de_k/dd + (gphi_mlp[u] + gphi(i,j) + gphi(j,i)) dphi/dd
//             + dEdd[u]  (the tabulated functions' share, table mode)
//   dE/du   = gu(i,j) - gu(j,i)                       (u_ji = -u_ij)
// (both from edge_g, or already taken together from pair_g)
//   Gp[u]   = dE/dd u + (dE/du - (dE/du . u) u) / d
__global__ void k_pair_vec(const float *__restrict__ pos, const float *__restrict__ box,
                           const int32_t *__restrict__ batch, const int2 *__restrict__ uij,
                           const int32_t *__restrict__ ue, const int32_t *__restrict__ rev,
                           const int32_t *__restrict__ nu, RadialParams rp, const float *__restrict__ ge,
                           const float *__restrict__ gphi_mlp, int64_t gphi_stride, const float4 *__restrict__ edge_g,
                           const float4 *__restrict__ pair_g, const float *__restrict__ dEdd,
                           float *__restrict__ Gp) {
    pdl_entry();
    const int U = *nu;
    // one thread per pair (a warp keeps 32 pairs' loads in flight); the
    // pair's row of dE/de is read as float4 when K allows
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < U; u += (int64_t)gridDim.x * blockDim.x) {
        const int2 p = uij[u];
        float x, y, zz;
        pair_vec(pos, box, batch, p.x, p.y, x, y, zz);
        const float d = sqrtf(norm2_rn(x, y, zz));
        const float phi = cutoff_phi(d, rp), dphi = cutoff_dphi(d, rp);
        float s = 0.f;
        if (ge) {
            const float *g = ge + u * rp.K;
            if ((rp.K & 3) == 0) {
                for (int k = 0; k < rp.K; k += 4) {
                    const float4 gv = *reinterpret_cast<const float4 *>(g + k);
                    const float gk[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float e, de;
                        expnorm_k(d, k + j, rp, phi, dphi, e, de);
                        s = fmaf(gk[j], de, s);
                    }
                }
            } else {
                for (int k = 0; k < rp.K; ++k) {
                    float e, de;
                    expnorm_k(d, k, rp, phi, dphi, e, de);
                    s = fmaf(g[k], de, s);
                }
            }
        }
        {
            float4 g;
            if (pair_g) {
                g = pair_g[u];
            } else {
                const int e = ue[u];
                const float4 a = edge_g[e], b = edge_g[rev[e]];
                g = make_float4(a.x + b.x, a.y - b.y, a.z - b.z, a.w - b.w);
            }
            const float gphi = (gphi_mlp ? gphi_mlp[u] + gphi_mlp[u + gphi_stride] : 0.f) + g.x;
            const float gd = s + gphi * dphi + (dEdd ? dEdd[u] : 0.f);
            const float inv = 1.0f / d;
            const float ux = x * inv, uy = y * inv, uz = zz * inv;
            const float gx = g.y, gy = g.z, gz = g.w;
            const float dot = gx * ux + gy * uy + gz * uz;
            Gp[3 * u] = gd * ux + (gx - dot * ux) * inv;
            Gp[3 * u + 1] = gd * uy + (gy - dot * uy) * inv;
            Gp[3 * u + 2] = gd * uz + (gz - dot * uz) * inv;
        }
    }
}

// F_i = -dE/dr_i = -sum over the active edges of row i of +-Gp[pair]
// (+ when i is the pair's first atom, r_ij = r_i - r_j), in row order, so the
// inactive edges of a skin list change nothing.  Eight lanes per atom load
// eight edges at a time and then add them up one after the other; a thread per
// atom spent its time on one chain of dependent loads (12 us at any size up to
// a few thousand atoms, 9 now).
constexpr int kForceLanes = 8;
__global__ void k_forces(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                         const int32_t *__restrict__ pair_of, const float *__restrict__ Gp, int N,
                         float *__restrict__ forces) {
    pdl_entry();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int i = (int)(t / kForceLanes), sub = (int)(t % kForceLanes);
    const unsigned group = 0xffu << (threadIdx.x & 24);
    if (i >= N) return;  // whole groups
    float fx = 0.f, fy = 0.f, fz = 0.f;
    const int e1 = row_ptr[i + 1];
    for (int e0 = row_ptr[i]; e0 < e1; e0 += kForceLanes) {
        const int e = e0 + sub;
        float gx = 0.f, gy = 0.f, gz = 0.f;
        if (e < e1) {
            const int u = pair_of[e];
            if (u >= 0) {
                const float sgn = col[e] > i ? 1.0f : -1.0f;
                gx = sgn * Gp[3LL * u];
                gy = sgn * Gp[3LL * u + 1];
                gz = sgn * Gp[3LL * u + 2];
            }
        }
#pragma unroll
        for (int k = 0; k < kForceLanes; ++k) {
            fx += __shfl_sync(group, gx, k, kForceLanes);
            fy += __shfl_sync(group, gy, k, kForceLanes);
            fz += __shfl_sync(group, gz, k, kForceLanes);
        }
    }
    if (sub == 0) {
        forces[3LL * i] = -fx;
        forces[3LL * i + 1] = -fy;
        forces[3LL * i + 2] = -fz;
    }
}

// Per-element sums of the pair-embedding adjoints (split over atom ranges):
// zpart[s][0][z][c] = sum_{i in split s, z_i = z} gA_atom[i][c], and [1] for gB.
__global__ void k_group_z(const int32_t *__restrict__ z, const float *__restrict__ gA,
                          const float *__restrict__ gB, int N, int F, int max_z, int splits,
                          float *__restrict__ zpart) {
    pdl_entry();
    const int zz = blockIdx.x, s = blockIdx.y, c = threadIdx.x;
    const int chunk = (N + splits - 1) / splits;
    const int i0 = s * chunk, i1 = min(N, i0 + chunk);
    float a = 0.f, b = 0.f;
    for (int i = i0; i < i1; ++i) {
        if (z[i] == zz) {
            a += gA[(int64_t)i * F + c];
            b += gB[(int64_t)i * F + c];
        }
    }
    zpart[(((int64_t)s * 2 + 0) * max_z + zz) * F + c] = a;
    zpart[(((int64_t)s * 2 + 1) * max_z + zz) * F + c] = b;
}

// A[z] = sum over splits of the receiver sums, B[z] likewise for senders.
__global__ void k_zreduce(const float *__restrict__ zpart, int splits, int F, int max_z, float *__restrict__ AB) {
    pdl_entry();
    const int zz = blockIdx.x, c = threadIdx.x;
    for (int h = 0; h < 2; ++h) {
        float acc = 0.f;
        for (int s = 0; s < splits; ++s) acc += zpart[(((int64_t)s * 2 + h) * max_z + zz) * F + c];
        AB[((int64_t)h * max_z + zz) * F + c] = acc;
    }
}

// Gradients of the atom embedding and the pair embedding Linear from the
// per-element sums A[z] (receiver) and B[z] (sender), Z_ij = W_e[emb_zi; emb_zj] + b_e.
// Blocks 0..F-1 give rows of dW_e (and db_e), blocks F..F+max_z-1 rows of demb.
__global__ void k_emb_tables_grad2(const float *__restrict__ AB, int F, int max_z, const float *__restrict__ emb,
                                   const float *__restrict__ We, float *__restrict__ g_emb,
                                   float *__restrict__ g_We, float *__restrict__ g_be) {
    pdl_entry();
    const int r = blockIdx.x, c = threadIdx.x;
    const float *A = AB, *B = AB + (int64_t)max_z * F;
    if (r < F) {
        // g_We[r][c] = sum_z A[z][r] emb[z][c];  g_We[r][F + c] = sum_z B[z][r] emb[z][c]
        float a = 0.f, b = 0.f;
        for (int zz = 0; zz < max_z; ++zz) {
            const float e = emb[(int64_t)zz * F + c];
            a = fmaf(A[(int64_t)zz * F + r], e, a);
            b = fmaf(B[(int64_t)zz * F + r], e, b);
        }
        g_We[(int64_t)r * 2 * F + c] = a;
        g_We[(int64_t)r * 2 * F + F + c] = b;
        if (r == 0) {
            float bb = 0.f;
            for (int zz = 0; zz < max_z; ++zz) bb += A[(int64_t)zz * F + c];
            g_be[c] = bb;
        }
    } else {
        // g_emb[z][c] = sum_r A[z][r] We[r][c] + B[z][r] We[r][F + c]
        const int zz = r - F;
        float a = 0.f;
        for (int q = 0; q < F; ++q)
            a += A[(int64_t)zz * F + q] * We[(int64_t)q * 2 * F + c] + B[(int64_t)zz * F + q] * We[(int64_t)q * 2 * F + F + c];
        g_emb[(int64_t)zz * F + c] = a;
    }
}

// dE/dE_i (seed of the system) and its products for the head gradients
__global__ void k_seed_atoms(const float *__restrict__ seed, const int32_t *__restrict__ batch, int N,
                             float *__restrict__ gEi) {
    pdl_entry();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) gEi[i] = seed ? seed[batch ? batch[i] : 0] : 1.0f;
}

// What a call makes of its weights before the first layer, in one launch: job
// j reads a [rows][cols] float matrix and writes a bf16 copy (mode 1), its
// TF32 split hi + lo (mode 2, the 3xTF32 GEMMs) or an FP32 copy (mode 3),
// transposed when tr[j] (backward operands).  perm[j] = F > 0: row p*F + c of
// the result is row c*3 + p of the source (the last radial layer, whose blob
// order is channel-major), so the per-pair filters g_ij and their adjoints are
// three contiguous F-channel planes I, A, S and the message kernels read and
// write them coalesced.  32 x 32 tiles through shared memory, so a transposed
// matrix is read and written along its rows.  The blocks past the jobs form
// the element tables (see elem_tables).
// Latency-bound; as three launches (filter rows, weight copies, tables with
// one block per element) 57 us a call at F = 128, now 10.
// at most 16 per layer (two filter copies, ten operands, two of them by class)
// of at most 8 layers, 4 + 2 + 8 beside them
constexpr int kMaxCvtJobs = 144;
static_assert(8 * 16 + 14 <= kMaxCvtJobs, "conversion jobs");
constexpr int kElemParts = 8;  // blocks per element
struct CvtJobs {
    const float *src[kMaxCvtJobs];
    void *hi[kMaxCvtJobs];
    void *lo[kMaxCvtJobs];
    int rows[kMaxCvtJobs], cols[kMaxCvtJobs];
    short perm[kMaxCvtJobs];
    signed char tr[kMaxCvtJobs], mode[kMaxCvtJobs];
    int n;
};
struct ElemTables {
    const float *emb, *W, *b;
    int F, max_z;
    float *Ta, *Tb;
};
struct WOp {  // a weight operand: bf16 matrix, or fp32 high part + residual
    const void *b;
    const void *blo;
};
__global__ void __launch_bounds__(256) k_prep_weights(const __grid_constant__ CvtJobs J, ElemTables E) {
    pdl_entry();
    __shared__ float tile[32][33];
    const int j = blockIdx.y;
    if (j >= J.n) {
        const int q = (j - J.n) * gridDim.x + blockIdx.x;
        if (q / kElemParts < E.max_z)
            elem_tables(q / kElemParts, q % kElemParts, kElemParts, E.emb, E.W, E.b, E.F, E.Ta, E.Tb);
        return;
    }
    const int R = J.rows[j], C = J.cols[j], pf = J.perm[j];
    const int tc = (C + 31) / 32, tiles = ((R + 31) / 32) * tc;
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    auto put = [&](int64_t o, float v) {
        if (J.mode[j] == 1) {
            static_cast<__nv_bfloat16 *>(J.hi[j])[o] = __float2bfloat16_rn(v);
        } else if (J.mode[j] == 3) {
            static_cast<float *>(J.hi[j])[o] = v;
        } else {
            float hi, lo;
            tf32_split(v, hi, lo);
            static_cast<float *>(J.hi[j])[o] = hi;
            static_cast<float *>(J.lo[j])[o] = lo;
        }
    };
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int r0 = (t / tc) * 32, c0 = (t % tc) * 32;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = r0 + row + 8 * k, c = c0 + lane;
            if (r < R && c < C) {
                const int sr = pf > 0 ? (r % pf) * 3 + r / pf : r;
                const float v = J.src[j][(int64_t)sr * C + c];
                if (J.tr[j]) tile[row + 8 * k][lane] = v;
                else put((int64_t)r * C + c, v);
            }
        }
        if (!J.tr[j]) continue;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + row + 8 * k, r = r0 + lane;
            if (r < R && c < C) put((int64_t)c * R + r, tile[lane][row + 8 * k]);
        }
    }
}

// FP32 plane-major copies of a layer's last radial weight and bias
static void filter_row_jobs(CvtJobs &J, const LayerW &L, int F, float *w3p, float *b3p) {
    const float *src[2] = {L.mlp3_w, L.mlp3_b};
    float *dst[2] = {w3p, b3p};
    for (int q = 0; q < 2; ++q) {
        const int j = J.n++;
        J.src[j] = src[q]; J.hi[j] = dst[q]; J.lo[j] = nullptr;
        J.rows[j] = 3 * F; J.cols[j] = q ? 1 : 2 * F; J.perm[j] = (short)F; J.tr[j] = 0; J.mode[j] = 3;
    }
}

// The tensor-core modes' weight operands, one set per call.
// WeightOps::x3 holds 3xTF32 operands: of the num_rbf-wide radial layers in
// both modes (rounding the narrow expnorm basis to bf16 costs more force
// accuracy than any other operand), and of the per-atom embedding and output
// MLPs in BF16 mode.  In the FP32-accurate mode those per-atom MLPs stay on
// FP32 FMA: they are cheap, and the energy is the quantity most sensitive to
// them (3xTF32 there costs an order of magnitude of energy accuracy).
struct LayerOps {
    WOp mlp2, mlp3, mlp2T, mlp3T, mix1, mix1T, mix2, mix2T, mlp1, mlp1T;
};
struct X3W {
    WOp dproj, dprojT, emb_mlp1, emb_mlp1T, emb_mlp2, emb_mlp2T, out, outT, head1, head1T;
};
struct WeightOps {
    LayerOps layer[8];
    WOp emix, emixT;
    X3W x3;
};
// Lays the operands out from wb and adds their jobs to J; returns the bytes
// they take (none in FP32 mode).  The workspace is sized by the same walk (wb
// NULL), so what a call lays out is what the context was given room for.
static int64_t weight_operands(const tnet_model_desc &d, const Weights &W, char *wb, CvtJobs &J, WeightOps &o) {
    o = WeightOps{};
    const int F = d.F, K = d.K, NL = d.L, H = F / 2, prec = d.precision;
    const bool tab = d.radial_table > 0;
    if (!prec) return 0;
    int64_t woff = 0;
    auto alloc = [&](int64_t elems, int esz) {
        void *p = wb ? wb + woff : nullptr;
        woff += (elems * esz + 255) & ~(int64_t)255;
        return p;
    };
    // forward operands keep the (out, in) = K-major layout; backward
    // operands are transposed
    auto job_m = [&](const float *src, int rows, int cols, int tr, int mode, int perm = 0) {
        WOp w{};
        const int esz = mode == 1 ? 2 : 4;
        void *hi = alloc((int64_t)rows * cols, esz);
        void *lo = mode == 2 ? alloc((int64_t)rows * cols, esz) : nullptr;
        J.src[J.n] = src; J.hi[J.n] = hi; J.lo[J.n] = lo;
        J.rows[J.n] = rows; J.cols[J.n] = cols; J.tr[J.n] = (signed char)tr; J.mode[J.n] = (signed char)mode;
        J.perm[J.n] = (short)perm;
        ++J.n;
        w.b = hi;
        w.blo = lo;
        return w;
    };
    auto job = [&](const float *src, int rows, int cols, int tr) { return job_m(src, rows, cols, tr, prec); };
    auto job3 = [&](const float *src, int rows, int cols, int tr) { return job_m(src, rows, cols, tr, 2); };
    // [3][F][F] -> per-class transposes; the three classes' high parts (and
    // residuals) must stay stacked contiguously [3F][F] for the GEMM
    auto job_classes_T = [&](const float *src) {
        const int64_t ff = (int64_t)F * F;
        const int esz = prec == 1 ? 2 : 4;
        char *hi = (char *)alloc(3 * ff, esz), *lo = prec == 2 ? (char *)alloc(3 * ff, esz) : nullptr;
        for (int q = 0; q < 3; ++q) {
            J.src[J.n] = src ? src + q * ff : nullptr;
            J.hi[J.n] = hi ? hi + q * ff * esz : nullptr;
            J.lo[J.n] = lo ? lo + q * ff * esz : nullptr;
            J.rows[J.n] = F; J.cols[J.n] = F; J.tr[J.n] = 1; J.mode[J.n] = (signed char)prec; J.perm[J.n] = 0;
            ++J.n;
        }
        return WOp{hi, lo};
    };
    o.emix = job(W.emb_mix_w, 3 * F, F, 0);
    o.emixT = job_classes_T(W.emb_mix_w);
    for (int l = 0; l < NL; ++l) {
        const LayerW &Lr = W.layer[l];
        LayerOps &lo = o.layer[l];
        lo.mix1 = job(Lr.mix1_w, 3 * F, F, 0);
        lo.mix1T = job_classes_T(Lr.mix1_w);
        lo.mix2 = job(Lr.mix2_w, 3 * F, F, 0);
        lo.mix2T = job_classes_T(Lr.mix2_w);
        if (tab) continue;  // no per-pair radial MLP
        lo.mlp2 = job(Lr.mlp2_w, 2 * F, F, 0);
        lo.mlp3 = job_m(Lr.mlp3_w, 3 * F, 2 * F, 0, prec, F);
        lo.mlp2T = job(Lr.mlp2_w, 2 * F, F, 1);
        lo.mlp3T = job_m(Lr.mlp3_w, 3 * F, 2 * F, 1, prec, F);
        lo.mlp1 = job3(Lr.mlp1_w, F, K, 0);
        lo.mlp1T = job3(Lr.mlp1_w, F, K, 1);
    }
    if (!tab) {
        o.x3.dproj = job3(W.dproj_w, 3 * F, K, 0);
        o.x3.dprojT = job3(W.dproj_w, 3 * F, K, 1);
    }
    if (prec == 1) {  // (see X3W)
        o.x3.emb_mlp1 = job3(W.emb_mlp1_w, 2 * F, F, 0);
        o.x3.emb_mlp1T = job3(W.emb_mlp1_w, 2 * F, F, 1);
        o.x3.emb_mlp2 = job3(W.emb_mlp2_w, 3 * F, 2 * F, 0);
        o.x3.emb_mlp2T = job3(W.emb_mlp2_w, 3 * F, 2 * F, 1);
        o.x3.out = job3(W.out_w, F, 3 * F, 0);
        o.x3.outT = job3(W.out_w, F, 3 * F, 1);
        o.x3.head1 = job3(W.head1_w, H, F, 0);
        o.x3.head1T = job3(W.head1_w, H, F, 1);
    }
    return woff;
}

int64_t weight_operand_bytes(const tnet_model_desc *d) {
    Weights W;
    weight_offsets(d, nullptr, &W);
    CvtJobs J;
    J.n = 0;
    WeightOps o;
    return weight_operands(*d, W, nullptr, J, o);
}

// Per-context kernel set-up (nothing needs opting in at present).
int tnet_kernel_setup(tnet_ctx *c) {
    (void)c;
    return TNET_OK;
}

// Tensor-core GEMM with the column tile chosen from N.
template <class Epi>
int tc_any(const tc::TcShape &P, const __nv_bfloat16 *A, int64_t a_rows, int64_t lda, const __nv_bfloat16 *B,
           int64_t b_rows, int64_t ldb, const Epi &epi, int32_t *status, cudaStream_t st, int sms, int bn = 0) {
    if (bn == 128 && P.N % 128 == 0) return tc::tc_gemm<128>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (bn == 192 && P.N % 192 == 0) return tc::tc_gemm<192>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (bn == 256 && P.N % 256 == 0) return tc::tc_gemm<256>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (P.N <= 32) return tc::tc_gemm<32>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (P.N <= 64) return tc::tc_gemm<64>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (P.N <= 128) return tc::tc_gemm<128>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (P.N % 256 == 0) return tc::tc_gemm<256>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (P.N % 192 == 0) return tc::tc_gemm<192>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    if (P.N % 128 == 0) return tc::tc_gemm<128>(P, A, a_rows, lda, B, b_rows, ldb, epi, status, st, sms);
    return TNET_ERR_ARG;
}

// Launch the thread-per-channel row kernels with 4 consecutive rows per block
// when rb >= 4 and the block fits (at most 1024 threads for the messages, 512
// for their adjoint, whose per-row staging is 37 KB at F = 128), else one.
// blocks1 is the grid the one-row-per-block launch would use.
template <int F, bool TAB, class... Args>
static void launch_message(int rb, int blocks1, cudaStream_t st, Args... args) {
    if constexpr (F * 4 <= 1024) {
        if (rb >= 4) {
            launch(k_message<F, TAB, 4>, (blocks1 + 3) / 4, F * 4, 0, st, args...);
            return;
        }
    }
    launch(k_message<F, TAB, 1>, blocks1, F, 0, st, args...);
}
template <int F, bool TAB, class... Args>
static void launch_message_bwd(int rb, int blocks1, cudaStream_t st, Args... args) {
    if constexpr (F * 4 <= 512) {
        if (rb >= 4) {
            launch(k_message_bwd<F, TAB, 4>, (blocks1 + 3) / 4, F * 4, 0, st, args...);
            return;
        }
    }
    launch(k_message_bwd<F, TAB, 1>, blocks1, F, 0, st, args...);
}

// ============================================== host-side launch sequence ===
static inline int grid_for(int64_t n, int threads, int num_sms) {
    int64_t g = (n + threads - 1) / threads;
    const int64_t cap = (int64_t)num_sms * 16;
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

#define TRY(...)                    \
    do {                            \
        int rc_ = (__VA_ARGS__);    \
        if (rc_) return rc_;        \
    } while (0)

// Radial-function tables (radial_table = n > 0): the projections f (table 0)
// and each layer's filter g (table 1 + l) as [n-1][4][3F] Hermite
// coefficients on the grid d_k = k h, h = rc/(n - 1).  f, g are functions of
// the pair distance alone (the expnorm basis, the cosine cutoff and the radial
// MLP of TensorNet Sec. 2.1.1); the chain runs in FP64 on the values and
// their d-derivatives.
int radial_tables_impl(tnet_ctx *ctx, const float *wblob, cudaStream_t st) {
    const tnet_model_desc &d = ctx->d;
    const Layout &Lw = ctx->lay;
    const int F = d.F, K = d.K, NL = d.L, nt = d.radial_table;
    const int sms = ctx->num_sms;
    if (nt <= 0) return TNET_ERR_ARG;
    Weights W;
    weight_offsets(&d, wblob, &W);
    auto f32 = [&](size_t off) { return wsp<float>(ctx, off); };
    const double rc = d.cutoff_upper, rl = d.cutoff_lower;
    RadialParams64 rp{rc, rl, 5.0 / (rc - rl), pow((2.0 / K) * (1.0 - exp(-(rc - rl))), -2.0), exp(-(rc - rl)),
                      (1.0 - exp(-(rc - rl))) / (K - 1), K};
    const double h = rc / (nt - 1);
    const int64_t per_fn = (int64_t)(nt - 1) * 4 * 3 * F;
    auto coef = [&](int j) { return reinterpret_cast<float4 *>(f32(Lw.tab) + j * per_fn); };
    const int64_t w3_per = 6LL * F * F + 3 * F;
    auto w3p = [&](int l) { return f32(Lw.w3p) + l * w3_per; };
    auto b3p = [&](int l) { return f32(Lw.w3p) + l * w3_per + 6LL * F * F; };
    if (NL > 0) {
        CvtJobs J;
        J.n = 0;
        for (int l = 0; l < NL; ++l) filter_row_jobs(J, W.layer[l], F, w3p(l), b3p(l));
        launch(k_prep_weights, dim3(64, J.n), 256, 0, st, J, ElemTables{});
        count_launch();
        TNET_LAUNCH_CHECK();
    }
    double *e_t = wsp<double>(ctx, Lw.tab_tmp), *de_t = e_t + (int64_t)nt * K, *phi_t = de_t + (int64_t)nt * K,
           *dphi_t = phi_t + nt, *h1_t = dphi_t + nt, *t1_t = h1_t + (int64_t)nt * F, *h2_t = t1_t + (int64_t)nt * F,
           *t2_t = h2_t + (int64_t)nt * 2 * F, *v_t = t2_t + (int64_t)nt * 2 * F, *dv_t = v_t + (int64_t)nt * 3 * F;
    launch(k_tab_rbf, grid_for((int64_t)nt * K, 256, sms), 256, 0, st, nt, h, rp, e_t, de_t, phi_t, dphi_t);
    count_launch();
    TNET_LAUNCH_CHECK();
    auto layer = [&](int Nout, int Kin, const double *x, const double *tx, const float *w, const float *b, int mode,
                     double *y, double *ty) {
        launch(k_tab_layer, dim3((Nout + 63) / 64, (nt + 63) / 64), 256, 0, st, nt, Nout, Kin, x, tx, w, b, mode,
               phi_t, dphi_t, y, ty);
        count_launch();
    };
    auto finish = [&](int j) {
        launch(k_tab_coef, grid_for((int64_t)(nt - 1) * 3 * F, 256, sms), 256, 0, st, nt, 3 * F, h, v_t, dv_t,
               coef(j));
        count_launch();
    };
    layer(3 * F, K, e_t, de_t, W.dproj_w, W.dproj_b, 1, v_t, dv_t);
    finish(0);
    for (int l = 0; l < NL; ++l) {
        const LayerW &Lr = W.layer[l];
        layer(F, K, e_t, de_t, Lr.mlp1_w, Lr.mlp1_b, 0, h1_t, t1_t);
        layer(2 * F, F, h1_t, t1_t, Lr.mlp2_w, Lr.mlp2_b, 0, h2_t, t2_t);
        layer(3 * F, 2 * F, h2_t, t2_t, w3p(l), b3p(l), 2, v_t, dv_t);
        finish(1 + l);
    }
    TNET_LAUNCH_CHECK();
    ctx->tab_ready = 1;
    return TNET_OK;
}

int energy_forces_impl(tnet_ctx *ctx, const float *wblob, int N, int S, const int32_t *z,
                       const float *pos, const int32_t *batch, const float *box,
                       const int32_t *row_ptr_in, const int32_t *col, const float *seed,
                       double *energy, float *forces, float *grad_w, int32_t *status,
                       cudaStream_t st) {
    const tnet_model_desc &d = ctx->d;
    const Layout &Lw = ctx->lay;
    const int F = d.F, K = d.K, NL = d.L, H = F / 2;
    // table mode: the radial functions are tabulated, which has no weight adjoint
    const int nt = d.radial_table;
    const bool tab = nt > 0;
    if (tab && grad_w) return TNET_ERR_UNSUPPORTED;
    const float th = tab ? ctx->rp.rc / (float)(nt - 1) : 0.f;
    const int sms = ctx->num_sms;
    const RadialParams rp = ctx->rp;
    const int gctas = sms * ctx->tune[T_GEMM_CTAS];
    const int bn3 = ctx->tune[T_TC_BN_3F], bn2 = ctx->tune[T_TC_BN_2F];
    const int pair_grid = sms * ctx->tune[T_PAIR_BLOCKS];
    Weights W, G;
    weight_offsets(&d, wblob, &W);
    weight_offsets(&d, grad_w, &G);
    auto gw = [](const float *p) { return const_cast<float *>(p); };
    auto f32 = [&](size_t off) { return wsp<float>(ctx, off); };
    auto i32 = [&](size_t off) { return wsp<int32_t>(ctx, off); };
    const int64_t n9 = Lw.node9;
    const int maxU = (int)Lw.maxU;
    float *wpart = f32(Lw.wpart);
    const int64_t wcap = Lw.wpart_floats;
    int32_t *sys_start = i32(Lw.sys_start), *sys_end = i32(Lw.sys_end);
    int32_t *rev = i32(Lw.rev), *pair_of = i32(Lw.pair_of), *ucnt = i32(Lw.ucnt);
    // every kernel below reads the clamped copy of the row offsets
    int32_t *row_ptr = i32(Lw.rp_safe);
    int32_t *nu = i32(Lw.nu), *ue = i32(Lw.ue);
    int2 *uij = wsp<int2>(ctx, Lw.uedge);
    float *Ta = f32(Lw.Ta), *Tb = f32(Lw.Tb);
    const int warps_grid = (int)(((int64_t)N * 32 + 255) / 256);
    // row-sum shapes for weight gradients
    auto rows1 = [&](int M_, int N_, int64_t R, const float *A, int64_t lda, const float *B, int64_t ldb,
                     const int32_t *rows_dev) {
        WgradShape P{};
        P.M = M_; P.N = N_; P.rows[0] = R; P.row0[0] = 0; P.rows_dev = rows_dev; P.rows_mul = 1;
        P.A = A; P.lda = lda; P.B = B; P.ldb = ldb; P.nclass = 1;
        return P;
    };
    auto rows3 = [&](const float *A, const float *B) {  // the I, A, S coordinate planes
        WgradShape P{};
        P.M = F; P.N = F;
        P.rows[0] = N; P.rows[1] = 3LL * N; P.rows[2] = 5LL * N;
        P.row0[0] = 0; P.row0[1] = N; P.row0[2] = 4LL * N;
        P.rows_dev = nullptr; P.rows_mul = 1;
        P.A = A; P.lda = F; P.B = B; P.ldb = F; P.nclass = 3;
        return P;
    };

    // ---- tensor-core modes: operand copies and weight copies
    //   precision 1 (BF16): bf16 operands, one MMA per k-step
    //   precision 2 (3xTF32): fp32 operands plus their TF32 residuals
    const int prec = d.precision;
    const bool tcm = prec != 0;
    const bool wg = grad_w != nullptr;
    // FP32 activations h1, h2 are read by the FP32 GEMMs and by the weight
    // gradients (the 3xTF32 GEMMs form them from a1, a2 when no weight
    // gradient is asked for); the BF16 GEMMs read only their bf16 copies
    const bool keep_h = prec != 1 || wg;
    // bf16 operand copies (BF16 mode only: the 3xTF32 GEMMs read the fp32
    // activations and form their residuals on chip)
    auto cp = [&](size_t off) { return prec == 1 ? OpCopy{(void *)(ctx->ws + off), 1} : OpCopy{nullptr, 0}; };
    // (the num_rbf-wide operands e(d) and dE/df stay FP32, so they get no copy)
    const OpCopy none{nullptr, 0};
    const OpCopy nbf = cp(Lw.nbf), eu_cp = none, ga3_cp = cp(Lw.ga3_bf), ga2_cp = cp(Lw.ga2_bf), ga1_cp = none,
                 gfu_cp = none;
    // per-layer radial-MLP activations (and their operand copies)
    const int64_t esz_cp = 2;
    // slab of layer l (one shared slab when the reverse pass recomputes them)
    const bool keep_act = !d.recompute_edges;
    auto slab = [&](int l) { return keep_act ? (int64_t)l : 0; };
    auto h1_cp = [&](int l) { return cp(Lw.h1_bf + (size_t)(slab(l) * maxU * F * esz_cp)); };
    auto h2_cp = [&](int l) { return cp(Lw.h2_bf + (size_t)(slab(l) * maxU * 2 * F * esz_cp)); };

    // ---- graph prep
    ProfSeq pf(ctx, st);
    pf.mark(P_PREP);
    const int64_t w3_per = 6LL * F * F + 3 * F;
    auto w3p = [&](int l) { return f32(Lw.w3p) + l * w3_per; };  // plane-major mlp3 weight
    auto b3p = [&](int l) { return f32(Lw.w3p) + l * w3_per + 6LL * F * F; };
    CvtJobs J;
    J.n = 0;
    if (!tab)
        for (int l = 0; l < NL; ++l) filter_row_jobs(J, W.layer[l], F, w3p(l), b3p(l));
    WeightOps wo;
    if (weight_operands(d, W, ctx->ws + Lw.wbf, J, wo) > Lw.wbf_bytes || J.n > kMaxCvtJobs) return TNET_ERR_WORKSPACE;
    const LayerOps *lb = wo.layer;
    const X3W &wx = wo.x3;
    const bool atom_x3 = prec == 1;  // per-atom MLPs on 3xTF32
    const WOp emix = wo.emix, emixT = wo.emixT;
    {
        const ElemTables et{W.emb, W.emb2_w, W.emb2_b, F, d.max_z, Ta, Tb};
        const int extra = (d.max_z * kElemParts + 63) / 64;  // grid rows of the element tables
        launch(k_prep_weights, dim3(64, J.n + extra), 256, 0, st, J, et);
        count_launch();
        TNET_LAUNCH_CHECK();
    }
    // 3xTF32 tensor-core GEMM: fp32 A (split in the kernel) against weight
    // operand w (its TF32 split)
    auto tcx3 = [&](const tc::TcShape &P, const float *A32, int64_t a_rows, int64_t lda, const WOp &w,
                    int64_t b_rows, int64_t ldb, const auto &epi, int bn = 0) -> int {
        const tc::TcOperands o{A32, w.b, w.blo, a_rows, lda, b_rows, ldb};
        if (P.N <= 32) return tc::tc_gemm_ops<32, true>(P, o, epi, status, st, sms);
        if (P.N <= 64) return tc::tc_gemm_ops<64, true>(P, o, epi, status, st, sms);
        // num_rbf-deep GEMMs (radial layer 1, the projections) are bound by
        // their epilogue, not their MMAs: they keep sixteen epilogue warps
        if (P.K <= 32) {
            if (P.N % 192 == 0 && bn != 128) return tc::tc_gemm_ops<192, true, true>(P, o, epi, status, st, sms);
            return tc::tc_gemm_ops<128, true, true>(P, o, epi, status, st, sms);
        }
        // 2F-wide outputs: one 256-wide tile when the knob asks for it (fewer
        // tile loads per MMA: 40 KB of TMA per 880 MMA cycles against 24 KB per
        // 440 at 128)
        if (P.N % 256 == 0 && bn == 256) return tc::tc_gemm_ops<256, true>(P, o, epi, status, st, sms);
        if (P.N % 192 == 0 && bn != 128) return tc::tc_gemm_ops<192, true>(P, o, epi, status, st, sms);
        return tc::tc_gemm_ops<128, true>(P, o, epi, status, st, sms);
    };
    // tensor-core GEMM of the mode: BF16 (A's bf16 copy) or 3xTF32 (A itself)
    auto tcg = [&](const tc::TcShape &P, const float *A32, const OpCopy &Acp, int64_t a_rows, int64_t lda,
                   const WOp &w, int64_t b_rows, int64_t ldb, const auto &epi, int bn = 0) -> int {
        if (prec == 1)
            return tc_any(P, (const __nv_bfloat16 *)Acp.p, a_rows, lda, (const __nv_bfloat16 *)w.b, b_rows, ldb,
                          epi, status, st, sms, bn);
        return tcx3(P, A32, a_rows, lda, w, b_rows, ldb, epi, bn);
    };
    // (sys_start, sys_end and rows_bad are adjacent in the layout)
    int32_t *rows_bad = i32(Lw.rows_bad);
    TNET_CUDA_TRY(cudaMemsetAsync(sys_start, 0, Lw.sysinfo - Lw.sys_start, st));
    launch(k_graph_rows, warps_grid, 256, 0, st, pos, box, batch, row_ptr_in, col, N, S, ctx->max_pairs, rp.rc, row_ptr,
           sys_start, sys_end, rows_bad, rev, pair_of, ucnt, status);
    count_launch();
    TNET_LAUNCH_CHECK();
    TRY(scan_exclusive_i32(ucnt, ucnt, N, i32(Lw.scan_tmp), nu, nullptr, st));
    launch(k_upper_assign, warps_grid, 256, 0, st, pos, box, batch, row_ptr, col, rev, N, rp.rc, ucnt, rows_bad, maxU,
           nu, pair_of, uij, ue);
    count_launch();
    TNET_LAUNCH_CHECK();
    float *eu = f32(Lw.eu), *phiu = f32(Lw.phiu), *fu = f32(Lw.fu);
    float4 *geo = wsp<float4>(ctx, Lw.geo);
    // table mode: function 0 is the projections f, function 1 + l layer l's
    // filter g, each [n-1][3F] float4 Hermite coefficients
    float *dist = f32(Lw.dist);
    auto tabfn = [&](int j) {
        if (!tab) return TabFn{nullptr, nullptr, 0, 0.f};
        return TabFn{reinterpret_cast<const float4 *>(f32(Lw.tab) + (int64_t)j * (nt - 1) * 4 * 3 * F), dist, nt,
                     1.0f / th};
    };
    const TabFn tf0 = tabfn(0);
    if (tab) {
        if (!ctx->tab_ready) return TNET_ERR_ARG;  // tnet_radial_tables not called
        launch(k_pair_geo, grid_for(maxU, 256, sms), 256, 0, st, pos, box, batch, uij, nu, rp, phiu, geo, dist);
        count_launch();
    } else {
        launch(k_edge_rbf, pair_grid, 256, 0, st, pos, box, batch, uij, nu, maxU, rp, eu, phiu, geo, eu_cp);
        count_launch();
    }
    TNET_LAUNCH_CHECK();
    if (!tab) {   // radial projections f^p = W^p e(d) + b^p, once per undirected pair
        // FP32 in both modes: K = num_rbf is small, and rounding the narrow
        // expnorm basis values to bf16 costs more force accuracy than any
        // other operand
        const EpiBiasAct ep{W.dproj_b, nullptr, 0, fu, 3 * F, 0, nullptr};
        if (tcm) {
            tc::TcShape tp = tc::tshape(maxU, 3 * F, K);
            tp.rows_dev = nu;
            TRY(tcx3(tp, eu, maxU, K, wx.dproj, 3 * F, K, EpiBulk{W.dproj_b, fu, 3 * F}, bn3));
        } else {
            GemmShape pp = gshape(maxU, 3 * F, K, eu, K, W.dproj_w, K);
            pp.rows_dev = nu;
            TRY(sgemm<true>(pp, ep, gctas, sms, st));
        }
    }

    // ---- embedding
    pf.mark(P_EMB_EDGE);
    float *Xraw = f32(Lw.Xraw), *Uemb = f32(Lw.Uemb), *n0 = f32(Lw.n0), *as1 = f32(Lw.as1),
          *hs1 = f32(Lw.hs1), *as2 = f32(Lw.as2), *s = f32(Lw.s), *q0 = f32(Lw.q0);
    float2 *ln0 = wsp<float2>(ctx, Lw.ln0);
    const int atom_blocks = N < sms * ctx->tune[T_ROW_BLOCKS] ? N : sms * ctx->tune[T_ROW_BLOCKS];
    // message kernels (and the pair-parallel embedding adjoint): knob 3 (or 0) =
    // the staged kernels (exact mode, F = 64 or 128, 32-bit offsets), 1 or 4 = that
    // many consecutive rows per block of F threads (one thread per channel)
    const int rows_pb = ctx->tune[T_MSG_KERNEL] == 4 ? 4 : 1;
    const bool warp_rows = (ctx->tune[T_MSG_KERNEL] == 0 || ctx->tune[T_MSG_KERNEL] == 3) && !tab &&
                           (F == 64 || F == 128) &&
                           9LL * N * F < (1LL << 31) && (int64_t)maxU * 3 * F < (1LL << 31);
#define EMB_FWD(FF)                                                                                           \
    if (tab)                                                                                                  \
        launch(k_emb_edges<FF, true>, atom_blocks, FF, 0, st, geo, z, row_ptr, col, pair_of, N, d.max_z, fu, tf0, Ta, \
                                                          Tb, Xraw, W.emb_ln_g, W.emb_ln_b, n0, ln0, q0, status, nbf); \
    else                                                                                                      \
        launch(k_emb_edges<FF, false>, atom_blocks, FF, 0, st, geo, z, row_ptr, col, pair_of, N, d.max_z, fu, tf0, Ta, \
                                                           Tb, Xraw, W.emb_ln_g, W.emb_ln_b, n0, ln0, q0, status, nbf)
    TNET_F_SWITCH(F, EMB_FWD);
#undef EMB_FWD
    count_launch();
    TNET_LAUNCH_CHECK();
    pf.mark(P_EMB_NODE);
    {
        const EpiBiasAct em1{W.emb_mlp1_b, as1, 2 * F, hs1, 2 * F, 1, nullptr};
        const EpiBiasAct em2{W.emb_mlp2_b, as2, 3 * F, s, 3 * F, 1, nullptr};
        if (atom_x3) {
            TRY(tcx3(tc::tshape(N, 2 * F, F), n0, N, F, wx.emb_mlp1, 2 * F, F, em1, bn2));
            TRY(tcx3(tc::tshape(N, 3 * F, 2 * F), hs1, N, 2 * F, wx.emb_mlp2, 3 * F, 2 * F, em2, bn3));
        } else {
            TRY(sgemm<true>(gshape(N, 2 * F, F, n0, F, W.emb_mlp1_w, F), em1, gctas, sms, st));
            TRY(sgemm<true>(gshape(N, 3 * F, 2 * F, hs1, 2 * F, W.emb_mlp2_w, 2 * F), em2, gctas, sms, st));
        }
    }
    if (tcm) TRY(tcg(tc::tshape_classes(N, F), Xraw, nbf, 9LL * N, F, emix, 3 * F, F, EpiBulk{nullptr, Uemb, F}));
    else TRY(sgemm<true>(gshape_classes(N, F, Xraw, W.emb_mix_w), EpiStore{Uemb, F, 0}, gctas, sms, st));
    const int ew = grid_for((int64_t)N * F, 256, sms);
    float *Xfin = f32(Lw.Xfin);  // the output model's input
    launch(k_emb_scale, ew, 256, 0, st, Uemb, s, N, F, Xfin, NL > 0 ? f32(Lw.qn) : nullptr, f32(Lw.Xn), nbf);
    count_launch();
    TNET_LAUNCH_CHECK();

    // ---- interaction layers
    // layer l's radial-MLP activations: [maxU][width] slabs
    auto act = [&](size_t off, int width, int l) { return f32(off) + slab(l) * maxU * width; };
    // The radial MLP of layer l over the undirected pairs.  Its last layer
    // stores only the pre-activation a3: the message kernels form the filter
    // g = phi SiLU(a3) themselves.  fwd_only (the forward pass when the reverse
    // pass recomputes the activations): a1 and a2 are not stored, since only
    // the reverse pass reads them.
    auto edge_mlp = [&](int l, bool fwd_only) -> int {
        const LayerW &Lr = W.layer[l];
        float *a1 = act(Lw.a1, F, l), *h1 = act(Lw.h1, F, l), *a2 = act(Lw.a2, 2 * F, l),
              *h2 = act(Lw.h2, 2 * F, l), *a3 = act(Lw.a3, 3 * F, l);
        if (tab) return TNET_OK;  // the message kernels evaluate g, dg/dd from the table
        const EpiBiasAct e3{b3p(l), a3, 3 * F, nullptr, 3 * F, 0, nullptr};
        const EpiBulk t3e{b3p(l), a3, 3 * F};
        if (tcm && prec == 2 && !wg) {
            // 3xTF32 without weight gradients: layers 1 and 2 store their
            // pre-activations alone; the next GEMM's converter warps form
            // h = silu_f(a) from them (bitwise the value the epilogue would
            // store), and the reverse pass reads only a1, a2
            const EpiBulk s1{Lr.mlp1_b, a1, F}, s2{Lr.mlp2_b, a2, 2 * F};
            tc::TcShape t1 = tc::tshape(maxU, F, K), t2 = tc::tshape(maxU, 2 * F, F), t3 = tc::tshape(maxU, 3 * F, 2 * F);
            t1.rows_dev = t2.rows_dev = t3.rows_dev = nu;
            t2.a_silu = t3.a_silu = 1;
            pf.mark(P_MLP1);
            TRY(tcx3(t1, eu, maxU, K, lb[l].mlp1, F, K, s1));
            pf.mark(P_MLP2);
            TRY(tcx3(t2, a1, maxU, F, lb[l].mlp2, 2 * F, F, s2, bn2));
            pf.mark(P_MLP3);
            TRY(tcx3(t3, a2, maxU, 2 * F, lb[l].mlp3, 3 * F, 2 * F, t3e, bn3));
            return TNET_OK;
        }
        const EpiBiasAct e1{Lr.mlp1_b, fwd_only ? nullptr : a1, F, keep_h ? h1 : nullptr, F, 1, nullptr, h1_cp(l), F};
        const EpiBiasAct e2{Lr.mlp2_b, fwd_only ? nullptr : a2, 2 * F, keep_h ? h2 : nullptr, 2 * F, 1, nullptr,
                            h2_cp(l), 2 * F};
        if (tcm) {
            tc::TcShape t2 = tc::tshape(maxU, 2 * F, F), t3 = tc::tshape(maxU, 3 * F, 2 * F);
            t2.rows_dev = t3.rows_dev = nu;
            pf.mark(P_MLP1);  // K = num_rbf: 3xTF32 in both modes (see the projections above)
            tc::TcShape t1 = tc::tshape(maxU, F, K);
            t1.rows_dev = nu;
            TRY(tcx3(t1, eu, maxU, K, lb[l].mlp1, F, K, e1));
            pf.mark(P_MLP2);
            TRY(tcg(t2, h1, h1_cp(l), maxU, F, lb[l].mlp2, 2 * F, F, e2, bn2));
            pf.mark(P_MLP3);
            TRY(tcg(t3, h2, h2_cp(l), maxU, 2 * F, lb[l].mlp3, 3 * F, 2 * F, t3e, bn3));
            return TNET_OK;
        }
        pf.mark(P_MLP1);
        GemmShape p1 = gshape(maxU, F, K, eu, K, Lr.mlp1_w, K);
        p1.rows_dev = nu;
        TRY(sgemm<true>(p1, e1, gctas, sms, st));
        pf.mark(P_MLP2);
        GemmShape p2 = gshape(maxU, 2 * F, F, h1, F, Lr.mlp2_w, F);
        p2.rows_dev = nu;
        TRY(sgemm<true>(p2, e2, gctas, sms, st));
        pf.mark(P_MLP3);
        GemmShape p3 = gshape(maxU, 3 * F, 2 * F, h2, 2 * F, w3p(l), 2 * F);
        p3.rows_dev = nu;
        TRY(sgemm<true>(p3, e3, gctas, sms, st));
        return TNET_OK;
    };
    for (int l = 0; l < NL; ++l) {
        float *Xn = f32(Lw.Xn) + l * n9;
        float *Y = f32(Lw.Y) + l * n9, *M = f32(Lw.M) + l * n9, *Tn = f32(Lw.Tn) + l * n9,
              *dX = f32(Lw.dX) + l * n9;
        pf.mark(P_NODE_MIX);
        if (tcm) TRY(tcg(tc::tshape_classes(N, F), Xn, nbf, 9LL * N, F, lb[l].mix1, 3 * F, F, EpiBulk{nullptr, Y, F}));
        else TRY(sgemm<true>(gshape_classes(N, F, Xn, W.layer[l].mix1_w), EpiStore{Y, F, 0}, gctas, sms, st));
        TRY(edge_mlp(l, !keep_act));
        pf.mark(P_MESSAGE);
        const float *a3l = act(Lw.a3, 3 * F, l);
#define MSG_FWD(FF)                                                                                          \
    if (tab) launch_message<FF, true>(rows_pb, atom_blocks, st, row_ptr, col, pair_of, a3l, phiu, tabfn(1 + l), Y, \
                                      N, M);                                                                 \
    else launch_message<FF, false>(rows_pb, atom_blocks, st, row_ptr, col, pair_of, a3l, phiu, tabfn(1 + l), Y, \
                                   N, M)
        auto staged = [&](auto channels) -> int {
            return message_tile<decltype(channels)::value, false>(sms, st, row_ptr, col, pair_of, a3l, phiu, Y, nullptr,
                                                                  N, M, none, nullptr, none, nullptr, 0, status);
        };
        if (warp_rows) TRY(F == 64 ? staged(Channels<64>{}) : staged(Channels<128>{}));
        else {
            TNET_F_SWITCH(F, MSG_FWD);
        }
#undef MSG_FWD
        count_launch();
        pf.mark(P_NODE_ELEM);
        launch(k_node_update, ew, 256, 0, st, Y, M, N, F, Tn, nbf);
        count_launch();
        TNET_LAUNCH_CHECK();
        pf.mark(P_NODE_MIX);
        if (tcm) TRY(tcg(tc::tshape_classes(N, F), Tn, nbf, 9LL * N, F, lb[l].mix2, 3 * F, F, EpiBulk{nullptr, dX, F}));
        else TRY(sgemm<true>(gshape_classes(N, F, Tn, W.layer[l].mix2_w), EpiStore{dX, F, 0}, gctas, sms, st));
        if (l + 1 < NL) {  // (the last layer's residual is formed by k_out_norms)
            pf.mark(P_NODE_ELEM);
            launch(k_residual, ew, 256, 0, st, Xn, dX, N, F, f32(Lw.qn) + (int64_t)(l + 1) * N * F, Xn + n9, nbf);
            count_launch();
            TNET_LAUNCH_CHECK();
        }
    }

    // ---- output model
    pf.mark(P_OUTPUT);
    float *h = f32(Lw.h), *hn = f32(Lw.hn), *ao = f32(Lw.ao), *o = f32(Lw.o), *at = f32(Lw.at),
          *t = f32(Lw.t), *Ei = f32(Lw.Ei);
    float2 *lno = wsp<float2>(ctx, Lw.lno);
    const float *dX_last = NL > 0 ? f32(Lw.dX) + (NL - 1) * n9 : nullptr;
    launch(k_out_norms, N, F, 0, st, NL > 0 ? f32(Lw.Xn) + (NL - 1) * n9 : Xfin, dX_last, N, F, W.out_ln_g, W.out_ln_b,
           Xfin, h, hn, lno);
    count_launch();
    TNET_LAUNCH_CHECK();
    {
        const EpiBiasAct eo{W.out_b, ao, F, o, F, 1, nullptr};
        const EpiBiasAct eh{W.head1_b, at, H, t, H, 1, nullptr};
        if (atom_x3) {
            TRY(tcx3(tc::tshape(N, F, 3 * F), hn, N, 3 * F, wx.out, F, 3 * F, eo));
            TRY(tcx3(tc::tshape(N, H, F), o, N, F, wx.head1, H, F, eh));
        } else {
            TRY(sgemm<true>(gshape(N, F, 3 * F, hn, 3 * F, W.out_w, 3 * F), eo, gctas, sms, st));
            TRY(sgemm<true>(gshape(N, H, F, o, F, W.head1_w, F), eh, gctas, sms, st));
        }
    }
    launch(k_head, warps_grid, 256, 0, st, t, N, H, W.head2_w, W.head2_b, Ei);
    count_launch();
    launch(k_energy, S, N / S > 1024 ? 1024 : 128, 0, st, Ei, sys_start, sys_end, energy);
    count_launch();
    TNET_LAUNCH_CHECK();
    if (!forces && !grad_w) return TNET_OK;

    // ---- reverse pass
    pf.mark(P_OUT_BWD);
    float *gat = f32(Lw.gat), *gao = f32(Lw.gao), *ghn = f32(Lw.ghn), *gEi = f32(Lw.gEi);
    float *gX = f32(Lw.gXa), *gdX = f32(Lw.gdX), *gTn = f32(Lw.gTn), *gM = f32(Lw.gM), *gY = f32(Lw.gY);
    float *gg = f32(Lw.gg), *ga2 = f32(Lw.ga2), *ga1 = f32(Lw.ga1), *ge = f32(Lw.ge), *gphiu = f32(Lw.gphiu);
    launch(k_head_bwd, grid_for((int64_t)N * H, 256, sms), 256, 0, st, at, N, H, W.head2_w, seed, batch, gat);
    count_launch();
    TNET_LAUNCH_CHECK();
    if (atom_x3) {
        TRY(tcx3(tc::tshape(N, F, H), gat, N, H, wx.head1T, F, H, EpiGradAct{ao, F, gao, F, 0}));
        TRY(tcx3(tc::tshape(N, 3 * F, F), gao, N, F, wx.outT, 3 * F, F, EpiStore{ghn, 3 * F, 0}, bn3));
    } else {
        TRY(sgemm<false>(gshape(N, F, H, gat, H, W.head1_w, F), EpiGradAct{ao, F, gao, F, 0}, gctas, sms, st));
        TRY(sgemm<false>(gshape(N, 3 * F, F, gao, F, W.out_w, 3 * F), EpiStore{ghn, 3 * F, 0}, gctas, sms, st));
    }
    launch(k_out_norms_bwd, N, F, 0, st, Xfin, h, ghn, lno, W.out_ln_g, N, F, gX, dX_last, gdX, nbf);
    count_launch();
    TNET_LAUNCH_CHECK();
    if (wg) {
        launch(k_seed_atoms, (N + 255) / 256, 256, 0, st, seed, batch, N, gEi);
        count_launch();
        TNET_LAUNCH_CHECK();
        TRY(wgrad_colsum(rows1(H, 1, N, t, H, nullptr, 0, nullptr), gEi, wpart, wcap, gw(G.head2_w), sms, st));
        TRY(wgrad_colsum(rows1(1, 1, N, gEi, 1, nullptr, 0, nullptr), nullptr, wpart, wcap, gw(G.head2_b), sms, st));
        TRY(wgrad_outer(rows1(H, F, N, gat, H, o, F, nullptr), wpart, wcap, gw(G.head1_w), gw(G.head1_b), sms, st));
        TRY(wgrad_outer(rows1(F, 3 * F, N, gao, F, hn, 3 * F, nullptr), wpart, wcap, gw(G.out_w), gw(G.out_b), sms, st));
        TRY(wgrad_layernorm(ghn, h, lno, N, 3 * F, wpart, wcap, gw(G.out_ln_g), sms, st));
    }
    // gphiu collects dE/dphi per pair (or, in table mode, dE/dd)
    if (NL > 0 || tab) TNET_CUDA_TRY(cudaMemsetAsync(gphiu, 0, sizeof(float) * 2 * maxU, st));
    for (int l = NL - 1; l >= 0; --l) {
        const LayerW &Lr = W.layer[l];
        const LayerW &Gr = G.layer[l];
        float *Xn = f32(Lw.Xn) + l * n9, *qn = f32(Lw.qn) + (int64_t)l * N * F;
        float *Y = f32(Lw.Y) + l * n9, *M = f32(Lw.M) + l * n9, *Tn = f32(Lw.Tn) + l * n9;
        // gX holds dE/dX_out of the layer and gdX (with its operand copy) its
        // residual adjoint; at the end gX holds dE/dX_n, whose normalisation
        // adjoint goes on to the layer before (or, at layer 0, into
        // k_emb_scale_bwd)
        auto norm_bwd = [&]() {
            if (l == 0) return;
            launch(k_node_norm_bwd, ew, 256, 0, st, Xn - n9, f32(Lw.dX) + (l - 1) * n9, qn, N, F, gX, gdX, nbf);
            count_launch();
        };
        pf.mark(P_NODE_BWD);
        if (tcm) TRY(tcg(tc::tshape_classes(N, F), gdX, nbf, 9LL * N, F, lb[l].mix2T, 3 * F, F, EpiBulk{nullptr, gTn, F}));
        else TRY(sgemm<false>(gshape_classes(N, F, gdX, Lr.mix2_w), EpiStore{gTn, F, 0}, gctas, sms, st));
        if (wg) TRY(wgrad_outer(rows3(gdX, Tn), wpart, wcap, gw(Gr.mix2_w), nullptr, sms, st));
        launch(k_T_bwd, ew, 256, 0, st, Y, M, gTn, N, F, gY, gM);
        count_launch();
        TNET_LAUNCH_CHECK();
        // this layer's radial-MLP activations: kept from the forward pass, or
        // recomputed here (same kernels, same inputs: bitwise the same values)
        if (!keep_act) TRY(edge_mlp(l, false));
        const float *a1 = act(Lw.a1, F, l), *h1 = act(Lw.h1, F, l), *a2 = act(Lw.a2, 2 * F, l),
                    *h2 = act(Lw.h2, 2 * F, l), *a3 = act(Lw.a3, 3 * F, l);
        pf.mark(P_MSG_BWD);
        // (the BF16 GEMMs read only the copy of ga3; the fp32 ga3 feeds the FP32
        // and 3xTF32 GEMMs and the weight gradients)
        float *ga3_out = (prec != 1 || wg) ? gg : nullptr;
#define MSG_BWD(FF)                                                                                          \
    launch_message_bwd<FF, false>(rows_pb, atom_blocks, st, row_ptr, col, pair_of, Y, gM, a3, phiu, tabfn(1 + l), \
                                  N, gY, nbf, ga3_out, ga3_cp, gphiu)
#define MSG_BWD_TAB(FF)                                                                                      \
    launch_message_bwd<FF, true>(rows_pb, atom_blocks, st, row_ptr, col, pair_of, Y, gM, a3, phiu, tabfn(1 + l), \
                                 N, gY, nbf, (float *)nullptr, none, gphiu)
        if (tab) {
            TNET_F_SWITCH(F, MSG_BWD_TAB);
        } else if (warp_rows) {
            auto staged = [&](auto channels) -> int {
                return message_tile<decltype(channels)::value, true>(sms, st, row_ptr, col, pair_of, a3, phiu, gM, Y, N,
                                                                     gY, nbf, ga3_out, ga3_cp, gphiu, maxU, status);
            };
            TRY(F == 64 ? staged(Channels<64>{}) : staged(Channels<128>{}));
        } else {
            TNET_F_SWITCH(F, MSG_BWD);
        }
#undef MSG_BWD
#undef MSG_BWD_TAB
        count_launch();
        TNET_LAUNCH_CHECK();
        if (tab) {  // no radial MLP to go back through
            pf.mark(P_NODE_BWD);
            if (tcm)
                TRY(tcg(tc::tshape_classes(N, F), gY, nbf, 9LL * N, F, lb[l].mix1T, 3 * F, F, EpiStore{gX, F, 1}));
            else TRY(sgemm<false>(gshape_classes(N, F, gY, Lr.mix1_w), EpiStore{gX, F, 1}, gctas, sms, st));
            norm_bwd();
            TNET_LAUNCH_CHECK();
            continue;
        }
        const EpiGradAct g3{a2, 2 * F, ga2, 2 * F, 0, ga2_cp, 2 * F};
        const EpiGradAct g2{a1, F, ga1, F, 0, ga1_cp, F};
        const EpiStore g1{ge, K, l != NL - 1};
        if (tcm) {
            tc::TcShape t3 = tc::tshape(maxU, 2 * F, 3 * F), t2 = tc::tshape(maxU, F, 2 * F);
            t2.rows_dev = t3.rows_dev = nu;
            pf.mark(P_MLP3_BWD);
            TRY(tcg(t3, gg, ga3_cp, maxU, 3 * F, lb[l].mlp3T, 2 * F, 3 * F, g3, bn2));
            pf.mark(P_MLP2_BWD);
            TRY(tcg(t2, ga2, ga2_cp, maxU, 2 * F, lb[l].mlp2T, F, 2 * F, g2));
            pf.mark(P_MLP1_BWD);  // N = num_rbf: 3xTF32 in both modes
            tc::TcShape u1 = tc::tshape(maxU, K, F);
            u1.rows_dev = nu;
            TRY(tcx3(u1, ga1, maxU, F, lb[l].mlp1T, K, F, g1));
        } else {
            pf.mark(P_MLP3_BWD);
            GemmShape q3 = gshape(maxU, 2 * F, 3 * F, gg, 3 * F, w3p(l), 2 * F);
            q3.rows_dev = nu;
            TRY(sgemm<false>(q3, g3, gctas, sms, st));
            pf.mark(P_MLP2_BWD);
            GemmShape q2 = gshape(maxU, F, 2 * F, ga2, 2 * F, Lr.mlp2_w, F);
            q2.rows_dev = nu;
            TRY(sgemm<false>(q2, g2, gctas, sms, st));
            pf.mark(P_MLP1_BWD);
            GemmShape q1 = gshape(maxU, K, F, ga1, F, Lr.mlp1_w, K);
            q1.rows_dev = nu;
            TRY(sgemm<false>(q1, g1, gctas, sms, st));
        }
        if (wg) {
            // gg is plane-major: map its rows back to the blob's c*3 + p order
            TRY(wgrad_outer(rows1(3 * F, 2 * F, maxU, gg, 3 * F, h2, 2 * F, nu), wpart, wcap, gw(Gr.mlp3_w), gw(Gr.mlp3_b), sms, st,
                            F));
            TRY(wgrad_outer(rows1(2 * F, F, maxU, ga2, 2 * F, h1, F, nu), wpart, wcap, gw(Gr.mlp2_w), gw(Gr.mlp2_b), sms, st));
            TRY(wgrad_outer(rows1(F, K, maxU, ga1, F, eu, K, nu), wpart, wcap, gw(Gr.mlp1_w), gw(Gr.mlp1_b), sms, st));
            TRY(wgrad_outer(rows3(gY, Xn), wpart, wcap, gw(Gr.mix1_w), nullptr, sms, st));
        }
        pf.mark(P_NODE_BWD);
        if (tcm) TRY(tcg(tc::tshape_classes(N, F), gY, nbf, 9LL * N, F, lb[l].mix1T, 3 * F, F, EpiStore{gX, F, 1}));
        else TRY(sgemm<false>(gshape_classes(N, F, gY, Lr.mix1_w), EpiStore{gX, F, 1}, gctas, sms, st));
        norm_bwd();
        TNET_LAUNCH_CHECK();
    }
    // embedding adjoint: gX holds dE/dX_n of layer 0 (without layers dE/dX0)
    pf.mark(P_EMB_NODE_BWD);
    float *gU = f32(Lw.gU), *gas2 = f32(Lw.gas2), *gas1 = f32(Lw.gas1), *gn0 = f32(Lw.gn0);
    float *gXraw = gdX;
    launch(k_emb_scale_bwd, ew, 256, 0, st, gX, NL > 0 ? f32(Lw.qn) : nullptr, Uemb, s, as2, N, F, gU, gas2, nbf);
    count_launch();
    TNET_LAUNCH_CHECK();
    if (atom_x3) {
        TRY(tcx3(tc::tshape(N, 2 * F, 3 * F), gas2, N, 3 * F, wx.emb_mlp2T, 2 * F, 3 * F,
                 EpiGradAct{as1, 2 * F, gas1, 2 * F, 0}, bn2));
        TRY(tcx3(tc::tshape(N, F, 2 * F), gas1, N, 2 * F, wx.emb_mlp1T, F, 2 * F, EpiStore{gn0, F, 0}));
    } else {
        TRY(sgemm<false>(gshape(N, 2 * F, 3 * F, gas2, 3 * F, W.emb_mlp2_w, 2 * F),
                                EpiGradAct{as1, 2 * F, gas1, 2 * F, 0}, gctas, sms, st));
        TRY(sgemm<false>(gshape(N, F, 2 * F, gas1, 2 * F, W.emb_mlp1_w, F), EpiStore{gn0, F, 0}, gctas, sms, st));
    }
    if (tcm) TRY(tcg(tc::tshape_classes(N, F), gU, nbf, 9LL * N, F, emixT, 3 * F, F, EpiBulk{nullptr, gXraw, F}));
    else TRY(sgemm<false>(gshape_classes(N, F, gU, W.emb_mix_w), EpiStore{gXraw, F, 0}, gctas, sms, st));
    launch(k_ln0_bwd, N, F, 0, st, Xraw, gn0, ln0, W.emb_ln_g, N, F, gXraw);
    count_launch();
    TNET_LAUNCH_CHECK();
    if (wg) {
        TRY(wgrad_outer(rows3(gU, Xraw), wpart, wcap, gw(G.emb_mix_w), nullptr, sms, st));
        TRY(wgrad_outer(rows1(3 * F, 2 * F, N, gas2, 3 * F, hs1, 2 * F, nullptr), wpart, wcap, gw(G.emb_mlp2_w), gw(G.emb_mlp2_b), sms, st));
        TRY(wgrad_outer(rows1(2 * F, F, N, gas1, 2 * F, n0, F, nullptr), wpart, wcap, gw(G.emb_mlp1_w), gw(G.emb_mlp1_b), sms, st));
        TRY(wgrad_layernorm(gn0, q0, ln0, N, F, wpart, wcap, gw(G.emb_ln_g), sms, st));
    }
    pf.mark(P_EMB_EDGE_BWD);
    float *gfu = f32(Lw.gfu), *Gp = f32(Lw.gp), *gA = f32(Lw.gA_atom), *gB = f32(Lw.gB_atom);
    float4 *edge_g = wsp<float4>(ctx, Lw.edge_g);
    const int bwd_blocks = grid_for((int64_t)N * 32, 256, sms);
    // weight gradients need per-atom sums of the pair-embedding adjoints
    // (atom-parallel kernel); forces alone use the pair-parallel kernel
#define EMB_BWD(CPL)                                                                                         \
    if (wg)                                                                                                  \
        launch(k_emb_bwd<CPL>, bwd_blocks, 256, 0, st, pos, box, batch, z, row_ptr, col, pair_of, N, d.max_z, rp, \
                                                   fu, Ta, Tb, gXraw, 1, gfu, edge_g, gA, gB, gfu_cp);        \
    else if (tab)                                                                                            \
        launch(k_emb_bwd_pairs<CPL, true>, pair_grid, 256, 0, st, geo, z, uij, ue, rev, nu, N, d.max_z, fu, tf0, Ta, \
                                                            Tb, gXraw, nullptr, edge_g, none, gphiu);               \
    else                                                                                                     \
        launch(k_emb_bwd_pairs<CPL, false>, pair_grid, 256, 0, st, geo, z, uij, ue, rev, nu, N, d.max_z, fu, tf0, Ta, \
                                                             Tb, gXraw, gfu, edge_g, gfu_cp, nullptr)
    const bool by_pair = !wg && !tab && warp_rows && F == 128;
    constexpr int pair_smem = 4 * kPairDepth * kPairBytes;
    if (by_pair) {
        TRY(ensure_smem_attr((const void *)k_emb_bwd_pairs_v4<128>, pair_smem));
        launch(k_emb_bwd_pairs_v4<128>, kPairBlocks * sms, 128, pair_smem, st, geo, z, uij, nu, N, d.max_z, fu, Ta, Tb, gXraw, gfu,
               edge_g);
    } else {
        switch (F / 32) {
            case 2: EMB_BWD(2); break;
            case 4: EMB_BWD(4); break;
            case 6: EMB_BWD(6); break;
            case 8: EMB_BWD(8); break;
            case 10: EMB_BWD(10); break;
            case 12: EMB_BWD(12); break;
            case 14: EMB_BWD(14); break;
            case 16: EMB_BWD(16); break;
            default: return TNET_ERR_ARG;
        }
    }
#undef EMB_BWD
    count_launch();
    TNET_LAUNCH_CHECK();
    if (!tab) {   // dE/de of the pair's radial basis also flows through the projections
        if (tcm) {
            tc::TcShape tg = tc::tshape(maxU, K, 3 * F);
            tg.rows_dev = nu;
            TRY(tcx3(tg, gfu, maxU, 3 * F, wx.dprojT, K, 3 * F, EpiStore{ge, K, NL > 0}));
        } else {
            GemmShape pg = gshape(maxU, K, 3 * F, gfu, 3 * F, W.dproj_w, K);
            pg.rows_dev = nu;
            TRY(sgemm<false>(pg, EpiStore{ge, K, NL > 0}, gctas, sms, st));
        }
    }
    if (wg) {
        TRY(wgrad_outer(rows1(3 * F, K, maxU, gfu, 3 * F, eu, K, nu), wpart, wcap, gw(G.dproj_w), gw(G.dproj_b), sms, st));
        const int zs = (int)Lw.zsplits;
        float *zpart = f32(Lw.zpart);
        launch(k_group_z, dim3(d.max_z, zs), F, 0, st, z, gA, gB, N, F, d.max_z, zs, zpart);
        count_launch();
        launch(k_zreduce, d.max_z, F, 0, st, zpart, zs, F, d.max_z, zpart);
        count_launch();
        launch(k_emb_tables_grad2, F + d.max_z, F, 0, st, zpart, F, d.max_z, W.emb, W.emb2_w, gw(G.emb), gw(G.emb2_w),
                                                      gw(G.emb2_b));
        count_launch();
        TNET_LAUNCH_CHECK();
    }
    if (!forces) return TNET_OK;
    pf.mark(P_FORCES);
    launch(k_pair_vec, pair_grid, 256, 0, st, pos, box, batch, uij, ue, rev, nu, rp, tab ? nullptr : ge,
           (NL > 0 && !tab) ? gphiu : nullptr, (int64_t)maxU, edge_g, by_pair ? edge_g : nullptr, tab ? gphiu : nullptr, Gp);
    count_launch();
    launch(k_forces, (unsigned)(((int64_t)N * kForceLanes + 127) / 128), 128, 0, st, row_ptr, col, pair_of, Gp, N, forces);
    count_launch();
    TNET_LAUNCH_CHECK();
    return TNET_OK;
}

}  // namespace tnet

extern "C" int tnet_debug_message_tile(int F, int backward, int n_atoms, const int32_t *row_ptr, const int32_t *col,
                                       const int32_t *pair_of, const float *a3, const float *phi, const float *V,
                                       const float *V2, float *out, float *ga3, float *gphi, int64_t n_pairs,
                                       uint32_t spin_limit, int hold_copies, int32_t *status, tnet_stream_t stream) {
    using namespace tnet;
    if ((F != 64 && F != 128) || n_atoms < 1 || 9LL * n_atoms * F >= (1LL << 31) || n_pairs < 0 ||
        n_pairs * 3 * F >= (1LL << 31) || (hold_copies && spin_limit < 1))
        return TNET_ERR_ARG;
    if (!row_ptr || !col || !pair_of || !a3 || !phi || !V || !out || !status || (backward && (!V2 || !ga3 || !gphi)))
        return TNET_ERR_ARG;
    int dev = 0, sms = 0;
    TNET_CUDA_TRY(cudaGetDevice(&dev));
    TNET_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const OpCopy none{nullptr, 0};
    auto run = [&](auto channels, auto bwd) -> int {
        return message_tile<decltype(channels)::value, decltype(bwd)::value>(
            sms, (cudaStream_t)stream, row_ptr, col, pair_of, a3, phi, V, V2, n_atoms, out, none, ga3, none, gphi,
            n_pairs, status, spin_limit, hold_copies);
    };
    TRY(F == 64 ? (backward ? run(Channels<64>{}, std::true_type{}) : run(Channels<64>{}, std::false_type{}))
                : (backward ? run(Channels<128>{}, std::true_type{}) : run(Channels<128>{}, std::false_type{})));
    TNET_LAUNCH_CHECK();
    return TNET_OK;
}
