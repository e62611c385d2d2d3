// Weight-gradient reductions: sums over rows (atoms, coordinate rows or
// undirected pairs) of outer products, column sums and LayerNorm parameter
// gradients.  Every reduction is split over row ranges into partial sums
// that a second kernel adds in a fixed order, so weight gradients are
// deterministic (no floating-point atomics).
#include "gemm.cuh"
#include "internal.cuh"

namespace tnet {

// out[m][n] = sum_r A[r][m] B[r][n] over one of `splits` row ranges per CTA: the
// rows are the GEMM's K, so both operands arrive as the tile reads them
// ([32 rows][columns], cp.async ring of three) and a thread keeps TM x (4 NB)
// outputs, two columns per packed FMA, in ascending row order.  The CTAs of
// the first column tile also add up their columns of A (the bias gradient,
// whose operand they hold anyway).
// What bounds it: FP32 FMA; the splits give every SM two 128 x 128 tiles.
template <int TM_, int NB_, int WM_, int WN_, int MINB_>
struct WgTile {
    static constexpr int TM = TM_, NB = NB_, WM = WM_, WN = WN_, MINB = MINB_, ST = 3, BK = 32;
    static constexpr int BM = 4 * TM * WM, BN = 32 * NB * WN, THREADS = 32 * WM * WN;
    static constexpr int SMEM = ST * (BM + BN) * BK * 4;
};

template <class C>
__global__ void __launch_bounds__(C::THREADS, C::MINB) k_wgrad(WgradShape P, int splits, float *__restrict__ partial,
                                                               float *__restrict__ partial_bias) {
    pdl_entry();
    constexpr int TM = C::TM, NB = C::NB, BM = C::BM, BN = C::BN, BK = C::BK, ST = C::ST, TH = C::THREADS;
    extern __shared__ __align__(128) float wg_smem[];
    float *sA = wg_smem, *sB = wg_smem + ST * BM * BK;
    const int z = blockIdx.z, s = blockIdx.y;
    int64_t R = z == 0 ? P.rows[0] : (z == 1 ? P.rows[1] : P.rows[2]);
    if (z == 0 && P.rows_dev) {
        const int64_t rd = (int64_t)(*P.rows_dev) * P.rows_mul;
        R = rd < R ? rd : R;
    }
    const int tilesN = (P.N + BN - 1) / BN;
    const int m0 = (blockIdx.x / tilesN) * BM, n0 = (blockIdx.x % tilesN) * BN;
    // equal row ranges of the true row count, in whole blocks
    const int64_t chunk = ((R + splits - 1) / splits + BK - 1) / BK * BK;
    const int64_t r_begin = s * chunk, r_end = r_begin + chunk < R ? r_begin + chunk : R;
    const int nk = r_end > r_begin ? (int)((r_end - r_begin + BK - 1) / BK) : 0;
    const int64_t rz = z == 0 ? P.row0[0] : (z == 1 ? P.row0[1] : P.row0[2]);
    const float *A = P.A + rz * P.lda;
    const float *B = P.B + rz * P.ldb;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int mrow = (w / C::WN) * 4 * TM + (lane >> 3) * TM, ncol = (w % C::WN) * 32 * NB + (lane & 7) * 4;
    auto load = [&](int kb) {
        const int st = kb % ST;
        if (kb < nk) {
            const int64_t r0 = r_begin + (int64_t)kb * BK;
#pragma unroll
            for (int t = tid; t < BK * BM / 4; t += TH) {
                const int r = t / (BM / 4), c = (t % (BM / 4)) * 4;
                const bool ok = r0 + r < r_end && m0 + c < P.M;
                sg_cp16(sg_addr(sA + (st * BK + r) * BM + c), ok ? A + (r0 + r) * P.lda + m0 + c : P.A, ok);
            }
#pragma unroll
            for (int t = tid; t < BK * BN / 4; t += TH) {
                const int r = t / (BN / 4), c = (t % (BN / 4)) * 4;
                const bool ok = r0 + r < r_end && n0 + c < P.N;
                sg_cp16(sg_addr(sB + (st * BK + r) * BN + c), ok ? B + (r0 + r) * P.ldb + n0 + c : P.B, ok);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint64_t acc[TM][NB][2];
    float cs = 0.f;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) acc[i][j][0] = acc[i][j][1] = 0;
    static_assert(TM == 8, "a lane of each row group per row of its column sums");
    const bool bias = partial_bias && n0 == 0 && w % C::WN == 0;
#pragma unroll
    for (int t = 0; t < ST - 1; ++t) load(t);
    for (int kb = 0; kb < nk; ++kb) {
        asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
        __syncthreads();
        load(kb + ST - 1);
        const float *a = sA + (kb % ST) * BM * BK, *b = sB + (kb % ST) * BN * BK;
        if (bias) {
            // one of the thread's TM rows of the output per lane of its row group,
            // a sum per block first: wide outputs leave few row ranges, and one
            // chain of additions over a range of thousands of rows would lose
            // what the blocks' shorter ones keep (20,000 equal rows in six
            // ranges: 4.9e-5 of the sum, 1.6e-6 by blocks)
            float blk = 0.f;
#pragma unroll 8
            for (int r = 0; r < BK; ++r) blk += a[r * BM + mrow + (lane & 7)];
            cs += blk;
        }
#pragma unroll 8
        for (int r = 0; r < BK; ++r) {
            float av[TM];
#pragma unroll
            for (int i = 0; i < TM; i += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(a + r * BM + mrow + i);
                av[i] = v.x; av[i + 1] = v.y; av[i + 2] = v.z; av[i + 3] = v.w;
            }
            uint64_t b2[NB][2];
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const float4 v = *reinterpret_cast<const float4 *>(b + r * BN + ncol + 32 * j);
                b2[j][0] = f2_pack(v.x, v.y);
                b2[j][1] = f2_pack(v.z, v.w);
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const uint64_t x2 = f2_pack(av[i], av[i]);
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    acc[i][j][0] = f2_fma(x2, b2[j][0], acc[i][j][0]);
                    acc[i][j][1] = f2_fma(x2, b2[j][1], acc[i][j][1]);
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    float *out = partial + ((int64_t)z * splits + s) * P.M * P.N;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + mrow + i;
        if (m >= P.M) continue;
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int n = n0 + ncol + 32 * j;
            if (n < P.N) *reinterpret_cast<float4 *>(out + (int64_t)m * P.N + n) = f2_four(acc[i][j]);
        }
    }
    const int mb = m0 + mrow + (lane & 7);
    if (bias && mb < P.M) partial_bias[(int64_t)s * P.M + mb] = cs;
}

// partial[(z*splits + s)][m] = sum over rows of split s of A[r][m] (* w[r])
__global__ void k_colsum(WgradShape P, int splits, const float *__restrict__ roww,
                         float *__restrict__ partial) {
    pdl_entry();
    const int z = blockIdx.z, s = blockIdx.y;
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= P.M) return;
    int64_t R = z == 0 ? P.rows[0] : (z == 1 ? P.rows[1] : P.rows[2]);
    if (z == 0 && P.rows_dev) {
        const int64_t rd = (int64_t)(*P.rows_dev) * P.rows_mul;
        R = rd < R ? rd : R;
    }
    const int64_t chunk = (R + splits - 1) / splits;
    const int64_t r_begin = s * chunk;
    int64_t r_end = r_begin + chunk;
    if (r_end > R) r_end = R;
    const float *A = P.A + (z == 0 ? P.row0[0] : (z == 1 ? P.row0[1] : P.row0[2])) * P.lda;
    float acc = 0.f;
#pragma unroll 8
    for (int64_t r = r_begin; r < r_end; ++r) acc += A[r * P.lda + m] * (roww ? roww[r] : 1.0f);
    partial[((int64_t)z * splits + s) * P.M + m] = acc;
}

// LayerNorm parameter gradients: dgamma[c] = sum_r gy[r][c] xhat[r][c],
// dbeta[c] = sum_r gy[r][c], xhat = (x - mean_r) * rstd_r
__global__ void k_ln_grad(const float *__restrict__ gy, const float *__restrict__ x,
                          const float2 *__restrict__ stats, int R, int C, int splits,
                          float *__restrict__ partial) {
    pdl_entry();
    const int s = blockIdx.y;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const int64_t chunk = ((int64_t)R + splits - 1) / splits;
    const int64_t r_begin = s * chunk;
    int64_t r_end = r_begin + chunk;
    if (r_end > R) r_end = R;
    float ag = 0.f, ab = 0.f;
#pragma unroll 4
    for (int64_t r = r_begin; r < r_end; ++r) {
        const float g = gy[r * C + c];
        const float2 st = stats[r];
        ag = fmaf(g, (x[r * C + c] - st.x) * st.y, ag);
        ab += g;
    }
    partial[(int64_t)s * 2 * C + c] = ag;
    partial[(int64_t)s * 2 * C + C + c] = ab;
}

// out[z][i] = sum_s partial[z][s][i] in split order, and likewise the bias
// sums (one class) that follow them.  With perm_f > 0 the rows m of the
// [3 perm_f][ncols] output come in plane-major order (m = p perm_f + c) and
// are written to row c*3 + p.
__global__ void k_split_reduce(const float *__restrict__ partial, int splits, int64_t per_class, int nclass,
                               float *__restrict__ out, int ncols, int perm_f, const float *__restrict__ partial_bias,
                               float *__restrict__ out_bias, int nbias) {
    pdl_entry();
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool b = t >= per_class * nclass;  // a bias entry
    if (b) {
        t -= per_class * nclass;
        if (t >= nbias) return;
        per_class = nbias;
        ncols = 1;
        partial = partial_bias;
        out = out_bias;
    }
    const int64_t z = b ? 0 : t / per_class, i = b ? t : t % per_class;
    int64_t o = t;
    if (perm_f > 0) {
        const int64_t m = i / ncols, n = i % ncols;
        o = z * per_class + ((m % perm_f) * 3 + m / perm_f) * ncols + n;
    }
    float acc = 0.f;
    const float *p = partial + z * splits * per_class + i;
#pragma unroll 8
    for (int s = 0; s < splits; ++s) acc += p[(int64_t)s * per_class];
    out[o] = acc;
}

// Row ranges: about `ctas` CTAs in all, at least min_rows rows each, partial
// sums within the scratch.
static int choose_splits(int64_t rows_cap, int64_t tiles, int min_rows, int64_t floats_per_split, int64_t partial_cap,
                         int64_t ctas) {
    int64_t splits = ctas / tiles;
    const int64_t max_by_rows = rows_cap / min_rows, max_by_mem = partial_cap / floats_per_split;
    if (splits > max_by_rows) splits = max_by_rows;
    if (splits > max_by_mem) splits = max_by_mem;
    return (int)(splits < 1 ? 1 : splits);
}

static int reduce_splits(const float *partial, int splits, int64_t per_class, int nclass, float *out, int ncols,
                         int perm_f, const float *partial_bias, float *out_bias, int nbias, cudaStream_t st) {
    const int64_t tot = nclass * per_class + nbias;
    launch(k_split_reduce, (unsigned)((tot + 255) / 256), 256, 0, st, partial, splits, per_class, nclass, out, ncols,
           perm_f, partial_bias, out_bias, nbias);
    count_launch();
    TNET_LAUNCH_CHECK();
    return TNET_OK;
}

template <class C>
static int wgrad_tile(const WgradShape &P, int64_t rows_cap, float *partial, int64_t partial_cap, float *out,
                      float *out_bias, int sms, cudaStream_t st, int perm_f) {
    const int64_t tiles = (int64_t)((P.M + C::BM - 1) / C::BM) * ((P.N + C::BN - 1) / C::BN);
    const int64_t per_split = (int64_t)P.nclass * P.M * P.N + (out_bias ? P.M : 0);
    const int splits = choose_splits(rows_cap, tiles * P.nclass, 64, per_split, partial_cap, (int64_t)C::MINB * sms);
    if (splits * per_split > partial_cap) return TNET_ERR_WORKSPACE;
    float *pb = out_bias ? partial + (int64_t)splits * P.M * P.N : nullptr;
    auto kern = k_wgrad<C>;
    const int rc = ensure_smem_attr((const void *)kern, C::SMEM);
    if (rc) return rc;
    launch(kern, dim3((unsigned)tiles, splits, P.nclass), C::THREADS, C::SMEM, st, P, splits, partial, pb);
    count_launch();
    TNET_LAUNCH_CHECK();
    return reduce_splits(partial, splits, (int64_t)P.M * P.N, P.nclass, out, P.N, perm_f, pb, out_bias,
                         out_bias ? P.M : 0, st);
}

int wgrad_outer(const WgradShape &P, float *partial, int64_t partial_cap, float *out, float *out_bias, int sms,
                cudaStream_t st, int perm_f) {
    int64_t rows_cap = 0;
    for (int z = 0; z < P.nclass; ++z) rows_cap = P.rows[z] > rows_cap ? P.rows[z] : rows_cap;
    if (rows_cap <= 0 || P.M <= 0 || P.N <= 0) return TNET_OK;
    if (P.M % 4 || P.N % 4 || P.lda % 4 || P.ldb % 4 || (out_bias && P.nclass != 1)) return TNET_ERR_ARG;
    // 128 x 128 tiles, two per SM; 128 x 32 for outputs of at most 64 columns
    // (the num_rbf-wide layers), four per SM
    if (P.N > 64)
        return wgrad_tile<WgTile<8, 2, 4, 2, 2>>(P, rows_cap, partial, partial_cap, out, out_bias, sms, st, perm_f);
    return wgrad_tile<WgTile<8, 1, 4, 1, 4>>(P, rows_cap, partial, partial_cap, out, out_bias, sms, st, perm_f);
}

int wgrad_colsum(const WgradShape &P, const float *roww, float *partial, int64_t partial_cap, float *out, int sms,
                 cudaStream_t st) {
    int64_t rows_cap = 0;
    for (int z = 0; z < P.nclass; ++z) rows_cap = P.rows[z] > rows_cap ? P.rows[z] : rows_cap;
    if (rows_cap <= 0 || P.M <= 0) return TNET_OK;
    const int64_t tiles = (P.M + 255) / 256;
    const int splits = choose_splits(rows_cap, tiles * P.nclass, 8, (int64_t)P.nclass * P.M, partial_cap, 2LL * sms);
    launch(k_colsum, dim3((unsigned)tiles, splits, P.nclass), 256, 0, st, P, splits, roww, partial);
    count_launch();
    TNET_LAUNCH_CHECK();
    return reduce_splits(partial, splits, P.M, P.nclass, out, 1, 0, nullptr, nullptr, 0, st);
}

// out_g[0..C) = dgamma, out_g[C..2C) = dbeta (gamma and beta are adjacent in
// the weight blob)
int wgrad_layernorm(const float *gy, const float *x, const float2 *stats, int R, int C, float *partial,
                    int64_t partial_cap, float *out_g, int sms, cudaStream_t st) {
    if (R <= 0) return TNET_OK;
    const int64_t tiles = (C + 255) / 256;
    const int splits = choose_splits(R, tiles, 8, 2LL * C, partial_cap, 2LL * sms);
    launch(k_ln_grad, dim3((unsigned)tiles, splits, 1), 256, 0, st, gy, x, stats, R, C, splits, partial);
    count_launch();
    TNET_LAUNCH_CHECK();
    return reduce_splits(partial, splits, 2LL * C, 1, out_g, 1, 0, nullptr, nullptr, 0, st);
}

}  // namespace tnet
