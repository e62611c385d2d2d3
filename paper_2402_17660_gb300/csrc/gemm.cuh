// FP32 SIMT GEMM with fused epilogues, used for the per-atom and per-edge
// dense layers of the FP32 path.
//
//   C[m][n] = epi( sum_k A[m*lda + k] B(k,n) )
//   B(k,n) = TB ? B[n*ldb + k] : B[k*ldb + n]      (TB: weights stored (out, in))
//
// Up to 3 "classes" (blockIdx.z) share one launch: class z uses rows
// [row0[z], row0[z] + rows[z]) of A and C and the weight B + z*strideB.
// This is how one launch mixes the I, A and S coordinate planes with their
// own matrices.  The row count of a class may be read from device memory
// (rows_dev, times rows_mul), so launches sized for a capacity stay valid
// inside a CUDA graph when the true count is only known on the device.
// Tiles are visited by a persistent grid-stride loop.
#pragma once
#include <cuda_bf16.h>

#include "internal.cuh"

namespace tnet {

struct GemmShape {
    int M[3];                // rows per class (capacity when rows_dev is set)
    int64_t row0[3];         // first row of each class in A and C
    const int32_t *rows_dev; // optional device row count (applies to class 0 only)
    int rows_mul;
    int N, K;
    const float *A;
    int64_t lda;
    const float *B;
    int64_t ldb, strideB;
    int nclass;
};

// --------------------------------------------------------------- epilogues
// Each epilogue receives 4 consecutive columns (n..n+3, all < N) of row m by
// value (a pointer would force the accumulator fragment into local memory).
// Optional bf16 operand copies feed the BF16 tensor-core GEMMs.
__device__ __forceinline__ void store_copy4(const OpCopy &c, int64_t idx, const float o[4]) {
    if (c.mode == 1) {
        __nv_bfloat162 a = __floats2bfloat162_rn(o[0], o[1]), b = __floats2bfloat162_rn(o[2], o[3]);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t *>(&a);
        u.y = *reinterpret_cast<uint32_t *>(&b);
        *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(c.p) + idx) = u;
    }
}

// Each functor splits into pre() (the loads: issued for several rows before
// the accumulator values arrive, so their latency overlaps) and post() (the
// arithmetic and stores); operator() runs both.  pre() may be given a row or
// column clamped into range, and its result is then unused.
struct EpiStore {  // C = v (+ C when accumulate)
    static constexpr bool BULK = false;
    float *C;
    int64_t ldc;
    int accumulate;
    struct Pre {
        float4 c;
    };
    __device__ Pre pre(int, int64_t m, int n) const {
        return Pre{accumulate ? *reinterpret_cast<const float4 *>(C + m * ldc + n) : make_float4(0.f, 0.f, 0.f, 0.f)};
    }
    __device__ void post(int, int64_t m, int n, float4 o, const Pre &p) const {
        if (accumulate) {
            o.x += p.c.x; o.y += p.c.y; o.z += p.c.z; o.w += p.c.w;
        }
        *reinterpret_cast<float4 *>(C + m * ldc + n) = o;
    }
    __device__ void operator()(int z, int64_t m, int n, float4 o) const { post(z, m, n, o, pre(z, m, n)); }
};

struct EpiBiasAct {  // a = v + bias; pre = a; out = act(a) * rowscale[m] (+ operand copy)
    static constexpr bool BULK = false;
    const float *bias;
    float *pre_out;
    int64_t ldp;
    float *out;
    int64_t ldo;
    int silu;
    const float *rowscale;
    OpCopy out_cp;
    int64_t ldoc;
    struct Pre {
        float4 b;
        float rs;
    };
    __device__ Pre pre(int, int64_t m, int n) const {
        return Pre{bias ? *reinterpret_cast<const float4 *>(bias + n) : make_float4(0.f, 0.f, 0.f, 0.f),
                   rowscale ? rowscale[m] : 1.0f};
    }
    __device__ void post(int, int64_t m, int n, float4 vv, const Pre &p) const {
        const float v[4] = {vv.x, vv.y, vv.z, vv.w};
        const float bv[4] = {p.b.x, p.b.y, p.b.z, p.b.w};
        float a[4], o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            a[q] = v[q] + bv[q];
            o[q] = (silu ? silu_f(a[q]) : a[q]) * p.rs;
        }
        if (pre_out) *reinterpret_cast<float4 *>(pre_out + m * ldp + n) = make_float4(a[0], a[1], a[2], a[3]);
        if (out) *reinterpret_cast<float4 *>(out + m * ldo + n) = make_float4(o[0], o[1], o[2], o[3]);
        if (out_cp.mode) store_copy4(out_cp, m * ldoc + n, o);
    }
    __device__ void operator()(int z, int64_t m, int n, float4 o) const { post(z, m, n, o, pre(z, m, n)); }
};

// C = v (+ bias) and nothing else: the tensor-core GEMM writes whole groups of
// 32 rows with bulk tensor stores
struct EpiBulk {
    static constexpr bool BULK = true;
    const float *bias;  // or NULL
    float *C;
    int64_t ldc;
    struct Pre {};
    __device__ Pre pre(int, int64_t, int) const { return Pre{}; }
    __device__ void post(int, int64_t, int, float4, const Pre &) const {}
};

struct EpiGradAct {  // out = v * silu'(pre)  (+ out when accumulate) (+ operand copy)
    static constexpr bool BULK = false;
    const float *pre_in;
    int64_t ldp;
    float *out;
    int64_t ldo;
    int accumulate;
    OpCopy out_cp;
    int64_t ldoc;
    struct Pre {
        float4 a, c;
    };
    __device__ Pre pre(int, int64_t m, int n) const {
        return Pre{*reinterpret_cast<const float4 *>(pre_in + m * ldp + n),
                   accumulate ? *reinterpret_cast<const float4 *>(out + m * ldo + n) : make_float4(0.f, 0.f, 0.f, 0.f)};
    }
    __device__ void post(int, int64_t m, int n, float4 vv, const Pre &p) const {
        float o[4] = {vv.x * silu_grad_f(p.a.x), vv.y * silu_grad_f(p.a.y), vv.z * silu_grad_f(p.a.z),
                      vv.w * silu_grad_f(p.a.w)};
        if (accumulate) {
            o[0] += p.c.x; o[1] += p.c.y; o[2] += p.c.z; o[3] += p.c.w;
        }
        *reinterpret_cast<float4 *>(out + m * ldo + n) = make_float4(o[0], o[1], o[2], o[3]);
        if (out_cp.mode) store_copy4(out_cp, m * ldoc + n, o);
    }
    __device__ void operator()(int z, int64_t m, int n, float4 o) const { post(z, m, n, o, pre(z, m, n)); }
};

// --------------------------------------------------------------- kernel ---
__device__ __forceinline__ uint32_t sg_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// asynchronous copies global -> shared, zero-filled when !ok
__device__ __forceinline__ void sg_cp16(uint32_t dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void sg_cp4(uint32_t dst, const void *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
// two FP32 values in one 64-bit register, and two FP32 FMAs in one instruction
// (each rounded like fmaf)
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_unpack(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float4 f2_four(const uint64_t v[2]) {
    const float2 a = f2_unpack(v[0]), b = f2_unpack(v[1]);
    return make_float4(a.x, a.y, b.x, b.y);
}

// One CTA: WM x WN warps (times KS groups of them that share the K range) on a
// (4 TM WM) x (32 NB WN) tile; a warp is 4 x 8 lanes, each with TM rows x NB
// blocks of four columns.  K runs in 32-deep blocks through an ST-stage
// cp.async ring: A as it lies ([m][32], 16-byte chunk c of row m at
// c ^ (m / TM), which keeps the four row groups a warp reads together on
// different banks), B as [32][n], transposed on the way in for TB by 4-byte
// copies (coalesced along k).  Products are packed two columns to an
// instruction.
// What bounds it: the FP32 pipe (70 TFLOP/s from registers alone, scalar or
// packed) and the issue slots beside it; packing halves the FMA instructions,
// which leaves the issue slots to the shared-memory loads.  Each output is one
// chain of FMAs in ascending k (KS = 1), so those tile sizes agree bit for bit;
// with KS > 1 the groups take every KS-th 4-deep slice and their sums are
// added in group order.  The tile follows from the rows a launch may have, so
// a system's bits depend on the company it is evaluated in and on the
// context's capacities (tnet.h says so); one chain in every tile (64 x 32 and
// 32 x 32 with more warps of fewer outputs instead) would end that at the same
// speed (32 atoms 307 us against 305, 3,000 atoms 3.51 ms against 3.52), but the
// shorter chains are the more exact: forces of 32 atoms are 8.6e-7 from 64-bit
// ones, 1.7e-6 with one chain.
// Measured (GB300, us, the former 128 x 64 tile with 8-deep blocks first):
//   M 82,000 N 384 K 256: 407 -> 318 (51 TFLOP/s); weights (out, in) 433 -> 353
//   M 96,000 N 128 K 384: 233 -> 209      M 82,000 N 32 K 384: 121 -> 60
//   M 3,000  N 128 K 384: 28.7 -> 14.4    M 32 N 128 K 384: 26.7 -> 8.3
template <int TM_, int NB_, int WM_, int WN_, int KS_, int ST_, int MINB_>
struct SgTile {
    static constexpr int TM = TM_, NB = NB_, WM = WM_, WN = WN_, KS = KS_, ST = ST_, MINB = MINB_;
    static constexpr int BM = 4 * TM * WM, BN = 32 * NB * WN, BK = 32, GROUP = 32 * WM * WN, THREADS = GROUP * KS;
    static constexpr int ldb(bool tb) { return tb ? BN + 4 : BN; }  // padded when B is transposed on the way in
    static constexpr int smem(bool tb) { return ST * (BM + ldb(tb)) * BK * 4; }
    static_assert((KS - 1) * GROUP * TM * NB * 4 * 4 <= ST * (BM + BN) * BK * 4, "partial sums reuse the ring");
};

template <class C, bool TB, class Epi>
__global__ void __launch_bounds__(C::THREADS, C::MINB) k_sgemm(GemmShape P, Epi epi) {
    pdl_entry();
    constexpr int TM = C::TM, NB = C::NB, BM = C::BM, BN = C::BN, BK = C::BK, ST = C::ST, KS = C::KS;
    constexpr int TH = C::THREADS, GROUP = C::GROUP, LB = C::ldb(TB);
    extern __shared__ __align__(128) float sg_smem[];
    float *sA = sg_smem, *sB = sg_smem + ST * BM * BK;
    const int z = blockIdx.z;
    // selects, not P.M[z]: a dynamically indexed parameter array is copied to local memory
    int M = z == 0 ? P.M[0] : (z == 1 ? P.M[1] : P.M[2]);
    if (z == 0 && P.rows_dev) {
        const int md = *P.rows_dev * P.rows_mul;
        M = md < M ? md : M;
    }
    const int64_t r0 = z == 0 ? P.row0[0] : (z == 1 ? P.row0[1] : P.row0[2]);
    const float *A = P.A + r0 * P.lda;
    const float *B = P.B + (int64_t)z * P.strideB;
    const int N = P.N, K = P.K;
    const int tilesN = (N + BN - 1) / BN, tilesM = (M + BM - 1) / BM, nk = (K + BK - 1) / BK;
    const int tid = threadIdx.x, lane = tid & 31, kg = tid / GROUP, gt = tid % GROUP, w = gt >> 5;
    const int mrow = (w / C::WN) * 4 * TM + (lane >> 3) * TM, ncol = (w % C::WN) * 32 * NB + (lane & 7) * 4;

    for (int tile = blockIdx.x; tile < tilesM * tilesN; tile += gridDim.x) {
        const int m0 = (tile / tilesN) * BM, n0 = (tile % tilesN) * BN;
        auto load = [&](int kb) {
            const int s = kb % ST, k0 = kb * BK;
            if (kb < nk) {
#pragma unroll
                for (int t = tid; t < BM * (BK / 4); t += TH) {
                    const int m = t / (BK / 4), c = t % (BK / 4);
                    const bool ok = m0 + m < M && k0 + 4 * c < K;
                    sg_cp16(sg_addr(sA + (s * BM + m) * BK + 4 * (c ^ ((m / TM) & 7))),
                            ok ? A + (int64_t)(m0 + m) * P.lda + k0 + 4 * c : A, ok);
                }
                if constexpr (TB) {
#pragma unroll
                    for (int t = tid; t < BN * BK; t += TH) {
                        const int n = t / BK, k = t % BK;
                        const bool ok = n0 + n < N && k0 + k < K;
                        sg_cp4(sg_addr(sB + (s * BK + k) * LB + n), ok ? B + (int64_t)(n0 + n) * P.ldb + k0 + k : B, ok);
                    }
                } else {
#pragma unroll
                    for (int t = tid; t < BK * BN / 4; t += TH) {
                        const int k = t / (BN / 4), n = (t % (BN / 4)) * 4;
                        const bool ok = n0 + n < N && k0 + k < K;
                        sg_cp16(sg_addr(sB + (s * BK + k) * LB + n), ok ? B + (int64_t)(k0 + k) * P.ldb + n0 + n : B, ok);
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        uint64_t acc[TM][NB][2];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) acc[i][j][0] = acc[i][j][1] = 0;
#pragma unroll
        for (int s = 0; s < ST - 1; ++s) load(s);
        for (int kb = 0; kb < nk; ++kb) {
            asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
            __syncthreads();  // block kb has landed for every thread, and block kb - 1 is consumed
            load(kb + ST - 1);
            const float *a = sA + (kb % ST) * BM * BK, *b = sB + (kb % ST) * LB * BK;
#pragma unroll
            for (int cc = 0; cc < BK / 4 / KS; ++cc) {
                const int c = cc * KS + kg;  // this group's 4-deep slice
                float4 av[TM], bv[4][NB];
#pragma unroll
                for (int i = 0; i < TM; ++i)
                    av[i] = *reinterpret_cast<const float4 *>(a + (mrow + i) * BK + 4 * (c ^ ((mrow / TM) & 7)));
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int j = 0; j < NB; ++j)
                        bv[k][j] = *reinterpret_cast<const float4 *>(b + (4 * c + k) * LB + ncol + 32 * j);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    uint64_t b2[NB][2];
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        b2[j][0] = f2_pack(bv[k][j].x, bv[k][j].y);
                        b2[j][1] = f2_pack(bv[k][j].z, bv[k][j].w);
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i) {
                        const float x = k == 0 ? av[i].x : (k == 1 ? av[i].y : (k == 2 ? av[i].z : av[i].w));
                        const uint64_t x2 = f2_pack(x, x);
#pragma unroll
                        for (int j = 0; j < NB; ++j) {
                            acc[i][j][0] = f2_fma(x2, b2[j][0], acc[i][j][0]);
                            acc[i][j][1] = f2_fma(x2, b2[j][1], acc[i][j][1]);
                        }
                    }
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        float4 *part = reinterpret_cast<float4 *>(sg_smem);  // [group - 1][i][j][thread]
        if (KS > 1) {
            if (kg > 0) {
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < NB; ++j) part[(((kg - 1) * TM + i) * NB + j) * GROUP + gt] = f2_four(acc[i][j]);
            }
            __syncthreads();
        }
        const int n = n0 + ncol;
        if (kg == 0) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    float4 o = f2_four(acc[i][j]);
#pragma unroll
                    for (int g = 0; g < KS - 1; ++g) {
                        const float4 p = part[((g * TM + i) * NB + j) * GROUP + gt];
                        o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w;
                    }
                    const int m = m0 + mrow + i;
                    if (m < M && n + 32 * j < N) epi(z, r0 + m, n + 32 * j, o);
                }
        }
        if (KS > 1) __syncthreads();  // the partial sums are read before the next tile's copies land on them
    }
}

template <class C, bool TB, class Epi>
int sgemm_tile(const GemmShape &P, const Epi &epi, int max_ctas, int64_t tiles, cudaStream_t st) {
    auto kern = k_sgemm<C, TB, Epi>;
    const int rc = ensure_smem_attr((const void *)kern, C::smem(TB));
    if (rc) return rc;
    const int64_t grid = tiles < max_ctas ? tiles : (max_ctas > 0 ? max_ctas : 1);
    launch(kern, dim3((unsigned)grid, 1, P.nclass), C::THREADS, C::smem(TB), st, P, epi);
    count_launch();
    TNET_LAUNCH_CHECK();
    return TNET_OK;
}

// Host launcher.  Persistent grid, sized from the capacity.
// max_ctas: size of the persistent grid (a tuning knob: SMs x CTAs per SM)
template <bool TB, class Epi>
inline int sgemm(const GemmShape &P, const Epi &epi, int max_ctas, int sms, cudaStream_t st) {
    using Large = SgTile<8, 2, 4, 2, 1, 3, 2>;  // 128 x 128
    using Wide = SgTile<8, 2, 4, 1, 1, 3, 4>;   // 128 x 64
    using Mid = SgTile<4, 1, 4, 1, 2, 4, 4>;    // 64 x 32, K shared by two groups
    using Small = SgTile<4, 1, 2, 1, 4, 4, 4>;  // 32 x 32, K shared by four
    int maxM = 0;
    for (int z = 0; z < P.nclass; ++z) maxM = P.M[z] > maxM ? P.M[z] : maxM;
    if (maxM <= 0 || P.N <= 0) return TNET_OK;
    if (P.K % 8 || P.N % 4) return TNET_ERR_ARG;
    // tiles over all classes, and of the largest class (the launch's grid.x)
    auto tiles = [&](int bm, int bn, int64_t &widest) {
        int64_t all = 0;
        widest = 0;
        for (int z = 0; z < P.nclass; ++z) {
            const int64_t t = (int64_t)((P.M[z] + bm - 1) / bm) * ((P.N + bn - 1) / bn);
            all += t;
            widest = t > widest ? t : widest;
        }
        return all;
    };
    // The largest tile that still gives every SM its share: 128 x 128 with two
    // tiles per SM (27,000 x 128 x 128 has 211 tiles: 28.8 us against 24.6 with
    // 128 x 64), 128 x 64 with about one (3,000 x 384 x 256, 144 tiles: 19.3 us
    // against 20.6 and 22.6 with the two below; 3,000 x 256 x 128, 96 tiles: 12.3
    // against 10.4), 64 x 32 with two (3,000 x 128 x 384, 188 tiles: 16.5 us
    // against 14.4), else 32 x 32.  At most 32 columns: never the wide tiles.
    int64_t w;
    if (P.N > 64 && tiles(128, 128, w) >= 2LL * sms) return sgemm_tile<Large, TB>(P, epi, max_ctas, w, st);
    if (P.N > 32 && 8 * tiles(128, 64, w) >= 7LL * sms) return sgemm_tile<Wide, TB>(P, epi, max_ctas, w, st);
    if (tiles(64, 32, w) >= 2LL * sms) return sgemm_tile<Mid, TB>(P, epi, max_ctas, w, st);
    tiles(32, 32, w);
    return sgemm_tile<Small, TB>(P, epi, max_ctas, w, st);
}

inline GemmShape gshape(int M, int N, int K, const float *A, int64_t lda, const float *B, int64_t ldb) {
    GemmShape P{};
    P.M[0] = M;
    P.row0[0] = 0;
    P.rows_dev = nullptr;
    P.rows_mul = 1;
    P.N = N;
    P.K = K;
    P.A = A;
    P.lda = lda;
    P.B = B;
    P.ldb = ldb;
    P.strideB = 0;
    P.nclass = 1;
    return P;
}

// The three coordinate classes of a node tensor buffer with N atoms:
// I rows [0, N), A rows [N, 4N), S rows [4N, 9N); weights W[3][F][F].
inline GemmShape gshape_classes(int N, int F, const float *A, const float *W) {
    GemmShape P{};
    P.M[0] = N; P.M[1] = 3 * N; P.M[2] = 5 * N;
    P.row0[0] = 0; P.row0[1] = N; P.row0[2] = 4LL * N;
    P.rows_dev = nullptr;
    P.rows_mul = 1;
    P.N = F;
    P.K = F;
    P.A = A;
    P.lda = F;
    P.B = W;
    P.ldb = F;
    P.strideB = (int64_t)F * F;
    P.nclass = 3;
    return P;
}

}  // namespace tnet
