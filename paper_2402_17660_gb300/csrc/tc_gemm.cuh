// Tensor-core GEMM for sm_103a: TMA tile loads into 128B-swizzled shared
// memory, tcgen05.mma issued by one elected lane with the FP32 accumulator in
// tensor memory (TMEM), and a tcgen05.ld epilogue that applies the same fused
// epilogue functors as the SIMT path, or hands a bias-only result to bulk
// tensor stores.
//
//   C[m][n] = epi( sum_k A[m][k] B[n][k] ),  A [rows][lda], B [rows][ldb},
//   both K-major (row-major with K contiguous).
//
// Two operand modes:
//   BF16   A, B bf16; one kind::f16 MMA per k-step.
//   TF32X3 fp32 A and the weights' TF32 split B = B_hi + B_lo (two fp32
//          arrays of TF32-representable values, see tf32_split); three
//          kind::tf32 MMAs per k-step, A_hi B_hi + A_lo B_hi + A_hi B_lo,
//          within about 3 * 2^-22 |a||b| per product of the fp32 product.
//          A's split is formed on the SM by converter warps: into TMEM for
//          tiles up to 192 columns, else each landed A tile is rewritten into
//          A_hi (in place) and A_lo (a second buffer) at the same byte offsets
//          (an elementwise map, so the swizzle carries over); they fence it
//          and release the stage to the MMA warp.  No split of an activation
//          ever goes through HBM.
//
// Persistent CTAs walk 128 x BN output tiles.  Warp 0 issues TMA loads into a
// shared-memory ring of 3 to 6 stages (k-blocks of 128-byte rows for BF16 and
// for 3xTF32 with A's split in TMEM; 64-byte rows for 3xTF32 with the split in
// shared memory, whose stage holds A, A_lo, B and B_lo), warp 1 owns TMEM and
// issues the MMAs (32-byte k-steps) into one of two accumulators, so the
// epilogue of a tile overlaps the MMAs of the next.  Sixteen epilogue warps
// (eight for 3xTF32 tiles but the num_rbf-deep ones) drain TMEM (warp w reads
// lanes 32*(w%4) .. +31, a quarter (half) of the tile's columns each) and run
// the fused epilogue.  Every mbarrier wait is bounded;
// on expiry the kernel records TNET_ERR_TIMEOUT, the other roles stop, the
// producer waits (bounded) for its own copies in flight, TMEM is freed and
// the kernel returns.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>
#include <utility>
#include <vector>

#include "internal.cuh"

namespace tnet {
namespace tc {

constexpr int BM = 128;
constexpr int STG_LD = 20;  // floats per staged row (16 + pad, keeps float4 alignment)
constexpr uint32_t kSpinLimit = 1u << 22;

struct TcShape {
    int M[3];                 // rows per class (capacity when rows_dev is set)
    int64_t row0[3];          // first row of each class in A and in the output
    int64_t brow0[3];         // first row of each class's weights in B
    const int32_t *rows_dev;  // optional device row count (class 0), times rows_mul
    int rows_mul;
    int N, K, nclass;
    // testing only (zero in every library call): a smaller bound on each
    // mbarrier wait, and an MMA issuer that issues nothing, so that the
    // bounded waits run out with no MMA and no unconsumed copy in flight
    uint32_t spin_limit;
    int skip_mma;
    // 3xTF32: the operand is SiLU(A) (the converter warps apply silu_f to each
    // landed element before the split), so a layer's activation need not be
    // stored beside its pre-activation
    int a_silu;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// bounded wait on the given phase parity; false when the limit (kSpinLimit
// tries unless `limit` is given) ran out or, when given, the CTA's abort flag
// was raised
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag = nullptr,
                                          uint32_t limit = 0) {
    const uint32_t addr = smem_u32(bar);
    const uint32_t n = limit ? limit : kSpinLimit;
    for (uint32_t it = 0; it < n; ++it) {
        if (abort_flag && (it & 1023u) == 1023u && *abort_flag) return false;
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(addr), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// the same for a converged warp: the verdict is the warp's, in a uniform register
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                               uint32_t limit) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, limit));
}
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The producer's and the MMA issuer's instructions take the elected lane as a
// predicate instead of standing in an `if (lane == 0)`: the warp stays
// converged, so descriptors, coordinates and addresses are computed and held in
// uniform registers, which these instructions read.  In a divergent branch every
// operand went through a vector register first: 85-105 cycles an MMA, whatever
// its width, where one of 32 columns takes 16 and one of 192 takes 96.
__device__ __forceinline__ uint32_t elect_lane() {
    uint32_t p;
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
    return p;
}
__device__ __forceinline__ void expect_tx_if(uint32_t lead, uint64_t *bar, uint32_t bytes) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(
            smem_u32(bar)),
        "r"(bytes), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d_if(uint32_t lead, void *dst, const CUtensorMap *map, int x, int y,
                                               uint64_t *bar) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n @q "
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n}\n" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar)), "r"(lead)
        : "memory");
}
// D (TMEM) (+)= A (smem desc) * B (smem desc)^T, kind::f16 with bf16 inputs
__device__ __forceinline__ void umma_bf16(uint32_t lead, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q "
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accum), "r"(lead)
        : "memory");
}
// the mbarrier arrives once all previously issued MMAs of this thread complete
__device__ __forceinline__ void umma_commit(uint32_t lead, uint64_t *bar) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n @q "
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar)),
        "r"(lead)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor: K-major tile with ROW-byte rows (128 or
// 64) stored in the matching swizzle layout TMA writes; 8-row groups 8 * ROW
// bytes apart.  Swizzle codes: 2 = 128-byte, 4 = 64-byte.
template <int ROW>
__device__ __forceinline__ uint64_t sdesc_sw(uint32_t saddr) {
    static_assert(ROW == 128 || ROW == 64, "row bytes");
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);         // start address / 16
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)((8 * ROW) >> 4) << 32;           // stride byte offset: 8 rows
    d |= (uint64_t)1 << 46;                          // descriptor version for tcgen05
    d |= (uint64_t)(ROW == 128 ? 2 : 4) << 61;       // swizzle mode
    return d;
}

// Instruction descriptor: D f32, A and B bf16 (format 1) or tf32 (format 2),
// both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D (TMEM) (+)= A * B^T, kind::tf32 (fp32 containers read as TF32)
__device__ __forceinline__ void umma_tf32(uint32_t lead, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q "
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accum), "r"(lead)
        : "memory");
}
// The same with A in TMEM: row m of A in lane m, one TF32 element of K per
// 32-bit column (8 columns per k-step)
__device__ __forceinline__ void umma_tf32_at(uint32_t lead, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q "
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accum), "r"(lead)
        : "memory");
}
// this thread's 16 consecutive 32-bit columns of its TMEM lane
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float v[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
        "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
        "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])),
        "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])),
        "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
        : "memory");
}

template <int BN, bool X3 = false, bool NK = false, bool BULK = false>
struct TileCfg {
    // 3xTF32 at BN <= 192 (K beyond two k-blocks): A's split goes to TMEM
    // instead of shared memory.  A set of four converter warps (one per TMEM
    // lane quadrant; two sets, see CONV) reads each landed A row, splits it and
    // stores A_hi and A_lo with tcgen05.st into a slot of columns after the two accumulators; the MMAs
    // then read only B from shared memory, and the stage needs no A_lo buffer.
    // The narrow tiles (32 or 64 output columns, whose k-blocks carry little
    // MMA work) gain most: their pace is set by splitting A.
    static constexpr bool A_TMEM = X3 && !NK && BN <= 192;
    // one k-block is ROW bytes of K per row: 64 bf16 or 32 fp32 (128-byte
    // rows), or 16 fp32 (64-byte rows) for 3xTF32 with A's split in shared
    // memory, whose stage holds A, A_lo, B and B_lo.  With A in TMEM the
    // 128-byte k-block halves the TMA rows, barrier round trips and loads
    // issued per MMA against 64-byte ones.
    static constexpr int ROW = (X3 && !A_TMEM) ? 64 : 128;
    static constexpr int BKE = ROW / (X3 ? 4 : 2);
    static constexpr int KSTEPS = ROW / 32;  // MMA k-steps (32 bytes of K) per k-block
    static constexpr uint32_t A_BYTES = BM * ROW;
    static constexpr uint32_t B_BYTES = BN * ROW;
    // bytes TMA brings per pipeline stage: A, B (+ B_lo for TF32X3; A_lo is
    // formed in shared memory or TMEM)
    static constexpr uint32_t STAGE_TX = A_BYTES + (X3 ? 2 : 1) * B_BYTES;
    // Converter warps.  A k-block's split takes four warps 780-1,370 cycles (with
    // SiLU), longer than its MMAs: with A in TMEM two sets of four take the
    // k-blocks in turn; in shared memory four warps share each (two for NK,
    // whose epilogue is the longer).  Per call at 96,000 atoms, before and after:
    // radial layer 3 (192) 4.04 -> 3.85 ms, its adjoint (256) 4.55 -> 4.25, the
    // 32-wide GEMMs 1.64 -> 1.50; eight in shared memory 4.33.
    static constexpr int CONV = A_TMEM ? 8 : (X3 && !NK ? 4 : 2);
    static constexpr int CONV_ARRIVE = A_TMEM ? 4 : CONV;  // converter warps per stage
    // A_TMEM: slot a holds a k-block's A_hi (ROW / 4 columns) then A_lo at
    // A_COL + a * A_SLOT_COLS; the slots fill TMEM beside the accumulators
    // (2 at BN = 192, 4 at 128) and are released by their own commit barriers
    static constexpr uint32_t A_COL = 2 * BN;
    static constexpr int A_SLOT_COLS = 2 * (ROW / 4);
    static constexpr int A_SLOTS = A_TMEM ? ((512 - 2 * BN) / A_SLOT_COLS > 4 ? 4 : (512 - 2 * BN) / A_SLOT_COLS) : 1;
    static constexpr uint32_t TMEM_COLS =
        A_TMEM ? 512 : (2 * BN <= 64 ? 64 : 2 * BN <= 128 ? 128 : 2 * BN <= 256 ? 256 : 512);
    // epilogue warps: 16, or 8 for 3xTF32, where the freed transpose buffers
    // make room for a deeper pipeline; NK (a K of at most two k-blocks, whose
    // epilogue outweighs its MMAs) keeps 16 and 4 stages
    static constexpr int EPI = (X3 && !NK && (BN >= 128 || A_TMEM)) ? 8 : 16;
    static constexpr int THREADS = 64 + 32 * (EPI + CONV);
    // epilogue buffers per warp: two bulk-store tiles, or a transpose (and no
    // more: the BF16 layer-3 adjoint, whose epilogue reads through L1, took
    // 0.81 ms a call instead of 0.67 at 24,000 atoms with 4 KB each)
    static constexpr int WARP_STAGE = BULK ? 4096 : 32 * STG_LD * 4;
    static constexpr uint32_t STAGE_BYTES = EPI * WARP_STAGE;
    // 3xTF32 with the split in shared memory (BN = 256, and NK): as many
    // 64-byte stages as fit beside the epilogue buffers, which is 4 at 256, and
    // 4 for NK.
    static constexpr int X3_FIT = (int)((232448 - 1024 - 1024 - STAGE_BYTES) / (STAGE_TX + A_BYTES));
    // A_TMEM: as many 128-byte stages as fit, at most four (six for the
    // narrow tiles, which stream A).  BF16: four stages (three at BN = 256,
    // where four do not fit beside the epilogue buffers)
    static constexpr int A_FIT = (int)((232448 - 1024 - 1024 - STAGE_BYTES) / STAGE_TX);
    static constexpr int A_CAP = BN <= 64 ? 6 : 4;
    static constexpr int STAGES = A_TMEM ? (A_FIT > A_CAP ? A_CAP : A_FIT)
                                         : X3 ? (BN >= 128 && !NK ? (X3_FIT > 6 ? 6 : X3_FIT) : 4)
                                              : (BN >= 256 ? 3 : 4);
    static_assert(CONV == CONV_ARRIVE || (A_SLOTS % 2 == 0 && A_SLOTS <= STAGES), "a converter set could miss a phase");
    static_assert(!A_TMEM || (A_SLOTS >= 2 && A_COL + A_SLOT_COLS * A_SLOTS <= 512), "A slots exceed TMEM");
    static_assert(STAGES >= 2 && 8 * (3 * STAGES + 5 + A_SLOTS) + 8 <= 256, "pipeline barriers exceed their block");
    static constexpr size_t SMEM =
        1024 + STAGES * (size_t)(STAGE_TX + (X3 && !A_TMEM ? A_BYTES : 0)) + 1024 + STAGE_BYTES;
    static_assert(SMEM <= 232448, "dynamic shared memory above 227 KB");
};

// Tile index -> (class, first row, first column); false past the last tile.
// Scalars and selects only: dynamically indexed arrays would live in local memory.
struct TileIter {
    int tilesN, nclass, mt0, mt1, mt2;
    __device__ __forceinline__ bool get(int t, int &z, int &m0, int &n0, int BN_) const {
        const int c0 = mt0 * tilesN, c1 = mt1 * tilesN, c2 = mt2 * tilesN;
        if (t < c0) z = 0;
        else if (nclass > 1 && t < c0 + c1) { z = 1; t -= c0; }
        else if (nclass > 2 && t < c0 + c1 + c2) { z = 2; t -= c0 + c1; }
        else return false;
        m0 = (t / tilesN) * BM;
        n0 = (t % tilesN) * BN_;
        return true;
    }
};
__device__ __forceinline__ int64_t sel3(int z, int64_t a, int64_t b, int64_t c) { return z == 0 ? a : (z == 1 ? b : c); }

template <int BN, class Epi, bool X3, bool NK = false>
__global__ void __launch_bounds__(TileCfg<BN, X3, NK, Epi::BULK>::THREADS, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmAlo, const __grid_constant__ CUtensorMap tmBlo,
              const __grid_constant__ CUtensorMap tmC, TcShape P, Epi epi, int32_t *status) {
    pdl_entry();
    using C = TileCfg<BN, X3, NK, Epi::BULK>;
    constexpr int STAGES = C::STAGES;
    constexpr int BK = C::BKE;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    // stage s: A at sA + s*A_BYTES, B at sB + s*B_BYTES; TF32X3 adds A_lo, B_lo
    uint8_t *sA = smem;
    uint8_t *sB = smem + STAGES * C::A_BYTES;
    uint8_t *sAlo = sB + STAGES * C::B_BYTES;
    uint8_t *sBlo = sAlo + (X3 && !C::A_TMEM ? STAGES * C::A_BYTES : 0);
    uint64_t *full = (uint64_t *)(sBlo + (X3 ? STAGES * C::B_BYTES : 0));
    uint64_t *empty = full + STAGES;
    uint64_t *acc_full = empty + STAGES;
    uint64_t *acc_empty = acc_full + 2;
    uint64_t *conv = acc_empty + 2;  // TF32X3: A_lo of the stage is ready
    uint64_t *drain = conv + STAGES;  // every MMA the issuer started has retired
    uint64_t *aempty = drain + 1;     // A_TMEM: the MMAs that read TMEM A slot a retired
    uint32_t *tmem_slot = (uint32_t *)(aempty + C::A_SLOTS);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    float *stage_all = (float *)((uint8_t *)full + 1024);

    // rows per class (class 0 may be bounded by a device-side count)
    int M0 = P.M[0];
    const int M1 = P.nclass > 1 ? P.M[1] : 0, M2 = P.nclass > 2 ? P.M[2] : 0;
    if (P.rows_dev) {
        const int md = *P.rows_dev * P.rows_mul;
        M0 = md < M0 ? md : M0;
    }
    M0 = __shfl_sync(0xffffffffu, M0, 0);  // (uniform registers: see elect_lane)
    TileIter it;
    it.tilesN = (P.N + BN - 1) / BN;
    it.nclass = P.nclass;
    it.mt0 = (M0 + BM - 1) / BM;
    it.mt1 = (M1 + BM - 1) / BM;
    it.mt2 = (M2 + BM - 1) / BM;
    const int nk = (P.K + BK - 1) / BK;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t lim = P.spin_limit;
    const int t_first = blockIdx.x, t_step = gridDim.x;
    auto next_tile = [&](int t, int &z, int &m0, int &n0) { return it.get(t, z, m0, n0, BN); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
            mbar_init(&conv[s], C::CONV_ARRIVE);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], C::EPI);
        }
        mbar_init(drain, 1);
        for (int a = 0; a < C::A_SLOTS; ++a) mbar_init(&aempty[a], 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tmem_slot, C::TMEM_COLS);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    if (warp == 0) {  // TMA producer
        const uint32_t lead = elect_lane();
        int kg = 0;
        int z, m0, n0;
        bool ok = true;
        for (int t = t_first; ok && next_tile(t, z, m0, n0); t += t_step) {
            const int ya = (int)(sel3(z, P.row0[0], P.row0[1], P.row0[2]) + m0);
            const int yb = (int)(sel3(z, P.brow0[0], P.brow0[1], P.brow0[2]) + n0);
            for (int kb = 0; kb < nk; ++kb, ++kg) {
                const int s = kg % STAGES;
                if (kg >= STAGES && !mbar_wait_warp(&empty[s], ((kg / STAGES) - 1) & 1, abort_flag, lim)) {
                    set_status(status, TNET_ERR_TIMEOUT);
                    *abort_flag = 1;
                    ok = false;
                    break;
                }
                expect_tx_if(lead, &full[s], C::STAGE_TX);
                tma_load_2d_if(lead, sA + s * C::A_BYTES, &tmA, kb * BK, ya, &full[s]);
                tma_load_2d_if(lead, sB + s * C::B_BYTES, &tmB, kb * BK, yb, &full[s]);
                if (X3) tma_load_2d_if(lead, sBlo + s * C::B_BYTES, &tmBlo, kb * BK, yb, &full[s]);
            }
        }
        // own copies must land before the CTA exits: a wait that runs out is
        // recorded and taken up again (bounded) on the same barrier
        for (int k = kg > STAGES ? kg - STAGES : 0; k < kg; ++k) {
            bool landed = false;
            for (int r = 0; r < 64 && !landed; ++r) {
                landed = mbar_wait_warp(&full[k % STAGES], (k / STAGES) & 1, nullptr, lim);
                if (!landed) set_status(status, TNET_ERR_TIMEOUT);
            }
        }
    } else if (warp == 1) {  // MMA issuer (one lane issues, the same throughout)
        const uint32_t lead = elect_lane();
        const uint32_t idesc = X3 ? idesc_tf32(BM, BN) : idesc_bf16(BM, BN);
        const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB), sAlo0 = smem_u32(sAlo), sBlo0 = smem_u32(sBlo);
        int kg = 0, lt = 0;
        int z, m0, n0;
        bool ok = true;
        for (int t = t_first; ok && !P.skip_mma && next_tile(t, z, m0, n0); t += t_step, ++lt) {
            const int buf = lt & 1;
            if (lt >= 2 && !mbar_wait_warp(&acc_empty[buf], ((lt >> 1) - 1) & 1, abort_flag, lim)) {
                ok = false;
                break;
            }
            fence_after();
            const uint32_t d = tmem + (uint32_t)(buf * BN);
            for (int kb = 0; kb < nk; ++kb, ++kg) {
                const int s = kg % STAGES;
                if (!mbar_wait_warp(&full[s], (kg / STAGES) & 1, abort_flag, lim) ||
                    (X3 && !mbar_wait_warp(&conv[s], (kg / STAGES) & 1, abort_flag, lim))) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint64_t da = sdesc_sw<C::ROW>(sA0 + s * C::A_BYTES), db = sdesc_sw<C::ROW>(sB0 + s * C::B_BYTES);
                const uint64_t dal = sdesc_sw<C::ROW>(sAlo0 + s * C::A_BYTES);
                const uint64_t dbl = sdesc_sw<C::ROW>(sBlo0 + s * C::B_BYTES);
                // slot kg mod A_SLOTS: A_hi, then A_lo ROW / 4 columns further
                const uint32_t ah = tmem + C::A_COL + (uint32_t)(C::A_SLOT_COLS * (kg % C::A_SLOTS));
                // 32-byte k-steps: four per 128-byte k-block, two per 64-byte one
                // (2 in the descriptors' 16-byte units)
#pragma unroll
                for (int k = 0; k < C::KSTEPS; ++k) {
                    const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
                    if constexpr (C::A_TMEM) {
                        umma_tf32_at(lead, d, ah + 8 * k, db + 2 * k, idesc, acc);
                        umma_tf32_at(lead, d, ah + 8 * k + C::ROW / 4, db + 2 * k, idesc, 1u);
                        umma_tf32_at(lead, d, ah + 8 * k, dbl + 2 * k, idesc, 1u);
                    } else if (X3) {
                        umma_tf32(lead, d, da + 2 * k, db + 2 * k, idesc, acc);
                        umma_tf32(lead, d, dal + 2 * k, db + 2 * k, idesc, 1u);
                        umma_tf32(lead, d, da + 2 * k, dbl + 2 * k, idesc, 1u);
                    } else {
                        umma_bf16(lead, d, da + 2 * k, db + 2 * k, idesc, acc);
                    }
                }
                umma_commit(lead, &empty[s]);
                if constexpr (C::A_TMEM) umma_commit(lead, &aempty[kg % C::A_SLOTS]);
            }
            if (!ok) break;
            umma_commit(lead, &acc_full[buf]);
        }
        if (!ok) {
            set_status(status, TNET_ERR_TIMEOUT);
            *abort_flag = 1;
        }
        // on every path: all MMAs this thread issued retire before the
        // block frees TMEM (a wait that runs out is taken up again)
        umma_commit(lead, drain);
        bool retired = false;
        for (int r = 0; r < 64 && !retired; ++r) {
            retired = mbar_wait_warp(drain, 0, nullptr, lim);
            if (!retired) set_status(status, TNET_ERR_TIMEOUT);
        }
    } else if (warp >= 2 + C::EPI) {
        if (X3) {  // converters: A -> (A_hi, A_lo) for every stage, in k order
            const int ct = threadIdx.x - 32 * (2 + C::EPI);
            int kg = 0;
            bool ok = true;
            int z, m0, n0;
            for (int t = t_first; ok && next_tile(t, z, m0, n0) && !*abort_flag; t += t_step) {
                for (int kb = 0; kb < nk; ++kb, ++kg) {
                    const int s = kg % STAGES;
                    // two sets of converter warps take the k-blocks in turn
                    if (C::CONV > C::CONV_ARRIVE && (kg & 1) != ct / (32 * C::CONV_ARRIVE)) continue;
                    // The slot's last readers, the MMAs of k-block kg - A_SLOTS, must
                    // have retired.  Waited for first: a set that sees every
                    // other k-block skips every other use of a stage when STAGES is
                    // odd, and a parity wait on `full` tells its phase from the
                    // next but not from the one after; with A_SLOTS <= STAGES the
                    // retired MMAs show that the stage's last use is over.
                    const int a = kg % C::A_SLOTS;
                    if (C::A_TMEM && kg >= C::A_SLOTS &&
                        !mbar_wait(&aempty[a], ((kg / C::A_SLOTS) - 1) & 1, abort_flag, lim)) {
                        ok = false;
                        break;
                    }
                    if (!mbar_wait(&full[s], (kg / STAGES) & 1, abort_flag, lim)) {
                        ok = false;
                        break;
                    }
                    if constexpr (C::A_TMEM) {
                        // this lane's row of the tile (= its TMEM lane): 32 fp32
                        // in eight 16-byte chunks, chunk c stored at c ^ (r & 7)
                        // (TMA's 128-byte swizzle)
                        const int q = warp & 3, r = 32 * q + lane;
                        const float4 *row = reinterpret_cast<const float4 *>(sA + s * C::A_BYTES + r * C::ROW);
                        fence_after();
                        const uint32_t ta =
                            tmem + ((uint32_t)(32 * q) << 16) + C::A_COL + (uint32_t)(C::A_SLOT_COLS * a);
#pragma unroll
                        for (int h16 = 0; h16 < C::ROW / 64; ++h16) {  // 16 elements (four chunks) at a time
                            float h[16], l[16];
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                float4 v = row[(4 * h16 + c) ^ (r & 7)];
                                if (P.a_silu) {
                                    v.x = silu_f(v.x); v.y = silu_f(v.y); v.z = silu_f(v.z); v.w = silu_f(v.w);
                                }
                                tf32_split(v.x, h[4 * c], l[4 * c]);
                                tf32_split(v.y, h[4 * c + 1], l[4 * c + 1]);
                                tf32_split(v.z, h[4 * c + 2], l[4 * c + 2]);
                                tf32_split(v.w, h[4 * c + 3], l[4 * c + 3]);
                            }
                            tmem_st16(ta + 16 * h16, h);
                            tmem_st16(ta + C::ROW / 4 + 16 * h16, l);
                        }
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                        fence_before();
                    } else {
                        float4 *hi = reinterpret_cast<float4 *>(sA + s * C::A_BYTES);
                        float4 *lo = reinterpret_cast<float4 *>(sAlo + s * C::A_BYTES);
#pragma unroll 4
                        for (int i = ct; i < (int)(C::A_BYTES / 16); i += 32 * C::CONV) {
                            float4 v = hi[i], l;
                            if (P.a_silu) {
                                v.x = silu_f(v.x); v.y = silu_f(v.y); v.z = silu_f(v.z); v.w = silu_f(v.w);
                            }
                            tf32_split(v.x, v.x, l.x);
                            tf32_split(v.y, v.y, l.y);
                            tf32_split(v.z, v.z, l.z);
                            tf32_split(v.w, v.w, l.w);
                            hi[i] = v;
                            lo[i] = l;
                        }
                        // make the generic-proxy writes visible to the tensor core
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&conv[s]);
                }
            }
            if (!ok) {
                set_status(status, TNET_ERR_TIMEOUT);
                *abort_flag = 1;
            }
        }
    } else {  // epilogue warps 2 .. 2 + C::EPI - 1
        const int q = warp & 3;                  // TMEM lane quadrant this warp may read
        // column slices of at least 16 (one tcgen05.ld.x16); warps past the last
        // slice only take part in the accumulator hand-off
        constexpr int NSLICE = (BN / 16) < (C::EPI / 4) ? (BN / 16) : (C::EPI / 4);
        constexpr int CW = BN / NSLICE;
        const int part = (warp - 2) >> 2;
        const int c_begin = part < NSLICE ? part * CW : 0, c_end = part < NSLICE ? c_begin + CW : 0;
        int lt = 0;
        uint32_t n_bulk = 0;  // bulk stores of this warp so far
        int z, m0, n0;
        for (int t = t_first; next_tile(t, z, m0, n0) && !*abort_flag; t += t_step, ++lt) {
            const int buf = lt & 1;
            if (!mbar_wait(&acc_full[buf], (lt >> 1) & 1, abort_flag, lim)) {
                set_status(status, TNET_ERR_TIMEOUT);
                *abort_flag = 1;
                break;
            }
            fence_after();
            const int Mrow = (int)sel3(z, M0, M1, M2);
            const int64_t rbase = sel3(z, P.row0[0], P.row0[1], P.row0[2]);
            // TMEM gives thread = row; a shared-memory transpose hands each lane
            // 4 columns of 4 rows instead, so every store instruction of the
            // warp writes 8 rows x 64 contiguous bytes
            float *stg = stage_all + (warp - 2) * (C::WARP_STAGE / 4);
            const int rsub = lane >> 2, csub = (lane & 3) * 4;
            if constexpr (Epi::BULK) {
                // lane = row, as TMEM gives it: 16 columns at a time into one of
                // two 64-byte-swizzled tiles of 32 rows, written out by a bulk
                // tensor store.  The transposing path reads every value back and
                // stores it (56 LSU wavefronts a 2 KB block against 20), which
                // bound the GEMMs of small K.  Per call at 96,000 atoms, before
                // and after: projections 1.03 -> 0.78 ms, radial layer 1 0.75 ->
                // 0.50, layer 2 2.39 -> 1.50, layer 3 3.85 -> 3.80.  A last
                // group of fewer than 32 rows of its class is stored by the lanes.
                const int rows = Mrow - m0 - 32 * q;
#pragma unroll 1
                for (int c0 = c_begin; c0 < c_end; c0 += 16) {
                    const int n = n0 + c0;
                    float4 bias[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        bias[j] = epi.bias ? *reinterpret_cast<const float4 *>(epi.bias + (n + 4 * j < P.N ? n + 4 * j : P.N - 4))
                                           : make_float4(-0.f, -0.f, -0.f, -0.f);
                    float v[16];
                    tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * BN + c0), v);
                    if (rows <= 0 || n >= P.N) continue;
                    float4 w[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        w[j] = make_float4(v[4 * j] + bias[j].x, v[4 * j + 1] + bias[j].y, v[4 * j + 2] + bias[j].z,
                                           v[4 * j + 3] + bias[j].w);
                    const int64_t row0 = rbase + m0 + 32 * q;
                    if (rows < 32) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (lane < rows && n + 4 * j < P.N)
                                *reinterpret_cast<float4 *>(epi.C + (row0 + lane) * epi.ldc + n + 4 * j) = w[j];
                        continue;
                    }
                    uint8_t *tile = reinterpret_cast<uint8_t *>(stg) + (n_bulk++ & 1) * 2048;
                    // the store before the last has read this tile
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<float4 *>(tile + lane * 64 + 16 * (j ^ ((lane >> 1) & 3))) = w[j];
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        asm volatile(
                            "cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                (uint64_t)&tmC),
                            "r"(n), "r"((int)row0), "r"(smem_u32(tile))
                            : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            } else
#pragma unroll 1
            for (int c0 = c_begin; c0 < c_end; c0 += 16) {
                const int n = n0 + c0 + csub;
                // the epilogue's loads for this lane's 4 rows first (rows and
                // columns clamped into range), so they overlap the TMEM read
                typename Epi::Pre pr[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int row = m0 + 32 * q + rsub + 8 * k;
                    pr[k] = epi.pre(z, rbase + (row < Mrow ? row : Mrow - 1), n < P.N ? n : P.N - 4);
                }
                float v[16];
                tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * BN + c0), v);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<float4 *>(stg + lane * STG_LD + 4 * j) =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = rsub + 8 * k;
                    const int row = m0 + 32 * q + r;
                    const float4 w = *reinterpret_cast<const float4 *>(stg + r * STG_LD + csub);
                    if (row < Mrow && n < P.N) epi.post(z, rbase + row, n, w, pr[k]);
                }
                __syncwarp();
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
        // own stores complete before the CTA exits
        if (Epi::BULK && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

// ------------------------------------------------------------------ host ---
using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn tensor_map_encoder();  // resolved once through the runtime (tc_gemm.cu)

// 2-D tensor maps (bf16 or fp32): `rows` rows of `cols` elements, row pitch
// `ld` elements, box of `box_rows` x 128 bytes, 128B swizzle, zero fill.
int make_map_bf16(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int64_t ld, int box_rows);
int make_map_f32(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int64_t ld, int box_rows,
                 int row_bytes);

// Operands of one GEMM: A, B and (TF32X3 only) B's split: B = B_hi, Blo = B_lo.
struct TcOperands {
    const void *A, *B, *Blo;
    int64_t a_rows, lda, b_rows, ldb;
};

// Launches one persistent GEMM: min(tiles, sms) CTAs, one per SM (`sms` is
// the SM count of the device the stream runs on).
template <int BN, bool X3, bool NK = false, class Epi>
int tc_gemm_ops(const TcShape &P, const TcOperands &o, const Epi &epi, int32_t *status, cudaStream_t st, int sms) {
    using C = TileCfg<BN, X3, NK, Epi::BULK>;
    const int esz = X3 ? 4 : 2;
    int maxM = 0;
    for (int z = 0; z < P.nclass; ++z) maxM = P.M[z] > maxM ? P.M[z] : maxM;
    if (maxM <= 0 || P.N <= 0) return TNET_OK;
    if (P.N % 4 || (o.lda * esz) % 16 || (o.ldb * esz) % 16 || ((uintptr_t)o.A & 15) || ((uintptr_t)o.B & 15))
        return TNET_ERR_ARG;
    if (X3 && (!o.Blo || ((uintptr_t)o.Blo & 15))) return TNET_ERR_ARG;
    CUtensorMap ma, mb, mal, mbl, mc;
    int rc;
    auto kern = k_tc_gemm<BN, Epi, X3, NK>;
    if ((rc = ensure_smem_attr((const void *)kern, (int)C::SMEM))) return rc;
    if (sms < 1) sms = 1;
    if (X3) {
        if ((rc = make_map_f32(&ma, o.A, o.a_rows, P.K, o.lda, BM, C::ROW))) return rc;
        if ((rc = make_map_f32(&mb, o.B, o.b_rows, P.K, o.ldb, BN, C::ROW))) return rc;
        if ((rc = make_map_f32(&mbl, o.Blo, o.b_rows, P.K, o.ldb, BN, C::ROW))) return rc;
        mal = ma;  // unused: A_lo is formed in shared memory or TMEM
    } else {
        if ((rc = make_map_bf16(&ma, o.A, o.a_rows, P.K, o.lda, BM))) return rc;
        if ((rc = make_map_bf16(&mb, o.B, o.b_rows, P.K, o.ldb, BN))) return rc;
        mal = ma;
        mbl = mb;
    }
    mc = ma;  // unused unless the epilogue stores in bulk
    if constexpr (Epi::BULK) {
        int64_t rows = 0;
        for (int z = 0; z < P.nclass; ++z) rows = P.row0[z] + P.M[z] > rows ? P.row0[z] + P.M[z] : rows;
        if (P.N % 4 || ((uintptr_t)epi.C & 15) || epi.ldc % 4) return TNET_ERR_ARG;
        if ((rc = make_map_f32(&mc, epi.C, rows, P.N, epi.ldc, 32, 64))) return rc;
    }
    int64_t tiles = 0;
    for (int z = 0; z < P.nclass; ++z) tiles += (int64_t)((P.M[z] + BM - 1) / BM) * ((P.N + BN - 1) / BN);
    launch(kern, (unsigned)(tiles < sms ? tiles : sms), C::THREADS, C::SMEM, st, ma, mb, mal, mbl, mc, P, epi, status);
    count_launch();
    TNET_LAUNCH_CHECK();
    return TNET_OK;
}

template <int BN, class Epi>
int tc_gemm(const TcShape &P, const __nv_bfloat16 *A, int64_t a_rows, int64_t lda, const __nv_bfloat16 *B,
            int64_t b_rows, int64_t ldb, const Epi &epi, int32_t *status, cudaStream_t st, int sms) {
    return tc_gemm_ops<BN, false>(P, TcOperands{A, B, nullptr, a_rows, lda, b_rows, ldb}, epi, status, st, sms);
}

inline TcShape tshape(int M, int N, int K) {
    TcShape P{};
    P.M[0] = M;
    P.rows_mul = 1;
    P.N = N;
    P.K = K;
    P.nclass = 1;
    return P;
}

// The three coordinate classes of a node tensor buffer with N atoms (rows
// [0,N), [N,4N), [4N,9N)) against weights stacked [3][F][F].
inline TcShape tshape_classes(int Natoms, int F) {
    TcShape P{};
    P.M[0] = Natoms; P.M[1] = 3 * Natoms; P.M[2] = 5 * Natoms;
    P.row0[0] = 0; P.row0[1] = Natoms; P.row0[2] = 4LL * Natoms;
    P.brow0[0] = 0; P.brow0[1] = F; P.brow0[2] = 2LL * F;
    P.rows_mul = 1;
    P.N = F;
    P.K = F;
    P.nclass = 3;
    return P;
}

}  // namespace tc
}  // namespace tnet
