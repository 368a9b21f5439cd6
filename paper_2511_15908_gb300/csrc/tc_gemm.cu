// tc_gemm.cu -- tcgen05 BF16 GEMMs fed by TMA through an mbarrier ring (see tc_gemm.cuh for the
// roles and the layout).
#include <cstring>

#include <cuda.h>

#include "sph_internal.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace sphgb {

namespace {

using namespace tcx;

constexpr int kStageA = kTcM * kTcKChunk * 2;          // 16 KB: 128 rows x 128 B
constexpr int kStageB = kTcMaxN * kTcKChunk * 2;       // 32 KB: up to 256 rows x 128 B
constexpr int kStageBytes = kStageA + kStageB;
// the ring, 1 KB of slack to align it to the 1024-byte swizzle period, and the barriers
constexpr int kSmemBytes = kTcStages * kStageBytes + 1024 + 256;

struct TcGroup {
    CUtensorMap a[kTcGroup], b[kTcGroup];
    TcGemm g[kTcGroup];
    int ntile[kTcGroup], cps[kTcGroup];   // columns per tile, K chunks per slice
    int first[kTcGroup + 1];              // the GEMM's first block
    int count;
    unsigned *status;
};

__global__ void __launch_bounds__(kTcThreads, 1) k_tc_gemm(const __grid_constant__ TcGroup group)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    chain_enter();
    int w = 0;
    while (w + 1 < group.count && (int)blockIdx.x >= group.first[w + 1]) ++w;
    const TcGemm &g = group.g[w];
    const int ntile = group.ntile[w], box_b = ntile;
    const int mt = (g.M + kTcM - 1) / kTcM, ct = (g.N + ntile - 1) / ntile;
    const int blk = (int)blockIdx.x - group.first[w];
    const int bm = blk % mt, bn = blk / mt % ct, bz = blk / mt / ct;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar = base + kTcStages * kStageBytes;   // full[S], empty[S], done
    auto full = [&](int s) { return bar + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar + 8u * (uint32_t)(kTcStages + s); };
    const uint32_t done = bar + 16u * kTcStages;

    const int m0 = bm * kTcM;
    const int n0 = bn * ntile;
    const int nt_raw = min(ntile, g.N - n0);
    const int nt = (nt_raw + 15) & ~15;              // UMMA N: multiple of 16
    int ncols = 32;
    while (ncols < nt) ncols <<= 1;                  // TMEM allocation: power of two >= 32
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nk = (g.K + kTcKChunk - 1) / kTcKChunk;
    const int kc0 = bz * group.cps[w];
    const int kc1 = min(nk, kc0 + group.cps[w]);
    const int row = m0 + warp * 32 + lane;
    float *C = g.C + (size_t)bz * g.split_stride;

    if (kc0 >= kc1) {
        // an empty K slice (more slices than chunks): its partial sum is zero
        if (row < g.M)
            for (int j = 0; j < nt_raw; ++j) C[(size_t)row * g.ldc + n0 + j] = 0.0f;
        return;
    }

    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < 2 * kTcStages + 1; ++s) mbar_init(bar + 8u * (uint32_t)s);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;

    if (threadIdx.x == 0) {
        // producer: chunk i goes to stage i % S once the MMAs of chunk i - S have read it
        const uint32_t tx = (uint32_t)(kTcM + box_b) * kTcKChunk * 2;
        for (int kc = kc0, i = 0; kc < kc1; ++kc, ++i) {
            const int s = i % kTcStages;
            if (i >= kTcStages && !mbar_wait(empty(s), ((i / kTcStages) & 1) ^ 1)) {
                s_fail = 1;
                break;
            }
            const uint32_t sa = base + (uint32_t)s * kStageBytes;
            mbar_expect_tx(full(s), tx);
            tma_load_2d(sa, &group.a[w], kc * kTcKChunk, m0, full(s));
            tma_load_2d(sa + kStageA, &group.b[w], kc * kTcKChunk, n0, full(s));
        }
    } else if (threadIdx.x == 32) {
        // MMA issuer: four K = 16 steps per chunk into the TMEM accumulator
        const uint32_t idesc = instr_desc(nt);
        for (int kc = kc0, i = 0; kc < kc1; ++kc, ++i) {
            const int s = i % kTcStages;
            if (!mbar_wait(full(s), (i / kTcStages) & 1)) {
                s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t sa = base + (uint32_t)s * kStageBytes, sb = sa + kStageA;
#pragma unroll
            for (int j = 0; j < kTcKChunk / 16; ++j) {
                const uint64_t ad = smem_desc_sw128(sa + 32u * (uint32_t)j);
                const uint64_t bd = smem_desc_sw128(sb + 32u * (uint32_t)j);
                mma_bf16(tmem, ad, bd, idesc, (i > 0 || j > 0) ? 1u : 0u);
            }
            mma_commit(empty(s));
        }
        mma_commit(done);                            // fires once every issued MMA completed
    }
    __syncwarp();
    if (!mbar_wait(done, 0)) s_fail = 1;
    asm volatile("tcgen05.fence::after_thread_sync;");
    __syncthreads();
    if (s_fail) {
        if (threadIdx.x == 0 && group.status) atomicOr(group.status, (unsigned)ST_TIMEOUT);
    } else {
        // thread = tile row (TMEM lane 32 warp + lane), 16 columns per load
        const bool vec_c = (g.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0 && (n0 & 3) == 0;
        for (int c0 = 0; c0 < nt; c0 += 16) {
            uint32_t r[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
            if (row >= g.M) continue;
            float *cp = C + (size_t)row * g.ldc + n0 + c0;
            if (c0 + 16 <= nt_raw && vec_c) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    reinterpret_cast<uint4 *>(cp)[q] = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
            } else {
                for (int j = 0; j < 16 && c0 + j < nt_raw; ++j) cp[j] = __uint_as_float(r[j]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

}  // namespace

// Tensor map of a K-contiguous BF16 operand [rows][K] (leading dimension ld elements): boxes
// of 64 K x box_rows rows with the 128-byte swizzle; out-of-range elements read as zero.
bool tc_operand_map(CUtensorMap *map, const __nv_bfloat16 *p, int rows, int K, int ld, int box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2u};
    const cuuint32_t box[2] = {(cuuint32_t)kTcKChunk, (cuuint32_t)box_rows};
    const cuuint32_t estride[2] = {1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(p), dims, strides, box, estride,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Columns per CTA tile: the widest of 256, 128, ..., 16 that still gives at least
// kTcMinCtas CTAs (row tiles x column tiles x K slices).  These GEMMs are small: a CTA's
// epilogue (one thread per row, one warp per SM sub-partition) is latency bound, so more,
// narrower tiles finish sooner than few wide ones; A is re-read from L2 per column tile.
static int ntile_of(const TcGemm &g)
{
    const int mt = (g.M + kTcM - 1) / kTcM;
    int nt = kTcMaxN;
    while (nt > 16 && mt * ((g.N + nt - 1) / nt) * g.ksplit < kTcMinCtas) nt >>= 1;
    return nt;
}

cudaError_t tc_gemm_group(const TcGemm *g, int count, unsigned *status, cudaStream_t s)
{
    static std::atomic<unsigned long long> configured{0};
    {
        cudaError_t e = smem_opt_in(k_tc_gemm, kSmemBytes, configured);
        if (e != cudaSuccess) return e;
    }
    if (count < 1 || count > kTcGroup) return cudaErrorInvalidValue;
    TcGroup grp;
    std::memset(&grp, 0, sizeof grp);
    grp.count = count;
    grp.status = status;
    for (int i = 0; i < count; ++i) {
        const TcGemm &q = g[i];
        if (!q.A || !q.B || !q.C || q.M < 1 || q.N < 1 || q.K < 1 || q.ksplit < 1 || (q.lda & 7) || (q.ldb & 7) ||
            q.lda < q.K || q.ldb < q.K || (reinterpret_cast<uintptr_t>(q.A) & 15u) ||
            (reinterpret_cast<uintptr_t>(q.B) & 15u))
            return cudaErrorInvalidValue;
        grp.g[i] = q;
        grp.ntile[i] = ntile_of(q);
        grp.cps[i] = ((q.K + kTcKChunk - 1) / kTcKChunk + q.ksplit - 1) / q.ksplit;
        if (!tc_operand_map(&grp.a[i], q.A, q.M, q.K, q.lda, kTcM) ||
            !tc_operand_map(&grp.b[i], q.B, q.N, q.K, q.ldb, grp.ntile[i]))
            return cudaErrorInvalidValue;
        const int ct = (q.N + grp.ntile[i] - 1) / grp.ntile[i];
        grp.first[i + 1] = grp.first[i] + (q.M + kTcM - 1) / kTcM * ct * q.ksplit;
    }
    return launch_after(s != nullptr, k_tc_gemm, grp.first[count], kTcThreads, kSmemBytes, s, grp);
}

}  // namespace sphgb
