// Tensor-core kernels of the learned lattice-size / amplitude model of the
// amplitude scan: a BF16 GEMM on the 5th-generation tensor cores and the
// elementwise kernels of an MLP's forward and backward passes and its Adam
// update.
//
// gemm: C[M][N] (fp32) = A[M][K] . B[N][K]^T with A, B bf16 and K-major
// (row-major [rows][K]). One CTA of 128 threads computes a 128 x N tile
// (N <= 256, multiple of 16; M a multiple of 128, K of 16) over a range of
// K (split-K when the M tiles alone cannot fill the GPU):
//  * thread 0 streams 64-wide K chunks of A (128 rows) and B (N rows) into a
//    4-stage shared-memory ring with TMA (cp.async.bulk.tensor, 128-byte
//    swizzle), each stage completing on a transaction-count mbarrier;
//  * thread 32 issues four tcgen05.mma (K = 16 each) per stage into an FP32
//    accumulator in tensor memory and frees the stage with tcgen05.commit;
//  * after the last commit all 4 warps read the accumulator back with
//    tcgen05.ld and store it.
// Split-K partials go to a workspace and a second kernel adds them in split
// order (deterministic). Every mbarrier wait has an iteration limit, after
// which the CTA records an error, waits for its copies in flight, frees its
// tensor memory and exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "../../include/qmc.h"

#include "qmc_device_once.h"
#include "qmc_internal.h"

#define QMC_E_INVAL_LOCAL QMC_E_INVAL
#define QMC_E_CUDA_LOCAL QMC_E_CUDA

namespace {

constexpr int kGemmThreads = 128;
constexpr int kStages = 4;
constexpr int kBK = 64;                                  // K elements per stage: one 128-byte swizzle span
constexpr int kTileM = 128;
constexpr int kMaxN = 256;
constexpr int kAStageBytes = kTileM * kBK * 2;           // 16 KB
constexpr int kBStageBytes = kMaxN * kBK * 2;            // 32 KB
constexpr int kStageBytes = kAStageBytes + kBStageBytes;
constexpr int kGemmSmem = kStages * kStageBytes + 1024;  // + slack to align the ring to 1024 B
static_assert(4 * 32 * (kMaxN + 4) * 4 <= kStages * kStageBytes, "the epilogue's blocks fit the ring");
// Polls of one mbarrier wait before it gives up (with 64 ns sleeps: a few
// seconds). The pipeline's waits take their limit from the launch (this value
// unless a caller asks for fewer); the clean-up after a timeout always waits
// with this one, so that copies and MMAs in flight land before the CTA frees
// its tensor memory and exits.
constexpr unsigned kWaitLimit = 1u << 26;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor (tcgen05) of a K-major operand in the
// 128-byte-swizzled layout that TMA writes: start address, stride between
// 8-row core-matrix groups 1024 B, fixed field 0b001 at bit 46, swizzle mode
// 2 (128 B) at bit 61; the leading-dimension offset is unused for swizzled
// K-major operands (set to 1).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase, unsigned limit) {
    for (unsigned it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(phase)
            : "memory");
        if (done) return true;
        if (it > 64) __nanosleep(64);
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(mbar)
        : "memory");
}

__global__ void __launch_bounds__(kGemmThreads, 1)
qmc_gemm_bf16_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, float *C,
                 int N, int K, int chunks_per_split, size_t split_stride, unsigned *err, unsigned wait_limit) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ int issued, consumed;
    unsigned char *ring = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * kTileM;
    const int nchunks = (K + kBK - 1) / kBK;
    const int c0 = blockIdx.y * chunks_per_split;
    const int nc = min(nchunks, c0 + chunks_per_split) - c0;   // >= 1 by the host's split choice
    float *Cs = C + (size_t)blockIdx.y * split_stride;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kMaxN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::);
        issued = 0;
        consumed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::);
    const uint32_t tmem = tmem_base;
    const uint32_t bytes_stage = (uint32_t)((kTileM + N) * kBK * 2);
    bool ok = true;

    if (tid == 0) {
        // producer: TMA into the ring, each stage reused once the MMAs reading it committed
        for (int i = 0; i < nc; ++i) {
            const int s = i % kStages;
            if (i >= kStages && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((i / kStages - 1) & 1), wait_limit)) {
                ok = false;
                break;
            }
            const uint32_t fb = smem_u32(&full[s]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(bytes_stage)
                         : "memory");
            const uint32_t sa = smem_u32(ring + s * kStageBytes);
            tma_load_2d(sa, &mapA, (c0 + i) * kBK, m0, fb);
            tma_load_2d(sa + kAStageBytes, &mapB, (c0 + i) * kBK, 0, fb);
            issued = i + 1;
        }
    } else if (tid == 32) {
        // MMA issuer
        const uint32_t idesc = instr_desc_bf16(kTileM, N);
        for (int i = 0; i < nc; ++i) {
            const int s = i % kStages;
            if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((i / kStages) & 1), wait_limit)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::);
            const uint32_t sa = smem_u32(ring + s * kStageBytes);
#pragma unroll
            for (int ks = 0; ks < kBK / 16; ++ks) {
                const uint64_t da = smem_desc_sw128(sa + ks * 32);
                const uint64_t db = smem_desc_sw128(sa + kAStageBytes + ks * 32);
                const uint32_t acc = (i > 0 || ks > 0) ? 1u : 0u;
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "setp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
                    "l"(da), "l"(db), "r"(idesc), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&empty[s]))
                         : "memory");
            consumed = i + 1;
        }
        // completion of every MMA issued so far
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(&done))
                     : "memory");
    }
    if (!mbar_wait(smem_u32(&done), 0, wait_limit)) ok = false;
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::);
    if (ok) {
        // warp w owns TMEM lanes 32w..32w+31 = rows m0 + 32w + lane. A lane holds
        // a row's columns, so stores straight from it would touch 32 rows at a
        // time (2048 x 256 x 256: they took most of the kernel's 22 us); the
        // warp turns its 32 x N block through the ring, which every MMA has
        // finished reading, and writes whole rows (10 us). Row stride N + 4
        // floats: 16-byte stores of eight lanes cover all banks.
        const int ldw = N + 4;
        float *blk = reinterpret_cast<float *>(ring) + (size_t)warp * 32 * ldw;
        for (int c = 0; c < N; c += 16) {
            uint32_t r[16];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                "%13, %14, %15}, [%16];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15])
                : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int q = 0; q < 16; q += 4)
                *reinterpret_cast<uint4 *>(blk + lane * ldw + c + q) = make_uint4(r[q], r[q + 1], r[q + 2], r[q + 3]);
        }
        __syncwarp();
        float *dst = Cs + (size_t)(m0 + warp * 32) * N;
        const bool vec = (reinterpret_cast<uintptr_t>(Cs) & 15) == 0;
        for (int row = 0; row < 32; ++row) {
            const float *src = blk + row * ldw;
            if (vec) {
                for (int c = 4 * lane; c < N; c += 128)
                    *reinterpret_cast<float4 *>(dst + (size_t)row * N + c) = *reinterpret_cast<const float4 *>(src + c);
            } else {
                for (int c = lane; c < N; c += 32) dst[(size_t)row * N + c] = src[c];
            }
        }
    } else {
        if (tid == 0) {
            atomicAdd(err, 1u);
            // copies still in flight land before the CTA's shared memory goes
            // away, and the MMAs issued so far finish before the accumulator's
            // tensor memory is freed (the MMA thread always commits `done`)
            for (int i = consumed; i < issued; ++i)
                mbar_wait(smem_u32(&full[i % kStages]), (uint32_t)((i / kStages) & 1), kWaitLimit);
            mbar_wait(smem_u32(&done), 0, kWaitLimit);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::);
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kMaxN));
}

// sum over splits of W[s][i], in split order (the loads eight at a time)
__device__ __forceinline__ float split_sum(const float *W, int splits, size_t stride, size_t i) {
    float acc = W[i];
    int s = 1;
    for (; s + 8 <= splits; s += 8) {
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = W[(size_t)(s + q) * stride + i];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc += v[q];
    }
    for (; s < splits; ++s) acc += W[(size_t)s * stride + i];
    return acc;
}

// C = sum over splits of W[s] (in split order)
__global__ void qmc_gemm_splitk_sum(const float *W, int splits, size_t stride, float *C, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        C[i] = split_sum(W, splits, stride, i);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// 2-D bf16 tensor [rows][K] (row stride K), box {64, box_rows}, 128-byte swizzle,
// zero fill beyond K
bool make_map(CUtensorMap *map, const void *ptr, int rows, int K, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// split-K workspace, grown on demand (one per process; calls on one device)
struct SplitWorkspace {
    std::mutex mu;
    float *ptr = nullptr;
    size_t cap = 0;
};
SplitWorkspace &workspace() {
    static SplitWorkspace w;
    return w;
}

}  // namespace

namespace {
// Splits of K when the M tiles leave most SMs idle: at most
// gemm_splits_most (grows with K), each of `per` chunks, at least one
int gemm_splits_most(int M, int K, int sms) {
    return std::max(1, std::min((K + kBK - 1) / kBK, sms / (M / kTileM)));
}
int gemm_splits(int M, int K, int sms, int &per) {
    const int nchunks = (K + kBK - 1) / kBK, splits = gemm_splits_most(M, K, sms);
    per = (nchunks + splits - 1) / splits;
    return (nchunks + per - 1) / per;
}
int gemm_sms() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}
bool gemm_shape_ok(const void *A, const void *B, int M, int N, int K) {
    if (M <= 0 || M % 128 || K <= 0 || K % 16 || N < 16 || N > 256 || N % 16) return false;
    return ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
}
// The product's splits, split s at out + s M N
int gemm_launch(const void *A, const void *B, float *out, int M, int N, int K, int splits, int per, unsigned *err_dev,
                cudaStream_t stream, unsigned wait_limit) {
    static std::atomic<uint64_t> done{0};
    if (!qmc_allow_smem(done, qmc_gemm_bf16_tc, kGemmSmem)) return -1;
    CUtensorMap mapA, mapB;
    if (!make_map(&mapA, A, M, K, kTileM) || !make_map(&mapB, B, N, K, N)) return -1;
    qmc_gemm_bf16_tc<<<dim3(M / kTileM, splits), kGemmThreads, kGemmSmem, stream>>>(
        mapA, mapB, out, N, K, per, (size_t)M * N, err_dev, wait_limit);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
}  // namespace

// C[M][N] = A[M][K] B[N][K]^T, device pointers; M % 128 == 0, K % 16 == 0,
// N % 16 == 0 and 16 <= N <= 256; A, B 16-byte aligned; C rows contiguous
// (ldc = N). Split-K when the M tiles leave most SMs idle.
extern "C" int qmc_k_gemm_bf16_limit(const void *A, const void *B, float *C, int M, int N, int K, unsigned *err_dev,
                                     void *stream, unsigned wait_limit) {
    if (!gemm_shape_ok(A, B, M, N, K)) return -2;
    int per = 1;
    const int splits = gemm_splits(M, K, gemm_sms(), per);
    const size_t mn = (size_t)M * N;
    float *out = C;
    std::unique_lock<std::mutex> lock(workspace().mu, std::defer_lock);
    if (splits > 1) {
        lock.lock();
        SplitWorkspace &w = workspace();
        if (w.cap < (size_t)splits * mn) {
            cudaStreamSynchronize((cudaStream_t)stream);
            cudaFree(w.ptr);
            w.ptr = nullptr;
            w.cap = 0;
            if (cudaMalloc(&w.ptr, (size_t)splits * mn * sizeof(float)) != cudaSuccess) return -1;
            w.cap = (size_t)splits * mn;
        }
        out = w.ptr;
    }
    if (gemm_launch(A, B, out, M, N, K, splits, per, err_dev, (cudaStream_t)stream, wait_limit)) return -1;
    if (splits > 1) {
        const unsigned blocks = (unsigned)std::min<size_t>((mn + 255) / 256, 4096);
        qmc_gemm_splitk_sum<<<blocks, 256, 0, (cudaStream_t)stream>>>(out, splits, mn, C, mn);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

extern "C" int qmc_k_gemm_bf16(const void *A, const void *B, float *C, int M, int N, int K, unsigned *err_dev,
                               void *stream) {
    return qmc_k_gemm_bf16_limit(A, B, C, M, N, K, err_dev, stream, kWaitLimit);
}

extern "C" int qmc_gemm_bf16_device(const void *A, const void *B, float *C, int M, int N, int K, unsigned *err_dev,
                                    void *stream) {
    if (!A || !B || !C || !err_dev) return QMC_E_INVAL_LOCAL;
    const int rc = qmc_k_gemm_bf16(A, B, C, M, N, K, err_dev, stream);
    return rc == -2 ? QMC_E_INVAL_LOCAL : (rc ? QMC_E_CUDA_LOCAL : 0);
}

extern "C" int qmc_gemm_bf16_device_limit(const void *A, const void *B, float *C, int M, int N, int K,
                                          unsigned *err_dev, void *stream, unsigned wait_limit) {
    if (!A || !B || !C || !err_dev) return QMC_E_INVAL_LOCAL;
    const int rc = qmc_k_gemm_bf16_limit(A, B, C, M, N, K, err_dev, stream, wait_limit);
    return rc == -2 ? QMC_E_INVAL_LOCAL : (rc ? QMC_E_CUDA_LOCAL : 0);
}

// Host-buffer wrapper (tests and small callers): copies in, runs, copies out.
extern "C" int qmc_gemm_bf16(const uint16_t *A, const uint16_t *B, float *C, int M, int N, int K) {
    if (!A || !B || !C) return QMC_E_INVAL_LOCAL;
    if (M <= 0 || M % 128 || K <= 0 || K % 16 || N < 16 || N > 256 || N % 16) return QMC_E_INVAL_LOCAL;
    void *dA = nullptr, *dB = nullptr;
    float *dC = nullptr;
    unsigned *derr = nullptr;
    int rc = 0;
    if (cudaMalloc(&dA, (size_t)M * K * 2) || cudaMalloc(&dB, (size_t)N * K * 2) ||
        cudaMalloc(&dC, (size_t)M * N * 4) || cudaMalloc(&derr, 4)) {
        rc = QMC_E_CUDA_LOCAL;
    } else {
        cudaMemcpy(dA, A, (size_t)M * K * 2, cudaMemcpyHostToDevice);
        cudaMemcpy(dB, B, (size_t)N * K * 2, cudaMemcpyHostToDevice);
        cudaMemset(derr, 0, 4);
        if (qmc_k_gemm_bf16(dA, dB, dC, M, N, K, derr, nullptr)) rc = QMC_E_CUDA_LOCAL;
        unsigned herr = 0;
        if (cudaMemcpy(C, dC, (size_t)M * N * 4, cudaMemcpyDeviceToHost) != cudaSuccess) rc = QMC_E_CUDA_LOCAL;
        if (cudaMemcpy(&herr, derr, 4, cudaMemcpyDeviceToHost) != cudaSuccess || herr) rc = QMC_E_CUDA_LOCAL;
    }
    cudaFree(dA);
    cudaFree(dB);
    cudaFree(dC);
    cudaFree(derr);
    return rc;
}

// ============================================================================
// The MLP: x (nin) -> tanh(W0 x + b0) -> [tanh(Wk h + bk)] x (depth-1) -> Wout h + bout
// Layer 0 (K = nin, tiny) runs on the CUDA cores in FP32; every other layer and
// every weight/activation gradient product runs through qmc_gemm_bf16_tc with
// bf16 operands and FP32 accumulation. FP32 master weights, Adam in FP32.
// Batches are padded to a multiple of 128 rows with zero loss weight.
// ============================================================================
namespace {

__device__ __forceinline__ __nv_bfloat16 bf(float x) { return __float2bfloat16_rn(x); }

// The elementwise kernels below work on 32 x 32 tiles (blocks of 32 x 8
// threads): the bf16 operands are wanted in both orders, and the transposed one
// goes through shared memory so that both are written in whole segments (2-byte
// stores one row apart filled a sixteenth of each sector). They read the GEMM's splits themselves, in split order, instead of a pass
// that sums them first.
struct Splits {
    const float *W;
    int n;
    size_t stride;
    __device__ __forceinline__ float at(size_t i) const { return split_sum(W, n, stride, i); }
};
constexpr int kTile = 32, kTileRows = 8;
// f(b, o) -> value, stored bf16 as hb [Bp][N] and, through the tile, hbT [N][Bp];
// one block per tile, the columns' tiles of 32 rows side by side (a grid's
// first dimension alone has room for more than two million rows)
template <class F>
__device__ __forceinline__ void tile_both(int Bp, int N, __nv_bfloat16 *hb, __nv_bfloat16 *hbT, F f) {
    __shared__ __nv_bfloat16 tile[kTile][kTile + 2];
    const int across = (N + kTile - 1) / kTile;
    const int o0 = blockIdx.x % across * kTile, b0 = blockIdx.x / across * kTile;
    const int o = o0 + threadIdx.x;
#pragma unroll
    for (int r = 0; r < kTile; r += kTileRows) {
        const int b = b0 + threadIdx.y + r;
        if (b < Bp && o < N) {
            const __nv_bfloat16 v = bf(f(b, o));
            hb[(size_t)b * N + o] = v;
            tile[threadIdx.y + r][threadIdx.x] = v;
        }
    }
    __syncthreads();
    const int bt = b0 + threadIdx.x;
#pragma unroll
    for (int r = 0; r < kTile; r += kTileRows) {
        const int ot = o0 + threadIdx.y + r;
        if (bt < Bp && ot < N) hbT[(size_t)ot * Bp + bt] = tile[threadIdx.x][threadIdx.y + r];
    }
}

// h0 = tanh(x W0^T + b0): f32 [Bp][H], bf16 [Bp][H] and [H][Bp]
__global__ void mlp_layer0_fwd(const float *x, const float *W0, const float *b0, int nin, int H, int Bp,
                               float *h, __nv_bfloat16 *hb, __nv_bfloat16 *hbT) {
    tile_both(Bp, H, hb, hbT, [=](int b, int o) {
        float z = b0[o];
        for (int k = 0; k < nin; ++k) z = fmaf(W0[o * nin + k], x[b * nin + k], z);
        const float a = tanhf(z);
        h[(size_t)b * H + o] = a;
        return a;
    });
}

// h = tanh(C + bias) for a GEMM output C [Bp][N]
__global__ void mlp_bias_tanh(Splits C, const float *bias, int N, int Bp, float *h, __nv_bfloat16 *hb,
                              __nv_bfloat16 *hbT) {
    tile_both(Bp, N, hb, hbT, [=](int b, int o) {
        const size_t i = (size_t)b * N + o;
        const float z = tanhf(C.at(i) + bias[o]);
        h[i] = z;
        return z;
    });
}

// out = C + bias for a GEMM output C [Bp][ldc] (columns < N used)
__global__ void mlp_bias_out(Splits C, const float *bias, int N, int ldc, int Bp, float *h) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Bp * N) return;
    const int b = i / N, o = i % N;
    h[i] = C.at((size_t)b * ldc + o) + bias[o];
}

// weighted squared error: loss += wt_o mask_b (out - y)^2 / B; dout = 2 wt_o
// mask_b (out - y) / B. One atomic per block (one per element, all on one
// address, took 400 us for 2048 x 144).
__global__ void mlp_loss(const float *out, const float *y, const float *wt, const float *mask, int No, int Nop,
                         int Bp, float invB, __nv_bfloat16 *dob, __nv_bfloat16 *dobT, float *dof, double *loss) {
    __shared__ double part[kTileRows];
    double mine = 0.0;
    tile_both(Bp, Nop, dob, dobT, [=, &mine](int b, int o) {
        float g = 0.f;
        if (o < No) {
            const float r = out[(size_t)b * No + o] - y[(size_t)b * No + o];
            const float w = wt[o] * mask[b];
            g = 2.f * w * r * invB;
            if (w != 0.f) mine += (double)(w * r * r * invB);
        }
        dof[(size_t)b * Nop + o] = g;
        return g;
    });
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, off);
    if (threadIdx.x == 0) part[threadIdx.y] = mine;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        double v = 0.0;
        for (int w = 0; w < kTileRows; ++w) v += part[w];
        atomicAdd(loss, v);
    }
}

// dz = dh (1 - h^2) for tanh layers: bf16 [Bp][H], bf16 [H][Bp], f32 [Bp][H]
__global__ void mlp_tanh_bwd(Splits dh, const float *h, int H, int Bp, __nv_bfloat16 *dzb,
                             __nv_bfloat16 *dzbT, float *dzf) {
    tile_both(Bp, H, dzb, dzbT, [=](int b, int o) {
        const size_t i = (size_t)b * H + o;
        const float a = h[i];
        const float g = dh.at(i) * (1.f - a * a);
        dzf[i] = g;
        return g;
    });
}

// Column sums over the batch in a fixed order: column o's terms f(b, o) go to
// 256 partial sums by b mod 256, added in b order, then pairwise by halves.
// A block takes kCols neighbouring columns, so that a row's segment is read
// whole, and 1024 threads, each with eight rows' loads in flight.
constexpr int kCols = 8, kColThreads = 1024;
// add(s, v, b) folds the loaded v of row b into s
template <class A>
__device__ __forceinline__ void column_sums(const float *dz, int N, int ld, int Bp, A add, float *out, int stride) {
    __shared__ float red[256][kCols];
    const int c = threadIdx.x % kCols, o = blockIdx.x * kCols + c;
    for (int t = threadIdx.x / kCols; t < 256; t += kColThreads / kCols) {
        float s = 0.f;
        if (o < N)
            for (int b = t; b < Bp; b += 8 * 256) {
                float v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = b + 256 * q < Bp ? dz[(size_t)(b + 256 * q) * ld + o] : 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (b + 256 * q < Bp) s = add(s, v[q], b + 256 * q);
            }
        red[t][c] = s;
    }
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        for (int i = threadIdx.x; i < w * kCols; i += kColThreads)
            red[i / kCols][i % kCols] += red[i / kCols + w][i % kCols];
        __syncthreads();
    }
    if (threadIdx.x < kCols && o < N) out[(size_t)o * stride] = red[0][c];
}

// db[o] = sum_b dz[b][o]
__global__ void mlp_colsum(const float *dz, int N, int ld, int Bp, float *db) {
    column_sums(dz, N, ld, Bp, [](float s, float v, int) { return s + v; }, db, 1);
}

// dW0[o][k] = sum_b dz0[b][o] x[b][k]
__global__ void mlp_layer0_bwd(const float *dz, const float *x, int nin, int H, int Bp, float *dW0) {
    const int k = blockIdx.y;
    column_sums(dz, H, H, Bp, [=](float s, float v, int b) { return fmaf(v, x[b * nin + k], s); }, dW0 + k, nin);
}

// copy a [H][Nop] GEMM result (dWout^T) into dWout [No][H]
__global__ void mlp_untranspose(Splits src, int H, int Nop, int No, float *dst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= No * H) return;
    const int o = i / H, k = i % H;
    dst[i] = src.at((size_t)k * Nop + o);
}

// bf16 copies of a weight matrix W [R][C] (rows >= R of the padded copy are 0)
__global__ void mlp_weights_bf16(const float *W, int R, int Rp, int C, __nv_bfloat16 *Wb, __nv_bfloat16 *WbT) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Rp * C) return;
    const int r = i / C, c = i % C;
    const float v = r < R ? W[(size_t)r * C + c] : 0.f;
    Wb[i] = bf(v);
    WbT[(size_t)c * Rp + r] = bf(v);
}

// Where each layer's weight matrix [R][C] lies in the parameters and its bf16
// copies (row count Rp of the padded ones); layer 0 has none
struct BfCopies {
    size_t off[17], end[17];
    int C[17], Rp[17];
    __nv_bfloat16 *Wb[17], *WbT[17];
    int layers;
};
// Adam, and the updated weights' bf16 copies (one launch instead of one per layer)
__global__ void mlp_adam(float *p, const float *g, float *m, float *v, size_t n, float lr, float b1, float b2,
                         float eps, float c1, float c2, const BfCopies L) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    for (int l = 0; l < L.layers; ++l)
        if (i >= L.off[l] && i < L.end[l]) {
            const int k = (int)(i - L.off[l]), r = k / L.C[l], c = k - r * L.C[l];
            L.Wb[l][k] = bf(w);
            L.WbT[l][(size_t)c * L.Rp[l] + r] = bf(w);
        }
}

inline unsigned nblk(size_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

uint64_t mlp_sm64(uint64_t &s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

}  // namespace

struct qmc_mlp {
    int device = 0, nin = 0, H = 0, D = 0, No = 0, Nop = 0;
    cudaStream_t stream = nullptr;
    size_t nparams = 0;
    std::vector<size_t> offW, offb;     // per layer (0..D-1 hidden, D = output)
    float *params = nullptr, *grads = nullptr, *am = nullptr, *av = nullptr;
    std::vector<__nv_bfloat16 *> Wb, WbT;   // layers 1..D (index by layer)
    int Bcap = 0;
    float *x = nullptr, *y = nullptr, *mask = nullptr;
    std::vector<float *> hf;                 // [D] f32 activations
    std::vector<__nv_bfloat16 *> hb, hbT;    // [D]
    float *out = nullptr, *dof = nullptr, *dz = nullptr;
    __nv_bfloat16 *dob = nullptr, *dobT = nullptr, *dzb = nullptr, *dzbT = nullptr;
    float *wt = nullptr;
    double *loss = nullptr;
    unsigned *err = nullptr;
    int t = 0;
    float *ws = nullptr;                     // GEMM splits (this network's own; stream ordered)
    size_t ws_cap = 0;
    int sms = 0;
};

namespace {

int mlp_free_batch(qmc_mlp *m) {
    cudaFree(m->x);
    cudaFree(m->y);
    cudaFree(m->mask);
    cudaFree(m->ws);
    cudaFree(m->out);
    cudaFree(m->dof);
    cudaFree(m->dz);
    cudaFree(m->dob);
    cudaFree(m->dobT);
    cudaFree(m->dzb);
    cudaFree(m->dzbT);
    for (float *p : m->hf) cudaFree(p);
    for (auto *p : m->hb) cudaFree(p);
    for (auto *p : m->hbT) cudaFree(p);
    m->hf.assign(m->D, nullptr);
    m->hb.assign(m->D, nullptr);
    m->hbT.assign(m->D, nullptr);
    m->x = m->y = m->mask = m->ws = m->out = m->dof = m->dz = nullptr;
    m->ws_cap = 0;
    m->dob = m->dobT = m->dzb = m->dzbT = nullptr;
    m->Bcap = 0;
    return 0;
}

int mlp_ensure_batch(qmc_mlp *m, int Bp) {
    if (Bp <= m->Bcap) return 0;
    mlp_free_batch(m);
    const size_t H = m->H, No = m->No, Nop = m->Nop;
    bool bad = false;
    auto A = [&](void **p, size_t bytes) { bad |= cudaMalloc(p, bytes) != cudaSuccess; };
    A((void **)&m->x, (size_t)Bp * m->nin * 4);
    A((void **)&m->y, (size_t)Bp * No * 4);
    A((void **)&m->mask, (size_t)Bp * 4);
    // the largest product's splits over the batch sizes up to Bp (splits fall
    // as the rows grow: bounded by all SMs' tiles, or one split of Bp rows)
    const size_t N = std::max(H, Nop);
    size_t cap = 0;
    for (int rows = kTileM; rows <= Bp; rows += kTileM)
        cap = std::max(cap, (size_t)gemm_splits_most(rows, (int)N, m->sms) * rows * N);
    cap = std::max(cap, (size_t)gemm_splits_most(m->H, Bp, m->sms) * H * N);
    A((void **)&m->ws, cap * 4);
    m->ws_cap = cap;
    A((void **)&m->out, (size_t)Bp * No * 4);
    A((void **)&m->dof, (size_t)Bp * Nop * 4);
    A((void **)&m->dz, (size_t)Bp * H * 4);
    A((void **)&m->dob, (size_t)Bp * Nop * 2);
    A((void **)&m->dobT, (size_t)Bp * Nop * 2);
    A((void **)&m->dzb, (size_t)Bp * H * 2);
    A((void **)&m->dzbT, (size_t)Bp * H * 2);
    for (int l = 0; l < m->D; ++l) {
        A((void **)&m->hf[l], (size_t)Bp * H * 4);
        A((void **)&m->hb[l], (size_t)Bp * H * 2);
        A((void **)&m->hbT[l], (size_t)Bp * H * 2);
    }
    if (bad) {
        mlp_free_batch(m);
        return -1;
    }
    m->Bcap = Bp;
    return 0;
}

// refresh the bf16 weight copies of the GEMM layers from the FP32 master weights
int mlp_sync_weights(qmc_mlp *m) {
    for (int l = 1; l <= m->D; ++l) {
        const int R = l == m->D ? m->No : m->H, Rp = l == m->D ? m->Nop : m->H;
        mlp_weights_bf16<<<nblk((size_t)Rp * m->H), 256, 0, m->stream>>>(m->params + m->offW[l], R, Rp, m->H,
                                                                        m->Wb[l], m->WbT[l]);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// A [M][K] B [N][K]^T into the network's workspace, as splits
int mlp_gemm(qmc_mlp *m, const void *A, const void *B, int M, int N, int K, Splits &out) {
    if (!gemm_shape_ok(A, B, M, N, K)) return -1;
    int per = 1;
    const int splits = gemm_splits(M, K, m->sms, per);
    if ((size_t)splits * M * N > m->ws_cap) return -1;
    out = Splits{m->ws, splits, (size_t)M * N};
    return gemm_launch(A, B, m->ws, M, N, K, splits, per, m->err, m->stream, kWaitLimit);
}
inline unsigned tiles(int N, int Bp) { return (unsigned)((N + kTile - 1) / kTile) * (unsigned)((Bp + kTile - 1) / kTile); }
// whether the launch before was accepted (asked at each: a later call may clear the error)
inline bool launched() { return cudaGetLastError() == cudaSuccess; }

// forward for Bp rows already in m->x; output in m->out [Bp][No]
int mlp_forward_dev(qmc_mlp *m, int Bp) {
    const int H = m->H;
    const dim3 tb(kTile, kTileRows);
    Splits C;
    mlp_layer0_fwd<<<tiles(H, Bp), tb, 0, m->stream>>>(m->x, m->params + m->offW[0], m->params + m->offb[0], m->nin, H,
                                                       Bp, m->hf[0], m->hb[0], m->hbT[0]);
    for (int l = 1; l < m->D; ++l) {
        if (!launched() || mlp_gemm(m, m->hb[l - 1], m->Wb[l], Bp, H, H, C)) return -1;
        mlp_bias_tanh<<<tiles(H, Bp), tb, 0, m->stream>>>(C, m->params + m->offb[l], H, Bp, m->hf[l], m->hb[l],
                                                          m->hbT[l]);
    }
    if (!launched() || mlp_gemm(m, m->hb[m->D - 1], m->Wb[m->D], Bp, m->Nop, H, C)) return -1;
    mlp_bias_out<<<nblk((size_t)Bp * m->No), 256, 0, m->stream>>>(C, m->params + m->offb[m->D], m->No, m->Nop, Bp,
                                                                 m->out);
    return launched() ? 0 : -1;
}

// loss (into *loss_dst) and gradients (into m->grads) for Bp rows with x, y, mask, wt in place
int mlp_backward_dev(qmc_mlp *m, int Bp, int B, double *loss_dst) {
    const int H = m->H, D = m->D, Nop = m->Nop, No = m->No;
    const dim3 tb(kTile, kTileRows);
    Splits C;
    cudaMemsetAsync(loss_dst, 0, sizeof(double), m->stream);
    mlp_loss<<<tiles(Nop, Bp), tb, 0, m->stream>>>(m->out, m->y, m->wt, m->mask, No, Nop, Bp, 1.f / B, m->dob, m->dobT,
                                                   m->dof, loss_dst);
    // output layer: dWout^T = h_{D-1}^T dout  ([H][Nop]), dbout, dh = dout Wout
    if (!launched() || mlp_gemm(m, m->hbT[D - 1], m->dobT, H, Nop, Bp, C)) return -1;
    mlp_untranspose<<<nblk((size_t)No * H), 256, 0, m->stream>>>(C, H, Nop, No, m->grads + m->offW[D]);
    mlp_colsum<<<(No + kCols - 1) / kCols, kColThreads, 0, m->stream>>>(m->dof, No, Nop, Bp, m->grads + m->offb[D]);
    if (!launched() || mlp_gemm(m, m->dob, m->WbT[D], Bp, H, Nop, C)) return -1;
    for (int l = D - 1; l >= 0; --l) {
        mlp_tanh_bwd<<<tiles(H, Bp), tb, 0, m->stream>>>(C, m->hf[l], H, Bp, m->dzb, m->dzbT, m->dz);
        mlp_colsum<<<H / kCols, kColThreads, 0, m->stream>>>(m->dz, H, H, Bp, m->grads + m->offb[l]);
        if (l == 0) {
            mlp_layer0_bwd<<<dim3(H / kCols, m->nin), kColThreads, 0, m->stream>>>(m->dz, m->x, m->nin, H, Bp,
                                                                           m->grads + m->offW[0]);
        } else {
            // dW_l = dz^T h_{l-1}  ([H][H]); dh_{l-1} = dz W_l
            if (!launched() || mlp_gemm(m, m->dzbT, m->hbT[l - 1], H, H, Bp, C)) return -1;
            qmc_gemm_splitk_sum<<<nblk((size_t)H * H), 256, 0, m->stream>>>(C.W, C.n, C.stride, m->grads + m->offW[l],
                                                                           C.stride);
            if (!launched() || mlp_gemm(m, m->dzb, m->WbT[l], Bp, H, H, C)) return -1;
        }
    }
    return launched() ? 0 : -1;
}

// stage a host batch (B rows) padded to Bp rows
int mlp_stage(qmc_mlp *m, const float *x, const float *y, const float *wt, int B, int Bp) {
    if (mlp_ensure_batch(m, Bp)) return -1;
    cudaMemsetAsync(m->x, 0, (size_t)Bp * m->nin * 4, m->stream);
    cudaMemcpyAsync(m->x, x, (size_t)B * m->nin * 4, cudaMemcpyHostToDevice, m->stream);
    if (y) {
        cudaMemsetAsync(m->y, 0, (size_t)Bp * m->No * 4, m->stream);
        cudaMemcpyAsync(m->y, y, (size_t)B * m->No * 4, cudaMemcpyHostToDevice, m->stream);
        std::vector<float> mk(Bp, 0.f);
        for (int b = 0; b < B; ++b) mk[b] = 1.f;
        cudaMemcpyAsync(m->mask, mk.data(), (size_t)Bp * 4, cudaMemcpyHostToDevice, m->stream);
        std::vector<float> w(m->No, 1.f);
        if (wt) w.assign(wt, wt + m->No);
        cudaMemcpyAsync(m->wt, w.data(), (size_t)m->No * 4, cudaMemcpyHostToDevice, m->stream);
        return cudaStreamSynchronize(m->stream) == cudaSuccess ? 0 : -1;   // host vectors go out of scope
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int mlp_check_err(qmc_mlp *m) {
    unsigned e = 0;
    if (cudaMemcpyAsync(&e, m->err, 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess) return -1;
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return -1;
    return e ? -1 : 0;
}

}  // namespace

extern "C" {

int qmc_mlp_create(qmc_mlp **out, int device, int nin, int width, int depth, int nout, uint64_t seed) {
    if (!out || nin < 1 || nin > 64 || width % 128 || width < 128 || width > 256 || depth < 1 || depth > 16 ||
        nout < 1 || nout > 256)
        return QMC_E_INVAL_LOCAL;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return QMC_E_CUDA_LOCAL;
    qmc_mlp *m = new qmc_mlp();
    m->device = device;
    cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, device);
    m->nin = nin;
    m->H = width;
    m->D = depth;
    m->No = nout;
    m->Nop = (nout + 15) / 16 * 16;
    m->hf.assign(depth, nullptr);
    m->hb.assign(depth, nullptr);
    m->hbT.assign(depth, nullptr);
    size_t off = 0;
    for (int l = 0; l <= depth; ++l) {
        const size_t fan_in = l == 0 ? nin : width, rows = l == depth ? nout : width;
        m->offW.push_back(off);
        off += rows * fan_in;
        m->offb.push_back(off);
        off += rows;
    }
    m->nparams = off;
    bool bad = cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking) != cudaSuccess;
    bad |= cudaMalloc(&m->params, off * 4) != cudaSuccess;
    bad |= cudaMalloc(&m->grads, off * 4) != cudaSuccess;
    bad |= cudaMalloc(&m->am, off * 4) != cudaSuccess;
    bad |= cudaMalloc(&m->av, off * 4) != cudaSuccess;
    bad |= cudaMalloc(&m->wt, 256 * 4) != cudaSuccess;
    bad |= cudaMalloc(&m->loss, sizeof(double)) != cudaSuccess;
    bad |= cudaMalloc(&m->err, 4) != cudaSuccess;
    m->Wb.assign(depth + 1, nullptr);
    m->WbT.assign(depth + 1, nullptr);
    for (int l = 1; l <= depth; ++l) {
        const size_t Rp = l == depth ? m->Nop : width;
        bad |= cudaMalloc(&m->Wb[l], Rp * width * 2) != cudaSuccess;
        bad |= cudaMalloc(&m->WbT[l], Rp * width * 2) != cudaSuccess;
    }
    if (bad) {
        qmc_mlp_destroy(m);
        return QMC_E_CUDA_LOCAL;
    }
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases, from splitmix64
    std::vector<float> p(off, 0.f);
    uint64_t st = seed;
    for (int l = 0; l <= depth; ++l) {
        const size_t fan_in = l == 0 ? nin : width, rows = l == depth ? nout : width;
        const double a = 1.0 / std::sqrt((double)fan_in);
        for (size_t i = 0; i < rows * fan_in; ++i)
            p[m->offW[l] + i] = (float)(a * (2.0 * ((mlp_sm64(st) >> 11) * (1.0 / 9007199254740992.0)) - 1.0));
    }
    cudaMemcpy(m->params, p.data(), off * 4, cudaMemcpyHostToDevice);
    cudaMemset(m->am, 0, off * 4);
    cudaMemset(m->av, 0, off * 4);
    cudaMemset(m->grads, 0, off * 4);
    cudaMemset(m->err, 0, 4);
    if (mlp_sync_weights(m) || cudaStreamSynchronize(m->stream) != cudaSuccess) {
        qmc_mlp_destroy(m);
        return QMC_E_CUDA_LOCAL;
    }
    *out = m;
    return 0;
}

void qmc_mlp_destroy(qmc_mlp *m) {
    if (!m) return;
    cudaSetDevice(m->device);
    if (m->stream) cudaStreamSynchronize(m->stream);
    mlp_free_batch(m);
    cudaFree(m->params);
    cudaFree(m->grads);
    cudaFree(m->am);
    cudaFree(m->av);
    cudaFree(m->wt);
    cudaFree(m->loss);
    cudaFree(m->err);
    for (auto *p : m->Wb) cudaFree(p);
    for (auto *p : m->WbT) cudaFree(p);
    if (m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

int qmc_mlp_num_params(const qmc_mlp *m, size_t *n) {
    if (!m || !n) return QMC_E_INVAL_LOCAL;
    *n = m->nparams;
    return 0;
}

int qmc_mlp_get_params(qmc_mlp *m, float *host, size_t n) {
    if (!m || !host || n != m->nparams) return QMC_E_INVAL_LOCAL;
    cudaSetDevice(m->device);
    if (cudaMemcpyAsync(host, m->params, n * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess)
        return QMC_E_CUDA_LOCAL;
    return 0;
}

int qmc_mlp_set_params(qmc_mlp *m, const float *host, size_t n) {
    if (!m || !host || n != m->nparams) return QMC_E_INVAL_LOCAL;
    cudaSetDevice(m->device);
    if (cudaMemcpyAsync(m->params, host, n * 4, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        mlp_sync_weights(m) || cudaStreamSynchronize(m->stream) != cudaSuccess)
        return QMC_E_CUDA_LOCAL;
    return 0;
}

int qmc_mlp_forward(qmc_mlp *m, const float *x, int B, float *y) {
    if (!m || !x || !y || B < 1) return QMC_E_INVAL_LOCAL;
    cudaSetDevice(m->device);
    cudaMemsetAsync(m->err, 0, 4, m->stream);
    const int Bp = (B + 127) / 128 * 128;
    if (mlp_stage(m, x, nullptr, nullptr, B, Bp) || mlp_forward_dev(m, Bp)) return QMC_E_CUDA_LOCAL;
    if (cudaMemcpyAsync(y, m->out, (size_t)B * m->No * 4, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
        return QMC_E_CUDA_LOCAL;
    return mlp_check_err(m) ? QMC_E_CUDA_LOCAL : 0;
}

int qmc_mlp_grad(qmc_mlp *m, const float *x, const float *y, const float *wt, int B, float *loss, float *grad) {
    if (!m || !x || !y || B < 1) return QMC_E_INVAL_LOCAL;
    cudaSetDevice(m->device);
    cudaMemsetAsync(m->err, 0, 4, m->stream);
    const int Bp = (B + 127) / 128 * 128;
    if (mlp_stage(m, x, y, wt, B, Bp) || mlp_forward_dev(m, Bp) || mlp_backward_dev(m, Bp, B, m->loss))
        return QMC_E_CUDA_LOCAL;
    double l = 0.0;
    cudaMemcpyAsync(&l, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
    if (grad) cudaMemcpyAsync(grad, m->grads, m->nparams * 4, cudaMemcpyDeviceToHost, m->stream);
    if (mlp_check_err(m)) return QMC_E_CUDA_LOCAL;
    if (loss) *loss = (float)l;
    return 0;
}

int qmc_mlp_train(qmc_mlp *m, const float *x, const float *y, const float *wt, int B, int steps, float lr,
                  float *losses) {
    if (!m || !x || !y || B < 1 || steps < 0 || !(lr > 0)) return QMC_E_INVAL_LOCAL;
    cudaSetDevice(m->device);
    cudaMemsetAsync(m->err, 0, 4, m->stream);
    const int Bp = (B + 127) / 128 * 128;
    if (mlp_stage(m, x, y, wt, B, Bp)) return QMC_E_CUDA_LOCAL;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    // per-step losses stay on the device until the end (no host round trip per step)
    double *hist = nullptr;
    if (cudaMalloc(&hist, (size_t)std::max(steps, 1) * sizeof(double)) != cudaSuccess) return QMC_E_CUDA_LOCAL;
    int rc = 0;
    BfCopies copies{};
    copies.layers = m->D;
    for (int l = 1; l <= m->D; ++l) {
        const int R = l == m->D ? m->No : m->H;
        copies.off[l - 1] = m->offW[l];
        copies.end[l - 1] = m->offW[l] + (size_t)R * m->H;
        copies.C[l - 1] = m->H;
        copies.Rp[l - 1] = l == m->D ? m->Nop : m->H;
        copies.Wb[l - 1] = m->Wb[l];
        copies.WbT[l - 1] = m->WbT[l];
    }
    for (int s = 0; s < steps && !rc; ++s) {
        if (mlp_forward_dev(m, Bp) || mlp_backward_dev(m, Bp, B, hist + s)) {
            rc = QMC_E_CUDA_LOCAL;
            break;
        }
        ++m->t;
        const float c1 = 1.f - std::pow(b1, (float)m->t), c2 = 1.f - std::pow(b2, (float)m->t);
        mlp_adam<<<nblk(m->nparams), 256, 0, m->stream>>>(m->params, m->grads, m->am, m->av, m->nparams, lr, b1,
                                                           b2, eps, c1, c2, copies);
        if (cudaGetLastError() != cudaSuccess) rc = QMC_E_CUDA_LOCAL;
    }
    if (!rc && losses && steps > 0) {
        std::vector<double> h(steps);
        if (cudaMemcpyAsync(h.data(), hist, steps * sizeof(double), cudaMemcpyDeviceToHost, m->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(m->stream) != cudaSuccess)
            rc = QMC_E_CUDA_LOCAL;
        for (int s = 0; s < steps && !rc; ++s) losses[s] = (float)h[s];
    }
    cudaStreamSynchronize(m->stream);
    cudaFree(hist);
    if (rc) return rc;
    return mlp_check_err(m) ? QMC_E_CUDA_LOCAL : 0;
}

}  // extern "C"
