// BF16 GEMM on the 5th-generation tensor cores (tcgen05 + TMEM) with TMA
// staging, for the surrogate MLP.  C[M x N] = A[M x K] . B[N x K]^T, FP32
// accumulation in tensor memory, the same fused epilogues as the mma.sync
// kernel in mlp.cu (plain, bias, bias+GELU, GELU derivative).  Either operand
// is row-major with K contiguous, or given transposed (row-major with M or N
// contiguous), so the weight gradient dY^T X and the input gradient dY W need
// no transposed copies (12 transposes, 77 us of a training step of 4096 rows).
// No counterpart in the paper.
//
// One CTA computes a 128 x BN tile with 128 threads:
//   thread 0    TMA producer: 64-wide K blocks of A and B (128B swizzle) into a
//               ring of shared-memory stages, completion tracked by mbarriers;
//   thread 32   MMA issuer: tcgen05.mma.cta_group::1.kind::f16 (M=128, N=BN,
//               K=16) from shared-memory descriptors into a BN-column TMEM
//               accumulator; tcgen05.commit frees each stage and finally
//               signals the epilogue;
//   all warps   epilogue: warp w reads TMEM lanes 32w..32w+31 (rows) with
//               tcgen05.ld.32x32b, turns each 32 x 32 block around in shared
//               memory and moves it four columns per lane (16-byte loads of
//               `pre`, 16- and 8-byte stores), eight rows in flight.
// What bounds it at the surrogate's sizes is latency, not the tensor cores: a
// tile has 16 to 64 K blocks and an epilogue of erf and exp, and there are at
// most about two tiles per SM.  So BN is the largest of 128, 64, 32 that still
// gives every SM a tile (a weight gradient of 1024 x 1024 is 64 tiles of 128
// columns), two CTAs share an SM with half the ring each when there are more
// tiles than SMs, and otherwise one CTA has the whole ring (about 190 KB in
// flight).  Training step of 4096 rows: GEMMs 400 us before.
// A transposed operand's stage holds 64-column blocks of 64 K rows (128 bytes
// each), 8 KB apart: the MN-major 128-byte-swizzle layout.
// Out-of-range rows, columns and K are zero-filled by TMA and skipped on
// store.  Every mbarrier wait gives up after a bounded number of polls and
// raises an error flag the host reads; TMEM is always released.

#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <mutex>

#include "pcv_common.cuh"
#include "tc_ptx.cuh"

namespace pcv {

namespace {

constexpr int TC_BM = 128, TC_BK = 64;
constexpr int TC_MAX_STAGES = 8;
constexpr int kTcSms = 152;
constexpr int TC_THREADS = 128;
constexpr uint32_t TC_RING_ONE = 192 * 1024, TC_RING_TWO = 96 * 1024;   // ring bytes with one, two CTAs per SM
constexpr long long TC_MAX_POLLS = 1ll << 22;                           // default bound of one mbarrier wait

struct TcArgs {
    int M, N, K;
    int at, bt;                       // operand given transposed (M or N contiguous)
    int stages;
    int vec;                          // bias, outputs and pre allow 4-column accesses
    const float* bias;
    float* outf; int ldo;
    __nv_bfloat16* outb; int ldob;
    const float* pre; int ldp;
    int* error;                       // set to the role that gave up (1 loads, 2 MMA, 3 epilogue, 4 clean-up)
    long long max_polls;              // bound of one mbarrier wait
};

using tcx::mbar_expect_tx;
using tcx::mbar_init;
using tcx::mbar_wait;
using tcx::sdesc_sw128;
using tcx::tma_load_2d;

__device__ __forceinline__ float gelu_tc(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_tc(float x)
{
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// Descriptor of an MN-major tile (128-byte swizzle): rows of one K, 64 MN
// values each; 8 K rows 1024 B apart, 64-value MN blocks 8 KB apart.
__device__ __forceinline__ uint64_t sdesc_mn_sw128(const void* p)
{
    uint64_t d = sdesc_sw128(p) & ~((uint64_t)0x3FFF << 16);
    return d | ((uint64_t)(8192 >> 4) << 16);
}

// One element of the epilogue.
template <int MODE>
__device__ __forceinline__ void epilogue_one(const TcArgs& a, float x, int row, int col)
{
    if constexpr (MODE == 0) a.outf[(size_t)row * a.ldo + col] = x;
    if constexpr (MODE == 2) a.outf[(size_t)row * a.ldo + col] = x + a.bias[col];
    if constexpr (MODE == 1) {
        x += a.bias[col];
        if (a.outf) a.outf[(size_t)row * a.ldo + col] = x;
        a.outb[(size_t)row * a.ldob + col] = __float2bfloat16_rn(gelu_tc(x));
    }
    if constexpr (MODE == 3)
        a.outb[(size_t)row * a.ldob + col] = __float2bfloat16_rn(x * gelu_grad_tc(a.pre[(size_t)row * a.ldp + col]));
}

__device__ __forceinline__ uint2 pack_bf16(float4 x)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
    uint2 r;
    r.x = *reinterpret_cast<const uint32_t*>(&lo);
    r.y = *reinterpret_cast<const uint32_t*>(&hi);
    return r;
}

template <int BN, int MODE, int KB>
__global__ void __launch_bounds__(TC_THREADS, 2)
gemm_bf16_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, const TcArgs a)
{
    constexpr uint32_t kABytes = TC_BM * TC_BK * 2, kBBytes = BN * TC_BK * 2, kStage = KB * (kABytes + kBBytes);
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte aligned ring of stages: KB blocks of A (128x64 bf16), then KB of B (BNx64)
    unsigned char* ring = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[TC_MAX_STAGES], empty_bar[TC_MAX_STAGES], done_bar, mma_done;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.y * TC_BM, n0 = blockIdx.x * BN;
    const int nk = (a.K + KB * TC_BK - 1) / (KB * TC_BK), stages = a.stages;

    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&done_bar, 1);
        mbar_init(&mma_done, 1);
        s_fail = 0;
        tcx::mbar_fence_init();
        tcx::prefetch_tmap(&mapA);
        tcx::prefetch_tmap(&mapB);
    }
    if (warp == 1) tcx::tmem_alloc(&tmem_base, BN);
    tcx::fence_before_sync();
    __syncthreads();
    tcx::fence_after_sync();
    const uint32_t tmem = tmem_base;
    const long long polls = a.max_polls;

    if (warp == 0 && tcx::elect_one()) {
        // ---------------- TMA producer
        int issued = 0;
        for (int kt = 0, st = 0, ph = 1; kt < nk && !s_fail; ++kt) {
            if (kt >= stages && !mbar_wait(&empty_bar[st], ph, polls)) { s_fail = 1; break; }
            unsigned char* sa = ring + st * kStage;
            unsigned char* sb = sa + KB * kABytes;
            mbar_expect_tx(&full_bar[st], kStage);
#pragma unroll
            for (int h = 0; h < KB; ++h) {             // blocks beyond K are zero-filled
                const int k0 = (kt * KB + h) * TC_BK;
                if (a.at) {
                    tma_load_2d(sa + h * kABytes, &mapA, &full_bar[st], m0, k0);
                    tma_load_2d(sa + h * kABytes + 8192, &mapA, &full_bar[st], m0 + 64, k0);
                } else {
                    tma_load_2d(sa + h * kABytes, &mapA, &full_bar[st], k0, m0);
                }
                if (a.bt) {
                    for (int j = 0; j < BN; j += 64)
                        tma_load_2d(sb + h * kBBytes + j * 128, &mapB, &full_bar[st], n0 + j, k0);
                } else {
                    tma_load_2d(sb + h * kBBytes, &mapB, &full_bar[st], k0, n0);
                }
            }
            ++issued;
            if (++st == stages) {
                st = 0;
                ph ^= 1;
            }
        }
        // the loads issued land in this CTA's shared memory before it may exit
        if (!tcx::wait_issued(full_bar, stages, (uint32_t)issued) && !s_fail) s_fail = 4;
    } else if (warp == 1 && tcx::elect_one()) {
        // ---------------- MMA issuer
        const uint32_t idesc = tcx::idesc_bf16(TC_BM, BN) | (a.at ? 1u << 15 : 0u) | (a.bt ? 1u << 16 : 0u);
        // 16 of K further: 32 B along a K-major row, 16 rows of 128 B of an MN-major tile (16-byte units)
        const uint32_t astep = a.at ? 128 : 2, bstep = a.bt ? 128 : 2;
        bool all = true;
        for (int kt = 0, st = 0, ph = 0; kt < nk; ++kt) {
            if (!mbar_wait(&full_bar[st], ph, polls)) { s_fail = 2; all = false; break; }
            tcx::fence_after_sync();
            const unsigned char* sa = ring + st * kStage;
            const unsigned char* sb = sa + KB * kABytes;
            const uint64_t ad = a.at ? sdesc_mn_sw128(sa) : sdesc_sw128(sa);
            const uint64_t bd = a.bt ? sdesc_mn_sw128(sb) : sdesc_sw128(sb);
#pragma unroll
            for (int kk = 0; kk < KB * TC_BK / 16; ++kk) {
                const int h = kk / (TC_BK / 16), j = kk % (TC_BK / 16);
                tcx::mma_bf16(tmem, ad + h * (kABytes >> 4) + j * astep, bd + h * (kBBytes >> 4) + j * bstep, idesc,
                              (kt > 0 || kk > 0) ? 1u : 0u);
            }
            tcx::mma_commit(&empty_bar[st]);
            if (++st == stages) {
                st = 0;
                ph ^= 1;
            }
        }
        // a complete accumulation goes to the epilogue; in every case the MMAs
        // issued finish before the tensor memory is released
        if (all) tcx::mma_commit(&done_bar);
        tcx::mma_commit(&mma_done);
        if (!mbar_wait(&mma_done, 0, tcx::kCleanupPolls) && !s_fail) s_fail = 4;
    }

    // The other lanes of the producer's and the issuer's warps park here: were
    // they to poll done_bar meanwhile, the warp would alternate between the two
    // paths and each K block's loads and MMAs would take about 400 cycles to
    // issue (K = 4096: 28.8 us however wide the tile).
    __syncwarp();

    // ---------------- epilogue (all warps)
    const bool ok = mbar_wait(&done_bar, 0, polls);
    if (!ok && lane == 0) s_fail = 3;
    tcx::fence_after_sync();
    __syncwarp();
    if (ok) {
        // Each warp moves its 32 rows x 32 columns through a padded shared tile
        // (the drained stage ring): a row per lane in, four columns per lane out
        // (8 lanes to a row).
        constexpr int kRow = 36;
        float* stage = reinterpret_cast<float*>(ring) + warp * (32 * kRow);
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 32) {
            const int col = n0 + c0 + (lane & 7) * 4, row0 = m0 + warp * 32 + (lane >> 3);
            const bool vec = a.vec && col + 4 <= a.N;
            float4 pre[8];
            if constexpr (MODE == 3) {
#pragma unroll
                for (int it = 0; it < 8; ++it)
                    if (vec && row0 + 4 * it < a.M)
                        pre[it] = *reinterpret_cast<const float4*>(a.pre + (size_t)(row0 + 4 * it) * a.ldp + col);
            }
            uint32_t r[32];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                  "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                  "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
            for (int j = 0; j < 32; j += 4)                                              // row = lane
                *reinterpret_cast<uint4*>(stage + lane * kRow + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
            __syncwarp();
            float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (MODE == 1 || MODE == 2)
                if (vec) bias = *reinterpret_cast<const float4*>(a.bias + col);
#pragma unroll
            for (int it = 0; it < 8; ++it) {
                const int row = row0 + 4 * it;
                if (row >= a.M) continue;
                float4 x = *reinterpret_cast<const float4*>(stage + ((lane >> 3) + 4 * it) * kRow + (lane & 7) * 4);
                if (!vec) {
                    const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (col + e < a.N) epilogue_one<MODE>(a, v[e], row, col + e);
                    continue;
                }
                if constexpr (MODE == 1 || MODE == 2) {
                    x.x += bias.x;
                    x.y += bias.y;
                    x.z += bias.z;
                    x.w += bias.w;
                }
                if constexpr (MODE == 3) {
                    x.x *= gelu_grad_tc(pre[it].x);
                    x.y *= gelu_grad_tc(pre[it].y);
                    x.z *= gelu_grad_tc(pre[it].z);
                    x.w *= gelu_grad_tc(pre[it].w);
                } else if (MODE != 1 || a.outf) {
                    *reinterpret_cast<float4*>(a.outf + (size_t)row * a.ldo + col) = x;
                }
                if constexpr (MODE == 1) x = make_float4(gelu_tc(x.x), gelu_tc(x.y), gelu_tc(x.z), gelu_tc(x.w));
                if constexpr (MODE == 1 || MODE == 3)
                    *reinterpret_cast<uint2*>(a.outb + (size_t)row * a.ldob + col) = pack_bf16(x);
            }
            __syncwarp();
        }
    }
    tcx::fence_before_sync();
    __syncthreads();
    if (warp == 1) tcx::tmem_dealloc(tmem, BN);
    if (tid == 0 && s_fail && a.error) atomicExch(a.error, s_fail);
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

cudaError_t get_encode()
{
    std::call_once(g_encode_once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    });
    return g_encode ? cudaSuccess : cudaErrorNotSupported;
}

// 2-D bf16 tensor map over `outer` rows of `inner` values (row stride ld), box
// 64 x box_rows, 128B swizzle.
cudaError_t make_map(CUtensorMap* map, const void* base, int inner, int outer, int ld, int box_rows)
{
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int BN, int MODE, int KB>
cudaError_t launch_tile(const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& a, size_t smem, cudaStream_t s)
{
    const cudaError_t e = allow_dynamic_smem((const void*)gemm_bf16_tc_kernel<BN, MODE, KB>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((a.N + BN - 1) / BN, (a.M + TC_BM - 1) / TC_BM);
    gemm_bf16_tc_kernel<BN, MODE, KB><<<grid, TC_THREADS, smem, s>>>(ma, mb, a);
    note_launches(1);
    return cudaGetLastError();
}

template <int BN, int KB>
cudaError_t launch_depth(const CUtensorMap& ma, const CUtensorMap& mb, int mode, TcArgs a, uint32_t ring, cudaStream_t s)
{
    constexpr uint32_t stage = KB * (TC_BM + BN) * TC_BK * 2;
    const int nk = (a.K + KB * TC_BK - 1) / (KB * TC_BK);
    a.stages = std::min<int>(std::min<int>(TC_MAX_STAGES, ring / stage), std::max(nk, 2));
    const size_t smem = std::max<size_t>((size_t)a.stages * stage, 4 * 32 * 36 * sizeof(float)) + 1024;
    switch (mode) {
    case 0: return launch_tile<BN, 0, KB>(ma, mb, a, smem, s);
    case 1: return launch_tile<BN, 1, KB>(ma, mb, a, smem, s);
    case 2: return launch_tile<BN, 2, KB>(ma, mb, a, smem, s);
    default: return launch_tile<BN, 3, KB>(ma, mb, a, smem, s);
    }
}

template <int BN>
cudaError_t launch_width(const CUtensorMap& ma, const CUtensorMap& mb, int mode, const TcArgs& a, int64_t tiles,
                         cudaStream_t s)
{
    if (tiles > kTcSms) return launch_depth<BN, 1>(ma, mb, mode, a, TC_RING_TWO, s);
    return a.K > 8 * TC_BK ? launch_depth<BN, 2>(ma, mb, mode, a, TC_RING_ONE, s)
                           : launch_depth<BN, 1>(ma, mb, mode, a, TC_RING_ONE, s);
}

bool aligned_to(const void* p, size_t n) { return (uintptr_t)p % n == 0; }

}  // namespace

cudaError_t launch_gemm_bf16_tc(const void* A, int lda, int at, const void* B, int ldb, int bt, int M, int N, int K,
                                int mode, const float* bias, float* outf, int ldo, void* outb, int ldob,
                                const float* pre, int ldp, int* error, cudaStream_t s)
{
    cudaError_t e = get_encode();
    if (e != cudaSuccess) return e;
    // the widest tile that still gives every SM one (a 32-wide tile cannot be
    // transposed: its stage would hold half a 64-column block)
    const int64_t rows = (M + TC_BM - 1) / TC_BM;
    int bn = 128;
    while (bn > (bt ? 64 : 32) && rows * ((N + bn - 1) / bn) < kTcSms) bn >>= 1;
    CUtensorMap ma, mb;
    e = at ? make_map(&ma, A, M, K, lda, TC_BK) : make_map(&ma, A, K, M, lda, TC_BM);
    if (e != cudaSuccess) return e;
    e = bt ? make_map(&mb, B, N, K, ldb, TC_BK) : make_map(&mb, B, K, N, ldb, bn);
    if (e != cudaSuccess) return e;
    TcArgs a;
    a.M = M; a.N = N; a.K = K; a.at = at; a.bt = bt;
    a.bias = bias; a.outf = outf; a.ldo = ldo; a.outb = (__nv_bfloat16*)outb; a.ldob = ldob; a.pre = pre; a.ldp = ldp;
    a.error = error;
    a.max_polls = wait_limit(TC_MAX_POLLS);
    a.vec = (!outf || (ldo % 4 == 0 && aligned_to(outf, 16))) && (!outb || (ldob % 4 == 0 && aligned_to(outb, 8))) &&
            (mode != 3 || (ldp % 4 == 0 && aligned_to(pre, 16))) && (mode == 0 || mode == 3 || aligned_to(bias, 16));
    const int64_t tiles = rows * ((N + bn - 1) / bn);
    if (bn == 128) return launch_width<128>(ma, mb, mode, a, tiles, s);
    if (bn == 64) return launch_width<64>(ma, mb, mode, a, tiles, s);
    return launch_width<32>(ma, mb, mode, a, tiles, s);
}

}  // namespace pcv

// Checks and launch of both entry points.
static int gemm_tc(const void* A, int lda, int at, const void* B, int ldb, int bt, int M, int N, int K, int mode,
                   const float* bias, float* outf, int ldo, void* outb, int ldob, const float* pre, int ldp, int* error,
                   void* stream)
{
    if (!A || !B || M < 1 || N < 1 || K < 16 || K % 8 != 0) {
        pcv::set_error("gemm_bf16_tc: sizes (K must be a positive multiple of 8)");
        return PCV_EINVAL;
    }
    if (lda % 8 || ldb % 8 || lda < (at ? M : K) || ldb < (bt ? N : K) || ((uintptr_t)A % 16) || ((uintptr_t)B % 16)) {
        pcv::set_error("gemm_bf16_tc: leading dimensions must be multiples of 8 >= K (>= M, N of a transposed operand) "
                       "and operands 16-byte aligned");
        return PCV_EINVAL;
    }
    if (mode < 0 || mode > 3 || ((mode == 0 || mode == 2) && !outf) || ((mode == 1 || mode == 3) && !outb) ||
        ((mode == 1 || mode == 2) && !bias) || (mode == 3 && !pre)) {
        pcv::set_error("gemm_bf16_tc: epilogue arguments");
        return PCV_EINVAL;
    }
    cudaError_t e = pcv::launch_gemm_bf16_tc(A, lda, at, B, ldb, bt, M, N, K, mode, bias, outf, ldo, outb, ldob, pre, ldp,
                                             error, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        char buf[200];
        snprintf(buf, sizeof buf, "gemm_bf16_tc: %s", cudaGetErrorString(e));
        pcv::set_error(buf);
        return PCV_ECUDA;
    }
    return PCV_OK;
}

extern "C" int pcv_gemm_bf16_tc(const void* A, int lda, const void* B, int ldb, int M, int N, int K, int mode,
                                const float* bias, float* outf, int ldo, void* outb, int ldob, const float* pre,
                                int ldp, int* error, void* stream)
{
    return gemm_tc(A, lda, 0, B, ldb, 0, M, N, K, mode, bias, outf, ldo, outb, ldob, pre, ldp, error, stream);
}

extern "C" int pcv_gemm_bf16_tc_t(const void* A, int lda, int a_transposed, const void* B, int ldb, int b_transposed,
                                  int M, int N, int K, int mode, const float* bias, float* outf, int ldo, void* outb,
                                  int ldob, const float* pre, int ldp, int* error, void* stream)
{
    return gemm_tc(A, lda, a_transposed != 0, B, ldb, b_transposed != 0, M, N, K, mode, bias, outf, ldo, outb, ldob, pre,
                   ldp, error, stream);
}
