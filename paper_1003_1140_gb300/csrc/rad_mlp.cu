// rad_mlp.cu -- the learned surrogate's network: a ReLU MLP with BF16 weights
// (FP32 master copy), BF16 GEMM operands and FP32 accumulation, trained with
// MSE and Adam, entirely on the device (C ABI in include/rad_mlp.h).
//
// GEMMs run on the 5th-generation tensor cores: one persistent kernel computes
// C = A B^T for BF16 operands A [M][K], B [N][K], one block of ten
// warps per SM taking 128 x 128 output tiles in turn:
//   * warp 0, one lane: TMA (cp.async.bulk.tensor.2d) loads of 128 x 64 tiles
//     of A and B in the 128-byte-swizzled layout into a five-stage ring,
//     completion on mbarriers;
//   * warp 1, one lane: four tcgen05.mma (kind::f16, BF16 x BF16 -> FP32,
//     M 128, N 128, K 16) per stage into one of two 128-column accumulators in
//     tensor memory (tiles alternate); tcgen05.commit frees the stage and,
//     after a tile's last stage, hands the accumulator to the epilogue;
//   * warps 2-9: tcgen05.ld of 32 accumulator rows x 64 columns each, a
//     transpose through shared memory into row-contiguous groups, the fused
//     epilogue (bias, ReLU, ReLU mask of the backward pass, FP32 and/or BF16
//     output) and coalesced global stores, after which the accumulator goes
//     back to warp 1 -- so a tile's epilogue overlaps the next tile's loads
//     and MMAs.
// Products with few output tiles and a long K (the input gradient of the wide
// output layer: 128 x 512 outputs over K = 393,216) split K across blocks:
// each slice writes raw FP32 partial sums and one reduction kernel adds the
// slices in a fixed order and applies the epilogue, so the result does not
// depend on scheduling.  An operand stored the other way round ([K][M] or
// [K][N]) is read in place as an M- (N-) major tile: the input gradient G W
// reads the same BF16 W as the forward pass, the weight gradient G^T H reads G
// and H as the passes left them.  The output layer's epilogue forms the loss and
// its gradient (training) or the output transform (prediction), so that its
// FP32 outputs never make a round trip through memory.
// Every wait on an mbarrier is bounded; on expiry the block raises an error
// word, drains what it issued and releases its tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <new>
#include <vector>

#include "rad_internal.cuh"
#include "rad_mlp.h"

namespace {

typedef __nv_bfloat16 bf16;
using rad::smem_addr;

constexpr int BM = 128, BN = 128, BK = 64;   // block tile; BK x 2 B = one 128-byte swizzle row
constexpr int kStages = 5;                   // TMA -> MMA pipeline depth
constexpr int kEpiWarps = 8;                 // epilogue warps: two per 32 TMEM lanes, each
                                             // storing half of the tile's columns
constexpr int kGemmThreads = (2 + kEpiWarps) * 32;   // TMA warp, MMA warp, epilogue warps
constexpr uint32_t kTileBytes = BM * BK * 2;               // 16 KB per operand per stage
constexpr uint32_t kStageBytes = 2 * kTileBytes;
constexpr uint32_t kTmemCols = 2 * BN;                     // two FP32 128 x 128 accumulators
constexpr size_t kEpiBytes = kEpiWarps * 32 * 32 * sizeof(float);   // transpose staging
constexpr int kChain = 2 * kEpiWarps * 2;    // column-sum hand-overs: accumulator, warp, 32 columns
constexpr size_t kChainBytes = kChain * 32 * sizeof(float);
constexpr size_t kGemmSmem = kStages * kStageBytes + kEpiBytes + kChainBytes +
                             1024 /* alignment */ + 512 /* barriers */;
constexpr int kMinSplitTiles = 4;            // K tiles (of 64) per slice at least

// Streaming multiprocessors of the current device (the persistent GEMM runs one
// block on each).
int device_sms()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
        cudaGetLastError();
        return 1;
    }
    return n;
}

// tcgen05 instruction descriptor, kind::f16: FP32 accumulator (bits 4-5 = 1),
// A and B BF16 (bits 7-9, 10-12 = 1), K-major (bits 15, 16 = 0; 1 for an M- or
// N-major operand), N / 8 in bits 17-22, M / 16 in bits 24-28.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                            ((uint32_t)(BM >> 4) << 24);

// Text of the last failure of a rad_mlp_* call on this host thread.
thread_local char g_last_error[256] = "";

int fail(int rc, const char* what, cudaError_t e = cudaSuccess)
{
    if (e != cudaSuccess)
        snprintf(g_last_error, sizeof g_last_error, "%s: %s", what, cudaGetErrorString(e));
    else
        snprintf(g_last_error, sizeof g_last_error, "%s", what);
    return rc;
}

// Raised (bit rad::kErrTimeout) by a GEMM block whose bounded wait expired.
__device__ int g_gemm_err;

int* gemm_err_word()
{
    void* p = nullptr;
    return cudaGetSymbolAddress(&p, g_gemm_err) == cudaSuccess ? static_cast<int*>(p) : nullptr;
}

// Reads and clears the error word (after the stream has been synchronised).
bool gemm_timed_out()
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_gemm_err, sizeof(int)) != cudaSuccess) return true;
    if (v) {
        const int zero = 0;
        cudaMemcpyToSymbol(g_gemm_err, &zero, sizeof(int));
    }
    return v != 0;
}

struct Epilogue {
    const float* bias = nullptr;    // [N] or null
    const float* mask = nullptr;    // [M][N] (z of the backward pass: keep where > 0) or null
    float* out_f32 = nullptr;       // [M][N] or null
    bf16* out_bf16 = nullptr;       // [M][N] or null
    int relu = 0;                   // apply ReLU before the BF16 store
    int rows = 0;                   // rows of out_f32 / target that exist (0: all M)
    // output transform: out_f32 = 10^(value sd + mu) per column
    const float* mu = nullptr;
    const float* sd = nullptr;
    // mean squared error: value becomes the gradient g = scale (value - target) on the
    // existing rows and 0 on the others (out_bf16, out_f32); each warp's (block's) share of
    // sum (value - target)^2 goes to loss_part, g's column sums to colsum if set
    const float* target = nullptr;
    float scale = 0.0f;
    float* colsum = nullptr;        // [N]; needs sums_in_epilogue()
    double* loss_part = nullptr;    // [loss_shares()]
};

// Number of K slices for an M x N x K product: enough tiles to fill the GPU
// twice over when the output alone gives too few, each slice kMinSplitTiles
// K tiles or more.
int split_count(int M, int N, int K)
{
    const int blocks = (M / BM) * (N / BN), nk = K / BK, target = 2 * device_sms();
    if (blocks >= target / 2) return 1;
    const int want = (target + blocks - 1) / blocks;
    return std::max(1, std::min(want, nk / kMinSplitTiles));
}

// Shared-memory matrix descriptor (without the tile's address / 16 in bits 0-13) of an
// operand tile stored by TMA with 128-byte swizzling; descriptor version 1 (bit 46), layout
// SWIZZLE_128B (2 in bits 61-63).  The tile base is 1024-B aligned.
// K-major: rows of 128 B, 8-row groups 1024 B apart (stride byte offset, bits 32-45), the
// leading byte offset (bits 16-29) unused for this layout (1); a slice of 16 K is 32 B.
// M- (N-) major: two halves of 64 K rows x 64 elements (128 B), 8192 B apart (leading byte
// offset: the next 64 elements along M); 8-row groups along K 1024 B apart (stride byte
// offset); a slice of 16 K rows is 2048 B.
constexpr uint64_t kSw128 = ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
constexpr uint64_t kDescK = kSw128 | ((uint64_t)1 << 16);
constexpr uint64_t kDescMN = kSw128 | ((uint64_t)((kTileBytes / 2) >> 4) << 16);

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrives on bar once every tcgen05.mma this thread issued before has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// Epilogues, each a kernel of its own: with all of them in one kernel the plain one, which
// bounds the wide layer's weight gradient (805 MB written), took 253 us instead of 151.
enum { kEpiPlain, kEpiPower, kEpiLoss };

// The kernels of a call run one after the other and most take a few microseconds: each is
// launched while its predecessor still runs (programmatic stream serialisation), sets up,
// and waits in chain_wait() for the predecessor's completion before it touches global
// memory; it lets its own successor do the same from the start.
// A prediction of 100 x 393,216 outputs (nine launches, 92 us of them the wide product):
// 137 us instead of 153.
__device__ __forceinline__ void chain_wait()
{
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
}

template <class... P, class... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Layout and order bits of a product.
constexpr int kAMajorM = 1;      // A stored [K][M]
constexpr int kBMajorN = 2;      // B stored [K][N]
constexpr int kRowsInner = 4;    // a block takes all row tiles of a column tile in turn

// Tile i of this block of C = A B^T (split into S slices along K): slice z, row tile m0,
// column tile n0, K tiles [kt0, kt1).  Column tiles vary fastest, so the blocks working at
// the same time share their A tile in L2; with kRowsInner the block keeps its B tile and
// takes the row tiles in order.  False past the last tile.
struct TileCoord {
    int z, m0, n0, kt0, kt1;
};

__device__ __forceinline__ bool tile_at(int i, int M, int N, int K, int S, int mode, TileCoord& c)
{
    const int mt = M / BM, ntl = N / BN, nk_all = K / BK;
    if (mode & kRowsInner) {
        const int q = i / mt, n = blockIdx.x + q * gridDim.x;
        c = {0, (i - q * mt) * BM, n * BN, 0, nk_all};
        return n < ntl;
    }
    const int t = blockIdx.x + i * gridDim.x;
    const int z = t / (mt * ntl), rem = t - z * mt * ntl;
    c.z = z;
    c.m0 = (rem / ntl) * BM;
    c.n0 = (rem % ntl) * BN;
    c.kt0 = (int)((int64_t)nk_all * z / S);
    c.kt1 = (int)((int64_t)nk_all * (z + 1) / S);
    return z < S;
}

// C = A B^T, persistent: each block takes its output tiles in turn (tile_at).
// Warp 0 (one lane) streams A and B tiles by TMA into a kStages-deep ring of
// shared-memory stages; warp 1 (one lane) issues the tcgen05 MMAs of a tile
// into one of two TMEM accumulators and commits it; warps 2-9 drain the other
// accumulator through the epilogue (two warps per 32-row quarter, 64 columns
// each), so that a tile's epilogue overlaps the next tile's loads and MMAs.  A and B come
// through the tensor maps (128-byte swizzle): K innermost, box 64 x 128, or
// (kAMajorM, kBMajorN) M / N innermost, two boxes 64 x 64.  Every wait is bounded: an
// expired wait raises the block's abort flag and err_word, every role leaves
// its loop, the TMA warp waits for its loads in flight and the MMA warp for its
// MMAs before the accumulators are released.
template <int EPI>
__global__ void __launch_bounds__(kGemmThreads, 1) umma_gemm_kernel(
    const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int M,
    int N, int K, int S, int mode, const Epilogue ep, float* partial, int* err_word)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* epi = reinterpret_cast<float*>(base + kStages * kStageBytes);
    float* chain = epi + kEpiBytes / sizeof(float);
    uint64_t* full = reinterpret_cast<uint64_t*>(chain + kChain * 32);
    uint64_t* empty = full + kStages;
    uint64_t* tfull = empty + kStages;    // [2] accumulator b holds a finished tile
    uint64_t* tempty = tfull + 2;         // [2] accumulator b has been drained
    uint64_t* mdone = tempty + 2;         // every MMA issued by this block is done
    uint64_t* linked = mdone + 1;         // [kChain] column-sum hand-over ready
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(linked + kChain);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            rad::mbar_init(&full[s], 1);
            rad::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            rad::mbar_init(&tfull[b], 1);
            rad::mbar_init(&tempty[b], kEpiWarps);
        }
        rad::mbar_init(mdone, 1);
        for (int q = 0; q < kChain; ++q) rad::mbar_init(&linked[q], 1);
        *abort_flag = 0;
        rad::fence_mbar_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    chain_wait();

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer: stage use counter `it` runs across tiles
            uint32_t it = 0;
            bool ok = true;
            TileCoord tc;
            for (int i = 0; ok && tile_at(i, M, N, K, S, mode, tc); ++i) {
                for (int kt = tc.kt0; kt < tc.kt1; ++kt, ++it) {
                    const int s = (int)(it % kStages);
                    const uint32_t u = it / kStages;
                    if (it >= (uint32_t)kStages &&
                        !rad::mbar_wait_bounded(&empty[s], (u - 1) & 1, abort_flag, err_word)) {
                        ok = false;
                        break;
                    }
                    rad::mbar_arrive_expect_tx(&full[s], kStageBytes);
                    unsigned char* st = base + s * kStageBytes;
                    if (mode & kAMajorM) {
                        tma_load_2d(st, &tmA, tc.m0, kt * BK, &full[s]);
                        tma_load_2d(st + kTileBytes / 2, &tmA, tc.m0 + 64, kt * BK, &full[s]);
                    } else {
                        tma_load_2d(st, &tmA, kt * BK, tc.m0, &full[s]);
                    }
                    st += kTileBytes;
                    if (mode & kBMajorN) {
                        tma_load_2d(st, &tmB, tc.n0, kt * BK, &full[s]);
                        tma_load_2d(st + kTileBytes / 2, &tmB, tc.n0 + 64, kt * BK, &full[s]);
                    } else {
                        tma_load_2d(st, &tmB, kt * BK, tc.n0, &full[s]);
                    }
                }
            }
            if (!ok || *abort_flag) {
                // never leave with a copy in flight: wait (bounded) for the last
                // kStages issued loads to land
                for (uint32_t j = it > (uint32_t)kStages ? it - kStages : 0; j < it; ++j)
                    rad::mbar_drain(&full[j % kStages], (j / kStages) & 1);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer: tile i of this block goes to accumulator i & 1
            uint32_t it = 0, i = 0;
            bool ok = true;
            const bool amn = mode & kAMajorM, bmn = mode & kBMajorN;
            const uint64_t ad = amn ? kDescMN : kDescK, bd = bmn ? kDescMN : kDescK;
            const uint32_t as = (amn ? 2048 : 32) >> 4, bs = (bmn ? 2048 : 32) >> 4;
            const uint32_t idesc = kIdesc | (amn ? 1u << 15 : 0u) | (bmn ? 1u << 16 : 0u);
            TileCoord tc;
            for (; ok && tile_at((int)i, M, N, K, S, mode, tc); ++i) {
                const int ab = (int)(i & 1);
                const uint32_t use = i >> 1;
                if (use >= 1 &&
                    !rad::mbar_wait_bounded(&tempty[ab], (use - 1) & 1, abort_flag, err_word))
                    break;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(ab * BN);
                for (int kt = tc.kt0; kt < tc.kt1; ++kt, ++it) {
                    const int s = (int)(it % kStages);
                    const uint32_t u = it / kStages;
                    if (!rad::mbar_wait_bounded(&full[s], u & 1, abort_flag, err_word)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a0 = smem_addr(base + s * kStageBytes);
                    const uint32_t b0 = a0 + kTileBytes;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        umma_bf16(d, ad + (a0 >> 4) + as * kk, bd + (b0 >> 4) + bs * kk, idesc,
                                  (kt > tc.kt0 || kk > 0) ? 1u : 0u);
                    umma_commit(&empty[s]);
                }
                if (ok) umma_commit(&tfull[ab]);
            }
            // completes once every MMA issued above is done (also after an abort)
            umma_commit(mdone);
            rad::mbar_drain(mdone, 0);
        }
    } else {
        // ---- epilogue: warp w may read TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31,
        // the accumulator rows of that quarter; warps 2-5 take columns 0-63 and
        // warps 6-9 columns 64-127.  Each 32 x 32 block goes TMEM ->
        // registers (one row per lane) -> this warp's staging (float4 slots
        // XOR-swizzled by row, conflict-free both ways) -> registers (four
        // consecutive columns per lane, eight lanes per row), so every global
        // access of a warp covers four whole 128-byte row segments.
        const int lg = warp & 3, cbase = ((warp - 2) >> 2) * (BN / 2);
        float* stage = epi + (warp - 2) * 32 * 32;
        const int qi = lane & 7, ri = lane >> 3;
        const int rows = ep.rows ? ep.rows : M;
        double loss = 0.0;
        uint32_t i = 0;
        bool up = true;
        TileCoord tc;
        for (; up && tile_at((int)i, M, N, K, S, mode, tc); ++i) {
            const int ab = (int)(i & 1);
            const int row0 = tc.m0 + lg * 32 + ri;       // this lane's rows: row0 + 4 k
            float4 ls = make_float4(0, 0, 0, 0);
            const bool ready = rad::mbar_wait_bounded(&tfull[ab], (i >> 1) & 1, abort_flag, err_word);
            // tcgen05.ld below is warp-collective: the whole warp goes on or stops
            if (!__all_sync(0xffffffffu, ready && !*abort_flag)) break;
            tc_fence_after();
#pragma unroll 1
            for (int c0 = cbase; up && c0 < cbase + BN / 2; c0 += 32) {
                const int n = tc.n0 + c0 + 4 * qi;
                // loss: the targets of all eight rows at once (one round of memory latency)
                float4 tg[8];
                if (EPI == kEpiLoss) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (row0 + 4 * k < rows)
                            tg[k] = __ldcs(reinterpret_cast<const float4*>(
                                ep.target + (size_t)(row0 + 4 * k) * N + n));
                }
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(ab * BN + c0), v);
                float4* srow = reinterpret_cast<float4*>(stage + lane * 32);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    srow[j ^ (lane & 7)] =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                __syncwarp();
                float4 b4 = make_float4(0, 0, 0, 0);
                if (ep.bias) b4 = *reinterpret_cast<const float4*>(ep.bias + n);
                if constexpr (EPI == kEpiLoss) {
                    // loss and its gradient (no other output)
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int r = 4 * k + ri;
                        float4& x = reinterpret_cast<float4*>(stage + r * 32)[qi ^ (r & 7)];
                        float g[4] = {0, 0, 0, 0};
                        if (row0 + 4 * k < rows) {
                            const float d[4] = {(x.x + b4.x) - tg[k].x, (x.y + b4.y) - tg[k].y,
                                                (x.z + b4.z) - tg[k].z, (x.w + b4.w) - tg[k].w};
                            ls.x = fmaf(d[0], d[0], ls.x);
                            ls.y = fmaf(d[1], d[1], ls.y);
                            ls.z = fmaf(d[2], d[2], ls.z);
                            ls.w = fmaf(d[3], d[3], ls.w);
#pragma unroll
                            for (int c = 0; c < 4; ++c) g[c] = ep.scale * d[c];
                        }
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(g[0], g[1]);
                        const __nv_bfloat162 hi = __floats2bfloat162_rn(g[2], g[3]);
                        *reinterpret_cast<uint2*>(ep.out_bf16 + (size_t)(row0 + 4 * k) * N + n) =
                            make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                                       *reinterpret_cast<const uint32_t*>(&hi));
                        const float4 g4 = make_float4(g[0], g[1], g[2], g[3]);
                        if (ep.out_f32)
                            *reinterpret_cast<float4*>(ep.out_f32 + (size_t)(row0 + 4 * k) * N + n) = g4;
                        if (ep.colsum) x = g4;
                    }
                    __syncwarp();
                    if (ep.colsum) {
                        // A lane adds one column's 32 rows, going on from the sum of the
                        // rows before: the warp of the previous 32, or the last warp's sum
                        // of the previous row tile.  Row order, so that the bias gradient
                        // does not depend on the tiling.  A slot is
                        // written again two tiles on, when its reader has handed the
                        // accumulator back (or, across tiles, has itself been read on).
                        float cv[32];
#pragma unroll
                        for (int r = 0; r < 32; ++r)
                            cv[r] = stage[r * 32 + (((lane >> 2) ^ (r & 7)) << 2) + (lane & 3)];
                        const int link = 4 * (cbase / 32) + (c0 - cbase) / 8 + lg;   // 4 of 32 columns
                        float sum = 0.0f;
                        if (lg || tc.m0) {
                            const uint32_t it = lg ? i : i - 1;
                            const int from = (int)(it & 1) * (kChain / 2) + (lg ? link - 1 : link + 3);
                            const bool got = rad::mbar_wait_bounded(&linked[from], (it >> 1) & 1,
                                                                    abort_flag, err_word);
                            up = __all_sync(0xffffffffu, got && !*abort_flag);
                            sum = chain[from * 32 + lane];
                        }
#pragma unroll
                        for (int r = 0; r < 32; ++r) sum += cv[r];
                        const int to = ab * (kChain / 2) + link;
                        chain[to * 32 + lane] = sum;
                        if (lg == 3 && tc.m0 + BM == M) ep.colsum[tc.n0 + c0 + lane] = sum;
                        __syncwarp();
                        if (lane == 0) rad::mbar_arrive(&linked[to]);
                    }
                } else {
#pragma unroll 2
                    for (int k = 0; k < 8; ++k) {
                        const int r = 4 * k + ri;
                        float4 x = reinterpret_cast<const float4*>(stage + r * 32)[qi ^ (r & 7)];
                        const size_t o = (size_t)(row0 + 4 * k) * N + n;
                        if (EPI == kEpiPower) {
                            if (row0 + 4 * k < rows) {
                                const float4 mu = *reinterpret_cast<const float4*>(ep.mu + n);
                                const float4 sd = *reinterpret_cast<const float4*>(ep.sd + n);
                                x.x = exp10f(fmaf(x.x + b4.x, sd.x, mu.x));
                                x.y = exp10f(fmaf(x.y + b4.y, sd.y, mu.y));
                                x.z = exp10f(fmaf(x.z + b4.z, sd.z, mu.z));
                                x.w = exp10f(fmaf(x.w + b4.w, sd.w, mu.w));
                                *reinterpret_cast<float4*>(ep.out_f32 + o) = x;
                            }
                            continue;
                        }
                        if (partial) {
                            *reinterpret_cast<float4*>(partial + (size_t)tc.z * M * N + o) = x;
                            continue;
                        }
                        x.x += b4.x;
                        x.y += b4.y;
                        x.z += b4.z;
                        x.w += b4.w;
                        if (ep.mask) {
                            const float4 q = *reinterpret_cast<const float4*>(ep.mask + o);
                            x.x = q.x > 0.0f ? x.x : 0.0f;
                            x.y = q.y > 0.0f ? x.y : 0.0f;
                            x.z = q.z > 0.0f ? x.z : 0.0f;
                            x.w = q.w > 0.0f ? x.w : 0.0f;
                        }
                        if (ep.out_f32 && row0 + 4 * k < rows) *reinterpret_cast<float4*>(ep.out_f32 + o) = x;
                        if (ep.out_bf16) {
                            if (ep.relu) {
                                x.x = fmaxf(x.x, 0.0f);
                                x.y = fmaxf(x.y, 0.0f);
                                x.z = fmaxf(x.z, 0.0f);
                                x.w = fmaxf(x.w, 0.0f);
                            }
                            const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y);
                            const __nv_bfloat162 hi = __floats2bfloat162_rn(x.z, x.w);
                            *reinterpret_cast<uint2*>(ep.out_bf16 + o) =
                                make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                                           *reinterpret_cast<const uint32_t*>(&hi));
                        }
                    }
                    __syncwarp();
                }
            }
            // this warp's reads of the accumulator are complete: hand it back
            tc_fence_before();
            __syncwarp();
            if (lane == 0) rad::mbar_arrive(&tempty[ab]);
            if (EPI == kEpiLoss) {
                float l = (ls.x + ls.y) + (ls.z + ls.w);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
                loss += (double)l;
            }
        }
        if (EPI == kEpiLoss && lane == 0) ep.loss_part[blockIdx.x * kEpiWarps + warp - 2] = loss;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols)
                     : "memory");
}

// Sum of the S slices' partials in slice order, then the epilogue of the
// unsplit kernel (four consecutive outputs per thread; N is a multiple of 128).
__global__ void splitk_reduce(const float* partial, int S, int M, int N, const Epilogue ep)
{
    chain_wait();
    const int64_t MN = (int64_t)M * N, n4 = MN / 4;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n4;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = 4 * q;
        float4 v = *reinterpret_cast<const float4*>(partial + o);
        for (int s = 1; s < S; ++s) {
            const float4 p = *reinterpret_cast<const float4*>(partial + s * MN + o);
            v.x += p.x;
            v.y += p.y;
            v.z += p.z;
            v.w += p.w;
        }
        float r[4] = {v.x, v.y, v.z, v.w};
        const int n = (int)(o % N);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (ep.bias) r[c] += ep.bias[n + c];
            if (ep.mask) r[c] = ep.mask[o + c] > 0.0f ? r[c] : 0.0f;
        }
        if (ep.mu) {
#pragma unroll
            for (int c = 0; c < 4; ++c) r[c] = exp10f(fmaf(r[c], ep.sd[n + c], ep.mu[n + c]));
        }
        if (ep.out_f32 && (!ep.rows || o / N < ep.rows))
            *reinterpret_cast<float4*>(ep.out_f32 + o) = make_float4(r[0], r[1], r[2], r[3]);
        if (ep.out_bf16) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (ep.relu) r[c] = fmaxf(r[c], 0.0f);
            __nv_bfloat162* d = reinterpret_cast<__nv_bfloat162*>(ep.out_bf16 + o);
            d[0] = __floats2bfloat162_rn(r[0], r[1]);
            d[1] = __floats2bfloat162_rn(r[2], r[3]);
        }
    }
}

// The loss epilogue of a split product (an output layer with few tiles and a long K): a
// block per 32 rows x 128 columns sums the slices in slice order, a warp per row.
__global__ void __launch_bounds__(256) splitk_loss(const float* partial, int S, int M, int N,
                                                   const Epilogue ep)
{
    chain_wait();
    __shared__ float share[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = blockIdx.x * 128 + 4 * lane;
    const size_t MN = (size_t)M * N;
    const float4 b4 = *reinterpret_cast<const float4*>(ep.bias + n);
    float l = 0.0f;
    for (int r = blockIdx.y * 32 + warp; r < (int)blockIdx.y * 32 + 32; r += 8) {
        const size_t o = (size_t)r * N + n;
        float4 g = make_float4(0, 0, 0, 0);
        if (r < ep.rows) {
            float4 v = *reinterpret_cast<const float4*>(partial + o);
            for (int s = 1; s < S; ++s) {
                const float4 p = *reinterpret_cast<const float4*>(partial + s * MN + o);
                v.x += p.x;
                v.y += p.y;
                v.z += p.z;
                v.w += p.w;
            }
            const float4 t = *reinterpret_cast<const float4*>(ep.target + o);
            const float4 d = make_float4((v.x + b4.x) - t.x, (v.y + b4.y) - t.y, (v.z + b4.z) - t.z,
                                         (v.w + b4.w) - t.w);
            l += (d.x * d.x + d.y * d.y) + (d.z * d.z + d.w * d.w);
            g = make_float4(ep.scale * d.x, ep.scale * d.y, ep.scale * d.z, ep.scale * d.w);
        }
        *reinterpret_cast<float4*>(ep.out_f32 + o) = g;
        __nv_bfloat162* out = reinterpret_cast<__nv_bfloat162*>(ep.out_bf16 + o);
        out[0] = __floats2bfloat162_rn(g.x, g.y);
        out[1] = __floats2bfloat162_rn(g.z, g.w);
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) share[warp] = l;
    __syncthreads();
    if (threadIdx.x) return;
    for (int w = 1; w < 8; ++w) l += share[w];
    ep.loss_part[blockIdx.y * gridDim.x + blockIdx.x] = (double)l;
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// Row-major BF16 [rows][ld] viewed as rows x cols; box 64 columns x box_rows, 128-byte
// swizzle.
bool make_map(CUtensorMap* map, const bf16* ptr, int rows, int cols, int ld, int box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(bf16)};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(ptr), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Whether a block takes the row tiles of its column tile in turn.  Pays when the row tiles
// share a B too wide for L2 (the output layer at a batch above 128: 403 MB of weights read
// once instead of once per 128 rows); the blocks then differ by a whole column of tiles,
// at most 1/8 of the work from eight columns per block on.
bool rows_inner(int M, int N) { return M > BM && N / BN >= 8 * device_sms(); }

// Whether the loss epilogue can form g's column sums: the row tiles of a column meet in one
// block, in order.
bool sums_in_epilogue(int M, int N, int K)
{
    return split_count(M, N, K) == 1 && (M == BM || rows_inner(M, N));
}

// Blocks of an M x N product split into S slices.
int gemm_grid(int M, int N, int S)
{
    return std::min(S == 1 && rows_inner(M, N) ? N / BN : (M / BM) * (N / BN) * S, device_sms());
}

// Entries of loss_part that the loss epilogue writes: one per epilogue warp, or when the
// product is split one per 32 x 128 outputs (fewer than device_sms() tiles then).
int loss_shares(int M, int N, int K)
{
    return split_count(M, N, K) > 1 ? (M / 32) * (N / 128) : gemm_grid(M, N, 1) * kEpiWarps;
}

// C [M][N] = A [M][K] B [N][K]^T with the fused epilogue.  mode: A is stored [M][lda], or
// with kAMajorM [K][lda]; B [N][ldb], or with kBMajorN [K][ldb].  work: FP32 scratch of at
// least split_count(M, N, K) * M * N floats, or null to run unsplit.
cudaError_t gemm_tn(const bf16* A, int lda, const bf16* B, int ldb, int mode, int M, int N, int K,
                    const Epilogue& ep, cudaStream_t st, float* work, int* err_word)
{
    const bool amn = mode & kAMajorM, bmn = mode & kBMajorN;
    if (M % BM || N % BN || K % BK || K < BK || lda % 8 || ldb % 8 || lda < (amn ? M : K) ||
        ldb < (bmn ? N : K) ||
        (reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) % 16 || !err_word) {
        fail(RAD_MLP_EINVAL, "gemm: shape, leading dimension or alignment not supported");
        return cudaErrorInvalidValue;
    }
    const int S = work ? split_count(M, N, K) : 1;
    const auto kernel = S > 1     ? umma_gemm_kernel<kEpiPlain>
                        : ep.target ? umma_gemm_kernel<kEpiLoss>
                        : ep.mu     ? umma_gemm_kernel<kEpiPower>
                                    : umma_gemm_kernel<kEpiPlain>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kGemmSmem);
    if (e != cudaSuccess) {
        fail(RAD_MLP_ECUDA, "gemm: shared-memory attribute", e);
        return e;
    }
    CUtensorMap ma, mb;
    if (!(amn ? make_map(&ma, A, K, M, lda, BK) : make_map(&ma, A, M, K, lda, BM)) ||
        !(bmn ? make_map(&mb, B, K, N, ldb, BK) : make_map(&mb, B, N, K, ldb, BN))) {
        fail(RAD_MLP_EINVAL, "gemm: tensor map encoding failed");
        return cudaErrorInvalidValue;
    }
    if (S == 1 && rows_inner(M, N)) mode |= kRowsInner;
    e = launch(kernel, gemm_grid(M, N, S), kGemmThreads, kGemmSmem, st, ma, mb, M, N, K, S, mode, ep,
               S > 1 ? work : nullptr, err_word);
    if (e == cudaSuccess && S > 1 && ep.target) {
        e = launch(splitk_loss, dim3(N / 128, M / 32), 256, 0, st, work, S, M, N, ep);
    } else if (e == cudaSuccess && S > 1) {
        const int64_t n4 = (int64_t)M * N / 4;
        // whole 4 KB rows per block: 64-thread blocks, which reach every SM, took twice as long
        // on 76 slices of 128 x 512 outputs
        const int blocks = (int)std::min<int64_t>((n4 + 255) / 256, 4 * device_sms());
        e = launch(splitk_reduce, blocks, 256, 0, st, work, S, M, N, ep);
    }
    if (e != cudaSuccess) fail(RAD_MLP_ECUDA, "gemm: launch", e);
    return e;
}

__global__ void to_bf16_rows(const float* x, bf16* y, int rows_valid, int rows, int cols)
{
    chain_wait();
    const int64_t n = (int64_t)rows * cols;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(i / cols);
        y[i] = __float2bfloat16_rn(r < rows_valid ? x[i] : 0.0f);
    }
}

// Input transform of rad_mlp_predict: h0 = BF16((log10(max(x, floor)) - mu) / sd)
// per feature (padded rows zero).
__global__ void log_standardise_rows(const float* __restrict__ x, bf16* __restrict__ y,
                                     const float* __restrict__ mu, const float* __restrict__ sd,
                                     float floor_v, int rows_valid, int rows, int cols)
{
    chain_wait();
    const int64_t n = (int64_t)rows * cols;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(i / cols), c = (int)(i - (int64_t)r * cols);
        float v = 0.0f;
        if (r < rows_valid) v = (log10f(fmaxf(x[i], floor_v)) - mu[c]) / sd[c];
        y[i] = __float2bfloat16_rn(v);
    }
}

// loss = sum of the n block shares / (rows_valid * cols), one block, fixed order.
__global__ void loss_sum(const double* part, int64_t n, double inv, double* loss)
{
    __shared__ double red[256];
    chain_wait();
    double a = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) a += part[i];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = red[0] * inv;
}

// Column sums db[n] = sum over rows of g[r][n] of several matrices in one launch: a warp per
// 32 columns, each thread adding its column in row order (unrolled: the loads of 16 rows
// are in flight at once).
constexpr int kMaxLayers = 16;
struct ColumnJobs {
    int n;
    const float* g[kMaxLayers];
    float* db[kMaxLayers];
    int cols[kMaxLayers], block0[kMaxLayers + 1];
};
__global__ void __launch_bounds__(32) column_sums(const ColumnJobs jobs, int rows)
{
    chain_wait();
    int q = 0;
    while (q + 1 < jobs.n && (int)blockIdx.x >= jobs.block0[q + 1]) ++q;
    const int cols = jobs.cols[q];
    const int n = ((int)blockIdx.x - jobs.block0[q]) * 32 + threadIdx.x;   // cols % 128 == 0
    const float* g = jobs.g[q] + n;
    float s = 0.0f;
#pragma unroll 16
    for (int r = 0; r < rows; ++r) s += g[(size_t)r * cols];
    jobs.db[q][n] = s;
}

// Adam on the FP32 master parameters of every layer in one launch; refreshes the BF16
// copies of the weights.  A block of 256 threads takes 1024 parameters, four per thread
// (16-byte accesses).  Bound by memory, 28 bytes per bias and 30 per weight: 201 M weights
// take 870 us, 6.9 TB/s (4-byte accesses with a transposed BF16 copy, 32 bytes: 1081 us).
// As an epilogue of the weight gradient it would save reading the gradient back, but that
// kernel's eight warps are too few for its divisions and square roots (2.2 ms against
// 151 + 870 us).
constexpr int kAdamBlock = 1024;
struct AdamJobs {
    int n;
    float* w[2 * kMaxLayers];
    bf16* wb[2 * kMaxLayers];       // null: no BF16 copy
    float* m[2 * kMaxLayers];
    float* v[2 * kMaxLayers];
    const float* g[2 * kMaxLayers];
    int64_t count[2 * kMaxLayers], block0[2 * kMaxLayers + 1];
};
__device__ __forceinline__ void adam_one(float g, float& m, float& v, float& w, float lr, float b1,
                                         float b2, float eps, float c1, float c2)
{
    m = __fmaf_rn(1.0f - b1, g, __fmul_rn(b1, m));
    v = __fmaf_rn(__fmul_rn(1.0f - b2, g), g, __fmul_rn(b2, v));
    w = w - lr * (m / c1) / (sqrtf(v / c2) + eps);
}
__global__ void __launch_bounds__(256) adam_update(const __grid_constant__ AdamJobs jobs, float lr,
                                                   float b1, float b2, float eps, float c1, float c2)
{
    chain_wait();
    int q = 0;
    while (q + 1 < jobs.n && (int64_t)blockIdx.x >= jobs.block0[q + 1]) ++q;
    const int64_t i = ((int64_t)blockIdx.x - jobs.block0[q]) * kAdamBlock + 4 * threadIdx.x;
    if (i >= jobs.count[q]) return;              // counts are multiples of 128
    const float4 g = __ldcs(reinterpret_cast<const float4*>(jobs.g[q] + i));
    float4 m = __ldcs(reinterpret_cast<const float4*>(jobs.m[q] + i));
    float4 v = __ldcs(reinterpret_cast<const float4*>(jobs.v[q] + i));
    float4 w = __ldcs(reinterpret_cast<const float4*>(jobs.w[q] + i));
    adam_one(g.x, m.x, v.x, w.x, lr, b1, b2, eps, c1, c2);
    adam_one(g.y, m.y, v.y, w.y, lr, b1, b2, eps, c1, c2);
    adam_one(g.z, m.z, v.z, w.z, lr, b1, b2, eps, c1, c2);
    adam_one(g.w, m.w, v.w, w.w, lr, b1, b2, eps, c1, c2);
    __stcs(reinterpret_cast<float4*>(jobs.m[q] + i), m);
    __stcs(reinterpret_cast<float4*>(jobs.v[q] + i), v);
    __stcs(reinterpret_cast<float4*>(jobs.w[q] + i), w);
    if (jobs.wb[q]) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y), hi = __floats2bfloat162_rn(w.z, w.w);
        *reinterpret_cast<uint2*>(jobs.wb[q] + i) = make_uint2(
            *reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
}

__global__ void f32_to_bf16(const float* x, bf16* y, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

int grid_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 4096); }

bool is_dev(const void* p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

struct rad_mlp {
    int L = 0;                      // layers
    std::vector<int> w;             // widths [L + 1]
    int max_rows = 0;               // max batch rounded up to 128
    cudaStream_t st = nullptr;
    // parameters: per layer, [out][in]
    std::vector<float*> W, b, Wm, Wv, bm, bv, dW, db;
    std::vector<bf16*> Wb;          // BF16 copy of W [out][in] (operand of both passes)
    int64_t step = 0;
    // activations: h[l] bf16 [rows][w[l]] (h[0] = input), z[l] fp32 [rows][w[l]] (l >= 1)
    std::vector<bf16*> h;
    std::vector<float*> z;
    float* t = nullptr;             // targets [rows][w[L]]
    std::vector<bf16*> gb;          // layer gradients bf16: gb[l] [rows][w[l]] for l >= 1
    double* loss = nullptr;
    double* loss_part = nullptr;    // loss shares of the output layer's epilogue
    float* xin = nullptr;           // staging for host inputs [rows][w[0]]
    float* work = nullptr;          // split-K partial sums (largest split product)
    float* in_mu = nullptr;         // rad_mlp_predict transforms [w[0]], [w[L]] (null: unset)
    float* in_sd = nullptr;
    float* out_mu = nullptr;
    float* out_sd = nullptr;
    float floor_v = 0.0f;
    int* err = nullptr;             // GEMM timeout word
    struct Back {                   // pinned: what a call reads back
        double loss;
        int err;
    }* back = nullptr;
};

#define MCU(call)                                                                  \
    do {                                                                           \
        const cudaError_t e_ = (call);                                             \
        if (e_ != cudaSuccess)                                                     \
            return e_ == cudaErrorInvalidValue ? fail(RAD_MLP_EINVAL, #call, e_)   \
                                               : fail(RAD_MLP_ECUDA, #call, e_);   \
    } while (0)

static int round128(int n) { return (n + 127) / 128 * 128; }

extern "C" {

int rad_mlp_init(rad_mlp** out, const int32_t* widths, int32_t n_layers, int32_t max_batch,
                 void* stream)
{
    if (!out || !widths || n_layers < 1 || n_layers > 16 || max_batch < 1) return RAD_MLP_EINVAL;
    *out = nullptr;
    for (int l = 0; l <= n_layers; ++l)
        if (widths[l] < 128 || widths[l] % 128) return RAD_MLP_EINVAL;
    rad_mlp* m = new (std::nothrow) rad_mlp();
    if (!m) return RAD_MLP_ENOMEM;
    m->L = n_layers;
    m->w.assign(widths, widths + n_layers + 1);
    m->max_rows = round128(max_batch);
    m->st = (cudaStream_t)stream;
    auto bail = [&](int rc) {
        rad_mlp_destroy(m);
        return rc;
    };
#define MAL(ptr, bytes)                                                          \
    do {                                                                         \
        cudaError_t e_ = cudaMalloc(&(ptr), (bytes));                            \
        if (e_ != cudaSuccess) return bail(e_ == cudaErrorMemoryAllocation ? RAD_MLP_ENOMEM : RAD_MLP_ECUDA); \
        cudaMemset((ptr), 0, (bytes));                                           \
    } while (0)
    const int R = m->max_rows;
    m->W.assign(n_layers, nullptr);
    m->b = m->Wm = m->Wv = m->bm = m->bv = m->dW = m->db = m->W;
    m->Wb.assign(n_layers, nullptr);
    m->h.assign(n_layers + 1, nullptr);
    m->z.assign(n_layers + 1, nullptr);
    m->gb.assign(n_layers + 1, nullptr);
    for (int l = 0; l < n_layers; ++l) {
        const size_t np = (size_t)m->w[l + 1] * m->w[l];
        MAL(m->W[l], np * 4);
        MAL(m->Wm[l], np * 4);
        MAL(m->Wv[l], np * 4);
        MAL(m->dW[l], np * 4);
        MAL(m->Wb[l], np * 2);
        MAL(m->b[l], (size_t)m->w[l + 1] * 4);
        MAL(m->bm[l], (size_t)m->w[l + 1] * 4);
        MAL(m->bv[l], (size_t)m->w[l + 1] * 4);
        MAL(m->db[l], (size_t)m->w[l + 1] * 4);
    }
    for (int l = 0; l <= n_layers; ++l) {
        MAL(m->h[l], (size_t)R * m->w[l] * 2);
        if (l >= 1) {
            MAL(m->z[l], (size_t)R * m->w[l] * 4);
            MAL(m->gb[l], (size_t)R * m->w[l] * 2);
        }
    }
    MAL(m->t, (size_t)R * m->w[n_layers] * 4);
    MAL(m->loss, sizeof(double));
    MAL(m->loss_part, (size_t)device_sms() * kEpiWarps * sizeof(double));
    MAL(m->xin, (size_t)R * m->w[0] * 4);
    // split-K scratch of the products that split: the forward and input-gradient products are
    // R rows wide (the weight gradient reduces over R itself and never splits)
    size_t work = 0;
    auto need = [&](int M, int N, int K) {
        const int S = split_count(M, N, K);
        if (S > 1) work = std::max(work, (size_t)S * M * N);
    };
    for (int l = 0; l < n_layers; ++l) {
        const int in = m->w[l], outw = m->w[l + 1];
        for (int rows = 128; rows <= R; rows += 128) {
            need(rows, outw, in);
            if (l > 0) need(rows, in, outw);
        }
    }
    MAL(m->work, work * 4);
#undef MAL
    m->err = gemm_err_word();
    if (!m->err) return bail(RAD_MLP_ECUDA);
    if (cudaMallocHost(reinterpret_cast<void**>(&m->back), sizeof *m->back) != cudaSuccess)
        return bail(RAD_MLP_ENOMEM);
    if (cudaDeviceSynchronize() != cudaSuccess) return bail(RAD_MLP_ECUDA);
    *out = m;
    return RAD_MLP_OK;
}

int rad_mlp_set_layer(rad_mlp* m, int32_t layer, const float* W, const float* b)
{
    if (!m || layer < 0 || layer >= m->L || !W || !b) return RAD_MLP_EINVAL;
    const size_t np = (size_t)m->w[layer + 1] * m->w[layer];
    MCU(cudaMemcpyAsync(m->W[layer], W, np * 4, cudaMemcpyDefault, m->st));
    MCU(cudaMemcpyAsync(m->b[layer], b, (size_t)m->w[layer + 1] * 4, cudaMemcpyDefault, m->st));
    f32_to_bf16<<<grid_for(np), 256, 0, m->st>>>(m->W[layer], m->Wb[layer], (int64_t)np);
    MCU(cudaGetLastError());
    // a new parameter set restarts the optimiser
    MCU(cudaMemsetAsync(m->Wm[layer], 0, np * 4, m->st));
    MCU(cudaMemsetAsync(m->Wv[layer], 0, np * 4, m->st));
    MCU(cudaMemsetAsync(m->bm[layer], 0, (size_t)m->w[layer + 1] * 4, m->st));
    MCU(cudaMemsetAsync(m->bv[layer], 0, (size_t)m->w[layer + 1] * 4, m->st));
    m->step = 0;
    MCU(cudaStreamSynchronize(m->st));
    return RAD_MLP_OK;
}

int rad_mlp_get_layer(rad_mlp* m, int32_t layer, float* W, float* b, float* dW, float* db)
{
    if (!m || layer < 0 || layer >= m->L) return RAD_MLP_EINVAL;
    const size_t np = (size_t)m->w[layer + 1] * m->w[layer];
    const size_t nb = (size_t)m->w[layer + 1] * 4;
    if (W) MCU(cudaMemcpyAsync(W, m->W[layer], np * 4, cudaMemcpyDefault, m->st));
    if (b) MCU(cudaMemcpyAsync(b, m->b[layer], nb, cudaMemcpyDefault, m->st));
    if (dW) MCU(cudaMemcpyAsync(dW, m->dW[layer], np * 4, cudaMemcpyDefault, m->st));
    if (db) MCU(cudaMemcpyAsync(db, m->db[layer], nb, cudaMemcpyDefault, m->st));
    MCU(cudaStreamSynchronize(m->st));
    return RAD_MLP_OK;
}

// Forward pass; the output layer's results go where `out` says (its bias is set here).
static int forward(rad_mlp* m, int32_t batch, const float* x, Epilogue out, bool transform = false)
{
    const int R = round128(batch);
    const float* xd = x;
    if (!is_dev(x)) {
        MCU(cudaMemcpyAsync(m->xin, x, (size_t)batch * m->w[0] * 4, cudaMemcpyHostToDevice, m->st));
        xd = m->xin;
    }
    if (transform)
        MCU(launch(log_standardise_rows, grid_for((int64_t)R * m->w[0]), 256, 0, m->st, xd, m->h[0],
                   m->in_mu, m->in_sd, m->floor_v, batch, R, m->w[0]));
    else
        MCU(launch(to_bf16_rows, grid_for((int64_t)R * m->w[0]), 256, 0, m->st, xd, m->h[0], batch, R,
                   m->w[0]));
    for (int l = 0; l < m->L; ++l) {
        Epilogue ep;
        if (l == m->L - 1) {
            ep = out;
        } else {
            ep.out_f32 = m->z[l + 1];
            ep.out_bf16 = m->h[l + 1];
            ep.relu = 1;
        }
        ep.bias = m->b[l];
        // z = h W^T + b: A = h [R][in], B = W [out][in].
        MCU(gemm_tn(m->h[l], m->w[l], m->Wb[l], m->w[l], 0, R, m->w[l + 1], m->w[l], ep, m->st,
                    m->work, m->err));
    }
    return RAD_MLP_OK;
}

// Waits for the call's work; the loss and the timeout word come back in the same wait (a
// second, blocking copy of the word cost 10 us per call).
static int finish(rad_mlp* m, double* loss)
{
    if (loss)
        MCU(cudaMemcpyAsync(&m->back->loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->st));
    MCU(cudaMemcpyAsync(&m->back->err, m->err, sizeof(int), cudaMemcpyDeviceToHost, m->st));
    MCU(cudaStreamSynchronize(m->st));
    if (loss) *loss = m->back->loss;
    if (!m->back->err) return RAD_MLP_OK;
    MCU(cudaMemset(m->err, 0, sizeof(int)));
    return RAD_MLP_ETIMEOUT;
}

// Memory of this device that the output layer's epilogue can write (read) in 16-byte
// accesses; anything else goes through a staging buffer.
static bool direct(const float* p)
{
    cudaPointerAttributes a;
    int dev = -1;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == dev)) &&
           reinterpret_cast<uintptr_t>(p) % 16 == 0;
}

int rad_mlp_forward(rad_mlp* m, int32_t batch, const float* x, float* y)
{
    if (!m || batch < 1 || batch > m->max_rows || !x || !y) return RAD_MLP_EINVAL;
    const bool in_place = direct(y);
    Epilogue out;
    out.out_f32 = in_place ? y : m->z[m->L];
    out.rows = batch;
    int rc = forward(m, batch, x, out);
    if (rc) return rc;
    if (!in_place)
        MCU(cudaMemcpyAsync(y, m->z[m->L], (size_t)batch * m->w[m->L] * 4, cudaMemcpyDefault, m->st));
    return finish(m, nullptr);
}

int rad_mlp_set_transform(rad_mlp* m, const float* in_mu, const float* in_sd, const float* out_mu,
                          const float* out_sd, float floor_value)
{
    if (!m || !in_mu || !in_sd || !out_mu || !out_sd || !(floor_value > 0.0f))
        return fail(RAD_MLP_EINVAL, "rad_mlp_set_transform: null statistics or floor <= 0");
    const int wi = m->w[0], wo = m->w[m->L];
    if (!m->in_mu) {
        MCU(cudaMalloc(&m->in_mu, (size_t)wi * 4));
        MCU(cudaMalloc(&m->in_sd, (size_t)wi * 4));
        MCU(cudaMalloc(&m->out_mu, (size_t)wo * 4));
        MCU(cudaMalloc(&m->out_sd, (size_t)wo * 4));
    }
    MCU(cudaMemcpyAsync(m->in_mu, in_mu, (size_t)wi * 4, cudaMemcpyDefault, m->st));
    MCU(cudaMemcpyAsync(m->in_sd, in_sd, (size_t)wi * 4, cudaMemcpyDefault, m->st));
    MCU(cudaMemcpyAsync(m->out_mu, out_mu, (size_t)wo * 4, cudaMemcpyDefault, m->st));
    MCU(cudaMemcpyAsync(m->out_sd, out_sd, (size_t)wo * 4, cudaMemcpyDefault, m->st));
    MCU(cudaStreamSynchronize(m->st));
    m->floor_v = floor_value;
    return RAD_MLP_OK;
}

int rad_mlp_predict(rad_mlp* m, int32_t batch, const float* x, float* y)
{
    if (!m || batch < 1 || batch > m->max_rows || !x || !y) return RAD_MLP_EINVAL;
    if (!m->in_mu) return fail(RAD_MLP_EINVAL, "rad_mlp_predict: no transform set");
    const int wo = m->w[m->L];
    const bool in_place = direct(y);
    Epilogue out;
    out.out_f32 = in_place ? y : m->z[m->L];
    out.rows = batch;
    out.mu = m->out_mu;
    out.sd = m->out_sd;
    int rc = forward(m, batch, x, out, true);
    if (rc) return rc;
    if (!in_place)
        MCU(cudaMemcpyAsync(y, m->z[m->L], (size_t)batch * wo * 4, cudaMemcpyDefault, m->st));
    return finish(m, nullptr);
}

// Forward, MSE and backward, enqueued on the stream (no host synchronisation).
static int backward(rad_mlp* m, int32_t batch, const float* x, const float* t)
{
    const int R = round128(batch);
    const int L = m->L, wo = m->w[L];
    // aligned device targets are read in place (only the batch's rows are touched)
    const float* td = t;
    if (!direct(t)) {
        MCU(cudaMemcpyAsync(m->t, t, (size_t)batch * wo * 4, cudaMemcpyDefault, m->st));
        td = m->t;
    }
    // forward pass whose output epilogue forms the loss shares, the BF16 output gradient
    // g = 2 (y - t) / (batch * out) and the FP32 gradient's column sums (or, where those
    // cannot be had there, the FP32 gradient)
    const bool summed = sums_in_epilogue(R, wo, m->w[L - 1]);
    Epilogue out;
    out.out_bf16 = m->gb[L];
    out.rows = batch;
    out.target = td;
    out.scale = (float)(2.0 / ((double)batch * wo));
    (summed ? out.colsum : out.out_f32) = summed ? m->db[L - 1] : m->z[L];
    out.loss_part = m->loss_part;
    const int rc = forward(m, batch, x, out);
    if (rc) return rc;
    MCU(launch(loss_sum, 1, 256, 0, m->st, m->loss_part, loss_shares(R, wo, m->w[L - 1]),
               1.0 / ((double)batch * wo), m->loss));
    for (int l = L - 1; l >= 0; --l) {
        const int in = m->w[l], outw = m->w[l + 1];
        if (l > 0) {
            // G_prev = (G W) * [z_l > 0]: A = G [R][out], B = W read [out][in]; the FP32
            // product lands in z_l's buffer for the bias sum
            Epilogue eg;
            eg.mask = m->z[l];
            eg.out_f32 = m->z[l];
            eg.out_bf16 = m->gb[l];
            MCU(gemm_tn(m->gb[l + 1], outw, m->Wb[l], in, kBMajorN, R, in, outw, eg, m->st, m->work,
                        m->err));
        }
        // dW = G^T H over the batch: G [R][out] and H [R][in] read batch-major in place
        Epilogue ew;
        ew.out_f32 = m->dW[l];
        MCU(gemm_tn(m->gb[l + 1], outw, m->h[l], in, kAMajorM | kBMajorN, outw, in, R, ew, m->st,
                    nullptr, m->err));
    }
    // the other bias gradients: column sums of the FP32 gradients
    ColumnJobs jobs{};
    for (int l = 0; l < (summed ? L - 1 : L); ++l) {
        jobs.g[l] = m->z[l + 1];
        jobs.cols[l] = m->w[l + 1];
        jobs.db[l] = m->db[l];
        jobs.block0[l + 1] = jobs.block0[l] + m->w[l + 1] / 32;
        jobs.n = l + 1;
    }
    if (jobs.n) MCU(launch(column_sums, jobs.block0[jobs.n], 32, 0, m->st, jobs, R));
    return RAD_MLP_OK;
}

int rad_mlp_gradients(rad_mlp* m, int32_t batch, const float* x, const float* t, double* loss)
{
    if (!m || batch < 1 || batch > m->max_rows || !x || !t) return RAD_MLP_EINVAL;
    const int rc = backward(m, batch, x, t);
    return rc ? rc : finish(m, loss);
}

// One Adam step of every layer from the stored gradients, enqueued.
static int adam_enqueue(rad_mlp* m, float lr, float beta1, float beta2, float eps)
{
    m->step += 1;
    const float c1 = 1.0f - std::pow(beta1, (float)m->step);
    const float c2 = 1.0f - std::pow(beta2, (float)m->step);
    AdamJobs jobs{};
    for (int l = 0; l < m->L; ++l)
        for (int bias = 0; bias < 2; ++bias) {
            const int q = jobs.n++;
            jobs.w[q] = bias ? m->b[l] : m->W[l];
            jobs.wb[q] = bias ? nullptr : m->Wb[l];
            jobs.m[q] = bias ? m->bm[l] : m->Wm[l];
            jobs.v[q] = bias ? m->bv[l] : m->Wv[l];
            jobs.g[q] = bias ? m->db[l] : m->dW[l];
            jobs.count[q] = (int64_t)m->w[l + 1] * (bias ? 1 : m->w[l]);
            jobs.block0[q + 1] = jobs.block0[q] + (jobs.count[q] + kAdamBlock - 1) / kAdamBlock;
        }
    MCU(launch(adam_update, (unsigned)jobs.block0[jobs.n], 256, 0, m->st, jobs, lr, beta1, beta2, eps,
               c1, c2));
    return RAD_MLP_OK;
}

static bool adam_args_ok(float lr, float beta1, float beta2)
{
    return lr > 0.0f && beta1 >= 0.0f && beta1 < 1.0f && beta2 >= 0.0f && beta2 < 1.0f;
}

int rad_mlp_adam(rad_mlp* m, float lr, float beta1, float beta2, float eps)
{
    if (!m || !adam_args_ok(lr, beta1, beta2)) return RAD_MLP_EINVAL;
    return adam_enqueue(m, lr, beta1, beta2, eps);
}

int rad_mlp_train_step(rad_mlp* m, int32_t batch, const float* x, const float* t, float lr,
                       float beta1, float beta2, float eps, double* loss)
{
    if (!m || batch < 1 || batch > m->max_rows || !x || !t || !adam_args_ok(lr, beta1, beta2))
        return RAD_MLP_EINVAL;
    int rc = backward(m, batch, x, t);
    if (!rc) rc = adam_enqueue(m, lr, beta1, beta2, eps);
    return rc ? rc : finish(m, loss);
}

int rad_mlp_gemm(int32_t a_kcontig, int32_t b_kcontig, int32_t M, int32_t N, int32_t K, const void* A,
                 const void* B, float* C)
{
    if (M < 1 || N < 1 || K < 1 || M % BM || N % BN || K % BK || !A || !B || !C)
        return fail(RAD_MLP_EINVAL, "rad_mlp_gemm: M, N must be multiples of 128 and K of 64");
    // the kernels load A and B by TMA and write C directly: host memory is
    // refused here instead of faulting inside a launch
    if (!is_dev(A) || !is_dev(B) || !is_dev(C))
        return fail(RAD_MLP_EINVAL, "rad_mlp_gemm: A, B and C must be device or managed memory");
    int* err = gemm_err_word();
    if (!err) return fail(RAD_MLP_ECUDA, "rad_mlp_gemm: error word");
    if (reinterpret_cast<uintptr_t>(C) % 16)
        return fail(RAD_MLP_EINVAL, "rad_mlp_gemm: C must be 16-byte aligned");
    Epilogue ep;
    ep.out_f32 = C;
    // scratch from the default stream's stream-ordered pool: split-K partials, and aligned
    // copies of M- or N-major operands that TMA cannot read where they are
    const int S = split_count(M, N, K);
    const bool ca = !a_kcontig && reinterpret_cast<uintptr_t>(A) % 16;
    const bool cb = !b_kcontig && reinterpret_cast<uintptr_t>(B) % 16;
    const size_t part = S > 1 ? (size_t)S * M * N * 4 : 0;
    const size_t at = ca ? (size_t)M * K * 2 : 0, bt = cb ? (size_t)N * K * 2 : 0;
    unsigned char* scratch = nullptr;
    if (part + at + bt &&
        cudaMallocAsync(reinterpret_cast<void**>(&scratch), part + at + bt, nullptr) != cudaSuccess)
        return fail(RAD_MLP_ENOMEM, "rad_mlp_gemm: scratch", cudaGetLastError());
    cudaError_t e = cudaSuccess;
    if (ca) {
        e = cudaMemcpyAsync(scratch + part, A, at, cudaMemcpyDefault, nullptr);
        A = scratch + part;
    }
    if (e == cudaSuccess && cb) {
        e = cudaMemcpyAsync(scratch + part + at, B, bt, cudaMemcpyDefault, nullptr);
        B = scratch + part + at;
    }
    if (e == cudaSuccess)
        e = gemm_tn(static_cast<const bf16*>(A), a_kcontig ? K : M, static_cast<const bf16*>(B),
                    b_kcontig ? K : N, (a_kcontig ? 0 : kAMajorM) | (b_kcontig ? 0 : kBMajorN), M, N, K, ep, nullptr,
                    part ? reinterpret_cast<float*>(scratch) : nullptr, err);
    if (scratch) cudaFreeAsync(scratch, nullptr);
    if (e == cudaErrorInvalidValue) return RAD_MLP_EINVAL;
    return e == cudaSuccess ? RAD_MLP_OK : RAD_MLP_ECUDA;
}

int rad_mlp_check(void)
{
    const cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return fail(RAD_MLP_ECUDA, "rad_mlp_check", e);
    return gemm_timed_out() ? fail(RAD_MLP_ETIMEOUT, "a GEMM block's bounded wait expired")
                            : RAD_MLP_OK;
}

const char* rad_mlp_last_error(void) { return g_last_error; }

void rad_mlp_destroy(rad_mlp* m)
{
    if (!m) return;
    if (m->st) cudaStreamSynchronize(m->st);
    for (auto* vv : {&m->W, &m->b, &m->Wm, &m->Wv, &m->bm, &m->bv, &m->dW, &m->db, &m->z})
        for (float* p : *vv)
            if (p) cudaFree(p);
    for (auto* vv : {&m->Wb, &m->h, &m->gb})
        for (bf16* p : *vv)
            if (p) cudaFree(p);
    for (void* p : {(void*)m->in_mu, (void*)m->in_sd, (void*)m->out_mu, (void*)m->out_sd})
        if (p) cudaFree(p);
    for (void* p : {(void*)m->t, (void*)m->loss, (void*)m->loss_part, (void*)m->xin,
                    (void*)m->work})
        if (p) cudaFree(p);
    if (m->back) cudaFreeHost(m->back);
    delete m;
}

}  // extern "C"
