// rad_internal.cuh -- structures and sm_103a device helpers shared by the
// kernels of the radiation-spectrum library (not part of the public ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

struct rad_ctx;   // the radiation context (rad_api.cu)

namespace rad {

// ---------------------------------------------------------------------------
// trajectory ring layout
// ---------------------------------------------------------------------------
// Both rings are tile-major: particle column col is particle p = col % 8 of tile
// col / 8.  Within each chunk of 32 slots the samples are innermost: element
// (tile, slot, c, p) sits at ((chunk * 8 + p) * comps + c) * 32 + slot % 32 with
// chunk = (tile * ring + slot) / 32, so that a warp reads one particle's chunk
// (contiguous, 1280 B in FP32) with lane = sample; the chunk of all eight particles is
// one contiguous block too.
// A chunk of the FP32 ring that single calls are filling is slot-major instead,
// [slot % 32][c][p], until a window closes: one call's values of a tile then are whole
// 32-byte sectors.  particle_major() turns it, in place, before the accumulation.
// comps is 10, or 11 when sample selectors are defined (the flags word); the
// precise-phase FP32 path adds dr's lo part as components 11-13 (comps 14).
// FP32 split path: slab[tile][chunk][p][c][slot % 32] float, c = 0..9 (10) =
//   dr (3)   : r_m - r_a, the offset from the block's FP64 anchor position
//   beta (3) : beta_m
//   bdot (3) : betadot_m (differenced in FP64 before the rounding)
//   g (1)    : 1/gamma_m^2 = 1/(1 + ubar^2)
//   flags (1): selector bits of the sample (bit i: inside selector i), stored as
//              the float with those bits (FP32 ring) or as an exact double (FP64)
// anc32[tile][blk][p][c] float, c = 0..5: r_a as hi (3) + lo (3) FP32 pairs at
//   the anchor samples a = K * blk (ring of ring/K blocks, tile-major like the
//   samples, so a chunk's anchors are one contiguous block too).
// FP64 path: slab64[tile][chunk][p][c][slot % 32] double with c = r (3, absolute unwrapped),
// beta (3), bdot (3), g (1), flags (1).
constexpr int kComps = 11;     // components at most (10 + the selector flags)
constexpr int kCompsPlain = 10;   // without selectors
constexpr int kCompsPrec = 14;    // precise-phase FP32 ring: + flags + the lo part of dr
constexpr int kTileP = 8;      // particles per tile: one warp each
constexpr int kChunk32 = 32;   // samples per chunk
constexpr int kComputeWarps = 8;
constexpr int kBlockThreads = (kComputeWarps + 1) * 32;  // + one TMA producer warp
constexpr int kMaxSpecies = 32;
constexpr int kFreqPad = 256;  // each grid's frequencies are padded with zeros to whole tiles

// error word bits
constexpr int kErrTimeout = 1;
constexpr int kErrNaN = 2;

// One unit of accumulation work: a window, a direction, a tile of the
// frequency grid and a run of particle tiles of one species.
struct WorkItem {
    int32_t win;      // window index
    int32_t dir;      // direction index (into the context's directions)
    int32_t ftile;    // frequency tile index within the window's grid
    int32_t sp;       // species index
    int32_t tile0;    // first particle tile (column / 8)
    int32_t ntiles;   // number of particle tiles
    int32_t row;      // output row of the direction in the window's [dirs][len] block
    int32_t kmul;     // FP32 path: phases anchored every K << kmul samples (K: the ring's)
    int32_t prec;     // FP32 path, precise-phase build for chosen items: 1 = this item
};

// Per-window constants the accumulation kernels read.
struct WinDev {
    int64_t s0, s1;      // sample range
    int32_t grid_off;    // offset of the frequency grid in the (padded) frequency arrays
    int32_t grid_len;    // frequencies in the grid
    int64_t out_off;     // offset of the window's [dirs][len] block in the accumulators
    int32_t sel;         // selector bit the samples must have, or -1 (all samples)
    int32_t pad_;
};

// A sample selector evaluated at ingest (positions as handed over, ubar).
constexpr int kMaxSelectors = 32;
struct SelectorDev {
    int32_t kind;        // 1: box, 2: cone
    int32_t pad_;
    double lo[3], hi[3]; // box: lo <= x < hi per component
    double axis[3];      // cone: unit axis
    double cos_lo, cos_hi;  // cone: cos(angle(ubar, axis)) in [cos_lo, cos_hi]
};

struct SpeciesDev {
    double qdt;          // q * dt
    int32_t col0;        // first column of the species in the ring
    int32_t count;       // particles
};

// ---------------------------------------------------------------------------
// float-float (double-single) helpers: error-free transformations of FP32
// arithmetic (Dekker/Knuth), used where FP64 accuracy is needed without the
// FP64 pipe
// ---------------------------------------------------------------------------
struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff two_prod(float a, float b)
{
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}

__device__ __forceinline__ ff two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z))};
}

// ---------------------------------------------------------------------------
// mbarrier / TMA helpers (inline PTX, sm_90+ forms valid on sm_103a)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_addr(bar)),
        "r"(bytes)
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: spins with a growing back-off for at most 2^18 polls.  A
// poll that fails costs about 4 us on GB300 (the try_wait's own suspension
// plus the back-off; 2^22 polls measured 17 s), so a wait expires after
// about a second, while every wait of a working kernel ends within
// microseconds.  On expiry it raises the block's abort flag and the device
// error word, and returns false; callers then carry on without waiting
// (results are flagged invalid) so that no thread is left behind at a barrier.
constexpr uint32_t kMaxPolls = 1u << 18;

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  volatile int* s_abort, int* err_word)
{
    if (mbar_try_wait(bar, parity)) return true;
    for (uint32_t it = 0; it < kMaxPolls; ++it) {
        if (*s_abort) return false;
        if (mbar_try_wait(bar, parity)) return true;
        __nanosleep(it < 64 ? 32 : 256);
    }
    *s_abort = 1;
    atomicOr(err_word, kErrTimeout);
    return false;
}

// Orders this thread's earlier generic-proxy accesses to shared memory before
// later async-proxy (bulk copy) writes to it.
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Bounded wait for a block's own copies still in flight before it exits: it
// polls at most kMaxPolls times and never raises flags.
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity)
{
    for (uint32_t it = 0; it < kMaxPolls; ++it) {
        if (mbar_try_wait(bar, parity)) return;
        __nanosleep(256);
    }
}

// 1-D bulk copy (TMA) of `bytes` contiguous bytes into shared memory,
// completion on `bar`.  Both addresses 16-byte aligned, bytes % 16 == 0.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_addr(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes),
        "r"(smem_addr(bar))
        : "memory");
}


// ---------------------------------------------------------------------------
// kernel parameter blocks and launchers
// ---------------------------------------------------------------------------
struct IngestParams {
    const double* x;        // [n_steps][3][n_in]
    const double* u;        // [n_steps][3][n_in]
    int64_t n_in;           // particles on the input axis
    int32_t n_steps;
    int64_t step0;          // absolute step of the first state in x/u
    double dt, idt;         // idt = 1 / dt
    double box_L;           // 0: no unwrapping
    float lim;              // crossing_limit(box_L)
    double* x_prev;         // [3][ncols] raw x of the previous call
    double* r_prev;         // [3][ncols] image count n of the previous call (r = x + L n)
    double* u_prev;         // [3][ncols] u of the previous call
    float* slab32;          // FP32 ring or nullptr
    double* slab64;         // FP64 ring or nullptr
    float* anc32;           // FP32 path: tile-major anchor ring (r_a as hi + lo)
    int64_t ncols;
    int64_t ring;           // samples in the ring
    // samples [keep0, keep1) -- whole chunks -- go into the ring, others only carry the
    // particle state on: the ring is as long as the windows' span, so two chunks outside
    // it may share a slot, and blocks of one launch would write it in no order
    int64_t keep0, keep1;
    // FP32 ring: whether the chunk of the launch's first sample, and those after it, are
    // slot-major (the first one's layout may be an earlier launch's choice)
    int32_t slot_major0, slot_major;
    int32_t turned;         // all chunks are to be particle-major
    int32_t comps;          // ring components per sample (10, or 11 with selector flags)
    int32_t K;              // anchor interval (FP32 path)
    int64_t nblk;           // anchor blocks in the ring
    int32_t n_species;
    int64_t in_off[kMaxSpecies + 1];
    int32_t col_off[kMaxSpecies];
    int32_t check;          // flag non-finite inputs
    int* err_word;
    const SelectorDev* sel; // selectors (device) or nullptr
    int32_t n_sel;
    int32_t nsub;           // sub-samples per PIC sample (<= 1: none)
    // particle range of this launch and layout of x/u (zero: all particles,
    // x/u holding every particle): particles first .. first + count - 1 are
    // processed; particle i is column i - xoff of x/u, whose particle axis
    // has stride ld
    int64_t first;
    int64_t count;
    int64_t ld;
    int64_t xoff;
    // time segments (one thread per particle and segment): segment 0 starts at
    // step0, segment g >= 1 at seg_first + (g - 1) seg_len (calls 1 + j seg_len:
    // anchor-aligned samples); wind [n_seg - 1][3][count] receives each
    // segment's change of the image count.  n_seg <= 1: one thread per particle.
    int64_t seg_first;
    int32_t seg_len;        // calls (batched launches: 32-sample chunks) per segment
    int32_t n_seg;
    int64_t tile0;          // batched launches: first tile and number of tiles
    int32_t n_tiles;
    int32_t* wind;
    double* state_out;      // [9][count]: the last segment's carry-over state,
                            // stored to x_prev/r_prev/u_prev after the launch
};

struct Accum32Params {
    const WorkItem* items;
    int32_t n_items;
    int* counter;             // dynamic item counter (zeroed before the launch)
    int32_t few;              // block-moment kernel: unit_grid's few
    const WinDev* wins;
    const SpeciesDev* species;
    const float* dirs32;      // [D][12]: n, e1, e2, n - (float)n
    const float* omega;       // [n_freq] rad per unit time
    const float* nu_hi;       // [n_freq] (omega / 2 pi) hi part
    const float* nu_lo;       // [n_freq] lo part
    const float* slab32;      // tile-major FP32 ring
    const float* anc32;       // tile-major anchor ring
    int64_t ring;
    int64_t nblk;
    int32_t comps;            // ring components per sample (10, or 11 with selector flags)
    float dt_hi, dt_lo;       // dt as a float-float pair
    double* acc;              // incoherent [n_out]; coherent [n_out][4]
    int* err_word;
    // failure-detection test hook (0: off): block 0's producer first waits on
    // a barrier nothing arrives on, so that its bounded wait expires
    int32_t fault_stall;
};

struct Accum64Params {
    const WorkItem* items;
    int32_t n_items;
    const WinDev* wins;
    const SpeciesDev* species;
    int* counter;             // dynamic unit counter (zeroed before the launch)
    int32_t few;              // unit_grid's few
    const double* dirs64;     // [D][9]: n, e1, e2
    const double* omega;      // [n_freq]
    const double* nu_hi;      // [n_freq] omega / 2 pi, hi and lo part
    const double* nu_lo;
    const double2* cis;       // [accum64_table()] cos, sin of 2 pi j / table
    const double* slab64;     // tile-major FP64 ring
    int64_t ring;
    int32_t comps;            // ring components per sample (10, or 11 with selector flags)
    double dt;
    double* acc;
    int* err_word;
    int32_t fault_stall;      // as in Accum32Params
};

// launch_ingest splits a launch in time below these sizes: 8-particle tiles (batches of
// calls), particles (sub-cycled samples).
constexpr int kSegMaxTiles = 608;
constexpr int64_t kSegMaxParticles = 32768;
cudaError_t launch_ingest(const IngestParams& p, cudaStream_t st);
float crossing_limit(double L);
// Whether launch_ingest takes the batch kernel (which fills whole chunks).
bool ingest_batched(const IngestParams& p);
// Chunks [c0, c1] of every tile from slot-major to particle-major, in place.
cudaError_t particle_major(float* slab, int64_t ncols, int64_t ring, int comps, int64_t c0, int64_t c1,
                           cudaStream_t st);
// The FP32 builds of the per-call ingest kernel (common and precise-phase ring, without and
// with sub-cycling); a kernel function pointer compares equal to the set when it is one.
struct IngestKernels {
    const void* build[4];
};
inline bool operator==(const void* f, const IngestKernels& k)
{
    return f == k.build[0] || f == k.build[1] || f == k.build[2] || f == k.build[3];
}
IngestKernels ingest_kernel_ptr();

// Stream a radiation context orders its work on (for in-library callers that
// hand it device buffers from another stream).
cudaStream_t ctx_stream(const rad_ctx* c);
// Particles a radiation context takes per call, and the step it expects next.
int64_t ctx_particles(const rad_ctx* c);
int64_t ctx_next_step(const rad_ctx* c);
// rad_accumulate of one step from device arrays whose components are ld particles apart
// (component c of particle i at x[c ld + i]), in the context's stream order.
int ctx_accumulate_strided(rad_ctx* c, int64_t step, const double* x, const double* u, int64_t ld);
// FP32 kernel variant: frequencies per thread, of which np by the FMA-pipe
// polynomial, anchor interval K, coherent sum, minimum resident blocks per SM.
struct Accum32Config {
    int ft, np, K;
    bool coh;
    int mb;
    bool band = false;   // items with anchor blocks of K << kmul (8 SFU frequencies per thread)
    int pm = 0;          // precise offset phase (8 SFU frequencies, K 32): 0 none, 1 every
                         // item, 2 the items whose WorkItem.prec is set
    bool mom = false;    // block-moment kernel (the automatic choice): 8 frequencies per
                         // thread, K 32
};
constexpr int kMomentBlocks = 4;   // its resident blocks per SM
bool accum32_moment(const Accum32Params* p, const Accum32Config& cfg, int grid,
                    cudaStream_t st, cudaError_t* err, int* nb);
bool accum32_ft8_sfu(const Accum32Params* p, const Accum32Config& cfg, int grid,
                     cudaStream_t st, cudaError_t* err, int* nb);
bool accum32_band(const Accum32Params* p, const Accum32Config& cfg, int grid,
                  cudaStream_t st, cudaError_t* err, int* nb);
bool accum32_precise(const Accum32Params* p, const Accum32Config& cfg, int grid,
                     cudaStream_t st, cudaError_t* err, int* nb);
bool accum32_ft8_mix(const Accum32Params* p, const Accum32Config& cfg, int grid,
                     cudaStream_t st, cudaError_t* err, int* nb);
bool accum32_ft16(const Accum32Params* p, const Accum32Config& cfg, int grid,
                  cudaStream_t st, cudaError_t* err, int* nb);
bool accum32_ft4(const Accum32Params* p, const Accum32Config& cfg, int grid,
                 cudaStream_t st, cudaError_t* err, int* nb);
// launch (p != nullptr) or occupancy query; false if the variant is not built
bool accum32_dispatch(const Accum32Params* p, const Accum32Config& cfg, int grid,
                      cudaStream_t st, cudaError_t* err, int* nb);
// FP64 kernel with ft frequency slots per lane (2, 4 or 8)
cudaError_t launch_accum64(const Accum64Params& p, int ft, bool coh, int grid, cudaStream_t st);
int accum64_blocks_per_sm(int ft, bool coh);
// Grid of the kernels whose warps take units (an item's particles) on their own: the full
// grid, so that all SMs get the same number of blocks.  few: under four units per warp,
// each unit is taken only when a warp is free for it.
inline int unit_grid(int64_t n_items, int total_blocks, int32_t* few)
{
    *few = n_items * kTileP < (int64_t)4 * 4 * total_blocks;
    return total_blocks;
}
int accum64_ft(int64_t particle_dirs, int n_omega, int sms);
int accum64_table();

}  // namespace rad
