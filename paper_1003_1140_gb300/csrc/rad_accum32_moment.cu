// rad_accum32_moment.cu -- FP32 split-phase accumulation with block moments: the
// automatic kernel choice.
//
// Same sum, phase split and ring as rad_accum32.cuh.  Within one 32-sample
// chunk the phase of sample m at frequency w is Theta + w dphi_m, so the
// chunk's contribution to an amplitude is
//   e^{i Theta} sum_m V_m e^{i w dphi_m} = e^{i Theta} sum_p c_p (i w h)^p M_p,
//   M_p = sum_m V_m (dphi_m / h)^p,   |dphi_m| <= h,
// with c_p the coefficients of polynomials for cos and sin on |w h| <= X0.
// The M_p (real, two components of V) do not depend on the frequency: one warp
// forms them once per chunk, lane = sample, and every frequency then costs P = 12
// multiply-adds per component and one rotation per chunk instead of 32 sines,
// cosines and 128 multiply-adds.  Larger w h are halved by splitting the chunk
// into two or four sub-blocks about their own centres; beyond that (or for
// non-finite offsets) the samples are summed directly, as in rad_accum32.cuh.
//
// The choice is made per warp (one particle), chunk and pair of 32-frequency
// slots from the largest |w| of the pair and the chunk's actual largest |dphi|,
// so it adapts to the direction: towards a beam 1 - n.beta is small and high
// frequencies take the moments too.
//
// Layout: every warp works on its own -- one particle of a work item at a time,
// taken from the list with an atomic counter -- so warps on cheap particles never
// wait for warps on dear ones and no barrier is left in the loop; direct sums (bound
// by the special-function unit) and moments (bound by instruction issue) of different
// warps overlap on an SM.  A chunk (32 samples x components of one particle, 1.3 KB
// contiguous in the ring) comes by bulk copies (TMA) two chunks ahead; lane = sample for the
// geometry and the moments, lane = chunk for the reference phases of the next 32
// chunks, lane = frequency for the rest, 8 frequency slots per lane kept as four
// pairs in packed f32x2 registers (two slots per instruction).  Frequency slots
// beyond the grid's end and particles beyond a species' count are skipped.  Particle
// sums run in float-float per warp and reach the FP64 accumulators once per work unit.
//
// Against the direct kernel (which the explicit variants still run): 8195 particles x 4096
// samples x 8 directions x 1024 omega, ingest included, 125.0 -> 77.4 ms; 1024 x 2000 x 192 x
// 2048 356 -> 221 ms; 1024 x 2000 x 12 x 64 3.49 -> 1.35 ms.  Issue slots 58% busy, the
// special-function pipe 65-69%, FMA 45%: dependent chains of four warps per scheduler, and the
// instruction cache, are what is left.  Tried and slower: eight sub-blocks of four samples for
// larger w h (dense map 225 -> 241 ms, shard 79.5 -> 87.1: 60 issue slots per sub-block against
// 68 for its direct sums, and more code); moments for the lower slot of the first direct pair (dense
// map 225 -> 267 ms); sines of one pair in four by polynomial (direct work 7.70 -> 7.25 ms, but
// mixed work 2.6% slower).
#include "rad_accum32.cuh"

namespace rad {
namespace {

typedef unsigned long long f2;   // a packed pair of FP32 values

__device__ __forceinline__ f2 pk(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f2 dup(float a) { return pk(a, a); }
__device__ __forceinline__ void upk(f2 v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// anchor_turns (rad_accum32.cuh) for two frequencies at once.
__device__ __forceinline__ f2 anchor_turns2(f2 nh, f2 nl, float2 an)
{
    const f2 ah = dup(an.x), mg = dup(kMagic), nmg = dup(-kMagic), m1 = dup(-1.0f);
    const f2 pr = mul2(nh, ah);
    const f2 pe = fma2(nh, ah, mul2(nh, dup(-an.x)));
    const f2 tl = fma2(nl, ah, fma2(nh, dup(an.y), pe));
    // pr - rint(pr) as a fused multiply-add by -1: in an addition of pr the packed
    // product and sum were re-formed as one fused operation, which counts pr's rounding
    // error (already in pe) twice
    f2 fr = fma2(add2(add2(pr, mg), nmg), m1, pr);
    fr = fma2(add2(add2(fr, mg), nmg), m1, fr);
    return add2(fr, tl);
}

constexpr int kFT = 8, kPairs = kFT / 2;
// 16 warps per SM at 128 registers.  Measured (2048 particles of the precision workload,
// 256 omega, kernel time; [0.1, 1] / [1, 10] / direct [300, 1000]): 2.69 / 5.18 / 7.70 ms;
// 20 warps at 96 registers 3.56 / 6.58 / 7.88 (register pairs no longer line up: a third
// more moves), 12 warps at 168 registers 3.01 / 5.72 / 8.03, 8-warp blocks 2.72 / 5.13 /
// 7.62 (slower as soon as units of different cost share a block).
constexpr int kWarps = 4, kBlocks = kMomentBlocks, kThreads = kWarps * 32;
constexpr int kMaxP = 12;    // moments per sub-block

// Polynomials cos t = sum_j C_j (-t^2)^j, sin t = t sum_j S_j (-t^2)^j, leading
// coefficients exactly 1, the rest minimax fits with successively rounded
// coefficients (fit_sincos.py, fit_moment): 12 terms to 6.1e-8 on |t| <= 2.5 -- an eighth
// of the special-function unit's own error, so the moments never lose accuracy against
// the direct sum.  (A second, 8-term form for |t| <= 0.85 was dropped: with its copies of
// the code gone, and those of direct ranges that end before the last pair, the kernel
// misses the instruction cache less -- coherent batch 9.06 -> 8.30 ms, precision shard
// 78.8 -> 77.7.)
constexpr float kX12 = 2.5f;
__device__ const float g_moment_coef[kMaxP] = {
    1.0f, 1.0f, 4.999995530e-01f, 1.666666120e-01f, 4.166565090e-02f, 8.333227597e-03f,
    1.388137927e-03f, 1.983425464e-04f, 2.455824688e-05f, 2.734730060e-06f, 2.393897489e-07f,
    2.211615246e-08f};

// The walk over (work unit, particle, chunk), advanced by lane 0 only; a unit is
// particle pp of every tile of an item.
struct MomCursor {
    const float* src;        // the particle's chunks in the ring
    int32_t ii, pp, t, nt;   // item (< 0: none left), particle of the tile, tile, tiles
    int32_t c, c0, c1;       // chunk, the window's first and last
    int32_t sc, sc0;         // their ring chunks
    int32_t lo, hi;          // first and last chunk's sample range ends
    int32_t ticket;          // the unit after that one, asked for early
};

// What lane 0 tells its warp about a chunk.
struct MomMeta {
    int32_t ii, pp, chunk, sc;   // item (< 0: no more work), particle, chunk, ring chunk
    int32_t lo, hi, flags;       // as ChunkMeta
    int32_t t;                   // tile of the item
};

template <bool COH>
struct __align__(128) WarpM {
    float raw[2][kComps * kChunk32];     // bulk-copy destinations: [component][sample]
    float4 geo[kChunk32 + 1];            // V1, V2, dphi per sample (direct sum)
    float4 mom[4][kMaxP];                // (M1, M1, M2, M2) per sub-block
    float2 ff[(COH ? 4 : 1) * kFT][32];  // particle sums (hi, lo)
    float dv[16];                        // n, e1, e2, n's lo part, q dt
    MomMeta meta[4];
    MomCursor cur;
    uint64_t full[2];
};

template <bool COH>
struct SmemM {
    WarpM<COH> w[kWarps];
    float coef[kMaxP];
    int abort_flag;
};

// 1 / x to about one ulp (x in the normal range): the special-function unit's
// reciprocal and one Newton step, without the divide's range checks.
__device__ __forceinline__ float rcp_nr(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}

// One level of the transposing reduction: n values per lane become n / 2, the
// lower lanes (bit o clear) keeping the first half, the upper the second.
template <int N>
__device__ __forceinline__ void fold(float (&v)[2 * kMaxP], int o, bool up)
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float a = v[i], b = v[i + N / 2];
        const float send = up ? a : b, keep = up ? b : a;
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
}

// Moments of sub-blocks of 2 o0 lanes (samples) each, o0 = 16, 8 or 4: P powers of
// tau times V1 and V2 per lane, summed over the sub-block by a transposing reduction
// (three halvings of the 2 P values, then plain sums over the lanes that are left),
// times the polynomial coefficient, as (M, M) pairs in out.  o0 is a run-time value
// to keep the kernel's code small: with a copy per block size and pair of slots the
// instruction cache was what bound mixed work.
template <int P>
__device__ __forceinline__ void moments(float V1, float V2, float tau, int o0, int lane,
                                        float4 (*out)[kMaxP], const float* coef)
{
    float v[2 * kMaxP];
    f2 w = pk(V1, V2);
    const f2 t2 = dup(tau);
    upk(w, v[0], v[1]);
#pragma unroll
    for (int p = 1; p < P; ++p) {
        w = mul2(w, t2);
        upk(w, v[2 * p], v[2 * p + 1]);
    }
    const int o1 = o0 >> 1, o2 = o0 >> 2;
    fold<2 * P>(v, o0, lane & o0);
    fold<P>(v, o1, lane & o1);
    fold<P / 2>(v, o2, lane & o2);
    constexpr int R = P / 4;             // values left per lane
#pragma unroll 1
    for (int o = o2 >> 1; o > 0; o >>= 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] += __shfl_xor_sync(0xffffffffu, v[r], o);
    }
    const int q0 = ((lane & o0) ? P : 0) + ((lane & o1) ? P / 2 : 0) + ((lane & o2) ? P / 4 : 0);
    __syncwarp();
    if ((lane & (o2 - 1)) == 0) {
        float2* dst = reinterpret_cast<float2*>(out[lane / (2 * o0)]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int q = q0 + r;                    // moment q / 2, component q & 1
            const float x = v[r] * coef[q >> 1];
            dst[q] = make_float2(x, x);
        }
    }
    __syncwarp();
}

// Adds one sub-block's moments to a pair of slots: theta the rotation (radians),
// x = w hs the scaled frequencies.
template <int P>
__device__ __forceinline__ void eval_moments(const float4* M, f2 x, f2 nx, f2 theta, f2& a1r, f2& a1i,
                                             f2& a2r, f2& a2i)
{
    const f2 z = mul2(x, nx);            // -x^2
    f2 E1, E2, O1, O2;
    {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(M + P - 2);
        const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(M + P - 1);
        E1 = e.x;
        E2 = e.y;
        O1 = o.x;
        O2 = o.y;
    }
#pragma unroll
    for (int j = P / 2 - 2; j >= 0; --j) {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(M + 2 * j);
        const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(M + 2 * j + 1);
        E1 = fma2(E1, z, e.x);
        E2 = fma2(E2, z, e.y);
        O1 = fma2(O1, z, o.x);
        O2 = fma2(O2, z, o.y);
    }
    O1 = mul2(O1, x);
    O2 = mul2(O2, x);
    float t0, t1, s0, s1, c0, c1;
    upk(theta, t0, t1);
    __sincosf(t0, &s0, &c0);
    __sincosf(t1, &s1, &c1);
    const f2 c = pk(c0, c1), s = pk(s0, s1), ns = pk(-s0, -s1);
    a1r = fma2(E1, c, a1r);
    a1i = fma2(E1, s, a1i);
    a2r = fma2(E2, c, a2r);
    a2i = fma2(E2, s, a2i);
    a1r = fma2(O1, ns, a1r);
    a1i = fma2(O1, c, a1i);
    a2r = fma2(O2, ns, a2r);
    a2i = fma2(O2, c, a2i);
}

// Direct sum of samples [lo, hi) for the slot pairs A .. B - 1.  With one or two pairs a
// sample's chain (load, phase, sine, sums) is not hidden by the other pairs': several samples
// at once (UNROLL) take the 64-frequency subset of 1024 particles from 1.51 to 1.38 ms; the
// coherent kernel, short of registers, gets slower by it (9.05 to 9.5 ms) and does without.
template <int A, int B, bool UNROLL>
__device__ __forceinline__ void direct_sum(const float4* geo, int lo, int hi, const f2 (&om)[kPairs],
                                           const f2 (&th)[kPairs], f2 (&a1r)[kPairs],
                                           f2 (&a1i)[kPairs], f2 (&a2r)[kPairs], f2 (&a2i)[kPairs])
{
    constexpr int U = !UNROLL || B - A > 2 ? 1 : 4 / (B - A);
    float4 g = geo[lo];
#pragma unroll U
    for (int l = lo; l < hi; ++l) {
        const float4 gn = geo[l + 1];    // [32] is padding
        const f2 v1 = dup(g.x), v2 = dup(g.y), dp = dup(g.z);
#pragma unroll
        for (int i = A; i < B; ++i) {
            float t0, t1, s0, s1, c0, c1;
            upk(fma2(om[i], dp, th[i]), t0, t1);
            __sincosf(t0, &s0, &c0);
            __sincosf(t1, &s1, &c1);
            const f2 c = pk(c0, c1), s = pk(s0, s1);
            a1r[i] = fma2(v1, c, a1r[i]);
            a1i[i] = fma2(v1, s, a1i[i]);
            a2r[i] = fma2(v2, c, a2r[i]);
            a2i[i] = fma2(v2, s, a2i[i]);
        }
        g = gn;
    }
}

template <bool COH>
__global__ void __launch_bounds__(kThreads, kBlocks) accum32_moment_kernel(const Accum32Params p)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto& SB = *reinterpret_cast<SmemM<COH>*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto& S = SB.w[warp];
    const int pstride = p.comps * kChunk32;              // one particle's chunk, floats
    const int rchunks = (int)(p.ring / kChunk32);        // chunks (and anchors) in the ring
    volatile int* abort_flag = &SB.abort_flag;

    if (lane == 0) {
        mbar_init(&S.full[0], 1);
        mbar_init(&S.full[1], 1);
        fence_mbar_init();
        S.geo[kChunk32] = make_float4(0, 0, 0, 0);
    }
    for (int v = lane; v < (int)(sizeof(S.ff) / 4); v += 32)
        reinterpret_cast<uint32_t*>(S.ff)[v] = 0u;
    if (tid == 0) SB.abort_flag = 0;
    if (tid < kMaxP) SB.coef[tid] = g_moment_coef[tid];
    __syncthreads();

    // ---- (lane 0) describe the cursor's chunk as chunk L, issue its copy and step on;
    // L < 0 only asks for the first unit.  False once there is no more work.
    auto issue = [&](int L) -> bool {
        MomCursor& C = S.cur;
        bool next_unit = L < 0;
        if (L >= 0) {
            const int buf = L & 1;
            MomMeta& M = S.meta[L & 3];
            M.ii = C.ii;
            if (C.ii < 0) {
                mbar_arrive(&S.full[buf]);
                return false;
            }
            const int c = C.c;
            const bool first = c == C.c0, last = c == C.c1;
            M.pp = C.pp;
            M.chunk = c;
            M.sc = C.sc;
            M.t = C.t;
            M.lo = first ? C.lo : 0;
            M.hi = last ? C.hi : kChunk32;
            M.flags = (first ? kFirstOfTile : 0) | (last ? kLastOfTile : 0) |
                      (first && C.t == 0 ? kFirstOfItem : 0) |
                      (last && C.t + 1 == C.nt ? kLastOfItem : 0);
            const uint32_t bytes = (uint32_t)(pstride * sizeof(float));
            fence_proxy_async();
            mbar_arrive_expect_tx(&S.full[buf], bytes);
            bulk_load(S.raw[buf], C.src + (int64_t)C.sc * (kTileP * pstride), bytes, &S.full[buf]);
            if (!last) {
                C.c = c + 1;
                C.sc = C.sc + 1 == rchunks ? 0 : C.sc + 1;
            } else if (++C.t < C.nt) {
                C.c = C.c0;
                C.sc = C.sc0;
                C.src += (int64_t)rchunks * kTileP * pstride;
            } else {
                next_unit = true;
            }
        }
        while (next_unit) {
            // (with few units none is asked for early: it would wait while other warps idle)
            const int v = L < 0 || p.few ? atomicAdd(p.counter, 1) : C.ticket;
            C.ii = -1;
            const int ii = v / kTileP;
            if (ii >= p.n_items) break;
            if (!p.few) C.ticket = atomicAdd(p.counter, 1);
            const WorkItem it = p.items[ii];
            const SpeciesDev sp = p.species[it.sp];
            C.pp = v % kTileP;
            // tiles of the item in which this particle exists
            const int left = sp.count - it.tile0 * kTileP - C.pp;
            L = 0;
            if (left <= 0) continue;
            C.ii = ii;
            C.nt = min(it.ntiles, (left - 1) / kTileP + 1);
            const int64_t s0 = p.wins[it.win].s0, s1 = p.wins[it.win].s1 - 1;
            C.src = p.slab32 +
                    ((int64_t)(sp.col0 / kTileP + it.tile0) * rchunks * kTileP + C.pp) * pstride;
            C.c0 = (int)(s0 / kChunk32);
            C.c1 = (int)(s1 / kChunk32);
            C.lo = (int)(s0 % kChunk32);
            C.hi = (int)(s1 % kChunk32) + 1;
            C.sc0 = (int)((uint32_t)C.c0 % (uint32_t)rchunks);
            C.t = 0;
            C.c = C.c0;
            C.sc = C.sc0;
            next_unit = false;
        }
        return true;
    };
    if (tid == 0 && p.fault_stall && blockIdx.x == 0) {
        // test hook: nothing has been issued, so nothing arrives and the wait expires
        mbar_wait_bounded(&S.full[0], 0, abort_flag, p.err_word);
    }
    bool feeding = lane == 0;    // lane 0: there may be more chunks to issue
    uint32_t issued = 0;         // chunks issued (lane 0)

    f2 a1r[kPairs], a1i[kPairs], a2r[kPairs], a2i[kPairs];
    float wm[kPairs];            // largest |omega| of the pair (warp-uniform); < 0: no slot in use
    const float* om0 = nullptr;  // this lane's frequency in slot 0 (read from `skip` on)
    const float *nh0 = nullptr, *nl0 = nullptr;
    int skip = 0, sel = -1;
    int kc = 0;                  // chunk of the particle
    float bh = 0.0f, bl = 0.0f;  // lane = chunk: reference phases but for the centre
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
        a1r[i] = a1i[i] = a2r[i] = a2i[i] = 0;
        wm[i] = -1.0f;
    }
    // L = -3 .. -1: the first unit and its first two copies (one code path for all)
#pragma unroll 1
    for (int L = -3;; ++L) {
        if (L < 0) {
            if (feeding) {
                feeding = issue(L + 2) && !*abort_flag;
                if (feeding && L > -3) ++issued;
            }
            __syncwarp();
            continue;
        }
        const int buf = L & 1;
        const bool ready = mbar_wait_bounded(&S.full[buf], (L >> 1) & 1, abort_flag, p.err_word);
        const MomMeta& M = S.meta[L & 3];
        const int ii = M.ii;
        // warp-collective from here: the whole warp goes on or stops
        if (!__all_sync(0xffffffffu, ready && ii >= 0 && !*abort_flag)) break;
        const int chunk = M.chunk, lo = M.lo, hi = M.hi, flags = M.flags;
        const bool first = flags & kFirstOfTile, last = flags & kLastOfTile;
        if (flags & kFirstOfItem) {
            const WorkItem it = p.items[ii];
            const WinDev w = p.wins[it.win];
            __syncwarp();
            if (lane < 12) S.dv[lane] = p.dirs32[12 * it.dir + lane];
            if (lane == 12) S.dv[12] = (float)p.species[it.sp].qdt;
            const int kb = it.ftile * (32 * kFT);
            sel = w.sel;
            // a grid's last tile fills the pairs from the end: the high frequencies then
            // always reach the last pair, whatever the grid's length
            skip = max(0, 32 * kFT - (w.grid_len - kb + 63) / 64 * 64);
            om0 = p.omega + w.grid_off + kb + lane - skip;
            nh0 = p.nu_hi + w.grid_off + kb + lane - skip;
            nl0 = p.nu_lo + w.grid_off + kb + lane - skip;
#pragma unroll
            for (int i = 0; i < kPairs; ++i) {
                wm[i] = -1.0f;
                if (64 * i < skip) continue;
                const float w0 = om0[64 * i], w1 = om0[64 * i + 32];
                wm[i] = __uint_as_float(__reduce_max_sync(
                    0xffffffffu, __float_as_uint(fmaxf(fabsf(w0), fabsf(w1)))));
            }
            __syncwarp();
        }
        if (first) {
#pragma unroll
            for (int i = 0; i < kPairs; ++i) a1r[i] = a1i[i] = a2r[i] = a2i[i] = 0;
        }
        const float4 q0 = *reinterpret_cast<const float4*>(S.dv);
        const float4 q1 = *reinterpret_cast<const float4*>(S.dv + 4);
        const float4 q2 = *reinterpret_cast<const float4*>(S.dv + 8);
        const float nh[3] = {q0.x, q0.y, q0.z}, nlo[3] = {q2.y, q2.z, q2.w};
        if (first) kc = 0;
        if ((kc & 31) == 0) {
            // reference phases of the next 32 chunks, lane = chunk: A dt - n . r_A at each
            // chunk's anchor in float-float (the chunk's centre is added below)
            const WorkItem it = p.items[ii];
            const int64_t tile = p.species[it.sp].col0 / kTileP + it.tile0 + M.t;
            const int cl = chunk + lane <= (int)((p.wins[it.win].s1 - 1) / kChunk32) ? lane : 0;
            int sl = M.sc + cl;
            if (sl >= rchunks) sl %= rchunks;
            const float2* ra = reinterpret_cast<const float2*>(
                p.anc32 + ((tile * rchunks + sl) * kTileP + M.pp) * 6);
            const float2 r0 = ra[0], r1 = ra[1], r2 = ra[2];
            const float rh[3] = {r0.x, r0.y, r1.x}, rl[3] = {r1.y, r2.x, r2.y};
            const float ta = (float)((int64_t)(chunk + cl) * kChunk32);
            const ff t = two_prod(ta, p.dt_hi);
            float sh = t.hi, e = fmaf(ta, p.dt_lo, t.lo);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const ff dd = two_prod(nh[q], rh[q]);
                const float dl = fmaf(nh[q], rl[q], fmaf(nlo[q], rh[q], dd.lo));
                const ff u = two_sum(sh, -dd.hi);
                sh = u.hi;
                e = e + (u.lo - dl);
            }
            bh = __fadd_rn(sh, e);
            bl = __fsub_rn(e, __fsub_rn(bh, sh));
        }

        // ---- geometry, lane = sample (see rad_accum32.cuh)
        float V1, V2, d;
        float2 an;
        {
            const float* tb = S.raw[buf] + lane;
            const float n0 = nh[0], n1 = nh[1], n2 = nh[2];
            const float dr[3] = {tb[0], tb[kChunk32], tb[2 * kChunk32]};
            const float ti = (float)lane;
            // centre of the block's offsets: the mean of its first and last in-window
            // offsets
            float h = 0.5f * (float)(kChunk32 - 1) * p.dt_hi;
            {
                const float o = ti * p.dt_hi - (n0 * dr[0] + n1 * dr[1] + n2 * dr[2]);
                const float hh = 0.5f * (__shfl_sync(0xffffffffu, o, lo) +
                                         __shfl_sync(0xffffffffu, o, hi - 1));
                if (fabsf(hh) <= (float)kChunk32 * p.dt_hi) h = hh;
            }
            // dphi = lane dt - h - n . dr, compensated
            {
                const ff t = two_prod(ti, p.dt_hi);
                float e = fmaf(ti, p.dt_lo, t.lo);
                const ff th = two_sum(t.hi, -h);
                float sh = th.hi;
                e = e + th.lo;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const ff dd = two_prod(nh[q], dr[q]);
                    const float dl = fmaf(nlo[q], dr[q], dd.lo);
                    const ff u = two_sum(sh, -dd.hi);
                    sh = u.hi;
                    e = e + (u.lo - dl);
                }
                d = sh + e;
            }
            {
                // phi_ref: the chunk's reference phase plus the centre
                const float ph = __shfl_sync(0xffffffffu, bh, kc & 31);
                const float pl = __shfl_sync(0xffffffffu, bl, kc & 31);
                const ff u = two_sum(ph, h);
                const float l = pl + u.lo;
                an.x = __fadd_rn(u.hi, l);
                an.y = __fsub_rn(l, __fsub_rn(an.x, u.hi));
            }
            const float b0 = tb[3 * kChunk32], b1 = tb[4 * kChunk32], b2 = tb[5 * kChunk32];
            const float d0 = tb[6 * kChunk32], d1 = tb[7 * kChunk32], d2 = tb[8 * kChunk32];
            const float g = tb[9 * kChunk32];
            const float e10 = q0.w, e11 = q1.x, e12 = q1.y, e20 = q1.z, e21 = q1.w, e22 = q2.x;
            const float bn = n0 * b0 + n1 * b1 + n2 * b2;
            const float p1 = e10 * b0 + e11 * b1 + e12 * b2;
            const float p2 = e20 * b0 + e21 * b1 + e22 * b2;
            const float dn = n0 * d0 + n1 * d1 + n2 * d2;
            const float t1 = e10 * d0 + e11 * d1 + e12 * d2;
            const float t2 = e20 * d0 + e21 * d1 + e22 * d2;
            const float kap = bn > 0.0f ? (g + p1 * p1 + p2 * p2) * rcp_nr(1.0f + bn) : 1.0f - bn;
            const float rk = rcp_nr(kap);
            const float inv = S.dv[12] * rk * rk;
            V1 = -(p1 * dn + t1 * kap) * inv;
            V2 = -(p2 * dn + t2 * kap) * inv;
            if (sel >= 0 && !((__float_as_uint(tb[10 * kChunk32]) >> sel) & 1u)) V1 = V2 = 0.0f;
        }
        // the buffer has been read: chunk L + 2 into it
        __syncwarp();
        if (feeding) {
            feeding = issue(L + 2);
            if (feeding) ++issued;
        }
        __syncwarp();
        if (lo > 0 || hi < kChunk32) {
            // samples outside the window carry nothing; their offset is the nearest
            // in-window one, so that they do not widen the block
            const int at = lane < lo ? lo : (lane >= hi ? hi - 1 : lane);
            d = __shfl_sync(0xffffffffu, d, at);
            if (at != lane) V1 = V2 = 0.0f;
        }

        // ---- mode of each pair: 0 direct, 1 moments of the whole chunk, 2 / 3 of two / four
        // sub-blocks, -1 no slot in use
        auto warp_max_abs = [&](float v) {       // NaN compares above everything
            return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v) & 0x7fffffffu));
        };
        const float h1 = warp_max_abs(d);
        int mode[kPairs];
        bool big = false;
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            const float x = wm[i] * h1;
            mode[i] = wm[i] < 0.0f ? -1 : (x <= kX12 ? 1 : 0);
            big = big || (mode[i] == 0 && x <= 5.0f * kX12);   // a quarter's may fit
        }
        float h2 = 0.0f, h4 = 0.0f, c2 = 0.0f, c4 = 0.0f;
        if (big) {
            c2 = 0.5f * (__shfl_sync(0xffffffffu, d, lane & 16) +
                         __shfl_sync(0xffffffffu, d, lane | 15));
            c4 = 0.5f * (__shfl_sync(0xffffffffu, d, lane & 24) +
                         __shfl_sync(0xffffffffu, d, lane | 7));
            h2 = warp_max_abs(d - c2);
            h4 = warp_max_abs(d - c4);
#pragma unroll
            for (int i = 0; i < kPairs; ++i)
                if (mode[i] == 0) mode[i] = wm[i] * h2 <= kX12 ? 2 : (wm[i] * h4 <= kX12 ? 3 : 0);
        }
        // direct pairs as one range up to the last (a pair above a direct one joins it)
        int da = kPairs;
#pragma unroll
        for (int i = kPairs - 1; i >= 0; --i)
            if (mode[i] == 0) da = i;
        // (the frequency arrays are padded with zeros to whole tiles of 256)
        auto freq = [&](int i) -> f2 {           // omega of a pair
            return pk(__ldg(om0 + 64 * i), __ldg(om0 + 64 * i + 32));
        };
        auto anchor = [&](int i) -> f2 {         // Theta of a pair, radians
            const f2 nh = pk(__ldg(nh0 + 64 * i), __ldg(nh0 + 64 * i + 32));
            const f2 nl = pk(__ldg(nl0 + 64 * i), __ldg(nl0 + 64 * i + 32));
            return mul2(anchor_turns2(nh, nl, an), dup(6.28318530717958647f));
        };

        // ---- moments and their evaluation, one block size after the other
        uint32_t has = 0;
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            if (i >= da) mode[i] = 0;
            if (mode[i] > 0) has |= 1u << mode[i];
        }
#pragma unroll 1
        for (int md = 1; has >> md; ++md) {
            if (!((has >> md) & 1u)) continue;
            const float hm = md == 1 ? h1 : (md == 2 ? h2 : h4);
            const float cc = md == 1 ? 0.0f : (md == 2 ? c2 : c4);
            const int o0 = 32 >> md;
            // a power of two above the largest offset: exact scalings
            const uint32_t hb = (__float_as_uint(hm) & 0x7f800000u) + 0x00800000u;
            const float hs = __uint_as_float(hb), ih = __uint_as_float(0x7f000000u - hb);
            moments<kMaxP>(V1, V2, (d - cc) * ih, o0, lane, S.mom, SB.coef);
#pragma unroll
            for (int i = 0; i < kPairs; ++i) {
                if (mode[i] != md) continue;
                const f2 om = freq(i), th = anchor(i);
                const f2 x = mul2(om, dup(hs)), nx = mul2(om, dup(-hs));
#pragma unroll 1
                for (int b = 0; b < 32; b += 2 * o0) {
                    const float cb = __shfl_sync(0xffffffffu, cc, b);
                    eval_moments<kMaxP>(S.mom[b / (2 * o0)], x, nx, fma2(om, dup(cb), th), a1r[i], a1i[i],
                                        a2r[i], a2i[i]);
                }
            }
        }
        if (da < kPairs) {
            __syncwarp();
            S.geo[lane] = make_float4(V1, V2, d, 0.0f);
            __syncwarp();
            f2 om[kPairs], th[kPairs];
#pragma unroll
            for (int i = 0; i < kPairs; ++i) {
                om[i] = th[i] = 0;
                if (i >= da) {
                    om[i] = freq(i);
                    th[i] = anchor(i);
                }
            }
            switch (da) {
                case 0: direct_sum<0, 4, !COH>(S.geo, lo, hi, om, th, a1r, a1i, a2r, a2i); break;
                case 1: direct_sum<1, 4, !COH>(S.geo, lo, hi, om, th, a1r, a1i, a2r, a2i); break;
                case 2: direct_sum<2, 4, !COH>(S.geo, lo, hi, om, th, a1r, a1i, a2r, a2i); break;
                default: direct_sum<3, 4, !COH>(S.geo, lo, hi, om, th, a1r, a1i, a2r, a2i); break;
            }
        }

        ++kc;
        if (last) {
            // ---- the particle's sums are complete: into the warp's running sums
            auto add = [&](float2& a, float v) {
                const ff u = two_sum(a.x, v);
                const float l = a.y + u.lo, hh = __fadd_rn(u.hi, l);
                a = make_float2(hh, __fsub_rn(l, __fsub_rn(hh, u.hi)));
            };
#pragma unroll
            for (int i = 0; i < kPairs; ++i) {
                float r[4][2];
                upk(a1r[i], r[0][0], r[0][1]);
                upk(a1i[i], r[1][0], r[1][1]);
                upk(a2r[i], r[2][0], r[2][1]);
                upk(a2i[i], r[3][0], r[3][1]);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (!COH) {
                        add(S.ff[2 * i + j][lane], r[0][j] * r[0][j] + r[1][j] * r[1][j] +
                                                       r[2][j] * r[2][j] + r[3][j] * r[3][j]);
                    } else {
#pragma unroll
                        for (int comp = 0; comp < 4; ++comp)
                            add(S.ff[4 * (2 * i + j) + comp][lane], r[comp][j]);
                    }
                }
            }
        }
        if (flags & kLastOfItem) {
            // ---- work unit done: the FP64 accumulators
            const WorkItem it = p.items[ii];
            const WinDev w = p.wins[it.win];
            const int64_t o = w.out_off + (int64_t)it.row * w.grid_len + it.ftile * (32 * kFT) + lane - skip;
            const int left = w.grid_len - it.ftile * (32 * kFT) - lane + skip;
#pragma unroll 1
            for (int s = 0; s < kFT; ++s) {
                constexpr int NC = COH ? 4 : 1;
                for (int comp = 0; comp < NC; ++comp) {
                    const float2 a = S.ff[NC * s + comp][lane];
                    S.ff[NC * s + comp][lane] = make_float2(0.0f, 0.0f);
                    if (32 * s >= skip && 32 * s < left)
                        atomicAdd(p.acc + NC * (o + 32 * s) + comp, (double)a.x + (double)a.y);
                }
            }
        }
    }
    // never leave the block with a copy in flight: a warp waits for every copy it
    // uses, so this only matters after an expired wait
    if (lane == 0 && *abort_flag)
        for (uint32_t j = issued > 2 ? issued - 2 : 0; j < issued; ++j)
            mbar_drain(&S.full[j & 1], (j >> 1) & 1);
}

template <bool COH>
bool moment_one(const Accum32Params* p, int grid, cudaStream_t st, cudaError_t* err, int* nb)
{
    auto kern = accum32_moment_kernel<COH>;
    const size_t smem = sizeof(SmemM<COH>) + 128;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (p) {
        if (e == cudaSuccess) {
            kern<<<grid, kThreads, smem, st>>>(*p);
            e = cudaGetLastError();
        }
        *err = e;
    } else if (e != cudaSuccess || cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                       nb, kern, kThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        *nb = 0;
    }
    return true;
}

}  // namespace

bool accum32_moment(const Accum32Params* p, const Accum32Config& cfg, int grid, cudaStream_t st,
                    cudaError_t* err, int* nb)
{
    if (cfg.ft != kFT || cfg.K != 32) return false;
    return cfg.coh ? moment_one<true>(p, grid, st, err, nb) : moment_one<false>(p, grid, st, err, nb);
}

}  // namespace rad
