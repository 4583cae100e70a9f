// rad_accum64.cu -- FP64 accumulation of the far-field amplitude.
//
// Same sum as the FP32 path (Sec. 2.2, Jackson retarded-time integrand) in FP64
// throughout: phi_m = m dt - n.r_m from the ring's absolute FP64 positions, FP64
// amplitudes and particle sums.  This is the GPU reference against which the FP32
// split path is judged; on GB300 it is bound by the FP64 pipe (1/64 of FP32: two lanes
// per clock and SM), so the kernel is arranged for few FP64 instructions per update:
//
// * Block moments, as in rad_accum32_moment.cu: within a chunk of 32 samples the phase
//   is w phi_c + w dphi_m, so where |w dphi| <= 2.5 (whole chunk, halves or quarters) a
//   warp forms moments sum_m V_m dphi_m^p once and every frequency costs 12, 16 or 20
//   multiply-adds per component and one rotation per (sub-)block: 2 to 9 FP64
//   instructions per update.
// * Elsewhere e^{i theta} comes from a table of 1024 points of the unit circle and short
//   polynomials of the remainder (|delta| <= pi / 1024): 18 FP64 instructions per update
//   with the accumulation, where CUDA's sincos took 34.  Phases are in table units
//   (1024 per turn); the chunk's reference phase w phi_c is reduced with its exact
//   product error, so the phase error is that of phi itself.
//
// Every warp works on its own (one particle of a work item at a time, taken from an
// atomic counter); lane = sample for geometry and moments, lane = frequency for the
// rest, 2 to 8 frequency slots per lane.  A chunk (32 samples x components of one particle,
// 2.5 KB contiguous in the ring) comes by bulk copies (TMA) two chunks ahead.
//
// Measured: 1024 electrons x 2000 samples x 256 omega in [0.1, 300], one direction,
// 33.4 -> 13.3 ms per launch; 301 + 47 particles, 8 directions, 150 omega, coherent, three
// windows 26.2 -> 6.8 ms.  Against an 80-bit evaluation (three draws each, relative L2, sincos
// kernel / this one): 96 particles of gamma 3, 2000 samples, omega to 300 8.7e-16 / 6.7e-16; 48
// summed coherently 4.4e-15 / 3.6e-15; 32, omega to 1000, 1.4e-15 / 1.2e-15, of gamma 10
// 1.14e-14 / 7.3e-15.  (A 64-bit evaluation that forms w phi as one rounded product, as the
// sincos kernel did, agrees better with that kernel than either does with the exact sum.)
#include "rad_internal.cuh"

namespace rad {
namespace {

constexpr int kWarps = 4, kBlocks = 3, kThreads = kWarps * 32;
constexpr int kMaxP = 20;              // moments per sub-block
constexpr int kTab = 1024;             // table points per turn
constexpr int kFirstOfTile = 1, kLastOfTile = 2, kFirstOfItem = 4, kLastOfItem = 8;
constexpr double kMagic = 6755399441055744.0;   // 1.5 * 2^52: x + kMagic - kMagic = rint(x)

// cos t = sum_j C_j (-t^2)^j, sin t = t sum_j S_j (-t^2)^j (C_0, S_0, C_1, ...): minimax
// fits (fit_sincos.py, fit_moment64), the larger error of the two 7.8e-17 with 12 terms on
// |t| <= 0.45, 2.9e-17 with 16 on 1.2, 7.2e-17 with 20 on 2.5.
__device__ const double g_coef64[3][kMaxP] = {
    {1.0, 1.0, 0.4999999999999825, 0.16666666666666435, 0.04166666666544268, 0.008333333333200448,
     0.0013888888610645155, 0.00019841269575805384, 2.480131122756528e-05, 2.7557078979925243e-06,
     2.7432934213223533e-07, 2.4951101621670652e-08, 0, 0, 0, 0, 0, 0, 0, 0},
    {1.0, 1.0, 0.4999999999999984, 0.16666666666666646, 0.04166666666663812, 0.008333333333330467,
     0.0013888888887176297, 0.00019841269839798658, 2.4801586814436715e-05, 2.7557318850581163e-06,
     2.755724509036157e-07, 2.505205633787126e-08, 2.087055278373164e-09, 1.6054983232036807e-10,
     1.1201163601728481e-11, 7.480625978115661e-13, 0, 0, 0, 0},
    {1.0, 1.0, 0.49999999999999856, 0.1666666666666665, 0.0416666666666574, 0.008333333333332454,
     0.00138888888886841, 0.000198412698411059, 2.4801587279386724e-05, 2.7557319208323927e-06,
     2.7557317861678203e-07, 2.5052107514794437e-08, 2.0876706458048e-09, 1.6059014026862612e-10,
     1.146958949098133e-11, 7.646525529615967e-13, 4.7634984499532814e-14, 2.8031185637892373e-15,
     1.4391004071714364e-16, 7.60997019323244e-18}};
constexpr float kX0 = 0.45f, kX1 = 1.2f, kX2 = 2.5f;

// The walk over (work unit, particle, chunk), advanced by lane 0 only; a unit is
// particle pp of every tile of an item.
struct Cursor64 {
    const double* src;       // the particle's chunks in the ring
    int32_t ii, pp, t, nt;   // item (< 0: none left), particle of the tile, tile, tiles
    int32_t c, c0, c1;       // chunk, the window's first and last
    int32_t sc, sc0;         // their ring chunks
    int32_t lo, hi;          // first and last chunk's sample range ends
    int32_t ticket;          // the unit after that one, asked for early
};

// What lane 0 tells its warp about a chunk.
struct Meta64 {
    int32_t ii, chunk;       // item (< 0: no more work), first sample / 32
    int32_t lo, hi, flags;
};

template <int kFT, bool COH>
struct __align__(128) Warp64 {
    double raw[2][kComps * kChunk32];        // bulk-copy destinations: [component][sample]
    double2 gv[kChunk32];                    // V1, V2 per sample (direct sum)
    double gd[kChunk32];                     // dphi
    double2 mom[4][kMaxP];                   // (M1, M2) per sub-block
    double run[(COH ? 4 : 1) * kFT][32];     // particle sums
    Meta64 meta[4];
    Cursor64 cur;
    uint64_t full[2];
};

template <int kFT, bool COH>
struct Smem64 {
    Warp64<kFT, COH> w[kWarps];
    int abort_flag;
};

// e^{i 2 pi u / kTab}: 11 FP64 instructions and a table look-up.
__device__ __forceinline__ void cis_table(double u, const double2* __restrict__ tab, double& c, double& s)
{
    const double t = u + kMagic;
    const double f = u - (t - kMagic);                   // in [-1/2, 1/2], exact
    const double2 e = __ldg(tab + (__double2loint(t) & (kTab - 1)));
    constexpr double h = 6.283185307179586476925286766559 / kTab;   // radians per unit
    const double f2 = f * f;
    const double cd = fma(f2, fma(f2, h * h * h * h / 24.0, -h * h / 2.0), 1.0);
    const double sd = f * fma(f2, fma(f2, h * h * h * h * h / 120.0, -h * h * h / 6.0), h);
    c = fma(e.x, cd, -(e.y * sd));
    s = fma(e.y, cd, e.x * sd);
}

template <int N>
__device__ __forceinline__ void fold(double (&v)[2 * kMaxP], int o, bool up)
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const double a = v[i], b = v[i + N / 2];
        const double send = up ? a : b, keep = up ? b : a;
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
}

// Moments of sub-blocks of 2 o0 samples (see rad_accum32_moment.cu).
template <int P>
__device__ __forceinline__ void moments(double V1, double V2, double tau, int o0, int lane,
                                        double2 (*out)[kMaxP], const double* coef)
{
    double v[2 * kMaxP];
    v[0] = V1;
    v[1] = V2;
#pragma unroll
    for (int p = 1; p < P; ++p) {
        v[2 * p] = v[2 * p - 2] * tau;
        v[2 * p + 1] = v[2 * p - 1] * tau;
    }
    const int o1 = o0 >> 1, o2 = o0 >> 2;
    fold<2 * P>(v, o0, lane & o0);
    fold<P>(v, o1, lane & o1);
    fold<P / 2>(v, o2, lane & o2);
    constexpr int R = P / 4;
#pragma unroll 1
    for (int o = o2 >> 1; o > 0; o >>= 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] += __shfl_xor_sync(0xffffffffu, v[r], o);
    }
    const int q0 = ((lane & o0) ? P : 0) + ((lane & o1) ? P / 2 : 0) + ((lane & o2) ? P / 4 : 0);
    __syncwarp();
    if ((lane & (o2 - 1)) == 0) {
        double* dst = reinterpret_cast<double*>(out[lane / (2 * o0)]);
#pragma unroll
        for (int r = 0; r < R; ++r) dst[q0 + r] = v[r] * coef[(q0 + r) >> 1];
    }
    __syncwarp();
}

// Adds one sub-block's P moments: u the rotation in table units, x = w hs.
__device__ __forceinline__ void eval_moments(const double2* M, int P, double x, double u,
                                             const double2* tab, double& a1r, double& a1i,
                                             double& a2r, double& a2i)
{
    const double z = -(x * x);
    double2 e = M[P - 2], o = M[P - 1];
#pragma unroll 2
    for (int j = P - 4; j >= 0; j -= 2) {
        const double2 en = M[j], on = M[j + 1];
        e.x = fma(e.x, z, en.x);
        e.y = fma(e.y, z, en.y);
        o.x = fma(o.x, z, on.x);
        o.y = fma(o.y, z, on.y);
    }
    o.x *= x;
    o.y *= x;
    double c, s;
    cis_table(u, tab, c, s);
    a1r = fma(e.x, c, fma(-o.x, s, a1r));
    a1i = fma(e.x, s, fma(o.x, c, a1i));
    a2r = fma(e.y, c, fma(-o.y, s, a2r));
    a2i = fma(e.y, s, fma(o.y, c, a2i));
}

template <int kFT, bool COH>
__global__ void __launch_bounds__(kThreads, kBlocks) accum64_kernel(const Accum64Params p)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto& SB = *reinterpret_cast<Smem64<kFT, COH>*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto& S = SB.w[warp];
    const int pstride = p.comps * kChunk32;              // one particle's chunk, values
    const int rchunks = (int)(p.ring / kChunk32);
    volatile int* abort_flag = &SB.abort_flag;
    const double2* __restrict__ tab = p.cis;

    if (lane == 0) {
        mbar_init(&S.full[0], 1);
        mbar_init(&S.full[1], 1);
        fence_mbar_init();
    }
    for (int s = 0; s < (COH ? 4 : 1) * kFT; ++s) S.run[s][lane] = 0.0;
    if (tid == 0) SB.abort_flag = 0;
    __syncthreads();

    // ---- (lane 0) describe the cursor's chunk as chunk L, issue its copy and step on;
    // L < 0 only asks for the first unit.  False once there is no more work.
    auto issue = [&](int L) -> bool {
        Cursor64& C = S.cur;
        bool next_unit = L < 0;
        if (L >= 0) {
            const int buf = L & 1;
            Meta64& M = S.meta[L & 3];
            M.ii = C.ii;
            if (C.ii < 0) {
                mbar_arrive(&S.full[buf]);
                return false;
            }
            const int c = C.c;
            const bool first = c == C.c0, last = c == C.c1;
            M.chunk = c;
            M.lo = first ? C.lo : 0;
            M.hi = last ? C.hi : kChunk32;
            M.flags = (first ? kFirstOfTile : 0) | (last ? kLastOfTile : 0) |
                      (first && C.t == 0 ? kFirstOfItem : 0) |
                      (last && C.t + 1 == C.nt ? kLastOfItem : 0);
            const uint32_t bytes = (uint32_t)(pstride * sizeof(double));
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
            C.src = p.slab64 +
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

    double a1r[kFT], a1i[kFT], a2r[kFT], a2i[kFT];
    float wm[kFT];               // largest |omega| of the slot (warp-uniform); < 0: unused
    const double *om0 = nullptr, *nh0 = nullptr, *nl0 = nullptr;   // this lane's first frequency
    int left = 0, sel = -1, dir = 0;
    double qdt = 0.0;
#pragma unroll
    for (int i = 0; i < kFT; ++i) {
        a1r[i] = a1i[i] = a2r[i] = a2i[i] = 0.0;
        wm[i] = -1.0f;
    }
    // L = -3 .. -1: the first unit and its first two copies
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
        const Meta64& M = S.meta[L & 3];
        const int ii = M.ii;
        // warp-collective from here: the whole warp goes on or stops
        if (!__all_sync(0xffffffffu, ready && ii >= 0 && !*abort_flag)) break;
        const int chunk = M.chunk, lo = M.lo, hi = M.hi, flags = M.flags;
        if (flags & kFirstOfItem) {
            const WorkItem it = p.items[ii];
            const WinDev w = p.wins[it.win];
            const int kb = it.ftile * (32 * kFT);
            dir = it.dir;
            qdt = p.species[it.sp].qdt;
            sel = w.sel;
            left = w.grid_len - kb - lane;
            // (the frequency arrays are padded with zeros to whole tiles)
            om0 = p.omega + w.grid_off + kb + lane;
            nh0 = p.nu_hi + w.grid_off + kb + lane;
            nl0 = p.nu_lo + w.grid_off + kb + lane;
#pragma unroll
            for (int i = 0; i < kFT; ++i) {
                // rounded up, so that the bound holds for the FP64 value
                const uint32_t m = __reduce_max_sync(
                    0xffffffffu, __float_as_uint(__double2float_ru(fabs(om0[32 * i]))));
                wm[i] = kb + 32 * i < w.grid_len ? __uint_as_float(m) : -1.0f;
            }
        }
        if (flags & kFirstOfTile) {
#pragma unroll
            for (int i = 0; i < kFT; ++i) a1r[i] = a1i[i] = a2r[i] = a2i[i] = 0.0;
        }
        // ---- geometry, lane = sample
        double V1, V2, d, phc;
        {
            const double* tb = S.raw[buf] + lane;
            const double* dv = p.dirs64 + 9 * dir;
            const double n0 = __ldg(dv + 0), n1 = __ldg(dv + 1), n2 = __ldg(dv + 2);
            const double e10 = __ldg(dv + 3), e11 = __ldg(dv + 4), e12 = __ldg(dv + 5);
            const double e20 = __ldg(dv + 6), e21 = __ldg(dv + 7), e22 = __ldg(dv + 8);
            const double r0 = tb[0], r1 = tb[kChunk32], r2 = tb[2 * kChunk32];
            const double b0 = tb[3 * kChunk32], b1 = tb[4 * kChunk32], b2 = tb[5 * kChunk32];
            const double d0 = tb[6 * kChunk32], d1 = tb[7 * kChunk32], d2 = tb[8 * kChunk32];
            const double g = tb[9 * kChunk32];
            const double bn = n0 * b0 + n1 * b1 + n2 * b2;
            const double p1 = e10 * b0 + e11 * b1 + e12 * b2;
            const double p2 = e20 * b0 + e21 * b1 + e22 * b2;
            const double dn = n0 * d0 + n1 * d1 + n2 * d2;
            const double q1 = e10 * d0 + e11 * d1 + e12 * d2;
            const double q2 = e20 * d0 + e21 * d1 + e22 * d2;
            const double kap = bn > 0.0 ? (g + p1 * p1 + p2 * p2) / (1.0 + bn) : 1.0 - bn;
            const double inv = qdt / (kap * kap);
            V1 = -(p1 * dn + q1 * kap) * inv;
            V2 = -(p2 * dn + q2 * kap) * inv;
            if (sel >= 0 && !(((uint32_t)tb[10 * kChunk32] >> sel) & 1u)) V1 = V2 = 0.0;
            const int64_t m = (int64_t)chunk * kChunk32 + lane;
            const double ph = (double)m * p.dt - (n0 * r0 + n1 * r1 + n2 * r2);
            // the chunk's centre: the mean of its first and last in-window phases (0 where
            // that is not finite); samples outside the window carry nothing, their
            // offset is the nearest in-window one
            phc = 0.5 * (__shfl_sync(0xffffffffu, ph, lo) + __shfl_sync(0xffffffffu, ph, hi - 1));
            if (!(fabs(phc) < 1e300)) phc = 0.0;
            d = ph - phc;
            if (lo > 0 || hi < kChunk32) {
                const int at = lane < lo ? lo : (lane >= hi ? hi - 1 : lane);
                d = __shfl_sync(0xffffffffu, d, at);
                if (at != lane) V1 = V2 = 0.0;
            }
        }
        // the buffer has been read: chunk L + 2 into it
        __syncwarp();
        if (feeding) {
            feeding = issue(L + 2);
            if (feeding) ++issued;
        }
        __syncwarp();

        // ---- mode of each slot: 0 direct, 1 / 2 / 3 moments of the whole chunk with 12 /
        // 16 / 20 terms, 4 / 5 of two / four sub-blocks, -1 not in use
        auto warp_max_abs = [&](double v) {      // rounded up; NaN compares above everything
            return __uint_as_float(__reduce_max_sync(
                0xffffffffu, __float_as_uint(__double2float_ru(fabs(v))) & 0x7fffffffu));
        };
        const float h1 = warp_max_abs(d);
        const double c2 = 0.5 * (__shfl_sync(0xffffffffu, d, lane & 16) +
                                 __shfl_sync(0xffffffffu, d, lane | 15));
        const double c4 = 0.5 * (__shfl_sync(0xffffffffu, d, lane & 24) +
                                 __shfl_sync(0xffffffffu, d, lane | 7));
        const float h2 = warp_max_abs(d - c2), h4 = warp_max_abs(d - c4);
        int mode[kFT];
        uint32_t has = 0;
        int terms = 1;                           // whole-chunk slots share one set of moments
#pragma unroll
        for (int i = 0; i < kFT; ++i) {
            const float w = wm[i];
            const int m1 = w * h1 <= kX0 ? 1 : (w * h1 <= kX1 ? 2 : 3);
            mode[i] = w < 0.0f ? -1
                               : (w * h1 <= kX2 ? m1 : (w * h2 <= kX2 ? 4 : (w * h4 <= kX2 ? 5 : 0)));
            if (mode[i] >= 1 && mode[i] <= 3) terms = max(terms, mode[i]);
        }
#pragma unroll
        for (int i = 0; i < kFT; ++i) {
            if (mode[i] >= 1 && mode[i] <= 3) mode[i] = terms;
            if (mode[i] >= 0) has |= 1u << mode[i];
        }
        // the reference phase w phi_c in table units, reduced to one turn: the product
        // nu phi_c with its rounding error and nu's lo part, its integer part removed
        auto anchor = [&](int i) -> double {
            const double nh = __ldg(nh0 + 32 * i);
            const double t = __dmul_rn(nh, phc);
            const double e = fma(__ldg(nl0 + 32 * i), phc, fma(nh, phc, -t));
            const double k = __dsub_rn(__dadd_rn(t, kMagic), kMagic);
            return (__dsub_rn(t, k) + e) * (double)kTab;
        };
#pragma unroll 1
        for (int md = 1; has >> md; ++md) {
            if (!((has >> md) & 1u)) continue;
            const float hm = md <= 3 ? h1 : (md == 4 ? h2 : h4);
            const double cc = md <= 3 ? 0.0 : (md == 4 ? c2 : c4);
            const int o0 = md <= 3 ? 16 : (md == 4 ? 8 : 4);
            const int P = md == 1 ? 12 : (md == 2 ? 16 : 20);
            // a power of two above the largest offset: exact scalings
            const uint32_t hb = (__float_as_uint(hm) & 0x7f800000u) + 0x00800000u;
            const double hs = (double)__uint_as_float(hb);
            const double ih = (double)__uint_as_float(0x7f000000u - hb);
            const double tau = (d - cc) * ih;
            if (md == 1)
                moments<12>(V1, V2, tau, o0, lane, S.mom, g_coef64[0]);
            else if (md == 2)
                moments<16>(V1, V2, tau, o0, lane, S.mom, g_coef64[1]);
            else
                moments<20>(V1, V2, tau, o0, lane, S.mom, g_coef64[2]);
#pragma unroll
            for (int i = 0; i < kFT; ++i) {
                if (mode[i] != md) continue;
                const double x = __ldg(om0 + 32 * i) * hs, th = anchor(i);
                const double nu = __ldg(nh0 + 32 * i) * (double)kTab;
#pragma unroll 1
                for (int b = 0; b < 32; b += 2 * o0)
                    eval_moments(S.mom[b / (2 * o0)], P, x,
                                 fma(nu, __shfl_sync(0xffffffffu, cc, b), th), tab, a1r[i], a1i[i],
                                 a2r[i], a2i[i]);
            }
        }
        if (has & 1u) {
            // ---- direct sum, one slot at a time
            __syncwarp();
            S.gv[lane] = make_double2(V1, V2);
            S.gd[lane] = d;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kFT; ++i) {
                if (mode[i] != 0) continue;
                const double th = anchor(i), nu = __ldg(nh0 + 32 * i) * (double)kTab;
#pragma unroll 1
                for (int l = lo; l < hi; ++l) {
                    const double2 v = S.gv[l];
                    double c, s;
                    cis_table(fma(nu, S.gd[l], th), tab, c, s);
                    a1r[i] = fma(v.x, c, a1r[i]);
                    a1i[i] = fma(v.x, s, a1i[i]);
                    a2r[i] = fma(v.y, c, a2r[i]);
                    a2i[i] = fma(v.y, s, a2i[i]);
                }
            }
        }

        if (flags & kLastOfTile) {
            // ---- the particle's sums are complete: into the warp's running sums
#pragma unroll
            for (int i = 0; i < kFT; ++i) {
                if (!COH) {
                    S.run[i][lane] += a1r[i] * a1r[i] + a1i[i] * a1i[i] + a2r[i] * a2r[i] +
                                      a2i[i] * a2i[i];
                } else {
                    S.run[4 * i + 0][lane] += a1r[i];
                    S.run[4 * i + 1][lane] += a1i[i];
                    S.run[4 * i + 2][lane] += a2r[i];
                    S.run[4 * i + 3][lane] += a2i[i];
                }
            }
        }
        if (flags & kLastOfItem) {
            // ---- work unit done: the accumulators
            constexpr int NC = COH ? 4 : 1;
            const WorkItem it = p.items[ii];
            const WinDev w = p.wins[it.win];
            const int64_t o = w.out_off + (int64_t)it.row * w.grid_len + it.ftile * (32 * kFT) + lane;
#pragma unroll 1
            for (int s = 0; s < kFT; ++s) {
                for (int comp = 0; comp < NC; ++comp) {
                    if (32 * s < left) atomicAdd(p.acc + NC * (o + 32 * s) + comp, S.run[NC * s + comp][lane]);
                    S.run[NC * s + comp][lane] = 0.0;
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

template <int kFT, bool COH>
cudaError_t one(const Accum64Params* p, int grid, cudaStream_t st, int* nb)
{
    auto kern = accum64_kernel<kFT, COH>;
    const size_t smem = sizeof(Smem64<kFT, COH>) + 128;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (!p) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, kern, kThreads, smem);
    kern<<<grid, kThreads, smem, st>>>(*p);
    return cudaGetLastError();
}

cudaError_t dispatch(const Accum64Params* p, int ft, bool coh, int grid, cudaStream_t st, int* nb)
{
    switch (ft) {
        case 8: return coh ? one<8, true>(p, grid, st, nb) : one<8, false>(p, grid, st, nb);
        case 4: return coh ? one<4, true>(p, grid, st, nb) : one<4, false>(p, grid, st, nb);
        case 2: return coh ? one<2, true>(p, grid, st, nb) : one<2, false>(p, grid, st, nb);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_accum64(const Accum64Params& p, int ft, bool coh, int grid, cudaStream_t st)
{
    if (p.n_items == 0) return cudaSuccess;
    return dispatch(&p, ft, coh, grid, st, nullptr);
}

int accum64_blocks_per_sm(int ft, bool coh)
{
    int nb = 0;
    if (dispatch(nullptr, ft, coh, 0, nullptr, &nb) != cudaSuccess) cudaGetLastError();
    return nb;
}

// Frequency slots per lane.  8 share the geometry and moments of a chunk best; with
// fewer (particle, direction, tile) units than the GPU has warps for them (12 per SM),
// narrower tiles: the FP64 pipe is divided among an SM's four sub-partitions, and 1024
// equal units left some with three or more of them (15.4 ms where narrower tiles take 13.3).
int accum64_ft(int64_t particle_dirs, int n_omega, int sms)
{
    for (int ft : {8, 4})
        if (particle_dirs * ((n_omega + 32 * ft - 1) / (32 * ft)) >= (int64_t)kWarps * kBlocks * sms)
            return ft;
    return 2;
}

int accum64_table() { return kTab; }

}  // namespace rad
