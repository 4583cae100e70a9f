// rad_ingest.cu -- per-step ingest: leapfrog states -> trajectory ring.
//
// Sec. 2.2 integrates E_ret exp(i w phi') over the particle history.  This
// kernel turns the states the PIC hands over (call s: x_s, u_{s-1/2}) into
// the samples the accumulation needs, one call late: sample m = s - 1 uses
//   r_m       = unwrapped x_m (minimum image in a periodic box),
//   beta_m    = ubar / sqrt(1 + ubar^2),  ubar = (u_{m-1/2} + u_{m+1/2}) / 2,
//   betadot_m = (beta_{m+1/2} - beta_{m-1/2}) / dt,
//   g_m       = 1/gamma_m^2 = 1 / (1 + ubar^2).
// The per-particle state arrays carry the previous raw position, the image count n
// (the unwrapped position is r = x + L n) and u_{s-1/2} between launches.  Two
// kernels:
//   * ingest_tile_kernel (batches of calls): a block turns chunks of 32 samples of one
//     8-particle tile into ring records, one thread per sample, and writes each
//     record as one contiguous block;
//   * ingest_kernel (a few calls, or sub-cycling): a thread walks one particle
//     through one time segment of the launch's steps.  One call's sample of a particle
//     would be ten 4-byte stores to as many sectors of the sample-innermost ring (181 us
//     per call of 557,056 particles); the chunk that is being filled is slot-major
//     instead, eight particles to a sector, and turned when a window closes (76 us, and
//     7.2 us per call for turning it; 135 us with four FP64 divisions per call and
//     particle and the slot-major ring of before).
// Both split a launch in time when the particles alone leave the GPU idle: a later
// segment's starting image count is the launch's initial count plus the integer
// changes of the earlier segments (wind kernels), so the split changes no result.
#include <algorithm>
#include <climits>

#include "rad_internal.cuh"

namespace rad {

// Whole box lengths in a displacement d, rint(d / L): the change of the image
// count (its nearest periodic image is d - L rint(d / L)).  A particle that did
// not cross the boundary has |d| <= L/2, where that is 0 exactly; only a
// crossing pays for the FP64 division, which this GPU runs on its 1/64-rate
// FP64 pipe.  Same value in every case; NaN where the displacement is not finite (or
// 2^30 boxes long): the particle's unwrapped position is lost from there on, whichever
// kernel takes its later calls.
__device__ __forceinline__ double image_jump(double d, double L, double half_L)
{
    if (!(L > 0.0) || fabs(d) <= half_L) return 0.0;
    const double j = rint(d / L);
    return fabs(j) < 1073741824.0 ? j : __longlong_as_double(0x7ff8000000000000ll);
}

// The binary exponent and leading 20 mantissa bits of a double as a float (truncated;
// magnitudes below the float range become 0, above it infinity): integer work only.
__device__ __forceinline__ float coarse(double v)
{
    const int hi = __double2hiint(v);
    const int t = (hi & 0x7fffffff) - (896 << 20);
    const uint32_t m = t <= 0 ? 0u : (t >= (255 << 20) ? 0x7f800000u : (uint32_t)t << 3);
    return __uint_as_float(m | ((uint32_t)hi & 0x80000000u));
}

// False only if the displacement b - a is surely within half a box (no crossing): the
// difference of the coarse values plus their truncation (2^-20 of each) against
// 0.4999 L.  Keeps the 1/64-rate FP64 pipe out of the common case.
__device__ __forceinline__ bool maybe_jump(double a, double b, float lim)
{
    const float fa = coarse(a), fb = coarse(b);
    return !(fmaf(fmaxf(fabsf(fa), fabsf(fb)), 1.9073486e-6f, fabsf(fb - fa)) <= lim);
}

// maybe_jump's limit for a box (on the host: FP64 work, also once per block, shows in the
// kernels' time); boxes whose lengths leave the float range take the exact test always.
float crossing_limit(double L)
{
    return L > 1e-30 && L < 1e30 ? 0.4999f * (float)L : -1.0f;
}

// Image counts as integers; kLost stands for NaN and stays.
constexpr int kLost = INT_MIN;
__device__ __forceinline__ int as_count(double v)
{
    return fabs(v) < 2147483648.0 ? (int)v : kLost;
}
__device__ __forceinline__ int add_count(int a, int b)
{
    return a == kLost || b == kLost ? kLost : a + b;
}
__device__ __forceinline__ int sub_count(int a, int b)
{
    return a == kLost || b == kLost ? kLost : a - b;
}
__device__ __forceinline__ double from_count(int n)
{
    return n == kLost ? __longlong_as_double(0x7ff8000000000000ll) : (double)n;
}

// Calls [s_begin, s_end) of segment g of the launch.
__device__ __forceinline__ void segment_range(const IngestParams& p, int g, int64_t& s_begin,
                                              int64_t& s_end)
{
    const int64_t end = p.step0 + p.n_steps;
    if (p.n_seg <= 1) {
        s_begin = p.step0;
        s_end = end;
        return;
    }
    s_begin = g == 0 ? p.step0 : p.seg_first + (int64_t)(g - 1) * p.seg_len;
    const int64_t e = p.seg_first + (int64_t)g * p.seg_len;
    s_end = e < end ? e : end;
}

// Change of the image count over each segment but the last (box_L > 0).
__global__ void __launch_bounds__(256) wind_kernel(const IngestParams p)
{
    const int64_t cnt = p.count ? p.count : p.n_in - p.first;
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= cnt * (p.n_seg - 1)) return;
    const int g = (int)(q / cnt);
    const int64_t k = q - (int64_t)g * cnt, i = p.first + k;
    const int64_t ld = p.ld ? p.ld : p.n_in;
    const int64_t xi = i - p.xoff;
    int sp = 0;
    while (sp + 1 < p.n_species && i >= p.in_off[sp + 1]) ++sp;
    const int64_t col = p.col_off[sp] + (i - p.in_off[sp]);
    int64_t s_begin, s_end;
    segment_range(p, g, s_begin, s_end);
    const double half_L = 0.5 * p.box_L;
    double xp[3];
    bool have = true;
    if (s_begin > p.step0) {
        for (int c = 0; c < 3; ++c) xp[c] = p.x[(s_begin - 1 - p.step0) * 3 * ld + c * ld + xi];
    } else if (p.step0 > 0) {
        for (int c = 0; c < 3; ++c) xp[c] = p.x_prev[c * p.ncols + col];
    } else {
        have = false;                       // call 0 has no predecessor
    }
    int32_t dn[3] = {0, 0, 0};
    for (int64_t s = s_begin; s < s_end; ++s) {
        for (int c = 0; c < 3; ++c) {
            const double xn = p.x[(s - p.step0) * 3 * ld + c * ld + xi];
            if (have) dn[c] = sub_count(dn[c], as_count(image_jump(xn - xp[c], p.box_L, half_L)));
            xp[c] = xn;
        }
        have = true;
    }
    for (int c = 0; c < 3; ++c) p.wind[((int64_t)g * 3 + c) * cnt + k] = dn[c];
}

// Selector bits of a sample: box tests on the position as handed over, cone
// tests on cos(angle(ubar, axis)) = ubar.axis / |ubar|, in FP64 without
// contraction (the oracle takes the same decisions bit for bit).
__device__ uint32_t selector_bits(const IngestParams& p, const double x[3], const double ub[3])
{
    uint32_t bits = 0;
    for (int i = 0; i < p.n_sel; ++i) {
        const SelectorDev& S = p.sel[i];
        bool in = false;
        if (S.kind == 1) {
            in = x[0] >= S.lo[0] && x[0] < S.hi[0] && x[1] >= S.lo[1] && x[1] < S.hi[1] &&
                 x[2] >= S.lo[2] && x[2] < S.hi[2];
        } else if (S.kind == 2) {
            const double par = __dadd_rn(__dadd_rn(__dmul_rn(ub[0], S.axis[0]), __dmul_rn(ub[1], S.axis[1])),
                                         __dmul_rn(ub[2], S.axis[2]));
            const double nrm = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ub[0], ub[0]), __dmul_rn(ub[1], ub[1])),
                                                    __dmul_rn(ub[2], ub[2])));
            const double cs = __ddiv_rn(par, nrm);
            in = cs >= S.cos_lo && cs <= S.cos_hi;
        }
        bits |= (in ? 1u : 0u) << i;
    }
    return bits;
}

// Component 0 of a sample in either ring (components are kChunk32 apart).
template <class T>
__device__ __forceinline__ T* slab_at(T* slab, const IngestParams& p, int64_t tile, int64_t slot,
                                      int64_t pp)
{
    return slab + (((tile * p.ring + slot) / kChunk32 * kTileP + pp) * p.comps) * kChunk32 +
           slot % kChunk32;
}

// 1 / gamma of a momentum, FP64.  Written with explicit fused operations: both ingest
// kernels have to give the same bits whatever surrounds the call.
__device__ __forceinline__ double inv_gamma(double a, double b, double c)
{
    return rsqrt(fma(a, a, fma(b, b, fma(c, c, 1.0))));
}

// 64-thread blocks (launch_ingest), 7 of them resident per SM: 146 registers hold the loop
// without spilling, and the warps left hide its FP64 latency (557,056 particles, us per call
// of 512-call batches / of single calls: 6 blocks 24.0 / 85.7, 7 26.2 / 78.7, 8 30.6 / 81.7;
// the FP64 instructions alone would take 17).
// MODE as in ingest_tile_kernel (1, the precise-phase ring, also takes the lo part of each
// position offset), SUB sub-cycled samples: builds of their own, so that the common one
// carries none of that work and none of its registers.
template <int MODE, bool SUB>
__global__ void __launch_bounds__(64, SUB ? 6 : 7) ingest_kernel(const IngestParams p)
{
    const int64_t cnt = p.count ? p.count : p.n_in - p.first;
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int nseg = p.n_seg > 1 ? p.n_seg : 1;
    if (q >= cnt * nseg) return;
    const int g = (int)(q / cnt);                // time segment
    const int64_t k = q - (int64_t)g * cnt;
    const int64_t i = p.first + k;
    const int64_t ld = p.ld ? p.ld : p.n_in;    // input particle stride
    const int64_t xi = i - p.xoff;              // input column of particle i
    int64_t s_begin, s_end;
    segment_range(p, g, s_begin, s_end);
    const int n_loc = (int)(s_end - s_begin);   // calls of this thread
    const int64_t t0 = s_begin - p.step0;       // its first input row
    int sp = 0;
    while (sp + 1 < p.n_species && i >= p.in_off[sp + 1]) ++sp;
    const int64_t col = p.col_off[sp] + (i - p.in_off[sp]);
    const int64_t nc = p.ncols;
    const int64_t tile = col / kTileP, pp = col % kTileP;

    double xp[3], off[3], rp[3], up[3], ra[3];   // off = L n
    int img[3];                          // image counts n
    const double half_L = 0.5 * p.box_L;
    const bool box = p.box_L > 0.0;
    const float lim = p.lim;
    const float idt = (float)p.idt;
    const bool have_state = s_begin > 0;
    // ring slot, position in the anchor block and anchor block of the next sample
    // (nsub = 1), advanced by counters instead of 64-bit divisions (a ring has far
    // fewer than 2^31 samples; nblk is 0 for an FP64 ring, which has no anchors)
    const int64_t m_next = s_begin > 0 ? s_begin - 1 : 0;
    const int ring = (int)p.ring, nblk = (int)p.nblk;
    int slot_n = (int)(m_next % p.ring), kpos_n = (int)(m_next % p.K);
    int blk_n = p.nblk > 0 ? (int)((m_next / p.K) % p.nblk) : 0;
    // this thread's calls whose sample the ring takes: [keep_a, keep_b)
    const int keep_a = (int)min(max(p.keep0 + 1 - s_begin, int64_t(0)), int64_t(n_loc));
    const int keep_b = (int)min(max(p.keep1 + 1 - s_begin, int64_t(0)), int64_t(n_loc));
    // the current chunk's layout (a chunk that starts here takes the launch's)
    bool sm = g == 0 ? p.slot_major0 : p.slot_major;
    // component 0 of a sample in FP32 ring slot `slot`; os: from component to component
    auto slab32_at = [&](int64_t slot, int& os) {
        if (slot % kChunk32 == 0) sm = p.slot_major;
        os = sm ? kTileP : kChunk32;
        return sm ? p.slab32 + (tile * p.ring + slot) * (p.comps * kTileP) + pp
                  : slab_at(p.slab32, p, tile, slot, pp);
    };
    if (have_state) {
        for (int c = 0; c < 3; ++c) {
            // image count at the launch start, plus the earlier segments' changes
            img[c] = box && p.step0 > 0 ? as_count(p.r_prev[c * nc + col]) : 0;
            for (int h = 0; h < g && box; ++h)
                img[c] = add_count(img[c], p.wind[((int64_t)h * 3 + c) * cnt + k]);
            off[c] = box ? p.box_L * from_count(img[c]) : 0.0;
            if (g == 0) {
                xp[c] = p.x_prev[c * nc + col];
                up[c] = p.u_prev[c * nc + col];
            } else {
                xp[c] = p.x[(t0 - 1) * 3 * ld + c * ld + xi];
                up[c] = p.u[(t0 - 1) * 3 * ld + c * ld + xi];
            }
            rp[c] = xp[c] + off[c];
        }
    }
    bool have_anchor = false, have_uf = false;
    float uf[3] = {0.0f, 0.0f, 0.0f};    // FP32 ring: u of the last sample's later call
    bool bad = false;

    // the next step's inputs are loaded while this step is being processed
    double xq[3], uq[3];
    const double *xs = p.x + t0 * 3 * ld + xi, *us = p.u + t0 * 3 * ld + xi;
    for (int c = 0; c < 3; ++c) {
        xq[c] = n_loc > 0 ? xs[c * ld] : 0.0;
        uq[c] = n_loc > 0 ? us[c * ld] : 0.0;
    }
    for (int t = 0; t < n_loc; ++t) {
        double xn[3], un[3], rn[3];
        for (int c = 0; c < 3; ++c) {
            xn[c] = xq[c];
            un[c] = uq[c];
        }
        if (t + 1 < n_loc) {
            xs += 3 * ld;
            us += 3 * ld;
            for (int c = 0; c < 3; ++c) {
                xq[c] = xs[c * ld];
                uq[c] = us[c * ld];
            }
        }
        if (p.check) {
            for (int c = 0; c < 3; ++c) bad |= !isfinite(xn[c]) || !isfinite(un[c]);
        }
        if (!have_state && t == 0) {     // call 0
            for (int c = 0; c < 3; ++c) {
                xp[c] = xn[c];
                img[c] = 0;
                off[c] = 0.0;
                rp[c] = xn[c];
                up[c] = un[c];
            }
            continue;
        }
        // unwrapped position of this call: r = x + L n, n counting box crossings
        for (int c = 0; c < 3; ++c) {
            if (box && maybe_jump(xp[c], xn[c], lim)) {
                const double jump = image_jump(xn[c] - xp[c], p.box_L, half_L);
                if (jump != 0.0) {
                    img[c] = sub_count(img[c], as_count(jump));
                    off[c] = p.box_L * from_count(img[c]);
                }
            }
            rn[c] = xn[c] + off[c];
        }

        // sample m = s - 1: r_m = rp, u_{m-1/2} = up, u_{m+1/2} = un
        const int slot = slot_n, kpos = kpos_n, blk = blk_n;
        if (++slot_n == ring) slot_n = 0;
        if (++kpos_n == p.K) {
            kpos_n = 0;
            if (++blk_n == nblk) blk_n = 0;
        }
        if (SUB) {
            // Sub-cycling (Sec. 2.2: tracked particles sub-cycled at
            // dt_synth <= dt_sim / 10): n sub-samples per PIC sample at
            // tau = (k + 1/2)/n - 1/2, u(tau) = ubar + tau du linear in time
            // between the half-step states, betadot the exact derivative of
            // u/gamma(u) for that u, r(tau) = r_m + dt * Simpson integral of
            // beta over [0, tau].  Sub-sample M = m n + k lives in ring slot
            // M mod ring; the samples' selector flags are those of sample m.
            double ub[3], du[3], b0[3];
            for (int c = 0; c < 3; ++c) {
                ub[c] = 0.5 * (up[c] + un[c]);
                du[c] = un[c] - up[c];
            }
            const double g0 = sqrt(1.0 + (ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2]));
            for (int c = 0; c < 3; ++c) b0[c] = ub[c] / g0;
            const uint32_t flags = p.n_sel ? selector_bits(p, xp, ub) : 0xffffffffu;
            const int64_t m = s_begin + t - 1;
            for (int k = 0; k < p.nsub; ++k) {
                const double tau = (k + 0.5) / p.nsub - 0.5;
                double uk[3], uh[3], bk[3], bh[3], bd[3], rk[3];
                for (int c = 0; c < 3; ++c) {
                    uk[c] = ub[c] + tau * du[c];
                    uh[c] = ub[c] + 0.5 * tau * du[c];
                }
                const double gk2 = 1.0 + (uk[0] * uk[0] + uk[1] * uk[1] + uk[2] * uk[2]);
                const double gk = sqrt(gk2);
                const double gh = sqrt(1.0 + (uh[0] * uh[0] + uh[1] * uh[1] + uh[2] * uh[2]));
                const double udot_u = (uk[0] * du[0] + uk[1] * du[1] + uk[2] * du[2]) / p.dt;
                for (int c = 0; c < 3; ++c) {
                    bk[c] = uk[c] / gk;
                    bh[c] = uh[c] / gh;
                    bd[c] = (du[c] / p.dt) / gk - uk[c] * udot_u / (gk2 * gk);
                    rk[c] = rp[c] + p.dt * (tau / 6.0) * (b0[c] + 4.0 * bh[c] + bk[c]);
                }
                const int64_t M = m * p.nsub + k;
                if (M < p.keep0 || M >= p.keep1) continue;
                const int64_t sl = M % p.ring;
                if (MODE != 2) {
                    float* an = p.anc32 + ((tile * p.nblk + (M / p.K) % p.nblk) * kTileP + pp) * 6;
                    if ((M % p.K) == 0 || !have_anchor) {
                        if ((M % p.K) == 0) {
                            for (int c = 0; c < 3; ++c) {
                                const float hi = (float)rk[c];
                                const float lo = (float)(rk[c] - (double)hi);
                                an[c] = hi;
                                an[3 + c] = lo;
                                ra[c] = (double)hi + (double)lo;
                            }
                        } else {
                            for (int c = 0; c < 3; ++c)
                                ra[c] = (double)an[c] + (double)an[3 + c];
                        }
                        have_anchor = true;
                    }
                    int os;
                    float* o = slab32_at(sl, os);
                    for (int c = 0; c < 3; ++c) {
                        const double d = rk[c] - ra[c];
                        const float dh = (float)d;
                        o[c * os] = dh;
                        if (MODE == 1) o[(11 + c) * os] = (float)(d - (double)dh);
                        o[(3 + c) * os] = (float)bk[c];
                        o[(6 + c) * os] = (float)bd[c];
                    }
                    o[9 * os] = (float)(1.0 / gk2);
                    if (p.comps > kCompsPlain) o[10 * os] = __uint_as_float(flags);
                } else {
                    double* o = slab_at(p.slab64, p, tile, sl, pp);
                    for (int c = 0; c < 3; ++c) {
                        o[c * kChunk32] = rk[c];
                        o[(3 + c) * kChunk32] = bk[c];
                        o[(6 + c) * kChunk32] = bd[c];
                    }
                    o[9 * kChunk32] = 1.0 / gk2;
                    if (p.comps > kCompsPlain) o[10 * kChunk32] = (double)flags;
                }
            }
        } else if (t < keep_a || t >= keep_b) {
            // no window needs the sample
        } else if (MODE != 2) {
            // FP32 ring: the only cancellation-prone quantities are differenced
            // in FP64 -- du = u_{m+1/2} - u_{m-1/2} and r_m - r_anchor -- and the
            // rest is evaluated in FP32 through the rearrangement
            //   beta_+ - beta_- = du/g_+ - u_- (du.(u_+ + u_-)) / (g_+ g_- (g_+ + g_-)),
            // which has no cancellation for the magnetic (du perpendicular to u)
            // and weakly parallel accelerations a frozen-field push produces.
            // anchor position r_a as an FP32 hi + lo pair; dr is taken relative
            // to exactly hi + lo, the value the accumulation kernel sees
            float* an = p.anc32 + ((tile * p.nblk + blk) * kTileP + pp) * 6;
            if (kpos == 0) {
                for (int c = 0; c < 3; ++c) {
                    const float hi = (float)rp[c];
                    const float lo = (float)(rp[c] - (double)hi);
                    an[c] = hi;
                    an[3 + c] = lo;
                    ra[c] = (double)hi + (double)lo;
                }
                have_anchor = true;
            } else if (!have_anchor) {
                for (int c = 0; c < 3; ++c) ra[c] = (double)an[c] + (double)an[3 + c];
                have_anchor = true;
            }
            float um[3], uq[3], du[3], ub[3];
            for (int c = 0; c < 3; ++c) {
                um[c] = have_uf ? uf[c] : (float)up[c];
                uq[c] = uf[c] = (float)un[c];
                du[c] = (float)(un[c] - up[c]);
                ub[c] = 0.5f * (um[c] + uq[c]);
            }
            have_uf = true;
            const float gm = sqrtf(1.0f + (um[0] * um[0] + um[1] * um[1] + um[2] * um[2]));
            const float gq = sqrtf(1.0f + (uq[0] * uq[0] + uq[1] * uq[1] + uq[2] * uq[2]));
            const float gb2 = 1.0f + (ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2]);
            const float igb = rsqrtf(gb2);
            const float dus = du[0] * (uq[0] + um[0]) + du[1] * (uq[1] + um[1]) +
                              du[2] * (uq[2] + um[2]);
            const float igq = 1.0f / gq;
            const float corr = dus / (gq * gm * (gq + gm));
            int os;
            float* o = slab32_at(slot, os);
            for (int c = 0; c < 3; ++c) {
                const double d = rp[c] - ra[c];
                const float dh = (float)d;
                o[c * os] = dh;
                // precise-phase ring: the rounding of the offset as its lo part
                if (MODE == 1) o[(11 + c) * os] = (float)(d - (double)dh);
            }
            o[3 * os] = ub[0] * igb;
            o[4 * os] = ub[1] * igb;
            o[5 * os] = ub[2] * igb;
            o[6 * os] = (du[0] * igq - um[0] * corr) * idt;
            o[7 * os] = (du[1] * igq - um[1] * corr) * idt;
            o[8 * os] = (du[2] * igq - um[2] * corr) * idt;
            o[9 * os] = 1.0f / gb2;
            if (p.comps > kCompsPlain) {
                double ubd[3] = {__dmul_rn(0.5, __dadd_rn(up[0], un[0])),
                                 __dmul_rn(0.5, __dadd_rn(up[1], un[1])),
                                 __dmul_rn(0.5, __dadd_rn(up[2], un[2]))};
                o[10 * os] = __uint_as_float(p.n_sel ? selector_bits(p, xp, ubd) : 0xffffffffu);
            }
        } else {
            double ub[3];
            for (int c = 0; c < 3; ++c) ub[c] = 0.5 * (up[c] + un[c]);
            const double igm = inv_gamma(up[0], up[1], up[2]), igp = inv_gamma(un[0], un[1], un[2]);
            const double igb = inv_gamma(ub[0], ub[1], ub[2]);
            double* o = slab_at(p.slab64, p, tile, slot, pp);
            for (int c = 0; c < 3; ++c) {
                o[c * kChunk32] = rp[c];
                o[(3 + c) * kChunk32] = ub[c] * igb;
                o[(6 + c) * kChunk32] =
                    __dmul_rn(__dsub_rn(__dmul_rn(un[c], igp), __dmul_rn(up[c], igm)), p.idt);
            }
            o[9 * kChunk32] = igb * igb;
            if (p.comps > kCompsPlain) {
                double ubd[3] = {__dmul_rn(0.5, __dadd_rn(up[0], un[0])),
                                 __dmul_rn(0.5, __dadd_rn(up[1], un[1])),
                                 __dmul_rn(0.5, __dadd_rn(up[2], un[2]))};
                o[10 * kChunk32] = (double)(p.n_sel ? selector_bits(p, xp, ubd) : 0xffffffffu);
            }
        }
        for (int c = 0; c < 3; ++c) {
            xp[c] = xn[c];
            rp[c] = rn[c];
            up[c] = un[c];
        }
    }
    if (g == nseg - 1) {                        // the launch's last segment carries the state on
        if (nseg > 1) {
            // segment 0 may still be reading the state arrays: stage it
            for (int c = 0; c < 3; ++c) {
                p.state_out[c * cnt + k] = xp[c];
                p.state_out[(3 + c) * cnt + k] = box ? from_count(img[c]) : 0.0;
                p.state_out[(6 + c) * cnt + k] = up[c];
            }
        } else {
            for (int c = 0; c < 3; ++c) {
                p.x_prev[c * nc + col] = xp[c];
                p.r_prev[c * nc + col] = box ? from_count(img[c]) : 0.0;
                p.u_prev[c * nc + col] = up[c];
            }
        }
    }
    if (bad) atomicOr(p.err_word, kErrNaN);
}

// The staged carry-over state of a segmented launch into the state arrays.
__global__ void store_state(const IngestParams p)
{
    const int64_t cnt = p.count ? p.count : p.n_in - p.first;
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= cnt) return;
    const int64_t i = p.first + k;
    int sp = 0;
    while (sp + 1 < p.n_species && i >= p.in_off[sp + 1]) ++sp;
    const int64_t col = p.col_off[sp] + (i - p.in_off[sp]);
    for (int c = 0; c < 3; ++c) {
        p.x_prev[c * p.ncols + col] = p.state_out[c * cnt + k];
        p.r_prev[c * p.ncols + col] = p.state_out[(3 + c) * cnt + k];
        p.u_prev[c * p.ncols + col] = p.state_out[(6 + c) * cnt + k];
    }
}

// Geometry of a batched launch: samples [m0, m1], chunks [c0, c1], calls up to s1.
struct BatchRange {
    int64_t m0, m1, s1, c0, c1;
};
__host__ __device__ __forceinline__ BatchRange batch_range(const IngestParams& p)
{
    BatchRange b;
    b.m0 = p.step0 > 0 ? p.step0 - 1 : 0;
    b.s1 = p.step0 + p.n_steps - 1;
    b.m1 = b.s1 - 1;
    b.c0 = b.m0 / kChunk32;
    b.c1 = b.m1 / kChunk32;
    return b;
}

// Particle of tile column col: its species' input index, or -1 (padding, or outside
// the launch's particle range).
__device__ __forceinline__ int64_t tile_particle(const IngestParams& p, int64_t col)
{
    int sp = 0;
    while (sp + 1 < p.n_species &&
           (col >= p.col_off[sp + 1] || p.in_off[sp + 1] == p.in_off[sp]))
        ++sp;
    const int64_t i = p.in_off[sp] + (col - p.col_off[sp]);
    const int64_t end = p.count ? p.first + p.count : p.n_in;
    return col >= p.col_off[sp] && i < p.in_off[sp + 1] && i >= p.first && i < end ? i : -1;
}

// Change of the image count over each segment but the last of a batched launch
// (box_L > 0): a block per tile and segment, a thread per particle and chunk of 32
// calls with eight calls' loads in flight (one thread per particle and whole segment
// took 60 us for 1024 particles x 2000 calls, a chain of 28 load rounds).
__global__ void __launch_bounds__(256) tile_wind_kernel(const IngestParams p)
{
    __shared__ int tot[3][kTileP], lost[3][kTileP];
    const int tid = threadIdx.x, pp = tid & (kTileP - 1);
    const int tile_l = (int)(blockIdx.x % p.n_tiles), g = (int)(blockIdx.x / p.n_tiles);
    const int64_t col = (p.tile0 + tile_l) * kTileP + pp;
    const int64_t i = tile_particle(p, col);
    const int64_t npart = p.count ? p.count : p.n_in - p.first;
    const int64_t ld = p.ld ? p.ld : p.n_in;
    const BatchRange b = batch_range(p);
    const float lim = p.lim;
    const double half_L = 0.5 * p.box_L;
    if (tid < 3 * kTileP) tot[tid >> 3][pp] = lost[tid >> 3][pp] = 0;
    __syncthreads();
    int dn[3] = {0, 0, 0};
    if (i >= 0) {
        const double* x = p.x + (i - p.xoff);
        for (int q = tid >> 3; q < p.seg_len; q += 32) {
            // calls (sa, sb] of chunk q of the segment
            const int64_t c = b.c0 + (int64_t)g * p.seg_len + q;
            const int64_t sa = max(b.m0, c * kChunk32), sb = (c + 1) * kChunk32;
            double xp[3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                xp[k] = sa >= p.step0 ? x[((sa - p.step0) * 3 + k) * ld] : p.x_prev[k * p.ncols + col];
            constexpr int U = 8;
            for (int64_t s = sa + 1; s <= sb; s += U) {
                double xn[U][3];
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        xn[u][k] = x[((min(s + u, sb) - p.step0) * 3 + k) * ld];
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (maybe_jump(xp[k], xn[u][k], lim))
                            dn[k] = sub_count(dn[k], as_count(image_jump(xn[u][k] - xp[k], p.box_L, half_L)));
                        xp[k] = xn[u][k];
                    }
            }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (dn[k] == kLost)
                lost[k][pp] = 1;
            else if (dn[k])
                atomicAdd(&tot[k][pp], dn[k]);
        }
    }
    __syncthreads();
    if (tid < 3 * kTileP && i >= 0)
        p.wind[((int64_t)g * 3 + (tid >> 3)) * npart + (i - p.first)] =
            lost[tid >> 3][pp] ? kLost : tot[tid >> 3][pp];
}

// One block: chunks [q0, q1) (32 samples each) of one 8-particle tile, thread = sample
// and particle.  Rows of 33 calls go through shared memory (a sample needs u of two
// calls); the image counts change only at a crossing, found with integer and FP32
// work, so the FP64 work per sample is one subtraction and two conversions per
// component of x and u (the previous kernel, one thread per particle for every call,
// ran 27 FP64 instructions per sample and a serial chain over the calls: 192 us for
// 1024 particles x 2000 calls).  The record of a chunk is staged in shared memory and
// written as one contiguous block.  MODE 0: FP32 ring, 1: the precise-phase FP32 ring
// (the offsets' lo part too), 2: FP64 ring (samples written directly, four to a sector).
template <int MODE>
__global__ void __launch_bounds__(256, MODE == 0 ? 4 : 2) ingest_tile_kernel(const IngestParams p)
{
    __shared__ double xs[kChunk32 + 1][3][kTileP], us[kChunk32 + 1][3][kTileP];
    __shared__ double ras[kChunk32 / 8][3][kTileP];
    __shared__ int cnt[3][kTileP], moved[3][kTileP];
    // FP32: [particle][comp][sample], padded; FP64: beta at the half steps.  Before that,
    // the crossings of a chunk that has any.
    extern __shared__ __align__(16) float outs[];
    int(*jc)[3][kTileP] = reinterpret_cast<int(*)[3][kTileP]>(outs);
    double(*bh)[3][kTileP] = reinterpret_cast<double(*)[3][kTileP]>(outs);
    const int tid = threadIdx.x, sm = tid >> 3, pp = tid & (kTileP - 1);
    const int tile_l = (int)(blockIdx.x % p.n_tiles), g = (int)(blockIdx.x / p.n_tiles);
    const int64_t tile = p.tile0 + tile_l, col = tile * kTileP + pp;
    const int64_t i = tile_particle(p, col);
    const int64_t npart = p.count ? p.count : p.n_in - p.first;
    const int64_t ld = p.ld ? p.ld : p.n_in, xi = i - p.xoff;
    const BatchRange b = batch_range(p);
    const int64_t q0 = b.c0 + (int64_t)g * p.seg_len;
    const int64_t q1 = min(q0 + p.seg_len, b.c1 + 1);
    const bool box = p.box_L > 0.0;
    const float lim = p.lim;
    const float idt = (float)p.idt;
    const int ostride = p.comps * kChunk32 + 4;
    bool bad = false;

    if (tid < 3 * kTileP) {
        const int c = tid >> 3;
        int n = 0;
        if (box && i >= 0) {
            if (p.step0 > 0) n = as_count(p.r_prev[c * p.ncols + col]);
            for (int h = 0; h < g; ++h)
                n = add_count(n, p.wind[((int64_t)h * 3 + c) * npart + (i - p.first)]);
        }
        cnt[c][pp] = n;
    }
    auto row = [&](int64_t s, int r, int c) {            // one value each of x and u
        double xv = 0.0, uv = 0.0;
        if (i >= 0 && s >= b.m0 && s <= b.s1) {
            if (s >= p.step0) {
                xv = p.x[((s - p.step0) * 3 + c) * ld + xi];
                uv = p.u[((s - p.step0) * 3 + c) * ld + xi];
                if (p.check) bad |= !isfinite(xv) || !isfinite(uv);
            } else {
                xv = p.x_prev[c * p.ncols + col];
                uv = p.u_prev[c * p.ncols + col];
            }
        }
        xs[r][c][pp] = xv;
        us[r][c][pp] = uv;
    };
    uint32_t rc = (uint32_t)(q0 % (p.ring / kChunk32));  // ring chunk of chunk q
    for (int64_t q = q0; q < q1; ++q) {
        const int64_t m = q * kChunk32 + sm, slot0 = (int64_t)rc * kChunk32;
        if (++rc == (uint32_t)(p.ring / kChunk32)) rc = 0;
        const bool valid = m >= b.m0 && m <= b.m1;
        const bool keep = q * kChunk32 >= p.keep0 && q * kChunk32 < p.keep1;
#pragma unroll
        for (int c = 0; c < 3; ++c) row(m, sm, c);
        if (tid < 3 * kTileP) row(q * kChunk32 + kChunk32, kChunk32, tid >> 3);
        __syncthreads();
        double x[3], up[3], un[3];
        bool jump = false;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[c] = xs[sm][c][pp];
            up[c] = us[sm][c][pp];
            un[c] = us[sm + 1][c][pp];
            jump |= box && valid && maybe_jump(x[c], xs[sm + 1][c][pp], lim);
        }
        // image counts: the chunk's starting count unless something crossed in it
        const bool any = __syncthreads_or(jump);
        int n[3] = {cnt[0][pp], cnt[1][pp], cnt[2][pp]};
        bool gone = false;               // a crossing count of the chunk is kLost
        if (any) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int j =
                    jump ? as_count(image_jump(xs[sm + 1][c][pp] - x[c], p.box_L, 0.5 * p.box_L)) : 0;
                jc[sm][c][pp] = j;
                gone |= j == kLost;
            }
            gone = __syncthreads_or(gone);
            if (!gone) {
                for (int r = 0; r < sm; ++r)
#pragma unroll
                    for (int c = 0; c < 3; ++c) n[c] -= jc[r][c][pp];
            } else {
#pragma unroll 1
                for (int r = 0; r < sm; ++r)
#pragma unroll
                    for (int c = 0; c < 3; ++c) n[c] = sub_count(n[c], jc[r][c][pp]);
            }
        }
        // a lost count makes the position NaN (its own count then is of no interest)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (cnt[c][pp] == kLost || n[c] == kLost) {
                x[c] = __longlong_as_double(0x7ff8000000000000ll);
                n[c] = 0;
            }
        // anchors: r_a as an FP32 hi + lo pair; offsets are relative to exactly hi + lo
        if (MODE != 2 && keep && sm % p.K == 0) {
            float* an = p.anc32 + ((tile * p.nblk + (slot0 + sm) / p.K) * kTileP + pp) * 6;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float hi = 0.0f, lo = 0.0f;
                if (valid && i >= 0) {
                    const double r = x[c] + p.box_L * (double)n[c];
                    hi = (float)r;
                    lo = (float)(r - (double)hi);
                    an[c] = hi;
                    an[3 + c] = lo;
                } else if (i >= 0 && m < b.m0) {         // written by an earlier launch
                    hi = an[c];
                    lo = an[3 + c];
                }
                const double ra = (double)hi + (double)lo;
                ras[sm / p.K][c][pp] = any ? ra : ra - p.box_L * (double)n[c];
            }
        }
        __syncthreads();                                 // ras; jc read by everyone
        if (any && tid < 3 * kTileP) {
            int t = 0;
            if (!gone) {
                for (int r = 0; r < kChunk32; ++r) t += jc[r][tid >> 3][pp];
            } else {
#pragma unroll 1
                for (int r = 0; r < kChunk32; ++r) t = add_count(t, jc[r][tid >> 3][pp]);
            }
            moved[tid >> 3][pp] = t;                     // zero beyond the last call
        }
        if (any) __syncthreads();
        if (!keep) {
            // no window needs the chunk
        } else if (MODE == 2) {
            // beta at the half steps, once per call (a sample uses two neighbouring ones):
            // one reciprocal square root where the samples took three square roots and
            // ten divisions between them (154 FP64 instructions each)
            auto half = [&](int r) {
                const double ig = inv_gamma(us[r][0][pp], us[r][1][pp], us[r][2][pp]);
                for (int c = 0; c < 3; ++c) bh[r][c][pp] = __dmul_rn(us[r][c][pp], ig);
            };
            half(sm);
            if (sm == 0) half(kChunk32);
            __syncthreads();
            if (valid && i >= 0) {
                double ub[3];
                for (int c = 0; c < 3; ++c) ub[c] = 0.5 * (up[c] + un[c]);
                const double igb = inv_gamma(ub[0], ub[1], ub[2]);
                double* o = slab_at(p.slab64, p, tile, slot0 + sm, pp);
                for (int c = 0; c < 3; ++c) {
                    o[c * kChunk32] = n[c] ? __dadd_rn(x[c], __dmul_rn(p.box_L, (double)n[c])) : x[c];
                    o[(3 + c) * kChunk32] = ub[c] * igb;
                    o[(6 + c) * kChunk32] = __dmul_rn(__dsub_rn(bh[sm + 1][c][pp], bh[sm][c][pp]), p.idt);
                }
                o[9 * kChunk32] = igb * igb;
                if (p.comps > kCompsPlain) {
                    double ubd[3] = {__dmul_rn(0.5, __dadd_rn(up[0], un[0])),
                                     __dmul_rn(0.5, __dadd_rn(up[1], un[1])),
                                     __dmul_rn(0.5, __dadd_rn(up[2], un[2]))};
                    const double xraw[3] = {xs[sm][0][pp], xs[sm][1][pp], xs[sm][2][pp]};
                    o[10 * kChunk32] = (double)(p.n_sel ? selector_bits(p, xraw, ubd) : 0xffffffffu);
                }
            }
        } else {
            // as ingest_kernel: only the cancellation-prone differences in FP64
            float* o = outs + pp * ostride + sm;
            float um[3], uq[3], du[3], ub[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double ra = ras[sm / p.K][c][pp];
                const double d = any ? (x[c] + p.box_L * (double)n[c]) - ra : x[c] - ra;
                const float dh = (float)d;
                o[c * kChunk32] = dh;
                if (MODE == 1) o[(11 + c) * kChunk32] = (float)(d - (double)dh);
                um[c] = (float)up[c];
                uq[c] = (float)un[c];
                du[c] = (float)(un[c] - up[c]);
                ub[c] = 0.5f * (um[c] + uq[c]);
            }
            const float gm = sqrtf(1.0f + (um[0] * um[0] + um[1] * um[1] + um[2] * um[2]));
            const float gq = sqrtf(1.0f + (uq[0] * uq[0] + uq[1] * uq[1] + uq[2] * uq[2]));
            const float gb2 = 1.0f + (ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2]);
            const float igb = rsqrtf(gb2);
            const float dus = du[0] * (uq[0] + um[0]) + du[1] * (uq[1] + um[1]) +
                              du[2] * (uq[2] + um[2]);
            const float igq = 1.0f / gq;
            const float corr = dus / (gq * gm * (gq + gm));
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o[(3 + c) * kChunk32] = ub[c] * igb;
                o[(6 + c) * kChunk32] = (du[c] * igq - um[c] * corr) * idt;
            }
            o[9 * kChunk32] = 1.0f / gb2;
            if (p.comps > kCompsPlain) {
                double ubd[3] = {__dmul_rn(0.5, __dadd_rn(up[0], un[0])),
                                 __dmul_rn(0.5, __dadd_rn(up[1], un[1])),
                                 __dmul_rn(0.5, __dadd_rn(up[2], un[2]))};
                const double xraw[3] = {xs[sm][0][pp], xs[sm][1][pp], xs[sm][2][pp]};
                o[10 * kChunk32] = __uint_as_float(p.n_sel ? selector_bits(p, xraw, ubd) : 0xffffffffu);
            }
            __syncthreads();
            float* dst = p.slab32 + (tile * p.ring + slot0) * (p.comps * kTileP);
            const int rec = p.comps * kChunk32;          // one particle's record
            if (q * kChunk32 >= b.m0 && q * kChunk32 + kChunk32 - 1 <= b.m1) {
                for (int v = tid; v < rec * kTileP / 4; v += 256) {
                    const int r = v / (rec / 4), w = v - r * (rec / 4);
                    reinterpret_cast<float4*>(dst)[v] =
                        *reinterpret_cast<const float4*>(outs + r * ostride + 4 * w);
                }
            } else if (valid && q == b.c0 && p.slot_major0) {   // this launch's samples only,
                for (int c = 0; c < p.comps; ++c)               // in the chunk's layout
                    dst[(sm * p.comps + c) * kTileP + pp] = outs[pp * ostride + c * kChunk32 + sm];
            } else if (valid) {
                for (int c = 0; c < p.comps; ++c)
                    dst[pp * rec + c * kChunk32 + sm] = outs[pp * ostride + c * kChunk32 + sm];
            }
        }
        if (q == b.c1 && tid < 3 * kTileP && i >= 0) {
            // the launch's last call is the state carried on (staged when other blocks
            // of the launch may still be reading the state arrays)
            const int c = tid >> 3, r = (int)(b.s1 - q * kChunk32);
            const double nn = from_count(sub_count(cnt[c][pp], any ? moved[c][pp] : 0));
            const int64_t k = i - p.first;
            double* sx = p.n_seg > 1 ? p.state_out + c * npart + k : p.x_prev + c * p.ncols + col;
            double* sr = p.n_seg > 1 ? p.state_out + (3 + c) * npart + k : p.r_prev + c * p.ncols + col;
            double* su = p.n_seg > 1 ? p.state_out + (6 + c) * npart + k : p.u_prev + c * p.ncols + col;
            *sx = xs[r][c][pp];
            *sr = nn;
            *su = us[r][c][pp];
        }
        __syncthreads();
        if (any && tid < 3 * kTileP)
            cnt[tid >> 3][pp] = sub_count(cnt[tid >> 3][pp], moved[tid >> 3][pp]);
    }
    if (bad) atomicOr(p.err_word, kErrNaN);
}

IngestKernels ingest_kernel_ptr()
{
    return {{reinterpret_cast<const void*>(&ingest_kernel<0, false>),
             reinterpret_cast<const void*>(&ingest_kernel<1, false>),
             reinterpret_cast<const void*>(&ingest_kernel<0, true>),
             reinterpret_cast<const void*>(&ingest_kernel<1, true>)}};
}

// Tiles of a launch's particles: all columns, or the range's (whole tiles of one species).
static void tile_range(IngestParams& q)
{
    q.tile0 = 0;
    q.n_tiles = (int32_t)(q.ncols / kTileP);
    if (q.count || q.first) {
        const int64_t cnt = q.count ? q.count : q.n_in - q.first;
        int sp = 0;
        while (sp + 1 < q.n_species && q.first >= q.in_off[sp + 1]) ++sp;
        const int64_t col = q.col_off[sp] + (q.first - q.in_off[sp]);
        q.tile0 = col / kTileP;
        q.n_tiles = (int32_t)((col + cnt - 1) / kTileP - q.tile0 + 1);
    }
}

// Batches of calls go through ingest_tile_kernel, a few calls (and sub-cycled samples)
// through ingest_kernel.  A batch costs the tile kernel a round per chunk and 608 tiles (4
// blocks on each SM), also for a chunk it fills in part only, so the shortest batch that pays
// grows with the tiles.  FP32, us per call, tile kernel / ingest_kernel: 8000 particles,
// batches of 16 calls 2.15 / 2.02, 32 1.38 / 1.78; 20,000, 64 2.17 / 1.86, 128 1.80 / 1.78
// (and 0.26 for turning the chunks); from about 40,000 particles on (512 calls 2.79 / 2.38 and
// 0.52; 65,536 4.38 / 3.31 and 0.85) never.  FP64, where ingest_kernel's three reciprocal
// square roots per sample cost most: 65,536, 16 calls 17.8 / 13.2, 32 12.4 / 12.9, 512
// 7.4 / 12.2.  Launches that may not leave slot-major chunks behind take the tile kernel
// from 8 calls on.
bool ingest_batched(const IngestParams& p)
{
    if (p.nsub > 1 || p.n_steps < 8) return false;
    if (p.turned) return true;
    IngestParams q = p;
    tile_range(q);
    const int64_t least = 20 * (int64_t)q.n_tiles / kSegMaxTiles - 12;
    if (!q.slab32) return p.n_steps >= std::min<int64_t>(32, least);
    return p.n_steps >= least && q.n_tiles < 4000;
}

// Slot-major chunks of the FP32 ring to particle-major, in place: a block per tile and chunk,
// through shared memory with rows padded to 33 (no bank conflicts on the way out).  Bound by
// memory: 65,536 particles x 320 samples take 272 us, 1.68 GB at 5.9 TB/s.
__global__ void __launch_bounds__(256) particle_major_kernel(float* slab, int n_tiles, int64_t rchunks,
                                                             int comps, int64_t c0)
{
    __shared__ float buf[kTileP * kCompsPrec * (kChunk32 + 1)];   // [particle][comp][slot], padded
    const int64_t tile = blockIdx.x % n_tiles, c = c0 + blockIdx.x / n_tiles;
    const int rec = comps * kChunk32, n4 = rec * kTileP / 4;
    float4* chunk = reinterpret_cast<float4*>(slab + (tile * rchunks + c % rchunks) * (rec * kTileP));
    for (int v = threadIdx.x; v < n4; v += 256) {
        const float4 a = chunk[v];
        const int q = v >> 1, slot = q / comps, comp = q - slot * comps, p = (v & 1) * 4;
        float* o = buf + (p * comps + comp) * (kChunk32 + 1) + slot;
        const int step = comps * (kChunk32 + 1);
        o[0] = a.x;
        o[step] = a.y;
        o[2 * step] = a.z;
        o[3 * step] = a.w;
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n4; v += 256) {
        const float* i = buf + (v >> 3) * (kChunk32 + 1) + (v & 7) * 4;
        chunk[v] = make_float4(i[0], i[1], i[2], i[3]);
    }
}

cudaError_t particle_major(float* slab, int64_t ncols, int64_t ring, int comps, int64_t c0, int64_t c1,
                           cudaStream_t st)
{
    const int64_t n_tiles = ncols / kTileP, per = std::max<int64_t>(1, (int64_t(1) << 30) / n_tiles);
    for (; c0 <= c1; c0 += per)
        particle_major_kernel<<<(unsigned)(n_tiles * std::min(per, c1 - c0 + 1)), 256, 0, st>>>(
            slab, (int)n_tiles, ring / kChunk32, comps, c0);
    return cudaGetLastError();
}

// A batch of calls through ingest_tile_kernel.
static cudaError_t launch_batch(IngestParams q, int64_t cnt, cudaStream_t st)
{
    const BatchRange b = batch_range(q);
    const int64_t chunks = b.c1 - b.c0 + 1;
    tile_range(q);
    // Time segments (whole chunks) until the launch has about 8 blocks for every SM; from
    // 608 tiles (4 blocks per SM) on the tiles alone do, and the extra pass over x for
    // the image counts costs more than the shorter blocks give.
    q.n_seg = 1;
    q.seg_len = (int32_t)chunks;
    if (q.n_tiles < kSegMaxTiles && q.state_out && (q.wind || !(q.box_L > 0.0))) {
        const int64_t want = std::min<int64_t>(std::min<int64_t>(chunks, 1216 / q.n_tiles + 1), 250);
        q.seg_len = (int32_t)((chunks + want - 1) / want);
        q.n_seg = (int32_t)((chunks + q.seg_len - 1) / q.seg_len);
    }
    if (q.n_seg > 1 && q.box_L > 0.0)
        tile_wind_kernel<<<(unsigned)((int64_t)q.n_tiles * (q.n_seg - 1)), 256, 0, st>>>(q);
    const unsigned blocks = (unsigned)((int64_t)q.n_tiles * q.n_seg);
    const size_t smem = q.slab32 ? (size_t)kTileP * (q.comps * kChunk32 + 4) * sizeof(float)
                                 : (size_t)(kChunk32 + 1) * 3 * kTileP * sizeof(double);
    if (!q.slab32)
        ingest_tile_kernel<2><<<blocks, 256, smem, st>>>(q);
    else if (q.comps >= kCompsPrec)
        ingest_tile_kernel<1><<<blocks, 256, smem, st>>>(q);
    else
        ingest_tile_kernel<0><<<blocks, 256, smem, st>>>(q);
    if (q.n_seg > 1) store_state<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(q);
    return cudaGetLastError();
}

cudaError_t launch_ingest(const IngestParams& p, cudaStream_t st)
{
    const int64_t cnt = p.count ? p.count : p.n_in - p.first;
    if (cnt <= 0 || p.n_steps == 0) return cudaSuccess;
    IngestParams q = p;
    q.n_seg = 1;
    if (ingest_batched(p)) return launch_batch(q, cnt, st);
    // time segments only when the particles alone leave the GPU idle: with
    // 32,768 or more one thread per particle already keeps the FP64 pipes of
    // all SMs busy, and the segments' extra pass only adds work (measured)
    if (p.wind && p.state_out && p.seg_len > 0 && cnt < kSegMaxParticles) {
        // boundaries at calls 1 + j seg_len strictly inside (step0, step0 + n_steps)
        // at most kMaxSeg segments (each thread sums the earlier segments' counts):
        // longer batches get longer segments, still multiples of seg_len
        constexpr int64_t kMaxSeg = 256;
        const int64_t end = p.step0 + p.n_steps;
        int64_t len = p.seg_len;
        const int64_t span = p.n_steps / (kMaxSeg - 1) + 1;
        if (span > len) len = (span + p.seg_len - 1) / p.seg_len * p.seg_len;
        const int64_t j0 = p.step0 < 1 ? 0 : (p.step0 - 1) / len + 1;
        const int64_t first = 1 + j0 * len;
        if (first < end) {
            q.seg_len = (int32_t)len;
            q.seg_first = first;
            q.n_seg = (int32_t)(1 + (end - first + len - 1) / len);
        }
    }
    // one thread per particle, small blocks: the kernel is bound by its FP64
    // work per SM, so the blocks must spread evenly over all 152 SMs (256-thread
    // blocks left 65,536 particles at two blocks on most SMs and one on the rest,
    // and a 16,384-particle share on 64 SMs)
    const int threads = 64;
    if (q.n_seg > 1 && q.box_L > 0.0) {
        const int64_t nw = cnt * (q.n_seg - 1);
        wind_kernel<<<(unsigned)((nw + 255) / 256), 256, 0, st>>>(q);
    }
    const int64_t blocks = (cnt * q.n_seg + threads - 1) / threads;
    const int mode = !q.slab32 ? 2 : (q.comps >= kCompsPrec ? 1 : 0);
    const auto kernel =
        q.nsub > 1 ? (mode == 2 ? ingest_kernel<2, true> : mode == 1 ? ingest_kernel<1, true> : ingest_kernel<0, true>)
                   : (mode == 2 ? ingest_kernel<2, false> : mode == 1 ? ingest_kernel<1, false> : ingest_kernel<0, false>);
    kernel<<<(unsigned)blocks, threads, 0, st>>>(q);
    if (q.n_seg > 1) store_state<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(q);
    return cudaGetLastError();
}

}  // namespace rad
