// rad_pic.cu -- the small live 2D3V PIC of the two-stream setup (Sec. 2.1)
// that drives the radiation diagnostic in situ (C ABI in include/rad_pic.h).
//
// One step (state x^n, u^{n-1/2}, E^n, B^n):
//   1. push_deposit: one thread per particle gathers E^n, B^n from the
//      staggered Yee points with linear weights, Boris-pushes u to n+1/2,
//      moves x to n+1 and deposits the charge-conserving current of the move
//      (Esirkepov's decomposition for linear shapes on the 3 x 3 nodes the old
//      and new positions share) with FP64 atomics, then wraps x;
//   2. ampere:  E^{n+1} = E^n + dt (curl B^{n+1/2} - J^{n+1/2}), J cleared;
//   3. faraday: B^{n+1} = B^{n+1/2} - dt/2 curl E^{n+1}, and with the same curl
//      B^{n+3/2} = B^{n+1} - dt/2 curl E^{n+1}, kept beside B^{n+1}.
// All fields are updated in place, at fixed addresses: a captured step can be replayed,
// also with direct steps between the replays.
// FP64 throughout (the diagnostic's FP64 parity chain reaches back into the
// particle state); a PIC step costs about 200 FP64 operations per particle,
// which this GPU's FP64 pipe (1/64 of FP32) sustains at about two billion
// particles per second.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstdio>
#include <new>
#include <string>
#include <vector>

#include "rad.h"
#include "rad_internal.cuh"
#include "rad_pic.h"

namespace {

constexpr int kMaxSpecies = 8;

struct PicDev {
    int n;
    double d, inv_d, dt, L;
    const double* E;   // [3][n][n]
    const double* B;
    double* J;
    double* x;         // [3][N]
    double* u;
    int64_t N;
    int n_species;
    int64_t off[kMaxSpecies + 1];
    double hqm[kMaxSpecies];  // q dt / 2 m
    double cx[kMaxSpecies];   // q w / (4 d^2)
    double cyz[kMaxSpecies];  // -q w / (2 d dt)
};

// The two grid points that bracket a coordinate, and the fraction between them, for
// the node points (floor of s) and the half points (floor of s - 1/2): one rounding
// to the nearest node serves both.  s >= 0 and far below 2^31.
struct Bracket {
    int n, h;            // lower node, lower half point (may be -1)
    double nd, fn, fh;   // the lower node as a number, fractions
};
__device__ __forceinline__ Bracket bracket(double s, int n)
{
    constexpr double kMagic = 6755399441055744.0;        // 1.5 * 2^52
    const double t = s + kMagic, rd = t - kMagic;
    const int r = min(max(__double2loint(t), 0), n);     // nearest node (clamped: NaN)
    const double f = s - rd;                             // in [-1/2, 1/2], exact
    const bool below = __double2hiint(f) < 0;
    Bracket b;
    b.n = below ? r - 1 : r;
    b.nd = below ? rd - 1.0 : rd;
    b.fn = s - b.nd;                                     // exact
    b.h = r - 1;
    b.fh = f + 0.5;
    return b;
}

// Weighted sum of the four points around a particle: offsets of the two y rows, z
// columns k0, k1.
__device__ __forceinline__ double interp(const double* __restrict__ F, int j0, int j1, int k0, int k1,
                                         double wy0, double wy1, double wz0, double wz1)
{
    return wy0 * fma(wz1, __ldg(F + j0 + k1), wz0 * __ldg(F + j0 + k0)) +
           wy1 * fma(wz1, __ldg(F + j1 + k1), wz0 * __ldg(F + j1 + k0));
}

__device__ __forceinline__ void add(double* a, double v)
{
    // zero test on the bits: the FP64 compare runs on the pipe that bounds the kernel
    if (((uint32_t)__double2hiint(v) << 1) | (uint32_t)__double2loint(v)) atomicAdd(a, v);
}

// CIC weights before (S0) and after (S1) a move along one axis on the three nodes the
// two supports share (a particle moves less than a cell); returns the first node
// relative to the old lower node (-1 or 0).  f: old fraction, r: new coordinate
// relative to the old lower node, in (-1, 2).
__device__ __forceinline__ int move_weights(double f, double r, double (&S0)[3], double (&S1)[3])
{
    const double g = 1.0 - f;
    const bool down = __double2hiint(r) < 0, up = r >= 1.0;
    const double f1 = down ? r + 1.0 : (up ? r - 1.0 : r), g1 = 1.0 - f1;
    S0[0] = down ? 0.0 : g;
    S0[1] = down ? g : f;
    S0[2] = down ? f : 0.0;
    S1[0] = up ? 0.0 : g1;
    S1[1] = up ? g1 : f1;
    S1[2] = up ? f1 : 0.0;
    return down ? -1 : 0;
}

// One thread per particle.  Bound by the FP64 pipe (1/64 of FP32 here: two lanes per
// clock and SM), so the work is arranged for few FP64 instructions, about 200 per
// particle where the first version had 700: one rounding per axis serves the node and
// half points, one reciprocal square root replaces each square root and its divisions,
// the current is deposited on the 3 x 3 nodes of the move as products of per-axis
// factors (the 4 x 4 form divided by 3 at every node), and sign and zero tests use
// integer instructions.  256 x 256 cells, 1,048,576 particles: 1.41 -> 0.378 ms
// (FP64 pipe 86% busy, 189 FP64 instructions per particle).
__global__ void __launch_bounds__(128) push_deposit(const PicDev p)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= p.N) return;
    int sp = 0;
    while (sp + 1 < p.n_species && i >= p.off[sp + 1]) ++sp;
    const int n = p.n;
    const int64_t N = p.N;
    const int64_t nn = (int64_t)n * n;
    const double x0 = p.x[i], y0 = p.x[N + i], z0 = p.x[2 * N + i];
    double u0 = p.u[i], u1 = p.u[N + i], u2 = p.u[2 * N + i];

    // ---- gather E^n, B^n at (y0, z0)
    const double sy = __dmul_rn(y0, p.inv_d), sz = __dmul_rn(z0, p.inv_d);
    const Bracket by = bracket(sy, n), bz = bracket(sz, n);
    auto wrap = [&](int a) { return a < 0 ? a + n : (a >= n ? a - n : a); };
    // rows and columns in [-1, n] before wrapping (y0, z0 in [0, L], rounding included)
    const int jn0 = wrap(by.n) * n, jn1 = wrap(by.n + 1) * n;
    const int jh0 = wrap(by.h) * n, jh1 = wrap(by.h + 1) * n;
    const int kn0 = wrap(bz.n), kn1 = wrap(bz.n + 1), kh0 = wrap(bz.h), kh1 = wrap(bz.h + 1);
    const double gyn = 1.0 - by.fn, gyh = 1.0 - by.fh, gzn = 1.0 - bz.fn, gzh = 1.0 - bz.fh;
    const double Ex = interp(p.E, jn0, jn1, kn0, kn1, gyn, by.fn, gzn, bz.fn);
    const double Ey = interp(p.E + nn, jh0, jh1, kn0, kn1, gyh, by.fh, gzn, bz.fn);
    const double Ez = interp(p.E + 2 * nn, jn0, jn1, kh0, kh1, gyn, by.fn, gzh, bz.fh);
    const double Bx = interp(p.B, jh0, jh1, kh0, kh1, gyh, by.fh, gzh, bz.fh);
    const double By = interp(p.B + nn, jn0, jn1, kh0, kh1, gyn, by.fn, gzh, bz.fh);
    const double Bz = interp(p.B + 2 * nn, jh0, jh1, kn0, kn1, gyh, by.fh, gzn, bz.fn);

    // ---- relativistic Boris
    const double h = p.hqm[sp];
    const double m0 = fma(h, Ex, u0), m1 = fma(h, Ey, u1), m2 = fma(h, Ez, u2);
    const double hg = h * rsqrt(fma(m0, m0, fma(m1, m1, fma(m2, m2, 1.0))));
    const double t0 = hg * Bx, t1 = hg * By, t2 = hg * Bz;
    const double tt = 2.0 / fma(t0, t0, fma(t1, t1, fma(t2, t2, 1.0)));
    const double p0 = m0 + fma(m1, t2, -(m2 * t1)), p1 = m1 + fma(m2, t0, -(m0 * t2)),
                 p2 = m2 + fma(m0, t1, -(m1 * t0));
    const double q0 = fma(tt, fma(p1, t2, -(p2 * t1)), m0), q1 = fma(tt, fma(p2, t0, -(p0 * t2)), m1),
                 q2 = fma(tt, fma(p0, t1, -(p1 * t0)), m2);
    u0 = fma(h, Ex, q0);
    u1 = fma(h, Ey, q1);
    u2 = fma(h, Ez, q2);
    const double ig = rsqrt(fma(u0, u0, fma(u1, u1, fma(u2, u2, 1.0))));
    const double v0 = u0 * ig, v1 = u1 * ig, v2 = u2 * ig;
    const double x1 = fma(p.dt, v0, x0), y1 = fma(p.dt, v1, y0), z1 = fma(p.dt, v2, z0);

    // ---- charge-conserving current of the move (y0, z0) -> (y1, z1): with S = (S0 + S1) / 2
    // and dS = S1 - S0 per axis, W_x = S_y S_z + dS_y dS_z / 12, and the y (z) current
    // is the running sum of dS_y (dS_z) times the other axis' S
    {
        double ay[3], az[3], dy[3], dz[3];
        // (the new coordinates relative to the old lower nodes are exact differences of
        // the scaled positions the next step starts from: the charge density implied by
        // this step's S1 and the next one's S0 is the same)
        const int ly = move_weights(by.fn, __dmul_rn(y1, p.inv_d) - by.nd, ay, dy);
        const int lz = move_weights(bz.fn, __dmul_rn(z1, p.inv_d) - bz.nd, az, dz);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double sy_ = ay[a] + dy[a], sz_ = az[a] + dz[a];
            dy[a] -= ay[a];
            dz[a] -= az[a];
            ay[a] = sy_;                                 // S0 + S1 (halves in the factors)
            az[a] = sz_;
        }
        const double cx = p.cx[sp] * v0, c12 = cx * (1.0 / 3.0);   // q w v_x / (4 d^2), and / 3
        const double cyz = p.cyz[sp];                    // -q w / (2 d dt)
        double cy[3], cz[3];
        cy[0] = cyz * dy[0];
        cy[1] = fma(cyz, dy[1], cy[0]);
        cz[0] = cyz * dz[0];
        cz[1] = fma(cyz, dz[1], cz[0]);
        int j[3], k[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            j[a] = wrap(by.n + ly + a) * n;
            k[a] = wrap(bz.n + lz + a);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double fa = cx * ay[a], fd = c12 * dy[a];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                double* Jc = p.J + j[a] + k[b];
                add(Jc, fma(fa, az[b], fd * dz[b]));
                if (a < 2) add(Jc + nn, cy[a] * az[b]);
                if (b < 2) add(Jc + 2 * nn, cz[b] * ay[a]);
            }
        }
    }

    // ---- wrap into [0, L) and store
    auto wrapL = [&](double c) {
        return __double2hiint(c) < 0 ? c + p.L : (c >= p.L ? c - p.L : c);
    };
    p.x[i] = wrapL(x1);
    p.x[N + i] = wrapL(y1);
    p.x[2 * N + i] = wrapL(z1);
    p.u[i] = u0;
    p.u[N + i] = u1;
    p.u[2 * N + i] = u2;
}

// One component of curl F at cell q = (j, k) by forward differences (d/dx = 0): jp, kp
// the offsets of the next row and column.
__device__ __forceinline__ double curl_fwd(const double* __restrict__ F, int64_t nn, int c, int64_t q,
                                           int64_t qjp, int64_t qkp, double inv_d)
{
    if (c == 0) return (F[2 * nn + qjp] - F[2 * nn + q]) * inv_d - (F[nn + qkp] - F[nn + q]) * inv_d;
    if (c == 1) return (F[qkp] - F[q]) * inv_d;
    return -(F[qjp] - F[q]) * inv_d;
}

// E += dt (curl Bh - J) with Bh the magnetic field at the half step; J is left at zero for
// the next step's deposit.
__global__ void ampere(double* __restrict__ E, const double* __restrict__ Bh, double* __restrict__ J,
                       int n, double inv_d, double dt)
{
    const int64_t nn = (int64_t)n * n;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nn;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(q / n), k = (int)(q - (int64_t)j * n);
        const int64_t qjm = j == 0 ? q + nn - n : q - n, qkm = k == 0 ? q + n - 1 : q - 1;
        const double bx = Bh[q], by = Bh[nn + q], bz = Bh[2 * nn + q];
        const double bxj = Bh[qjm], bxk = Bh[qkm], byk = Bh[nn + qkm], bzj = Bh[2 * nn + qjm];
        E[q] = E[q] + dt * ((bz - bzj) * inv_d - (by - byk) * inv_d - J[q]);
        E[nn + q] = E[nn + q] + dt * ((bx - bxk) * inv_d - J[nn + q]);
        E[2 * nn + q] = E[2 * nn + q] + dt * (-(bx - bxj) * inv_d - J[2 * nn + q]);
        J[q] = J[nn + q] = J[2 * nn + q] = 0.0;
    }
}

// With c = dt / 2 and the new E: B = Bh - c curl E (the second half of this step), then
// Bh = B - c curl E (the first half of the next one, which starts from the same E).
__global__ void faraday(const double* __restrict__ E, double* __restrict__ B, double* __restrict__ Bh,
                        int n, double inv_d, double c)
{
    const int64_t nn = (int64_t)n * n;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nn;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(q / n), k = (int)(q - (int64_t)j * n);
        const int64_t qjp = j + 1 == n ? q + n - nn : q + n, qkp = k + 1 == n ? q + 1 - n : q + 1;
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            const double r = curl_fwd(E, nn, comp, q, qjp, qkp, inv_d);
            const double b = Bh[comp * nn + q] - c * r;
            B[comp * nn + q] = b;
            Bh[comp * nn + q] = b - c * r;
        }
    }
}

// Bh = B - c curl E of fields that were set from outside.
__global__ void half_step(const double* __restrict__ E, const double* __restrict__ B,
                          double* __restrict__ Bh, int n, double inv_d, double c)
{
    const int64_t nn = (int64_t)n * n;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nn;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(q / n), k = (int)(q - (int64_t)j * n);
        const int64_t qjp = j + 1 == n ? q + n - nn : q + n, qkp = k + 1 == n ? q + 1 - n : q + 1;
#pragma unroll
        for (int comp = 0; comp < 3; ++comp)
            Bh[comp * nn + q] = B[comp * nn + q] - c * curl_fwd(E, nn, comp, q, qjp, qkp, inv_d);
    }
}

// Positions into [0, L) (init: the kernels' index arithmetic relies on it; the
// push keeps it, moving particles by under one cell per step).
__global__ void wrap_positions(double* x, int64_t n3, double L)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n3;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double v = x[i];
        double w = v - L * floor(v / L);
        if (!(w >= 0.0 && w < L)) w = 0.0;    // non-finite input, or rounding up to L
        x[i] = w;
    }
}

__global__ void gather_range(const double* __restrict__ x, const double* __restrict__ u, int64_t N,
                             int64_t first, int64_t count, double* __restrict__ xo,
                             double* __restrict__ uo)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xo[c * count + i] = x[c * N + first + i];
            uo[c * count + i] = u[c * N + first + i];
        }
    }
}

// out[0] += sum (E^2 + B^2)/2 d^2, out[1] += sum w m (gamma - 1)
__global__ void energy_kernel(const PicDev p, const double* __restrict__ mw, double* out)
{
    const int64_t nn = (int64_t)p.n * p.n;
    double ef = 0.0, ek = 0.0;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < 3 * nn;
         q += (int64_t)gridDim.x * blockDim.x)
        ef += 0.5 * (p.E[q] * p.E[q] + p.B[q] * p.B[q]) * p.d * p.d;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < p.N;
         i += (int64_t)gridDim.x * blockDim.x) {
        int sp = 0;
        while (sp + 1 < p.n_species && i >= p.off[sp + 1]) ++sp;
        const double a = p.u[i], b = p.u[p.N + i], c = p.u[2 * p.N + i];
        ek += mw[sp] * (sqrt(1.0 + (a * a + b * b + c * c)) - 1.0);
    }
    for (int o = 16; o > 0; o >>= 1) {
        ef += __shfl_down_sync(0xffffffffu, ef, o);
        ek += __shfl_down_sync(0xffffffffu, ek, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(out, ef);
        atomicAdd(out + 1, ek);
    }
}

int grid_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 4096); }

bool is_dev(const void* ptr)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

struct rad_pic {
    PicDev dev{};
    double* E = nullptr;
    double* B = nullptr;
    double* Bh = nullptr;       // B half a step on (B - dt/2 curl E)
    double* J = nullptr;
    double* x = nullptr;
    double* u = nullptr;
    double* mw = nullptr;       // per-species m w (device)
    double* en = nullptr;       // energy accumulators (device)
    double* xt = nullptr;       // staging for the tracked particles
    double* ut = nullptr;
    int64_t staged = 0;
    int64_t steps = 0;
    cudaEvent_t staged_ev = nullptr;   // staging buffers written (PIC stream)
    cudaEvent_t read_ev = nullptr;     // staging buffers read (radiation stream)
    cudaStream_t side = nullptr;       // field updates of a coupled run on one stream
    cudaEvent_t pushed_ev = nullptr;   // the push before them
    cudaEvent_t fields_ev = nullptr;   // their end
    cudaStream_t st = nullptr;
    std::string err;
};

static int pfail(rad_pic* p, int rc, const std::string& what, cudaError_t e = cudaSuccess)
{
    if (p) p->err = e != cudaSuccess ? what + ": " + cudaGetErrorString(e) : what;
    return rc;
}

#define PCU(call)                                                        \
    do {                                                                 \
        const cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return pfail(p, RAD_PIC_ECUDA, #call, e_); \
    } while (0)

static int pic_push(rad_pic* p)
{
    if (p->dev.N > 0) push_deposit<<<(unsigned)((p->dev.N + 127) / 128), 128, 0, p->st>>>(p->dev);
    PCU(cudaGetLastError());
    return RAD_PIC_OK;
}

// The rest of the step, from the currents that pic_push() deposited.
static int pic_fields(rad_pic* p, cudaStream_t st)
{
    const int64_t nn = (int64_t)p->dev.n * p->dev.n;
    const double inv_d = p->dev.inv_d, dt = p->dev.dt;
    const unsigned cells = (unsigned)((nn + 127) / 128);
    ampere<<<cells, 128, 0, st>>>(p->E, p->Bh, p->J, p->dev.n, inv_d, dt);
    faraday<<<cells, 128, 0, st>>>(p->E, p->B, p->Bh, p->dev.n, inv_d, 0.5 * dt);
    PCU(cudaGetLastError());
    ++p->steps;
    return RAD_PIC_OK;
}

extern "C" {

int rad_pic_init(rad_pic** out, int32_t n, double d, double dt, const rad_pic_species* sp,
                 int32_t n_species, const double* x, const double* u, void* cuda_stream)
{
    if (!out) return RAD_PIC_EINVAL;
    *out = nullptr;
    if (n < 4 || n > 16384 || !(d > 0.0) || !(dt > 0.0) || !std::isfinite(d) ||
        !std::isfinite(dt) || !(dt < d / std::sqrt(2.0)) ||
        n_species < 0 || n_species > kMaxSpecies || (n_species > 0 && !sp))
        return RAD_PIC_EINVAL;
    int64_t N = 0;
    for (int s = 0; s < n_species; ++s) {
        if (sp[s].count < 0 || !(sp[s].mass > 0.0) || !std::isfinite(sp[s].charge) ||
            !std::isfinite(sp[s].weight))
            return RAD_PIC_EINVAL;
        N += sp[s].count;
    }
    if (N > 0 && (!x || !u)) return RAD_PIC_EINVAL;
    rad_pic* p = new (std::nothrow) rad_pic();
    if (!p) return RAD_PIC_ENOMEM;
    p->st = (cudaStream_t)cuda_stream;
    const int64_t nn = (int64_t)n * n;
    auto bail = [&](int rc) {
        rad_pic_destroy(p);
        return rc;
    };
#define PMAL(ptr, bytes)                                                              \
    do {                                                                              \
        if (cudaMalloc(&(ptr), (bytes) > 0 ? (bytes) : 8) != cudaSuccess) {           \
            cudaGetLastError();                                                       \
            return bail(RAD_PIC_ENOMEM);                                              \
        }                                                                             \
    } while (0)
    PMAL(p->E, 3 * nn * sizeof(double));
    PMAL(p->B, 3 * nn * sizeof(double));
    PMAL(p->Bh, 3 * nn * sizeof(double));
    PMAL(p->J, 3 * nn * sizeof(double));
    PMAL(p->x, 3 * N * sizeof(double));
    PMAL(p->u, 3 * N * sizeof(double));
    PMAL(p->mw, kMaxSpecies * sizeof(double));
    PMAL(p->en, 2 * sizeof(double));
#undef PMAL
    if (cudaMemset(p->E, 0, 3 * nn * sizeof(double)) != cudaSuccess ||
        cudaMemset(p->B, 0, 3 * nn * sizeof(double)) != cudaSuccess ||
        cudaMemset(p->Bh, 0, 3 * nn * sizeof(double)) != cudaSuccess ||
        cudaMemset(p->J, 0, 3 * nn * sizeof(double)) != cudaSuccess ||
        (N > 0 && (cudaMemcpy(p->x, x, 3 * N * sizeof(double), cudaMemcpyDefault) != cudaSuccess ||
                   cudaMemcpy(p->u, u, 3 * N * sizeof(double), cudaMemcpyDefault) != cudaSuccess)))
        return bail(RAD_PIC_ECUDA);
    PicDev& D = p->dev;
    D.n = n;
    D.d = d;
    D.inv_d = 1.0 / d;
    D.dt = dt;
    D.L = n * d;
    D.E = p->E;
    D.B = p->B;
    D.J = p->J;
    D.x = p->x;
    D.u = p->u;
    D.N = N;
    D.n_species = n_species;
    double mw[kMaxSpecies] = {0};
    D.off[0] = 0;
    for (int s = 0; s < n_species; ++s) {
        D.off[s + 1] = D.off[s] + sp[s].count;
        D.hqm[s] = 0.5 * (sp[s].charge / sp[s].mass) * dt;
        D.cx[s] = 0.25 * sp[s].charge * sp[s].weight / (d * d);
        D.cyz[s] = -0.5 * sp[s].charge * sp[s].weight / (d * dt);
        mw[s] = sp[s].mass * sp[s].weight;
    }
    if (cudaMemcpy(p->mw, mw, sizeof mw, cudaMemcpyHostToDevice) != cudaSuccess)
        return bail(RAD_PIC_ECUDA);
    if (N > 0) {
        wrap_positions<<<grid_for(3 * N), 256>>>(p->x, 3 * N, D.L);
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
            return bail(RAD_PIC_ECUDA);
    }
    *out = p;
    return RAD_PIC_OK;
}

int rad_pic_set_fields(rad_pic* p, const double* E, const double* B)
{
    if (!p) return RAD_PIC_EINVAL;
    const size_t bytes = 3 * (size_t)p->dev.n * p->dev.n * sizeof(double);
    if (E) PCU(cudaMemcpyAsync(p->E, E, bytes, cudaMemcpyDefault, p->st));
    if (B) PCU(cudaMemcpyAsync(p->B, B, bytes, cudaMemcpyDefault, p->st));
    half_step<<<grid_for((int64_t)p->dev.n * p->dev.n), 256, 0, p->st>>>(
        p->E, p->B, p->Bh, p->dev.n, p->dev.inv_d, 0.5 * p->dev.dt);
    PCU(cudaGetLastError());
    PCU(cudaStreamSynchronize(p->st));
    return RAD_PIC_OK;
}

int rad_pic_get_fields(rad_pic* p, double* E, double* B)
{
    if (!p) return RAD_PIC_EINVAL;
    const size_t bytes = 3 * (size_t)p->dev.n * p->dev.n * sizeof(double);
    if (E) PCU(cudaMemcpyAsync(E, p->E, bytes, cudaMemcpyDefault, p->st));
    if (B) PCU(cudaMemcpyAsync(B, p->B, bytes, cudaMemcpyDefault, p->st));
    PCU(cudaStreamSynchronize(p->st));
    return RAD_PIC_OK;
}

int rad_pic_get_particles(rad_pic* p, double* x, double* u)
{
    if (!p) return RAD_PIC_EINVAL;
    const size_t bytes = 3 * (size_t)p->dev.N * sizeof(double);
    if (x && bytes) PCU(cudaMemcpyAsync(x, p->x, bytes, cudaMemcpyDefault, p->st));
    if (u && bytes) PCU(cudaMemcpyAsync(u, p->u, bytes, cudaMemcpyDefault, p->st));
    PCU(cudaStreamSynchronize(p->st));
    return RAD_PIC_OK;
}

int rad_pic_step(rad_pic* p, int32_t n_steps)
{
    if (!p || n_steps < 0) return pfail(p, RAD_PIC_EINVAL, "rad_pic_step: bad arguments");
    for (int32_t s = 0; s < n_steps; ++s) {
        int rc = pic_push(p);
        if (!rc) rc = pic_fields(p, p->st);
        if (rc) return rc;
    }
    return RAD_PIC_OK;
}

int64_t rad_pic_steps_done(const rad_pic* p) { return p ? p->steps : -1; }

int rad_pic_tracked(rad_pic* p, int64_t first, int64_t count, double* x_out, double* u_out)
{
    if (!p || first < 0 || count < 0 || first + count > p->dev.N || !x_out || !u_out ||
        !is_dev(x_out) || !is_dev(u_out))
        return pfail(p, RAD_PIC_EINVAL, "rad_pic_tracked: range or device buffers");
    if (count == 0) return RAD_PIC_OK;
    gather_range<<<grid_for(count), 256, 0, p->st>>>(p->x, p->u, p->dev.N, first, count, x_out, u_out);
    PCU(cudaGetLastError());
    return RAD_PIC_OK;
}

int rad_pic_run_coupled(rad_pic* p, rad_ctx* r, int64_t first, int64_t count, int32_t n_steps)
{
    if (!p || !r || n_steps < 0 || first < 0 || count < 1 || first + count > p->dev.N)
        return pfail(p, RAD_PIC_EINVAL, "rad_pic_run_coupled: bad arguments");
    if (rad::ctx_particles(r) != count)
        return pfail(p, RAD_PIC_EINVAL, "rad_pic_run_coupled: count differs from the radiation "
                                        "context's particle count");
    // the radiation context may order its work on another stream: its reads of
    // the staging buffers wait for the gather, and the next gather waits for
    // those reads
    const cudaStream_t rs = rad::ctx_stream(r);
    const bool other = rs != p->st;
    if (other) {
        if (p->staged < count) {
            if (p->xt) cudaFree(p->xt);
            if (p->ut) cudaFree(p->ut);
            p->xt = p->ut = nullptr;
            p->staged = 0;
            if (cudaMalloc(&p->xt, 3 * count * sizeof(double)) != cudaSuccess ||
                cudaMalloc(&p->ut, 3 * count * sizeof(double)) != cudaSuccess) {
                cudaGetLastError();
                return pfail(p, RAD_PIC_ENOMEM, "rad_pic_run_coupled: staging buffers");
            }
            p->staged = count;
        }
        if (!p->staged_ev) {
            PCU(cudaEventCreateWithFlags(&p->staged_ev, cudaEventDisableTiming));
            PCU(cudaEventCreateWithFlags(&p->read_ev, cudaEventDisableTiming));
        }
    }
    auto hand_over = [&]() -> int {
        // a state the context has already received (the final state of a previous run)
        if (rad::ctx_next_step(r) == p->steps + 1) return RAD_PIC_OK;
        if (!other) {
            // one stream: the ingest reads the particle arrays in place (particle stride
            // N), in order before the push that changes them
            const int rc = rad::ctx_accumulate_strided(r, p->steps, p->x + first, p->u + first, p->dev.N);
            if (rc != RAD_OK) return pfail(p, RAD_PIC_ERAD, std::string("rad_accumulate: ") + rad_last_error(r));
            return RAD_PIC_OK;
        }
        PCU(cudaStreamWaitEvent(p->st, p->read_ev, 0));
        gather_range<<<grid_for(count), 256, 0, p->st>>>(p->x, p->u, p->dev.N, first, count, p->xt,
                                                         p->ut);
        PCU(cudaGetLastError());
        PCU(cudaEventRecord(p->staged_ev, p->st));
        PCU(cudaStreamWaitEvent(rs, p->staged_ev, 0));
        const int rc = rad_accumulate(r, p->steps, p->xt, p->ut);
        if (rc != RAD_OK) return pfail(p, RAD_PIC_ERAD, std::string("rad_accumulate: ") + rad_last_error(r));
        PCU(cudaEventRecord(p->read_ev, rs));
        return RAD_PIC_OK;
    };
    // On one stream the field update runs beside the hand-over of the state that the push
    // has just made (neither touches what the other reads or writes; each is far too small
    // to fill the GPU): 65,536 particles with 4096 tracked take 51 us per step instead
    // of 57.  A stream under capture is left in one piece.
    bool fork = false;
    if (!other && n_steps > 0) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        PCU(cudaStreamIsCapturing(p->st, &cap));
        fork = cap == cudaStreamCaptureStatusNone;
        if (fork && !p->side) {
            PCU(cudaStreamCreateWithFlags(&p->side, cudaStreamNonBlocking));
            PCU(cudaEventCreateWithFlags(&p->pushed_ev, cudaEventDisableTiming));
            PCU(cudaEventCreateWithFlags(&p->fields_ev, cudaEventDisableTiming));
        }
    }
    auto step = [&]() -> int {
        int rc = pic_push(p);
        if (rc || !fork) return rc ? rc : pic_fields(p, p->st);
        PCU(cudaEventRecord(p->pushed_ev, p->st));
        PCU(cudaStreamWaitEvent(p->side, p->pushed_ev, 0));
        rc = pic_fields(p, p->side);
        PCU(cudaEventRecord(p->fields_ev, p->side));
        return rc;
    };
    // the next push, and whatever the caller does next, comes after the fields
    auto join = [&](int rc) -> int {
        if (fork) PCU(cudaStreamWaitEvent(p->st, p->fields_ev, 0));
        return rc;
    };
    int rc = hand_over();
    for (int32_t s = 0; s < n_steps && !rc; ++s) {
        rc = step();
        if (!rc) rc = hand_over();
        rc = join(rc);
    }
    return rc;
}

int rad_pic_energy(rad_pic* p, double* field, double* kinetic)
{
    if (!p) return RAD_PIC_EINVAL;
    PCU(cudaMemsetAsync(p->en, 0, 2 * sizeof(double), p->st));
    energy_kernel<<<grid_for(std::max<int64_t>(p->dev.N, 3 * (int64_t)p->dev.n * p->dev.n)), 256, 0,
                    p->st>>>(p->dev, p->mw, p->en);
    PCU(cudaGetLastError());
    double h[2];
    PCU(cudaMemcpyAsync(h, p->en, sizeof h, cudaMemcpyDeviceToHost, p->st));
    PCU(cudaStreamSynchronize(p->st));
    if (field) *field = h[0];
    if (kinetic) *kinetic = h[1];
    return RAD_PIC_OK;
}

const char* rad_pic_last_error(const rad_pic* p) { return p ? p->err.c_str() : "null context"; }

void rad_pic_destroy(rad_pic* p)
{
    if (!p) return;
    if (p->st) cudaStreamSynchronize(p->st);
    for (double* q : {p->E, p->B, p->Bh, p->J, p->x, p->u, p->mw, p->en, p->xt, p->ut})
        if (q) cudaFree(q);
    if (p->staged_ev) cudaEventDestroy(p->staged_ev);
    if (p->read_ev) cudaEventDestroy(p->read_ev);
    if (p->pushed_ev) cudaEventDestroy(p->pushed_ev);
    if (p->fields_ev) cudaEventDestroy(p->fields_ev);
    if (p->side) cudaStreamDestroy(p->side);
    delete p;
}

}  // extern "C"
