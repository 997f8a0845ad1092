// common.cuh -- device-side model functions and shared types of the MIUGKS
// CUDA library (arXiv 1704.03151).  Units: R = 1/2, lambda = 1/T, p = rho T / 2;
// 2-D monatomic gas with one internal degree of freedom carried by the reduced
// distributions G (comp 0) and H (comp 1).
#pragma once
#include <cuda_runtime.h>
#include <cooperative_groups.h>
#include <stdint.h>

namespace miugks {

constexpr int kKint = 1;                       // internal degrees of freedom
constexpr double kPi = 3.14159265358979323846;
constexpr int kMaxLevels = 8;
constexpr int kMaxBcs = 64;                    // boundary conditions per solver
constexpr int kMaxLine = 512;                  // longest grid line (cells) of the micro sweep kernels

enum BcType { BC_WALL = 0, BC_SYMMETRY = 1, BC_FARFIELD = 2, BC_OUTFLOW = 3 };

struct BcDev { int type; double rho, u, v, t; };

// velocity space: k = a * nvv + b, u_k = ua[a], v_k = vb[b]
struct VelDev {
    int nu, nvv, nv;
    const double *u, *v, *w;     // per discrete velocity
    const double *ua, *vb;       // per-axis nodes (ascending)
    const double *wa, *wb;       // per-axis weights, w = wa wb
    const float *uf, *vf, *wf;   // u, v, w rounded to FP32 (for the mixed-precision kernels)
    double umax, vmax;           // largest |u|, |v|
    int ld;                      // row stride of per-velocity arrays: nv rounded up to a multiple of 16 (the tables
                                 // u, v, w, uf, vf, wf go on with zeros to ld)
    // per pass (0 forward, 1 backward) and axis: the nodes of that axis that leave
    // through a boundary face on the sweep side (u_n > 0): the first ones of the
    // axis in pass 0, the last ones in pass 1
    int nleave[2][2];
    // wall sums of the line cells (k_line_rho): velocities and weights w u_n (storage type) of the chains' steps
    const int* chain;
    const void* wchain;
};

// one grid level (all device pointers)
struct LevelDev {
    int nx, ny, nc, nfx, nfy;
    const double *xn, *yn, *xc, *yc, *dx, *dy;
    const int *fbx, *fby;        // face BC id, -1 interior (or inactive: no fluid cell on either side)
    const double *rdx, *rdy;     // 1/dx, 1/dy
    const unsigned char* solid;  // per cell: 1 inside a body (no state, never updated)
    const int* ubc;              // fluid cells with a boundary face on the east or north side
    int nubc;
};

// The fluid cell of boundary x-face (axis 0, i in 0..nx) or y-face (axis 1,
// j in 0..ny) and the sign of the face's outward normal seen from it: the face
// lies on the domain edge or between a fluid cell and a body.
__device__ __forceinline__ void bface_side(const LevelDev& L, int axis, int i, int j, int& c, int& outsign)
{
    const int nx = L.nx;
    if (axis == 0) {
        const bool lo = i > 0 && !L.solid[j * nx + i - 1];
        c = lo ? j * nx + i - 1 : j * nx + i;
        outsign = lo ? 1 : -1;
    } else {
        const bool lo = j > 0 && !L.solid[(j - 1) * nx + i];
        c = lo ? (j - 1) * nx + i : j * nx + i;
        outsign = lo ? 1 : -1;
    }
}
// a face without a BC id that does not join two fluid cells (inside a body)
__device__ __forceinline__ bool inactive_face(const LevelDev& L, int axis, int i, int j)
{
    const int nx = L.nx;
    if (axis == 0) return i == 0 || i == nx || L.solid[j * nx + i - 1] || L.solid[j * nx + i];
    return j == 0 || j == L.ny || L.solid[(j - 1) * nx + i] || L.solid[j * nx + i];
}

struct GasDev { double mu_ref, omega, pr; };

// per-velocity nodes and weights in the arithmetic type
template <typename F> struct VelT;
template <> struct VelT<double> {
    static __device__ __forceinline__ const double* u(const VelDev& V) { return V.u; }
    static __device__ __forceinline__ const double* v(const VelDev& V) { return V.v; }
    static __device__ __forceinline__ const double* w(const VelDev& V) { return V.w; }
};
template <> struct VelT<float> {
    static __device__ __forceinline__ const float* u(const VelDev& V) { return V.uf; }
    static __device__ __forceinline__ const float* v(const VelDev& V) { return V.vf; }
    static __device__ __forceinline__ const float* w(const VelDev& V) { return V.wf; }
};


// ---------------------------------------------------------------------------
// gas model
__device__ __forceinline__ void prim4(const double* W, double& rho, double& U, double& V, double& lam)
{
    rho = W[0];
    double ir = 1.0 / W[0];
    U = W[1] * ir;
    V = W[2] * ir;
    double eint = W[3] - 0.5 * (W[1] * U + W[2] * V);
    lam = (kKint + 2) * rho / (4.0 * eint);
}

__device__ __forceinline__ double tau_of(const GasDev& g, double rho, double lam)
{
    double T = 1.0 / lam;
    return g.mu_ref * pow(T, g.omega) / (0.5 * rho * T);
}
// the same in FP32 (mixed-precision face scalars)
__device__ __forceinline__ float tau_of_f(const GasDev& g, float rho, float lam)
{
    float T = 1.0f / lam;
    return (float)g.mu_ref * powf(T, (float)g.omega) / (0.5f * rho * T);
}

// moments dw (already divided by rho) -> slope coefficients of a Maxwellian at (U, V, lam)
template <typename T>
__device__ __forceinline__ void micro_slope_t(const T dw[4], T U, T V, T lam, T a[4])
{
    const T Kp2 = T(kKint + 2.0);
    T c = U * U + V * V + Kp2 / (T(2) * lam);
    T R4 = T(2) * dw[3] - c * dw[0];
    T R3 = dw[2] - V * dw[0];
    T R2 = dw[1] - U * dw[0];
    a[3] = T(4) * lam * lam / Kp2 * (R4 - T(2) * U * R2 - T(2) * V * R3);
    a[2] = T(2) * lam * R3 - V * a[3];
    a[1] = T(2) * lam * R2 - U * a[3];
    a[0] = dw[0] - U * a[1] - V * a[2] - T(0.5) * a[3] * c;
}
__device__ __forceinline__ void micro_slope(const double dw[4], double U, double V, double lam, double a[4])
{
    micro_slope_t<double>(dw, U, V, lam, a);
}

// Reciprocal by one third-order step y <- y + y (e + e^2), e = 1 - x y, from a
// single-precision seed: e is below 2^-22, so the truncation e^3 is below 2^-66
// and the result within 1 ulp of 1/x.  Outside the seed's exponent range (tested
// on the exponent bits: a comparison would take the FP64 pipe twice) the IEEE
// division is used.
__device__ __forceinline__ double rcp64(double x)
{
    const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    if (ex - (1023u - 99u) > 198u) return 1.0 / x;
    float s;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"((float)x));
    const double y = (double)s, e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// ---------------------------------------------------------------------------
// Per-thread accumulator of velocity sums: plain FP64 in the FP64 form, a
// Kahan-compensated FP32 sum in the mixed form (its value is taken in FP64).
template <typename T> struct Acc;
template <> struct Acc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct Acc<float> {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        float y = x - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// ---------------------------------------------------------------------------
// error-free sum of two floats: a + b = s + e
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = a + b;
    float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Sums of N per-thread values over a warp: at every step a lane sends half of its
// values and keeps the other half, so N values take about 1.4 N exchanges instead
// of 5 N.  Afterwards the lane holds the sum of value `which` (none: which >= N).
// FP32 values are float-float pairs throughout.
template <int N>
__device__ __forceinline__ double warp_sums(Acc<double> (&a)[N], int& which)
{
    const int lane = threadIdx.x & 31;
    double v[N];
    #pragma unroll
    for (int q = 0; q < N; ++q) v[q] = a[q].s;
    which = 0;
    int n = N, mine = N;              // slots in use, and how many of this lane's hold a value
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int h = (n + 1) / 2;
        const bool up = n > 1 && (lane & o);             // with one value left: a plain exchange
        #pragma unroll
        for (int q = 0; q < N; ++q) {
            if (q >= h) break;
            const double hi = n == 1 ? v[q] : q + h < n ? v[q + h] : 0.0;
            const double r = __shfl_xor_sync(0xffffffffu, up ? v[q] : hi, o);
            v[q] = (up ? hi : v[q]) + r;
        }
        which += up ? h : 0;
        mine = up ? mine - h : min(mine, h);
        n = h;
    }
    if (mine <= 0) which = N;
    return v[0];
}
template <int N>
__device__ __forceinline__ float2 warp_sums(Acc<float> (&a)[N], int& which)
{
    const int lane = threadIdx.x & 31;
    float vh[N], vl[N];
    #pragma unroll
    for (int q = 0; q < N; ++q) { vh[q] = a[q].s; vl[q] = -a[q].c; }
    which = 0;
    int n = N, mine = N;              // slots in use, and how many of this lane's hold a value
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int h = (n + 1) / 2;
        const bool up = n > 1 && (lane & o);             // with one value left: a plain exchange
        #pragma unroll
        for (int q = 0; q < N; ++q) {
            if (q >= h) break;
            const float th = n == 1 ? vh[q] : q + h < n ? vh[q + h] : 0.0f, tl = n == 1 ? vl[q] : q + h < n ? vl[q + h] : 0.0f;
            const float rh = __shfl_xor_sync(0xffffffffu, up ? vh[q] : th, o), rl = __shfl_xor_sync(0xffffffffu, up ? vl[q] : tl, o);
            float s, e;
            two_sum(up ? th : vh[q], rh, s, e);
            vl[q] = (up ? tl : vl[q]) + rl + e;
            vh[q] = s;
        }
        which += up ? h : 0;
        mine = up ? mine - h : min(mine, h);
        n = h;
    }
    if (mine <= 0) which = N;
    return make_float2(vh[0], vl[0]);
}
// deterministic block reduction of N doubles (fixed tree order); every thread
// receives the result.  scratch: (warps + 1) * N doubles of shared memory.
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double* scratch)
{
    const int warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    Acc<double> a[N];
    #pragma unroll
    for (int q = 0; q < N; ++q) a[q].s = v[q];
    int which;
    const double x = warp_sums<N>(a, which);
    __syncthreads();
    if (which < N) scratch[warp * N + which] = x;        // (lanes with the same value agree)
    __syncthreads();
    // one thread per value adds the warps' sums (an FP64 addition costs a warp as much as 32 of them)
    if (threadIdx.x < N) {
        double t = scratch[threadIdx.x];
        for (int w = 1; w < nw; ++w) t += scratch[w * N + threadIdx.x];
        scratch[nw * N + threadIdx.x] = t;
    }
    __syncthreads();
    #pragma unroll
    for (int q = 0; q < N; ++q) v[q] = scratch[nw * N + q];
    __syncthreads();
}

// Block reduction of per-thread velocity sums into FP64 totals, broadcast to
// every thread.  FP64 form: block_sum.  Mixed form: float-float pairs (error-free
// TwoSum) within the warps and over them, one conversion to FP64 per value at the
// end; at most eight warps.  scratch: (warps + 1) * N doubles.
template <int N>
__device__ __forceinline__ void block_total(Acc<float> (&a)[N], double* scratch, double (&out)[N])
{
    const int warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    float2* fs = reinterpret_cast<float2*>(scratch);
    int which;
    const float2 v = warp_sums<N>(a, which);
    if (which < N) fs[warp * N + which] = v;
    __syncthreads();
    if (threadIdx.x < N) {
        // the warps' pairs (at most eight) as a tree, 4, 2 and 1 apart
        float2 t[8];
        #pragma unroll
        for (int w = 0; w < 8; ++w) t[w] = w < nw ? fs[w * N + threadIdx.x] : make_float2(0.0f, 0.0f);
        #pragma unroll
        for (int o = 4; o > 0; o >>= 1)
            #pragma unroll
            for (int w = 0; w < o; ++w) {
                float s, e;
                two_sum(t[w].x, t[w + o].x, s, e);
                t[w] = make_float2(s, t[w].y + t[w + o].y + e);
            }
        scratch[nw * N + threadIdx.x] = (double)t[0].x + (double)t[0].y;
    }
    __syncthreads();
    #pragma unroll
    for (int q = 0; q < N; ++q) out[q] = scratch[nw * N + q];
    __syncthreads();
}

template <int N>
__device__ __forceinline__ void block_total(Acc<double> (&a)[N], double* scratch, double (&out)[N])
{
    #pragma unroll
    for (int q = 0; q < N; ++q) out[q] = a[q].s;
    block_sum<N>(out, scratch);
}

} // namespace miugks
