// flux.cu -- Step 1 of the MIUGKS iteration (arXiv 1704.03151, Sec. 2.1):
// time-averaged UGKS interface fluxes of every discrete velocity (Eqs.
// macroResidualCalc, microResidualDef) and the macroscopic residual R
// (Eq. macroResidualDef), plus its RMS (Eq. Residual_Def).
//
// One CTA per face; a thread keeps one velocity of the second axis and strides
// over the first, so every load of f is coalesced and whatever depends on the
// second axis only stays in registers.  Two passes over the velocities: the
// first reconstructs the face values and takes their moments, the second forms
// the flux and its moments.
#include "kernels.cuh"
#include <algorithm>
#include <type_traits>

namespace miugks {

__constant__ double c_series[5][28];   // power-series coefficients of the time integrals
__constant__ float c_series_f[5][28];  // the same rounded to FP32

void upload_series_coefficients()
{
    // q1/dt  = sum_{n>=1} (-1)^{n+1} x^n/(n+1)!
    // q2/dt2 = sum_{n>=1} (-1)^n n x^n/(n+2)!
    // q3/dt2 = sum_{n>=1} (-1)^{n+1} x^n/(n+2)!
    // q4/dt  = sum_{n>=0} (-1)^n x^n/(n+1)!
    // q5/dt2 = sum_{n>=0} (-1)^{n+1} (n+1) x^n/(n+2)!
    double c[5][28] = {};
    double fact[32];
    fact[0] = 1.0;
    for (int n = 1; n < 32; ++n) fact[n] = fact[n - 1] * n;
    for (int n = 0; n < 28; ++n) {
        double s = (n % 2) ? -1.0 : 1.0;                 // (-1)^n
        c[0][n] = n >= 1 ? -s / fact[n + 1] : 0.0;
        c[1][n] = n >= 1 ? s * n / fact[n + 2] : 0.0;
        c[2][n] = n >= 1 ? -s / fact[n + 2] : 0.0;
        c[3][n] = s / fact[n + 1];
        c[4][n] = -s * (n + 1) / fact[n + 2];
    }
    cudaMemcpyToSymbol(c_series, c, sizeof c);
    float cf[5][28];
    for (int m = 0; m < 5; ++m)
        for (int n = 0; n < 28; ++n) cf[m][n] = (float)c[m][n];
    cudaMemcpyToSymbol(c_series_f, cf, sizeof cf);
}

// one of the five time integrals (series below x = dt/tau = 1, closed form above)
__device__ __forceinline__ double time_coeff_one(double dt, double tau, int m)
{
    double x = dt / tau;
    if (x < 1.0) {
        double acc = c_series[m][27];
        #pragma unroll
        for (int n = 26; n >= 0; --n) acc = fma(acc, x, c_series[m][n]);
        return (m == 0 || m == 3) ? dt * acc : dt * dt * acc;
    }
    double e = exp(-x), E1 = -expm1(-x);
    switch (m) {
    case 0: return dt - tau * E1;
    case 1: return -tau * dt * (1.0 + e) + 2.0 * tau * tau * E1;
    case 2: return 0.5 * dt * dt - tau * dt + tau * tau * E1;
    case 3: return tau * E1;
    default: return tau * dt * e - tau * tau * E1;
    }
}

// FP32 form of time_coeff_one (mixed-precision face scalars)
__device__ __forceinline__ float time_coeff_one_f(float dt, float tau, int m)
{
    float x = dt / tau;
    if (x < 1.0f) {
        float acc = c_series_f[m][27];
        #pragma unroll
        for (int n = 26; n >= 0; --n) acc = fmaf(acc, x, c_series_f[m][n]);
        return (m == 0 || m == 3) ? dt * acc : dt * dt * acc;
    }
    float e = expf(-x), E1 = -expm1f(-x);
    switch (m) {
    case 0: return dt - tau * E1;
    case 1: return -tau * dt * (1.0f + e) + 2.0f * tau * tau * E1;
    case 2: return 0.5f * dt * dt - tau * dt + tau * tau * E1;
    case 3: return tau * E1;
    default: return tau * dt * e - tau * tau * E1;
    }
}

// van Leer limited slope 2 s1 s2 / (s1 + s2) when s1 s2 > 0, else 0
__device__ __forceinline__ double vl_limited(double s1, double s2)
{
    const double p = s1 * s2;      // (the sign is looked at in the bits: a comparison would take the FP64 pipe)
    return __double_as_longlong(p) > 0 ? (p + p) * rcp64(s1 + s2) : 0.0;
}
__device__ __forceinline__ float vl_limited(float s1, float s2)
{
    float p = s1 * s2;   // s1 + s2 has no cancellation here; the fast quotient is within 2 ulp
    return p > 0.0f ? __fdividef(2.0f * p, s1 + s2) : 0.0f;
}

// Sums over the block: out[q] in shared memory, valid after the caller's next barrier
template <int N>
__device__ __forceinline__ void block_sums(Acc<double> (&a)[N], double* scratch, double* out)
{
    int which;
    const double v = warp_sums<N>(a, which);
    const int warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if (which < N) scratch[warp * N + which] = v;        // (lanes with the same value agree)
    __syncthreads();
    if (threadIdx.x < N) {
        double t = scratch[threadIdx.x];
        for (int w = 1; w < nw; ++w) t += scratch[w * N + threadIdx.x];
        out[threadIdx.x] = t;
    }
}
template <int N>
__device__ __forceinline__ void block_sums(Acc<float> (&a)[N], double* scratch, double* out)
{
    int which;
    const float2 v = warp_sums<N>(a, which);
    float2* fs = reinterpret_cast<float2*>(scratch);
    const int warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if (which < N) fs[warp * N + which] = v;
    __syncthreads();
    if (threadIdx.x < N) {
        float2 t = fs[threadIdx.x];
        for (int w = 1; w < nw; ++w) {
            const float2 r = fs[w * N + threadIdx.x];
            float s, e;
            two_sum(t.x, r.x, s, e);
            t = make_float2(s, t.y + r.y + e);
        }
        out[threadIdx.x] = (double)t.x + (double)t.y;
    }
}

// Constants of the flux per node of the velocity axis normal to the face, and per
// node of the tangential axis (k_face_flux, second pass)
template <typename F> struct alignas(16) NormalNode { F un, E, P, C, Z, hZ, xZ, Fq, S, q5u; };
template <typename F> struct alignas(16) TangentNode { F ut, h, E, Fq, S; };   // h = u_t / 2

// Per-velocity arithmetic runs in F (FP64, or FP32 in the mixed form); the
// velocity sums are FP64 (or Kahan-compensated FP32) per thread and combined in
// FP64; the per-face scalars (interface state, slopes, time integrals) are FP64.
//
// What is done per velocity is kept small, since the kernel is bound by the issue
// of its arithmetic (FP64: two lanes per clock and SM):
//   * only the upwind side of a velocity is reconstructed (three cells of the
//     four), with mirrored constants for the velocities that come from above;
//   * the heat flux needs no pass of its own: it follows from moments about the
//     mean velocity of the two cells, taken with the face values (about that
//     velocity, not about zero, so that nothing cancels in a fast flow);
//   * the compatibility sums of the equilibrium's slopes, sum w u_n psi (a.psi) g,
//     are products of one-axis sums, because g, w and the powers of u and v
//     separate: nu + nv terms by one warp instead of nu nv by all;
//   * the equilibrium part of the flux is g times a polynomial whose coefficients
//     depend on one axis each (NormalNode, TangentNode).
// CACHE keeps the face values and slopes of every velocity in shared memory
// between the passes; without it (a velocity grid too large for shared memory)
// the second pass reconstructs again.
// Per launch against three passes that reconstructed both sides of every velocity:
// square cylinder (89x89) mixed 4.3 -> 2.1 ms, flat plate (48x48) mixed 0.73 ->
// 0.51 ms, FP64 13.1 -> 4.8 ms, 64x64 cavity (32x32) mixed 131 -> 103 us, FP64 1.92
// -> 0.72 ms, square cylinder at half size FP64 21.4 -> 10.1 ms.
template <typename F, bool CACHE>
__global__ void __launch_bounds__(256, sizeof(F) == 4 ? 4 : 2) k_face_flux(FaceFluxArgs<F> A)
{
    extern __shared__ double sm[];
    const LevelDev& L = A.L;
    const VelDev& Vg = A.V;
    const int nv = Vg.nv, nu = Vg.nu, nvv = Vg.nvv, tid = threadIdx.x, bs = blockDim.x;
    const size_t ld = Vg.ld;
    const int axis = A.axis, fi = blockIdx.x;
    const int nx = L.nx, ny = L.ny;
    const size_t nc = L.nc, nf = axis == 0 ? L.nfx : L.nfy;
    double* red = sm;                       // 32 * 9
    double* par = red + 288;                // face scalars (FP64), [48]
    double* tot = par + 48;                 // block sums, [16]
    F* pf = reinterpret_cast<F*>(tot + 16); // face constants in F, [64]
    NormalNode<F>* tn = reinterpret_cast<NormalNode<F>*>(pf + 64);   // per node of the first axis (or TangentNodes)
    F* ta = reinterpret_cast<F*>(tn + nu);  // per node of the first axis: u - U_s, (u - U_s)^2 / 2, [nu][2]
    F* wE = ta + 2 * nu;                    // exponentials per node, [nu] then [nvv]
    F* f0s = wE + nu + nvv;                 // [2][nv] (CACHE)
    F* sgs = f0s + 2 * nv;                  // [2][nv] (CACHE)
    const int i = axis == 0 ? fi % (nx + 1) : fi % nx;
    const int j = axis == 0 ? fi / (nx + 1) : fi / nx;
    const int bcid = (axis == 0 ? L.fbx : L.fby)[fi];
    const F* __restrict__ fG = A.f;
    const F* __restrict__ fH = A.f + nc * ld;
    F* __restrict__ phG = A.ph + (size_t)fi * ld;
    F* __restrict__ phH = A.ph + (nf + fi) * ld;

    if (bcid >= 0) {
        // ---------------- boundary face: free transport of the face distribution
        int outsign, c;
        bface_side(L, axis, i, j, c, outsign);
        const BcDev B = A.bc[bcid];
        const double* Cb = A.Cw + (size_t)bcid * nv;
        const double Hfac = kKint * B.t / 4.0;   // K / (4 lambda_b)
        double rhow = B.rho;
        if (B.type == BC_WALL) {
            double s[2] = {0.0, 0.0};
            for (int k = tid; k < nv; k += bs) {
                double uo = outsign * (axis == 0 ? Vg.u[k] : Vg.v[k]);
                if (uo > 0) s[0] += Vg.w[k] * uo * (double)fG[c * ld + k];
                else if (uo < 0) s[1] += Vg.w[k] * uo * Cb[k];
            }
            block_sum<2>(s, red);
            rhow = -s[0] / s[1];
        }
        double Fm[4] = {0, 0, 0, 0};
        for (int k = tid; k < nv; k += bs) {
            double un = axis == 0 ? Vg.u[k] : Vg.v[k];
            double uo = outsign * un;
            double g, h;
            if (uo >= 0 || B.type == BC_OUTFLOW) {
                g = fG[c * ld + k]; h = fH[c * ld + k];
            } else if (B.type == BC_SYMMETRY) {
                int a = k / Vg.nvv, b = k - a * Vg.nvv;
                int km = axis == 0 ? (Vg.nu - 1 - a) * Vg.nvv + b : a * Vg.nvv + (Vg.nvv - 1 - b);
                g = fG[c * ld + km]; h = fH[c * ld + km];
            } else {   // wall (rho_w C) or farfield (rho_inf C)
                g = rhow * Cb[k]; h = g * Hfac;
            }
            double pg = un * g, ph = un * h;
            phG[k] = (F)pg; phH[k] = (F)ph;
            double u = Vg.u[k], v = Vg.v[k], w = Vg.w[k];
            Fm[0] += w * pg; Fm[1] += w * u * pg; Fm[2] += w * v * pg;
            Fm[3] += w * (0.5 * (u * u + v * v) * pg + ph);
        }
        block_sum<4>(Fm, red);
        if (tid == 0)
            for (int m = 0; m < 4; ++m) A.Fm[4 * (size_t)fi + m] = Fm[m];
        return;
    }

    if (inactive_face(L, axis, i, j)) {   // inside a body: no flux
        for (int k = tid; k < nv; k += bs) { phG[k] = F(0); phH[k] = F(0); }
        if (tid == 0)
            for (int m = 0; m < 4; ++m) A.Fm[4 * (size_t)fi + m] = 0.0;
        return;
    }
    // ---------------- interior face between cL (lower) and cR (upper)
    // Face constants are computed once (by one thread or one lane each) and
    // broadcast through shared memory as F: an FP64 instruction occupies a
    // GB300 SM sub-partition for as long for one lane as for thirty-two.
    const F* __restrict__ vw = VelT<F>::w(Vg);
    // a cell behind that does not exist is the upwind cell itself: its difference is zero, and so is the slope
    int cL, cR, cLL, cRR;
    if (axis == 0) {
        cL = j * nx + i - 1; cR = cL + 1;
        cLL = i - 1 > 0 && L.fbx[fi - 1] < 0 ? cL - 1 : cL;
        cRR = i + 1 < nx && L.fbx[fi + 1] < 0 ? cR + 1 : cR;
    } else {
        cL = (j - 1) * nx + i; cR = cL + nx;
        cLL = j - 1 > 0 && L.fby[fi - nx] < 0 ? cL - nx : cL;
        cRR = j + 1 < ny && L.fby[fi + nx] < 0 ? cR + nx : cR;
    }
    // the face's mesh constants (kFluxGeo): par[32..40] in FP64, the first five also in F
    if (tid < kFluxGeo - 1) {
        const double gv = A.geo[(size_t)fi * kFluxGeo + tid];
        par[32 + tid] = gv;
        if (tid < 5) pf[tid] = (F)gv;
    }
    // U_s, V_s: mean velocity of the two cells, rounded to FP32 (any value near the interface's serves)
    if (tid >= 32 && tid < 34) {
        const int m = tid - 31;
        const double *wl = A.W + 4 * (size_t)cL, *wr = A.W + 4 * (size_t)cR;
        pf[4 + m] = (F)(0.5f * ((float)wl[m] / (float)wl[0] + (float)wr[m] / (float)wr[0]));
    }
    __syncthreads();
    const F Us = pf[5], Vs = pf[6];
    for (int a = tid; a < nu; a += bs) {
        const F d = (F)Vg.ua[a] - Us;
        ta[2 * a] = d;
        ta[2 * a + 1] = F(0.5) * d * d;
    }
    __syncthreads();
    // threads: columns tx of the second axis, rows ty of the first
    const int bw = min(nvv, bs), rows = bs / bw, tx = tid % bw, ty = tid / bw;
    // nodes ascend: the first nneg of the normal axis come from above, the last ones from below
    const int nneg = Vg.nleave[0][axis], npos0 = (axis == 0 ? nu : nvv) - Vg.nleave[1][axis];
    const F r1 = pf[0], r2 = pf[1], r3 = pf[2], fhL = pf[3], fhR = pf[4];
    const size_t oL = cL * ld, oR = cR * ld, oLL = cLL * ld, oRR = cRR * ld;
    // face value f0 and slope sg of velocity k, reconstructed in its upwind cell (n: index on the normal axis)
    auto recon = [&](int k, int n, F (&f0)[2], F (&sg)[2]) {
        const bool neg = n < nneg;
        const size_t om = neg ? oRR : oLL, o0 = neg ? oR : oL, op = neg ? oL : oR;
        const F rm = neg ? -r3 : r1, rp = neg ? -r2 : r2, h = neg ? -fhR : fhL;
        #pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const F* fc = (cp == 0 ? fG : fH) + k;
            const F fu = fc[o0], s1 = (fu - fc[om]) * rm, s2 = (fc[op] - fu) * rp;
            sg[cp] = vl_limited(s1, s2);
            f0[cp] = fu + sg[cp] * h;
        }
        if (n >= nneg && n < npos0) {            // u_n = 0: the mean of both sides
            #pragma unroll
            for (int cp = 0; cp < 2; ++cp) {
                const F* fc = (cp == 0 ? fG : fH) + k;
                const F fu = fc[oR], s = vl_limited((fc[oRR] - fu) * r3, (fu - fc[oL]) * r2);
                f0[cp] = F(0.5) * (f0[cp] + (fu - s * fhR));
                sg[cp] = F(0.5) * (sg[cp] + s);
            }
        }
    };

    // pass 1: reconstruction and moments about (U_s, V_s): 1, a, b, e; a e, b e; a^2, a b, b^2
    // with (a, b) the shifted velocity and e its energy with the internal one
    Acc<F> M[9];
    if (ty < rows)
        for (int b = tx; b < nvv; b += bw) {
            const F db = (F)Vg.vb[b] - Vs, hb = F(0.5) * db * db;
            #pragma unroll 2
            for (int a = ty; a < nu; a += rows) {
                const int k = a * nvv + b;
                const F w = vw[k], da = ta[2 * a], ha = ta[2 * a + 1];
                F f0[2], sg[2];
                recon(k, axis == 0 ? a : b, f0, sg);
                if constexpr (CACHE) {
                    f0s[k] = f0[0]; f0s[nv + k] = f0[1];
                    sgs[k] = sg[0]; sgs[nv + k] = sg[1];
                }
                const F g = w * f0[0], we = w * ((ha + hb) * f0[0] + f0[1]), ga = g * da, gb = g * db;
                M[0].add(g); M[1].add(ga); M[2].add(gb); M[3].add(we);
                M[4].add(we * da); M[5].add(we * db);
                M[6].add(ga * da); M[7].add(ga * db); M[8].add(gb * db);
            }
        }
    block_sums<9>(M, red, tot);
    __syncthreads();
    // face scalars, spread over the lanes of warp 0: lane 0 the collision time and
    // time step, lanes 1 and 2 the left and right equilibrium slopes, lane 3 the heat flux
    if (tid < 4) {
        const double m0 = tot[0], m1 = tot[1], m2 = tot[2], m3 = tot[3], us = (double)Us, vs = (double)Vs;
        const double ir = rcp64(m0), dx = m1 * ir, dy = m2 * ir;
        const double U = us + dx, V = vs + dy;
        const double lam = (0.25 * (kKint + 2)) * m0 * rcp64(m3 - 0.5 * (m1 * dx + m2 * dy));
        if (tid == 0) {
            par[0] = m0; par[1] = U; par[2] = V; par[3] = lam;
            if constexpr (sizeof(F) == 8) par[4] = tau_of(A.gas, m0, lam);
            else par[4] = (double)tau_of_f(A.gas, (float)m0, (float)lam);
            par[5] = par[37];
            if (A.shock) {
                double rl, ul, vl, ll, rr, ur, vr, lr;
                prim4(A.W + 4 * (size_t)cL, rl, ul, vl, ll);
                prim4(A.W + 4 * (size_t)cR, rr, ur, vr, lr);
                const double pl = rl / (2.0 * ll), pr = rr / (2.0 * lr);
                par[4] += par[5] * fabs(pl - pr) / (pl + pr);
            }
        } else if (tid < 3) {
            const double* Wc = A.W + 4 * (size_t)(tid == 1 ? cL : cR);
            const double W0[4] = {m0, m1 + us * m0, m2 + vs * m0, m3 + us * m1 + vs * m2 + 0.5 * (us * us + vs * vs) * m0};
            const double hf = (tid == 1 ? ir : -ir) * (tid == 1 ? par[39] : par[40]);
            double dw[4];
            for (int m = 0; m < 4; ++m) dw[m] = (W0[m] - Wc[m]) * hf;
            if constexpr (sizeof(F) == 8) {
                micro_slope(dw, U, V, lam, par + (tid == 1 ? 8 : 12));
            } else {
                float dwf[4] = {(float)dw[0], (float)dw[1], (float)dw[2], (float)dw[3]}, af[4];
                micro_slope_t<float>(dwf, (float)U, (float)V, (float)lam, af);
                for (int m = 0; m < 4; ++m) par[(tid == 1 ? 8 : 12) + m] = af[m];
            }
        } else {
            // moments about (U, V) = (U_s, V_s) + (dx, dy)
            const double d2 = 0.5 * (dx * dx + dy * dy), es = m3 - dx * m1 - dy * m2 + d2 * m0;
            par[6] = tot[4] - dx * tot[6] - dy * tot[7] + d2 * m1 - dx * es;
            par[7] = tot[5] - dx * tot[7] - dy * tot[8] + d2 * m2 - dy * es;
        }
    }
    __syncthreads();
    {
        // warp 0: constants of the equilibrium in F, and one time integral per lane; the others: the exponentials
        const double rho0 = par[0], U0 = par[1], V0 = par[2], lam0 = par[3];
        if (tid < 32) {
            F val = F(0);
            if (tid < 8) val = (F)par[8 + tid];          // aL, aR
            else if (tid == 8) val = (F)U0;
            else if (tid == 9) val = (F)V0;
            else if (tid == 14) val = (F)par[6];
            else if (tid == 15) val = (F)par[7];
            else if constexpr (sizeof(F) == 8) {
                if (tid == 10) val = rho0 * lam0 / kPi;
                else if (tid == 11) val = kKint / (4.0 * lam0);
                else if (tid == 12) val = kKint * (kKint + 2.0) / (16.0 * lam0 * lam0);
                else if (tid == 13) val = (1.0 - A.gas.pr) * 4.0 * lam0 * lam0 / (5.0 * rho0);
                else if (tid >= 16 && tid < 21) val = time_coeff_one(par[5], par[4], tid - 16) * par[38];   // q_i / dt
            } else {                                      // FP32 constants need no FP64 division
                const float fl = (float)lam0;
                if (tid == 10) val = (float)rho0 * fl * (float)(1.0 / kPi);
                else if (tid == 11) val = (float)(kKint / 4.0) / fl;
                else if (tid == 12) val = (float)(kKint * (kKint + 2.0) / 16.0) / (fl * fl);
                else if (tid == 13) val = (float)((1.0 - A.gas.pr) * 0.8) * (fl * fl) / (float)rho0;
                else if (tid >= 16 && tid < 21) val = (float)((double)time_coeff_one_f((float)par[5], (float)par[4], tid - 16) * par[38]);
            }
            if (tid == 21) val = (F)lam0;
            if (tid < 22) pf[8 + tid] = val;
        } else {
            for (int e = tid - 32; e < nu + nvv; e += bs - 32) {
                const bool isu = e < nu;
                const double d = isu ? Vg.ua[e] - U0 : Vg.vb[e - nu] - V0;
                if constexpr (sizeof(F) == 8) {
                    wE[e] = exp(-lam0 * d * d);
                } else {
                    const float df = (float)d;
                    wE[e] = expf(-(float)lam0 * df * df);
                }
            }
        }
    }
    __syncthreads();
    const F fU0 = pf[16], fV0 = pf[17], gnorm = pf[18], hfac = pf[19], xi4q = pf[20], shk = pf[21], qx = pf[22], qy = pf[23];
    const F q1 = pf[24], q2 = pf[25], q3 = pf[26], q4 = pf[27], q5 = pf[28], lam = pf[29];
    // warp 0: one-axis sums N_i = sum w E u_n^i (i = 1..5, each side) and T_i = sum w E u_t^i (i = 0..4),
    // then the compatibility sums and the time slope
    if (tid < 32) {
        const F* En = axis == 0 ? wE : wE + nu;
        const F* Et = axis == 0 ? wE + nu : wE;
        const int Nn = axis == 0 ? nu : nvv, Nt = axis == 0 ? nvv : nu;
        Acc<F> T[15];
        for (int n = tid; n < Nn; n += 32) {
            const F u = (F)(axis == 0 ? Vg.ua : Vg.vb)[n];
            F p = (F)(axis == 0 ? Vg.wa : Vg.wb)[n] * En[n] * u;
            const bool neg = n < nneg;
            #pragma unroll
            for (int m = 0; m < 5; ++m) {
                T[m].add(neg ? F(0) : p);
                T[5 + m].add(neg ? p : F(0));
                p *= u;
            }
        }
        for (int n = tid; n < Nt; n += 32) {
            const F u = (F)(axis == 0 ? Vg.vb : Vg.ua)[n];
            F p = (F)(axis == 0 ? Vg.wb : Vg.wa)[n] * Et[n];
            #pragma unroll
            for (int m = 0; m < 5; ++m) { T[10 + m].add(p); p *= u; }
        }
        int which;
        const auto v = warp_sums<15>(T, which);
        F* NT = pf + 40;                                         // N_1 .. N_5 of both sides, T_0 .. T_4
        if (which < 15) {
            if constexpr (sizeof(F) == 8) NT[which] = v;
            else NT[which] = v.x + v.y;
        }
        __syncwarp();
        // sums of u_n^i u_t^j (c + a_n u_n + a_t u_t + a_3 (u_n^2 + u_t^2) / 2) w u_n E E: one (side, i, j, c) per lane,
        // lane 8 side + p: p 0 .. 4 with c = a_0 + a_3 K/(4 lambda) and (i, j) = 00, 10, 01, 20, 02; 5 with c = a_0; 6 a_3 alone
        const int side = tid >> 3 & 1, p = tid & 7;
        const F* as = pf + (side == 0 ? 8 : 12);
        const F* N = NT + 5 * side;
        const F* Tt = NT + 10;
        const int ii = p == 1 ? 1 : p == 3 ? 2 : 0, jj = p == 2 ? 1 : p == 4 ? 2 : 0;
        const F a3 = p == 6 ? F(0) : as[3], an = p == 6 ? F(0) : as[1 + axis], at = p == 6 ? F(0) : as[2 - axis];
        const F c = p == 6 ? as[3] : p == 5 ? as[0] : fma(as[3], hfac, as[0]);
        F S = (c * N[ii] + an * N[ii + 1] + F(0.5) * a3 * N[ii + 2]) * Tt[jj] + N[ii] * (at * Tt[jj + 1] + F(0.5) * a3 * Tt[jj + 2]);
        S += __shfl_down_sync(0xffffffffu, S, 8);
        // time slope A from -sum / rho, with g = rho lambda / pi E E
        F dwt[4];
        const F nrm = -lam * F(1.0 / kPi);
        #pragma unroll
        for (int m = 0; m < 4; ++m) {
            const F x = __shfl_sync(0xffffffffu, S, m), s4 = __shfl_sync(0xffffffffu, S, 4), s5 = __shfl_sync(0xffffffffu, S, 5),
                    s6 = __shfl_sync(0xffffffffu, S, 6);
            dwt[m] = nrm * (m < 3 ? x : F(0.5) * (x + s4) + hfac * s5 + xi4q * s6);
        }
        const F d1 = axis == 0 ? dwt[1] : dwt[2], d2 = axis == 0 ? dwt[2] : dwt[1];
        const F dw[4] = {dwt[0], d1, d2, dwt[3]};
        F As[4];
        micro_slope_t<F>(dw, fU0, fV0, lam, As);
        if (tid == 0)
            for (int m = 0; m < 4; ++m) pf[32 + m] = As[m];
    }
    __syncthreads();
    // nodes of the normal and the tangential axis
    auto normal = [&](int n, NormalNode<F>& N) {
        const F u = (F)(axis == 0 ? Vg.ua : Vg.vb)[n], c = u - (axis == 0 ? fU0 : fV0), qn = axis == 0 ? qx : qy;
        const F* as = pf + (n < nneg ? 12 : 8);
        const F an = as[1 + axis], at = as[2 - axis], a3 = as[3];
        const F* As = pf + 32;
        const F q2u = q2 * u;
        N.un = u;
        N.E = gnorm * (axis == 0 ? wE[n] : wE[nu + n]);
        N.P = q1 + q2u * (as[0] + u * (an + F(0.5) * a3 * u)) + q3 * (As[0] + u * (As[1 + axis] + F(0.5) * As[3] * u));
        N.C = q2u * at + q3 * As[2 - axis];
        N.Z = q2u * a3 + q3 * As[3];
        N.hZ = hfac * N.Z;
        N.xZ = xi4q * N.Z;
        N.Fq = q1 * shk * (c * qn);
        N.S = F(2) * lam * (c * c) - F(4);
        N.q5u = q5 * u;
    };
    auto tangent = [&](int n, TangentNode<F>& N) {
        const F u = (F)(axis == 0 ? Vg.vb : Vg.ua)[n], c = u - (axis == 0 ? fV0 : fU0), qt = axis == 0 ? qy : qx;
        N.ut = u;
        N.h = F(0.5) * u;
        N.E = axis == 0 ? wE[nu + n] : wE[n];
        N.Fq = q1 * shk * (c * qt);
        N.S = F(2) * lam * (c * c);
    };
    for (int a = tid; a < nu; a += bs) {
        if (axis == 0) normal(a, tn[a]);
        else tangent(a, reinterpret_cast<TangentNode<F>*>(tn)[a]);
    }
    __syncthreads();

    // pass 2: time-averaged flux of every discrete velocity and its moments
    Acc<F> Fa[4];
    auto sweep = [&](auto ax) {
        constexpr int AX = decltype(ax)::value;
        for (int b = tx; b < nvv; b += bw) {
            NormalNode<F> N;
            TangentNode<F> T;
            if (AX == 0) tangent(b, T); else normal(b, N);
            const F vb = (F)Vg.vb[b], hv2 = F(0.5) * vb * vb;
            #pragma unroll 2
            for (int a = ty; a < nu; a += rows) {
                const int k = a * nvv + b;
                const F w = vw[k];
                if (AX == 0) N = tn[a];
                else T = reinterpret_cast<const TangentNode<F>*>(tn)[a];
                F f0[2], sg[2];
                if constexpr (CACHE) {
                    f0[0] = f0s[k]; f0[1] = f0s[nv + k]; sg[0] = sgs[k]; sg[1] = sgs[nv + k];
                } else {
                    recon(k, AX == 0 ? a : b, f0, sg);
                }
                const F gM = N.E * T.E, Fq = N.Fq + T.Fq, S = N.S + T.S;
                const F Y = fma(Fq, S, fma(T.ut, fma(T.h, N.Z, N.C), N.P));
                const F eG = gM * (Y + N.hZ), eH = gM * fma(hfac, fma(F(2), Fq, Y), N.xZ);
                const F pg = N.un * fma(q4, f0[0], fma(N.q5u, sg[0], eG));
                const F ph = N.un * fma(q4, f0[1], fma(N.q5u, sg[1], eH));
                phG[k] = pg; phH[k] = ph;
                const F u = AX == 0 ? N.un : T.ut, wg = w * pg;
                Fa[0].add(wg); Fa[1].add(wg * u); Fa[2].add(wg * vb);
                Fa[3].add(fma(wg, fma(F(0.5) * u, u, hv2), w * ph));
            }
        }
    };
    if (ty < rows) {
        if (axis == 0) sweep(std::integral_constant<int, 0>());
        else sweep(std::integral_constant<int, 1>());
    }
    block_sums<4>(Fa, red, tot);
    if (tid < 4) A.Fm[4 * (size_t)fi + tid] = tot[tid];      // (written by this thread)
}

template <typename F>
cudaError_t launch_face_flux(const FaceFluxArgs<F>& a, cudaStream_t st)
{
    constexpr size_t kSmemMax = 227 * 1024;
    // the cache pays while it leaves room for two CTAs per SM; beyond that the face values are
    // reconstructed again in the second pass (which costs a third of the arithmetic, where the split
    // of a face over a cluster, each CTA caching its share, repeats the face's serial phases)
    constexpr size_t kCacheMax = 110 * 1024;
    const size_t base = sizeof(double) * (288 + 48 + 16) + sizeof(F) * (64 + 3 * (size_t)a.V.nu + a.V.nvv) +
                        sizeof(NormalNode<F>) * (size_t)a.V.nu;
    const size_t full = base + sizeof(F) * 4 * (size_t)a.V.nv;
    const bool cache = full <= kCacheMax;
    const size_t smem = cache ? full : base;
    if (smem > kSmemMax) return cudaErrorInvalidValue;
    auto kern = cache ? k_face_flux<F, true> : k_face_flux<F, false>;
    if (smem > 47 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int nf = a.axis == 0 ? a.L.nfx : a.L.nfy;
    // whole rows of the second velocity axis, about 128 threads for a small velocity grid (more faces
    // overlap their serial phases on an SM) and 256 for a large one
    const int want = a.V.nv <= 1536 ? 128 : 256, rows = std::max(1, want / a.V.nvv);
    const int threads = std::min(256, std::max(64, (rows * a.V.nvv + 31) / 32 * 32));
    kern<<<nf, threads, smem, st>>>(a);
    return cudaGetLastError();
}
template cudaError_t launch_face_flux<double>(const FaceFluxArgs<double>&, cudaStream_t);
template cudaError_t launch_face_flux<float>(const FaceFluxArgs<float>&, cudaStream_t);

// R_i = -(1/V_i) sum_j S_ij F_ij
__global__ void k_cell_residual(LevelDev L, const double* __restrict__ Fx, const double* __restrict__ Fy,
                                double* __restrict__ R)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.nc) return;
    int i = c % L.nx, j = c / L.nx;
    if (L.solid[c]) {
        for (int m = 0; m < 4; ++m) R[4 * (size_t)c + m] = 0.0;
        return;
    }
    double V = L.dx[i] * L.dy[j];
    const double* FW = Fx + 4 * (size_t)(j * (L.nx + 1) + i);
    const double* FE = FW + 4;
    const double* FS = Fy + 4 * (size_t)(j * L.nx + i);
    const double* FN = Fy + 4 * (size_t)((j + 1) * L.nx + i);
    for (int m = 0; m < 4; ++m)
        R[4 * (size_t)c + m] = -(L.dy[j] * (FE[m] - FW[m]) + L.dx[i] * (FN[m] - FS[m])) / V;
}

cudaError_t launch_cell_residual(const LevelDev& L, const double* Fx, const double* Fy, double* R, cudaStream_t st)
{
    k_cell_residual<<<(L.nc + 127) / 128, 128, 0, st>>>(L, Fx, Fy, R);
    return cudaGetLastError();
}

// sum of squares of R per component: per-block partials, then one block
// partial sums of R^2 per component and the count of unphysical cells
// (non-positive density or internal energy, or NaN) per CTA
__global__ void k_rms_partial(const double* __restrict__ R, const double* __restrict__ W, int nc,
                              double* __restrict__ part)
{
    __shared__ double red[32 * 5];
    double s[5] = {0, 0, 0, 0, 0};
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
        for (int m = 0; m < 4; ++m) s[m] += R[4 * (size_t)c + m] * R[4 * (size_t)c + m];
        const double* w = W + 4 * (size_t)c;
        // rho e_int = E - |m|^2 / (2 rho), tested as rho E - |m|^2 / 2 > 0 with rho > 0
        const double e2 = w[3] * w[0] - 0.5 * (w[1] * w[1] + w[2] * w[2]);
        if (!(w[0] > 0.0) || !(e2 > 0.0)) s[4] += 1.0;
    }
    block_sum<5>(s, red);
    if (threadIdx.x == 0)
        for (int m = 0; m < 5; ++m) part[5 * blockIdx.x + m] = s[m];
}

__global__ void k_rms_final(const double* __restrict__ part, int nblk, int nfluid, double* __restrict__ out)
{
    __shared__ double red[32 * 5];
    double s[5] = {0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x)
        for (int m = 0; m < 5; ++m) s[m] += part[5 * b + m];
    block_sum<5>(s, red);
    if (threadIdx.x == 0) {
        for (int m = 0; m < 4; ++m) out[m] = sqrt(s[m] / nfluid);
        out[4] = s[4];
    }
}

// RMS over the fluid cells (R is zero in bodies)
cudaError_t launch_rms(const double* R, const double* W, int nc, int nfluid, double* part, double* out, cudaStream_t st)
{
    int nblk = 64;
    k_rms_partial<<<nblk, 256, 0, st>>>(R, W, nc, part);
    k_rms_final<<<1, 64, 0, st>>>(part, nblk, nfluid, out);
    return cudaGetLastError();
}

} // namespace miugks
