// flux.cu -- Step 1 of the MIUGKS iteration (arXiv 1704.03151, Sec. 2.1):
// time-averaged UGKS interface fluxes of every discrete velocity (Eqs.
// macroResidualCalc, microResidualDef) and the macroscopic residual R
// (Eq. macroResidualDef), plus its RMS (Eq. Residual_Def).
//
// One CTA per face.  FP64 (k_face_flux) is bound by the issue of its arithmetic and
// the mixed form (k_face_flux_mixed) by how exactly FP32 can take the interface's
// sums, so the two are different kernels.
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
    const double p = s1 * s2;      // p > 0 is looked at in the bits (a comparison would take the FP64 pipe); a NaN is not > 0
    return (unsigned long long)(__double_as_longlong(p) - 1) < 0x7ff0000000000000ull ? (p + p) * rcp64(s1 + s2) : 0.0;
}
// (sum: s1 + s2, as the caller rounds it)
__device__ __forceinline__ float vl_limited(float s1, float s2, float sum)
{
    float p = s1 * s2;   // the sum has no cancellation here; the fast quotient is within 2 ulp
    return p > 0.0f ? __fdividef(2.0f * p, sum) : 0.0f;
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

// A boundary face (free transport of the face distribution) or a face inside a body (no
// flux); false at an interior face.  FP64 in both forms.  red: block_sum's scratch
template <typename F>
__device__ bool outer_face(const FaceFluxArgs<F>& A, int fi, int i, int j, double* red)
{
    const LevelDev& L = A.L;
    const VelDev& Vg = A.V;
    const int axis = A.axis, nv = Vg.nv, tid = threadIdx.x, bs = blockDim.x;
    const size_t ld = Vg.ld, nc = L.nc, nf = axis == 0 ? L.nfx : L.nfy;
    const int bcid = (axis == 0 ? L.fbx : L.fby)[fi];
    const F* __restrict__ fG = A.f;
    const F* __restrict__ fH = A.f + nc * ld;
    F* __restrict__ phG = A.ph + (size_t)fi * ld;
    F* __restrict__ phH = A.ph + (nf + fi) * ld;
    if (bcid >= 0) {
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
        return true;
    }

    if (inactive_face(L, axis, i, j)) {   // inside a body: no flux
        for (int k = tid; k < nv; k += bs) { phG[k] = F(0); phH[k] = F(0); }
        if (tid == 0)
            for (int m = 0; m < 4; ++m) A.Fm[4 * (size_t)fi + m] = 0.0;
        return true;
    }
    return false;
}

// Constants of the flux per node of the velocity axis normal to the face, and per
// node of the tangential axis (k_face_flux, second pass)
struct alignas(16) NormalNode { double un, E, P, C, Z, hZ, xZ, Fq, S, q5u; };
struct alignas(16) TangentNode { double ut, h, E, Fq, S; };   // h = u_t / 2

// FP64 form.  A thread keeps one velocity of the second axis and strides over the
// first, so every load of f is coalesced and whatever depends on the second axis only
// stays in registers.  Two passes over the velocities: the first reconstructs the face
// values and takes their moments, the second forms the flux and its moments.
//
// What is done per velocity is kept small, since the kernel is bound by the issue of its
// FP64 arithmetic (two lanes per clock and SM):
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
// the second pass reconstructs again.  Without TABLES (a first axis of more than
// about 2,200 nodes) the node constants are formed where they are used, too.
// Per launch against three passes that reconstructed both sides of every velocity: flat
// plate (48x48) 13.1 -> 4.8 ms, 64x64 cavity (32x32) 1.92 -> 0.72 ms, square cylinder at
// half size (89x89) 21.4 -> 10.1 ms.
template <bool CACHE, bool TABLES>
__global__ void __launch_bounds__(256, 2) k_face_flux(FaceFluxArgs<double> A)
{
    using F = double;
    extern __shared__ double sm[];
    const LevelDev& L = A.L;
    const VelDev& Vg = A.V;
    const int nv = Vg.nv, nu = Vg.nu, nvv = Vg.nvv, tid = threadIdx.x, bs = blockDim.x;
    const size_t ld = Vg.ld;
    const int axis = A.axis, fi = blockIdx.x;
    const int nx = L.nx, ny = L.ny;
    const size_t nc = L.nc, nf = axis == 0 ? L.nfx : L.nfy;
    double* red = sm;                       // 32 * 9
    double* par = red + 288;                // face scalars, [48]
    double* tot = par + 48;                 // block sums, [16]
    F* pf = tot + 16;                       // face constants, [64]
    F* wE = pf + 64;                        // exponentials per node, [nu] then [nvv], to an even number
    NormalNode* tn = reinterpret_cast<NormalNode*>(wE + ((nu + nvv + 1) & ~1));   // per node of the first axis (or TangentNodes)
    F* ta = reinterpret_cast<F*>(tn + (TABLES ? nu : 0));   // per node of the first axis: u - U_s, (u - U_s)^2 / 2, [nu][2]
    F* f0s = ta + (TABLES ? 2 * nu : 0);    // [2][nv] (CACHE)
    F* sgs = f0s + 2 * nv;                  // [2][nv] (CACHE)
    const int i = axis == 0 ? fi % (nx + 1) : fi % nx;
    const int j = axis == 0 ? fi / (nx + 1) : fi / nx;
    const F* __restrict__ fG = A.f;
    const F* __restrict__ fH = A.f + nc * ld;
    F* __restrict__ phG = A.ph + (size_t)fi * ld;
    F* __restrict__ phH = A.ph + (nf + fi) * ld;

    if (outer_face<double>(A, fi, i, j, red)) return;
    // ---------------- interior face between cL (lower) and cR (upper)
    // Face constants are computed once (by one thread or one lane each) and
    // broadcast through shared memory: an FP64 instruction occupies a
    // GB300 SM sub-partition for as long for one lane as for thirty-two.
    const F* __restrict__ vw = Vg.w;
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
    // the face's mesh constants (kFluxGeo): par[32..40], the first five also in pf
    if (tid < kFluxGeo - 1) {
        const double gv = A.geo[(size_t)fi * kFluxGeo + tid];
        par[32 + tid] = gv;
        if (tid < 5) pf[tid] = gv;
    }
    // U_s, V_s: mean velocity of the two cells, rounded to FP32 (any value near the interface's serves)
    if (tid >= 32 && tid < 34) {
        const int m = tid - 31;
        const double *wl = A.W + 4 * (size_t)cL, *wr = A.W + 4 * (size_t)cR;
        pf[4 + m] = (F)(float)(0.5 * (wl[m] * rcp64(wl[0]) + wr[m] * rcp64(wr[0])));
    }
    __syncthreads();
    const F Us = pf[5], Vs = pf[6];
    auto shifted = [&](int a, F& d, F& h) { d = Vg.ua[a] - Us; h = F(0.5) * d * d; };
    if constexpr (TABLES) {
        for (int a = tid; a < nu; a += bs) shifted(a, ta[2 * a], ta[2 * a + 1]);
        __syncthreads();
    }
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
                const F w = vw[k];
                F da, ha;
                if constexpr (TABLES) { da = ta[2 * a]; ha = ta[2 * a + 1]; }
                else shifted(a, da, ha);
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
            par[4] = tau_of(A.gas, m0, lam);
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
            micro_slope(dw, U, V, lam, par + (tid == 1 ? 8 : 12));
        } else {
            // moments about (U, V) = (U_s, V_s) + (dx, dy)
            const double d2 = 0.5 * (dx * dx + dy * dy), es = m3 - dx * m1 - dy * m2 + d2 * m0;
            par[6] = tot[4] - dx * tot[6] - dy * tot[7] + d2 * m1 - dx * es;
            par[7] = tot[5] - dx * tot[7] - dy * tot[8] + d2 * m2 - dy * es;
        }
    }
    __syncthreads();
    {
        // warp 0: constants of the equilibrium, and one time integral per lane; the others: the exponentials
        const double rho0 = par[0], U0 = par[1], V0 = par[2], lam0 = par[3];
        if (tid < 32) {
            F val = F(0);
            if (tid < 8) val = par[8 + tid];             // aL, aR
            else if (tid == 8) val = U0;
            else if (tid == 9) val = V0;
            else if (tid == 10) val = rho0 * lam0 / kPi;
            else if (tid == 11) val = kKint / (4.0 * lam0);
            else if (tid == 12) val = kKint * (kKint + 2.0) / (16.0 * lam0 * lam0);
            else if (tid == 13) val = (1.0 - A.gas.pr) * 4.0 * lam0 * lam0 / (5.0 * rho0);
            else if (tid == 14) val = par[6];
            else if (tid == 15) val = par[7];
            else if (tid < 21) val = time_coeff_one(par[5], par[4], tid - 16) * par[38];   // q_i / dt
            else if (tid == 21) val = lam0;
            if (tid < 22) pf[8 + tid] = val;
        } else {
            for (int e = tid - 32; e < nu + nvv; e += bs - 32) {
                const bool isu = e < nu;
                const double d = isu ? Vg.ua[e] - U0 : Vg.vb[e - nu] - V0;
                wE[e] = exp(-lam0 * d * d);
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
        const F v = warp_sums<15>(T, which);
        F* NT = pf + 40;                                         // N_1 .. N_5 of both sides, T_0 .. T_4
        if (which < 15) NT[which] = v;
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
    auto normal = [&](int n, NormalNode& N) {
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
    auto tangent = [&](int n, TangentNode& N) {
        const F u = (F)(axis == 0 ? Vg.vb : Vg.ua)[n], c = u - (axis == 0 ? fV0 : fU0), qt = axis == 0 ? qy : qx;
        N.ut = u;
        N.h = F(0.5) * u;
        N.E = axis == 0 ? wE[nu + n] : wE[n];
        N.Fq = q1 * shk * (c * qt);
        N.S = F(2) * lam * (c * c);
    };
    if constexpr (TABLES) {
        for (int a = tid; a < nu; a += bs) {
            if (axis == 0) normal(a, tn[a]);
            else tangent(a, reinterpret_cast<TangentNode*>(tn)[a]);
        }
        __syncthreads();
    }

    // pass 2: time-averaged flux of every discrete velocity and its moments
    Acc<F> Fa[4];
    auto sweep = [&](auto ax) {
        constexpr int AX = decltype(ax)::value;
        for (int b = tx; b < nvv; b += bw) {
            NormalNode N;
            TangentNode T;
            if (AX == 0) tangent(b, T); else normal(b, N);
            const F vb = (F)Vg.vb[b], hv2 = F(0.5) * vb * vb;
            #pragma unroll 2
            for (int a = ty; a < nu; a += rows) {
                const int k = a * nvv + b;
                const F w = vw[k];
                if constexpr (!TABLES) {
                    if (AX == 0) normal(a, N);
                    else tangent(a, T);
                } else if (AX == 0) {
                    N = tn[a];
                } else {
                    T = reinterpret_cast<const TangentNode*>(tn)[a];
                }
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

// (a . psi) g split into the reduced components: b gM + a4 hM and b hM + a4 <xi^4>/4 gM
template <typename F>
__device__ __forceinline__ void slope_mom(const F* a, F u, F v, F gM, F hM, F xi4q, F& mG, F& mH)
{
    F b = a[0] + a[1] * u + a[2] * v + F(0.5) * a[3] * (u * u + v * v);
    mG = b * gM + a[3] * hM;
    mH = b * hM + a[3] * xi4q * gM;
}

// Mixed form.  Per-velocity arithmetic in FP32; every sum over the velocities is Kahan
// compensated per thread, reduced as float-float pairs and rounded to FP64 once, and the
// face's state, slopes and their compatibility sums are FP64 until they are rounded to FP32
// as constants of the next pass.  Three passes over the velocities, threads striding over
// them: interface state; heat flux and compatibility moments, about the state just found;
// the flux and its moments.  The equilibrium comes from per-axis exponentials (nu + nv per
// face instead of nu nv).
//
// The FP64 form's one-axis sums are not used here.  Rounded to FP32 and multiplied together
// they lose what the FP64 totals keep: the raw powers of the velocities, up to the fifth,
// cancel in a fast flow, where the time slope A had about eighteen times this form's error
// (Mach 5 free stream, 89x89 velocities).  From a marginally stable start such a difference
// decides which cells keep their prediction.
//
// Only the upwind side of a velocity is reconstructed (three cells of the four).  CACHE
// keeps the face values and slopes in shared memory between the passes; without it (a
// velocity grid whose cache leaves too few CTAs per SM) each pass reconstructs them.
// Bound by the issue of its FP32 arithmetic.  Flux per iteration against reconstructing both
// sides: square cylinder (89x89) 8.7 -> 6.1 ms, flat plate (48x48) 1.46 -> 1.03 ms, 64x64 cavity
// (32x32) 0.26 -> 0.18 ms.
template <bool CACHE>
__global__ void __launch_bounds__(256, 4) k_face_flux_mixed(FaceFluxArgs<float> A)
{
    using F = float;
    extern __shared__ double sm[];
    const LevelDev& L = A.L;
    const VelDev& Vg = A.V;
    const int nv = Vg.nv, tid = threadIdx.x, bs = blockDim.x;
    const size_t ld = Vg.ld;
    const int axis = A.axis, fi = blockIdx.x;
    const int nx = L.nx, ny = L.ny;
    const size_t nc = L.nc, nf = axis == 0 ? L.nfx : L.nfy;
    double* red = sm;                       // 32 * 8
    double* par = red + 256;                // face scalars (FP64), [48]
    F* pf = reinterpret_cast<F*>(par + 48); // face constants in FP32, [64]
    F* f0s = pf + 64;                       // [2][nv] (CACHE)
    F* sgs = f0s + (CACHE ? 2 * nv : 0);    // [2][nv] (CACHE)
    F* Eu = sgs + (CACHE ? 2 * nv : 0);     // [nu]
    F* Ev = Eu + Vg.nu;                     // [nvv]
    const int i = axis == 0 ? fi % (nx + 1) : fi % nx;
    const int j = axis == 0 ? fi / (nx + 1) : fi / nx;
    const F* __restrict__ fG = A.f;
    const F* __restrict__ fH = A.f + nc * ld;
    F* __restrict__ phG = A.ph + (size_t)fi * ld;
    F* __restrict__ phH = A.ph + (nf + fi) * ld;

    if (outer_face<float>(A, fi, i, j, red)) return;
    // ---------------- interior face between cL (lower) and cR (upper)
    // Face constants are computed once (by one thread or one lane each) and
    // broadcast through shared memory as F: an FP64 instruction occupies a
    // GB300 SM sub-partition for as long for one lane as for thirty-two.
    const F* __restrict__ vu = Vg.uf;
    const F* __restrict__ vv = Vg.vf;
    const F* __restrict__ vw = Vg.wf;
    int cL, cR, cLL = -1, cRR = -1;
    if (axis == 0) {
        cL = j * nx + i - 1; cR = cL + 1;
        if (i - 1 > 0 && L.fbx[fi - 1] < 0) cLL = cL - 1;
        if (i + 1 < nx && L.fbx[fi + 1] < 0) cRR = cR + 1;
    } else {
        cL = (j - 1) * nx + i; cR = cL + nx;
        if (j - 1 > 0 && L.fby[fi - nx] < 0) cLL = cL - nx;
        if (j + 1 < ny && L.fby[fi + nx] < 0) cRR = cR + nx;
    }
    // the face's mesh constants (kFluxGeo): par[32..40] in FP64, the first five also in F
    if (tid < kFluxGeo - 1) {
        const double gv = A.geo[(size_t)fi * kFluxGeo + tid];
        par[32 + tid] = gv;
        if (tid < 5) pf[tid] = (F)gv;
    }
    __syncthreads();
    const F r1 = pf[0], r2 = pf[1], r3 = pf[2], fhL = pf[3], fhR = pf[4];
    // the cells' rows, from the lower cell's: the upper one's, and those behind (a missing one is the upwind
    // cell itself: its difference is zero, and so is the slope)
    const F* __restrict__ gL = fG + cL * ld;
    const F* __restrict__ hL = fH + cL * ld;
    const int oR = (cR - cL) * Vg.ld, oLL = cLL >= 0 ? -oR : 0, oRR = cRR >= 0 ? 2 * oR : oR;
    // face value f0 and slope sg of G and H of velocity k, reconstructed in its upwind cell (van Leer); the sum of the
    // slopes is rounded once, the inner product fused into it, where the value is kept, and from both products else
    auto recon = [&](int k, F (&f0)[2], F (&sg)[2]) {
        const F un = axis == 0 ? vu[k] : vv[k];
        const bool neg = un < F(0);
        const int om = neg ? oRR : oLL, o0 = neg ? oR : 0, op = neg ? 0 : oR;
        const F rm = neg ? -r3 : r1, rp = neg ? -r2 : r2, h = neg ? -fhR : fhL;
        #pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const F* fc = (cp == 0 ? gL : hL) + k;
            const F fu = fc[o0], d1 = fu - fc[om], d2 = fc[op] - fu, s1 = __fmul_rn(d1, rm), s2 = __fmul_rn(d2, rp);
            sg[cp] = vl_limited(s1, s2, CACHE ? fmaf(d2, rp, s1) : s1 + s2);
            f0[cp] = fmaf(sg[cp], h, fu);
        }
        if (un == F(0)) {                        // the mean of both sides
            #pragma unroll
            for (int cp = 0; cp < 2; ++cp) {
                const F* fc = (cp == 0 ? gL : hL) + k;
                const F fu = fc[oR], d1 = fc[oRR] - fu, d2 = fu - fc[0], s1 = __fmul_rn(d1, r3), s2 = __fmul_rn(d2, r2);
                const F s = vl_limited(s1, s2, CACHE ? fmaf(d2, r2, s1) : s1 + s2);
                f0[cp] = F(0.5) * (f0[cp] + fmaf(-s, fhR, fu));
                sg[cp] = F(0.5) * (sg[cp] + s);
            }
        }
    };
    auto face_vals = [&](int k, F (&f0)[2], F (&sg)[2]) {
        if constexpr (CACHE) {
            f0[0] = f0s[k]; f0[1] = f0s[nv + k]; sg[0] = sgs[k]; sg[1] = sgs[nv + k];
        } else {
            recon(k, f0, sg);
        }
    };

    // pass 1: reconstruction, upwinding, interface conservative variables
    // (unrolled so that the loads of the next velocity are in flight with this one's arithmetic)
    Acc<F> W0a[4];
    #pragma unroll 2
    for (int k = tid; k < nv; k += bs) {
        F f0[2], sg[2];
        recon(k, f0, sg);
        if constexpr (CACHE) {
            f0s[k] = f0[0]; f0s[nv + k] = f0[1];
            sgs[k] = sg[0]; sgs[nv + k] = sg[1];
        }
        const F w = vw[k], u = vu[k], v = vv[k], g = f0[0];
        W0a[0].add(w * g); W0a[1].add(w * u * g); W0a[2].add(w * v * g);
        W0a[3].add(w * (F(0.5) * (u * u + v * v) * g + f0[1]));
    }
    double W0[4];
    block_total<4>(W0a, red, W0);
    // face scalars, spread over the lanes of warp 0: lane 0 the collision time and
    // time step, lanes 1 and 2 the left and right equilibrium slopes
    if (tid < 3) {
        double rho = W0[0], ir = rcp64(rho);
        double U = W0[1] * ir, V = W0[2] * ir;
        double lam = (kKint + 2) * rho * rcp64(4.0 * (W0[3] - 0.5 * (W0[1] * U + W0[2] * V)));
        if (tid == 0) {
            par[0] = rho; par[1] = U; par[2] = V; par[3] = lam;
            par[4] = (double)tau_of_f(A.gas, (float)rho, (float)lam);
            par[5] = par[37];
            if (A.shock) {
                double rl, ul, vl, ll, rr, ur, vr, lr;
                prim4(A.W + 4 * (size_t)cL, rl, ul, vl, ll);
                prim4(A.W + 4 * (size_t)cR, rr, ur, vr, lr);
                const double pl = rl / (2.0 * ll), pr = rr / (2.0 * lr);
                par[4] += par[5] * fabs(pl - pr) / (pl + pr);
            }
        } else {
            const double* Wc = A.W + 4 * (size_t)(tid == 1 ? cL : cR);
            double hf, dw[4];
            hf = (tid == 1 ? 1.0 : -1.0) * ir * (tid == 1 ? par[39] : par[40]);
            for (int m = 0; m < 4; ++m) dw[m] = (W0[m] - Wc[m]) * hf;
            float dwf[4] = {(float)dw[0], (float)dw[1], (float)dw[2], (float)dw[3]}, af[4];
            micro_slope_t<float>(dwf, (float)U, (float)V, (float)lam, af);
            for (int m = 0; m < 4; ++m) par[(tid == 1 ? 8 : 12) + m] = af[m];
        }
    }
    __syncthreads();
    {
        // warp 0: constants of the equilibrium in F; the other warps: the per-axis exponentials
        const double rho0 = par[0], U0 = par[1], V0 = par[2], lam0 = par[3];
        if (tid < 32) {
            F val = F(0);
            if (tid < 8) val = (F)par[8 + tid];          // aL, aR
            else if (tid == 8) val = (F)U0;
            else if (tid == 9) val = (F)V0;
            else {                                        // (no FP64 division for FP32 constants)
                const float fl = (float)lam0;
                if (tid == 10) val = (float)rho0 * fl * (float)(1.0 / kPi);
                else if (tid == 11) val = (float)(kKint / 4.0) / fl;
                else if (tid == 12) val = (float)(kKint * (kKint + 2.0) / 16.0) / (fl * fl);
            }
            if (tid < 13) pf[8 + tid] = val;
        } else {
            for (int e = tid - 32; e < Vg.nu + Vg.nvv; e += bs - 32) {
                const bool isu = e < Vg.nu;
                const double d = isu ? Vg.ua[e] - U0 : Vg.vb[e - Vg.nu] - V0;
                const float df = (float)d;
                Eu[e] = expf(-(float)lam0 * df * df);    // Ev follows Eu
            }
        }
    }
    __syncthreads();
    const F fU0 = pf[16], fV0 = pf[17], gnorm = pf[18], hfac = pf[19], xi4q = pf[20];
    F aL[4], aR[4];
    #pragma unroll
    for (int m = 0; m < 4; ++m) { aL[m] = pf[8 + m]; aR[m] = pf[12 + m]; }

    // velocity k = a * nvv + b of this thread, stepped by the block size without a division
    const int ka0 = tid / Vg.nvv, kb0 = tid - ka0 * Vg.nvv;
    const int sa = bs / Vg.nvv, sb = bs - sa * Vg.nvv;
    // pass 2: heat flux of the interface distribution, compatibility moments for A
    Acc<F> s6a[6];
    for (int k = tid, a = ka0, b = kb0; k < nv; k += bs, a += sa, b += sb) {
        if (b >= Vg.nvv) { b -= Vg.nvv; ++a; }
        const F u = vu[k], v = vv[k], w = vw[k];
        F cx = u - fU0, cy = v - fV0, c2 = cx * cx + cy * cy;
        F f0[2], sg[2];
        face_vals(k, f0, sg);
        F e = F(0.5) * c2 * f0[0] + f0[1];
        s6a[0].add(w * cx * e);
        s6a[1].add(w * cy * e);
        F un = axis == 0 ? u : v;
        if (un != F(0)) {
            F gM = gnorm * Eu[a] * Ev[b], hM = gM * hfac, mG, mH;
            slope_mom<F>(un > F(0) ? aL : aR, u, v, gM, hM, xi4q, mG, mH);
            F wu = w * un;
            s6a[2].add(wu * mG); s6a[3].add(wu * u * mG); s6a[4].add(wu * v * mG);
            s6a[5].add(wu * (F(0.5) * (u * u + v * v) * mG + mH));
        }
    }
    double s6[6];
    block_total<6>(s6a, red, s6);
    // lane 0: time slope A from compatibility; lanes 1-5: one time integral each
    if (tid < 6) {
        const double rho0 = par[0], U0 = par[1], V0 = par[2], lam0 = par[3];
        if (tid == 0) {
            double dwt[4], ir = -rcp64(rho0);
            for (int m = 0; m < 4; ++m) dwt[m] = s6[2 + m] * ir;
            float dwf[4] = {(float)dwt[0], (float)dwt[1], (float)dwt[2], (float)dwt[3]}, af[4];
            micro_slope_t<float>(dwf, (float)U0, (float)V0, (float)lam0, af);
            for (int m = 0; m < 4; ++m) par[16 + m] = af[m];
            par[6] = s6[0]; par[7] = s6[1];
        } else {
            par[20 + tid - 1] = time_coeff_one_f((float)par[5], (float)par[4], tid - 1);
        }
    }
    __syncthreads();
    if (tid < 32) {
        const double rho0 = par[0], lam0 = par[3];
        F val = F(0);
        if (tid < 4) val = (F)par[16 + tid];             // A
        else if (tid < 9) val = (F)(par[20 + tid - 4] * par[38]);   // q_i / dt
        else if (tid == 9) {
            val = (float)((1.0 - A.gas.pr) * 0.8) * ((float)lam0 * (float)lam0) / (float)rho0;
        }
        else if (tid == 10) val = (F)par[6];
        else if (tid == 11) val = (F)par[7];
        else if (tid == 12) val = (F)(2.0 * lam0);
        if (tid < 13) pf[24 + tid] = val;
    }
    __syncthreads();
    F As[4];
    #pragma unroll
    for (int m = 0; m < 4; ++m) As[m] = pf[24 + m];
    const F q1 = pf[28], q2 = pf[29], q3 = pf[30], q4 = pf[31], q5 = pf[32];
    const F shk = pf[33], qx = pf[34], qy = pf[35], flam2 = pf[36];

    // pass 3: time-averaged flux of every discrete velocity and its moments
    Acc<F> Fa[4];
    for (int k = tid, a = ka0, b = kb0; k < nv; k += bs, a += sa, b += sb) {
        if (b >= Vg.nvv) { b -= Vg.nvv; ++a; }
        const F u = vu[k], v = vv[k], w = vw[k];
        const F un = axis == 0 ? u : v;
        F cx = u - fU0, cy = v - fV0, c2 = cx * cx + cy * cy;
        F gM = gnorm * Eu[a] * Ev[b], hM = gM * hfac;
        F Fq = shk * (cx * qx + cy * qy);
        F gP = gM * (F(1) + Fq * (flam2 * c2 - F(4)));
        F hP = hM * (F(1) + Fq * (flam2 * c2 - F(2)));
        F mGa, mHa, mGA, mHA;
        slope_mom<F>(un > F(0) ? aL : aR, u, v, gM, hM, xi4q, mGa, mHa);
        slope_mom<F>(As, u, v, gM, hM, xi4q, mGA, mHA);
        F f0[2], sg[2];
        face_vals(k, f0, sg);
        F pg = un * (q1 * gP + q2 * un * mGa + q3 * mGA + q4 * f0[0] + q5 * un * sg[0]);
        F ph = un * (q1 * hP + q2 * un * mHa + q3 * mHA + q4 * f0[1] + q5 * un * sg[1]);
        phG[k] = pg; phH[k] = ph;
        Fa[0].add(w * pg); Fa[1].add(w * u * pg); Fa[2].add(w * v * pg);
        Fa[3].add(w * (F(0.5) * (u * u + v * v) * pg + ph));
    }
    double Fm[4];
    block_total<4>(Fa, red, Fm);
    if (tid == 0)
        for (int m = 0; m < 4; ++m) A.Fm[4 * (size_t)fi + m] = Fm[m];
}

template <>
cudaError_t launch_face_flux<double>(const FaceFluxArgs<double>& a, cudaStream_t st)
{
    constexpr size_t kSmemMax = 227 * 1024;
    // the cache pays while it leaves room for two CTAs per SM; beyond that the face values are
    // reconstructed again in the second pass (which costs a third of the arithmetic, where the split
    // of a face over a cluster, each CTA caching its share, repeats the face's serial phases)
    constexpr size_t kCacheMax = 110 * 1024;
    const size_t nodes = sizeof(double) * (288 + 48 + 16 + 64 + (((size_t)a.V.nu + a.V.nvv + 1) & ~(size_t)1));
    const size_t base = nodes + (sizeof(double) * 2 + sizeof(NormalNode)) * (size_t)a.V.nu;
    const size_t full = base + sizeof(double) * 4 * (size_t)a.V.nv;
    const bool cache = full <= kCacheMax, tables = base <= kSmemMax;
    const size_t smem = cache ? full : tables ? base : nodes;
    if (smem > kSmemMax) return cudaErrorInvalidValue;
    auto kern = cache ? k_face_flux<true, true> : tables ? k_face_flux<false, true> : k_face_flux<false, false>;
    if (smem > 47 * 1024) {
        const cudaError_t e = allow_shared_memory((const void*)kern);
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

template <>
cudaError_t launch_face_flux<float>(const FaceFluxArgs<float>& a, cudaStream_t st)
{
    constexpr size_t kSmemMax = 227 * 1024;
    // the cache pays while it leaves room for several CTAs per SM; beyond it (89x89) one CTA per face that
    // reconstructs in each pass beats a face split over a cluster.  Measured with both sides of a face
    // reconstructed, per iteration: 64x64 cavity with 32x32 velocities 0.34 with the cache, 0.42 ms without,
    // flat plate with 48x48 1.48 and 2.08 ms, square cylinder 8.7 ms without and 11.8 ms split
    constexpr size_t kCacheMax = 64 * 1024;
    const size_t base = sizeof(double) * (256 + 48) + sizeof(float) * (64 + (size_t)a.V.nu + a.V.nvv);
    const size_t full = base + sizeof(float) * 4 * (size_t)a.V.nv;
    const bool cache = full <= kCacheMax;
    const size_t smem = cache ? full : base;
    if (smem > kSmemMax) return cudaErrorInvalidValue;
    auto kern = cache ? k_face_flux_mixed<true> : k_face_flux_mixed<false>;
    if (smem > 47 * 1024) {
        const cudaError_t e = allow_shared_memory((const void*)kern);
        if (e != cudaSuccess) return e;
    }
    const int nf = a.axis == 0 ? a.L.nfx : a.L.nfy;
    // a small velocity grid: 128 threads, so that more faces overlap their serial scalar phases on an
    // SM (0.27 against 0.34 ms); from 48x48 on 256 are faster (flat plate 1.48 against 1.72 ms)
    kern<<<nf, a.V.nv <= 1536 ? 128 : 256, smem, st>>>(a);
    return cudaGetLastError();
}

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
