// micro.cu -- evolution step of MIUGKS (arXiv 1704.03151, Secs. 2.1.2, 2.3,
// 2.4, 3.2): the microscopic residual with the predicted equilibrium (Eq.
// microResidualDef, Shakhov equilibrium), the upwind implicit operator (Eqs.
// microUpwind, microFinalDefect, evolutionCoefficients), its LU-SGS smoother,
// the residual renewal of the CS cycle (Eq. renewResidualMicro), and the
// moment update (Steps 6-7).
//
// LU-SGS on the GPU.  The sweep order is the serial lexicographic one; every
// cell depends only on its two lower (forward) or upper (backward) neighbours,
// so anti-diagonals can run in parallel.  Discrete velocities are independent
// except at boundary cells, where the diffuse-wall ghost (Eq. delta_f_on_wall)
// couples the incoming velocities of a cell to a sum over its outgoing ones.
// On the lower side (forward sweep) the boundary cells form two lines, the
// first column and the first row, and each line only depends on itself; the
// same holds for the last column and row in the backward sweep.  At a line
// cell, the velocities leaving through the boundary face (outgoing) need no
// ghost, and the incoming ones need only the cell's wall density, a sum over
// the outgoing ones.  Each sweep is therefore three launches:
//   * k_sgs_edge walks the lines for their outgoing velocities;
//   * k_line_rho sums up the wall densities of their cells;
//   * k_sgs_wave sweeps all cells, every CTA for its own velocities and with
//     no synchronisation between CTAs; the incoming velocities of line cells
//     are ordinary updates there, their ghost term being known.
// Which products are fused into sums, and the order of the wall sums, are written
// out: the mixed form's roundings are part of its result, since a marginally stable
// flow (a hot channel under the F cycle) amplifies them from one iteration to the next.
//
// Rows of velocities are padded to a multiple of sixteen (VelDev::ld), four lanes
// of 16 bytes in FP32, so that a block of the wavefront never leaves its row; the
// padding is zero and stays so.
#include "kernels.cuh"
#include "async.cuh"
#include <algorithm>
#include <array>
#include <type_traits>

namespace miugks {

// asynchronous 4- or 8-byte global -> shared copies (LDGSTS), completed per commit group
template <typename F>
__device__ __forceinline__ void cp_async_elem(F* sdst, const F* gsrc)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
    if constexpr (sizeof(F) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gsrc) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gsrc) : "memory");
}
// a product that is not fused into a sum
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

// (1/V) sum over the faces with u_n > 0 of u_n S = |u|/dx + |v|/dy
template <typename F>
__device__ __forceinline__ F geomD_r(F rdxi, F rdyj, F u, F v)
{
    return fma(fabs(u), rdxi, mul_rn(fabs(v), rdyj));
}

// coefficient (1/V) u_n S of a neighbour (or ghost) through the face with outward normal
// outsign * e_axis, zero unless u_n < 0; rS = S/V = 1/dx (x-faces) or 1/dy (y-faces)
template <typename F>
__device__ __forceinline__ F Dface(int axis, int outsign, F rS, F u, F v)
{
    F un = (axis == 0 ? u : v);
    un = outsign < 0 ? -un : un;
    return un < F(0) ? un * rS : F(0);
}

__device__ __forceinline__ double recip(double x) { return rcp64(x); }
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }

// ---------------------------------------------------------------------------
// Steps 3-4 on the finest level
template <typename F>
__global__ void __launch_bounds__(256) k_micro_residual(MicroArgs M, GasDev gas, const double* __restrict__ Wt,
                                                        const double* __restrict__ q, const F* __restrict__ f,
                                                        const F* __restrict__ phx, const F* __restrict__ phy,
                                                        double dtn_inv, double* __restrict__ inv_tau,
                                                        F* __restrict__ invD, F* __restrict__ r)
{
    extern __shared__ double sm[];
    const LevelDev& L = M.L;
    const VelDev& Vg = M.V;
    const int c = blockIdx.x, nv = Vg.nv, nx = L.nx;
    const size_t ld = Vg.ld;
    const int i = c % nx, j = c / nx;
    const size_t nc = L.nc;
    // cell constants: FP64 state from thread 0, then one constant per lane of warp 0
    // (an FP64 instruction costs a warp as much as thirty-two lanes of it)
    double* cs = sm;                            // cell scalars (FP64), [8]
    F* cf = reinterpret_cast<F*>(sm + 8);       // cell constants in F, [16]
    F* Eu = reinterpret_cast<F*>(sm + 24);
    F* Ev = Eu + Vg.nu;
    if (threadIdx.x == 0) {
        double rho, U, V, lam;
        prim4(Wt + 4 * (size_t)c, rho, U, V, lam);
        double it;
        if constexpr (sizeof(F) == 8) it = 1.0 / tau_of(gas, rho, lam);
        else it = (double)(1.0f / tau_of_f(gas, (float)rho, (float)lam));
        cs[0] = rho; cs[1] = U; cs[2] = V; cs[3] = lam; cs[4] = it;
        inv_tau[c] = it + dtn_inv;
    }
    __syncthreads();
    {
        const double rho = cs[0], U = cs[1], V = cs[2], lam = cs[3], itau = cs[4];
        const int t = threadIdx.x;
        if (t < 32) {
            F val = F(0);
            switch (t) {
            case 0: val = (F)(rho * lam / kPi); break;
            case 1: val = (F)(kKint / (4.0 * lam)); break;
            case 2: val = (F)(2.0 * lam); break;
            case 3: val = (F)((1.0 - gas.pr) * 4.0 * lam * lam / (5.0 * rho)); break;
            case 4: val = (F)q[2 * (size_t)c]; break;
            case 5: val = (F)q[2 * (size_t)c + 1]; break;
            case 6: val = (F)U; break;
            case 7: val = (F)V; break;
            case 8: val = (F)L.rdx[i]; break;
            case 9: val = (F)L.rdy[j]; break;
            case 10: val = (F)itau; break;
            case 11: val = (F)(itau + dtn_inv); break;
            default: break;
            }
            if (t < 12) cf[t] = val;
        } else {
            for (int e = t - 32; e < Vg.nu + Vg.nvv; e += blockDim.x - 32) {
                const bool isu = e < Vg.nu;
                const double d = isu ? Vg.ua[e] - U : Vg.vb[e - Vg.nu] - V;
                F ex;
                if constexpr (sizeof(F) == 8) ex = exp(-lam * d * d);
                else ex = expf((float)(-lam * d * d));
                (isu ? Eu[e] : Ev[e - Vg.nu]) = ex;
            }
        }
    }
    __syncthreads();
    const F gnorm = cf[0], hfac = cf[1], flam2 = cf[2], shk = cf[3], qx = cf[4], qy = cf[5], fU = cf[6], fV = cf[7];
    const F rdxi = cf[8], rdyj = cf[9], fitau = cf[10], fdiag = cf[11];
    const F* __restrict__ vu = VelT<F>::u(Vg);
    const F* __restrict__ vv = VelT<F>::v(Vg);
    const size_t nfx = L.nfx, nfy = L.nfy;
    const size_t fW = (size_t)j * (nx + 1) + i, fE = fW + 1, fS = (size_t)j * nx + i, fN = (size_t)(j + 1) * nx + i;
    const bool body = L.solid[c];   // cells in a body: zero residual
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        int a = k / Vg.nvv, b = k - a * Vg.nvv;
        const F u = vu[k], v = vv[k];
        F cx = u - fU, cy = v - fV, c2 = cx * cx + cy * cy;
        F gM = gnorm * Eu[a] * Ev[b], hM = gM * hfac;
        F Fq = shk * (cx * qx + cy * qy);
        F gt[2] = {gM * (F(1) + Fq * (flam2 * c2 - F(4))), hM * (F(1) + Fq * (flam2 * c2 - F(2)))};
        #pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            const F* px = phx + cp * nfx * ld;
            const F* py = phy + cp * nfy * ld;
            F div = (px[fE * ld + k] - px[fW * ld + k]) * rdxi + (py[fN * ld + k] - py[fS * ld + k]) * rdyj;
            r[(cp * nc + c) * ld + k] = body ? F(0) : (gt[cp] - f[(cp * nc + c) * ld + k]) * fitau - div;
        }
        invD[(size_t)c * ld + k] = recip(fdiag + geomD_r<F>(rdxi, rdyj, u, v));
    }
}

template <typename F>
cudaError_t launch_micro_residual(const MicroArgs& m, GasDev gas, const double* Wt, const double* q, const F* f,
                                  const F* phx, const F* phy, double dtn_inv, double* inv_tau, F* invD, F* r,
                                  cudaStream_t st)
{
    size_t smem = sizeof(double) * 24 + sizeof(F) * (m.V.nu + m.V.nvv);
    k_micro_residual<F><<<m.L.nc, m.V.nv >= 256 ? 256 : 128, smem, st>>>(m, gas, Wt, q, f, phx, phy, dtn_inv,
                                                                          inv_tau, invD, r);
    return cudaGetLastError();
}
template cudaError_t launch_micro_residual<double>(const MicroArgs&, GasDev, const double*, const double*,
                                                   const double*, const double*, const double*, double, double*,
                                                   double*, double*, cudaStream_t);
template cudaError_t launch_micro_residual<float>(const MicroArgs&, GasDev, const double*, const double*,
                                                  const float*, const float*, const float*, double, double*, float*,
                                                  float*, cudaStream_t);

template <typename F>
__global__ void k_coarse_coeffs(MicroArgs M, GasDev gas, const double* __restrict__ Wt, double dtn_inv,
                                double* __restrict__ inv_tau, F* __restrict__ invD)
{
    const LevelDev& L = M.L;
    const int c = blockIdx.x, i = c % L.nx, j = c / L.nx;
    __shared__ F sc[3];
    if (threadIdx.x == 0) {
        double rho, U, V, lam;
        prim4(Wt + 4 * (size_t)c, rho, U, V, lam);
        double it;
        if constexpr (sizeof(F) == 8) it = 1.0 / tau_of(gas, rho, lam);
        else it = (double)(1.0f / tau_of_f(gas, (float)rho, (float)lam));
        it += dtn_inv;
        inv_tau[c] = it;
        sc[0] = (F)it; sc[1] = (F)L.rdx[i]; sc[2] = (F)L.rdy[j];
    }
    __syncthreads();
    const F fit = sc[0], rdxi = sc[1], rdyj = sc[2];
    const F* __restrict__ vu = VelT<F>::u(M.V);
    const F* __restrict__ vv = VelT<F>::v(M.V);
    for (int k = threadIdx.x; k < M.V.nv; k += blockDim.x)
        invD[(size_t)c * M.V.ld + k] = recip(fit + geomD_r<F>(rdxi, rdyj, vu[k], vv[k]));
}

template <typename F>
cudaError_t launch_coarse_coeffs(const MicroArgs& m, GasDev gas, const double* Wt, double dtn_inv, double* inv_tau,
                                 F* invD, cudaStream_t st)
{
    k_coarse_coeffs<F><<<m.L.nc, 128, 0, st>>>(m, gas, Wt, dtn_inv, inv_tau, invD);
    return cudaGetLastError();
}
template cudaError_t launch_coarse_coeffs<double>(const MicroArgs&, GasDev, const double*, double, double*, double*,
                                                  cudaStream_t);
template cudaError_t launch_coarse_coeffs<float>(const MicroArgs&, GasDev, const double*, double, double*, float*,
                                                 cudaStream_t);

// ---------------------------------------------------------------------------
// boundary faces of a cell on one sweep side (0 lower = west/south, 1 upper = east/north)
struct BFace { int bc, axis, outsign; double rS; };   // rS = face area / cell volume

// (of a fluid cell: its faces with a BC id, on the domain edge or on a body)
__device__ __forceinline__ int side_faces(const LevelDev& L, int i, int j, int side, BFace* bf)
{
    int n = 0;
    const int nx = L.nx;
    const int w = L.fbx[j * (nx + 1) + i], e = L.fbx[j * (nx + 1) + i + 1];
    const int so = L.fby[j * nx + i], no = L.fby[(j + 1) * nx + i];
    if (side != 1 && w >= 0) bf[n++] = {w, 0, -1, L.rdx[i]};
    if (side != 1 && so >= 0) bf[n++] = {so, 1, -1, L.rdy[j]};
    if (side != 0 && e >= 0) bf[n++] = {e, 0, 1, L.rdx[i]};
    if (side != 0 && no >= 0) bf[n++] = {no, 1, 1, L.rdy[j]};
    return n;
}

// ---------------------------------------------------------------------------
// The evolution smoother's sweeps.
__device__ __forceinline__ void cp_async16_if(bool on, void* sdst, const void* gsrc)   // zeros when off
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(sdst)), "l"(gsrc), "r"(on ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void ld16(const float* p, float* v)
{
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld16(const double* p, double* v)
{
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void st16(float* p, const float* v) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st16(double* p, const double* v) { *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]); }

// Walk of boundary lines.  On the sweep side of a pass, the cells of a line
// each have one boundary face of the same orientation (the domain edge's column
// and row, and runs along bodies).  A velocity that leaves through that face is
// coupled only along the line: one thread per line and leaving velocity walks the
// line (inputs streamed RA cells ahead by asynchronous copies) and keeps the values
// in S.xline, from which the wall densities (k_line_rho), the mirrored ghosts of
// symmetry faces and the line cells' final values are taken.
//
// Edge lines start in the corner cell, whose two faces couple its velocities
// (a 2x2 system for two walls, substitution otherwise): every CTA solves it for
// itself from the cell's inputs (a few loads per thread), which costs less than
// a cluster exchange.  Lines along bodies start from a cell that the wavefront
// has finished.
//
// Bound by latency: the corner, then one load latency and a short recurrence per
// RA cells.  64x64 cavity, 32x32 velocities, mixed: 11 us, and 6 us for the wall sums, against 34 us
// for the walk by clusters of eight CTAs with its fold launch that this replaces (17 us with the
// corner's sums in two rounds of loads and its divisions in one thread).  Levels of 20x8 cells and
// less, 47x13 velocities, FP64: 17 us and 6 us, against 27 us and 7 us.
template <typename F> struct EdgeRing { static constexpr int RA = 128 / (int)sizeof(F); };

// GENERAL: a symmetry or outflow face at the corner (without them the code is half as
// long, and a short kernel is mostly instruction fetches).
template <typename F, bool GENERAL>
__global__ void __launch_bounds__(128) k_sgs_edge(MicroArgs M, const double* __restrict__ Zw, const F* __restrict__ invD,
                                                  const F* __restrict__ r, const F* __restrict__ x, SweepScratch<F> S,
                                                  int pass, int q0, int nchunk)
{
    constexpr int RA = EdgeRing<F>::RA, U = 8, NB = RA / U, B = 128;
    extern __shared__ __align__(16) unsigned char esm[];
    F* ring = reinterpret_cast<F*>(esm);              // [RA][3][B]
    __shared__ F nbS[kMaxLine], itS[kMaxLine];
    __shared__ F red[sizeof(F) == 4 ? 32 : 4][4];
    const LevelDev& L = M.L;
    const VelDev& V = M.V;
    const int nx = L.nx, ny = L.ny, nv = V.nv, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t nc = L.nc, ld = V.ld;
    const F* __restrict__ vu = VelT<F>::u(V);
    const F* __restrict__ vv = VelT<F>::v(V);
    const F* __restrict__ vw = VelT<F>::w(V);
    const int q = q0 + (int)blockIdx.x / nchunk, chunk = (int)blockIdx.x % nchunk;
    // the line; the edge's two follow from the mesh (a load less before the first inputs can be asked for)
    const bool edge = q < 2;
    int i0 = pass == 0 ? 0 : nx - 1, j0 = pass == 0 ? 0 : ny - 1, di = q == 1 ? (pass == 0 ? 1 : -1) : 0,
        dj = q == 0 ? (pass == 0 ? 1 : -1) : 0, len = q == 0 ? ny : nx, axis = q, ebase = q == 0 ? 0 : ny;
    if (!edge) {
        const int* ln = M.P.lines[pass] + 8 * q;
        i0 = ln[0]; j0 = ln[1]; di = ln[2]; dj = ln[3]; len = ln[4]; axis = ln[5]; ebase = ln[6];
    }
    const long c0 = (long)j0 * nx + i0, cstep = (long)dj * nx + di;
    const F* src = pass == 0 ? r : x;
    // the velocities that leave (zero ones among them): nodes ascend, so the first (pass 0) or last ones of that axis
    const int naxis = axis == 0 ? V.nu : V.nvv, nl1 = naxis - V.nleave[1 - pass][axis], other = axis == 0 ? V.nvv : V.nu;
    const int v = chunk * B + tid;
    const bool on = v < nl1 * other;
    int k = 0;
    if (on) {
        if (axis == 0) k = (pass == 0 ? 0 : (V.nu - nl1) * V.nvv) + v;
        else { const int a = v / nl1; k = a * V.nvv + (pass == 0 ? 0 : V.nvv - nl1) + v - a * nl1; }
    }
    const long pst = cstep * (long)ld;
    const F *pi = invD + (c0 + cstep) * (long)ld + k, *ps = src + (c0 + cstep) * (long)ld + k;
    auto issue = [&](int b) {                         // cells 1 + U b .. U (b + 1), one copy group
        F* d = ring + (b % NB) * U * 3 * B + tid;
        #pragma unroll
        for (int u = 0; u < U; ++u) {
            if (1 + U * b + u < len && on) {
                cp_async_elem(d + u * 3 * B, pi);
                cp_async_elem(d + u * 3 * B + B, ps);
                cp_async_elem(d + u * 3 * B + 2 * B, ps + nc * ld);
            }
            pi += pst;
            ps += pst;
        }
        cp_async_commit();
    };
    for (int b = 0; b < NB - 1; ++b) issue(b);
    // per cell: 1/d along the line and the collision frequency, asked for early
    for (int st = tid; st < len; st += B) {
        nbS[st] = (F)(axis == 0 ? L.rdy[j0 + st * dj] : L.rdx[i0 + st * di]);
        itS[st] = (F)M.inv_tau[c0 + st * cstep];
    }
    F xp[2] = {F(0), F(0)};
    if (edge) {
        // the corner cell: face 0 its x-face, face 1 its y-face
        const int c = pass == 0 ? 0 : (int)nc - 1, ci = pass == 0 ? 0 : nx - 1, cj = pass == 0 ? 0 : ny - 1;
        const int bc0 = M.P.cbc[pass][0], bc1 = M.P.cbc[pass][1];
        const BcDev B0 = M.bc[bc0], B1 = M.bc[bc1];
        const F rx = (F)L.rdx[ci], ry = (F)L.rdy[cj], itau = (F)M.inv_tau[c];
        const bool w0 = B0.type == BC_WALL, w1 = B1.type == BC_WALL, two = w0 && w1;
        const bool y0 = GENERAL && B0.type == BC_SYMMETRY, y1 = GENERAL && B1.type == BC_SYMMETRY;
        const bool o0 = GENERAL && B0.type == BC_OUTFLOW, o1 = GENERAL && B1.type == BC_OUTFLOW;
        const F sg = pass == 0 ? F(-1) : F(1);
        // a velocity of the corner: outward normal speeds, weight, 1/D, right-hand sides, the walls' Maxwellians
        struct Vel { F ux, uy, w, den, b[2]; double C[2]; };
        const double* __restrict__ C0 = M.Cw + (size_t)bc0 * nv;
        const double* __restrict__ C1 = M.Cw + (size_t)bc1 * nv;
        auto fetch = [&](int kk, Vel& p) {           // independent loads, used once all are asked for
            p.ux = vu[kk];
            p.uy = vv[kk];
            p.w = vw[kk];
            p.den = invD[(size_t)c * ld + kk];
            p.b[0] = src[(size_t)c * ld + kk];
            p.b[1] = src[(nc + c) * ld + kk];
            p.C[0] = w0 ? C0[kk] : 0.0;
            p.C[1] = w1 ? C1[kk] : 0.0;
        };
        // coefficient of the ghost behind face f (zero unless the velocity enters there)
        auto Dg = [&](int f, const Vel& p) { return f == 0 ? mul_rn(min(p.ux, F(0)), rx) : mul_rn(min(p.uy, F(0)), ry); };
        auto finish = [&](Vel& p) {
            p.ux *= sg;
            p.uy *= sg;
            if (pass == 1 || o0 || o1) {
                const F D = itau + geomD_r<F>(rx, ry, p.ux, p.uy);
                if (o0 || o1) {
                    F d = D;
                    if (o0) d += Dg(0, p);
                    if (o1) d += Dg(1, p);
                    p.den = recip(d);
                }
                if (pass == 1) { p.b[0] = mul_rn(D, p.b[0]); p.b[1] = mul_rn(D, p.b[1]); }
            }
        };
        auto wallC = [&](int f, const Vel& p, int cp) {
            return cp == 0 ? (F)p.C[f] : (F)(p.C[f] * (kKint * (f == 0 ? B0.t : B1.t) / 4.0));
        };
        auto mirror = [&](int f, int kk) {
            const int a = kk / V.nvv, b = kk - a * V.nvv;
            return f == 0 ? (V.nu - 1 - a) * V.nvv + b : a * V.nvv + (V.nvv - 1 - b);
        };
        F rho0 = F(0), rho1 = F(0);
        if (w0 || w1) {
            // sums over the velocities: in the mixed form eight groups of row pairs (a, nu - 1 - a) a group apart, a
            // thread's share of a group in order, then warps and groups by exchange; in FP64, where the groups'
            // exchanges would take longer than the sums, a thread's velocities, then warps.  At a time RB velocities,
            // their loads in flight together.
            constexpr bool GROUPS = sizeof(F) == 4;
            constexpr int RB = GROUPS ? 8 : 4, NA = GROUPS ? 8 : 1;
            const int ngroups = (V.nu + 1) / 2, per = 2 * V.nvv, nloc = GROUPS ? (ngroups + 7) / 8 * per : nv;
            const double z0 = w0 ? Zw[bc0 * 4 + pass] : 0.0, z1 = w1 ? Zw[bc1 * 4 + 2 + pass] : 0.0;
            const F iz = (F)(Zw + 4 * kMaxBcs)[w0 ? bc0 * 4 + pass : bc1 * 4 + 2 + pass];
            F acc[NA][4];
            #pragma unroll
            for (int rr = 0; rr < NA; ++rr)
                #pragma unroll
                for (int m = 0; m < 4; ++m) acc[rr][m] = F(0);
            #pragma unroll 1
            for (int m = tid; m < nloc; m += GROUPS ? B : RB * B) {
                const int sl = m / per, rem = m - sl * per, side = rem >= V.nvv, b = rem - side * V.nvv;
                Vel p[RB];
                int kk[RB];
                #pragma unroll
                for (int rr = 0; rr < RB; ++rr) {
                    const int g = rr + sl * 8, a = side ? V.nu - 1 - g : g;
                    if (GROUPS) kk[rr] = g < ngroups && !(side && a == g) ? a * V.nvv + b : -1;
                    else kk[rr] = m + rr * B < nv ? m + rr * B : -1;
                    fetch(max(kk[rr], 0), p[rr]);
                }
                #pragma unroll
                for (int rr = 0; rr < RB; ++rr) {
                    if (kk[rr] < 0) continue;
                    F* s = acc[GROUPS ? rr : 0];
                    finish(p[rr]);
                    const F wx = mul_rn(p[rr].w, max(p[rr].ux, F(0))), wy = mul_rn(p[rr].w, max(p[rr].uy, F(0)));
                    if (two) {
                        s[0] = fma(mul_rn(wx, p[rr].b[0]), p[rr].den, s[0]);
                        s[1] = fma(mul_rn(wy, p[rr].b[0]), p[rr].den, s[1]);
                        s[2] = fma(mul_rn(mul_rn(wx, Dg(1, p[rr])), wallC(1, p[rr], 0)), p[rr].den, s[2]);
                        s[3] = fma(mul_rn(mul_rn(wy, Dg(0, p[rr])), wallC(0, p[rr], 0)), p[rr].den, s[3]);
                    } else {
                        F val = p[rr].b[0];
                        if (y0 || y1) {              // beside a symmetry face: the mirrored ghost of a velocity that enters through it
                            const F d = Dg(y0 ? 0 : 1, p[rr]);
                            if (d != F(0)) {
                                Vel mv;
                                fetch(mirror(y0 ? 0 : 1, kk[rr]), mv);
                                finish(mv);
                                val = fma(-d, mul_rn(mv.b[0], mv.den), val);
                            }
                        }
                        val = mul_rn(val, p[rr].den);
                        s[0] = fma(w0 ? wx : wy, val, s[0]);
                    }
                }
            }
            #pragma unroll
            for (int rr = 0; rr < NA; ++rr)
                #pragma unroll
                for (int m = 0; m < 4; ++m) {
                    #pragma unroll
                    for (int o = 16; o > 0; o >>= 1) acc[rr][m] += __shfl_xor_sync(0xffffffffu, acc[rr][m], o);
                    if (lane == 0) red[rr * 4 + warp][m] = acc[rr][m];
                }
            __syncthreads();
            F t[4];
            #pragma unroll
            for (int m = 0; m < 4; ++m) {
                t[m] = red[lane % (4 * NA)][m];
                #pragma unroll
                for (int o = 2 * NA; o > 0; o >>= 1) t[m] += __shfl_xor_sync(0xffffffffu, t[m], o);
            }
            // (the same in every thread)
            if (two) {
                // rho_0 = k_0 + m_0 rho_1, rho_1 = k_1 + m_1 rho_0; lane 0 .. 3 of a warp divides for k_0, k_1, m_0, m_1
                const F tl = (lane & 3) == 0 ? -t[0] : (lane & 3) == 1 ? -t[1] : (lane & 3) == 2 ? t[2] : t[3];
                const double d = (double)tl / (lane & 1 ? z1 : z0);
                const double k0 = __shfl_sync(0xffffffffu, d, 0), k1 = __shfl_sync(0xffffffffu, d, 1);
                const double m0 = __shfl_sync(0xffffffffu, d, 2), m1 = __shfl_sync(0xffffffffu, d, 3);
                const double r0 = (k0 + m0 * k1) / (1.0 - m0 * m1);
                rho0 = (F)r0;
                rho1 = (F)(k1 + m1 * r0);
            } else {
                rho0 = rho1 = -t[0] * iz;
            }
        }
        // value of a velocity with its ghosts: a wall's from its density, a symmetry face's from the mirrored velocity,
        // which leaves there and may itself enter through the other face
        auto value = [&](auto&& self, auto depth, int kk, F (&out)[2]) {
            Vel p;
            fetch(kk, p);
            finish(p);
            F a[2] = {p.b[0], p.b[1]};
            #pragma unroll
            for (int f = 0; f < 2; ++f) {
                const F d = Dg(f, p);
                if (d == F(0)) continue;
                if (f == 0 ? w0 : w1) {
                    #pragma unroll
                    for (int cp = 0; cp < 2; ++cp) a[cp] = fma(-mul_rn(d, wallC(f, p, cp)), f == 0 ? rho0 : rho1, a[cp]);
                } else if (f == 0 ? y0 : y1) {
                    if constexpr (GENERAL && decltype(depth)::value > 0) {
                        F g[2];
                        self(self, std::integral_constant<int, decltype(depth)::value - 1>(), mirror(f, kk), g);
                        #pragma unroll
                        for (int cp = 0; cp < 2; ++cp) a[cp] = fma(-d, g[cp], a[cp]);
                    }
                }
            }
            out[0] = mul_rn(a[0], p.den);
            out[1] = mul_rn(a[1], p.den);
        };
        const std::integral_constant<int, GENERAL ? 2 : 0> deep;
        if (on) value(value, deep, k, xp);
        if (q == 0) {                                // the corner's values for the wavefront, a slice per CTA
            const int per = (nv + nchunk - 1) / nchunk;
            #pragma unroll 1
            for (int kk = chunk * per + tid; kk < min(nv, (chunk + 1) * per); kk += B) {
                F t[2];
                value(value, deep, kk, t);
                S.corner[kk] = t[0];
                S.corner[ld + kk] = t[1];
            }
        }
    } else if (on) {
        xp[0] = x[c0 * ld + k];
        xp[1] = x[(nc + c0) * ld + k];
    }
    __syncthreads();                                 // nbS, itS
    // an: coefficient of the previous cell of the line; D = 1/tau + (|u|/dx + |v|/dy), the line's fixed spacing in gfix
    const F s1 = axis == 0 ? vv[k] : vu[k], an = min(pass == 0 ? -s1 : s1, F(0)), gvar = fabs(s1);
    const F gfix = axis == 0 ? mul_rn(fabs(vu[k]), (F)L.rdx[i0]) : mul_rn(fabs(vv[k]), (F)L.rdy[j0]);
    const int nbat = (len - 1 + U - 1) / U;
    F* xo = S.xline + (size_t)(ebase + 1) * 2 * ld + k;
    for (int b = 0; b < nbat; ++b) {
        issue(b + NB - 1);
        cp_async_wait_n<NB - 1>();
        const F* d = ring + (b % NB) * U * 3 * B + tid;
        #pragma unroll
        for (int u = 0; u < U; ++u) {
            const int st = 1 + U * b + u;
            if (st < len && on) {
                const F id = d[u * 3 * B], Dn = mul_rn(an, nbS[st]), D = itS[st] + fma(gvar, nbS[st], gfix);
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                    const F in = d[u * 3 * B + (1 + cp) * B];
                    xp[cp] = mul_rn(pass == 0 ? fma(-Dn, xp[cp], in) : fma(D, in, -mul_rn(Dn, xp[cp])), id);
                    xo[cp * ld] = xp[cp];
                }
                xo += 2 * ld;
            }
        }
    }
    cp_async_wait_n<0>();
}

// Wall densities of the line cells [e0, e0 + gridDim.x), rho = -sum / Z with the sum of
// w u_n x over the velocities that leave through the wall, one CTA per cell.  Order of the
// sum: eight groups of row pairs of the velocity grid, in a group P shares (128 over the
// line's cells, in FP64 eight, less those without a velocity) of eight interleaved chains
// each, a chain in order; then the chains as a tree, the shares and the groups in order.
// The tables hold the chains side by side, a step of all of them after the other, so that
// a thread's loads are known ahead.
// A kernel of its own because all of a line's walks have to be done; bound by latency
// (mixed: 64x64 cavity with 32x32 velocities 6 us, square cylinder's body lines 8 us; FP64:
// square cylinder at half size 9 us, against 22 us with as many shares as the mixed form).
template <typename F>
__global__ void __launch_bounds__(512) k_line_rho(MicroArgs M, const double* __restrict__ Zw, SweepScratch<F> S, int pass, int e0)
{
    __shared__ F part[8 * 128];                      // [group][share]
    const VelDev& V = M.V;
    const int e = e0 + (int)blockIdx.x, tid = threadIdx.x;
    const int4 lc = M.P.lcell[pass][e];              // {cell, line axis, bc id, 0 at the corner}
    const int4 ls = M.P.lsum[pass][e];               // {place in the tables, shares, steps, short chains}
    if (ls.y == 0) return;                           // no wall there: the density is not asked for
    constexpr int U = sizeof(F) == 8 ? 4 : 16;       // (512 threads in FP64: chains of a few steps)
    const int P = ls.y, nch = 64 * P;
    const F iz = (F)(Zw + 4 * kMaxBcs)[lc.z * 4 + lc.y * 2 + pass];
    const F* __restrict__ x = S.xline + (size_t)e * 2 * V.ld;
    const int* __restrict__ chain = V.chain + ls.x;
    const F* __restrict__ weight = reinterpret_cast<const F*>(V.wchain) + ls.x;
    auto finish = [&](int t, F acc) {                // the tree over the eight chains of share t / 8
        #pragma unroll
        for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((t & 7) == 0) part[t >> 3] = acc;
    };
    // U steps of a chain or one step of G chains at a time, their loads in flight together
    constexpr int G = 8;
    if (ls.w == 0) {
        for (int t = tid; t < nch; t += blockDim.x) {    // (whole warps)
            F acc = F(0);
            for (int n = 0; n < ls.z; n += U) {
                F w[U], v[U];
                int k[U];
                #pragma unroll
                for (int q = 0; q < U; ++q) {        // (a chain that has ended goes on with weight zero)
                    const int at = min(n + q, ls.z - 1) * nch + t;
                    k[q] = chain[at];
                    w[q] = n + q < ls.z ? weight[at] : F(0);
                }
                #pragma unroll
                for (int q = 0; q < U; ++q) v[q] = x[k[q]];
                #pragma unroll
                for (int q = 0; q < U; ++q) acc = w[q] != F(0) ? fma(w[q], v[q], acc) : acc;
            }
            finish(t, acc);
        }
    } else {
        for (int t0 = tid; t0 < nch; t0 += G * blockDim.x) {
            F acc[G];
            #pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = F(0);
            for (int n = 0; n < ls.z; ++n) {
                F w[G], v[G];
                int k[G];
                #pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int t = t0 + g * (int)blockDim.x, at = n * nch + min(t, nch - 1);
                    k[g] = chain[at];
                    w[g] = t < nch ? weight[at] : F(0);
                }
                #pragma unroll
                for (int g = 0; g < G; ++g) v[g] = x[k[g]];
                #pragma unroll
                for (int g = 0; g < G; ++g) acc[g] = w[g] != F(0) ? fma(w[g], v[g], acc[g]) : acc[g];
            }
            #pragma unroll
            for (int g = 0; g < G; ++g)
                if (t0 + g * (int)blockDim.x < nch) finish(t0 + g * (int)blockDim.x, acc[g]);   // (whole warps)
        }
    }
    __syncthreads();
    if (tid < 8) {
        F t = F(0);
        #pragma unroll 8
        for (int p = 0; p < P; ++p) t += part[tid * P + p];
        part[tid * P] = t;
    }
    __syncthreads();
    if (tid == 0) {
        F t = F(0);
        for (int g = 0; g < 8; ++g) t += part[g * P];
        S.rho[e] = -t * iz;
    }
}

// Wavefront steps [dd0, dd1) of one sweep over every cell.  A CTA owns 16 LPC
// bytes of consecutive velocities and the whole mesh; its warps own strips of
// 32 / LPC grid lines, LPC lanes per line, and walk along the lines one cell per
// step: the cells of a step lie on an anti-diagonal, the neighbour along the line
// is the lane's own last result, the one across comes from the line before by
// shuffles (from the strip before through a shared ring), so there is no barrier.
// Strips follow each other; their counters are looked at every kWaveChunk steps.
// Inputs stream through a ring of R steps by asynchronous copies, every lane its own.
//   forward   x = (b - C_a x_a - C_l x_l) / D, b the residual,
//   backward  x = b - (C_a x_a + C_l x_l) / D, b the forward value,
// with the coefficients zero where the neighbour lies downwind: a CTA whose
// velocities need no neighbour across hands none on, and in the backward pass
// one that needs neither only takes over the line cells' values.
// Of the two products, the neighbour's along x is fused into their sum.
// Boundary-line cells take b and 1/D from the fold, which the CTA makes for its
// velocities before it starts, from the wall densities of the line walk: the
// entries [e0, e0 + ne) of the lines walked last.  1/D = 0 marks a value that is
// final: the corner cell, a line cell's leaving velocities (the walk's own values),
// and the zeros that stand for a cell in a body or a step outside a line.  They are
// chosen, not computed, so that nothing that overflowed ahead of a body gets into
// it; a zero in the body in turn drops it as a neighbour.
// What bounds it: on large levels the L1 look-ups of the copies and stores (one per
// cell and warp access, see LPC in launch_micro_sgs), on small ones the
// instructions of a step, as an SM sub-partition has one warp.  Square cylinder,
// mixed: 8.7 ms per iteration for all levels, against 16.4 ms for the wavefront of
// 4-velocity CTAs with a barrier per diagonal and the line kernel beside it that
// this replaces; 64x64 cavity 26 us per launch against 32 us.
constexpr int kWaveChunk = 4;
constexpr int kWaveEdge = 16;                       // results of a strip's last line in flight to the next strip

// false once limit_ns of global time (or kWaitRounds looks) have gone by
__device__ __forceinline__ bool wave_wait(const int* flag, int need, uint64_t limit_ns)
{
    const unsigned a = smem_addr(flag);
    uint64_t t0 = 0;
    for (int it = 0; it < kWaitRounds; ++it) {
        int v;
        asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];\n" : "=r"(v) : "r"(a) : "memory");
        if (v >= need) return true;
        __nanosleep(20);                             // (a spinning strip takes issue slots from the working ones)
        if ((it & 31) == 31) {
            const uint64_t t = global_ns();
            if (t0 == 0) t0 = t;
            else if (t - t0 > limit_ns) return false;
        }
    }
    return false;
}
__device__ __forceinline__ void wave_post(int* flag, int v)
{
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;\n" ::"r"(smem_addr(flag)), "r"(v) : "memory");
}

// 64 bits of velocities: two floats (packed arithmetic, rounded as the scalar one) or a double
template <typename F> struct Pack;
template <> struct Pack<float> {
    using T = unsigned long long;
    static __device__ __forceinline__ T make(float a, float b) { T r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
    static __device__ __forceinline__ T splat(float a) { return make(a, a); }
    static __device__ __forceinline__ void split(T v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
    static __device__ __forceinline__ T pick(T iv, T v, T b)                // v where 1/D is given, else b
    {
        float i0, i1, v0, v1, b0, b1;
        split(iv, i0, i1);
        split(v, v0, v1);
        split(b, b0, b1);
        return make(i0 > 0.0f ? v0 : b0, i1 > 0.0f ? v1 : b1);
    }
    static __device__ __forceinline__ T load(const float* p) { return make(p[0], p[1]); }
    static __device__ __forceinline__ T mul(T a, T b) { T r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
    static __device__ __forceinline__ T add(T a, T b) { T r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
    static __device__ __forceinline__ T fma(T a, T b, T c)
    {
        T r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
        return r;
    }
};
template <> struct Pack<double> {
    using T = double;
    static __device__ __forceinline__ T pick(T iv, T v, T b) { return iv > 0.0 ? v : b; }
    static __device__ __forceinline__ T splat(double a) { return a; }
    static __device__ __forceinline__ T load(const double* p) { return p[0]; }
    static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return ::fma(a, b, c); }
};
__device__ __forceinline__ void ld_pair(const void* p, unsigned long long* v)
{
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void ld_pair(const void* p, double* v)
{
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void st_pair(void* p, const unsigned long long* v)
{
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v[0], v[1]);
}
__device__ __forceinline__ void st_pair(void* p, const double* v) { *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]); }

// the same under a predicate (a branch would have to be resolved on the path of a step)
__device__ __forceinline__ unsigned long long bits(unsigned long long v) { return v; }
__device__ __forceinline__ unsigned long long bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ void st_pair_if(bool on, void* p, unsigned long long a, unsigned long long b)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p st.global.v2.b64 [%0], {%1, %2};\n}\n"
                 ::"l"(p), "l"(a), "l"(b), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void sts_pair_if(bool on, unsigned p, unsigned long long a, unsigned long long b)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p st.shared.v2.b64 [%0], {%1, %2};\n}\n"
                 ::"r"(p), "l"(a), "l"(b), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void lds_pair_if(bool on, unsigned p, unsigned long long* v)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p ld.shared.v2.b64 {%0, %1}, [%2];\n}\n"
                 : "+l"(v[0]), "+l"(v[1]) : "r"(p), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void lds_pair_if(bool on, unsigned p, double* v)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p ld.shared.v2.f64 {%0, %1}, [%2];\n}\n"
                 : "+d"(v[0]), "+d"(v[1]) : "r"(p), "r"((unsigned)on) : "memory");
}

// Fold of the boundary-line cells [e0, e0 + ne) for the CTA's velocities (k_sgs_wave)
template <typename F, int PASS, int LPC>
__device__ void wave_fold(const MicroArgs& M, const F* __restrict__ invD, const F* __restrict__ src, const SweepScratch<F>& S,
                          F* __restrict__ fold, int k0, int e0, int ne)
{
    constexpr int V16 = 16 / (int)sizeof(F), KB = LPC * V16;            // a thread's and the CTA's velocities
    const LevelDev& L = M.L;
    const VelDev& V = M.V;
    const int nx = L.nx, nv = V.nv;
    const size_t nc = L.nc, ld = V.ld;
    const F* __restrict__ vu = VelT<F>::u(V);
    const F* __restrict__ vv = VelT<F>::v(V);
    const int part = (int)threadIdx.x % LPC;
    k0 += part * V16;
    for (int e = e0 + (int)threadIdx.x / LPC; e < e0 + ne; e += (int)blockDim.x / LPC) {
        const int4 lc = M.P.lcell[PASS][e];         // {cell, line axis, bc id, 0 at the corner}
        const int c = lc.x, axis = lc.y, i = c % nx, j = c / nx;
        F b[2][V16], iv[V16];
        const F* fin = lc.w == 0 ? S.corner : S.xline + (size_t)e * 2 * ld;   // final values: the corner, leaving velocities
        const size_t o1 = (size_t)c * ld + k0;
        ld16(src + o1, b[0]);
        ld16(src + nc * ld + o1, b[1]);
        ld16(invD + o1, iv);
        const int bc = lc.z;
        const BcDev Bc = M.bc[bc];
        const F rx = (F)L.rdx[i], ry = (F)L.rdy[j], rS = axis == 0 ? rx : ry, itau = (F)M.inv_tau[c], rho = S.rho[e];
        #pragma unroll
        for (int q = 0; q < V16; ++q) {
            const int k = k0 + q;
            const F u = vu[k], v = vv[k];
            F un = axis == 0 ? u : v;
            un = PASS == 0 ? -un : un;
            if (k >= nv) {
                b[0][q] = b[1][q] = iv[q] = F(0);
            } else if (lc.w == 0 || un >= F(0)) {
                b[0][q] = fin[k];
                b[1][q] = fin[ld + k];
                iv[q] = F(0);
            } else {
                const F Db = mul_rn(un, rS), D = itau + geomD_r<F>(rx, ry, u, v);
                F g[2] = {F(0), F(0)};
                if (Bc.type == BC_WALL) {
                    const double C = M.Cw[(size_t)bc * nv + k];
                    g[0] = mul_rn(Db, mul_rn((F)C, rho));
                    g[1] = mul_rn(Db, mul_rn((F)(C * (kKint * Bc.t / 4.0)), rho));
                } else if (Bc.type == BC_SYMMETRY) {
                    const int a2 = k / V.nvv, b2 = k - a2 * V.nvv;
                    const int km = axis == 0 ? (V.nu - 1 - a2) * V.nvv + b2 : a2 * V.nvv + (V.nvv - 1 - b2);
                    g[0] = mul_rn(Db, fin[km]);
                    g[1] = mul_rn(Db, fin[ld + km]);
                } else if (Bc.type == BC_OUTFLOW) {
                    iv[q] = recip(D + Db);
                }
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp) b[cp][q] = PASS == 0 ? b[cp][q] - g[cp] : fma(D, b[cp][q], -g[cp]) * iv[q];
            }
        }
        F* o = fold + (size_t)e * 3 * KB + part * V16;
        st16(o, b[0]);
        st16(o + KB, b[1]);
        st16(o + 2 * KB, iv);
    }
}

// LPC: lanes per cell, 16 bytes of velocities each; XL: the lines are columns
template <typename F, int R, int PASS, bool BODIES, int LPC, bool XL>
__global__ void __launch_bounds__(512) k_sgs_wave(MicroArgs M, const F* __restrict__ invD, const F* __restrict__ r,
                                                  F* __restrict__ x, SweepScratch<F> S, int dd0, int dd1, int e0, int ne)
{
    using P = Pack<F>;
    using T = typename P::T;
    constexpr int V16 = 16 / (int)sizeof(F), K = LPC * V16, NL = 32 / LPC, step_bytes = 3 * 512, ebytes = 32 * LPC;
    extern __shared__ __align__(16) unsigned char wsm[];
    const LevelDev& L = M.L;
    const VelDev& V = M.V;
    const int nx = L.nx, ny = L.ny, k0 = (int)blockIdx.x * K;
    const int ns = XL ? nx : ny, nt = XL ? ny : nx, nw = (int)blockDim.x >> 5;
    const size_t nc = L.nc, ld = V.ld;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, ll = lane / LPC, part = lane % LPC, s = NL * w + ll;
    unsigned char* ring = wsm + (size_t)w * R * step_bytes + lane * 16;
    unsigned char* edges = wsm + (size_t)nw * R * step_bytes;                   // [strip][kWaveEdge][2][LPC] x 16 bytes
    F* ral = reinterpret_cast<F*>(edges + (size_t)nw * kWaveEdge * ebytes);     // [nt] -1/d along the lines
    int* prog = reinterpret_cast<int*>(ral + nt);                               // per strip: edge values there
    int* cons = prog + nw;                                                      // per strip: edge values taken
    if (M.wait_ns == 0) {                           // gives up before its first step
        if (threadIdx.x == 0) *M.flag = 1.0;
        return;
    }
    const F* src = PASS == 0 ? r : x;
    const F* __restrict__ vu = VelT<F>::u(V);
    const F* __restrict__ vv = VelT<F>::v(V);
    const int kl = k0 + part * V16;                 // first velocity of this lane
    // coefficients per unit face: across and along the lines (zero where that neighbour lies downwind)
    F ca[V16], cl[V16];
    bool any_a = false, any_l = false;
    #pragma unroll
    for (int q = 0; q < V16; ++q) {
        const F u = vu[kl + q], v = vv[kl + q];     // the tables are padded with zeros
        const F cu = min(PASS == 0 ? -u : u, F(0)), cv = min(PASS == 0 ? -v : v, F(0));
        ca[q] = XL ? cu : cv;
        cl[q] = XL ? cv : cu;
        any_a = any_a || ca[q] != F(0);
        any_l = any_l || cl[q] != F(0);
    }
    any_a = __any_sync(0xffffffffu, any_a);
    any_l = __any_sync(0xffffffffu, any_l);
    F* fold = S.fold + (size_t)blockIdx.x * S.nl * 3 * K;
    wave_fold<F, PASS, LPC>(M, invD, src, S, fold, k0, e0, ne);
    if (PASS == 1 && !any_a && !any_l) {            // (the same in every warp)
        for (int e = e0 + (int)threadIdx.x / LPC; e < e0 + ne; e += (int)blockDim.x / LPC) {   // (a thread's own entries)
            const size_t o = (size_t)M.P.lcell[PASS][e].x * ld + kl;
            const F* f = fold + (size_t)e * 3 * K + part * V16;
            F v[V16];
            ld16(f, v);
            st16(x + o, v);
            ld16(f + K, v);
            st16(x + nc * ld + o, v);
        }
        return;
    }
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
        const int p = PASS == 0 ? t : nt - 1 - t;
        ral[t] = -(F)(XL ? L.rdy[p] : L.rdx[p]);
    }
    if (lane == 0) prog[w] = cons[w] = max(0, dd0 + 1 - NL * w);
    __threadfence();                                // the fold is read by asynchronous copies of other threads
    __syncthreads();
    // ---- this strip's steps of the segment: step k sweeps the strip's diagonal NL w + k
    const int kb = max(0, dd0 - NL * w), ke = min(nt + NL - 1, dd1 - NL * w);
    if (kb >= ke) return;
    const bool line = s < ns;
    const int sp = PASS == 0 ? s : ns - 1 - s, tp = PASS == 0 ? 0 : nt - 1;
    const long cfirst = line ? (XL ? (long)tp * nx + sp : (long)sp * nx + tp) : 0;   // the line's cell t = 0
    const long cst = (PASS == 0 ? 1 : -1) * (XL ? (long)nx : 1L);
    const long pst = cst * (long)ld;                // from a cell of the line to the next, in values
    const F rac = line && s > 0 ? -(XL ? (F)L.rdx[sp] : (F)L.rdy[sp]) : F(0);
    T nca[2], ncl[2];
    #pragma unroll
    for (int q = 0; q < V16; ++q) ca[q] *= rac;
    #pragma unroll
    for (int q = 0; q < 2; ++q) { nca[q] = P::load(ca + q * (V16 / 2)); ncl[q] = P::load(cl + q * (V16 / 2)); }
    const int ea = XL ? 0 : ny, eb = XL ? ny + s : s;   // fold entries of line 0 (+ t) and of the cells t = 0
    const int* __restrict__ code = M.P.code[PASS];
    auto code_of = [&](int k) {
        const int t = k - ll;
        return line && (unsigned)t < (unsigned)nt && k < ke ? code[cfirst + t * cst] : -2;
    };
    int cd0 = 0, cd1 = 0, cd2 = 0, cd3 = 0;         // codes of the next four cells to be copied
    if constexpr (BODIES) { cd0 = code_of(kb); cd1 = code_of(kb + 1); cd2 = code_of(kb + 2); cd3 = code_of(kb + 3); }
    const size_t hoff = nc * ld;
    // running addresses of the next cell to be copied (before and after the line they are not used)
    const F* pb = src + (cfirst + (kb - ll) * cst) * (long)ld + kl;
    const F* pi = invD + (cfirst + (kb - ll) * cst) * (long)ld + kl;
    const F* safe = src + kl;
    auto issue = [&](int k, int stage) {
        const int t = k - ll;
        bool on = line && (unsigned)t < (unsigned)nt && k < ke;
        const F *p0 = pb, *p1 = pb + hoff, *p2 = pi;
        pb += pst;
        pi += pst;
        if constexpr (BODIES) {
            on = on && cd0 != -2;
            if (cd0 >= 0) {
                p0 = fold + (long)cd0 * 3 * K + part * V16;
                p1 = p0 + K;
                p2 = p0 + 2 * K;
            }
            cd0 = cd1; cd1 = cd2; cd2 = cd3; cd3 = code_of(k + 4);
        } else if (w == 0 || k < NL) {              // (the other steps of a strip hold no line cell)
            if (s == 0 || t == 0) {
                p0 = fold + (long)(s == 0 ? ea + t : eb) * 3 * K + part * V16;
                p1 = p0 + K;
                p2 = p0 + 2 * K;
            }
        }
        if (!on) p0 = p1 = p2 = safe;               // nothing is read from it
        unsigned char* d = ring + stage * step_bytes;
        cp_async16_if(on, d, p0);
        cp_async16_if(on, d + 512, p1);
        cp_async16_if(on, d + 1024, p2);
        cp_async_commit();
    };
    T ac[2][2], al[2][2];
    #pragma unroll
    for (int q = 0; q < 2; ++q) ac[0][q] = ac[1][q] = al[0][q] = al[1][q] = P::splat(F(0));
    #pragma unroll
    for (int q = 0; q < R - 1; ++q) issue(kb + q, q);
    if (dd0 > 0 && kb + NL * w == dd0) {
        // the segment goes on from the diagonal before it
        const int t = kb - ll;
        const bool hl = line && t >= 1 && t <= nt, ha = s >= 1 && s <= ns && t >= 0 && t < nt;
        const long c_l = cfirst + (long)(t - 1) * cst;
        const int sa = PASS == 0 ? s - 1 : ns - s, ta = PASS == 0 ? t : nt - 1 - t;
        const long c_a = XL ? (long)ta * nx + sa : (long)sa * nx + ta;
        #pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
            if (hl) ld_pair(x + (cp * nc + c_l) * ld + kl, al[cp]);
            if (ha) ld_pair(x + (cp * nc + c_a) * ld + kl, ac[cp]);
        }
    }
    const bool takes = any_a && w > 0, feeds = any_a && w + 1 < nw;
    const int tfirst = max(0, dd0 + 1 - NL * w);    // edge values from here on come through the ring
    const unsigned etake = smem_addr(edges + (size_t)w * kWaveEdge * ebytes + part * 32);
    const unsigned efeed = smem_addr(edges + (size_t)(w + 1) * kWaveEdge * ebytes + part * 32);
    F* xo = x + (cfirst + (kb - ll) * cst) * (long)ld + kl;
    for (int kc = kb; kc < ke; kc += 8) {
        #pragma unroll
        for (int kk = 0; kk < 8; ++kk) {             // steps beyond ke copy zeros and store nothing
            const int k = kc + kk, t = k - ll;
            if (kk % kWaveChunk == 0) {
                const int kn = min(k + kWaveChunk, ke);
                bool got = true;
                if (takes) got = wave_wait(prog + w, min(nt, kn), M.wait_ns);
                if (feeds) got = got && wave_wait(cons + w + 1, min(nt, kn - (NL - 1)) - kWaveEdge, M.wait_ns);
                if (!__all_sync(0xffffffffu, got)) { if (lane == 0) *M.flag = 1.0; cp_async_wait_n<0>(); return; }
            }
            cp_async_wait_n<R - 2>();
            T b[2][2], iv[2];
            const unsigned char* d = ring + (kk % R) * step_bytes;
            ld_pair(d, b[0]);
            ld_pair(d + 512, b[1]);
            ld_pair(d + 1024, iv);
            const bool tk = takes && ll == 0 && k >= tfirst && k < nt;
            const unsigned ea_ = etake + (unsigned)(k % kWaveEdge) * ebytes;
            lds_pair_if(tk, ea_, ac[0]);
            lds_pair_if(tk, ea_ + 16, ac[1]);
            issue(k + R - 1, (kk + R - 1) % R);
            // minus the neighbours' terms (line 0 has no neighbour across: its coefficient is zero)
            const T ra = P::splat(ral[min(max(t, 0), nt - 1)]);
            #pragma unroll
            for (int q = 0; q < 2; ++q) {
                const T g = P::mul(ncl[q], ra);
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                    const T n = XL ? P::fma(nca[q], ac[cp][q], P::mul(g, al[cp][q])) : P::fma(g, al[cp][q], P::mul(nca[q], ac[cp][q]));
                    al[cp][q] = PASS == 0 ? P::mul(P::add(b[cp][q], n), iv[q]) : P::fma(n, iv[q], b[cp][q]);
                }
            }
            if (BODIES || w == 0 || k < NL)          // (the other steps of a strip hold no final value)
                #pragma unroll
                for (int q = 0; q < 2; ++q) {
                    al[0][q] = P::pick(iv[q], al[0][q], b[0][q]);
                    al[1][q] = P::pick(iv[q], al[1][q], b[1][q]);
                }
            const bool on = line && (unsigned)t < (unsigned)nt && k < ke;
            st_pair_if(on, xo, bits(al[0][0]), bits(al[0][1]));
            st_pair_if(on, xo + hoff, bits(al[1][0]), bits(al[1][1]));
            xo += pst;
            if (any_a) {
                const bool fd = feeds && ll == NL - 1 && on;
                const unsigned ed = efeed + (unsigned)(t & (kWaveEdge - 1)) * ebytes;
                sts_pair_if(fd, ed, bits(al[0][0]), bits(al[0][1]));
                sts_pair_if(fd, ed + 16, bits(al[1][0]), bits(al[1][1]));
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp)
                    #pragma unroll
                    for (int q = 0; q < 2; ++q) ac[cp][q] = __shfl_up_sync(0xffffffffu, al[cp][q], LPC);
            }
            if ((kk + 1) % kWaveChunk == 0 && (feeds || takes)) {
                const int kn = min(k + 1, ke);
                __syncwarp();                        // every lane's edge values are stored, or read
                if (feeds && lane == 31) wave_post(prog + w + 1, min(nt, kn - (NL - 1)));
                if (takes && lane == 0) wave_post(cons + w, min(nt, kn));
            }
        }
    }
    cp_async_wait_n<0>();
}

// sweep scratch: values of the storage type per solver (the largest level)
size_t micro_scratch_elems(int ld, int nl)
{
    return 2 * (size_t)ld + (((size_t)nl + 15) & ~(size_t)15) + 5 * (size_t)ld * nl;
}
template <typename F>
SweepScratch<F> sweep_scratch(F* base, int ld, int nl)
{
    SweepScratch<F> S;
    S.corner = base;
    S.rho = S.corner + 2 * (size_t)ld;
    S.fold = S.rho + (((size_t)nl + 15) & ~(size_t)15);
    S.xline = S.fold + 3 * (size_t)ld * nl;
    S.nl = nl;
    return S;
}
// CTAs of the line walk per line: the leaving velocities of a pass and axis, zero ones among them
static int edge_chunks(const VelDev& V)
{
    int m = 1;
    for (int p = 0; p < 2; ++p)
        for (int a = 0; a < 2; ++a)
            m = std::max(m, (((a == 0 ? V.nu : V.nvv) - V.nleave[1 - p][a]) * (a == 0 ? V.nvv : V.nu) + 127) / 128);
    return m;
}

template <typename F>
cudaError_t launch_micro_sgs(const MicroArgs& m, const SweepPlanHost& plan, const double* Zw, const F* invD,
                             const F* r, F* x, F* scratch, cudaStream_t st)
{
    if (m.L.nx > kMaxLine || m.L.ny > kMaxLine) return cudaErrorInvalidValue;
    const int ns = std::min(m.L.nx, m.L.ny), nt = std::max(m.L.nx, m.L.ny), nchunk = edge_chunks(m.V);
    const SweepScratch<F> S = sweep_scratch<F>(scratch, m.V.ld, plan.nl);
    constexpr size_t kSmemMax = 227 * 1024;
    constexpr size_t esmem = sizeof(F) * EdgeRing<F>::RA * 3 * 128;
    // Lanes per cell: an asynchronous copy or store of a warp costs its SM's L1 one look-up per cell, so
    // the more lanes share a cell the better (64 bytes of a cell with four), as long as the strips fit a
    // CTA of 16 warps and the CTAs fill the SMs.  Finest level and coarser ones together, per
    // iteration, 1 / 2 / 4 lanes: square cylinder mixed 21.5 / 12.6 / 8.7 ms, plate mixed 2.8 / 2.0 / 1.6 ms;
    // 64x64 cavity with 32x32 velocities (64 CTAs with four lanes) 0.55 / 0.53 / 0.58 ms.
    constexpr int V16 = 16 / (int)sizeof(F);
    const int LPC = ns <= 128 && m.V.ld / (4 * V16) > 128 ? 4 : ns <= 256 ? 2 : 1;
    if (m.V.ld % (LPC * V16)) return cudaErrorInvalidValue;   // a block of velocities would leave its row
    const int nblk = m.V.ld / (LPC * V16), nw = (ns * LPC + 31) / 32;
    // ring depth: eight steps in flight where they fit, else four
    const size_t fixed = (size_t)nw * kWaveEdge * 32 * LPC + sizeof(F) * nt + 2 * sizeof(int) * nw + 16, slot = (size_t)nw * 1536;
    const int R = fixed + 8 * slot <= kSmemMax ? 8 : 4;
    const size_t wsmem = fixed + R * slot;
    if (wsmem > kSmemMax) return cudaErrorInvalidValue;
    using Wave = void (*)(MicroArgs, const F*, const F*, F*, SweepScratch<F>, int, int, int, int);
    const bool xl = m.L.nx <= m.L.ny;
    if (R == 4 && LPC != 4) return cudaErrorInvalidValue;   // (eight steps always fit with fewer lanes)
    auto pick = [&](auto h, auto bodies, auto cols) {
        constexpr int HH = decltype(h)::value;
        constexpr bool BB = decltype(bodies)::value, XX = decltype(cols)::value;
        std::array<Wave, 2> f = {k_sgs_wave<F, 8, 0, BB, HH, XX>, k_sgs_wave<F, 8, 1, BB, HH, XX>};
        if constexpr (HH == 4)
            if (R == 4) f = {k_sgs_wave<F, 4, 0, BB, HH, XX>, k_sgs_wave<F, 4, 1, BB, HH, XX>};
        return f;
    };
    auto by_lanes = [&](auto bodies, auto cols) {
        return LPC == 4 ? pick(std::integral_constant<int, 4>(), bodies, cols)
               : LPC == 2 ? pick(std::integral_constant<int, 2>(), bodies, cols) : pick(std::integral_constant<int, 1>(), bodies, cols);
    };
    auto by_axis = [&](auto bodies) { return xl ? by_lanes(bodies, std::true_type()) : by_lanes(bodies, std::false_type()); };
    const std::array<Wave, 2> wave = m.P.bodies ? by_axis(std::true_type()) : by_axis(std::false_type());
    for (int p = 0; p < 2; ++p) {
        const cudaError_t e = allow_shared_memory((const void*)wave[p]);
        if (e != cudaSuccess) return e;
    }
    using Edge = void (*)(MicroArgs, const double*, const F*, const F*, const F*, SweepScratch<F>, int, int, int);
    const Edge walk[2] = {k_sgs_edge<F, false>, k_sgs_edge<F, true>};
    cudaError_t e = cudaSuccess;
    for (int g = 0; g < 2; ++g)
        if ((e = allow_shared_memory((const void*)walk[g])) != cudaSuccess) return e;
    // timing mode: an event pair around a launch, with the cell-velocity pairs it sweeps
    auto timed = [&](double units, auto&& launch) {
        SweepTimer* T = plan.timer;
        if (!T) { launch(); return cudaGetLastError(); }
        while ((int)T->ev.size() < 2 * (T->used + 1)) {
            cudaEvent_t ev;
            cudaError_t ce = cudaEventCreate(&ev);
            if (ce != cudaSuccess) return ce;
            T->ev.push_back(ev);
        }
        if ((int)T->units.size() <= T->used) T->units.resize(T->used + 1);
        cudaError_t ce = cudaEventRecord(T->ev[2 * T->used], st);
        if (ce != cudaSuccess) return ce;
        launch();
        if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
        if ((ce = cudaEventRecord(T->ev[2 * T->used + 1], st)) != cudaSuccess) return ce;
        T->units[T->used] = units;
        T->used++;
        return cudaSuccess;
    };
    const int nd = m.L.nx + m.L.ny - 1;
    for (int pass = 0; pass < 2; ++pass) {
        walk[m.P.general[pass]]<<<2 * nchunk, 128, esmem, st>>>(m, Zw, invD, r, x, S, pass, 0, nchunk);
        // (a thread per chain, up to 512)
        if (m.P.shares[pass]) k_line_rho<F><<<m.P.nl[pass], std::min(512, 64 * m.P.shares[pass]), 0, st>>>(m, Zw, S, pass, 0);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // wavefront segments between the body lines' walks
        int dd = 0, e0 = 0, ne = m.P.nl[pass];
        for (int b = 0; b <= plan.nbrk[pass]; ++b) {
            const int end = b < plan.nbrk[pass] ? plan.brk[pass][b].dd : nd;
            double cells = 0.0;                        // cells on the segment's diagonals
            for (int q = dd; q < end; ++q) {
                const int d = pass == 0 ? q : nd - 1 - q;
                cells += std::min(m.L.nx - 1, d) - std::max(0, d - (m.L.ny - 1)) + 1;
            }
            if ((e = timed(cells * m.V.nv, [&] {
                    wave[pass]<<<nblk, 32 * nw, wsmem, st>>>(m, invD, r, x, S, dd, end, e0, ne);
                })) != cudaSuccess)
                return e;
            dd = end;
            if (b < plan.nbrk[pass]) {
                const SweepBreak& k = plan.brk[pass][b];
                walk[m.P.general[pass]]<<<k.nq * nchunk, 128, esmem, st>>>(m, Zw, invD, r, x, S, pass, 2 + k.q0, nchunk);
                if (k.shares) k_line_rho<F><<<k.ne, std::min(512, 64 * k.shares), 0, st>>>(m, Zw, S, pass, k.e0);
                if ((e = cudaGetLastError()) != cudaSuccess) return e;
                e0 = k.e0;
                ne = k.ne;
            }
        }
    }
    return cudaSuccess;
}
template cudaError_t launch_micro_sgs<double>(const MicroArgs&, const SweepPlanHost&, const double*, const double*,
                                              const double*, double*, double*, cudaStream_t);
template cudaError_t launch_micro_sgs<float>(const MicroArgs&, const SweepPlanHost&, const double*, const float*,
                                             const float*, float*, float*, cudaStream_t);

// Sum of squares of n values (deterministic: fixed grid, fixed per-thread order,
// fixed reduction tree), for the decisions of the adaptive multigrid cycle.
constexpr int kSumsqBlocks = 128;
template <typename T>
__global__ void k_sumsq_part(const T* __restrict__ a, size_t n, double* __restrict__ part)
{
    __shared__ double red[32];
    double s[1] = {0.0};
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
        const double v = (double)a[q];
        s[0] += v * v;
    }
    block_sum<1>(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}
__global__ void k_sumsq_final(const double* __restrict__ part, int nb, double* __restrict__ out)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double t = 0.0;
        for (int b = 0; b < nb; ++b) t += part[b];
        *out = t;
    }
}
template <typename T>
cudaError_t launch_sumsq(const T* a, size_t n, double* part, double* out, cudaStream_t st)
{
    k_sumsq_part<T><<<kSumsqBlocks, 256, 0, st>>>(a, n, part);
    k_sumsq_final<<<1, 32, 0, st>>>(part, kSumsqBlocks, out);
    return cudaGetLastError();
}
template cudaError_t launch_sumsq<float>(const float*, size_t, double*, double*, cudaStream_t);
template cudaError_t launch_sumsq<double>(const double*, size_t, double*, double*, cudaStream_t);

// ---------------------------------------------------------------------------
// r -= A x (full operator with every neighbour and ghost), acc += x
template <typename F>
__global__ void __launch_bounds__(256) k_micro_renew(MicroArgs M, const double* __restrict__ Zw, const F* __restrict__ x,
                                                     F* __restrict__ r, F* __restrict__ acc, int renew)
{
    __shared__ double red[32 * 4];
    const LevelDev& L = M.L;
    const VelDev& Vg = M.V;
    const int c = blockIdx.x, nx = L.nx, nv = Vg.ld, i = c % nx, j = c / nx;   // rows with their padding
    const size_t nc = L.nc;
    constexpr int V16 = 16 / (int)sizeof(F);
    const bool inner = renew && !L.solid[c] && L.fbx[j * (nx + 1) + i] < 0 && L.fbx[j * (nx + 1) + i + 1] < 0 &&
                       L.fby[j * nx + i] < 0 && L.fby[(j + 1) * nx + i] < 0;
    if (inner) {
        // A cell without boundary faces.
        const F* __restrict__ vu = VelT<F>::u(Vg);
        const F* __restrict__ vv = VelT<F>::v(Vg);
        const F itau = (F)M.inv_tau[c], rdxi = (F)L.rdx[i], rdyj = (F)L.rdy[j];
        const size_t hoff = nc * (size_t)nv, xrow = (size_t)nx * nv;
        const F* xb = x + (size_t)c * nv;
        F* rb = r + (size_t)c * nv;
        F* ab = acc ? acc + (size_t)c * nv : nullptr;
        if constexpr (sizeof(F) == 4) {
            // FP32 is bound by memory: all four neighbours are read, so that every load can be issued at
            // once (choosing the two that a velocity sees first made the square cylinder's renewals
            // 16.0 -> 21.6 ms per three iterations)
            const bool four = (Vg.nv & 3) == 0;
            for (int k0 = threadIdx.x * V16; k0 < nv; k0 += blockDim.x * V16) {
                F u[V16], v[V16], cW[V16], cE[V16], cS[V16], cN[V16], dg[V16];
                ld16(vu + k0, u);
                ld16(vv + k0, v);
                #pragma unroll
                for (int q = 0; q < V16; ++q) {
                    dg[q] = itau + geomD_r<F>(rdxi, rdyj, u[q], v[q]);
                    cW[q] = min(-u[q], F(0)) * rdxi;
                    cE[q] = min(u[q], F(0)) * rdxi;
                    cS[q] = min(-v[q], F(0)) * rdyj;
                    cN[q] = min(v[q], F(0)) * rdyj;
                }
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                    const F* p = xb + cp * hoff + k0;
                    F xc[V16], xw[V16], xe[V16], xs[V16], xn[V16], rr[V16], aa[V16];
                    ld16(p, xc);
                    ld16(p - nv, xw);
                    ld16(p + nv, xe);
                    ld16(p - xrow, xs);
                    ld16(p + xrow, xn);
                    ld16(rb + cp * hoff + k0, rr);
                    if (ab) ld16(ab + cp * hoff + k0, aa);
                    #pragma unroll
                    for (int q = 0; q < V16; ++q) {
                        // (which of the first two products is rounded before the sum follows the row's length)
                        F a = four ? fma(dg[q], xc[q], mul_rn(cW[q], xw[q])) : fma(cW[q], xw[q], mul_rn(dg[q], xc[q]));
                        a = fma(cE[q], xe[q], a);
                        a = fma(cS[q], xs[q], a);
                        a = fma(cN[q], xn[q], a);
                        rr[q] = rr[q] - a;
                        aa[q] = ab ? aa[q] + xc[q] : F(0);
                    }
                    st16(rb + cp * hoff + k0, rr);
                    if (ab) st16(ab + cp * hoff + k0, aa);
                }
            }
            return;
        }
        // FP64 is bound by its arithmetic: of its four neighbours a velocity sees the two it comes from, and
        // the other two are neither read nor multiplied.  Where the velocities of an access (16 bytes) come
        // from the same sides, which their index tells, the access is one group; else one by one.
        // (64x64 cavity with 32x32 velocities 252 -> 158 us on the finest level, half-size square cylinder
        // 22.0 -> 16.2 ms per two iterations)
        const int nvv = Vg.nvv, nun = Vg.nleave[0][0], nvn = Vg.nleave[0][1];
        for (int k0 = threadIdx.x * V16; k0 < Vg.nv; k0 += blockDim.x * V16) {
            const int a = k0 / nvv, b = k0 - a * nvv;
            if (b + V16 <= nvv && (b >= nvn || b + V16 <= nvn)) {
                const F* pu = xb + k0 + (a < nun ? (long)nv : -(long)nv);
                const F* pv = xb + k0 + (b < nvn ? (long)xrow : -(long)xrow);
                F u[V16], v[V16], xc[2][V16], xu[2][V16], xv[2][V16], rr[2][V16], aa[2][V16];
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                    ld16(xb + cp * hoff + k0, xc[cp]);
                    ld16(pu + cp * hoff, xu[cp]);
                    ld16(pv + cp * hoff, xv[cp]);
                    ld16(rb + cp * hoff + k0, rr[cp]);
                    if (ab) ld16(ab + cp * hoff + k0, aa[cp]);
                }
                ld16(vu + k0, u);
                ld16(vv + k0, v);
                #pragma unroll
                for (int q = 0; q < V16; ++q) {
                    const F du = fabs(u[q]) * rdxi, dv = fabs(v[q]) * rdyj, dg = itau + (du + dv);
                    #pragma unroll
                    for (int cp = 0; cp < 2; ++cp) {
                        rr[cp][q] -= fma(-dv, xv[cp][q], fma(-du, xu[cp][q], dg * xc[cp][q]));
                        if (ab) aa[cp][q] += xc[cp][q];
                    }
                }
                #pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                    st16(rb + cp * hoff + k0, rr[cp]);
                    if (ab) st16(ab + cp * hoff + k0, aa[cp]);
                }
            } else {
                #pragma unroll 1
                for (int k = k0; k < min(k0 + V16, Vg.nv); ++k) {
                    const F u = vu[k], v = vv[k], du = fabs(u) * rdxi, dv = fabs(v) * rdyj, dg = itau + (du + dv);
                    const long ou = u < F(0) ? (long)nv : -(long)nv, ov = v < F(0) ? (long)xrow : -(long)xrow;
                    for (int cp = 0; cp < 2; ++cp) {
                        const F* p = xb + cp * hoff + k;
                        rb[cp * hoff + k] -= fma(-dv, p[ov], fma(-du, p[ou], dg * p[0]));
                        if (ab) ab[cp * hoff + k] += p[0];
                    }
                }
            }
        }
        return;
    }
    if (acc)
        for (int cp = 0; cp < 2; ++cp)
            for (int k0 = threadIdx.x * V16; k0 < nv; k0 += blockDim.x * V16) {
                const size_t id = (cp * nc + c) * nv + k0;
                F xa[V16], aa[V16];
                ld16(x + id, xa);
                ld16(acc + id, aa);
                #pragma unroll
                for (int q = 0; q < V16; ++q) aa[q] += xa[q];
                st16(acc + id, aa);
            }
    if (!renew || L.solid[c]) return;   // a body keeps a zero residual
    BFace bf[4];
    int nb = side_faces(L, i, j, 2, bf);
    __shared__ F srho[4], sgeo[3];
    const F* __restrict__ vu = VelT<F>::u(Vg);
    const F* __restrict__ vv = VelT<F>::v(Vg);
    const F* __restrict__ vw = VelT<F>::w(Vg);
    int nwall = 0;
    for (int b = 0; b < nb; ++b) nwall += M.bc[bf[b].bc].type == BC_WALL;
    if (nwall > 0) {
        Acc<F> sa[4];
        for (int k = threadIdx.x; k < Vg.nv; k += blockDim.x)
            for (int b = 0; b < nb; ++b) {
                if (M.bc[bf[b].bc].type != BC_WALL) continue;
                F uo = bf[b].axis == 0 ? vu[k] : vv[k];
                uo = bf[b].outsign < 0 ? -uo : uo;
                if (uo > F(0)) sa[b].add(vw[k] * uo * x[c * (size_t)nv + k]);
            }
        double sd[4];
        block_total<4>(sa, red, sd);
        if (threadIdx.x == 0)
            for (int b = 0; b < 4; ++b)
                srho[b] = b < nb && M.bc[bf[b].bc].type == BC_WALL
                              ? (F)(-sd[b] / Zw[bf[b].bc * 4 + bf[b].axis * 2 + (bf[b].outsign > 0)]) : F(0);
    }
    if (threadIdx.x == 0) {
        sgeo[0] = (F)M.inv_tau[c]; sgeo[1] = (F)L.rdx[i]; sgeo[2] = (F)L.rdy[j];
        if (nwall == 0) srho[0] = srho[1] = srho[2] = srho[3] = F(0);
    }
    __syncthreads();
    F rho[4] = {srho[0], srho[1], srho[2], srho[3]};
    const F itau = sgeo[0], rdxi = sgeo[1], rdyj = sgeo[2];
    // interior neighbours (faces without a BC id)
    const bool hw = L.fbx[j * (nx + 1) + i] < 0, he = L.fbx[j * (nx + 1) + i + 1] < 0;
    const bool hs = L.fby[j * nx + i] < 0, hn = L.fby[(j + 1) * nx + i] < 0;
    for (int cp = 0; cp < 2; ++cp) {
        const F* xb = x + cp * nc * nv;
        F* rb = r + cp * nc * nv;
        for (int k = threadIdx.x; k < Vg.nv; k += blockDim.x) {
            const F u = vu[k], v = vv[k];
            size_t id = (size_t)c * nv + k;
            F a = (itau + geomD_r<F>(rdxi, rdyj, u, v)) * xb[id];
            if (hw) a += Dface<F>(0, -1, rdxi, u, v) * xb[id - nv];
            if (he) a += Dface<F>(0, 1, rdxi, u, v) * xb[id + nv];
            if (hs) a += Dface<F>(1, -1, rdyj, u, v) * xb[id - (size_t)nx * nv];
            if (hn) a += Dface<F>(1, 1, rdyj, u, v) * xb[id + (size_t)nx * nv];
            for (int b = 0; b < nb; ++b) {
                F Db = Dface<F>(bf[b].axis, bf[b].outsign, (F)bf[b].rS, u, v);
                if (Db == F(0)) continue;
                int ty = M.bc[bf[b].bc].type;
                if (ty == BC_WALL)
                    a += Db * (F)(M.Cw[(size_t)bf[b].bc * Vg.nv + k] * (cp == 0 ? 1.0 : kKint * M.bc[bf[b].bc].t / 4.0)) * rho[b];
                else if (ty == BC_SYMMETRY) {
                    int aa = k / Vg.nvv, bb = k - aa * Vg.nvv;
                    int km = bf[b].axis == 0 ? (Vg.nu - 1 - aa) * Vg.nvv + bb : aa * Vg.nvv + (Vg.nvv - 1 - bb);
                    a += Db * xb[(size_t)c * nv + km];
                } else if (ty == BC_OUTFLOW) {
                    a += Db * xb[id];
                }
            }
            rb[id] = rb[id] - a;
        }
    }
}

template <typename F>
cudaError_t launch_micro_renew(const MicroArgs& m, const double* Zw, const F* x, F* r, F* acc, int renew,
                                 cudaStream_t st)
{
    k_micro_renew<F><<<m.L.nc, m.V.nv >= 256 ? 256 : 128, 0, st>>>(m, Zw, x, r, acc, renew);
    return cudaGetLastError();
}
template cudaError_t launch_micro_renew<double>(const MicroArgs&, const double*, const double*, double*, double*,
                                                int, cudaStream_t);
template cudaError_t launch_micro_renew<float>(const MicroArgs&, const double*, const float*, float*, float*, int,
                                               cudaStream_t);

// ---------------------------------------------------------------------------
// Steps 6-7: f += df (when df != null), then W = sum w psi f and q = sum w c (c^2 G/2 + H)
template <typename F>
__global__ void __launch_bounds__(256) k_update_moments(LevelDev L, VelDev Vg, F* __restrict__ f, const F* __restrict__ df,
                                                        double* __restrict__ W, double* __restrict__ q)
{
    // Two passes over f + df: its moments, then, about the velocity they give, the heat flux, which also
    // commits f + df.  W and q depend on the committed f alone, so that a state read back gives the same.
    // FP64 is bound by its products and shares their factors; in the mixed form each term keeps its own
    // products and roundings, which the prediction amplifies from a marginally stable start.
    __shared__ double red[32 * 4];
    __shared__ F sUV[2];
    __shared__ int sok;
    const int c = blockIdx.x, nv = Vg.nv, bs = blockDim.x;
    const size_t nc = L.nc, ld = Vg.ld;
    F* fG = f + (size_t)c * ld;
    F* fH = f + (nc + c) * ld;
    const F* dG = df ? df + (size_t)c * ld : nullptr;
    const F* dH = df ? df + (nc + c) * ld : nullptr;
    const F* __restrict__ vu = VelT<F>::u(Vg);
    const F* __restrict__ vv = VelT<F>::v(Vg);
    const F* __restrict__ vw = VelT<F>::w(Vg);
    // four velocities a block apart per round, their loads issued before the arithmetic
    auto load = [&](int k0, bool with, F (&g)[4], F (&h)[4]) {
        #pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int k = k0 + t * bs;
            g[t] = h[t] = F(0);
            if (k < nv) {
                g[t] = fG[k]; h[t] = fH[k];
                if (with) { g[t] += dG[k]; h[t] += dH[k]; }
            }
        }
    };
    double s[4];
    auto moments = [&](bool with) {
        Acc<F> sa[4];
        for (int k0 = threadIdx.x; k0 < nv; k0 += 4 * bs) {
            F g[4], h[4];
            load(k0, with, g, h);
            #pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int k = k0 + t * bs;
                if (k < nv) {
                    const F w = vw[k], u = vu[k], v = vv[k];
                    if constexpr (sizeof(F) == 8) {
                        const F wg = w * g[t], gu = wg * u, gv = wg * v;
                        sa[0].add(wg); sa[1].add(gu); sa[2].add(gv);
                        sa[3].add(fma(w, h[t], F(0.5) * fma(gu, u, gv * v)));
                    } else {
                        sa[0].add(w * g[t]); sa[1].add(w * u * g[t]); sa[2].add(w * v * g[t]);
                        sa[3].add(w * (F(0.5) * (u * u + v * v) * g[t] + h[t]));
                    }
                }
            }
        }
        block_total<4>(sa, red, s);
    };
    moments(df != nullptr);
    bool commit = df != nullptr;
    if (df) {
        // commit f + df, unless it would leave the cell with non-positive density or
        // internal energy: then the cell keeps f and its moments are those of f
        if (threadIdx.x == 0) sok = s[0] > 0.0 && s[3] * s[0] - 0.5 * (s[1] * s[1] + s[2] * s[2]) > 0.0;
        __syncthreads();
        commit = sok;
        if (!commit) moments(false);
    }
    if (threadIdx.x == 0) {
        const double ir = rcp64(s[0]);
        sUV[0] = (F)(s[1] * ir);
        sUV[1] = (F)(s[2] * ir);
    }
    __syncthreads();
    const F fU = sUV[0], fV = sUV[1];
    Acc<F> ta[2];
    for (int k0 = threadIdx.x; k0 < nv; k0 += 4 * bs) {
        F g[4], h[4];
        load(k0, commit, g, h);
        #pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int k = k0 + t * bs;
            if (k < nv) {
                if (commit) { fG[k] = g[t]; fH[k] = h[t]; }
                const F cx = vu[k] - fU, cy = vv[k] - fV;
                if constexpr (sizeof(F) == 8) {
                    const F we = vw[k] * fma(F(0.5) * fma(cx, cx, cy * cy), g[t], h[t]);
                    ta[0].add(we * cx);
                    ta[1].add(we * cy);
                } else {
                    const F e = F(0.5) * (cx * cx + cy * cy) * g[t] + h[t];
                    ta[0].add(vw[k] * cx * e);
                    ta[1].add(vw[k] * cy * e);
                }
            }
        }
    }
    double t[2];
    block_total<2>(ta, red, t);
    if (threadIdx.x == 0) {
        for (int m = 0; m < 4; ++m) W[4 * (size_t)c + m] = s[m];
        q[2 * (size_t)c] = t[0];
        q[2 * (size_t)c + 1] = t[1];
    }
}

template <typename F>
cudaError_t launch_update_moments(const LevelDev& L, const VelDev& V, F* f, const F* df, double* W, double* q,
                                  cudaStream_t st)
{
    // FP64: fewer warps per cell, so that fewer repeat the reductions in the FP64 pipe
    k_update_moments<F><<<L.nc, V.nv >= (sizeof(F) == 8 ? 2048 : 256) ? 256 : 128, 0, st>>>(L, V, f, df, W, q);
    return cudaGetLastError();
}
template <typename F>
cudaError_t launch_moments(const LevelDev& L, const VelDev& V, const F* f, double* W, double* q, cudaStream_t st)
{
    return launch_update_moments<F>(L, V, const_cast<F*>(f), nullptr, W, q, st);
}
template cudaError_t launch_update_moments<double>(const LevelDev&, const VelDev&, double*, const double*, double*,
                                                   double*, cudaStream_t);
template cudaError_t launch_moments<double>(const LevelDev&, const VelDev&, const double*, double*, double*,
                                            cudaStream_t);
template cudaError_t launch_update_moments<float>(const LevelDev&, const VelDev&, float*, const float*, double*,
                                                  double*, cudaStream_t);
template cudaError_t launch_moments<float>(const LevelDev&, const VelDev&, const float*, double*, double*,
                                           cudaStream_t);

// discrete Maxwellian of (rho, U, V, T) per cell
// Full-multigrid start-up: a fine cell whose prolonged state f has
// non-positive density or internal energy takes the f of its coarse cell
// (fc, the next coarser mesh with ncx cells per row).  One CTA per fine cell.
template <typename F>
__global__ void __launch_bounds__(256) k_state_fallback(LevelDev L, VelDev Vg, int ncx, size_t ncc,
                                                        const F* __restrict__ fc, F* __restrict__ f)
{
    __shared__ double red[32 * 4];
    const int c = blockIdx.x, nv = Vg.nv, i = c % L.nx, j = c / L.nx;
    const size_t nc = L.nc, ld = Vg.ld, cc = (size_t)(j / 2) * ncx + i / 2;
    const F* __restrict__ vu = VelT<F>::u(Vg);
    const F* __restrict__ vv = VelT<F>::v(Vg);
    const F* __restrict__ vw = VelT<F>::w(Vg);
    Acc<F> sa[4];
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        const F g = f[(size_t)c * ld + k], h = f[(nc + c) * ld + k], u = vu[k], v = vv[k], w = vw[k];
        sa[0].add(w * g); sa[1].add(w * u * g); sa[2].add(w * v * g);
        sa[3].add(w * (F(0.5) * (u * u + v * v) * g + h));
    }
    double s[4];
    block_total<4>(sa, red, s);
    if (s[0] > 0.0 && s[3] * s[0] - 0.5 * (s[1] * s[1] + s[2] * s[2]) > 0.0) return;
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        f[(size_t)c * ld + k] = fc[cc * ld + k];
        f[(nc + c) * ld + k] = fc[(ncc + cc) * ld + k];
    }
}
template <typename F>
cudaError_t launch_state_fallback(const LevelDev& L, const VelDev& V, int ncx, size_t ncc, const F* fc, F* f,
                                  cudaStream_t st)
{
    k_state_fallback<F><<<L.nc, V.nv >= 256 ? 256 : 128, 0, st>>>(L, V, ncx, ncc, fc, f);
    return cudaGetLastError();
}
template cudaError_t launch_state_fallback<double>(const LevelDev&, const VelDev&, int, size_t, const double*,
                                                   double*, cudaStream_t);
template cudaError_t launch_state_fallback<float>(const LevelDev&, const VelDev&, int, size_t, const float*, float*,
                                                  cudaStream_t);

template <typename F>
// The Maxwellian of velocity k = a nv_y + b factors into rho lam/pi e^{-lam (u_a - U)^2}
// times e^{-lam (v_b - V)^2}: nu + nv_y exponentials per cell (in FP64, tabled in shared
// memory), then two FP64 products per velocity.
__global__ void k_init_maxwell(LevelDev L, VelDev Vg, const double* __restrict__ prim, F* __restrict__ f)
{
    extern __shared__ double etab[];      // [nu] rho lam/pi e^{-lam (u_a - U)^2}, [nvv] e^{-lam (v_b - V)^2}
    const int c = blockIdx.x, nv = Vg.nv, nu = Vg.nu, nvv = Vg.nvv, tid = threadIdx.x, bs = blockDim.x;
    const size_t nc = L.nc, ld = Vg.ld;
    const double rho = prim[4 * c], U = prim[4 * c + 1], V = prim[4 * c + 2], lam = 1.0 / prim[4 * c + 3];
    const double hfac = kKint / (4.0 * lam);
    for (int e = tid; e < nu + nvv; e += bs) {
        if (e < nu) {
            const double d = Vg.ua[e] - U;
            etab[e] = rho * (lam / kPi) * exp(-lam * d * d);
        } else {
            const double d = Vg.vb[e - nu] - V;
            etab[e] = exp(-lam * d * d);
        }
    }
    __syncthreads();
    // velocity k = a * nvv + b of this thread, stepped by the block size without a division
    const int sa = bs / nvv, sb = bs - sa * nvv;
    int a = tid / nvv, b = tid - a * nvv;
    for (int k = tid; k < nv; k += bs, a += sa, b += sb) {
        if (b >= nvv) { b -= nvv; ++a; }
        const double g = etab[a] * etab[nu + b];
        f[(size_t)c * ld + k] = (F)g;
        f[(nc + c) * ld + k] = (F)(g * hfac);
    }
}
template <typename F>
cudaError_t launch_init_maxwell(const LevelDev& L, const VelDev& V, const double* prim, F* f, cudaStream_t st)
{
    k_init_maxwell<F><<<L.nc, V.nv >= 256 ? 256 : 128, (V.nu + V.nvv) * sizeof(double), st>>>(L, V, prim, f);
    return cudaGetLastError();
}
template cudaError_t launch_init_maxwell<double>(const LevelDev&, const VelDev&, const double*, double*, cudaStream_t);
template cudaError_t launch_init_maxwell<float>(const LevelDev&, const VelDev&, const double*, float*, cudaStream_t);

// wall pressure, shear and heat flux of the faces in `faces` (axis * 2^30 + face index)
template <typename F>
__global__ void k_wall_quantities(LevelDev L, VelDev Vg, const BcDev* __restrict__ bc, const double* __restrict__ Cw,
                                  const F* __restrict__ f, int bcid, const int* __restrict__ faces,
                                  double* __restrict__ out)
{
    __shared__ double red[32 * 4];
    const int code = faces[blockIdx.x];
    const int axis = code >> 30, fi = code & ((1 << 30) - 1);
    const int nx = L.nx, nv = Vg.nv;
    const size_t nc = L.nc, ld = Vg.ld;
    int i = axis == 0 ? fi % (nx + 1) : fi % nx, j = axis == 0 ? fi / (nx + 1) : fi / nx;
    int outsign, c;
    bface_side(L, axis, i, j, c, outsign);
    const BcDev B = bc[bcid];
    const double* Cb = Cw + (size_t)bcid * nv;
    double s[2] = {0, 0};
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        double uo = outsign * (axis == 0 ? Vg.u[k] : Vg.v[k]);
        if (uo > 0) s[0] += Vg.w[k] * uo * (double)f[(size_t)c * ld + k];
        else if (uo < 0) s[1] += Vg.w[k] * uo * Cb[k];
    }
    block_sum<2>(s, red);
    double rhow = -s[0] / s[1];
    double t[3] = {0, 0, 0};
    double Uwt = axis == 0 ? B.v : B.u;
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        double u = Vg.u[k], v = Vg.v[k];
        double uo = outsign * (axis == 0 ? u : v), ut = axis == 0 ? v : u;
        double g, h;
        if (uo >= 0) { g = f[(size_t)c * ld + k]; h = f[(nc + c) * ld + k]; }
        else { g = rhow * Cb[k]; h = g * kKint * B.t / 4.0; }
        double du = u - B.u, dv = v - B.v;
        t[0] += Vg.w[k] * uo * uo * g;
        t[1] += Vg.w[k] * uo * (ut - Uwt) * g;
        t[2] += Vg.w[k] * uo * (0.5 * (du * du + dv * dv) * g + h);
    }
    block_sum<3>(t, red);
    if (threadIdx.x == 0)
        for (int m = 0; m < 3; ++m) out[3 * blockIdx.x + m] = t[m];
}
template <typename F>
cudaError_t launch_wall_quantities(const LevelDev& L, const VelDev& V, const BcDev* bc, const double* Cw, const F* f,
                                   int bcid, const int* faces, int nfaces, double* out, cudaStream_t st)
{
    if (nfaces == 0) return cudaSuccess;
    k_wall_quantities<F><<<nfaces, 128, 0, st>>>(L, V, bc, Cw, f, bcid, faces, out);
    return cudaGetLastError();
}
template cudaError_t launch_wall_quantities<double>(const LevelDev&, const VelDev&, const BcDev*, const double*,
                                                    const double*, int, const int*, int, double*, cudaStream_t);
template cudaError_t launch_wall_quantities<float>(const LevelDev&, const VelDev&, const BcDev*, const double*,
                                                   const float*, int, const int*, int, double*, cudaStream_t);

} // namespace miugks
