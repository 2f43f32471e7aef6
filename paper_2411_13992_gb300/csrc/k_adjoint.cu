// k_adjoint.cu -- reverse-mode adjoint of the libsphtv step (not in the
// paper; derivatives of Eq. 2-8 and 14-16 taken by hand), with each step's
// neighbour set and step size frozen.
//
// One reverse step, in the cell-sorted order of the forward step it undoes
// (forward values come from a per-step tape), cotangents kept in FP64 in the
// caller's particle order:
//   k_adj_prep    : A_i = abar'_i + dt/2 vbar'_i (the closing kick), and the
//                   cotangent of the residual R_i from that of the
//                   displacement dr_i = xi chi(s) H^2 R_i, s = H^2 |R_i|^2
//   k_adj_pairs   : gather form of the pair terms: particle k collects the
//                   derivatives of its own sums (k as i) and of each fluid
//                   neighbour's sums (k as j), so no atomics are needed;
//                   also the density cotangent and d/d(eta) partials
//   k_adj_density : the density sum rho_k = rho0 sum_j W_kj / sigma0_k, then
//                   the reverse of the drift and the opening kick; its first
//                   block adds the step's d/d(eta) (fixed-order reduction)
//
// Both walks run over the neighbour list that the step's density pass left in
// the tape (the FP64 form scanned the 5^D cells with its exact test before:
// 570 and 176 us per reverse step of 4,096 particles), and in the FP64 form
// with a group of L lanes per particle (adj_lanes64 below), since one thread's
// chain of FP64 operations is the bound of a problem of some thousand
// particles.
//
// Subgradients: d beta/d dU = eta_R / c inside 0 < eta_R dU / c < 1, else 0
// (Eq. 6); d chi/d s = C inside thresh < s < 1/C, else 0 (Eq. 15).
#include <type_traits>

#include "common.cuh"
#include "launch.h"
#include "pair_physics.cuh"
#include "pair_walk.cuh"

namespace sphtv {

template <typename Real>
using AccOf = typename std::conditional<sizeof(Real) == 4, KSum, PlainD>::type;

// Sum of a group's accumulators, in every lane of the group (a fixed tree).
template <int L>
__device__ __forceinline__ void group_sum(KSum& a)
{
#pragma unroll
    for (int o = L / 2; o >= 1; o >>= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, a.s, o);
        const float c2 = __shfl_xor_sync(0xffffffffu, a.c, o);
        ksum_merge(a.s, a.c, s2, c2);
    }
    if (L > 1) {
        a.s = __fsub_rn(a.s, a.c);
        a.c = 0.f;
    }
}

template <int L>
__device__ __forceinline__ void group_sum(PlainD& a)
{
#pragma unroll
    for (int o = L / 2; o >= 1; o >>= 1) a.s += __shfl_xor_sync(0xffffffffu, a.s, o);
}

// The cotangents Abar_k and Rbar_k of a particle as one record of
// kAbStride<DIM> values ({Abar, Rbar}, padded to a whole number of 16-byte
// vectors in the FP32 form), so that the pair kernel gathers a neighbour's
// with one or two vector loads.
template <int DIM> constexpr int kAbStride = DIM == 3 ? 8 : 4;

template <typename Real, int DIM>
__device__ __forceinline__ void load_ab(const Real* AR, int k, Real* Ab, Real* Rb)
{
    const Real* p = AR + (size_t)k * kAbStride<DIM>;
    if constexpr (sizeof(Real) == 4) {
        const float4 a = *(const float4*)p;
        if (DIM == 2) {
            Ab[0] = a.x; Ab[1] = a.y; Rb[0] = a.z; Rb[1] = a.w;
        } else {
            const float4 b = *(const float4*)(p + 4);
            Ab[0] = a.x; Ab[1] = a.y; Ab[2] = a.z; Rb[0] = a.w; Rb[1] = b.x; Rb[2] = b.y;
        }
    } else {
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            Ab[d] = p[d];
            Rb[d] = p[DIM + d];
        }
    }
}

// Forward values of one step.
template <typename Real>
struct Tape {
    const int32_t* id;
    const int8_t* kind;
    const double* x;       // [DIM][n] positions after the drift (FP64)
    const double* h;
    const double* m;
    const double* s0;
    const typename Vec4<Real>::T* vr;   // {half-step v, rho - rho0 (+inf: wall)}
    const Real* R;         // [DIM][n] residual
    const int32_t* start;  // cell ranges
    const float4* pos4;    // FP32 form: cell-relative positions
    const int32_t* cell;   // cell of each particle
    const double* dt;      // step size of the step
    const uint32_t* nbl;   // the step's force-neighbour list (transposed)
    const int32_t* nbc;    // and its counts
};

// Visit the neighbours j != k of particle k with 0 < r < 2 h_kj, decided
// exactly as the forward pass decided them: f(j, rv[3] = x_k - x_j, r, 1/r,
// w_j, load(j)) with w_j = pos4[j].w (FP32 form: m_j at uniform resolution,
// else h_j) and load(j) whatever else of j the caller gathers, which the FP32
// list walk requests one neighbour ahead.
// Lane q of a group of L takes the list's entries q, q + L, ...; a particle
// with more neighbours than the list holds is walked over its cells, in the
// FP64 form cells q, q + L, ... by lane q.
// FP32 form: 1/r from rsqrt and r = r^2/r, as the forward force pass takes
// them; FP64 form: 1/r within one rounding, r = r^2 (1/r).
template <typename Real, int DIM, int L, typename Load, typename F>
__device__ __forceinline__ void adj_visit(int n, int k, int q, const Grid& G, const Consts<Real>& K,
                                          const Tape<Real>& T, Load& load, F& f)
{
    const int cnt = T.nbc[k];
    const bool listed = cnt <= list_capacity(DIM);
    if constexpr (sizeof(Real) == 4) {
        const float4 pk = T.pos4[k];
        const float ok[3] = {pk.x, pk.y, pk.z};
        if (listed) {
            // the list holds exactly the pairs the density pass's walk
            // accepted, in the walk's order; the pair vector and r^2 with the
            // walk's arithmetic
            const float ex = G.edgef[0], ey = G.edgef[1], ez = G.edgef[2];
            // the lane's entry two ahead and the neighbour's data one ahead in flight
            const size_t row = (size_t)L * n;
            const uint32_t* lp = T.nbl + k + (size_t)q * n;
            uint32_t e_n = q < cnt ? lp[0] : 0u;
            uint32_t e_nn = q + L < cnt ? lp[row] : 0u;
            float4 p_n = T.pos4[e_n >> kCodeBits];
            auto d_n = load((int)(e_n >> kCodeBits));
            lp += 2 * row;
            for (int t = q; t < cnt; t += L, lp += row) {
                const uint32_t e = e_n;
                const float4 pj = p_n;
                const auto dj = d_n;
                e_n = e_nn;
                if (t + L < cnt) {
                    p_n = T.pos4[e_n >> kCodeBits];
                    d_n = load((int)(e_n >> kCodeBits));
                }
                e_nn = t + 2 * L < cnt ? *lp : 0u;
                const int j = (int)(e >> kCodeBits);
                const uint32_t code = e & ((1u << kCodeBits) - 1u);
                const int dx = (int)(code % kSide) - kStencilR, dy = (int)((code / kSide) % kSide) - kStencilR,
                          dz = (int)(code / (kSide * kSide)) - kStencilR;
                const float2 rxy = __fadd2_rn(__ffma2_rn(make_float2(pj.x, pj.y), make_float2(-1.f, -1.f),
                                                         make_float2(ok[0], ok[1])),
                                              make_float2(-(float)dx * ex, -(float)dy * ey));
                const float2 qq = __fmul2_rn(rxy, rxy);
                float r2 = qq.x + qq.y;
                float rz = 0.f;
                if (DIM == 3) {
                    rz = (ok[2] - pj.z) + -(float)dz * ez;
                    r2 = fmaf(rz, rz, r2);
                }
                const Real rv[3] = {rxy.x, rxy.y, rz};
                const float inv_r = rsqrtf(r2);
                f(j, rv, r2 * inv_r, inv_r, pj.w, dj);
            }
            return;
        }
        if (q) return;
        // the clipped row walk of the forward density pass, with its
        // arithmetic for r^2, so the pairs are exactly the forward's
        const float hk = (float)T.h[k];
        const float reach = K.uniform_h ? 2.f * K.h_u : 2.f * pair_h(K, hk, K.h_u);
        auto g = [&](int j, uint32_t, const float4& pj, float r2, float rx, float ry, float rz) {
            float lim;
            if (K.uniform_h) lim = K.four_h2_u;
            else {
                const float hh = pair_h(K, hk, pj.w);
                lim = 4.f * hh * hh;
            }
            if (!(r2 < lim) || !(r2 > 0.f)) return;
            const Real rv[3] = {rx, ry, rz};
            const float inv_r = rsqrtf(r2);
            f(j, rv, r2 * inv_r, inv_r, pj.w, load(j));
        };
        for_candidates_rows<DIM, false>(ok, reach, T.cell[k], G, T.start, T.cell, T.pos4, g);
    } else {
        double xk[3] = {0, 0, 0};
#pragma unroll
        for (int d = 0; d < DIM; ++d) xk[d] = T.x[(size_t)d * n + k];
        int c[3];
        cell_decode(G, T.cell[k], c);
        if (listed) {
            // the list of the density pass's exact test; the stencil step of
            // j's cell fixes the periodic image
            for (int t = q; t < cnt; t += L) {
                const uint32_t e = T.nbl[(size_t)t * n + k];
                const int j = (int)(e >> kCodeBits);
                const int code = (int)(e & ((1u << kCodeBits) - 1u));
                const int step[3] = {code % kSide - kStencilR, (code / kSide) % kSide - kStencilR,
                                     code / (kSide * kSide) - kStencilR};
                Real rv[3] = {0, 0, 0};
                double r2 = 0.0;
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    double y = __dsub_rn(xk[d], T.x[(size_t)d * n + j]);
                    if (G.periodic[d]) {
                        const int sc = c[d] + step[d];
                        if (sc >= G.nc[d]) y = __dsub_rn(y, G.L[d]);
                        else if (sc < 0) y = __dadd_rn(y, G.L[d]);
                    }
                    rv[d] = y;
                    r2 += y * y;
                }
                const double inv_r = rsqrt_pos(r2);
                f(j, rv, r2 * inv_r, inv_r, 0.f, load(j));
            }
            return;
        }
        // the exact test of the forward pass over the cells q, q + L, ... of the
        // stencil (minimum image, sqrt(r^2) < 2 h_kj by the same root)
        constexpr int cells = DIM == 3 ? kSide * kSide * kSide : kSide * kSide;
        for (int t = q; t < cells; t += L) {
            const int cx = cell_step(G, c[0], t % kSide - kStencilR, 0);
            const int cy = cell_step(G, c[1], t / kSide % kSide - kStencilR, 1);
            const int cz = DIM == 3 ? cell_step(G, c[2], t / (kSide * kSide) - kStencilR, 2) : 0;
            if (cx < 0 || cy < 0 || cz < 0) continue;
            const int cell = cx + G.nc[0] * (cy + G.nc[1] * cz);
            for (int j = T.start[cell]; j < T.start[cell + 1]; ++j) {
                if (j == k) continue;
                Real rv[3] = {0, 0, 0};
                double r2 = 0.0;
                for (int d = 0; d < DIM; ++d) {
                    rv[d] = min_image(G, xk[d], T.x[(size_t)d * n + j], d);
                    r2 += rv[d] * rv[d];
                }
                if (!(r2 > 0.0)) continue;
                const double hij = pair_h(K, T.h[k], T.h[j]);
                if (!(sqrt_pos(r2) < 2.0 * hij)) continue;
                const double inv_r = rsqrt_pos(r2);
                f(j, rv, r2 * inv_r, inv_r, 0.f, load(j));
            }
        }
    }
}

// Reverse of one pair term of a_i (Eq. 3, 5-7) and R_i (Eq. 14) for the pair
// (i, j), given the cotangents Ai of a_i and Rbi of R_i.  rv = x_i - x_j,
// r = |rv|, inv_r = 1/r, w = W'(r), w2 = W''(r); rho_j, p_j and vj are the
// stand-ins of a wall neighbour when j is a wall; inv_rho_i, inv_rho_j are
// the reciprocals of the densities (each division once per pair or per
// particle, not six times per call).  Outputs: rb (cotangent of rv), dvb
// (of v_i - v_j), rho_ib, rho_jb (of rho_i, rho_j), etab (of eta).
template <typename Real, int DIM>
__device__ __forceinline__ void pair_adjoint(const Consts<Real>& K, const Real* rv, Real r, Real inv_r, Real w,
                                             Real w2, const Real* vi, Real rho_i, Real inv_rho_i, Real p_i,
                                             const Real* vj, Real rho_j, Real inv_rho_j, Real p_j, Real m_j,
                                             const Real* Ai, const Real* Rbi, Real* rb, Real* dvb, Real& rho_ib,
                                             Real& rho_jb, Real& etab)
{
    Real u[3] = {0, 0, 0}, dv[3] = {0, 0, 0};
    Real udv = 0, Au = 0, Adv = 0, Ru = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        u[d] = rv[d] * inv_r;
        dv[d] = vi[d] - vj[d];
        udv += u[d] * dv[d];
        Au += Ai[d] * u[d];
        Adv += Ai[d] * dv[d];
        Ru += Rbi[d] * u[d];
    }
    const Real dU = -udv;                               // U_l - U_r
    const Real slope = K.beta_slope * K.inv_c;
    const Real braw = slope * dU;
    const Real beta = braw > Real(0) ? (braw < Real(1) ? braw : Real(1)) : Real(0);
    const Real dbeta = (braw > Real(0) && braw < Real(1)) ? slope : Real(0);
    const Real rbar = Real(0.5) * (rho_i + rho_j);
    const Real pstar = Real(0.5) * (p_i + p_j) + Real(0.5) * beta * rbar * K.c * dU;
    const Real Kf = m_j * (inv_rho_i * inv_rho_j);      // m_j / (rho_i rho_j)
    const Real Vj = m_j * inv_rho_j;
    const Real wq = w * inv_r;
    const Real Pb = Real(-2) * Kf * w * Au;
    const Real Kb = Real(-2) * pstar * w * Au + K.two_eta * wq * Adv;
    const Real wb = Real(-2) * Kf * pstar * Au + Vj * Ru;
    const Real wqb = K.two_eta * Kf * Adv;
    etab = Real(2) * Kf * wq * Adv;
    const Real dUb = Pb * Real(0.5) * rbar * K.c * (beta + dU * dbeta);
    const Real rbarb = Pb * Real(0.5) * beta * K.c * dU;
    rho_ib = -Kf * inv_rho_i * Kb + Real(0.5) * rbarb + K.c2 * Real(0.5) * Pb;
    rho_jb = -Kf * inv_rho_j * Kb + Real(0.5) * rbarb + K.c2 * Real(0.5) * Pb - Vj * inv_rho_j * w * Ru;
    Real ub[3] = {0, 0, 0};
    Real uu = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        ub[d] = Real(-2) * Kf * pstar * w * Ai[d] + Vj * w * Rbi[d] - dUb * dv[d];
        dvb[d] = K.two_eta * Kf * wq * Ai[d] - dUb * u[d];
        uu += ub[d] * u[d];
    }
    const Real radial = w2 * wb + (w2 * inv_r - w * inv_r * inv_r) * wqb;
#pragma unroll
    for (int d = 0; d < DIM; ++d) rb[d] = (ub[d] - uu * u[d]) * inv_r + radial * u[d];
}

// 1/x: rcp.approx in the FP32 form (as its forward pass takes reciprocals),
// the correctly rounded division in the FP64 form.
__device__ __forceinline__ float recip(float x) { return rcp_approx(x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

// W'(r) and W''(r) of the pair (k, j); w_j = pos4[j].w of the FP32 form (h_j
// at variable resolution).  The FP64 form at uniform resolution takes them
// from the constant C = -5 a_D h^-(D+2): W' = C r t^3 and W'' = C t^2 (1 - 2q)
// with t = 1 - q/2.
template <typename Real, int DIM>
__device__ __forceinline__ void pair_kernels(const Consts<Real>& K, const Tape<Real>& T, int k, int j, Real hk,
                                             float w_j, Real r, Real& w, Real& w2)
{
    Real inv_h;
    if constexpr (sizeof(Real) == 4) {
        inv_h = K.uniform_h ? K.inv_h_u : 1.f / pair_h(K, hk, w_j);
    } else {
        if (K.uniform_h) {
            const double t = fma(-K.half_inv_h_u, r, 1.0), t2 = t * t;
            w = K.dwr_coef_u * r * (t2 * t);
            w2 = K.dwr_coef_u * t2 * fma(-K.two_inv_h_u, r, 1.0);
            return;
        }
        inv_h = 1.0 / pair_h(K, hk, T.h[j]);
    }
    w = wendland_dW<DIM, Real>(r, inv_h);
    w2 = wendland_d2W<DIM, Real>(r, inv_h);
}

template <typename Real>
__device__ __forceinline__ Real mass_of(const Consts<Real>& K, const Tape<Real>& T, int j, float w_j)
{
    // at uniform resolution the position record of the FP32 form holds the
    // same FP32 mass (a conversion fewer on the FP64 pipe per pair)
    if constexpr (sizeof(Real) == 4) return K.uniform_h ? w_j : (float)T.m[j];
    else return T.m[j];
}

// ------------------------------------------------------------------- prep

template <typename Real, int DIM>
__global__ void __launch_bounds__(256) k_adj_prep(int n, Tape<Real> T, Consts<Real> K, int step_mode,
                                                  const double* vc, const double* ac,
                                                  const double* drc, Real* AR)
{
    pdl_wait();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int i = T.id[k];
    Real* const ar = AR + (size_t)k * kAbStride<DIM>;
    if (T.kind[k]) {
        for (int q = 0; q < kAbStride<DIM>; ++q) ar[q] = Real(0);
        return;
    }
    const double hdt = step_mode ? 0.5 * *T.dt : 0.0;
    const Real H = K.tv_h_particle ? (Real)T.h[k] : K.h_min;
    const Real H2 = H * H;
    Real R[3] = {0, 0, 0}, D[3] = {0, 0, 0};
    Real s = 0, DR = 0;
    for (int d = 0; d < DIM; ++d) {
        R[d] = T.R[(size_t)d * n + k];
        D[d] = (Real)drc[(size_t)d * n + i];
        s += R[d] * R[d];
        DR += D[d] * R[d];
    }
    s *= H2;
    const Real chi = tv_limiter(K, s);
    const Real dchi = (K.tv_mode == SPH_TV_LIMITED && s > K.tv_thresh && K.tv_C * s < Real(1)) ? K.tv_C : Real(0);
    for (int d = 0; d < DIM; ++d) {
        ar[d] = (Real)(ac[(size_t)d * n + i] + hdt * vc[(size_t)d * n + i]);
        ar[DIM + d] = K.tv_xi * H2 * (chi * D[d] + dchi * DR * Real(2) * H2 * R[d]);
    }
    for (int q = 2 * DIM; q < kAbStride<DIM>; ++q) ar[q] = Real(0);
}

// ------------------------------------------------------------------ pairs

constexpr int kAdjTPB = 128;

// What the pair kernel gathers of a neighbour besides its position.
template <typename Real>
struct Neighbour {
    typename Vec4<Real>::T vr;
    Real Ab[3], Rb[3];
};

template <typename Real, int DIM, int L>
__global__ void __launch_bounds__(kAdjTPB) k_adj_pairs(int n, Tape<Real> T, Grid G, Consts<Real> K,
                                                   const Real* AR,
                                                   Real* xbp, Real* vbp,
                                                   Real* sigb, double* partials)
{
    pdl_wait();
    using Acc = AccOf<Real>;
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) / L, q = threadIdx.x % L;
    const bool fluid = k < n && !T.kind[k];
    Acc ax[DIM], av[DIM], arho;
    double eta = 0.0;
    if (fluid) {
        const auto mk = T.vr[k];
        const Real vk[3] = {mk.x, mk.y, mk.z};
        const Real rho_k = K.rho0 + mk.w;
        const Real p_k = K.c2 * mk.w;
        const Real inv_rho_k = Real(1) / rho_k;
        const Real m_k = (Real)T.m[k];
        const Real h_k = K.uniform_h ? K.h_u : (Real)T.h[k];
        Real Ak[3] = {0, 0, 0}, Rk[3] = {0, 0, 0};
        load_ab<Real, DIM>(AR, k, Ak, Rk);
        auto load = [&](int j) {
            Neighbour<Real> d = {};
            d.vr = T.vr[j];
            load_ab<Real, DIM>(AR, j, d.Ab, d.Rb);       // zero for a wall
            return d;
        };
        auto pair = [&](int j, const Real* rv, Real r, Real inv_r, float w_j, const Neighbour<Real>& nb) {
            Real w, w2;
            pair_kernels<Real, DIM>(K, T, k, j, h_k, w_j, r, w, w2);
            const auto mj = nb.vr;
            const Real vj[3] = {mj.x, mj.y, mj.z};
            const bool wall = isinf(mj.w);
            const Real rho_j = wall ? rho_k : K.rho0 + mj.w;
            const Real inv_rho_j = wall ? inv_rho_k : recip(rho_j);
            const Real p_j = wall ? p_k : K.c2 * mj.w;
            Real rb[3], dvb[3], rib, rjb, eb;
            // k's own sums (k as i)
            pair_adjoint<Real, DIM>(K, rv, r, inv_r, w, w2, vk, rho_k, inv_rho_k, p_k, vj, rho_j, inv_rho_j, p_j,
                                    mass_of(K, T, j, w_j), Ak, Rk, rb, dvb, rib, rjb, eb);
            for (int d = 0; d < DIM; ++d) {
                ax[d].add(rb[d]);
                av[d].add(dvb[d]);
            }
            arho.add(wall ? rib + rjb : rib);
            eta += (double)eb;
            if (wall) return;
            // the fluid neighbour's sums (j as i, k as j): r_jk = -r_kj
            const Real *Aj = nb.Ab, *Rj = nb.Rb;
            Real mrv[3] = {0, 0, 0};
            for (int d = 0; d < DIM; ++d) mrv[d] = -rv[d];
            pair_adjoint<Real, DIM>(K, mrv, r, inv_r, w, w2, vj, rho_j, inv_rho_j, p_j, vk, rho_k, inv_rho_k, p_k,
                                    m_k, Aj, Rj, rb, dvb, rib, rjb, eb);
            for (int d = 0; d < DIM; ++d) {
                ax[d].add(-rb[d]);
                av[d].add(-dvb[d]);
            }
            arho.add(rjb);
        };
        adj_visit<Real, DIM, L>(n, k, q, G, K, T, load, pair);
    }
    __syncwarp();
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        group_sum<L>(ax[d]);
        group_sum<L>(av[d]);
    }
    group_sum<L>(arho);
    if (k < n && q == 0) {
        for (int d = 0; d < DIM; ++d) {
            xbp[(size_t)d * n + k] = ax[d].value();
            vbp[(size_t)d * n + k] = av[d].value();
        }
        sigb[k] = fluid ? arho.value() * K.rho0 / (Real)T.s0[k] : Real(0);
    }
    // the block's d/d(eta), in a fixed order
    __shared__ double wsum[kAdjTPB / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) eta += __shfl_down_sync(0xffffffffu, eta, off);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = eta;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)blockDim.x / 32; ++w) eta += wsum[w];
        partials[blockIdx.x] = eta;
    }
}

// ------------------------------------------------- density + drift / kick

template <typename Real, int DIM, int L>
__global__ void __launch_bounds__(kAdjTPB) k_adj_density(int n, Tape<Real> T, Grid G, Consts<Real> K,
                                                     const Real* sigb, const Real* xbp,
                                                     const Real* vbp, int step_mode,
                                                     double* xc, double* vc,
                                                     double* ac, double* drc,
                                                     const double* partials, int nblocks,
                                                     double* eta)
{
    pdl_wait();
    using Acc = AccOf<Real>;
    if (blockIdx.x == 0) {
        // block 0 first adds the pair kernel's per-block d/d(eta) partials to
        // eta (a fixed order: strided per thread, then the warps, then the
        // block's warps by thread 0)
        __shared__ double wsum[kAdjTPB / 32];
        double v = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v += partials[b];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)blockDim.x / 32; ++w) t += wsum[w];
            *eta += t;
        }
    }
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) / L, q = threadIdx.x % L;
    const bool fluid = k < n && !T.kind[k];
    Acc acc[DIM];
    if (fluid) {
        const Real sk = sigb[k];
        const Real h_k = K.uniform_h ? K.h_u : (Real)T.h[k];
        auto load = [&](int j) { return sigb[j]; };           // 0 for a wall
        auto pair = [&](int j, const Real* rv, Real r, Real inv_r, float w_j, Real sj) {
            Real w, w2;
            pair_kernels<Real, DIM>(K, T, k, j, h_k, w_j, r, w, w2);
            const Real g = (sk + sj) * w * inv_r;
            for (int d = 0; d < DIM; ++d) acc[d].add(g * rv[d]);
        };
        adj_visit<Real, DIM, L>(n, k, q, G, K, T, load, pair);
    }
    __syncwarp();
#pragma unroll
    for (int d = 0; d < DIM; ++d) group_sum<L>(acc[d]);
    if (k >= n || q) return;
    const int i = T.id[k];
    if (!fluid) {
        if (step_mode)
            for (int d = 0; d < 3; ++d) {
                const size_t o = (size_t)d * n + i;
                xc[o] = vc[o] = ac[o] = drc[o] = 0.0;
            }
        return;
    }
    const double dt = step_mode ? *T.dt : 0.0;
    const double hdt = 0.5 * dt;
    for (int d = 0; d < DIM; ++d) {
        const size_t o = (size_t)d * n + i, so = (size_t)d * n + k;
        const double xb = xc[o] + (double)xbp[so] + (double)acc[d].value();   // cotangent of x'
        double vh = vc[o] + (double)vbp[so];                                  // of the half-step v
        if (step_mode) {
            drc[o] = xb;              // x' = x + dt v_h + dr
            vh += dt * xb;
            ac[o] = hdt * vh;         // v_h = v + dt/2 a
        }
        xc[o] = xb;
        vc[o] = vh;
    }
}

// -------------------------------------------------------------- the tape

// The forward values of a step that the reverse sweep reads, from the
// context's buffers into a tape slot: one kernel for what eleven copies did
// (each a node of the segment's graph).
template <typename Real, int DIM>
__global__ void __launch_bounds__(256) k_save_tape(int n, int nstart, StateSet<Real> S,
                                                   const typename Vec4<Real>::T* vr,
                                                   const Real* R, const int32_t* start,
                                                   const float4* pos4, const int32_t* cell,
                                                   Tape<Real> T)
{
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nstart) const_cast<int32_t*>(T.start)[i] = start[i];
    if (i >= n) return;
    const_cast<int32_t*>(T.id)[i] = S.id[i];
    const_cast<int8_t*>(T.kind)[i] = S.kind[i];
    const_cast<double*>(T.h)[i] = S.h[i];
    const_cast<double*>(T.m)[i] = S.m[i];
    const_cast<double*>(T.s0)[i] = S.s0[i];
    const_cast<typename Vec4<Real>::T*>(T.vr)[i] = vr[i];
    const_cast<int32_t*>(T.cell)[i] = cell[i];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const size_t o = (size_t)d * n + i;
        const_cast<Real*>(T.R)[o] = R[o];
        if (sizeof(Real) == 8) const_cast<double*>(T.x)[o] = S.x[o];
    }
    if (sizeof(Real) == 4) const_cast<float4*>(T.pos4)[i] = pos4[i];
}

// -------------------------------------------------------------- launchers

static inline int nblk(int n, int t) { return (n + t - 1) / t; }

// Lanes per particle of the reverse kernels in the FP64 form: as many as give
// every SM some 500 threads (the FP64 pipe is full with few warps).  The FP32
// form keeps one: its compensated sums stay in the order of the list.
static int adj_lanes64(int n, int sms)
{
    if (sms <= 0) sms = 152;
    return n >= sms * 512 ? 1 : (n >= sms * 128 ? 4 : 8);
}

// Blocks of the pair kernel at most (eight lanes per particle).
size_t adj_partials(int n) { return ((size_t)n + kAdjTPB / 8 - 1) / (kAdjTPB / 8); }

template <typename Real>
static Tape<Real> make_tape(const TapeView& V)
{
    Tape<Real> T;
    T.id = V.id; T.kind = V.kind; T.x = V.x; T.h = V.h; T.m = V.m; T.s0 = V.s0;
    T.vr = (const typename Vec4<Real>::T*)V.vr;
    T.R = (const Real*)V.R;
    T.start = V.start; T.pos4 = V.pos4; T.cell = V.cell; T.dt = V.dt;
    T.nbl = V.nbl; T.nbc = V.nbc;
    return T;
}

template <typename Real, int DIM, int L>
static void adjoint_step_l(int n, const Tape<Real>& T, const Grid& G, const Consts<Real>& K, const AdjView& A,
                           int step_mode, cudaStream_t st)
{
    const int nb = nblk(n, kAdjTPB / L);
    launch(k_adj_pairs<Real, DIM, L>, nb, kAdjTPB, 0, st, n, T, G, K, (const Real*)A.AR, (Real*)A.xbp, (Real*)A.vbp,
                                                      (Real*)A.sigb, A.partials);
    launch(k_adj_density<Real, DIM, L>, nb, kAdjTPB, 0, st, n, T, G, K, (const Real*)A.sigb, (const Real*)A.xbp,
                                                        (const Real*)A.vbp, step_mode, A.xc, A.vc, A.ac, A.drc,
                                                        A.partials, nb, A.eta);
}

template <typename Real, int DIM>
static void adjoint_step_t(int n, const TapeView& V, const Grid& G, const Consts<Real>& K, const AdjView& A,
                           int step_mode, cudaStream_t st)
{
    const Tape<Real> T = make_tape<Real>(V);
    launch(k_adj_prep<Real, DIM>, nblk(n, 256), 256, 0, st, n, T, K, step_mode, A.vc, A.ac, A.drc, (Real*)A.AR);
    if constexpr (sizeof(Real) == 8) {
        const int L = adj_lanes64(n, G.sms);
        if (L == 8) return adjoint_step_l<Real, DIM, 8>(n, T, G, K, A, step_mode, st);
        if (L == 4) return adjoint_step_l<Real, DIM, 4>(n, T, G, K, A, step_mode, st);
    }
    adjoint_step_l<Real, DIM, 1>(n, T, G, K, A, step_mode, st);
}

template <typename Real>
static void save_tape_t(int dim, int n, int nstart, const void* S, const void* vr, const void* R,
                        const int32_t* start, const float4* pos4, const int32_t* cell, const TapeView& V,
                        cudaStream_t st)
{
    const Tape<Real> T = make_tape<Real>(V);
    const auto s = *(const StateSet<Real>*)S;
    const auto v = (const typename Vec4<Real>::T*)vr;
    const int nb = nblk(n > nstart ? n : nstart, 256);
    if (dim == 2) launch(k_save_tape<Real, 2>, nb, 256, 0, st, n, nstart, s, v, (const Real*)R, start, pos4, cell, T);
    else launch(k_save_tape<Real, 3>, nb, 256, 0, st, n, nstart, s, v, (const Real*)R, start, pos4, cell, T);
}

cudaError_t launch_save_tape(int prec, int dim, int n, int nstart, const void* S, const void* vr, const void* R,
                             const int32_t* start, const float4* pos4, const int32_t* cell, const TapeView& V,
                             cudaStream_t st)
{
    if (prec == 64) save_tape_t<double>(dim, n, nstart, S, vr, R, start, pos4, cell, V, st);
    else save_tape_t<float>(dim, n, nstart, S, vr, R, start, pos4, cell, V, st);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_step(int prec, int dim, int n, const TapeView& V, const Grid& G, const void* K,
                                const AdjView& A, int step_mode, cudaStream_t st)
{
    if (prec == 64) {
        const Consts<double>& k = *(const Consts<double>*)K;
        if (dim == 2) adjoint_step_t<double, 2>(n, V, G, k, A, step_mode, st);
        else adjoint_step_t<double, 3>(n, V, G, k, A, step_mode, st);
    } else {
        const Consts<float>& k = *(const Consts<float>*)K;
        if (dim == 2) adjoint_step_t<float, 2>(n, V, G, k, A, step_mode, st);
        else adjoint_step_t<float, 3>(n, V, G, k, A, step_mode, st);
    }
    return cudaGetLastError();
}

}  // namespace sphtv
