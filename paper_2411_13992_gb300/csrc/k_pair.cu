// k_pair.cu -- the pair passes of libsphtv, one thread per cell-sorted
// particle, neighbours from the (2R+1)^D block of cells around it.
//
//   k_density : sigma_i = sum_j W(r_ij, h_ij) (self and walls included),
//               rho_i = rho0 sigma_i / sigma0_i (Eq. 8), stored as
//               rho_i - rho0 beside the half-step velocity (p = c^2 (rho -
//               rho0), Eq. 2, is formed where it is used).
//   k_forces  : for every fluid i, over j != i:
//                 Riemann interface pressure P* with the dissipation
//                 limiter (Eq. 5-6), pressure acceleration (Eq. 3),
//                 viscous acceleration (Eq. 7), residual R_i = sum_j V_j
//                 grad_i W_ij (Eq. 14); then the limiter chi_i (Eq. 15), the
//                 displacement dr_i = xi chi_i h^2 R_i (Eq. 16), the closing
//                 half kick, and FP64 partials of the diagnostics, folded in a
//                 fixed order by the blocks that finish last, which also set
//                 the next step size min(dt_ad, dt_ac) (Eq. 9-11, h = h_min).
//
// Readings: e_ij points from i to j (Riemann states); grad W_ij is
// grad_i W_ij = W'(r) (x_i - x_j)/r; V_j = m_j / rho_j; rho_bar is the mean
// density, c_bar = c; h_ij = (h_i + h_j)/2 (or max); a wall j stands in with
// rho_j = rho_i, p_j = p_i, V_j = m_j / rho_i and its prescribed velocity.
//
// FP64 form (this file): absolute FP64 positions, the nearest periodic
// image of each pair (fixed by the stencil step of its cell), plain sums;
// 1/rho_i once per particle.  FP32 form: k_pair32.cu.
#include <cmath>

#include "common.cuh"
#include "launch.h"
#include "pair_physics.cuh"
#include "pair_walk.cuh"

namespace sphtv {

// ============================================================== FP64 form

// Lanes per particle.  L = 1: one thread per particle, which at 38,912
// particles or more (256 threads on each of 152 SMs) keeps the FP64 pipe of
// every SM busy.  L > 1: a group of L consecutive lanes per particle for
// smaller problems, whose passes are bound by the latency of one thread's
// chain of FP64 operations (a few hundred per particle, some 60 cycles each):
// 2,500 particles with one thread each left half the SMs without a warp and
// one warp on the others.  The lanes of a group share the particle's
// candidates and neighbours; the per-particle work before and after the sums
// is done by one thread per particle in full warps, since the FP64 pipe
// serves a warp instruction whole, however few of its lanes are active.
// Measured, us a step (start of the comparison -> L = 1 / 4 / 8): 2-D 2,500
// particles 116 -> 99 / 48 / 42, 8,100: 115 -> 100 / 55 / 55, 20,000: 120 ->
// 103 / 102 / 113, 40,000: 250 -> 151 / 161 / 186; 3-D 4,096: 391 -> 358 /
// 122 / 93, 17,576: 397 -> 363 / 259 / 276, 64,000: 889 (now 809) / 823; 3-D
// with 8 / 16 lanes 343: 72.9 / 55.1, 1,331: 74.0 / 59.4, 2,197: 77.0 / 69.5.
template <int L> struct Lanes {
    static constexpr int kThreads = L == 1 ? 256 : 512;    // most threads of a block
};

// Threads of a block with L > 1 lanes per particle: what spreads the particles
// evenly over the SMs, whole warps; past that, blocks of 128 (L = 4) or 256.
static int lane_threads(int L, int n, int sms)
{
    const int64_t t = ((int64_t)n * L + sms - 1) / sms;
    const int full = L >= 8 ? 512 : 128;          // 64 particles a block: 32 KB of row bounds in 3-D
    return t > full ? (L >= 8 ? 256 : 128) : (t < 32 ? 32 : (int)((t + 31) / 32 * 32));
}

// Exact FP64 test and kernel value of the density pass for particle i: the
// candidate's image (the periodic image of the stencil step, which is the
// nearest one of every neighbour), r < 2 h_ij, and W added to sigma; true for
// a force neighbour (j != i, 0 < r < 2 h_ij).  The comparisons of
// non-negative doubles are made on their bit patterns (same order) by the
// integer ALU, off the FP64 pipe.  At uniform resolution sigma collects
// W / (a_D h^-D), the constant applied once at the end.
template <int DIM>
struct Density64 {
    int n, i;
    const Grid& G;
    const Consts<double>& K;
    const StateSet<double>& S;
    double xi[3];
    int ci[3];
    double hi;
    double sigma;

    __device__ __forceinline__ Density64(int n_, int i_, const Grid& G_, const Consts<double>& K_,
                                         const StateSet<double>& S_, int cell_i)
        : n(n_), i(i_), G(G_), K(K_), S(S_), sigma(0.0)
    {
#pragma unroll
        for (int d = 0; d < 3; ++d) xi[d] = d < DIM ? S.x[(size_t)d * n + i] : 0.0;
        hi = S.h[i];
        cell_decode(G, cell_i, ci);
    }

    // the largest support radius 2 h_ij of any pair of i (h_j <= h_max)
    __device__ __forceinline__ float reach() const
    {
        return K.uniform_h ? K.reach_u : (float)(2.0 * pair_h(K, hi, K.h_u));
    }

    __device__ __forceinline__ bool exact(int j, uint32_t code)
    {
        const bool uni = K.uniform_h != 0;
        const int step[3] = {(int)(code % kSide) - kStencilR, (int)((code / kSide) % kSide) - kStencilR,
                             (int)(code / (kSide * kSide)) - kStencilR};
        double r2 = 0.0;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            double t = __dsub_rn(xi[d], S.x[(size_t)d * n + j]);
            if (G.periodic[d]) {
                const int sc = ci[d] + step[d];
                if (sc >= G.nc[d]) t = __dsub_rn(t, G.L[d]);
                else if (sc < 0) t = __dadd_rn(t, G.L[d]);
            }
            r2 += t * t;
        }
        const bool apart = __double_as_longlong(r2) != 0;                // r2 >= +0
        const double r = apart ? sqrt_pos(r2) : 0.0;
        // r < 2 h_ij (a NaN has a pattern above every finite value's)
        const unsigned long long rb = (unsigned long long)__double_as_longlong(r);
        if (uni) {
            if (!(rb < (unsigned long long)__double_as_longlong(K.two_h_u))) return false;
            // t = 1 - q/2 and 2q + 1 with q = r/h, each one fused operation
            const double t = fma(-K.half_inv_h_u, r, 1.0);
            const double t2 = t * t;
            sigma = fma(t2 * t2, fma(K.two_inv_h_u, r, 1.0), sigma);
        } else {
            const double hij = pair_h(K, hi, S.h[j]);
            if (!(rb < (unsigned long long)__double_as_longlong(2.0 * hij))) return false;
            sigma += wendland_W<DIM, double>(r, 1.0 / hij);
        }
        return j != i && apart;
    }
};

// FP32 prefilter of a candidate (1e-4 margin): the squared bound of the pair
// (i, j), pj_w = (float)h_j when h varies.
__device__ __forceinline__ float prefilter2(const Consts<double>& K, float hi_f, float pj_w)
{
    if (K.uniform_h) return K.prefilter2_u;
    const float lim = 2.f * (K.h_pair_max ? fmaxf(hi_f, pj_w) : 0.5f * (hi_f + pj_w));
    return lim * lim * 1.0001f;
}

// End of the density pass for particle i: rho_i (Eq. 8), its velocity record
// {v, rho - rho0} (+inf marks a wall), and V_i = m_i / rho_i for the force
// pass.
template <int DIM>
__device__ __forceinline__ void density64_end(int n, int i, const Consts<double>& K, const StateSet<double>& S,
                                              double sigma, double4_32a* vr, double* vol)
{
    double vi[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < DIM; ++d) vi[d] = S.v[(size_t)d * n + i];
    if (S.kind[i]) {
        vr[i] = make_double4_32a(vi[0], vi[1], vi[2], __longlong_as_double(0x7ff0000000000000ll));
        return;
    }
    if (K.uniform_h) sigma *= K.w_norm_u;
    const double rho = __ddiv_rn(__dmul_rn(K.rho0, sigma), S.s0[i]);
    const double w = __dsub_rn(rho, K.rho0);
    vr[i] = make_double4_32a(vi[0], vi[1], vi[2], w);
    if (vol) vol[i] = S.m[i] / (K.rho0 + w);
}

// Candidates come from the clipped FP32 row walk over the cell-relative
// positions (pos4); a loose FP32 test drops the far ones and the exact FP64
// test (minimum image, sqrt(r2) < 2 h_ij) decides the rest.  The walk visits
// candidates in the order of the cell scan (cells by dz, dy, dx, then index),
// so sigma is summed in the same order as a plain scan would.  With nbl
// non-null it also writes the particle's neighbour list (j != i,
// 0 < r < 2 h_ij), transposed (entry k at nbl[k * n + i] = j << kCodeBits),
// and the count (which may exceed cap); the FP64 force pass walks it.
template <int DIM>
__device__ __forceinline__ double density64_thread(int n, int i, const StateSet<double>& S,
                                                   const int32_t* start, const Grid& G,
                                                   const Consts<double>& K, const float4* pos4,
                                                   const int32_t* cell_of, uint32_t* nbl,
                                                   int32_t* nbc, int cap, bool two_pass)
{
    const float4 pi = pos4[i];
    const float oi[3] = {pi.x, pi.y, pi.z};
    const int cell_i = cell_of[i];
    Density64<DIM> D(n, i, G, K, S, cell_i);
    const float reach = D.reach();
    const float hi_f = K.uniform_h ? 0.f : (float)D.hi;      // read at variable resolution only
    int cnt = 0;
    bool staged = false;
    if (nbl && two_pass) {
        // two passes: the walk stages the candidates that pass the prefilter
        // in the particle's list, then the exact FP64 test runs over them
        // with every lane busy (the FP64 pipe serves a warp instruction
        // whole, however few of its lanes are active), and the list is
        // compacted in place to the force neighbours.  Same tests, in the
        // same order, as the one pass.
        int nf = 0;
        uint32_t* lp = nbl + i;
        auto stage = [&](int j, uint32_t code, const float4& pj, float r2f, float, float, float) {
            if (!(r2f <= prefilter2(K, hi_f, pj.w))) return;
            if (nf < cap) {
                *lp = ((uint32_t)j << kCodeBits) | code;
                lp += n;
            }
            ++nf;
        };
        for_candidates_rows<DIM, false>(oi, reach, cell_i, G, start, cell_of, pos4, stage);
        if (nf <= cap) {
            staged = true;
            for (int k = 0; k < nf; ++k) {
                const uint32_t e = nbl[(size_t)k * n + i];
                const int j = (int)(e >> kCodeBits);
                if (D.exact(j, e & ((1u << kCodeBits) - 1u))) {
                    if (cnt != k) nbl[(size_t)cnt * n + i] = e;     // entries before a rejected one stay in place
                    ++cnt;
                }
            }
        }
    }
    if (!staged) {
        // one pass: the exact test inside the walk (the lanes whose candidate
        // passed the prefilter run it while the others wait)
        auto visit = [&](int j, uint32_t code, const float4& pj, float r2f, float, float, float) {
            if (!(r2f <= prefilter2(K, hi_f, pj.w))) return;
            if (D.exact(j, code) && nbl) {
                if (cnt < cap) nbl[(size_t)cnt * n + i] = ((uint32_t)j << kCodeBits) | code;
                ++cnt;
            }
        };
        for_candidates_rows<DIM, false>(oi, reach, cell_i, G, start, cell_of, pos4, visit);
    }
    if (nbc) nbc[i] = cnt;
    return D.sigma;
}

// The density pass of a particle by a group of L lanes: the lanes first find
// the bounds of the stencil rows (one row per lane at a time, so that the
// loads of all rows are in flight together), then walk each row L candidates
// at a time, staging the ones that pass the prefilter in the particle's list
// in the order of the walk (a ballot gives each its place), then run the
// exact test over the staged ones L at a time, compacting the list.  Returns
// the lane's part of sigma.  Called by whole warps; `active` is the same for
// all lanes of a group.
template <int DIM, int L>
__device__ __forceinline__ double density64_group(int n, int i, bool active, RowRuns* rows,
                                                  const StateSet<double>& S, const int32_t* start,
                                                  const Grid& G, const Consts<double>& K,
                                                  const float4* pos4,
                                                  const int32_t* cell_of, uint32_t* nbl,
                                                  int32_t* nbc, int cap)
{
    constexpr int R = kStencilR, NR = DIM == 3 ? kSide * kSide : kSide;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, q = lane & (L - 1);
    const unsigned below = (1u << lane) - 1u, group = ((L == 32 ? 0u : (1u << L)) - 1u) << (lane - q);
    const float4 pi = pos4[i];
    const float oi[3] = {pi.x, pi.y, pi.z};
    const int cell_i = cell_of[i];
    Density64<DIM> D(n, i, G, K, S, cell_i);
    const float reach = D.reach();
    const float hi_f = K.uniform_h ? 0.f : (float)D.hi;      // read at variable resolution only
    for (int r = q; r < NR; r += L) {
        RowRuns rr = {0, 0, 0, 0, 0};
        if (active) rr = row_runs<DIM>(r, oi, reach, D.ci, G, start);
        rows[r] = rr;
    }
    __syncwarp();
    const float ex = G.edgef[0], ey = G.edgef[1], ez = G.edgef[2];
    // the rows' candidates that pass the prefilter, L at a time, in the order of
    // the walk: `keep` says which of them to count and to list
    auto walk_rows = [&](bool walk, auto&& keep) {
        int got = 0;
        for (int r = 0; r < NR; ++r) {
            const RowRuns rr = rows[r];
            const int len = walk ? rr.n0 + rr.n1 : 0;
            const int most = __reduce_max_sync(kAll, len);
            const int dy = r % kSide - R, dz = DIM == 3 ? r / kSide - R : 0;
            for (int f0 = 0; f0 < most; f0 += L) {
                const int f = f0 + q;
                bool take = false;
                uint32_t e = 0;
                if (f < len) {
                    const int j = f < rr.n0 ? rr.j0 + f : rr.j1 + (f - rr.n0);
                    const float4 pj = pos4[j];
                    int dx = cell_of[j] - rr.row - D.ci[0];
                    if (dx > R) dx -= G.nc[0];                    // across the periodic x boundary
                    else if (dx < -R) dx += G.nc[0];
                    const float rx = (oi[0] - pj.x) - (float)dx * ex;
                    const float ry = (oi[1] - pj.y) - (float)dy * ey;
                    float r2 = rx * rx + ry * ry;
                    if (DIM == 3) {
                        const float rz = (oi[2] - pj.z) - (float)dz * ez;
                        r2 += rz * rz;
                    }
                    const uint32_t code = (uint32_t)((dx + R) + kSide * (dy + R) + kSide * kSide * (dz + R));
                    e = ((uint32_t)j << kCodeBits) | code;
                    take = r2 <= prefilter2(K, hi_f, pj.w) && keep(j, code);
                }
                const unsigned m = __ballot_sync(kAll, take) & group;
                const int at = got + __popc(m & below);
                if (take && at < cap) nbl[(size_t)at * n + i] = e;
                got += __popc(m);
            }
        }
        return got;
    };
    const int nf = walk_rows(true, [](int, uint32_t) { return true; });
    __syncwarp();
    int cnt = 0;
    const bool fits = nf <= cap;
    const int most = __reduce_max_sync(kAll, fits ? nf : 0);
    for (int k0 = 0; k0 < most; k0 += L) {
        const int k = k0 + q;
        bool keep = false;
        uint32_t e = 0;
        if (fits && k < nf) {
            e = nbl[(size_t)k * n + i];
            const int j = (int)(e >> kCodeBits);
            keep = D.exact(j, e & ((1u << kCodeBits) - 1u));
        }
        const unsigned m = __ballot_sync(kAll, keep) & group;
        const int at = cnt + __popc(m & below);
        if (keep && at != k) nbl[(size_t)at * n + i] = e;
        cnt += __popc(m);
    }
    // more candidates than the list holds: the lanes walk them again with the
    // exact test inside the walk (as the force pass shares the cells; by one lane
    // alone a step of 32^3 particles at h = 1.82 dp took 12.96 ms, shared 3.96,
    // with one thread per particle 4.21)
    if (__any_sync(kAll, active && !fits)) {
        const int again = walk_rows(active && !fits, [&](int j, uint32_t code) { return D.exact(j, code); });
        if (!fits) cnt = again;
    }
    if (active && q == 0) nbc[i] = cnt;
    return D.sigma;
}

template <int DIM, int L>
__global__ void __launch_bounds__(Lanes<L>::kThreads, L == 1 ? 4 : 1) k_density_f64(int n, StateSet<double> S,
                                                     const int32_t* start, Grid G, Consts<double> K,
                                                     double4_32a* vr, const float4* pos4,
                                                     const int32_t* cell_of, uint32_t* nbl,
                                                     int32_t* nbc, int cap, double* vol)
{
    pdl_wait();
    if constexpr (L == 1) {
        const int i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i >= n) return;
        double sigma = 0.0;
        if (S.kind[i]) {
            if (nbc) nbc[i] = 0;
        } else {
            sigma = density64_thread<DIM>(n, i, S, start, G, K, pos4, cell_of, nbl, nbc, cap, true);
        }
        density64_end<DIM>(n, i, K, S, sigma, vr, vol);
    } else {
        // shared memory: each particle's row bounds, then its lanes' sums
        constexpr int NR = DIM == 3 ? kSide * kSide : kSide;
        extern __shared__ __align__(16) unsigned char smem64[];
        RowRuns* rows = reinterpret_cast<RowRuns*>(smem64);
        double* sums = reinterpret_cast<double*>(smem64 + ((size_t)(blockDim.x / L) * NR * sizeof(RowRuns) + 15) / 16 * 16);
        const int P = blockDim.x / L, p = threadIdx.x / L;
        const int i = blockIdx.x * P + p;
        const bool active = i < n && S.kind[i] == 0;
        sums[threadIdx.x] = density64_group<DIM, L>(n, min(i, n - 1), active, rows + (size_t)p * NR, S, start, G, K,
                                                    pos4, cell_of, nbl, nbc, cap);
        __syncthreads();
        const int ie = blockIdx.x * P + threadIdx.x;
        if (threadIdx.x < P && ie < n) {
            if (S.kind[ie]) nbc[ie] = 0;
            double sigma = 0.0;
            for (int k = 0; k < L; ++k) sigma += sums[threadIdx.x * L + k];
            density64_end<DIM>(n, ie, K, S, sigma, vr, vol);
        }
    }
}

// The pair sums of particle i over its neighbours k0, k0 + dk, ... of the
// list, or over the stencil's cells k0, k0 + dk, ... when there is no list (or
// more neighbours than it holds).
template <int DIM>
__device__ __forceinline__ void forces64_sums(int n, int i, const StateSet<double>& S,
                                              const int32_t* start, const Grid& G,
                                              const Consts<double>& K, const double4_32a* vr,
                                              const int32_t* cell_of,
                                              const uint32_t* nbl, int cnt, int cap, int k0, int dk,
                                              const double* vol, PairSums64<DIM>& sums)
{
    double xi[3] = {0, 0, 0}, vi[3] = {0, 0, 0};
    const double4_32a me = vr[i];
    vi[0] = me.x; vi[1] = me.y; vi[2] = me.z;
#pragma unroll
    for (int d = 0; d < DIM; ++d) xi[d] = S.x[(size_t)d * n + i];
    const double hi = S.h[i];
    // uniform resolution: h_ij = h for every pair, and W'/r = C t^3 (t = 1 - r
    // / 2h) leaves C out of the sums
    const bool uni = K.uniform_h != 0;
    int ci[3];
    cell_decode(G, cell_of[i], ci);
    const PairI64 I = pair_i64(K, me.w);
    // a neighbour j (0 < r < 2 h_ij) at rv = x_i - x_j, r2 = |rv|^2
    auto body = [&](int j, const double* rv, double r2) {
        const double inv_r = rsqrt_pos(r2);
        const double r = r2 * inv_r;
        double g;
        if (uni) {
            const double t = fma(-K.half_inv_h_u, r, 1.0);
            g = t * t * t;
        } else {
            g = wendland_dW<DIM, double>(r, 1.0 / pair_h(K, hi, S.h[j])) * inv_r;
        }
        const double4_32a oj = vr[j];
        const double vj[3] = {oj.x, oj.y, oj.z};
        double w_j = oj.w, V_j = vol[j];
        const bool wall = is_wall(w_j);
        if (__any_sync(__activemask(), wall)) {
            // a wall stands in with rho_j = rho_i: w_j = w_i, V_j = m_j / rho_i
            if (wall) {
                w_j = me.w;
                V_j = S.m[j] / (K.rho0 + me.w);
            }
        }
        pair_force64<DIM>(K, I, rv, inv_r, g, vi, vj, w_j, V_j, sums);
    };
    if (cnt <= cap) {
        // the density pass's list: exactly the pairs with 0 < r < 2 h_ij
        // (its exact FP64 test), in the order of the cell scan below, so
        // no test is repeated here.  The stencil step of j's cell fixes
        // the periodic image (the nearest one for every neighbour: the
        // same operations as min_image).
        for (int k = k0; k < cnt; k += dk) {
            const uint32_t e = nbl[(size_t)k * n + i];
            const int j = (int)(e >> kCodeBits);
            const int code = (int)(e & ((1u << kCodeBits) - 1u));
            const int step[3] = {code % kSide - kStencilR, (code / kSide) % kSide - kStencilR,
                                 code / (kSide * kSide) - kStencilR};
            double rv[3] = {0, 0, 0};
            double r2 = 0.0;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                double t = __dsub_rn(xi[d], S.x[(size_t)d * n + j]);
                if (G.periodic[d]) {
                    const int sc = ci[d] + step[d];
                    if (sc >= G.nc[d]) t = __dsub_rn(t, G.L[d]);
                    else if (sc < 0) t = __dadd_rn(t, G.L[d]);
                }
                rv[d] = t;
                r2 += t * t;
            }
            body(j, rv, r2);
        }
    } else {
        // no list (or more neighbours than it holds): scan the cells k0, k0 + dk,
        // ... of the stencil with the minimum image and the support test
        constexpr int cells = DIM == 3 ? kSide * kSide * kSide : kSide * kSide;
        for (int t = k0; t < cells; t += dk) {
            const int cx = cell_step(G, ci[0], t % kSide - kStencilR, 0);
            const int cy = cell_step(G, ci[1], t / kSide % kSide - kStencilR, 1);
            const int cz = DIM == 3 ? cell_step(G, ci[2], t / (kSide * kSide) - kStencilR, 2) : 0;
            if (cx < 0 || cy < 0 || cz < 0) continue;
            const int cell = cx + G.nc[0] * (cy + G.nc[1] * cz);
            for (int j = start[cell]; j < start[cell + 1]; ++j) {
                if (j == i) continue;
                double rv[3] = {0, 0, 0};
                double r2 = 0.0;
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    rv[d] = min_image(G, xi[d], S.x[(size_t)d * n + j], d);
                    r2 += rv[d] * rv[d];
                }
                const double hij = uni ? K.h_u : pair_h(K, hi, S.h[j]);
                if (r2 > 4.0 * hij * hij * (1.0 + 1e-12)) continue;
                if (!(r2 > 0.0)) continue;
                if (!(sqrt_pos(r2) < 2.0 * hij)) continue;     // as the density pass decides
                body(j, rv, r2);
            }
        }
    }
}

// L lanes per particle (see Lanes): lane q of a group takes the neighbours
// q, q + L, ...; their sums meet in shared memory, where one thread per
// particle adds them in lane order and ends the particle's step.
template <int DIM, int L>
__global__ void __launch_bounds__(Lanes<L>::kThreads, L == 1 ? 2 : 1) k_forces_f64(int n, StateSet<double> S,
                                                    const int32_t* start, Grid G, Consts<double> K,
                                                    const double4_32a* vr,
                                                    const int32_t* cell_of,
                                                    const uint32_t* nbl, const int32_t* nbc,
                                                    int cap, const double* dt_ptr, int kick_on,
                                                    int write_ad, double* Rout,
                                                    double* chi_out, GridSum B, DtConsts Dc,
                                                    double* diag, double* dt_next, int count_step,
                                                    const double* vol)
{
    pdl_wait();
    const int P = blockDim.x / L;
    PairSums64<DIM> sums;
    if constexpr (L == 1) {
        const int i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i < n && S.kind[i] == 0)
            forces64_sums<DIM>(n, i, S, start, G, K, vr, cell_of, nbl, nbl ? nbc[i] : cap + 1, cap, 0, 1, vol, sums);
    } else {
        extern __shared__ __align__(16) unsigned char smem64[];
        double* part = reinterpret_cast<double*>(smem64);       // [3 DIM][blockDim.x]
        const int i = blockIdx.x * P + threadIdx.x / L;
        if (i < n && S.kind[i] == 0)
            forces64_sums<DIM>(n, i, S, start, G, K, vr, cell_of, nbl, nbc[i], cap, threadIdx.x % L, L, vol, sums);
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            part[(3 * d + 0) * blockDim.x + threadIdx.x] = sums.P[d];
            part[(3 * d + 1) * blockDim.x + threadIdx.x] = sums.V[d];
            part[(3 * d + 2) * blockDim.x + threadIdx.x] = sums.R[d];
        }
        __syncthreads();
        sums = PairSums64<DIM>();
        if (threadIdx.x < P) {
#pragma unroll
            for (int d = 0; d < DIM; ++d)
                for (int q = 0; q < L; ++q) {
                    sums.P[d] += part[(3 * d + 0) * blockDim.x + threadIdx.x * L + q];
                    sums.V[d] += part[(3 * d + 1) * blockDim.x + threadIdx.x * L + q];
                    sums.R[d] += part[(3 * d + 2) * blockDim.x + threadIdx.x * L + q];
                }
        }
    }
    // the end of the step, one thread per particle
    const int i = blockIdx.x * P + threadIdx.x;
    double part[kNPart];
#pragma unroll
    for (int k = 0; k < kNPart; ++k) part[k] = 0.0;
    const double dt = *dt_ptr;
    const double hdt = kick_on ? 0.5 * dt : 0.0;
    if (threadIdx.x < P && i < n) {
        if (S.kind[i] == 0) {
            const double4_32a me = vr[i];
            const double vi[3] = {me.x, me.y, me.z};
            const double rho_i = K.rho0 + me.w;
            const double inv_rho_i = 1.0 / rho_i;
            const double hi = S.h[i];
            // W'/r = C t^3 at uniform resolution, C = -5 a_D h^-(D+2): C leaves the sums
            const double C = K.uniform_h ? K.dwr_coef_u : 1.0;
            const double fp = (-2.0 * C) * inv_rho_i, fv = (K.two_eta * C) * inv_rho_i;
            double a[3] = {0, 0, 0}, R[3] = {0, 0, 0};
            double R2 = 0.0;
            const double m_i = S.m[i];
            // free-stream forcing lambda(x) (U_inf - v) of the fringe region
            const double lam = K.fr_on ? fringe_rate<double>(K, S.x[i]) : 0.0;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                const double pair_a = fma(fp, sums.P[d], fv * sums.V[d]);
                // the fluid's momentum rate from its pair terms: minus the force on the walls
                if (K.body_force) part[9 + d] = m_i * pair_a;
                a[d] = K.g[d] + pair_a;
                if (K.fr_on) a[d] += lam * (K.fr_u[d] - vi[d]);
                R[d] = C * sums.R[d];
                R2 += R[d] * R[d];
            }
            const double htv = K.tv_h_particle ? hi : K.h_min;
            const double htv2 = htv * htv;
            const double chi = tv_limiter(K, htv2 * R2);
            // Eq. 12 (background pressure p0 = rho0 c^2): dr = dt^2/2 a_bg = -(dt^2 p0 / rho_i) R_i
            const bool bgmode = K.tv_mode == SPH_TV_BACKGROUND;
            const double bg = bgmode ? -(dt * dt * (K.rho0 * K.c2) / rho_i) : 0.0;
            // 1/dt once per particle: the transport speed is a diagnostic
            const double inv_dt = dt > 0.0 ? 1.0 / dt : 0.0;
            double v2 = 0.0, vt2 = 0.0, dr2 = 0.0;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                size_t o = (size_t)d * n + i;
                double dr = bgmode ? bg * R[d] : K.tv_xi * chi * htv2 * R[d];
                double vn = __dadd_rn(vi[d], __dmul_rn(hdt, a[d]));
                if (write_ad) {
                    S.a[o] = a[d];
                    S.dr[o] = dr;
                }
                S.v[o] = vn;
                Rout[o] = R[d];
                part[1 + d] = m_i * vn;
                v2 += vn * vn;
                dr2 += dr * dr;
                const double vt = fma(dr, inv_dt, vn);
                vt2 += vt * vt;
            }
            chi_out[i] = chi;
            part[0] = m_i;
            part[4] = 0.5 * m_i * v2;
            part[5] = chi > 0.0 ? 1.0 : 0.0;
            part[6] = v2;                 // squares: the roots are taken at the very end
            part[7] = vt2;
            part[8] = dr2;
        } else {
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                if (write_ad) {
                    S.a[(size_t)d * n + i] = 0.0;
                    S.dr[(size_t)d * n + i] = 0.0;
                }
                Rout[(size_t)d * n + i] = 0.0;
            }
            chi_out[i] = 0.0;
        }
    }
    __shared__ double total[kNPart];
    if (grid_partials(part, B, total, true, K.body_force != 0)) finish_step(total, Dc, diag, dt_next, count_step);
}

// ================================================ diagnostics only

// FP64 partials of the diagnostics from the stored v and dr (no pair work):
// used when the caller supplied a and dr, so no force pass is needed.
template <typename Real, int DIM>
__global__ void __launch_bounds__(256) k_diag_only(int n, StateSet<Real> S, GridSum B, DtConsts D,
                                                   double* diag, double* dt_next, int count_step)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    double part[kNPart];
#pragma unroll
    for (int k = 0; k < kNPart; ++k) part[k] = 0.0;
    if (i < n && S.kind[i] == 0) {
        const double m_i = S.m[i];
        double v2 = 0.0, dr2 = 0.0;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            double v = (double)S.v[(size_t)d * n + i];
            double dr = (double)S.dr[(size_t)d * n + i];
            part[1 + d] = m_i * v;
            v2 += v * v;
            dr2 += dr * dr;
        }
        part[0] = m_i;
        part[4] = 0.5 * m_i * v2;
        part[6] = v2;                 // squares: block_partials takes the roots
        part[7] = v2;
        part[8] = dr2;
    }
    __shared__ double total[kNPart];
    if (grid_partials(part, B, total)) finish_step(total, D, diag, dt_next, count_step);
}

// The rows of a large grid (see GridSum), and the end of the step.
__global__ void __launch_bounds__(256) k_fold_step(GridSum B, int nrows, DtConsts D, double* diag,
                                                   double* dt_ptr, int count_step)
{
    pdl_wait();
    __shared__ double total[kNPart];
    if (fold_grid(B, nrows, total)) finish_step(total, D, diag, dt_ptr, count_step);
}

// ============================================================ launchers

static inline int nblk(int n, int t) { return (n + t - 1) / t; }

// Threads per block of the pair passes: 256 (FP64) or 128 (FP32) when the
// particles fill every SM at that size; smaller blocks (down to one warp)
// when they do not, so that a small problem still spreads over all SMs
// instead of queueing its FP64 work on a few.  FP64 between one and eight
// full blocks per SM: 64, since the FP64 pipe is the bound and a pass takes
// as long as the SM with the most blocks (40,000 particles: 157 blocks of 256
// on 152 SMs, 208 us a step against 151 with 64; 64,000 in 3-D: 889 against
// 809 us; 96^3: the same).
int pair_threads(int prec, int n, int sms)
{
    const int full = prec == 64 ? 256 : 128;
    if (sms <= 0) sms = 152;
    if ((int64_t)n >= (int64_t)sms * full) return prec == 64 && (int64_t)n < (int64_t)sms * full * 8 ? 64 : full;
    int t = ((n + sms - 1) / sms + 31) / 32 * 32;
    return t < 32 ? 32 : (t > full ? full : t);
}

// The FP64 pair passes with neighbour lists: lanes per particle (see Lanes),
// threads per block and blocks.
struct Lane64 {
    int L, T, blocks;
};

static Lane64 lanes64(int dim, int n, int sms)
{
    if (sms <= 0) sms = 152;
    const int L = n >= sms * 256 ? 1 : (n >= sms * 64 ? 4 : (dim == 2 || n >= sms * 16 ? 8 : 16));
    const int T = L == 1 ? pair_threads(64, n, sms) : lane_threads(L, n, sms);
    return Lane64{L, T, nblk(n, T / L)};
}

#define SPH_LANES64(kernel, DIM, L) \
    ((L) == 1 ? kernel<DIM, 1> : (L) == 4 ? kernel<DIM, 4> : (L) == 8 ? kernel<DIM, 8> : kernel<DIM, (DIM) == 3 ? 16 : 8>)

int pair_blocks(int prec, int n, int sms) { return nblk(n, pair_threads(prec, n, sms)); }

GridSum grid_sum(const FinishArgs& F, int nblocks)
{
    int group = nblocks;
    if (nblocks > kInlineBlocks) group = 0;
    else if (nblocks > kFoldRows) group = (int)std::ceil(std::sqrt((double)nblocks));
    return GridSum{F.partials, F.rows, F.counters, group};
}

int grid_groups() { return kMaxGroups; }

DtConsts dt_consts(const sph_params& P)
{
    const double nu = P.eta / P.rho0;
    return DtConsts{std::fmax(nu / P.h_min, P.u_ref), P.cfl_ad * P.h_min, P.cfl_ac * P.h_min, P.c0, P.fixed_dt};
}

cudaError_t launch_density(int prec, int dim, int n, void* S, const int32_t* start, const Grid& G, const void* K,
                           void* vr, const float4* pos4, const int32_t* cell_of, uint32_t* nbl, int32_t* nbc,
                           cudaStream_t st, double* vol, const float4* pos4c, int tiles)
{
    if (prec == 32) return launch_density32(dim, n, S, start, G, K, vr, pos4, cell_of, nbl, nbc, st, pos4c, tiles);
    auto s = *(StateSet<double>*)S;
    auto k = *(const Consts<double>*)K;
    const int cap = nbl_capacity(dim);
    const Lane64 Q = nbl ? lanes64(dim, n, G.sms) : Lane64{1, pair_threads(64, n, G.sms), nblk(n, pair_threads(64, n, G.sms))};
    const size_t smem = Q.L == 1 ? 0 : ((size_t)(Q.T / Q.L) * (dim == 3 ? kSide * kSide : kSide) * sizeof(RowRuns) + 15) / 16 * 16 +
                                           Q.T * sizeof(double);
    auto kern = dim == 2 ? SPH_LANES64(k_density_f64, 2, Q.L) : SPH_LANES64(k_density_f64, 3, Q.L);
    launch(kern, Q.blocks, Q.T, smem, st, n, s, start, G, k, (double4_32a*)vr, pos4, cell_of, nbl, nbc, cap, vol);
    return cudaGetLastError();
}

cudaError_t launch_forces(int prec, int dim, int n, void* S, const int32_t* start, const Grid& G, const void* K,
                          const float* mf, const void* vr, const float4* pos4, const int32_t* cell_of,
                          const uint32_t* nbl, const int32_t* nbc, int kick_on, int write_ad,
                          void* Rout, void* chi, const FinishArgs& F, cudaStream_t st, const double* vol)
{
    if (prec == 32)
        return launch_forces32(dim, n, S, start, G, K, mf, vr, pos4, cell_of, nbl, nbc, kick_on, write_ad, Rout, chi,
                               F, st);
    auto s = *(StateSet<double>*)S;
    auto k = *(const Consts<double>*)K;
    const int cap = nbl_capacity(dim);
    const Lane64 Q = lanes64(dim, n, G.sms);
    const GridSum B = grid_sum(F, Q.blocks);
    const DtConsts D = dt_consts(*F.P);
    const size_t smem = Q.L == 1 ? 0 : (size_t)3 * dim * Q.T * sizeof(double);
    auto kern = dim == 2 ? SPH_LANES64(k_forces_f64, 2, Q.L) : SPH_LANES64(k_forces_f64, 3, Q.L);
    launch(kern, Q.blocks, Q.T, smem, st, n, s, start, G, k, (const double4_32a*)vr, cell_of, nbl, nbc, cap, F.dt, kick_on,
                                      write_ad, (double*)Rout, (double*)chi, B, D, F.diag, F.dt, F.count_step, vol);
    return cudaGetLastError();
}

cudaError_t launch_finish_step(int prec, int n, int sms, const FinishArgs& F, cudaStream_t st, int64_t* launches)
{
    // (the FP64 passes of more than kInlineBlocks blocks have one lane per particle)
    const int nb = pair_blocks(prec, n, sms);
    const GridSum B = grid_sum(F, nb);
    if (B.group) return cudaSuccess;      // the pass folded its partials itself
    launch(k_fold_step, kFoldBlocks, 256, 0, st, B, nb, dt_consts(*F.P), F.diag, F.dt, F.count_step);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_diag_only(int prec, int dim, int n, void* S, const FinishArgs& F, int sms, cudaStream_t st)
{
    const int T = pair_threads(prec, n, sms);   // one partials row per block of the force pass
    const GridSum B = grid_sum(F, nblk(n, T));
    const DtConsts D = dt_consts(*F.P);
    if (prec == 64) {
        auto s = *(StateSet<double>*)S;
        if (dim == 2) launch(k_diag_only<double, 2>, nblk(n, T), T, 0, st, n, s, B, D, F.diag, F.dt, F.count_step);
        else launch(k_diag_only<double, 3>, nblk(n, T), T, 0, st, n, s, B, D, F.diag, F.dt, F.count_step);
    } else {
        auto s = *(StateSet<float>*)S;
        if (dim == 2) launch(k_diag_only<float, 2>, nblk(n, T), T, 0, st, n, s, B, D, F.diag, F.dt, F.count_step);
        else launch(k_diag_only<float, 3>, nblk(n, T), T, 0, st, n, s, B, D, F.diag, F.dt, F.count_step);
    }
    return cudaGetLastError();
}

}  // namespace sphtv
