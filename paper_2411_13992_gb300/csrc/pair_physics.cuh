// pair_physics.cuh -- per-pair arithmetic of the method used by the pair
// kernels: pair smoothing length, the transport-velocity limiter (Eq. 15),
// one neighbour's contribution to the pressure (Eq. 3, 5-6) and viscous
// (Eq. 7) accelerations and to the residual of Eq. 14 in the FP64 form (the
// FP32 form is pair_force32 in k_pair32.cu), and the block reduction of the
// FP64 diagnostics partials.
//
// Readings of the paper: e_ij points from i to j (Riemann states U_l, U_r);
// grad W_ij is grad_i W_ij = W'(r) (x_i - x_j)/r; V_j = m_j / rho_j;
// rho_bar = (rho_i + rho_j)/2, c_bar = c; a wall neighbour stands in with
// rho_j = rho_i, p_j = p_i (so V_j = m_j / rho_i) and its prescribed velocity.
#pragma once

#include "common.cuh"

namespace sphtv {

template <typename Real>
__device__ __forceinline__ Real pair_h(const Consts<Real>& K, Real hi, Real hj)
{
    return K.h_pair_max ? (hi > hj ? hi : hj) : Real(0.5) * (hi + hj);
}

template <typename Real>
__device__ __forceinline__ Real tv_limiter(const Consts<Real>& K, Real s)
{
    if (K.tv_mode == SPH_TV_OFF) return Real(0);
    if (K.tv_mode == SPH_TV_UNLIMITED || K.tv_mode == SPH_TV_BACKGROUND) return Real(1);
    if (s > K.tv_thresh) {
        Real t = K.tv_C * s;
        return t < Real(1) ? t : Real(1);
    }
    return Real(0);
}

// 1/sqrt(x) and sqrt(x) for a normal x > 0 in six FP64 operations: the
// hardware's approximation y0 (from the upper word of x only), then one step
// of Householder's third-order iteration for x^(-1/2), y0 (1 + e/2 + 3 e^2/8)
// with e = 1 - x y0^2.  The error left by the iteration is O(e^3) < 2^-58, so
// that both results are within one unit in the last place of the exact values
// (largest errors found over all exponents 0.98 and 0.76).  For a
// subnormal x (a pair closer than 1.5e-154) the seed is that of the smallest
// normal number (an integer maximum on the upper word), and both results are
// finite.
__device__ __forceinline__ double rsqrt_seed(double x)
{
    double y;
    const double xn = __hiloint2double(max(__double2hiint(x), 0x00100000), __double2loint(x));
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(xn));
    return y;
}

__device__ __forceinline__ double sqrt_pos(double x)
{
    const double y0 = rsqrt_seed(x);
    const double g = x * y0;
    const double e = fma(-g, y0, 1.0);
    return fma(g * e, fma(0.375, e, 0.5), g);
}

__device__ __forceinline__ double rsqrt_pos(double x)
{
    const double y0 = rsqrt_seed(x);
    const double e = fma(-(x * y0), y0, 1.0);
    return fma(y0 * e, fma(0.375, e, 0.5), y0);
}

// Per-particle values of i shared by all pairs of i in the FP64 force pass.
struct PairI64 {
    double w;          // rho_i - rho0
    double hp;         // p_i / 2 = (c^2 / 2) w_i
    double crho;       // (c/2)(rho0 + w_i / 2): (c/2) rho_bar = crho + (c/4) w_j
};

__device__ __forceinline__ PairI64 pair_i64(const Consts<double>& K, double w)
{
    PairI64 I;
    I.w = w;
    I.hp = K.half_c2 * w;
    I.crho = K.half_c * fma(0.5, w, K.rho0);
    return I;
}

// The pair sums of particle i in the FP64 force pass, without the factors
// that all pairs of i share: P = sum V_j g P*_ij r_ij, V = sum V_j g v_ij,
// R = sum V_j g r_ij, where W'/r = C g (C a constant of the particle's
// resolution, 1 at variable resolution).  Then a_i = -2 C / rho_i P + 2 eta C
// / rho_i V and R_i = C R.
template <int DIM>
struct PairSums64 {
    double P[DIM], V[DIM], R[DIM];
    __device__ __forceinline__ PairSums64()
    {
#pragma unroll
        for (int d = 0; d < DIM; ++d) P[d] = V[d] = R[d] = 0.0;
    }
};

// min(max(x, 0), 1) by the sign and order of the binary64 bit pattern (the
// order of non-negative doubles is that of their patterns): integer selects
// instead of two FP64 comparisons.
__device__ __forceinline__ double clamp01(double x)
{
    const long long b = __double_as_longlong(x);
    if (b < 0) return 0.0;
    if (b >= 0x3ff0000000000000LL) return 1.0;
    return x;
}

// w = +inf marks a wall particle in the velocity record (a bit test: no
// FP64 comparison).
__device__ __forceinline__ bool is_wall(double w)
{
    return (__double_as_longlong(w) & 0x7fffffffffffffffLL) == 0x7ff0000000000000LL;
}

// Contribution of neighbour j to the sums of i in the FP64 form: Eq. 3
// (pressure, with P* of Eq. 5-6), Eq. 7 (viscous) and the residual of
// Eq. 14, arranged for the FP64 pipe (1/74 of the FP32 rate here): P* from
// the density deviations (p_i + p_j = c^2 (w_i + w_j), rho_bar = rho0 +
// (w_i + w_j)/2), the limiter's clamp on the integer ALU, one product V_j g
// that the three sums share, and every factor of i alone out of the pair
// (39 FP64 operations in 3-D).  rv = x_i - x_j, inv_r = 1/r, g = W'(r, h_ij)
// / (r C); w_j = rho_j - rho0 and V_j = m_j / rho_j, for a wall neighbour w_i
// and m_j / rho_i (the caller substitutes them).
template <int DIM>
__device__ __forceinline__ void pair_force64(const Consts<double>& K, const PairI64& I, const double* rv,
                                             double inv_r, double g, const double* vi, const double* vj,
                                             double w_j, double V_j, PairSums64<DIM>& S)
{
    double dv[3] = {0.0, 0.0, 0.0};
    double dvr = 0.0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        dv[d] = vi[d] - vj[d];
        dvr += dv[d] * rv[d];
    }
    const double du = -dvr * inv_r;                                   // U_l - U_r
    const double beta = clamp01(K.beta_k * du);
    const double hpsum = fma(K.half_c2, w_j, I.hp);                   // (p_i + p_j) / 2
    const double crhobar = fma(K.quarter_c, w_j, I.crho);               // (c/2) rho_bar
    const double pstar = fma(beta * du, crhobar, hpsum);
    const double vw = V_j * g;                                        // V_j W'/(r C)
    const double vwp = vw * pstar;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        S.P[d] = fma(vwp, rv[d], S.P[d]);
        S.V[d] = fma(vw, dv[d], S.V[d]);
        S.R[d] = fma(vw, rv[d], S.R[d]);
    }
}

// Free-stream forcing rate of the fringe region technique (Nordstrom, Nordin
// & Henningson 1999): lambda(x) = lambda_max [S((x - x0)/rise) - S((x -
// x1)/fall + 1)] with the smooth step S(t) = 1/(1 + exp(1/(t - 1) + 1/t)) on
// (0, 1), 0 below, 1 above; the acceleration gets lambda(x) (U_inf - v).
template <typename Real>
__device__ __forceinline__ Real fringe_step(Real t)
{
    if (t <= Real(0)) return Real(0);
    if (t >= Real(1)) return Real(1);
    return Real(1) / (Real(1) + exp(Real(1) / (t - Real(1)) + Real(1) / t));
}

template <typename Real>
__device__ __forceinline__ Real fringe_rate(const Consts<Real>& K, Real x)
{
    return K.fr_lambda *
           (fringe_step<Real>((x - K.fr_x[0]) / K.fr_x[2]) - fringe_step<Real>((x - K.fr_x[1]) / K.fr_x[3] + Real(1)));
}

// Block reduction of the diagnostics partials into out_block (layout: 0
// mass, 1-3 momentum, 4 KE, 5 n_chi, 6 max|v|, 7 max|v + dr/dt|, 8 max|dr|,
// 9-11 the fluid's momentum rate from its pair terms, sum m_i (a_i - g -
// forcing), whose negative is the force on the walls; zero unless the pass
// computes it).  On entry slot 5 is a 0/1 flag and slots 6-8 are the SQUARES
// of the magnitudes; in out_block slot 5 is an int64 count in a double's bits
// and slots 6-8 are still squares (the root of the largest square is the
// largest root, so one root per slot, taken at the very end, replaces one per
// block).  The sums are FP64 shuffle trees in a fixed order; the flags are
// counted with a ballot and the maxima of the non-negative squares are
// integer maxima of their bit patterns (a NaN counts as 0, as fmax ignores
// it), which keeps both off the FP64 pipe (1/74 of the FP32 rate on this
// part).  sums = false (the same for every thread of the grid) when the
// caller's sums are all zero: they are skipped, as in a warp without mass.
constexpr int kMaxWarps = 16;         // warps of a block of any pass that writes partials

__device__ __forceinline__ void block_partials(double* vals, double* out_block, bool sums = true, bool body = false)
{
    __shared__ double sh[kMaxWarps][kNPart];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    // slot 0 is a mass: a warp in which it is zero everywhere holds no fluid particle
    if (!sums || !__any_sync(0xffffffffu, __double_as_longlong(vals[0]) != 0)) {
        // the caller's sums are all zero: skip them
        if (lane == 0)
            for (int k = 0; k < 5; ++k) sh[w][k] = 0.0;
    } else {
        // the five sums as a transposing reduction: at each of the first three
        // levels a lane keeps half of its values and adds its partner's copy
        // of them (4 + 2 + 1 additions instead of 5 per level), then the last
        // two levels reduce one value per group of four lanes; value g ends in
        // lane 4 g (eight slots, the last three zero)
        double v8[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v8[k] = k < 5 ? vals[k] : 0.0;
        const bool hi16 = lane & 16, hi8 = lane & 8, hi4 = lane & 4;
        double a4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const double send = hi16 ? v8[j] : v8[4 + j];
            const double keep = hi16 ? v8[4 + j] : v8[j];
            a4[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
        double a2[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const double send = hi8 ? a4[j] : a4[2 + j];
            const double keep = hi8 ? a4[2 + j] : a4[j];
            a2[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
        double a1;
        {
            const double send = hi4 ? a2[0] : a2[1];
            const double keep = hi4 ? a2[1] : a2[0];
            a1 = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
        a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
        a1 += __shfl_xor_sync(0xffffffffu, a1, 1);
        const int g = (lane >> 2);   // value index held by this group of four lanes
        if ((lane & 3) == 0 && g < 5) sh[w][g] = a1;
    }
    // slots 9-11 (uniform over the grid: body is the same for every thread)
    if (body) {
#pragma unroll
        for (int k = 9; k < 12; ++k) {
            double x = vals[k];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
            if (lane == 0) sh[w][k] = x;
        }
    } else if (lane == 0) {
        for (int k = 9; k < 12; ++k) sh[w][k] = 0.0;
    }
    const unsigned flags = __ballot_sync(0xffffffffu, __double_as_longlong(vals[5]) != 0);
    if (lane == 0) sh[w][5] = __longlong_as_double((long long)__popc(flags));
#pragma unroll
    for (int k = 6; k <= 8; ++k) {
        long long b = __double_as_longlong(vals[k]);
        if ((b & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL) b = 0;      // NaN
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) b = max(b, __shfl_down_sync(0xffffffffu, b, off));
        if (lane == 0) sh[w][k] = __longlong_as_double(b);
    }
    __syncthreads();
    if (threadIdx.x < kNPart) {
        const int k = threadIdx.x;
        double x = sh[0][k];
        for (int t = 1; t < nw; ++t) {
            const double y = sh[t][k];
            if (k >= 5 && k <= 8) {
                const long long a = __double_as_longlong(x), b = __double_as_longlong(y);
                x = __longlong_as_double(k == 5 ? a + b : max(a, b));
            } else {
                x = x + y;
            }
        }
        out_block[k] = x;
    }
}

// The grid's partials folded without a one-block kernel.  A grid of up to
// kInlineBlocks blocks folds them itself: blocks are cut into groups of
// `group` consecutive ones, the block of a group that finishes last folds the
// group's rows, and the group that finishes last folds the groups' rows.  A
// larger grid leaves the rows to k_fold, which does the same over kFoldBlocks
// chunks of rows.  Which block folds depends on timing, what it adds and in
// which order does not.  The former reduction (a kernel of 256 blocks, then
// one block of 8 warps that added 12 columns on every lane: a warp's FP64
// addition holds an SM's FP64 pipe for about 19 cycles) took 10-15 us of
// every step; folding in the grid takes 1-2 us.  Every block that counts
// itself waits for its own stores first (about 1.2 us), which a grid of many
// waves pays once a wave: 23 us at 128^3 (16,384 blocks of 128), against
// about 6 us for k_fold; hence the line at about two waves.
struct GridSum {
    double* partials;     // [blocks][kNPart]
    double* rows;         // [groups][kNPart]
    unsigned* counters;   // [1 + groups], zero between launches
    int group;            // blocks per group; 0: k_fold folds the rows
};

constexpr int kInlineBlocks = 2048;
constexpr int kFoldRows = 256;       // rows one block folds before the grid is cut into groups
constexpr int kFoldBlocks = 128;     // blocks of k_fold
constexpr int kMaxGroups = 128;      // groups of a grid that folds itself (46), blocks of k_fold

// Rows of partials folded into out (shared memory, [kNPart]) by one block:
// eight lanes per row, one per FP64 sum (slots 0-4 and 9-11), so that every
// lane of an FP64 addition works; the count and the maxima (slots 5-8) on the
// integer ALU.
__device__ __forceinline__ void fold_rows(const double* rows, int count, double* out)
{
    __shared__ double shs[kMaxWarps][8];
    __shared__ long long shi[kMaxWarps][4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int c = lane & 7;
    const int cs = c < 5 ? c : c + 4;          // FP64 column of this lane
    const int ci = 5 + (c & 3);                // integer column (lanes of c >= 4 repeat it)
    double s = 0.0;
    long long b = 0;
#pragma unroll 4
    for (int r = 4 * w + (lane >> 3); r < count; r += 4 * nw) {
        const double x = __ldcg(rows + (size_t)r * kNPart + cs);
        const long long y = __double_as_longlong(__ldcg(rows + (size_t)r * kNPart + ci));
        s += x;
        b = ci == 5 ? b + y : max(b, y);
    }
#pragma unroll
    for (int off = 8; off < 32; off <<= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, off);
        const long long y = __shfl_xor_sync(0xffffffffu, b, off);
        b = ci == 5 ? b + y : max(b, y);
    }
    if (lane < 8) shs[w][lane] = s;
    if (lane < 4) shi[w][lane] = b;
    __syncthreads();
    if (threadIdx.x < 8) {
        double t = shs[0][threadIdx.x];
        for (int k = 1; k < nw; ++k) t += shs[k][threadIdx.x];
        out[threadIdx.x < 5 ? threadIdx.x : threadIdx.x + 4] = t;
    } else if (threadIdx.x < 12) {
        const int q = threadIdx.x - 8;
        long long t = shi[0][q];
        for (int k = 1; k < nw; ++k) t = q == 0 ? t + shi[k][q] : max(t, shi[k][q]);
        out[5 + q] = __longlong_as_double(t);
    }
    __syncthreads();
}

// Folded slots as the finishing code reads them: the count as a double, the
// roots of the squares.
__device__ __forceinline__ void totals_of(double* out)
{
    if (threadIdx.x == 5) out[5] = (double)__double_as_longlong(out[5]);
    if (threadIdx.x >= 6 && threadIdx.x <= 8) out[threadIdx.x] = sqrt(out[threadIdx.x]);
    __syncthreads();
}

// True in exactly one block of a grid that folds itself (B.group > 0), the
// one that finishes last, for all its threads and with the grid's totals in out (shared memory, [kNPart]:
// slot 5 as a double, slots 6-8 the magnitudes).  Every thread of every block
// calls it, after its last read of anything the finishing block writes.
__device__ __forceinline__ bool grid_partials(double* vals, const GridSum& B, double* out, bool sums = true,
                                              bool body = false)
{
    __shared__ int is_last;
    block_partials(vals, B.partials + (size_t)blockIdx.x * kNPart, sums, body);
    if (B.group == 0) return false;
    const int g = blockIdx.x / B.group, ngroups = (gridDim.x + B.group - 1) / B.group;
    const int size = min(B.group, (int)gridDim.x - g * B.group);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        is_last = atomicAdd(B.counters + 1 + g, 1u) == (unsigned)size - 1u;
        if (is_last) B.counters[1 + g] = 0u;
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    fold_rows(B.partials + (size_t)g * B.group * kNPart, size, out);
    if (ngroups > 1) {
        if (threadIdx.x < kNPart) B.rows[(size_t)g * kNPart + threadIdx.x] = out[threadIdx.x];
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            is_last = atomicAdd(B.counters, 1u) == (unsigned)ngroups - 1u;
            if (is_last) B.counters[0] = 0u;
        }
        __syncthreads();
        if (!is_last) return false;
        __threadfence();
        fold_rows(B.rows, ngroups, out);
    }
    totals_of(out);
    return true;
}

// k_fold's part: block b folds its chunk of the rows, the block that finishes
// last folds the chunks.  True in that block, with the totals in out.
__device__ __forceinline__ bool fold_grid(const GridSum& B, int nrows, double* out)
{
    __shared__ int is_last;
    const int chunk = (nrows + gridDim.x - 1) / gridDim.x;
    const int r0 = min(nrows, (int)blockIdx.x * chunk);
    fold_rows(B.partials + (size_t)r0 * kNPart, min(chunk, nrows - r0), out);
    if (threadIdx.x < kNPart) B.rows[(size_t)blockIdx.x * kNPart + threadIdx.x] = out[threadIdx.x];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        is_last = atomicAdd(B.counters, 1u) == gridDim.x - 1u;
        if (is_last) B.counters[0] = 0u;
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    fold_rows(B.rows, gridDim.x, out);
    totals_of(out);
    return true;
}

// Constants of the step sizes (Eq. 9-11 with h = h_min): dt_ad = ad / max(max|v|, v_floor),
// dt_ac = ac / (max|v| + c), with v_floor = max(nu / h_min, U_ref).
struct DtConsts {
    double v_floor, ad, ac, c, fixed_dt;
};

// Diagnostics and the next step size of a kick-drift-kick step (or of
// sph_build_cells, count_step = 0) from the grid's totals.
__device__ __forceinline__ void finish_step(const double* out, const DtConsts& D, double* diag,
                                            double* dt_ptr, int count_step)
{
    const double dt_used = *dt_ptr;
    __syncthreads();                      // thread 0 writes *dt_ptr below
    const int k = threadIdx.x;
    if (k == 0) {
        const double vmax = out[6];
        const double dt_ad = D.ad / fmax(vmax, D.v_floor);
        const double dt_ac = D.ac / (vmax + D.c);
        const double dt_next = D.fixed_dt > 0.0 ? D.fixed_dt : fmin(dt_ad, dt_ac);
        diag[DG_DT] = count_step ? dt_used : 0.0;
        diag[DG_DTNEXT] = dt_next;
        diag[DG_STEPS] = count_step ? diag[DG_STEPS] + 1.0 : 0.0;
        diag[DG_TIME] = count_step ? diag[DG_TIME] + dt_used : 0.0;    // simulated time since sph_build_cells
        *dt_ptr = dt_next;
    } else if (k < 10) {
        // slots 0-8 of the totals are in the order of the diagnostics but for n_chi
        const int q = k - 1;
        const int to = q < 5 ? DG_MASS + q : (q == 5 ? DG_NCHI : DG_VMAX + (q - 6));
        diag[to] = out[q];
    } else if (k < 13) {
        // force on the walls, and the body's impulse since sph_build_cells (the
        // time integral of the force over the steps, each step's force times its dt)
        const int d = k - 10;
        diag[DG_FBODY + d] = -out[9 + d];
        diag[DG_IMPULSE + d] = count_step ? diag[DG_IMPULSE + d] - out[9 + d] * dt_used : 0.0;
    }
}

}  // namespace sphtv
