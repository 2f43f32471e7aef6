// k_io.cu -- state transfer kernels of libsphtv: the load of a state in the
// caller's order ([n][3] rows into per-component arrays, wall velocities, the
// input checks), the way back from the cell order, the adjoint's cotangents,
// and the per-particle reference sums sigma0 of Eq. 8 (the perfect-lattice sum
// at the particle's own spacing dp = (m/rho0)^(1/D) and smoothing length h).
#include "common.cuh"
#include "launch.h"

namespace sphtv {

// Exact FP64 value of a stored component, off the FP64 pipe: the read-back is
// bound by its conversions otherwise, those of outputs not asked for among them
// (density alone of 128^3 in FP32 38.6 -> 14.8 us).  Below kWideFrom particles a
// thread's chain of operations counts for more than the pipe (2,916 particles:
// 0.5 us), and the hardware converts.
constexpr int kWideFrom = 20000;
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) { return f2d_exact(x); }

template <typename Real, int DIM>
__global__ void k_vec_in(int n, const double* src3, Real* dst)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int d = 0; d < DIM; ++d) dst[(size_t)d * n + i] = (Real)src3[3 * (size_t)i + d];
}

// pos[id[k]] = k: where the particle the caller gave as number i sits in
// the cell order.
__global__ void k_inverse_perm(int n, const int32_t* id, int32_t* pos)
{
    pdl_wait();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) pos[id[k]] = k;
}

// k_vec_out by gathering: dst3 row i (the caller's order) from the sorted
// position pos[i], so the writes of a warp are contiguous (the destination
// may be page-locked host memory written across the host link).
template <typename Real, int DIM>
__global__ void k_vec_out_gather(int n, const Real* src, const int32_t* pos,
                                 double* dst3)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const size_t k = (size_t)pos[i];
    // the loads before the first store: none could be moved past a store that
    // may alias it (all five arrays of 200^3 427 -> 387 us)
    double q[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) q[d] = d < DIM ? wide(src[(size_t)d * n + k]) : 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) dst3[3 * (size_t)i + d] = q[d];
}

template <typename V4>
__global__ void k_rho_out_gather(int n, const V4* vr, const int8_t* kind,
                                 const int32_t* pos, double rho0, double* dst)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = pos[i];
    dst[i] = kind[k] ? rho0 : rho0 + wide(vr[k].w);
}

// Smoothing lengths (in units of dp) from which the lattice sum is taken at its
// limit, the kernel's integral: sigma0 = dp^-D.  The two differ by 1.2e-15 of
// the value at 500 in 2-D and 4e-14 at 100 in 3-D, falling with the 5th and 6th
// power (the decay of the kernel's transform), below the rounding of the sum's
// million and eight million terms.  Without the line the sum over the lattice
// of a mass near or at 0 or of an infinite h has no end in practice, and the
// load would never come to the check that reports them.
template <int DIM> constexpr double kLatticeMax = DIM == 2 ? 500.0 : 100.0;

template <int DIM>
__device__ double sigma0_of(double h, double m, double rho0)
{
    const double vol = m / rho0;
    const double dp = DIM == 2 ? sqrt(vol) : cbrt(vol);
    const double ratio = h / dp;               // smoothing length in units of dp
    if (ratio >= kLatticeMax<DIM>) return 1.0 / (DIM == 2 ? dp * dp : dp * dp * dp);
    // (a negative ratio or NaN, whose particle the load rejects: no point, or one)
    const double reach2 = 4.0 * ratio * ratio;
    const int K = (int)ceil(2.0 * ratio);
    const double inv = 1.0 / ratio;
    // One octant of the integer lattice; each point stands for its 2^(number
    // of non-zero coordinates) mirror images.
    double s = 0.0;
    const int kz1 = DIM == 3 ? K : 0;
    for (int kz = 0; kz <= kz1; ++kz)
        for (int ky = 0; ky <= K; ++ky)
            for (int kx = 0; kx <= K; ++kx) {
                double r2 = (double)(kx * kx + ky * ky + kz * kz);
                if (r2 >= reach2) continue;
                double mult = (kx ? 2.0 : 1.0) * (ky ? 2.0 : 1.0) * (kz ? 2.0 : 1.0);
                s += mult * wendland_W<DIM, double>(sqrt(r2), inv);
            }
    return s / (DIM == 2 ? dp * dp : dp * dp * dp);
}

// sigma0_of by a whole warp for one (h, m): one lattice point per lane, the
// terms added in sigma0_of's order (the products by 2, 4 and 8 are exact, so
// the sum is sigma0_of's bit for bit).  FP64 work: a thread's own sum takes
// some 400 operations, a warp's shared one about 60.
template <int DIM>
__device__ __forceinline__ double sigma0_shared(double h, double m, double rho0)
{
    const double vol = m / rho0;
    const double dp = DIM == 2 ? sqrt(vol) : cbrt(vol);
    const double ratio = h / dp;
    if (!(ratio > 0.0 && ratio < kLatticeMax<DIM>)) return sigma0_of<DIM>(h, m, rho0);   // at most 8 million points below
    const double reach2 = 4.0 * ratio * ratio;
    const int side = (int)ceil(2.0 * ratio) + 1;
    const double inv = 1.0 / ratio;
    const int points = DIM == 3 ? side * side * side : side * side, lane = threadIdx.x & 31;
    double s = 0.0;
    for (int base = 0; base < points; base += 32) {
        const int p = base + lane;
        const int kx = p % side, ky = (p / side) % side, kz = p / (side * side);
        const double r2 = (double)(kx * kx + ky * ky + kz * kz);
        double term = 0.0;
        if (p < points && r2 < reach2) {
            const double mult = (kx ? 2.0 : 1.0) * (ky ? 2.0 : 1.0) * (kz ? 2.0 : 1.0);
            term = mult * wendland_W<DIM, double>(sqrt(r2), inv);
        }
        for (int t = 0; t < min(32, points - base); ++t) s += __shfl_sync(0xffffffffu, term, t);
    }
    return s / (DIM == 2 ? dp * dp : dp * dp * dp);
}

// The reference sum depends on (h, m) only: particle 0's value is computed
// once, by one warp, and stands for every particle with the same h and m; the
// others share theirs among the lanes of a warp that want the same one, or,
// where a warp wants more than four, compute their own.
template <int DIM>
__device__ __forceinline__ double sigma0_in_warp(double h, double m, double rho0, bool want)
{
    const int lane = threadIdx.x & 31;
    const unsigned same = __match_any_sync(0xffffffffu, __double_as_longlong(h)) &
                          __match_any_sync(0xffffffffu, __double_as_longlong(m)) &
                          __ballot_sync(0xffffffffu, want);
    unsigned leaders = __ballot_sync(0xffffffffu, want && lane == __ffs(same) - 1);
    double s0 = 0.0;
    if (__popc(leaders) > 4) {
        if (want) s0 = sigma0_of<DIM>(h, m, rho0);
        return s0;
    }
    while (leaders) {
        const int l = __ffs(leaders) - 1;
        leaders &= leaders - 1;
        const double v = sigma0_shared<DIM>(__shfl_sync(0xffffffffu, h, l), __shfl_sync(0xffffffffu, m, l), rho0);
        if (want && (same >> l & 1u)) s0 = v;
    }
    return s0;
}

template <int DIM>
__global__ void k_sigma0_first(const double* h, const double* m, double rho0, double* s0_first, uint32_t* varies)
{
    pdl_wait();
    const double v = sigma0_shared<DIM>(h[0], m[0], rho0);
    if (threadIdx.x == 0) {
        *s0_first = v;
        *varies = 0u;
    }
}

// One particle's load, everything sph_set_state (or the adjoint's reload)
// brings, in the caller's order: positions and velocities (walls: the
// prescribed velocity) into the components, accelerations and displacements
// or zeros, h, m, sigma0 and kind into both state sets (the sort leaves them
// where they are when they do not vary), ids, the adjoint's copies; checks h
// and m (h in [h_min, h_max], which sizes the cell edge; m positive and
// finite) and sets *varies (cleared before) when a particle's h, m or sigma0
// differs from particle 0's or a particle is a wall particle.  One kernel for
// eight and the copies between them: loading 3,000 particles is launches, not
// bytes.
template <typename Real, int DIM>
__global__ void __launch_bounds__(256) k_load_state(int n, LoadArgs A, StateSet<Real> S0, StateSet<Real> S1,
                                                    double rho0, double h_min, double h_max, uint32_t* err)
{
    pdl_wait();
    const int at = blockIdx.x * blockDim.x + threadIdx.x, i = min(at, n - 1);
    const double h = A.h[i], m = A.m[i], h0 = A.h[0], m0 = A.m[0];
    const int8_t kind = A.kind ? A.kind[i] : 0;
    double s0, s00;
    if (A.sigma0) {
        s0 = A.sigma0[i];
        s00 = A.sigma0[0];
    } else {
        s00 = s0 = *A.s0_first;
        const bool other = h != h0 || m != m0;
        if (__any_sync(0xffffffffu, other)) {
            const double own = sigma0_in_warp<DIM>(h, m, rho0, other);
            if (other) s0 = own;
        }
    }
    const bool varies = kind != 0 || h != h0 || m != m0 || s0 != s00;
    const unsigned b = __ballot_sync(0xffffffffu, varies);
    if (b && (threadIdx.x & 31) == 0) atomicOr(err + 1, 1u);
    if (at >= n) return;
    if (!(h >= h_min && h <= h_max && m > 0.0 && isfinite(m))) atomicOr(err, ERRB_INPUT);
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const size_t o = (size_t)d * n + i;
        if (A.x) S0.x[o] = A.x[3 * (size_t)i + d];
        if (kind) S0.v[o] = A.vw ? (Real)A.vw[3 * (size_t)i + d] : Real(0);
        else if (A.v) S0.v[o] = (Real)A.v[3 * (size_t)i + d];
        else if (A.zero_v) S0.v[o] = Real(0);
        if (A.a) {
            S0.a[o] = (Real)A.a[3 * (size_t)i + d];
            S0.dr[o] = (Real)A.dr[3 * (size_t)i + d];
        } else if (A.zero_ad) {
            S0.a[o] = Real(0);
            S0.dr[o] = Real(0);
        }
    }
    S0.h[i] = S1.h[i] = h;
    S0.m[i] = S1.m[i] = m;
    S0.s0[i] = S1.s0[i] = s0;
    S0.kind[i] = S1.kind[i] = kind;
    S0.id[i] = i;
    if (S0.drho) S0.drho[i] = Real(0);
    if (A.orig_h) {
        A.orig_h[i] = h;
        A.orig_m[i] = m;
        A.orig_s0[i] = s0;
        A.orig_kind[i] = kind;
#pragma unroll
        for (int d = 0; d < 3; ++d) A.orig_vw[3 * (size_t)i + d] = A.vw ? A.vw[3 * (size_t)i + d] : 0.0;
    }
}

// The whole state out into device memory, in the caller's order (each of the
// outputs may be null): one kernel for an inverse permutation and five
// gathers.  The reads are in the sorted order, each particle's rows of 24
// bytes go where its id says; for how much output, see kScatterBytes.  (With a
// row's loads before the stores of the one before, the scattered stores came in
// longer bursts: 64^3 shuffled 35 -> 56 us.)
template <typename Real, int DIM, bool WIDE>
__global__ void __launch_bounds__(256) k_store_state(int n, StateSet<Real> S, const typename Vec4<Real>::T* vr,
                                                     double rho0, double* x, double* v, double* a, double* dr,
                                                     double* rho)
{
    pdl_wait();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const size_t i = (size_t)S.id[k];
    auto fp64 = [](auto q) { return WIDE ? wide(q) : (double)q; };
    auto row = [&](double* dst, const auto* src) {
        if (!dst) return;
#pragma unroll
        for (int d = 0; d < 3; ++d) dst[3 * i + d] = d < DIM ? fp64(src[(size_t)d * n + k]) : 0.0;
    };
    row(x, S.x);
    row(v, S.v);
    row(a, S.a);
    row(dr, S.dr);
    if (rho) rho[i] = S.kind[k] ? rho0 : rho0 + fp64(vr[k].w);
}

// The adjoint's four cotangents between the caller's rows and [3][n]
// (components past DIM are zero on the way in).
__global__ void __launch_bounds__(256) k_cotangents_in(int n, int dim, Four<const double> src, Four<double> dst)
{
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (!src.p[q]) continue;
        for (int d = 0; d < 3; ++d) dst.p[q][(size_t)d * n + i] = d < dim ? src.p[q][3 * (size_t)i + d] : 0.0;
    }
}

__global__ void __launch_bounds__(256) k_cotangents_out(int n, Four<const double> src, Four<double> dst)
{
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (!dst.p[q]) continue;
        for (int d = 0; d < 3; ++d) dst.p[q][3 * (size_t)i + d] = src.p[q][(size_t)d * n + i];
    }
}

template <typename V4>
__global__ void k_rho_out(int n, const V4* vr, const int8_t* kind,
                          const int32_t* id, double rho0, double* dst)
{
    pdl_wait();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    dst[id[k]] = kind[k] ? rho0 : rho0 + (double)vr[k].w;
}

template <typename Real>
__global__ void k_scalar_out(int n, const Real* src, const int32_t* id,
                             double* dst)
{
    pdl_wait();
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) dst[id[k]] = (double)src[k];
}

// Caller-order scalar in (walls get 0); used before the first sort, when the
// internal order is the caller's.
template <typename Real>
__global__ void k_scalar_in(int n, const double* src, const int8_t* kind,
                            Real* dst)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = kind[i] ? Real(0) : (Real)src[i];
}

static inline int nblk(int n, int t) { return (n + t - 1) / t; }

cudaError_t launch_vec_in(int prec, int dim, int n, const double* src3, void* dst, cudaStream_t st)
{
    const int T = 256;
    if (prec == 64) {
        if (dim == 2) launch(k_vec_in<double, 2>, nblk(n, T), T, 0, st, n, src3, (double*)dst);
        else launch(k_vec_in<double, 3>, nblk(n, T), T, 0, st, n, src3, (double*)dst);
    } else {
        if (dim == 2) launch(k_vec_in<float, 2>, nblk(n, T), T, 0, st, n, src3, (float*)dst);
        else launch(k_vec_in<float, 3>, nblk(n, T), T, 0, st, n, src3, (float*)dst);
    }
    return cudaGetLastError();
}

cudaError_t launch_load_state(int prec, int dim, int n, const LoadArgs& A, void* S0, void* S1, double rho0,
                              double h_min, double h_max, uint32_t* err, cudaStream_t st, int64_t* launches)
{
    if (A.sigma0) {
        const cudaError_t e = cudaMemsetAsync(err + 1, 0, sizeof(uint32_t), st);
        if (e != cudaSuccess) return e;
    } else {
        launch(dim == 2 ? k_sigma0_first<2> : k_sigma0_first<3>, 1, 32, 0, st, A.h, A.m, rho0, A.s0_first, err + 1);
        ++*launches;
    }
    const int T = 256, nb = nblk(n, T);
    if (prec == 64) {
        const auto a = *(const StateSet<double>*)S0, b = *(const StateSet<double>*)S1;
        launch(dim == 2 ? k_load_state<double, 2> : k_load_state<double, 3>, nb, T, 0, st, n, A, a, b, rho0, h_min,
               h_max, err);
    } else {
        const auto a = *(const StateSet<float>*)S0, b = *(const StateSet<float>*)S1;
        launch(dim == 2 ? k_load_state<float, 2> : k_load_state<float, 3>, nb, T, 0, st, n, A, a, b, rho0, h_min,
               h_max, err);
    }
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_store_state(int prec, int dim, int n, const void* S, const void* vr, double rho0, double* x,
                               double* v, double* a, double* dr, double* rho, cudaStream_t st)
{
    const int T = 256, nb = nblk(n, T);
    if (prec == 64) {
        launch(dim == 2 ? k_store_state<double, 2, false> : k_store_state<double, 3, false>, nb, T, 0, st, n,
               *(const StateSet<double>*)S, (const double4_32a*)vr, rho0, x, v, a, dr, rho);
        return cudaGetLastError();
    }
    auto kern = n < kWideFrom ? (dim == 2 ? k_store_state<float, 2, false> : k_store_state<float, 3, false>)
                              : (dim == 2 ? k_store_state<float, 2, true> : k_store_state<float, 3, true>);
    launch(kern, nb, T, 0, st, n, *(const StateSet<float>*)S, (const float4*)vr, rho0, x, v, a, dr, rho);
    return cudaGetLastError();
}

cudaError_t launch_cotangents_in(int n, int dim, const Four<const double>& src, const Four<double>& dst,
                                 cudaStream_t st)
{
    launch(k_cotangents_in, nblk(n, 256), 256, 0, st, n, dim, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_cotangents_out(int n, const Four<const double>& src, const Four<double>& dst, cudaStream_t st)
{
    launch(k_cotangents_out, nblk(n, 256), 256, 0, st, n, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_rho_out(int prec, int n, const void* vr, const int8_t* kind, const int32_t* id, double rho0,
                           double* dst, cudaStream_t st)
{
    if (prec == 64) launch(k_rho_out<double4_32a>, nblk(n, 256), 256, 0, st, n, (const double4_32a*)vr, kind, id, rho0, dst);
    else launch(k_rho_out<float4>, nblk(n, 256), 256, 0, st, n, (const float4*)vr, kind, id, rho0, dst);
    return cudaGetLastError();
}

cudaError_t launch_inverse_perm(int n, const int32_t* id, int32_t* pos, cudaStream_t st)
{
    launch(k_inverse_perm, nblk(n, 256), 256, 0, st, n, id, pos);
    return cudaGetLastError();
}

cudaError_t launch_vec_out_gather(int prec, int dim, int n, const void* src, const int32_t* pos, double* dst3,
                                  cudaStream_t st)
{
    const int T = 256;
    if (prec == 64) {
        if (dim == 2) launch(k_vec_out_gather<double, 2>, nblk(n, T), T, 0, st, n, (const double*)src, pos, dst3);
        else launch(k_vec_out_gather<double, 3>, nblk(n, T), T, 0, st, n, (const double*)src, pos, dst3);
    } else {
        if (dim == 2) launch(k_vec_out_gather<float, 2>, nblk(n, T), T, 0, st, n, (const float*)src, pos, dst3);
        else launch(k_vec_out_gather<float, 3>, nblk(n, T), T, 0, st, n, (const float*)src, pos, dst3);
    }
    return cudaGetLastError();
}

cudaError_t launch_rho_out_gather(int prec, int n, const void* vr, const int8_t* kind, const int32_t* pos,
                                  double rho0, double* dst, cudaStream_t st)
{
    if (prec == 64)
        launch(k_rho_out_gather<double4_32a>, nblk(n, 256), 256, 0, st, n, (const double4_32a*)vr, kind, pos, rho0, dst);
    else launch(k_rho_out_gather<float4>, nblk(n, 256), 256, 0, st, n, (const float4*)vr, kind, pos, rho0, dst);
    return cudaGetLastError();
}

cudaError_t launch_scalar_in(int prec, int n, const double* src, const int8_t* kind, void* dst, cudaStream_t st)
{
    if (prec == 64) launch(k_scalar_in<double>, nblk(n, 256), 256, 0, st, n, src, kind, (double*)dst);
    else launch(k_scalar_in<float>, nblk(n, 256), 256, 0, st, n, src, kind, (float*)dst);
    return cudaGetLastError();
}

cudaError_t launch_scalar_out(int prec, int n, const void* src, const int32_t* id, double* dst, cudaStream_t st)
{
    if (prec == 64) launch(k_scalar_out<double>, nblk(n, 256), 256, 0, st, n, (const double*)src, id, dst);
    else launch(k_scalar_out<float>, nblk(n, 256), 256, 0, st, n, (const float*)src, id, dst);
    return cudaGetLastError();
}

}  // namespace sphtv
