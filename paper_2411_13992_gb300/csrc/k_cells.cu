// k_cells.cu -- the kick-drift stage and the cell-linked list of libsphtv.
//
// Per step, three kernels:  kick + drift + bin key, with each bin's particles
// counted and linked into a list  ->  exclusive scan of the bin counts  ->
// each particle ranks itself by id among its bin's list (so the sorted order
// never depends on atomic timing) and moves its arrays to the new order (and,
// in both forms, emits its FP32 position relative to its cell's origin).
//
// The kick-drift follows the kick-drift-kick scheme the paper names (Sec. 1,
// Sec. 3): v += dt/2 a; x += dt v + dr, where dr is the transport-velocity
// displacement of the previous step (Eq. 16), applied once per step.  With the
// dual-criteria integrator (Sec. 2.4) the substeps have moved the particles
// already and this stage only wraps the periodic axes.
#include "common.cuh"
#include "launch.h"

namespace sphtv {

// A non-negative int as a double, exactly, on the integer ALU: the leading
// one sets the binary64 exponent, the bits below it the fraction.
__device__ __forceinline__ double i2d_exact(int c)
{
    if (c <= 0) return 0.0;                   // callers pass cell coordinates >= 0
    const int e = 31 - __clz(c);
    const unsigned long long frac = ((unsigned long long)c << (52 - e)) & 0xfffffffffffffULL;
    return __longlong_as_double((long long)(((unsigned long long)(e + 1023) << 52) | frac));
}

template <typename Real>
__device__ __forceinline__ Real kick(Real v, double hdt, Real a);

template <>
__device__ __forceinline__ double kick<double>(double v, double hdt, double a)
{
    return __dadd_rn(v, __dmul_rn(hdt, a));
}

template <>
__device__ __forceinline__ float kick<float>(float v, double hdt, float a)
{
    return __fadd_rn(v, __fmul_rn(d2f_rn(hdt), a));
}

// FP64 value of a velocity or displacement component (exact either way).
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(float x) { return f2d_exact(x); }

// -1 for x < lo, +1 for x >= hi, else 0: the periodic wrap of axis d, as
// integer comparisons of order keys (dkey).
__device__ __forceinline__ int wrap_side(const Grid& G, double x, int d)
{
    const long long kx = dkey(x);
    return kx < dkey(G.lo[d]) ? -1 : (kx >= dkey(G.hi[d]) ? 1 : 0);
}

template <typename Real, int DIM>
__global__ void k_kick_drift_key(int n, StateSet<Real> S, const double* dt_ptr, int drift, Grid G,
                                 int32_t* key, int32_t* count,
                                 int32_t* head, int32_t* next, uint32_t* err)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double xs[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int d = 0; d < DIM; ++d) xs[d] = S.x[(size_t)d * n + i];
    uint32_t e = 0;
    if (drift == 2 && S.kind[i] == 0) {
        // dual-criteria integrator: the substeps moved the particles; only
        // the periodic wrap is left to do here
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            if (!G.periodic[d]) continue;
            const int w = wrap_side(G, xs[d], d);
            if (__any_sync(__activemask(), w != 0) && w != 0) {
                xs[d] = w < 0 ? __dadd_rn(xs[d], G.L[d]) : __dsub_rn(xs[d], G.L[d]);
                S.x[(size_t)d * n + i] = xs[d];
            }
        }
    } else if (drift == 1) {
        // every load issued before the kind test and the arithmetic
        Real vv[3] = {0, 0, 0}, aa[3] = {0, 0, 0}, rr[3] = {0, 0, 0};
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const size_t o = (size_t)d * n + i;
            vv[d] = S.v[o];
            aa[d] = S.a[o];
            rr[d] = S.dr[o];
        }
        const double dt = *dt_ptr;
        if (S.kind[i] == 0) {
            const double hdt = 0.5 * dt;
            // FP32 form: the displacement dt v + dr in FP32 (one rounding, from
            // FP32 inputs), accumulated into the FP64 position
            const float dt_f = d2f_rn(dt);
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                size_t o = (size_t)d * n + i;
                Real vh = kick<Real>(vv[d], hdt, aa[d]);
                S.v[o] = vh;
                double xn;
                if (sizeof(Real) == 4)
                    xn = __dadd_rn(xs[d], to_double(__fmaf_rn(dt_f, (float)vh, (float)rr[d])));
                else
                    xn = __dadd_rn(__dadd_rn(xs[d], __dmul_rn(dt, to_double(vh))), to_double(rr[d]));
                if (G.periodic[d]) {
                    // the wrap only in warps where a particle left the box (the
                    // FP64 operation would otherwise be issued for every warp)
                    const int w = wrap_side(G, xn, d);
                    if (__any_sync(__activemask(), w != 0) && w != 0)
                        xn = w < 0 ? __dadd_rn(xn, G.L[d]) : __dsub_rn(xn, G.L[d]);
                }
                xs[d] = xn;
                S.x[o] = xn;
            }
        }
    }
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        if (!finite_bits(xs[d])) e |= ERRB_NAN;
        else if (!G.periodic[d] && (dkey(xs[d]) < dkey(G.lo[d]) || dkey(xs[d]) > dkey(G.hi[d]))) e |= ERRB_DOMAIN;
    }
    if (e) atomicOr(err, e);
    int k = sort_key<DIM>(G, xs);
    key[i] = k;
    // count the bin, and put the particle at the front of the bin's list (two
    // atomics per particle: with the sub-cell bins a warp's lanes seldom share
    // one, and aggregating them by __match_any_sync cost more than it saved).
    // A list is followed for as many members as its bin counts, so its end and
    // an empty bin's head need no mark and no clearing.
    atomicAdd(&count[k], 1);
    next[i] = atomicExch(&head[k], i);
}

// ------------------------------------------------------- exclusive scan

constexpr int kScanThreads = 512;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

size_t scan_temp_elems(int n) { return (size_t)(n + kScanTile - 1) / kScanTile; }

// In-place exclusive scan over the block of one value per thread: returns the
// sum of the threads before, *total the block's sum.
__device__ __forceinline__ int32_t block_scan(int32_t s, int32_t* warp_tot, int32_t* total)
{
    constexpr int nw = kScanThreads / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t incl = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int32_t t = lane < nw ? warp_tot[lane] : 0;
        int32_t ti = t;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, ti, off);
            if (lane >= off) ti += u;
        }
        if (lane < nw) warp_tot[lane] = ti - t;
        if (lane == nw - 1) warp_tot[nw] = ti;
    }
    __syncthreads();
    *total = warp_tot[nw];
    return warp_tot[w] + incl - s;
}

// The sort's scan: prefix[k] = the sum of count[0, k) within k's tile of
// kScanTile bins, tile_off[b] the sum of the tiles before tile b, so that the
// start of bin k is prefix[k] + tile_off[k / kScanTile] (the readers add the
// two: no pass over the bins for it).  Clears the counts as it reads them.
// The block that finishes last scans the tiles' sums (one kernel where there
// were two or three); a single tile needs no such scan (step of 2,304
// particles 27.9 -> 25.8 us, of 4,096 in 3-D 50.1 -> 48.1).  Where each reading warp scanned up to 32 sums itself
// instead, the step of a small problem took as long and the permute 3 us more
// at 128^3.
__global__ void __launch_bounds__(kScanThreads) k_bin_scan(int32_t* count, int32_t* prefix,
                                                           int32_t* tile_off, unsigned* done, int n)
{
    pdl_wait();
    __shared__ int32_t warp_tot[kScanThreads / 32 + 1];
    __shared__ int is_last;
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    static_assert(kScanItems % 4 == 0, "16-byte vectors");
    __align__(16) int32_t vals[kScanItems];          // moved as int4, wherever the compiler keeps it
    const bool whole = base + kScanItems <= n;      // base is a multiple of 16: 64-byte aligned
    if (whole) {
        int4* c4 = reinterpret_cast<int4*>(count + base);
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) *reinterpret_cast<int4*>(vals + 4 * k) = c4[k];
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) c4[k] = make_int4(0, 0, 0, 0);
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            vals[k] = base + k < n ? count[base + k] : 0;
            if (base + k < n) count[base + k] = 0;
        }
    }
    int32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const int32_t v = vals[k];
        vals[k] = s;
        s += v;
    }
    int32_t total;
    const int32_t pre = block_scan(s, warp_tot, &total);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) vals[k] += pre;
    if (whole) {
        int4* p4 = reinterpret_cast<int4*>(prefix + base);
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) p4[k] = *reinterpret_cast<int4*>(vals + 4 * k);
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k)
            if (base + k < n) prefix[base + k] = vals[k];
    }
    const int nt = gridDim.x;
    if (nt == 1) {
        if (threadIdx.x == 0) tile_off[0] = 0;
        return;
    }
    if (threadIdx.x == 0) {
        tile_off[blockIdx.x] = total;
        __threadfence();
        is_last = atomicAdd(done, 1u) == (unsigned)nt - 1u;
        if (is_last) *done = 0u;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    int32_t carry = 0;
    for (int t0 = 0; t0 < nt; t0 += kScanThreads) {
        const int t = t0 + threadIdx.x;
        const int32_t v = t < nt ? __ldcg(tile_off + t) : 0;
        const int32_t p = carry + block_scan(v, warp_tot, &total);
        if (t < nt) tile_off[t] = p;
        carry += total;
        __syncthreads();                        // warp_tot is used again
    }
}

cudaError_t launch_bin_scan(int32_t* count, int32_t* prefix, int n, int32_t* tile_off, unsigned* done,
                            cudaStream_t st)
{
    launch(k_bin_scan, (n + kScanTile - 1) / kScanTile, kScanThreads, 0, st, count, prefix, tile_off, done, n);
    return cudaGetLastError();
}

// ------------------------------------------------------ order and permute

// One thread per particle, in the old order: its slot in the new order is its
// bin's start plus the number of its bin's particles with a smaller id (ids
// are unique), found by following the bin's list; bins hold less than one
// particle on average.  The particle's arrays are read in the old order, in
// which neighbouring threads read neighbouring words, and written to the
// slots, which are nearly in the same order after one step's motion.  One
// kernel where there were three (scatter by atomics, order of each bin,
// permute by gathering), without their passes over two permutations.
//
// The threads also write the bins' starts (thread nbin the end, n); with
// sub-cells (G.sub_shift > 0) the thread of a cell's first sub-cell also
// writes the cell's start.
//
// pos4 = {offset from the cell origin, h} (uniform resolution:
// {offset, m}, since h is then a constant), mf = m in FP32, cell_out = key;
// pos4c (when given: the FP32 form at uniform resolution) = {offset, bits of
// the cell index}, which the FP32 density walk reads instead of pos4 and
// cell_out.  When *varies is 0 every particle has particle 0's h, m and
// sigma0 and is a fluid particle, and both state sets hold these arrays
// (set by sph_set_state): they are left where they are.
//
// The order a state is loaded in may have nothing to do with space (a shuffled
// load, a checkpoint of a mixed flow): the first sort of a state that does not
// fit the L2 would spend its time on parts of sectors written all over memory.
// It runs as two kernels (HOW): one ranks the particles and notes where each
// slot's comes from, the other moves them in the new order by gathering.
// sph_build_cells of 128^3 particles in the order of space / disordered by 0.2 dp
// / shuffled by one kernel 1451 / 1708 / 2014 us, by two 1458 / 1691 / 1573; of
// 200^3 in the order of space / shuffled 5373 / 8962 and 5380 / 6785.
enum : int { kRankAndMove, kRank, kMove };

template <typename Real, int DIM, bool CARRY_AD, int HOW>
__global__ void __launch_bounds__(256) k_order_permute(int n, int nbin, const int32_t* key,
                                const int32_t* prefix, const int32_t* tile_off,
                                const int32_t* head, const int32_t* next,
                                int32_t* bin_start, int32_t* cell_start,
                                StateSet<Real> src, StateSet<Real> dst, Grid G, float4* pos4,
                                int32_t* cell_out, float* mf, int uniform_h,
                                float4* pos4c, const uint32_t* varies, int32_t* old_of)
{
    pdl_wait();
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
    auto start_of = [&](int k) { return prefix[k] + tile_off[k / kScanTile]; };
    if (HOW != kMove && t0 <= nbin) {
        const int s = start_of(t0);
        bin_start[t0] = s;
        if (G.sub_shift && (t0 & ((1 << G.sub_shift) - 1)) == 0) cell_start[t0 >> G.sub_shift] = s;
    }
    if (t0 >= n) return;
    const int i = HOW == kMove ? old_of[t0] : t0;
    const int bin = key[i];
    const int id = src.id[i];
    const bool moves = HOW != kRank && *varies != 0;
    double xs[3] = {0.0, 0.0, 0.0};
    Real vs[3] = {0, 0, 0};
    if (HOW != kRank) {
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            xs[d] = src.x[(size_t)d * n + i];
            vs[d] = src.v[(size_t)d * n + i];
        }
    }
    int k = t0;
    if (HOW != kMove) {
        k = start_of(bin);
        const int members = start_of(bin + 1) - k;
        if (members > 1) {
            int t = head[bin];
            for (int q = 1; ; ++q) {
                k += src.id[t] < id;
                if (q == members) break;
                t = next[t];
            }
        }
    }
    if (HOW == kRank) {
        old_of[k] = i;
        return;
    }
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const size_t so = (size_t)d * n + i, dof = (size_t)d * n + k;
        dst.x[dof] = xs[d];
        dst.v[dof] = vs[d];
        if (CARRY_AD) {
            dst.a[dof] = src.a[so];
            dst.dr[dof] = src.dr[so];
        }
    }
    if (src.drho) dst.drho[k] = src.drho[i];
    const double h = moves ? src.h[i] : src.h[0];
    const double m = moves ? src.m[i] : src.m[0];
    if (moves) {
        dst.h[k] = h;
        dst.m[k] = m;
        dst.s0[k] = src.s0[i];
        dst.kind[k] = src.kind[i];
    }
    dst.id[k] = id;
    const int cell = bin >> G.sub_shift;   // the cell of the sort key
    int c[3];
    cell_decode(G, cell, c);
    float o[3] = {0.f, 0.f, 0.f};
    // the conversions on the integer ALU (the same values as the hardware
    // conversions, which run on the FP64 pipe)
#pragma unroll
    for (int d = 0; d < DIM; ++d) o[d] = d2f_rn(xs[d] - (G.lo[d] + i2d_exact(c[d]) * G.edge[d]));
    const float m_f = d2f_rn(m);
    pos4[k] = make_float4(o[0], o[1], o[2], uniform_h ? m_f : d2f_rn(h));
    if (pos4c) pos4c[k] = make_float4(o[0], o[1], o[2], __int_as_float(cell));
    cell_out[k] = cell;
    mf[k] = m_f;
}

// The cell-relative FP32 records of sorted particles by themselves, as
// k_order_permute writes them (the FP64 form's adjoint, whose tape does not
// hold them).
template <int DIM>
__global__ void __launch_bounds__(256) k_offsets(int n, const double* x, const double* h, const double* m,
                                                 const int32_t* cell, Grid G, int uniform_h, float4* pos4)
{
    pdl_wait();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int c[3];
    cell_decode(G, cell[k], c);
    float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < DIM; ++d) o[d] = d2f_rn(x[(size_t)d * n + k] - (G.lo[d] + i2d_exact(c[d]) * G.edge[d]));
    pos4[k] = make_float4(o[0], o[1], o[2], d2f_rn(uniform_h ? m[k] : h[k]));
}

// ------------------------------------------------------------- launchers

static inline int nblk(int n, int t) { return (n + t - 1) / t; }

cudaError_t launch_kick_drift_key(int prec, int dim, int n, void* S, const double* dt, int drift, const Grid& G,
                                  int32_t* key, int32_t* count, int32_t* head, int32_t* next, uint32_t* err,
                                  cudaStream_t st)
{
    const int T = 256;
    if (prec == 64) {
        auto s = *(StateSet<double>*)S;
        if (dim == 2) launch(k_kick_drift_key<double, 2>, nblk(n, T), T, 0, st, n, s, dt, drift, G, key, count, head, next, err);
        else launch(k_kick_drift_key<double, 3>, nblk(n, T), T, 0, st, n, s, dt, drift, G, key, count, head, next, err);
    } else {
        auto s = *(StateSet<float>*)S;
        if (dim == 2) launch(k_kick_drift_key<float, 2>, nblk(n, T), T, 0, st, n, s, dt, drift, G, key, count, head, next, err);
        else launch(k_kick_drift_key<float, 3>, nblk(n, T), T, 0, st, n, s, dt, drift, G, key, count, head, next, err);
    }
    return cudaGetLastError();
}

template <typename Real>
static void order_permute_t(int dim, int n, int nbin, const SortBufs& B, void* src, void* dst, const Grid& G,
                            float4* pos4, int32_t* cell, float* mf, int uh, int carry_ad, cudaStream_t st,
                            float4* pos4c, const uint32_t* varies, int32_t* old_of)
{
    auto s = *(StateSet<Real>*)src;
    auto d = *(StateSet<Real>*)dst;
    int32_t* cs = G.sub_shift ? B.cell_start : nullptr;
    int32_t* bs = G.sub_shift ? B.sub_start : B.cell_start;
    const int T = 256, all = n > nbin ? n : nbin + 1;
    auto go = [&](auto* kern, int threads) {
        launch(kern, nblk(threads, T), T, 0, st, n, nbin, B.key, B.prefix, B.tile_off, B.head, B.next, bs, cs, s, d, G,
               pos4, cell, mf, uh, pos4c, varies, old_of);
    };
    if (old_of) {
        go(dim == 2 ? k_order_permute<Real, 2, false, kRank> : k_order_permute<Real, 3, false, kRank>, all);
        if (dim == 2) go(carry_ad ? k_order_permute<Real, 2, true, kMove> : k_order_permute<Real, 2, false, kMove>, n);
        else go(carry_ad ? k_order_permute<Real, 3, true, kMove> : k_order_permute<Real, 3, false, kMove>, n);
        return;
    }
    constexpr int both = kRankAndMove;
    if (dim == 2) go(carry_ad ? k_order_permute<Real, 2, true, both> : k_order_permute<Real, 2, false, both>, all);
    else go(carry_ad ? k_order_permute<Real, 3, true, both> : k_order_permute<Real, 3, false, both>, all);
}

cudaError_t launch_order_permute(int prec, int dim, int n, int nbin, const SortBufs& B, void* src, void* dst,
                                 const Grid& G, float4* pos4, int32_t* cell, float* mf, int uniform_h, int carry_ad,
                                 cudaStream_t st, const uint32_t* varies, float4* pos4c, int32_t* old_of)
{
    if (prec == 64)
        order_permute_t<double>(dim, n, nbin, B, src, dst, G, pos4, cell, mf, uniform_h, carry_ad, st, pos4c, varies, old_of);
    else
        order_permute_t<float>(dim, n, nbin, B, src, dst, G, pos4, cell, mf, uniform_h, carry_ad, st, pos4c, varies, old_of);
    return cudaGetLastError();
}

cudaError_t launch_offsets(int dim, int n, const double* x, const double* h, const double* m, const int32_t* cell,
                           const Grid& G, int uniform_h, float4* pos4, cudaStream_t st)
{
    launch(dim == 2 ? k_offsets<2> : k_offsets<3>, nblk(n, 256), 256, 0, st, n, x, h, m, cell, G, uniform_h, pos4);
    return cudaGetLastError();
}

}  // namespace sphtv
