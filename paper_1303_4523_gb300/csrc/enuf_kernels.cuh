// enuf_kernels.cuh -- sm_103a kernels of the ENUF-DPD hot path, templated on
// the working precision R (float or double). Energies, virials and charge
// sums are always reduced in double.
//
// Stages (Table 2 step 4, Eq. 14-25 of the paper):
//   bin      : charged beads -> tile bins of the oversampled grid
//   spread   : transposed NFFT part 1, by global reductions (or in shared-memory tiles)
//   fft_x/y  : forward R2C/C2C passes, pruned to |k_t| <= n_c
//   fft_z    : forward z, influence x deconvolution multiply, FP64 energy and
//              virial, -i D F and kz times it, inverse z (conjugated NFFT part 1)
//   fft_iy/ix: inverse passes to three real fields
//   gather   : conjugated NFFT part 2, warp per bead, F_i += kappa 2 q_i/L^2 * sum psi h
//   real     : erfc Ewald + Slater correction pairs (Eq. 31, 27-28) on the tile bins
//   dpd      : conservative, dissipative and random pair forces (Eq. 2-7) + bonds
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "enuf_fft.cuh"
#include "enuf_internal.h"

namespace enuf {

template <typename R> struct V4;
template <> struct V4<float> { using T = float4; };
template <> struct V4<double> { using T = double4_32a; };

__device__ __forceinline__ float int_as_real(int v, float) { return __int_as_float(v); }
__device__ __forceinline__ double int_as_real(int v, double) { return __longlong_as_double((long long)v); }
__device__ __forceinline__ int real_as_int(float v) { return __float_as_int(v); }
__device__ __forceinline__ int real_as_int(double v) { return (int)__double_as_longlong(v); }

__device__ __forceinline__ const WinK<float>& win_k(const Geo& g, float) { return g.wkf; }
__device__ __forceinline__ const WinK<double>& win_k(const Geo& g, double) { return g.wkd; }
__device__ __forceinline__ const DpdK<float>& dpd_k(const DpdDev& d, float) { return d.kf; }
__device__ __forceinline__ const DpdK<double>& dpd_k(const DpdDev& d, double) { return d.kd; }
__device__ __forceinline__ float dpd_cinv(const DpdDev& d, float) { return d.cinvf; }
__device__ __forceinline__ double dpd_cinv(const DpdDev& d, double) { return d.cinv; }

// Programmatic dependent launch (sm_90 and later): every kernel first waits
// until the grid before it in the stream has completed and its writes are
// visible (griddepcontrol.wait, a no-op when it was launched without the
// programmatic attribute). Nothing touches global memory before the wait. No
// kernel triggers its dependents early: CTAs of the next grid parked in the
// wait would hold shared memory that the other stream's kernels need, so the
// next grid launches at completion, with its launch work already done.
__device__ __forceinline__ void pdl_enter() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Asynchronous 16-byte global -> shared copies (both addresses 16-byte aligned),
// grouped by commit; wait_prior waits for all groups but the most recent one.
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gsrc) : "memory");
}
// nbytes (a multiple of 8) from global to shared memory by the whole block:
// 16-byte granules when both ends and the size allow, else 8-byte ones; the
// caller commits the group
__device__ __forceinline__ void cp_async_block(void* sdst, const void* gsrc, int nbytes) {
    char* d = static_cast<char*>(sdst);
    const char* src = static_cast<const char*>(gsrc);
    if (((reinterpret_cast<size_t>(d) | reinterpret_cast<size_t>(src) | (size_t)nbytes) & 15) == 0) {
        for (int e = threadIdx.x; e < nbytes / 16; e += blockDim.x) cp_async16(d + 16 * e, src + 16 * e);
    } else {
        for (int e = threadIdx.x; e < nbytes / 8; e += blockDim.x) cp_async8(d + 8 * e, src + 8 * e);
    }
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The block a kernel body works on: its index and the number of blocks of
// its launch for this system. A single-system launch passes (blockIdx.x,
// gridDim.x); a batched launch over many systems passes the block's index
// within its system's share of the grid and that share's size.
struct Blk {
    int id, n;
};

__device__ __forceinline__ float r_exp(float x) { return expf(x); }
__device__ __forceinline__ double r_exp(double x) { return exp(x); }
__device__ __forceinline__ float r_erfc(float x) { return erfcf(x); }
__device__ __forceinline__ double r_erfc(double x) { return erfc(x); }
__device__ __forceinline__ float r_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double r_sqrt(double x) { return sqrt(x); }
// 1/sqrt: the hardware approximation in float (2 ulp). In double, Newton's
// iteration for x^{-1/2}, y <- y + y (1/2 - (x/2) y^2), from the float value:
// the relative error e goes to ~(3/2) e^2 per step, 2^-21 -> 2^-41 -> rounding
// (within 2 ulp), in 3 multiplies and 4 fused multiply-adds on the FP64 units
// instead of a correctly rounded square root and quotient. Outside the normal
// float range of x the quotient is taken.
__device__ __forceinline__ float r_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double r_rsqrt(double x) {
    const float xf = (float)x;
    if (!(xf > 1e-30f && xf < 1e30f)) return 1.0 / sqrt(x);
    double y = (double)rsqrtf(xf);
    const double h = 0.5 * x;
    y = fma(y, fma(-h, y * y, 0.5), y);
    y = fma(y, fma(-h, y * y, 0.5), y);
    return y;
}

// ---------------------------------------------------------------------------
// Coordinates. FP64 wraps and grid coordinates follow the exact operation
// sequence of the definition (no fused multiply-add), FP32 ones are formed in
// float with error terms, so the integer decisions (grid base, tile, cell) are
// reproducible.
// ---------------------------------------------------------------------------
// q = floor(x / L) comes from a float quotient (off by at most one for
// |x| < 2^20 L) corrected in double until 0 <= x - L q < L: the same q and w
// as an FP64 division would give, without one (an FP64 division is a long
// sequence on this part's few FP64 units, and DPD positions drift out of the
// box, so most steps wrap many beads).
__device__ __forceinline__ double wrap_pos(double x, double L) {
    if (x >= 0.0 && x < L) return x;
    double q = (double)floorf(__fdiv_rn((float)x, (float)L));
    double w = __dsub_rn(x, __dmul_rn(L, q));
    if (w < 0.0) {
        q -= 1.0;
        w = __dsub_rn(x, __dmul_rn(L, q));
    } else if (w >= L) {
        q += 1.0;
        w = __dsub_rn(x, __dmul_rn(L, q));
    }
    if (w >= L || w < 0.0) w = 0.0;
    return w;
}

// Wrapped position in the working precision, in [0, L). Inside [0, L) the value
// is kept as is (decided in float for float: x <= xmaxf, the largest float
// below L). FP32: a value within half a unit of L, which only float(L) >= L could
// hold, is 0, the same point of the periodic box to within its rounding.
// FP32: x - L q in float arithmetic with error terms, L = Lhi + Llo: the product
// q Lhi and the difference x - fl(q Lhi) are taken with their exact rounding
// errors (fused multiply-add; two-sum), which are added back with q Llo before
// the one rounding that counts. The terms added back are below 2^-22 |x| and
// carry an error below 2^-45 |x|, so a result of at least 2^-16 |x| is the FP64
// wrap rounded to float but within 1/32 unit of a tie; a smaller one, one at a
// face and one whose q is off by one take the FP64 wrap. That costs ~8 FP64
// instructions per coordinate (16 cycles of the SM each), and DPD positions
// drift out of the box, so nearly every warp wraps some bead, but a bead k boxes
// away takes it once in 65536 / k times only.
__device__ __forceinline__ float wrap_diff(float x, float q, float Lhi, float Llo) {
    const float p = __fmul_rn(q, Lhi);
    const float pe = __fmaf_rn(q, Lhi, -p);          // q Lhi = p + pe
    const float d = __fsub_rn(x, p);
    const float bb = __fsub_rn(d, x);                // two-sum: x - p = d + de
    const float de = __fsub_rn(__fsub_rn(x, __fsub_rn(d, bb)), __fadd_rn(p, bb));
    return __fadd_rn(d, __fsub_rn(__fsub_rn(de, pe), __fmul_rn(q, Llo)));
}
__device__ __forceinline__ float wrap_r(float x, double L, float xmaxf, float Lhi, float Llo) {
    if (x >= 0.0f && x <= xmaxf) return x;
    const float w = wrap_diff(x, floorf(__fdiv_rn(x, Lhi)), Lhi, Llo);
    if (w >= fabsf(x) * 0x1p-16f && w < xmaxf) return w;
    const float v = __double2float_rn(wrap_pos((double)x, L));
    return v > xmaxf ? 0.0f : v;   // NaN is kept
}
__device__ __forceinline__ double wrap_r(double x, double L, float, float, float) { return wrap_pos(x, L); }

// Grid coordinate u = x_w * (n/L) in [0, n): one FP64 product and one floor
// (n/L formed once on the host). Where the product rounds to n, u and the
// coordinate itself become 0: a bead is stored with the coordinate that its
// tile (its grid base) holds, because the real-space sweep takes the image
// shift of a run of candidates from the tiles.
__device__ __forceinline__ void grid_coord(double& xw, double ratio, int n, int& base, double& frac) {
    double u = __dmul_rn(xw, ratio);
    if (u >= (double)n) {
        u = __dsub_rn(u, (double)n);
        xw = 0.0;
    }
    const double bb = floor(u);
    base = max((int)bb, 0);   // not a number converts to the smallest int: base 0, the fraction stays
    frac = __dsub_rn(u, bb);
}

// FP32 path: the same floor decided in float on a compensated product. With
// n/L = rhi + rlo (two floats), p = fl(x rhi) and t = fl(x rlo + (x rhi - p))
// represent u = p + t to ~1e-13 relative; floor(u) = floor(p), less one when
// p is an integer and t < 0 (u just below n: base n - 1, the coordinate stays).
__device__ __forceinline__ void grid_coord_f(float& x, float rhi, float rlo, int n, int& base, float& frac) {
    float p = __fmul_rn(x, rhi);
    const float e = __fmaf_rn(x, rhi, -p);
    const float t = __fmaf_rn(x, rlo, e);
    const bool over = p >= (float)n;
    if (over) p = __fsub_rn(p, (float)n);
    float b = floorf(p);
    if (p == b && t < 0.0f) b = __fsub_rn(b, 1.0f);
    frac = __fadd_rn(__fsub_rn(p, b), t);
    if (b < 0.0f) b = __fadd_rn(b, (float)n);
    else if (over) x = 0.0f;
    base = (int)b;
}

// Grid base and fraction in the working precision.
__device__ __forceinline__ void grid_coord_r(float& xw, const Geo& g, int& base, float& frac) {
    grid_coord_f(xw, g.rhi, g.rlo, g.n, base, frac);
}
__device__ __forceinline__ void grid_coord_r(double& xw, const Geo& g, int& base, double& frac) {
    grid_coord(xw, g.ratio, g.n, base, frac);
}

// Minimum-image difference and squared distance. For float the sequence is
// fixed with explicit intrinsics (the same sequence decides the cutoff in the
// oracle's float mode).
__device__ __forceinline__ float min_image(float a, float b, float L, float hL) {
    float d = __fsub_rn(a, b);
    if (d > hL) d = __fsub_rn(d, L);
    else if (d < -hL) d = __fadd_rn(d, L);
    return d;
}
__device__ __forceinline__ double min_image(double a, double b, double L, double hL) {
    double d = a - b;
    if (d > hL) d -= L;
    else if (d < -hL) d += L;
    return d;
}
__device__ __forceinline__ float dist2(float x, float y, float z) {
    return __fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)));
}
__device__ __forceinline__ double dist2(double x, double y, double z) { return x * x + y * y + z * z; }

// ---------------------------------------------------------------------------
// Reductions
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <typename R>
__device__ __forceinline__ R warp_sum_r(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Block sum of two doubles; result valid in thread 0. Uses 64 doubles of shared memory.
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double red[2][32];
    // warps holding only zeros skip their shuffle tree (its adds run on the
    // few FP64 units); the branch is uniform over the warp
    if (__any_sync(0xffffffffu, a != 0.0 || b != 0.0)) {
        a = warp_sum(a);
        b = warp_sum(b);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) { red[0][w] = a; red[1][w] = b; }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = l < nw ? red[0][l] : 0.0;
        b = l < nw ? red[1][l] : 0.0;
        a = warp_sum(a);
        b = warp_sum(b);
    }
}

// Block sum, in double, of two values per thread held in the working
// precision; result valid in thread 0. FP32: the values go to shared memory as
// they are and one warp converts and adds them (8 conversions and additions
// per lane and one shuffle tree per quantity for a block of 8 warps), so that
// the other warps spend nothing on the FP64 units (a tree in every warp is 10
// double additions each, 16 cycles of the SM's FP64 units apiece).
constexpr int kSumThreads = 256;
template <typename R>
__device__ __forceinline__ void block_sum2_r(R va, R vb, double& a, double& b) {
    if constexpr (sizeof(R) == 8) {
        a = va;
        b = vb;
        block_sum2(a, b);
    } else {
        __shared__ float vals[2][kSumThreads];   // blockDim.x <= kSumThreads
        __shared__ double bsum;
        const int tid = threadIdx.x;
        vals[0][tid] = va;
        vals[1][tid] = vb;
        __syncthreads();
        if (tid < 64) {   // warp 0: a, warp 1: b
            const int w = tid >> 5, l = tid & 31;
            double s = 0.0;
            for (int k = l; k < (int)blockDim.x; k += 32) s += (double)vals[w][k];
            s = warp_sum(s);
            if (tid == 0) a = s;
            if (tid == 32) bsum = s;
        }
        __syncthreads();
        if (tid == 0) b = bsum;
    }
}

struct Kahan {
    double s = 0.0, c = 0.0;
    __device__ __forceinline__ void add(double x) {
        const double y = x - c;
        const double t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

// Totals quantity qd (0-8) of the 9 (Sum q, Sum q^2, E_real, W_real, E_recip,
// W_recip, E_c, E_bond, E_kin): where its per-block partials sit.
__device__ __forceinline__ void totals_src(const TotalsArgs& t, int qd, int& off, int& cnt, int& stride) {
    if (qd < 2) { off = t.off_q + qd; cnt = t.nq; stride = 2; }
    else if (qd < 4) { off = t.off_real + (qd - 2); cnt = t.nreal; stride = 2; }
    else if (qd < 6) { off = t.off_recip + (qd - 4); cnt = t.nrecip; stride = 2; }
    else if (qd < 8) { off = t.off_dpd + (qd - 6); cnt = t.ndpd; stride = 2; }
    else { off = t.off_kin; cnt = t.nkin; stride = 1; }
}

// Kahan sum, per lane, of the partials i = first, first + step, ... of
// quantity qd (eight independent loads in flight; partials come from other
// blocks and kernels: loads bypass L1).
__device__ __forceinline__ double kahan_lane(const TotalsArgs& t, int qd, int first, int step) {
    int off, cnt, stride;
    totals_src(t, qd, off, cnt, stride);
    Kahan k;
    for (int i0 = first; i0 < cnt; i0 += 8 * step) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + step * u;
            v[u] = i < cnt ? __ldcg(&t.part[off + stride * i]) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) k.add(v[u]);
    }
    return k.s;
}

// Final FP64 totals (Kahan over the per-block partials) by one block of any
// multiple of 32 threads: warp w reduces the quantities qd with qd mod (warps)
// = w among the 9 (with t.pre: quantities 0-7 are read from pre and the
// warps share the kinetic partials).
// Edev: [0] E_real [1] E_recip [2] E_self+E_neutral [3] E_elec [4] E_conservative
//       [5] E_bond [6] E_kinetic [7] virial_elec
static __device__ void totals_block(const Geo& g, const TotalsArgs& t) {
    __shared__ double vals[9];
    __shared__ double kin[32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (t.pre) {
        if (threadIdx.x < 8) vals[threadIdx.x] = __ldcg(&t.pre[threadIdx.x]);
        const double v = warp_sum(kahan_lane(t, 8, threadIdx.x, blockDim.x));
        if (l == 0) kin[w] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int k = 0; k < nw; ++k) s += kin[k];
            vals[8] = s;
        }
    } else {
        for (int qd = w; qd < 9; qd += nw) {
            const double v = warp_sum(kahan_lane(t, qd, l, 32));
            if (l == 0) vals[qd] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double* Edev = t.Edev;
        // constants formed on the host: no FP64 division or square root here
        const double Q = vals[0], Q2 = vals[1];
        const double e_self = g.c_self * Q2;
        const double e_neut = g.c_neut * Q * Q;
        const double e_real = vals[2], e_recip = g.c_recip * vals[4];
        Edev[0] = e_real;
        Edev[1] = e_recip;
        Edev[2] = e_self + e_neut;
        Edev[3] = e_real + e_recip + e_self + e_neut;
        Edev[4] = vals[6];
        Edev[5] = vals[7];
        Edev[6] = vals[8];
        Edev[7] = vals[3] + g.c_recip * vals[5] + 3.0 * e_neut;
        for (int i = 8; i < 16; ++i) Edev[i] = 0.0;
    }
}

// Quantities 0-7 of a DPD step's totals, one block per quantity, launched on
// the side stream once the pair kernels and the reciprocal (z) pass have
// written their partials, so that it runs beside the gather; the step's
// closing totals then add the kinetic partials only (t.pre).
static __global__ void __launch_bounds__(256) k_totals_pre(TotalsArgs t) {
    pdl_enter();
    __shared__ double ws[8];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const double v = warp_sum(kahan_lane(t, blockIdx.x, threadIdx.x, blockDim.x));
    if (l == 0) ws[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += ws[k];
        t.pre[blockIdx.x] = s;
    }
}

// The last block of a kernel to finish (arrival counter) runs the totals;
// nblk: the blocks of the launch that count on this ticket.
__device__ __forceinline__ void totals_if_last(const Geo& g, const TotalsArgs& t, int nblk) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(t.ticket, 1) == nblk - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    totals_block(g, t);
    if (threadIdx.x == 0) *t.ticket = 0;
}


// ---------------------------------------------------------------------------
// a1: binning of the charged beads into tiles of the oversampled grid, a
// counting sort in two kernels (three with many tiles):
// k_bin_count: each block compacts the charged beads of its share (warp
//   ballots into a shared list), computes their grid coordinates on dense
//   warps and takes each bead's rank in its tile from the tile's counter (one
//   global add per charged bead, spread over the tiles).
// k_bin_scatter: every block scans the tile counters for itself (up to
//   kBinScanTiles of them; more go through k_scan_mb), moves its records to
//   their slots (tile start + rank) and, in FP32 single evaluations, computes
//   their window weights. The last block to have read the counters clears
//   them for the next evaluation.
// Per-block tile histograms with a last block that turned them into offsets
// (the form before) cost that block a walk over tiles x blocks counts, or two
// more launches. The stage with the window weights, FP32: 81k beads 22.0 ->
// 15.7 us, 524k 32.5 -> 23.6, 3M 75 -> 51; FP64: 375k 75 -> 55, 3000 28 -> 18.
// ---------------------------------------------------------------------------
constexpr int kBinThreads = 256;

// In-place exclusive scan of count ints in shared memory (data[count] = total)
// by the whole block: contiguous chunks per thread, warp and block scans.
__device__ __forceinline__ void block_exclusive_scan(int* data, int count) {
    __shared__ int wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nwarp = (blockDim.x + 31) >> 5;
    const int per = (count + blockDim.x - 1) / blockDim.x;
    const int i0 = tid * per, i1 = min(count, i0 + per);
    int sum = 0;
    for (int i = i0; i < i1; ++i) sum += data[i];
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int run = x - sum, total = 0;
    for (int k = 0; k < nwarp; ++k) {
        if (k < w) run += wsum[k];
        total += wsum[k];
    }
    for (int i = i0; i < i1; ++i) {
        const int v = data[i];
        data[i] = run;
        run += v;
    }
    if (tid == 0) data[count] = total;
    __syncthreads();
}

// Tile coordinate of a grid line: base < 1024, so the float quotient of
// base + 1/2 is exact.
__device__ __forceinline__ int tile_of(int base, float rT) { return (int)(((float)base + 0.5f) * rT); }

template <typename R>
__device__ __forceinline__ void k_bin_count_body(Geo g, int N, const R* __restrict__ pos,
                                                   const R* __restrict__ q, int* __restrict__ cnt_blk,
                                                   int* __restrict__ tcnt, int* __restrict__ crank,
                                                   typename V4<R>::T* __restrict__ cpos,
                                                   typename V4<R>::T* __restrict__ cfrac, int* __restrict__ cbase,
                                                   R* __restrict__ Fzero, double* __restrict__ qpart,
                                                   R* __restrict__ gzero, Blk blk) {
    pdl_enter();
    extern __shared__ int slist[];   // [chunk]
    __shared__ int scount;
    if (threadIdx.x == 0) scount = 0;
    __syncthreads();
    const int b = blk.id, lane = threadIdx.x & 31;
    const int i0 = b * g.chunk;   // the block's region of the compacted arrays
    double s1 = 0.0, s2 = 0.0;
    // the beads, in groups of 32 consecutive ones (one warp's coalesced load),
    // are dealt to the blocks round robin: charged beads that sit together in
    // the input order (chains, counterions, salt) are spread over all blocks
    // (at most chunk / 32 groups per block: chunk is a multiple of 32)
    constexpr int U = 4;   // groups in flight per warp
    const int nwarp = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const int ngroups = (N + 31) >> 5, step = nwarp * blk.n;
    for (int g0 = b + warp * blk.n; g0 < ngroups; g0 += U * step) {
        R qv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = (g0 + u * step) * 32 + lane;   // i < N + 32 U step: within an int
            qv[u] = g0 + u * step < ngroups && i < N ? q[i] : (R)0;
        }
        if (Fzero) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = (g0 + u * step) * 32 + lane;
                if (g0 + u * step < ngroups && i < N) {
                    Fzero[3 * i] = (R)0;
                    Fzero[3 * i + 1] = (R)0;
                    Fzero[3 * i + 2] = (R)0;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool charged = qv[u] != (R)0;
            const unsigned m = __ballot_sync(0xffffffffu, charged);
            int basei = 0;
            if (lane == 0 && m) basei = atomicAdd(&scount, __popc(m));
            basei = __shfl_sync(0xffffffffu, basei, 0);
            if (charged) slist[basei + __popc(m & ((1u << lane) - 1u))] = (g0 + u * step) * 32 + lane;
        }
    }
    __syncthreads();
    if (gzero) {   // clear the grid for the reduction form of the spreading (n even: n^3 is a multiple of 8)
        const int n4 = g.n * g.n * g.n / 4;
        typename V4<R>::T z4;
        z4.x = z4.y = z4.z = z4.w = (R)0;
        for (int e = b * blockDim.x + threadIdx.x; e < n4; e += blk.n * blockDim.x)
            reinterpret_cast<typename V4<R>::T*>(gzero)[e] = z4;
    }
    const int nc = scount;
    const float rT = 1.0f / (float)g.T;
    for (int k = threadIdx.x; k < nc; k += blockDim.x) {
        if (!ENUF_GUARD(g.check, k < g.chunk, 1)) continue;   // the compacted list holds a chunk
        const int i = slist[k];
        R xw[3], fr[3];
        int bs[3];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            xw[t] = wrap_r(pos[3 * i + t], g.L, g.xmaxf, g.Lhi, g.Llo);
            grid_coord_r(xw[t], g, bs[t], fr[t]);
        }
        const int tile = (tile_of(bs[2], rT) * g.ntd + tile_of(bs[1], rT)) * g.ntd + tile_of(bs[0], rT);
        if (!ENUF_GUARD(g.check, (unsigned)tile < (unsigned)g.ntiles, 0)) continue;
        const int o = i0 + k;
        crank[o] = atomicAdd(&tcnt[tile], 1);
        typename V4<R>::T a, c;
        a.x = xw[0]; a.y = xw[1]; a.z = xw[2]; a.w = q[i];
        // charge sums over the compacted beads: only the block's first warps
        // hold nonzero partials, the rest skip the reduction tree
        s1 += (double)a.w;
        s2 = fma((double)a.w, (double)a.w, s2);
        c.x = fr[0]; c.y = fr[1]; c.z = fr[2]; c.w = int_as_real(i, (R)0);
        cpos[o] = a;
        cfrac[o] = c;
        cbase[o] = bs[0] | (bs[1] << 10) | (bs[2] << 20);
    }
    if (threadIdx.x == 0) cnt_blk[b] = nc;
    block_sum2(s1, s2);
    if (threadIdx.x == 0) {
        qpart[2 * b] = s1;
        qpart[2 * b + 1] = s2;
    }
}

template <typename R>
__global__ void __launch_bounds__(kBinThreads) k_bin_count(Geo g, int N, const R* __restrict__ pos,
                                                   const R* __restrict__ q, int* __restrict__ cnt_blk,
                                                   int* __restrict__ tcnt, int* __restrict__ crank,
                                                   typename V4<R>::T* __restrict__ cpos,
                                                   typename V4<R>::T* __restrict__ cfrac, int* __restrict__ cbase,
                                                   R* __restrict__ Fzero, double* __restrict__ qpart,
                                                   R* __restrict__ gzero) {
    k_bin_count_body<R>(g, N, pos, q, cnt_blk, tcnt, crank, cpos, cfrac, cbase, Fzero, qpart, gzero, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// Exclusive scan of in[0, count) into out[0, count], out[count] = total; one
// CTA of 1024 threads, 16 elements per thread and round (four 16-byte loads).
// aux, when given, receives a copy of out.
static __global__ void __launch_bounds__(1024) k_scan(const int* __restrict__ in, int* __restrict__ out, int count,
                                                      int* __restrict__ aux) {
    pdl_enter();
    constexpr int IPT = 16;
    __shared__ int wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int carry = 0;
    for (int base = 0; base < count; base += 1024 * IPT) {
        const int i0 = base + IPT * tid;
        int v[IPT];
        if (i0 + IPT <= count) {
#pragma unroll
            for (int k = 0; k < IPT; k += 4) {
                const int4 x = *reinterpret_cast<const int4*>(in + i0 + k);
                v[k] = x.x; v[k + 1] = x.y; v[k + 2] = x.z; v[k + 3] = x.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < IPT; ++k) v[k] = i0 + k < count ? in[i0 + k] : 0;
        }
        int sum = 0;
#pragma unroll
        for (int k = 0; k < IPT; ++k) sum += v[k];
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            int z = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, z, o);
                if (lane >= o) z += y;
            }
            wsum[lane] = z;
        }
        __syncthreads();
        int run = carry + (x - sum) + (w > 0 ? wsum[w - 1] : 0);
        const int total = wsum[31];
        if (i0 + IPT <= count) {
#pragma unroll
            for (int k = 0; k < IPT; k += 4) {
                int4 o4;
                o4.x = run; run += v[k];
                o4.y = run; run += v[k + 1];
                o4.z = run; run += v[k + 2];
                o4.w = run; run += v[k + 3];
                *reinterpret_cast<int4*>(out + i0 + k) = o4;
                if (aux) *reinterpret_cast<int4*>(aux + i0 + k) = o4;
            }
        } else {
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const int idx = i0 + k;
                if (idx < count) {
                    out[idx] = run;
                    if (aux) aux[idx] = run;
                }
                run += v[k];
            }
        }
        carry += total;
        __syncthreads();
    }
    if (tid == 0) {
        out[count] = carry;
        if (aux) aux[count] = carry;
    }
}

// Exclusive scan of in[0, count) into out[0, count] and aux (out[count] =
// total) by ceil(count / kScanMbSpan) CTAs of 1024 threads, 4 elements per
// thread: every CTA adds up all elements before its own span (16-byte loads)
// and scans its span, so no CTA waits on another (for counts where that
// redundant prefix read stays small; in must be 16-byte aligned and is not
// modified).
constexpr int kScanMbSpan = 4096;
constexpr int kScanMbMax = 16 * kScanMbSpan;
static __global__ void __launch_bounds__(1024) k_scan_mb(const int* __restrict__ in, int* __restrict__ out, int count,
                                                         int* __restrict__ aux) {
    pdl_enter();
    __shared__ int wsum[32];
    __shared__ int spre;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int base = blockIdx.x * kScanMbSpan;
    int pre = 0;
    for (int k = tid; k < base / 4; k += 1024) {
        const int4 x = reinterpret_cast<const int4*>(in)[k];
        pre += x.x + x.y + x.z + x.w;
    }
    pre = __reduce_add_sync(0xffffffffu, pre);
    if (lane == 0) wsum[w] = pre;
    __syncthreads();
    if (w == 0) {
        const int z = __reduce_add_sync(0xffffffffu, wsum[lane]);
        if (lane == 0) spre = z;
    }
    __syncthreads();
    const int i0 = base + 4 * tid;
    int v[4];
    if (i0 + 4 <= count) {
        const int4 x = *reinterpret_cast<const int4*>(in + i0);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = i0 + k < count ? in[i0 + k] : 0;
    }
    const int sum = v[0] + v[1] + v[2] + v[3];
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) {
        int z = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) z += y;
        }
        wsum[lane] = z;
    }
    __syncthreads();
    int run = spre + (x - sum) + (w > 0 ? wsum[w - 1] : 0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (i0 + k < count) {
            out[i0 + k] = run;
            if (aux) aux[i0 + k] = run;
        }
        run += v[k];
    }
    if (tid == 0 && base + kScanMbSpan >= count) {
        out[count] = spre + wsum[31];
        if (aux) aux[count] = spre + wsum[31];
    }
}

// Window weights of one (bead, dimension) (Eq. 14): out[a] = psi(f + p - 1 - a)
// for the 2p taps a, f the fractional grid coordinate. FP32: an exponential per
// tap. FP64: e^{-(f + m)^2/b} = e^{-f^2/b} (e^{-2f/b})^m e^{-m^2/b} (the fast
// Gaussian gridding of Greengard & Lee, SIAM Rev. 46, 2004): three exponentials
// and products instead of 2p exponentials on the few FP64 units (375k beads,
// p = 4: the binning stage 75 -> 55 us with it); |m| <= p <= 8 keeps the
// products within a few ulp, the rounding that (f + m)^2/b itself brings to the
// direct form.
template <typename R>
__device__ __forceinline__ void window_row(const Geo& g, R f, R* __restrict__ out) {
    const int p = g.p, P2 = 2 * g.p;
    if constexpr (sizeof(R) == 8) {
        const double rb = g.rb;
        const double e0 = exp(-f * f * rb);
        const double up = exp(-2.0 * f * rb), dn = exp(2.0 * f * rb);
        double t = e0;
        for (int m = 0; m < p; ++m) {   // m = 0 .. p - 1: tap p - 1 - m
            out[p - 1 - m] = t * g.e3[m];
            t *= up;
        }
        t = e0;
        for (int m = 1; m <= p; ++m) {   // -m: tap p - 1 + m
            t *= dn;
            out[p - 1 + m] = t * g.e3[m];
        }
    } else {
        const float rb = g.wkf.rb, wn = g.wkf.wn;
        if ((P2 & 3) == 0) {
            for (int a = 0; a < P2; a += 4) {
                float w4[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float u = f + (float)(p - 1 - (a + k));
                    w4[k] = wn * r_exp(-u * u * rb);
                }
                *reinterpret_cast<float4*>(out + a) = make_float4(w4[0], w4[1], w4[2], w4[3]);
            }
        } else {
            for (int a = 0; a < P2; ++a) {
                const float u = f + (float)(p - 1 - a);
                out[a] = wn * r_exp(-u * u * rb);
            }
        }
    }
}

// W: the window weights as well, one thread per (bead, dimension).
template <typename R, bool W>
__device__ __forceinline__ void k_bin_scatter_body(Geo g, const int* __restrict__ cnt_blk, int* __restrict__ tcnt,
                                                     int* __restrict__ tstart, const int* __restrict__ crank,
                                                     const typename V4<R>::T* __restrict__ cpos,
                                                     const typename V4<R>::T* __restrict__ cfrac,
                                                     const int* __restrict__ cbase,
                                                     typename V4<R>::T* __restrict__ sq,
                                                     typename V4<R>::T* __restrict__ sw, int* __restrict__ sb,
                                                     float4* __restrict__ spf, R* __restrict__ wb,
                                                     int* __restrict__ ticket, Blk blk) {
    pdl_enter();
    extern __shared__ int pre[];   // [ntiles + 1] tile starts (g.bin_scan)
    const int b = blk.id;
    const int* ts = tstart;
    if (g.bin_scan) {
        __shared__ int last;
        for (int t = threadIdx.x; t < g.ntiles; t += blockDim.x) pre[t] = __ldcg(&tcnt[t]);
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == blk.n - 1;
        block_exclusive_scan(pre, g.ntiles);   // contains barriers
        if (last) {   // every block has its copy of the counters
            for (int t = threadIdx.x; t < g.ntiles; t += blockDim.x) tcnt[t] = 0;
            if (threadIdx.x == 0) *ticket = 0;
        }
        if (b == 0)
            for (int t = threadIdx.x; t <= g.ntiles; t += blockDim.x) tstart[t] = pre[t];
        ts = pre;
    } else {   // tstart comes from the scan kernel
        for (int t = b * blockDim.x + threadIdx.x; t < g.ntiles; t += blk.n * blockDim.x) tcnt[t] = 0;
    }
    const int nc = cnt_blk[b];
    const int i0 = b * g.chunk;
    const float rT = 1.0f / (float)g.T;
    constexpr int D = W ? 3 : 1;
    for (int e = threadIdx.x; e < D * nc; e += blockDim.x) {
        const int k = e / D, d = e - D * k;
        const int o = i0 + k;
        const int pb = cbase[o];
        const int t = (tile_of((pb >> 20) & 1023, rT) * g.ntd + tile_of((pb >> 10) & 1023, rT)) * g.ntd +
                      tile_of(pb & 1023, rT);
        if (!ENUF_GUARD(g.check, (unsigned)t < (unsigned)g.ntiles, 2)) continue;
        const int slot = ts[t] + crank[o];
        if (!ENUF_GUARD(g.check, (unsigned)slot < (unsigned)g.nmax, 2)) continue;
        const typename V4<R>::T c = cfrac[o];
        if (d == 0) {
            const typename V4<R>::T a = cpos[o];
            sq[slot] = a;
            sw[slot] = c;
            sb[slot] = pb;
            // FP64: a float copy of the position for the real-space cutoff pre-test
            if (sizeof(R) == 8 && spf) spf[slot] = make_float4((float)a.x, (float)a.y, (float)a.z, 0.f);
        }
        if constexpr (W)
            window_row<R>(g, d == 0 ? c.x : (d == 1 ? c.y : c.z), wb + ((size_t)slot * 3 + d) * (2 * g.p));
    }
}

template <typename R, bool W>
__global__ void __launch_bounds__(kBinThreads) k_bin_scatter(Geo g, const int* __restrict__ cnt_blk, int* __restrict__ tcnt,
                                                     int* __restrict__ tstart, const int* __restrict__ crank,
                                                     const typename V4<R>::T* __restrict__ cpos,
                                                     const typename V4<R>::T* __restrict__ cfrac,
                                                     const int* __restrict__ cbase,
                                                     typename V4<R>::T* __restrict__ sq,
                                                     typename V4<R>::T* __restrict__ sw, int* __restrict__ sb,
                                                     float4* __restrict__ spf, R* __restrict__ wb,
                                                     int* __restrict__ ticket) {
    k_bin_scatter_body<R, W>(g, cnt_blk, tcnt, tstart, crank, cpos, cfrac, cbase, sq, sw, sb, spf, wb, ticket,
                             Blk{(int)blockIdx.x, (int)gridDim.x});
}

// Window weights of every sorted charged bead, computed once and read by the
// spreading and gathering kernels: wb[s][d][a]. One thread per (bead,
// dimension) writes its 2p consecutive weights; all SMs (in FP64 the
// exponentials run on the FP64 units).
template <typename R>
__device__ __forceinline__ void k_bin_weights_body(Geo g, const int* __restrict__ tstart,
                                                    const typename V4<R>::T* __restrict__ sw, R* __restrict__ wb, Blk blk) {
    pdl_enter();
    const int nq = tstart[g.ntiles];
    const int tot = 3 * nq;   // (bead, dimension) pairs; nq <= n_max < 2^29
    for (int e = blk.id * blockDim.x + threadIdx.x; e < tot; e += blk.n * blockDim.x) {
        const int s = e / 3, d = e - 3 * s;
        const typename V4<R>::T fr = sw[s];
        window_row<R>(g, d == 0 ? fr.x : (d == 1 ? fr.y : fr.z), wb + (size_t)e * (2 * g.p));
    }
}

template <typename R>
__global__ void __launch_bounds__(256) k_bin_weights(Geo g, const int* __restrict__ tstart,
                                                    const typename V4<R>::T* __restrict__ sw, R* __restrict__ wb) {
    k_bin_weights_body<R>(g, tstart, sw, wb, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---------------------------------------------------------------------------
// a2: spreading g(l) = sum_j q_j prod_t psi(u_jt - l_t)   (Eq. 14/19, first half)
// One CTA owns one T^3 tile of the grid: it visits the beads of the (up to)
// 27 neighbouring bins, deposits the taps that fall inside its tile into
// shared memory, and writes the finished tile once. No global atomics.
// ---------------------------------------------------------------------------
constexpr int kSpreadThreads = 256;
constexpr int kMaxTaps = 16;
constexpr int kSpreadCap = 512;   // beads staged in shared memory per round
// Shared slots of the work-item kernel's tile: T^3 rounded up to a multiple of
// 4, so that the regions after it (the int2 work items last) stay 16-byte
// aligned for odd T as well.
__host__ __device__ constexpr int spread_tile_slots(int T) { return (T * T * T + 3) & ~3; }

// Taps of a bead (base b, 2p taps from b - p + 1) that fall in the tile [o, o+T)
// of a periodic grid of n points, as a bit mask over the taps. With at least
// 3 tiles per dimension the window (2p <= 2T) meets tile tb - 1, tb or tb + 1
// of the bead's tile tb in one contiguous run, found arithmetically; otherwise
// the taps are tested one by one.
__device__ __forceinline__ unsigned tap_mask(int b, int o, int T, int n, int ntd, int p) {
    const int P2 = 2 * p;
    if (ntd >= 3) {
        const int tb = b / T, tc = o / T;
        int dt = tc - tb;
        if (dt > 1) dt -= ntd;
        else if (dt < -1) dt += ntd;
        if (dt < -1 || dt > 1) return 0u;
        const int ou = (tb + dt) * T;        // tile origin in the bead's unwrapped frame
        const int l0 = b - p + 1;
        const int a0 = max(0, ou - l0), a1 = min(P2, ou + T - l0);
        if (a1 <= a0) return 0u;
        return ((a1 - a0) >= 32 ? 0xffffffffu : ((1u << (a1 - a0)) - 1u)) << a0;
    }
    unsigned m = 0u;
    for (int a = 0; a < P2; ++a) {
        int l = b - p + 1 + a;
        l = l < 0 ? l + n : (l >= n ? l - n : l);
        if ((unsigned)(l - o) < (unsigned)T) m |= 1u << a;
    }
    return m;
}

// Slots [lo, lo + cnt) of the tile (lines o .. o + T - 1) that hold the taps in
// mask m != 0: contiguous taps on contiguous slots, else (taps or slots wrap
// around a grid of few tiles) the whole tile, whose other slots weigh 0.
__device__ __forceinline__ int tap_slots(unsigned m, int b, int o, int T, int n, int p) {
    const int t0 = __ffs(m) - 1, t1 = 31 - __clz(m), c = __popc(m);
    int s0 = b - p + 1 + t0 - o;   // in (-n - p, n + p)
    s0 += s0 < 0 ? n : 0;
    s0 -= s0 >= n ? n : 0;
    const bool run = c == t1 - t0 + 1 && s0 + c <= T;
    return run ? (s0 | c << 5) : (T << 5);
}

template <typename R>
__global__ void __launch_bounds__(kSpreadThreads, 5) k_spread(Geo g, const int* __restrict__ tstart,
                                                           const typename V4<R>::T* __restrict__ sq,
                                                           const typename V4<R>::T* __restrict__ sw,
                                                           const int* __restrict__ sb,
                                                           R* __restrict__ grid) {
    pdl_enter();
    using V = typename V4<R>::T;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int T = g.T, T3 = T * T * T;
    constexpr int NW = kSpreadThreads / 32;
    V* stg = reinterpret_cast<V*>(smraw);                          // [cap] (fx, fy, fz, q)
    R* acc = reinterpret_cast<R*>(stg + kSpreadCap);                // [T^3], padded to spread_tile_slots(T)
    R* wts = acc + spread_tile_slots(T);                            // [NW][3][16]
    int* lix = reinterpret_cast<int*>(wts + NW * 3 * kMaxTaps);     // [NW][3][16]
    int* sbase = lix + NW * 3 * kMaxTaps;                           // [cap]
    int2* items = reinterpret_cast<int2*>(sbase + kSpreadCap);      // [cap] (bead | x mask, y mask | z mask)
    __shared__ int nb_start[27], nb_pre[28];
    __shared__ int nnb, nitems;

    const int tile = blockIdx.x;
    const int tx = tile % g.ntd, ty = (tile / g.ntd) % g.ntd, tz = tile / (g.ntd * g.ntd);
    const int o[3] = {tx * T, ty * T, tz * T};
    for (int e = threadIdx.x; e < T3; e += blockDim.x) acc[e] = (R)0;
    const int no = g.ntd >= 3 ? 3 : g.ntd;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {   // neighbouring bins (<= 27): starts and an exclusive prefix of their sizes
        const int cntn = no * no * no;
        int st = 0, c = 0;
        if (lane < cntn) {
            const int dx = lane % no, dy = (lane / no) % no, dz = lane / (no * no);
            const int nz = g.ntd >= 3 ? (tz + dz - 1 + g.ntd) % g.ntd : dz;
            const int ny = g.ntd >= 3 ? (ty + dy - 1 + g.ntd) % g.ntd : dy;
            const int nx = g.ntd >= 3 ? (tx + dx - 1 + g.ntd) % g.ntd : dx;
            const int nt = (nz * g.ntd + ny) * g.ntd + nx;
            st = tstart[nt];
            c = tstart[nt + 1] - st;
        }
        int x = c;
#pragma unroll
        for (int of = 1; of < 32; of <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, of);
            if (lane >= of) x += y;
        }
        if (lane < cntn) {
            nb_start[lane] = st;
            nb_pre[lane] = x - c;
        }
        if (lane == cntn - 1) {
            nb_pre[cntn] = x;
            nnb = cntn;
        }
    }
    __syncthreads();
    R* myw = wts + warp * 3 * kMaxTaps;
    int* myl = lix + warp * 3 * kMaxTaps;
    const int P2 = 2 * g.p;
    const int total = nb_pre[nnb];
    const R rb = win_k(g, (R)0).rb, wn = win_k(g, (R)0).wn;
    for (int cb = 0; cb < total; cb += kSpreadCap) {
        const int cn = min(kSpreadCap, total - cb);
        if (threadIdx.x == 0) nitems = 0;
        // stage this round's candidates: one thread per bead, its bin by binary search
        for (int idx = threadIdx.x; idx < cn; idx += blockDim.x) {
            const int f = cb + idx;
            int lo = 0, hi = nnb;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (nb_pre[mid] <= f) lo = mid; else hi = mid;
            }
            const int j = nb_start[lo] + f - nb_pre[lo];
            V v = sw[j];
            v.w = sq[j].w;
            stg[idx] = v;
            sbase[idx] = sb[j];
        }
        __syncthreads();
        // phase A: one lane per candidate; beads whose window meets this tile become work items
        for (int c0 = 0; c0 < cn; c0 += blockDim.x) {
            const int c = c0 + threadIdx.x;
            unsigned mx = 0u, my = 0u, mz = 0u;
            if (c < cn) {
                const int pb = sbase[c];
                mx = tap_mask(pb & 1023, o[0], T, g.n, g.ntd, g.p);
                if (mx) my = tap_mask((pb >> 10) & 1023, o[1], T, g.n, g.ntd, g.p);
                if (my) mz = tap_mask((pb >> 20) & 1023, o[2], T, g.n, g.ntd, g.p);
            }
            const bool keep = mz != 0u;
            const unsigned bal = __ballot_sync(0xffffffffu, keep);
            int basei = 0;
            if (lane == 0 && bal) basei = atomicAdd(&nitems, __popc(bal));
            basei = __shfl_sync(0xffffffffu, basei, 0);
            if (keep) items[basei + __popc(bal & ((1u << lane) - 1u))] = make_int2(c | (int)(mx << 16), (int)(my | (mz << 16)));
        }
        __syncthreads();
        const int ni = nitems;
        // phase B: one warp per work item
        for (int it = warp; it < ni; it += NW) {
            const int2 e = items[it];
            const int c = e.x & 0xffff;
            const unsigned msk[3] = {(unsigned)e.x >> 16, (unsigned)e.y & 0xffffu, (unsigned)e.y >> 16};
            const V wv = stg[c];
            const int pb = sbase[c];
            if (lane < P2) {
                const int base[3] = {pb & 1023, (pb >> 10) & 1023, (pb >> 20) & 1023};
                const R fr[3] = {wv.x, wv.y, wv.z};
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    if ((msk[t] >> lane) & 1u) {
                        const int slot = __popc(msk[t] & ((1u << lane) - 1u));
                        int l = base[t] - g.p + 1 + lane;
                        l = l < 0 ? l + g.n : (l >= g.n ? l - g.n : l);
                        const R d = fr[t] + (R)(g.p - 1 - lane);
                        myw[t * kMaxTaps + slot] = wn * r_exp(-d * d * rb);
                        myl[t * kMaxTaps + slot] = l - o[t];
                    }
                }
            }
            __syncwarp();
            const int cx = __popc(msk[0]), cy = __popc(msk[1]), cz = __popc(msk[2]);
            const int cxy = cx * cy;
            // xy -> (ix, iy) by a float reciprocal: xy < 256 and the true quotient of
            // xy + 1/2 is at least 1/32 away from an integer, far above the error
            const float icx = 1.0f / (float)cx;
            const R qj = wv.w;
            for (int xy = lane; xy < cxy; xy += 32) {
                const int iy = (int)(((float)xy + 0.5f) * icx);
                const int ix = xy - iy * cx;
                const R wxy = qj * myw[ix] * myw[kMaxTaps + iy];
                const int rowo = myl[kMaxTaps + iy] * T + myl[ix];
                for (int iz = 0; iz < cz; ++iz)
                    atomicAdd(&acc[myl[2 * kMaxTaps + iz] * T * T + rowo], wxy * myw[2 * kMaxTaps + iz]);
            }
            __syncwarp();
        }
        __syncthreads();
    }
    const int n = g.n;
    // write-back, one row of T <= 24 points per warp iteration
    int ly = warp, lz = 0;
    while (ly >= T) { ly -= T; ++lz; }
    while (lz < T) {
        if (lane < T) grid[((size_t)(o[2] + lz) * n + (o[1] + ly)) * n + (o[0] + lane)] = acc[(lz * T + ly) * T + lane];
        ly += NW;
        while (ly >= T) { ly -= T; ++lz; }
    }
}

// Column-stationary spreading for the common tile edges T (template): one CTA
// per T^3 tile; candidates are the charged beads of the 27 neighbouring bins;
// those whose window meets the tile become items; per batch of items the
// per-dimension weights restricted to the tile (T slots each, zero outside
// the item's taps, q folded into z) are laid out in shared memory from the
// per-bead weights; each thread owns one (x, y) column of the tile and adds
// w_x w_y w_z(z) for every item into T registers. No atomics; the tile is
// written once.
constexpr int kColCand = 512;    // candidates staged per round
constexpr int kColItems = 128;   // items per weight batch

//
// SLAB (the FP64 form): the same staging, but the tile is accumulated in
// shared memory and each of the 4 warps owns a slab of z-planes; per item a
// warp whose slab meets the item's z-range spreads the item's footprint
// (its slots in x and y, lanes over the footprint's columns) into its planes.
// The FP64 units are then spent on the item's taps only: the column form
// multiplies every column of the tile by every z-slot, zero or not, and on
// GB300's few FP64 units that was ~4x the instructions.
constexpr int kSlabThreads = 128;
__host__ __device__ constexpr int col_threads(int T) { return T * T <= 128 ? 128 : ((T * T + 31) / 32) * 32; }
template <bool SLAB>
__host__ __device__ constexpr int spread2_threads(int T) { return SLAB ? kSlabThreads : col_threads(T); }

template <typename R>
__host__ __device__ constexpr int col_smem(int T, bool slab = false) {
    return kColCand * (4 + 4 + 8 + (int)sizeof(R)) + kColItems * 3 * T * (int)sizeof(R) +
           (slab ? T * T * T * (int)sizeof(R) : 0);
}

template <typename R, int T, bool SLAB>
__device__ __forceinline__ void k_spread_col_body(Geo g, const int* __restrict__ tstart,
                                                                        const typename V4<R>::T* __restrict__ sq,
                                                                        const int* __restrict__ sb,
                                                                        const R* __restrict__ wb,
                                                                        R* __restrict__ grid, Blk blk) {
    pdl_enter();
    constexpr int NT = spread2_threads<SLAB>(T);
    constexpr int NW = NT / 32;
    constexpr int SZ = (T + NW - 1) / NW;   // SLAB: z-planes per warp
    extern __shared__ __align__(16) unsigned char smraw[];
    R* wt = reinterpret_cast<R*>(smraw);                        // [kColItems][3][T]
    R* cq = wt + kColItems * 3 * T;                             // [kColCand] charges
    int* cslot = reinterpret_cast<int*>(cq + kColCand);         // [kColCand] sorted slots
    int* cbase = cslot + kColCand;                              // [kColCand] packed bases
    int2* items = reinterpret_cast<int2*>(cbase + kColCand);    // [kColCand] (candidate, slot ranges)
    R* acc_s = reinterpret_cast<R*>(items + kColCand);          // SLAB: [T][T][T] tile
    __shared__ int nb_start[27], nb_pre[28];
    __shared__ int nnb, nitems;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blk.id;
    const int tx = tile % g.ntd, ty = (tile / g.ntd) % g.ntd, tz = tile / (g.ntd * g.ntd);
    const int o[3] = {tx * T, ty * T, tz * T};
    const int no = g.ntd >= 3 ? 3 : g.ntd;
    if (warp == 0) {   // neighbouring bins (<= 27): starts and an exclusive prefix of their sizes
        const int cntn = no * no * no;
        int st = 0, c = 0;
        if (lane < cntn) {
            const int dx = lane % no, dy = (lane / no) % no, dz = lane / (no * no);
            const int nz = g.ntd >= 3 ? (tz + dz - 1 + g.ntd) % g.ntd : dz;
            const int ny = g.ntd >= 3 ? (ty + dy - 1 + g.ntd) % g.ntd : dy;
            const int nx = g.ntd >= 3 ? (tx + dx - 1 + g.ntd) % g.ntd : dx;
            const int nt = (nz * g.ntd + ny) * g.ntd + nx;
            st = tstart[nt];
            c = tstart[nt + 1] - st;
        }
        int x = c;
#pragma unroll
        for (int of = 1; of < 32; of <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, of);
            if (lane >= of) x += y;
        }
        if (lane < cntn) {
            nb_start[lane] = st;
            nb_pre[lane] = x - c;
        }
        if (lane == cntn - 1) {
            nb_pre[cntn] = x;
            nnb = cntn;
        }
    }
    __syncthreads();
    const int P2 = 2 * g.p, n = g.n;
    const int cx = tid % T, cy = tid / T;   // this thread's column (tid < T^2)
    const bool owner = !SLAB && tid < T * T;
    R acc[SLAB ? 1 : T];
    const int z0w = warp * SZ, z1w = min(T, z0w + SZ);   // SLAB: this warp's planes
    if constexpr (SLAB) {
        for (int e = z0w * T * T + lane; e < z1w * T * T; e += 32) acc_s[e] = (R)0;
    } else {
#pragma unroll
        for (int z = 0; z < T; ++z) acc[z] = (R)0;
    }
    const int total = nb_pre[nnb];
    for (int cb = 0; cb < total; cb += kColCand) {
        const int cn = min(kColCand, total - cb);
        if (tid == 0) nitems = 0;
        for (int idx = tid; idx < cn; idx += NT) {   // stage: one thread per candidate
            const int f = cb + idx;
            int lo = 0, hi = nnb;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (nb_pre[mid] <= f) lo = mid; else hi = mid;
            }
            const int j = nb_start[lo] + f - nb_pre[lo];
            cslot[idx] = j;
            cbase[idx] = sb[j];
            cq[idx] = sq[j].w;
        }
        __syncthreads();
        for (int c0 = 0; c0 < cn; c0 += NT) {   // items: candidates whose window meets the tile
            const int c = c0 + tid;
            unsigned mx = 0u, my = 0u, mz = 0u;
            if (c < cn) {
                const int pb = cbase[c];
                mx = tap_mask(pb & 1023, o[0], T, n, g.ntd, g.p);
                if (mx) my = tap_mask((pb >> 10) & 1023, o[1], T, n, g.ntd, g.p);
                if (my) mz = tap_mask((pb >> 20) & 1023, o[2], T, n, g.ntd, g.p);
            }
            const bool keep = mz != 0u;
            int rg = 0;   // SLAB: slot ranges (lo | cnt << 5) of x, y, z at bits 0, 10, 20
            if (SLAB && keep) {
                const int pb = cbase[c];
                rg = tap_slots(mx, pb & 1023, o[0], T, n, g.p) | tap_slots(my, (pb >> 10) & 1023, o[1], T, n, g.p) << 10 |
                     tap_slots(mz, (pb >> 20) & 1023, o[2], T, n, g.p) << 20;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, keep);
            int basei = 0;
            if (lane == 0 && bal) basei = atomicAdd(&nitems, __popc(bal));
            basei = __shfl_sync(0xffffffffu, basei, 0);
            const int at = basei + __popc(bal & ((1u << lane) - 1u));
            if (keep && ENUF_GUARD(g.check, at < kColCand, 3)) items[at] = make_int2(c, rg);
        }
        __syncthreads();
        const int ni = nitems;
        for (int ib = 0; ib < ni; ib += kColItems) {
            const int nb = min(kColItems, ni - ib);
            // weights restricted to the tile: slot s of dimension d holds the weight of the
            // tap on grid line o_d + s, or 0 when that line is outside the item's window
            for (int e = tid; e < nb * 3 * T; e += NT) {
                const int i = e / (3 * T), r = e - i * (3 * T);
                const int d = r / T, sl = r - d * T;
                const int c = items[ib + i].x;
                const int base = (cbase[c] >> (10 * d)) & 1023;
                int a = o[d] + sl - base + g.p - 1;
                if (a < 0) a += n;
                else if (a >= n) a -= n;
                R v = (R)0;
                if (a < P2) v = wb[(size_t)cslot[c] * 3 * P2 + d * P2 + a];
                if (d == 2) v *= cq[c];
                wt[e] = v;
            }
            __syncthreads();
            if constexpr (SLAB) {
                for (int i = 0; i < nb; ++i) {
                    const int rg = items[ib + i].y;
                    const int lz = (rg >> 20) & 31, hz = lz + ((rg >> 25) & 31);
                    const int za = max(lz, z0w), zb = min(hz, z1w);
                    if (za >= zb) continue;   // warp-uniform
                    const int lx = rg & 31, nx = (rg >> 5) & 31, ly = (rg >> 10) & 31, ny = (rg >> 15) & 31;
                    const R* wi = wt + i * 3 * T;
                    // xy -> (ix, iy) by a float reciprocal: xy < 576 and the true quotient of
                    // xy + 1/2 is at least 1/48 away from an integer, far above the error
                    const float inx = 1.0f / (float)nx;
                    for (int xy = lane; xy < nx * ny; xy += 32) {
                        const int iy = (int)(((float)xy + 0.5f) * inx);
                        const int x = lx + xy - iy * nx, y = ly + iy;
                        if (!ENUF_GUARD(g.check, x < T && y < T && zb <= T, 4)) continue;
                        const R w = wi[x] * wi[T + y];
                        R* a = acc_s + y * T + x;
                        for (int z = za; z < zb; ++z) a[z * T * T] += w * wi[2 * T + z];
                    }
                }
            } else if (owner) {
                for (int i = 0; i < nb; ++i) {
                    const R* wi = wt + i * 3 * T;
                    const R w = wi[cx] * wi[T + cy];
                    if (w != (R)0) {
#pragma unroll
                        for (int z = 0; z < T; ++z) acc[z] += w * wi[2 * T + z];
                    }
                }
            }
            __syncthreads();
        }
    }
    if constexpr (SLAB) {   // each warp writes its own planes, rows of T points
        const size_t n2 = (size_t)n * n;
        for (int e = z0w * T * T + lane; e < z1w * T * T; e += 32) {
            const int z = e / (T * T), r = e - z * T * T, y = r / T, x = r - y * T;
            grid[(size_t)(o[2] + z) * n2 + (size_t)(o[1] + y) * n + (o[0] + x)] = acc_s[e];
        }
    } else if (owner) {
        R* col = grid + ((size_t)o[2] * n + (o[1] + cy)) * n + (o[0] + cx);
        const size_t n2 = (size_t)n * n;
#pragma unroll
        for (int z = 0; z < T; ++z) col[z * n2] = acc[z];
    }
}

template <typename R, int T, bool SLAB>
__global__ void __launch_bounds__(spread2_threads<SLAB>(T)) k_spread_col(Geo g, const int* __restrict__ tstart,
                                                                        const typename V4<R>::T* __restrict__ sq,
                                                                        const int* __restrict__ sb,
                                                                        const R* __restrict__ wb,
                                                                        R* __restrict__ grid) {
    k_spread_col_body<R, T, SLAB>(g, tstart, sq, sb, wb, grid, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---------------------------------------------------------------------------
// a2, scatter form (FP32; large grids with few beads per grid point). One CTA
// owns a region of RT^3 tiles, edge E = RT T (a template constant), held in
// shared memory. Its candidates are the charged beads of the (RT + 2)^3 bins
// around it: a window of 2p <= T taps reaches no farther than the next tile.
// Warps test 32 candidates at a time against the region and append the beads
// whose window meets it to a shared list; the list is then spread bead by
// bead, a warp per bead: lanes over its (x, y) taps, a loop over the z taps
// inside the region, each product q w_x w_y w_z added to the region. Work is
// spent only on taps that land in the region (the column form multiplies
// every column of its tile by every z slot, which at ~100 grid points per
// charged bead is mostly zeros).
//
// The region accumulates in 32-bit fixed point with native integer shared
// atomics (a float add to shared memory is a compare-and-swap loop): scale
// S = 2^k with S B <= 2^30, B = sum over the region's beads of |q| w_max^3
// bounding every point (w_max = the window's peak, psi(0)). Each term is
// rounded to 1/S: at most B 2^-31 per term, below the float rounding of the
// larger terms; the region is written once, rows of E points as 16-byte
// stores, converted back to float.
// The host admits it when 2p = PT, E is a multiple of T, RT <= 2 divides the
// tiles per dimension ntd >= RT + 2, n % 4 = 0 and n >= 2 (E + T + PT): a
// window's offset from the region origin is then unique modulo n.
// ---------------------------------------------------------------------------
constexpr int kScThreads = 256;
constexpr int kScCap = 1024;   // listed beads per round = candidates per round

// x pitch of the region in shared memory: the 8 x taps x 4 y rows of one
// update land on 32 distinct banks when the pitch is 8 or 24 modulo 32
__host__ __device__ constexpr int sc_pitch(int E) { return (E % 32 == 8 || E % 32 == 24) ? E : sc_pitch(E + 4); }
__host__ __device__ constexpr int sc_smem(int E) { return E * E * sc_pitch(E) * (int)sizeof(int) + kScCap * 16; }

template <int E, int PT>
__global__ void __launch_bounds__(kScThreads) k_spread_sc(Geo g, const int* __restrict__ tstart,
                                                          const float4* __restrict__ sq, const int* __restrict__ sb,
                                                          const float* __restrict__ wb, float* __restrict__ grid) {
    pdl_enter();
    static_assert(E % 4 == 0 && PT >= 2 && PT <= 16, "region edge and window");
    constexpr int EP = sc_pitch(E);
    constexpr int BPR = 32 / PT;               // y taps per round of lanes
    constexpr int NR = (PT + BPR - 1) / BPR;   // rounds
    constexpr int NW = kScThreads / 32;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) int acc[];            // [E][E][EP] fixed point
    int4* items = reinterpret_cast<int4*>(acc + E * E * EP);   // [kScCap] (bead, offsets, q, -)
    __shared__ int nb_start[64], nb_pre[65];
    __shared__ int nitems;
    __shared__ float wsum[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int T = g.T, RT = E / T, nr = g.ntd / RT;
    const int rx = blockIdx.x % nr, ry = (blockIdx.x / nr) % nr, rz = blockIdx.x / (nr * nr);
    const int ox = rx * E, oy = ry * E, oz = rz * E;
    for (int e = tid; e < E * E * EP / 4; e += kScThreads) reinterpret_cast<int4*>(acc)[e] = make_int4(0, 0, 0, 0);
    const int nbd = RT + 2, nbins = nbd * nbd * nbd;   // <= 64
    if (warp == 0) {   // the bins, their bead ranges and an exclusive prefix of their sizes
        int run = 0;
        for (int k0 = 0; k0 < nbins; k0 += 32) {
            const int k = k0 + lane;
            int st = 0, cnt = 0;
            if (k < nbins) {
                const int dx = k % nbd, dy = (k / nbd) % nbd, dz = k / (nbd * nbd);
                const int bx = (rx * RT + dx - 1 + g.ntd) % g.ntd;
                const int by = (ry * RT + dy - 1 + g.ntd) % g.ntd;
                const int bz = (rz * RT + dz - 1 + g.ntd) % g.ntd;
                const int t = (bz * g.ntd + by) * g.ntd + bx;
                st = tstart[t];
                cnt = tstart[t + 1] - st;
            }
            int x = cnt;
#pragma unroll
            for (int of = 1; of < 32; of <<= 1) {
                const int y = __shfl_up_sync(FULL, x, of);
                if (lane >= of) x += y;
            }
            if (k < nbins) {
                nb_start[k] = st;
                nb_pre[k] = run + x - cnt;
            }
            run += __shfl_sync(FULL, x, 31);
        }
        if (lane == 0) {
            nb_pre[nbins] = run;
            nitems = 0;
        }
    }
    __syncthreads();
    const int p = g.p, n = g.n, hn = n >> 1;
    const int total = nb_pre[nbins];
    // Candidates [f0, f1) of the bins' concatenation, 32 per warp step: the beads
    // whose window meets the region, appended to the list (list) and/or their
    // |q| summed.
    auto scan = [&](int f0, int f1, bool list, float& qsum) {
        for (int fb = f0 + 32 * warp; fb < f1; fb += 32 * NW) {
            const int f = fb + lane;
            bool hit = false;
            int pk = 0, j = 0;
            if (f < f1) {
                // its bin: the last k with nb_pre[k] <= f (a non-empty bin)
                int k = 0;
#pragma unroll
                for (int st = 32; st > 0; st >>= 1)
                    if (k + st < nbins && nb_pre[k + st] <= f) k += st;
                j = nb_start[k] + f - nb_pre[k];
                const int pb = sb[j];
                int d0 = (pb & 1023) - p + 1 - ox, d1 = ((pb >> 10) & 1023) - p + 1 - oy;
                int d2 = ((pb >> 20) & 1023) - p + 1 - oz;
                d0 += d0 < -hn ? n : (d0 >= hn ? -n : 0);
                d1 += d1 < -hn ? n : (d1 >= hn ? -n : 0);
                d2 += d2 < -hn ? n : (d2 >= hn ? -n : 0);
                hit = d0 > -PT && d0 < E && d1 > -PT && d1 < E && d2 > -PT && d2 < E;
                pk = (d0 + PT) | (d1 + PT) << 8 | (d2 + PT) << 16;   // each in [1, E + PT) < 256
            }
            const float qj = hit ? sq[j].w : 0.f;
            qsum += fabsf(qj);
            if (list) {
                const unsigned m = __ballot_sync(FULL, hit);
                int at = 0;
                if (lane == 0 && m) at = atomicAdd(&nitems, __popc(m));
                at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (hit) items[at] = make_int4(j, pk, __float_as_int(qj), 0);
            }
        }
    };
    // Spread the listed beads, q pre-multiplied by the scale S.
    auto spread = [&](float S) {
        const int a = lane % PT, b = lane / PT;
        const bool lane_on = lane < BPR * PT;
        const int ni = nitems;
        for (int it = warp; it < ni; it += NW) {
            const int4 rec = items[it];
            const int dx = (rec.y & 255) - PT, dy = ((rec.y >> 8) & 255) - PT, dz = (rec.y >> 16) - PT;
            const float w = lane < 3 * PT ? wb[(size_t)rec.x * (3 * PT) + lane] : 0.f;   // x, y, z taps
            const float wxq = __shfl_sync(FULL, w, a) * (__int_as_float(rec.z) * S);
            const int x = dx + a;
            const bool vx = lane_on && (unsigned)x < (unsigned)E;
            float wxy[NR];
            int i0[NR];
            bool v[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int bb = b + r * BPR;
                const float wy = __shfl_sync(FULL, w, PT + (bb < PT ? bb : PT - 1));
                const int y = dy + bb;
                v[r] = vx && bb < PT && (unsigned)y < (unsigned)E;
                wxy[r] = wxq * wy;
                i0[r] = (dz * E + y) * EP + x;
            }
            const int clo = max(0, -dz), chi = min(PT, E - dz);   // z taps inside the region
#pragma unroll
            for (int r = 0; r < NR; ++r) i0[r] += clo * E * EP;
            for (int c = clo; c < chi; ++c) {
                const float wzc = __shfl_sync(FULL, w, 2 * PT + c);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    if (v[r]) atomicAdd(&acc[i0[r]], __float2int_rn(wxy[r] * wzc));
                    i0[r] += E * EP;
                }
            }
        }
    };
    // the scale from the sum of |q| over the region's beads: in the listing pass
    // when all candidates fit one round, else from a pass of its own
    const bool one_round = total <= kScCap;
    float qs = 0.f;
    scan(0, total, one_round, qs);
#pragma unroll
    for (int of = 16; of > 0; of >>= 1) qs += __shfl_xor_sync(FULL, qs, of);
    if (lane == 0) wsum[warp] = qs;
    __syncthreads();
    float B = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) B += wsum[w];
    const float wm = g.wkf.wn;
    B *= wm * wm * wm;
    int ex = 0;
    frexpf(B, &ex);                                   // B < 2^ex
    const float S = B > 0.f ? ldexpf(1.f, min(126, 30 - ex)) : 1.f;   // S B < 2^30
    if (one_round) {
        spread(S);
    } else {
        for (int f0 = 0; f0 < total; f0 += kScCap) {
            __syncthreads();
            if (tid == 0) nitems = 0;
            __syncthreads();
            float dummy = 0.f;
            scan(f0, min(total, f0 + kScCap), true, dummy);
            __syncthreads();
            spread(S);
        }
    }
    __syncthreads();
    const float iS = 1.f / S;   // a power of two: exact
    constexpr int Q = E / 4;    // 16-byte pieces per row
    for (int e = tid; e < E * E * Q; e += kScThreads) {
        const int row = e / Q, cq = e - row * Q;
        const int z = row / E, y = row - z * E;
        const int4 v = *reinterpret_cast<const int4*>(acc + (z * E + y) * EP + 4 * cq);
        *reinterpret_cast<float4*>(grid + ((size_t)(oz + z) * n + (oy + y)) * n + ox + 4 * cq) =
            make_float4((float)v.x * iS, (float)v.y * iS, (float)v.z * iS, (float)v.w * iS);
    }
}

// ---------------------------------------------------------------------------
// a2, reduction form: a warp per charged bead adds its (2p)^3 products
// q w_x w_y w_z to the zeroed grid by global reductions, which the L2 executes;
// lanes over (x, y) taps (rows of 2p consecutive points), a loop over the z
// taps. No work on points outside a window, none repeated for neighbouring
// tiles, and in FP64 the additions do not run on the SM's FP64 units at all
// (one product per point does). Bound by the L2's reductions (~190 G sectors/s:
// groups of four points per reduction, half the instructions on 1.4x the
// sectors, took 44 against 34 us at 524k beads) and, at few beads, by latency.
// Stage alone against the forms it replaces as the automatic choice (tile form
// below n = 128, scatter form from there, slab form in FP64): FP32 3000 beads
// 16.3 -> 6.1 us, 24k 28.6 -> 8.2, 81k 20.5 -> 10.2, 192k 32.7 -> 16.3, 524k
// 57 -> 34, 3M 208 -> 190; FP64 3000 beads 61 -> 7.9, 375k 190 -> 52. The grid is
// cleared by the count kernel (up to 16 16- or 32-byte stores a thread) or, when
// it is large for its beads, by a memset beside the binning.
// ---------------------------------------------------------------------------
constexpr int kRedThreads = 256;

// PT = 2p fixed at compile time (unrolled), or 0: any 2p <= 16.
template <typename R, int PT>
__device__ __forceinline__ void k_spread_red_body(const Geo& g, const int* __restrict__ tstart,
                                                  const typename V4<R>::T* __restrict__ sq, const int* __restrict__ sb,
                                                  const R* __restrict__ wb, R* __restrict__ grid, Blk blk) {
    pdl_enter();
    constexpr int NW = kRedThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nq = tstart[g.ntiles], n = g.n, n2 = n * n, P2 = PT ? PT : 2 * g.p, p = P2 / 2;
    const int rpi = 32 / P2;                    // y taps per round of lanes
    const int nr = (P2 + rpi - 1) / rpi;        // rounds
    const int b0 = lane / P2, a = lane - b0 * P2;
    const bool on = b0 < rpi;
    for (int s = blk.id * NW + warp; s < nq; s += blk.n * NW) {
        const int pb = sb[s];
        const R* w = wb + (size_t)s * 3 * P2;
        const R wq = on ? sq[s].w * w[a] : (R)0;
        const R wzl = lane < P2 ? w[2 * P2 + lane] : (R)0;
        int x = (pb & 1023) - p + 1 + a;
        x = x < 0 ? x + n : (x >= n ? x - n : x);
        const int y0 = ((pb >> 10) & 1023) - p + 1;
        int z = ((pb >> 20) & 1023) - p + 1;
        z += z < 0 ? n : 0;
        auto column = [&](int b) {   // the z taps of the lane's column in row b
            const bool v = on && b < P2;
            int y = y0 + (v ? b : 0);
            y = y < 0 ? y + n : (y >= n ? y - n : y);
            const R wxy = v ? wq * w[P2 + b] : (R)0;
            R* col = grid + y * n + x;
            int zz = z;
#pragma unroll
            for (int c = 0; c < (PT ? PT : kMaxTaps); ++c) {
                if (!PT && c >= P2) break;
                const R wz = __shfl_sync(0xffffffffu, wzl, c);
                if (v && ENUF_GUARD(g.check, (unsigned)zz < (unsigned)n, 4)) atomicAdd(col + zz * n2, wxy * wz);
                zz = zz + 1 == n ? 0 : zz + 1;
            }
        };
        if constexpr (PT > 0) {
            constexpr int RPI = 32 / PT, NR = (PT + RPI - 1) / RPI;
#pragma unroll
            for (int r = 0; r < NR; ++r) column(b0 + r * RPI);
        } else {
            for (int r = 0; r < nr; ++r) column(b0 + r * rpi);
        }
    }
}

template <typename R, int PT>
__global__ void __launch_bounds__(kRedThreads) k_spread_red(Geo g, const int* __restrict__ tstart,
                                                            const typename V4<R>::T* __restrict__ sq,
                                                            const int* __restrict__ sb, const R* __restrict__ wb,
                                                            R* __restrict__ grid) {
    k_spread_red_body<R, PT>(g, tstart, sq, sb, wb, grid, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---------------------------------------------------------------------------
// a3: forward FFT pass along x (R2C, two real rows per complex line), keep
// k_x = 0..nc; output spec1[z][kx][y].
// ---------------------------------------------------------------------------
template <typename R, bool CR = false>
__global__ void __launch_bounds__(256) k_fft_x(Geo g, FftPlanDev fp, const R* __restrict__ grid,
                                              const typename Cx<R>::T* __restrict__ twg,
                                              typename Cx<R>::T* __restrict__ spec1, int LP) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc1 = g.nc + 1;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // padded, swizzled lines (the split reads across lines)
    C* b0 = tw + n;
    C* b1 = b0 + LP * ls;
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const float rn = 1.0f / (float)n;
    const int row0 = blockIdx.x * 2 * LP;     // first real row (z*n + y), y even
    const int nrows = n * n;
    const int nl = min(LP, (nrows - row0) / 2);
    const float rnl = 1.0f / (float)max(nl, 1);
    for (int idx = threadIdx.x; idx < nl * n; idx += blockDim.x) {
        const int c = qdiv(idx, n, rn), x = idx - c * n;
        C v;
        v.x = grid[(size_t)(row0 + 2 * c) * n + x];
        v.y = grid[(size_t)(row0 + 2 * c + 1) * n + x];
        b0[c * ls + swz<C>(x)] = v;
    }
    __syncthreads();
    C* res = fft_lines<R, false, CR>(b0, b1, tw, fp, nl, ls);
    // split the two real transforms: A = (Z_k + conj Z_{n-k})/2, B = -i (Z_k - conj Z_{n-k})/2
    for (int idx = threadIdx.x; idx < nl * nc1; idx += blockDim.x) {
        const int k = qdiv(idx, nl, rnl), c = idx - k * nl;
        const C z = res[c * ls + swz<C>(k)];
        const C zm = res[c * ls + swz<C>(k == 0 ? 0 : n - k)];
        C A, B;
        A.x = (R)0.5 * (z.x + zm.x);
        A.y = (R)0.5 * (z.y - zm.y);
        B.x = (R)0.5 * (z.y + zm.y);
        B.y = (R)0.5 * (zm.x - z.x);
        const int row = row0 + 2 * c;
        const int zz = qdiv(row, n, rn), y = row - zz * n;
        C* dst = spec1 + ((size_t)zz * nc1 + k) * n + y;
        dst[0] = A;
        dst[1] = B;
    }
}

// forward pass along y for lines (z, kx), keep |ky| <= nc; output spec2[kx][ky][z]
template <typename R, bool CR = false>
__global__ void __launch_bounds__(256) k_fft_y(Geo g, FftPlanDev fp, const typename Cx<R>::T* __restrict__ spec1,
                                              const typename Cx<R>::T* __restrict__ twg,
                                              typename Cx<R>::T* __restrict__ spec2, int LB) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc1 = g.nc + 1, K = g.K;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // padded, swizzled lines (the output reads across lines)
    C* b0 = tw + n;
    C* b1 = b0 + LB * ls;
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const float rn = 1.0f / (float)n;
    const int kx = blockIdx.x;
    const int z0 = blockIdx.y * LB;
    const int nl = min(LB, n - z0);
    const float rnl = 1.0f / (float)max(nl, 1);
    for (int idx = threadIdx.x; idx < nl * n; idx += blockDim.x) {
        const int c = qdiv(idx, n, rn), y = idx - c * n;
        b0[c * ls + swz<C>(y)] = spec1[((size_t)(z0 + c) * nc1 + kx) * n + y];
    }
    __syncthreads();
    C* res = fft_lines<R, false, CR>(b0, b1, tw, fp, nl, ls);
    for (int idx = threadIdx.x; idx < nl * K; idx += blockDim.x) {
        const int ki = qdiv(idx, nl, rnl), c = idx - ki * nl;
        const int ky = ki - g.nc;
        spec2[((size_t)kx * K + ki) * n + z0 + c] = res[c * ls + swz<C>(ky < 0 ? ky + n : ky)];
    }
}

// z pass: forward z; E += w D |F|^2, W += w D v |F|^2 (FP64, Kahan); the
// fields G = -i D F and kz G of Eq. 24 (the later passes take x and y as kx G
// and ky G; see spec3_array) or, in gradient mode, the one field G = D F; the
// CTA's lines of both inverse-transformed together; output spec3[a][z][kx][ky].
template <typename R, bool CR = false>
__global__ void __launch_bounds__(256) k_fft_z(Geo g, FftPlanDev fp, const typename Cx<R>::T* __restrict__ spec2,
                                              const typename Cx<R>::T* __restrict__ twg,
                                              const double* __restrict__ tab, const double* __restrict__ tabv,
                                              const R* __restrict__ tabr, typename Cx<R>::T* __restrict__ spec3,
                                              double* __restrict__ epart, int LB, int plane_major) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc = g.nc, K = g.K, nf = g.nf;
    const int NL = (nc + 1) * K;
    const float rK = 1.0f / (float)K, rn = 1.0f / (float)n;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // padded, swizzled lines (loads and stores go across lines)
    C* b0 = tw + n;               // [LB][ls] forward lines
    C* b1 = b0 + LB * ls;         // [LB][ls] scratch
    const int nz = nf == 3 ? 2 : 1;
    C* X = b1 + LB * ls;          // [nz][LB][ls] fields
    C* Y = X + nz * LB * ls;      // [nz][LB][ls] scratch
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const int l0 = blockIdx.x * LB;
    const int nl = min(LB, NL - l0);
    const float rnl = 1.0f / (float)max(nl, 1);
    if (plane_major) {   // spec2[z][l]: lines gathered across planes
        for (int idx = threadIdx.x; idx < nl * n; idx += blockDim.x) {
            const int z = qdiv(idx, nl, rnl), c = idx - z * nl;
            b0[c * ls + swz<C>(z)] = spec2[(size_t)z * NL + l0 + c];
        }
    } else {             // spec2[l][z]: lines contiguous
        for (int idx = threadIdx.x; idx < nl * n; idx += blockDim.x) {
            const int c = qdiv(idx, n, rn), z = idx - c * n;
            b0[c * ls + swz<C>(z)] = spec2[(size_t)l0 * n + idx];
        }
    }
    __syncthreads();
    C* Fh = fft_lines<R, false, CR>(b0, b1, tw, fp, nl, ls);
    // energy and virial of the kept modes (half space kx >= 0, kx > 0 counted twice)
    Kahan ke, kw;
    for (int idx = threadIdx.x; idx < nl * K; idx += blockDim.x) {
        const int c = qdiv(idx, K, rK), kzi = idx - c * K;
        const int l = l0 + c;
        const int kx = qdiv(l, K, rK);
        const int kz = kzi - nc;
        const C f = Fh[c * ls + swz<C>(kz < 0 ? kz + n : kz)];
        const double a2 = (double)f.x * (double)f.x + (double)f.y * (double)f.y;
        const double wgt = kx == 0 ? 1.0 : 2.0;
        ke.add(wgt * tab[(size_t)l * K + kzi] * a2);
        kw.add(wgt * tabv[(size_t)l * K + kzi] * a2);
    }
    double se = ke.s, sv = kw.s;
    block_sum2(se, sv);
    if (threadIdx.x == 0) {
        epart[2 * blockIdx.x] = se;
        epart[2 * blockIdx.x + 1] = sv;
    }
    // fields: line a * nl + c of X, only the half that the transform reads
    const bool half = fft_half(fp) >= 0;
    const int cnt = half ? n / 2 : n;
    const int hper = nl * cnt, per = nl * n;
    const float rhper = 1.0f / (float)max(hper, 1), rper = 1.0f / (float)max(per, 1), rcnt = 1.0f / (float)cnt;
    for (int idx = threadIdx.x; idx < nz * hper; idx += blockDim.x) {
        const int a = qdiv(idx, hper, rhper), e = idx - a * hper;
        const int c = qdiv(e, cnt, rcnt), i = e - c * cnt;
        const int m = half && i >= n / 4 ? i + n / 2 : i;
        const int kz = m <= n / 2 ? m : m - n;
        C v;
        v.x = (R)0;
        v.y = (R)0;
        if (kz >= -nc && kz <= nc) {
            const int l = l0 + c;
            const R d = tabr[(size_t)l * K + (kz + nc)];
            const C f = Fh[c * ls + swz<C>(m)];
            if (nf == 1) {
                v.x = d * f.x;     // D F
                v.y = d * f.y;
            } else {
                const R s = a == 0 ? d : (R)kz * d;
                v.x = s * f.y;     // -i D F, -i kz D F
                v.y = -s * f.x;
            }
        }
        X[(a * nl + c) * ls + swz<C>(m)] = v;
    }
    __syncthreads();
    C* res = fft_lines<R, true, CR, true>(X, Y, tw, fp, nz * nl, ls);
    for (int idx = threadIdx.x; idx < nz * per; idx += blockDim.x) {
        const int a = qdiv(idx, per, rper), e = idx - a * per;
        const int z = qdiv(e, nl, rnl), c = e - z * nl;
        spec3[((size_t)a * n + z) * NL + l0 + c] = res[(a * nl + c) * ls + swz<C>(z)];
    }
}

// Forward x and y passes of one z-plane in shared memory (small grids): the
// n real rows as n/2 complex lines (two rows each), FFT along x, split into
// the two half spectra kx = 0..nc, FFT of the nc + 1 columns along y, keep
// |ky| <= nc; output spec2[z][kx][ky] (plane-major).
template <typename R, bool CR = false>
__global__ void __launch_bounds__(512) k_fft_xy(Geo g, FftPlanDev fp, const R* __restrict__ grid,
                                               const typename Cx<R>::T* __restrict__ twg,
                                               typename Cx<R>::T* __restrict__ spec2) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc = g.nc, nc1 = nc + 1, K = g.K, h = n / 2;
    const float rn = 1.0f / (float)n, rh = 1.0f / (float)h, rK = 1.0f / (float)K;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // padded, swizzled lines
    C* L0 = tw + n;        // [n/2][ls]
    C* L1 = L0 + h * ls;   // [n/2][ls]
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const int z = blockIdx.x;
    const R* gz = grid + (size_t)z * n * n;
    for (int idx = threadIdx.x; idx < h * n; idx += blockDim.x) {
        const int c = qdiv(idx, n, rn), x = idx - c * n;
        C v;
        v.x = gz[(size_t)(2 * c) * n + x];
        v.y = gz[(size_t)(2 * c + 1) * n + x];
        L0[c * ls + swz<C>(x)] = v;
    }
    __syncthreads();
    C* X = fft_lines<R, false, CR>(L0, L1, tw, fp, h, ls);
    C* P = X == L0 ? L1 : L0;   // [nc+1][ls] columns over y, then scratch
    C* S = P + nc1 * ls;        // 2 (nc + 1) = n/2: P and S fill the other buffer
    // split the two real transforms: A = (Z_k + conj Z_{n-k})/2, B = -i (Z_k - conj Z_{n-k})/2
    for (int idx = threadIdx.x; idx < nc1 * h; idx += blockDim.x) {
        const int k = qdiv(idx, h, rh), c = idx - k * h;
        const C zk = X[c * ls + swz<C>(k)];
        const C zm = X[c * ls + swz<C>(k == 0 ? 0 : n - k)];
        C A, B;
        A.x = (R)0.5 * (zk.x + zm.x);
        A.y = (R)0.5 * (zk.y - zm.y);
        B.x = (R)0.5 * (zk.y + zm.y);
        B.y = (R)0.5 * (zm.x - zk.x);
        P[k * ls + swz<C>(2 * c)] = A;
        P[k * ls + swz<C>(2 * c + 1)] = B;
    }
    __syncthreads();
    C* Y = fft_lines<R, false, CR>(P, S, tw, fp, nc1, ls);
    C* out = spec2 + (size_t)z * nc1 * K;
    for (int idx = threadIdx.x; idx < nc1 * K; idx += blockDim.x) {
        const int kx = qdiv(idx, K, rK), ki = idx - kx * K;
        const int ky = ki - nc;
        out[idx] = Y[kx * ls + swz<C>(ky < 0 ? ky + n : ky)];
    }
}

// Inverse y and x passes of one (field, z-plane) in shared memory (small
// grids): the plane spec3[a][z][kx][ky], zero-padded to n along y, inverse
// FFT of the nc + 1 columns, then two Hermitian rows per complex line
// (C2R) inverse along x; output h[a][z][y][x].
template <typename R, bool CR = false>
__global__ void __launch_bounds__(512) k_fft_yx(Geo g, FftPlanDev fp, const typename Cx<R>::T* __restrict__ spec3,
                                               const typename Cx<R>::T* __restrict__ twg, R* __restrict__ h) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc = g.nc, nc1 = nc + 1, K = g.K, hn = n / 2;
    const float rn = 1.0f / (float)n;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // padded, swizzled lines
    C* L0 = tw + n;         // [n/2][ls]: the nc + 1 columns and their scratch
    C* L1 = L0 + hn * ls;   // [n/2][ls]: the x lines
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const int az = blockIdx.x;   // a * n + z
    const int a = qdiv(az, n, rn), z = az - a * n;
    const C* in = spec3 + ((size_t)spec3_array(g.nf, a) * n + z) * nc1 * K;
    C* P = L0;                   // [nc+1][ls] columns over y
    C* S = L0 + nc1 * ls;
    for (int idx = threadIdx.x; idx < nc1 * n; idx += blockDim.x) {
        const int kx = qdiv(idx, n, rn), m = idx - kx * n;
        const int ky = m <= n / 2 ? m : m - n;
        C v;
        v.x = (R)0;
        v.y = (R)0;
        if (ky >= -nc && ky <= nc) {
            v = in[kx * K + (ky + nc)];
            const R f = spec3_factor<R>(g.nf, a, kx, ky);
            v.x *= f;
            v.y *= f;
        }
        P[kx * ls + swz<C>(m)] = v;
    }
    __syncthreads();
    C* Yc = fft_lines<R, true, CR>(P, S, tw, fp, nc1, ls);   // [kx][y], in L0
    // x lines: row pair (2c, 2c+1) as A + i B with the Hermitian extension
    for (int idx = threadIdx.x; idx < hn * n; idx += blockDim.x) {
        const int c = qdiv(idx, n, rn), m = idx - c * n;
        C a, b;
        a.x = a.y = b.x = b.y = (R)0;
        if (m == 0) {
            a.x = Yc[swz<C>(2 * c)].x;
            b.x = Yc[swz<C>(2 * c + 1)].x;
        } else if (m <= nc) {
            a = Yc[m * ls + swz<C>(2 * c)];
            b = Yc[m * ls + swz<C>(2 * c + 1)];
        } else if (m >= n - nc) {
            a = Yc[(n - m) * ls + swz<C>(2 * c)];
            a.y = -a.y;
            b = Yc[(n - m) * ls + swz<C>(2 * c + 1)];
            b.y = -b.y;
        }
        C zz;
        zz.x = a.x - b.y;   // A + i B
        zz.y = a.y + b.x;
        L1[c * ls + swz<C>(m)] = zz;
    }
    __syncthreads();
    C* Xr = fft_lines<R, true, CR>(L1, L0, tw, fp, hn, ls);
    R* out = h + (size_t)az * n * n;
    for (int idx = threadIdx.x; idx < hn * n; idx += blockDim.x) {
        const int c = qdiv(idx, n, rn), x = idx - c * n;
        const C v = Xr[c * ls + swz<C>(x)];
        out[(size_t)(2 * c) * n + x] = v.x;
        out[(size_t)(2 * c + 1) * n + x] = v.y;
    }
}

// inverse pass along y for lines (a, z, kx): K inputs zero-padded to n; output spec4[a][z][y][kx]
template <typename R, bool CR = false>
__global__ void __launch_bounds__(256) k_fft_iy(Geo g, FftPlanDev fp, const typename Cx<R>::T* __restrict__ spec3,
                                               const typename Cx<R>::T* __restrict__ twg,
                                               typename Cx<R>::T* __restrict__ spec4, int LB) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc = g.nc, nc1 = nc + 1, K = g.K;
    const int NLT = g.nf * n * nc1;
    const float rnc1 = 1.0f / (float)nc1;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // padded, swizzled lines (the output reads across lines)
    C* b0 = tw + n;
    C* b1 = b0 + LB * ls;
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const float rn = 1.0f / (float)n;
    // the wave numbers as R: a conversion per element would cost the FP64 pipe as
    // much as an addition
    R* kr = reinterpret_cast<R*>(b1 + LB * ls);
    for (int t = threadIdx.x; t < nc1; t += blockDim.x) kr[t] = (R)t;
    __syncthreads();
    const int l0 = blockIdx.x * LB;
    const int nl = min(LB, NLT - l0);
    const float rnl = 1.0f / (float)max(nl, 1);
    const bool half = fft_half(fp) >= 0;
    const int cnt = half ? n / 2 : n;   // the half that the transform reads
    const float rcnt = 1.0f / (float)cnt;
    for (int idx = threadIdx.x; idx < nl * cnt; idx += blockDim.x) {
        const int c = qdiv(idx, cnt, rcnt), i = idx - c * cnt;
        const int m = half && i >= n / 4 ? i + n / 2 : i;
        const int ky = m <= n / 2 ? m : m - n;
        C v;
        v.x = (R)0;
        v.y = (R)0;
        if (ky >= -nc && ky <= nc) {
            const int l = l0 + c, az = qdiv(l, nc1, rnc1), kx = l - az * nc1;
            const int a = az >= 2 * n ? 2 : (az >= n ? 1 : 0);
            v = spec3[(size_t)(l - (a - spec3_array(g.nf, a)) * n * nc1) * K + (ky + nc)];
            if (g.nf == 3 && a < 2) {
                const R f = kr[a == 0 ? kx : abs(ky)];
                v.x *= f;
                v.y *= f;
                if (a == 1 && ky < 0) {
                    v.x = -v.x;
                    v.y = -v.y;
                }
            }
        }
        b0[c * ls + swz<C>(m)] = v;
    }
    __syncthreads();
    C* res = fft_lines<R, true, CR, true>(b0, b1, tw, fp, nl, ls);
    for (int idx = threadIdx.x; idx < nl * n; idx += blockDim.x) {
        const int y = qdiv(idx, nl, rnl), c = idx - y * nl;
        const int l = l0 + c;
        const int az = qdiv(l, nc1, rnc1), kx = l - az * nc1;
        spec4[((size_t)az * n + y) * nc1 + kx] = res[c * ls + swz<C>(y)];
    }
}

// inverse pass along x (C2R, two Hermitian rows per complex line); output h[a][z][y][x]
template <typename R, bool CR = false>
__global__ void __launch_bounds__(256) k_fft_ix(Geo g, FftPlanDev fp, const typename Cx<R>::T* __restrict__ spec4,
                                               const typename Cx<R>::T* __restrict__ twg,
                                               R* __restrict__ h, int LP) {
    pdl_enter();
    using C = typename Cx<R>::T;
    extern __shared__ unsigned char smraw[];
    const int n = g.n, nc = g.nc, nc1 = nc + 1;
    const int nrows = g.nf * n * n;
    C* tw = reinterpret_cast<C*>(smraw);
    const int ls = line_stride<C>(n);   // swizzled lines
    C* b0 = tw + n;
    C* b1 = b0 + LP * ls;
    for (int t = threadIdx.x; t < n; t += blockDim.x) tw[t] = twg[t];
    const float rn = 1.0f / (float)n;
    const int row0 = blockIdx.x * 2 * LP;
    const int nl = min(LP, (nrows - row0) / 2);
    const float rnl = 1.0f / (float)max(nl, 1);
    const bool half = fft_half(fp) >= 0;
    const int cnt = half ? n / 2 : n;   // the half that the transform reads
    const float rcnt = 1.0f / (float)cnt;
    for (int idx = threadIdx.x; idx < nl * cnt; idx += blockDim.x) {
        const int c = qdiv(idx, cnt, rcnt), i = idx - c * cnt;
        const int m = half && i >= n / 4 ? i + n / 2 : i;
        const C* A = spec4 + (size_t)(row0 + 2 * c) * nc1;
        const C* B = A + nc1;
        C a, b;
        a.x = a.y = b.x = b.y = (R)0;
        if (m == 0) {
            a.x = A[0].x;
            b.x = B[0].x;
        } else if (m <= nc) {
            a = A[m];
            b = B[m];
        } else if (m >= n - nc) {
            a = A[n - m];
            a.y = -a.y;
            b = B[n - m];
            b.y = -b.y;
        }
        C z;
        z.x = a.x - b.y;   // A + i B
        z.y = a.y + b.x;
        b0[c * ls + swz<C>(m)] = z;
    }
    __syncthreads();
    C* res = fft_lines<R, true, CR, true>(b0, b1, tw, fp, nl, ls);
    for (int idx = threadIdx.x; idx < nl * n; idx += blockDim.x) {
        const int c = qdiv(idx, n, rn), x = idx - c * n;
        const C v = res[c * ls + swz<C>(x)];
        h[(size_t)(row0 + 2 * c) * n + x] = v.x;
        h[(size_t)(row0 + 2 * c + 1) * n + x] = v.y;
    }
}

// ---------------------------------------------------------------------------
// a6: gather (conjugated NFFT part 2, Eq. 25). Warp per charged bead.
// ---------------------------------------------------------------------------
constexpr int kGatherThreads = 256;

// PT > 0: the window's tap count 2p fixed at compile time. The tap loops are
// then unrolled: the z taps' offsets and weights sit in registers and the
// 3 x 2p loads of a column are all in flight at once (the runtime-count loop
// waits on each tap's loads before the next: at 3M beads the gather was
// bound by that latency, not by DRAM).
template <typename R, int PT = 0>
__device__ __forceinline__ void k_gather_body(Geo g, const int* __restrict__ tstart,
                                                           const typename V4<R>::T* __restrict__ sq,
                                                           const typename V4<R>::T* __restrict__ sw,
                                                           const int* __restrict__ sb, const R* __restrict__ wb,
                                                           const R* __restrict__ h, R* __restrict__ F,
                                                           TotalsArgs tot, Blk blk) {
    pdl_enter();
    // with totals the launch has one more block, the first, which reduces the
    // energies while the others gather (their partials are all written by then)
    if (tot.Edev) {
        if (blk.id == 0) {
            totals_block(g, tot);
            return;
        }
        blk.id -= 1;
        blk.n -= 1;
    }
    constexpr int NW = kGatherThreads / 32;
    __shared__ R wts[NW][3][kMaxTaps];
    __shared__ R dwts[NW][3][kMaxTaps];   // gradient mode: psi'(d) = -(2 d / b) psi(d)
    __shared__ int lix[NW][3][kMaxTaps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Nq = tstart[g.ntiles];
    const int n = g.n;
    const size_t n3 = (size_t)n * n * n;   // n <= 1024: one grid's offsets fit an int
    const R* __restrict__ h0 = h;
    const R* __restrict__ h1 = g.nf == 3 ? h + n3 : h;
    const R* __restrict__ h2 = g.nf == 3 ? h + 2 * n3 : h;
    const int P2 = 2 * g.p;
    const float iP2 = 1.0f / (float)P2;
    const R rb = win_k(g, (R)0).rb, wn = win_k(g, (R)0).wn;
    const R pref = win_k(g, (R)0).pref;
    const bool grad = g.nf == 1;
    // the whole grid sweeps the tile-sorted beads in order (bead s by warp s mod
    // the grid's warps): the fields' working set at any moment is a band of
    // neighbouring tiles, which stays in L2 (measured: giving each block a
    // contiguous run instead spread the working set over the whole grid and
    // read 2.4x the DRAM bytes at 3M beads)
    for (int s = blk.id * NW + warp; s < Nq; s += blk.n * NW) {
        const typename V4<R>::T wv = sw[s];
        const R qs = sq[s].w;
        const int pb = sb[s];
        if (lane < P2) {
            const int base[3] = {pb & 1023, (pb >> 10) & 1023, (pb >> 20) & 1023};
            const R fr[3] = {wv.x, wv.y, wv.z};
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                int l = base[t] - g.p + 1 + lane;
                l = l < 0 ? l + n : (l >= n ? l - n : l);
                lix[warp][t][lane] = t == 2 ? l * n * n : l;
                const R d = fr[t] + (R)(g.p - 1 - lane);   // n x - l
                const R w = wb ? wb[(size_t)s * 3 * P2 + t * P2 + lane] : wn * r_exp(-d * d * rb);
                wts[warp][t][lane] = w;
                if (grad) dwts[warp][t][lane] = (R)-2 * d * rb * w;
            }
        }
        __syncwarp();
        R ax = 0, ay = 0, az = 0;
        // lanes over the (x, y) taps, the z taps summed first and weighted by
        // the column's x-y weight once; ab -> (a, b) by a float reciprocal
        // (ab < 256, so the quotient of ab + 1/2 is 1/32 from an integer)
        if constexpr (PT > 0) {
            constexpr int NAB = PT * PT;
            constexpr int NRD = (NAB + 31) / 32;   // rounds of lanes over the (x, y) taps
            R wz[PT], dz[PT];
            int oz[PT];
#pragma unroll
            for (int c = 0; c < PT; ++c) {
                wz[c] = wts[warp][2][c];
                dz[c] = grad ? dwts[warp][2][c] : (R)0;
                oz[c] = lix[warp][2][c];
            }
            if (sizeof(R) == 4 && g.h4) {
                // interleaved fields: a point's three values by one 16-byte load, a round's
                // 2p loads issued before the sums (planar fields cost three loads of 32-byte
                // rows each: twice the L1 lookups)
                const float4* __restrict__ h4 = reinterpret_cast<const float4*>(h);
#pragma unroll
                for (int r = 0; r < NRD; ++r) {
                    const int ab = lane + 32 * r;
                    const bool on = NAB % 32 == 0 || ab < NAB;
                    const int b = on ? ab / PT : 0, a = on ? ab - b * PT : 0;
                    const int rowo = lix[warp][1][b] * n + lix[warp][0][a];
                    float4 v[PT];
#pragma unroll
                    for (int c = 0; c < PT; ++c) {
                        int off = oz[c] + rowo;
                        if (!ENUF_GUARD(g.check, (size_t)off < n3, 5)) off = 0;
                        v[c] = h4[off];
                    }
                    R s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
                    for (int c = 0; c < PT; ++c) {
                        s0 = fma(wz[c], (R)v[c].x, s0);
                        s1 = fma(wz[c], (R)v[c].y, s1);
                        s2 = fma(wz[c], (R)v[c].z, s2);
                    }
                    const R wab = on ? wts[warp][0][a] * wts[warp][1][b] : (R)0;
                    ax = fma(wab, s0, ax);
                    ay = fma(wab, s1, ay);
                    az = fma(wab, s2, az);
                }
            } else {
#pragma unroll
                for (int r = 0; r < NRD; ++r) {
                    const int ab = lane + 32 * r;
                    if (NAB % 32 != 0 && ab >= NAB) break;
                    const int b = ab / PT, a = ab - b * PT;
                    const int rowo = lix[warp][1][b] * n + lix[warp][0][a];
                    const R wx = wts[warp][0][a], wy = wts[warp][1][b];
                    if (grad) {   // one field: sum_l grad Psi(n x - l) h(l)
                        R hv[PT];
#pragma unroll
                        for (int c = 0; c < PT; ++c) {
                            const int off = oz[c] + rowo;
                            hv[c] = ENUF_GUARD(g.check, (size_t)off < n3, 5) ? h0[off] : (R)0;
                        }
                        R s0 = 0, s1 = 0;
#pragma unroll
                        for (int c = 0; c < PT; ++c) {
                            s0 = fma(wz[c], hv[c], s0);
                            s1 = fma(dz[c], hv[c], s1);
                        }
                        ax = fma(dwts[warp][0][a] * wy, s0, ax);
                        ay = fma(wx * dwts[warp][1][b], s0, ay);
                        az = fma(wx * wy, s1, az);
                    } else {
                        R h0v[PT], h1v[PT], h2v[PT];
#pragma unroll
                        for (int c = 0; c < PT; ++c) {
                            int off = oz[c] + rowo;
                            if (!ENUF_GUARD(g.check, (size_t)off < n3, 5)) off = 0;
                            h0v[c] = h0[off];
                            h1v[c] = h1[off];
                            h2v[c] = h2[off];
                        }
                        R s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
                        for (int c = 0; c < PT; ++c) {
                            s0 = fma(wz[c], h0v[c], s0);
                            s1 = fma(wz[c], h1v[c], s1);
                            s2 = fma(wz[c], h2v[c], s2);
                        }
                        const R wab = wx * wy;
                        ax = fma(wab, s0, ax);
                        ay = fma(wab, s1, ay);
                        az = fma(wab, s2, az);
                    }
                }
            }
        } else if (grad) {   // one field: sum_l grad Psi(n x - l) h(l)
            for (int ab = lane; ab < P2 * P2; ab += 32) {
                const int b = (int)(((float)ab + 0.5f) * iP2);
                const int a = ab - b * P2;
                const int rowo = lix[warp][1][b] * n + lix[warp][0][a];
                R s0 = 0, s1 = 0;   // sum_z psi h, sum_z psi' h
                for (int c = 0; c < P2; ++c) {
                    const int off = lix[warp][2][c] + rowo;
                    if (!ENUF_GUARD(g.check, (size_t)off < n3, 5)) continue;
                    const R hv = h0[off];
                    s0 = fma(wts[warp][2][c], hv, s0);
                    s1 = fma(dwts[warp][2][c], hv, s1);
                }
                const R wx = wts[warp][0][a], wy = wts[warp][1][b];
                ax = fma(dwts[warp][0][a] * wy, s0, ax);
                ay = fma(wx * dwts[warp][1][b], s0, ay);
                az = fma(wx * wy, s1, az);
            }
        } else {
            for (int ab = lane; ab < P2 * P2; ab += 32) {
                const int b = (int)(((float)ab + 0.5f) * iP2);
                const int a = ab - b * P2;
                const int rowo = lix[warp][1][b] * n + lix[warp][0][a];
                R s0 = 0, s1 = 0, s2 = 0;   // sum_z psi h_a
                for (int c = 0; c < P2; ++c) {
                    const R w = wts[warp][2][c];
                    const int off = lix[warp][2][c] + rowo;   // z index pre-scaled by n^2
                    if (!ENUF_GUARD(g.check, (size_t)off < n3, 5)) continue;
                    if (sizeof(R) == 4 && g.h4) {
                        const float4 v = reinterpret_cast<const float4*>(h)[off];
                        s0 = fma(w, (R)v.x, s0);
                        s1 = fma(w, (R)v.y, s1);
                        s2 = fma(w, (R)v.z, s2);
                        continue;
                    }
                    s0 = fma(w, h0[off], s0);
                    s1 = fma(w, h1[off], s1);
                    s2 = fma(w, h2[off], s2);
                }
                const R wab = wts[warp][0][a] * wts[warp][1][b];
                ax = fma(wab, s0, ax);
                ay = fma(wab, s1, ay);
                az = fma(wab, s2, az);
            }
        }
        if constexpr (sizeof(R) == 8) {   // each lane's share as a global reduction (a warp
            const int i = real_as_int(wv.w);   // sum would run 15 adds on the FP64 units)
            const R f = pref * qs;
            atomicAdd(&F[3 * i], f * ax);
            atomicAdd(&F[3 * i + 1], f * ay);
            atomicAdd(&F[3 * i + 2], f * az);
        } else {
        ax = warp_sum_r(ax);
        ay = warp_sum_r(ay);
        az = warp_sum_r(az);
        if (lane < 3) {   // a reduction each: nothing waits for F's old value
            const R f = pref * qs * (lane == 0 ? ax : (lane == 1 ? ay : az));
            atomicAdd(&F[3 * real_as_int(wv.w) + lane], f);
        }
        }
        __syncwarp();
    }
}

// Four CTAs per SM: the launch's 4 x 152 blocks are one wave (FP32 windows up
// to 8 taps, one round's loads in flight per lane; both rounds' took 88 registers,
// two CTAs per SM and a second wave). Whole calls with that and with F by
// reductions: 1M beads at p = 2 380 -> 361 us, 150,000 at p = 6 154 -> 147, 3000
// at p = 2 34.6 -> 33.4, 60,000 with a quarter charged in FP64 328 -> 317; the
// others within 1%.
template <typename R, int PT>
constexpr int gather_ctas() { return sizeof(R) == 4 && PT > 0 && PT <= 8 ? 4 : 2; }
template <typename R, int PT = 0>
__global__ void __launch_bounds__(kGatherThreads, gather_ctas<R, PT>()) k_gather(Geo g, const int* __restrict__ tstart,
                                                           const typename V4<R>::T* __restrict__ sq,
                                                           const typename V4<R>::T* __restrict__ sw,
                                                           const int* __restrict__ sb, const R* __restrict__ wb,
                                                           const R* __restrict__ h, R* __restrict__ F,
                                                           TotalsArgs tot) {
    k_gather_body<R, PT>(g, tstart, sq, sw, sb, wb, h, F, tot, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---------------------------------------------------------------------------
// a7 (electrostatic part): real-space erfc + Slater-correction pairs on the
// tile bins (Eq. 31, corrected Eq. 32, Eq. 27-28).
//
// S lanes per charged bead (S a power of 2, chosen per launch), 32 / S
// consecutive beads of the sorted order per warp. The tiles around a bead's
// tile form one contiguous run of sorted beads per (y, z) row of tiles; the
// bead's lanes walk the runs and read the candidates straight from the sorted
// array (the lanes of beads of one tile read the same lines). What passes the
// cutoff test goes to shared memory:
//   FP32: each lane notes its candidates in a list of its own (one predicated
//     store, no ballot); the lists are evaluated in step, each lane adding
//     into its own registers, and the S shares of a bead are summed once.
//     Issue-bound.
//   FP64: pairs of all the warp's beads go to one ring and are evaluated on
//     full warps, each pair once, because every FP64 instruction costs the
//     whole warp's 16 cycles of the SM's few FP64 units; +f and -f go out by
//     global reductions.
// The form before it staged the 27-tile halo of every tile in shared memory
// (27 staged beads per central bead at 3M beads, and as many CTAs as tiles:
// 8 for a 3000-bead box). Alone: FP32 3M beads 473 -> 229 us, 524k 94 -> 67,
// 192k 85 -> 51, 24k 62 -> 22; FP64 375k 264 -> 156, 3000 beads 49 -> 18 us (375k 92
// alone with more lanes per bead, before the plan's present real_lanes).
// ---------------------------------------------------------------------------
constexpr int kRealThreads = 256;
constexpr int kRealQ = 32;      // FP32: noted candidates per lane
constexpr int kRealU = 4;       // candidates per lane and iteration (loads in flight)
constexpr int kRealRing = 256;  // FP64: pair ring per warp (>= 31 + 32 kRealU, a power of 2)
static_assert(kRealRing >= 31 + 32 * kRealU && (kRealRing & (kRealRing - 1)) == 0, "pair ring");
template <typename R>
constexpr int real_smem_bytes() {
    return sizeof(R) == 8 ? (kRealThreads / 32) * kRealRing * (int)sizeof(int2)
                          : kRealThreads * kRealQ * (int)sizeof(int);
}

// Kernel table: per interval [j h, (j + 1) h] of [0, r_c] the power-basis
// coefficients c_0..c_5 of the quintic Hermite interpolant of J in t = r/h - j
// (J, J', J'' matched at both ends); kKtStride64 / kKtStride32 values per
// interval (16-byte aligned rows: 6 doubles, or 6 floats padded to 8).
template <typename R>
__device__ __forceinline__ void kt_load(const R* __restrict__ kt, int j, R (&c)[6]) {
    if constexpr (sizeof(R) == 8) {
        const double2* a = reinterpret_cast<const double2*>(kt + kKtStride64 * j);
        const double2 a0 = __ldg(a), a1 = __ldg(a + 1), a2 = __ldg(a + 2);
        c[0] = a0.x; c[1] = a0.y; c[2] = a1.x; c[3] = a1.y; c[4] = a2.x; c[5] = a2.y;
    } else {
        const float4* a = reinterpret_cast<const float4*>(kt + kKtStride32 * j);
        const float4 a0 = __ldg(a), a1 = __ldg(a + 1);
        c[0] = a0.x; c[1] = a0.y; c[2] = a0.z; c[3] = a0.w; c[4] = a1.x; c[5] = a1.y;
    }
}

// Pair energy u(r) and radial force f(r) = -du/dr of the real-space sum,
// u = J(r)/r with J = erfc(alpha r) - (1 + beta r) e^{-2 beta r} (the
// Slater correction, beta > 0), or with the Slater form factor in k space
// J = B1 - I. With a table (kt != null: FP64, and the k-space form factor)
// J and dJ/dt come from one Horner pass over the interval's coefficients and
// f = (J - J' r)/r^2; otherwise erfc and exp are evaluated directly.
template <typename R>
__device__ __forceinline__ void real_pair(R r2, R al, R c2a, R be, bool slater, R& u, R& fr_over_r, R& f_r,
                                          const R* __restrict__ kt = nullptr, int kn = 0, R kinv = 0) {
    const R ir = r_rsqrt(r2);
    const R r = r2 * ir;
    if (kt) {
        const R x = r * kinv;
        int j = (int)x;
        j = j >= kn ? kn - 1 : j;   // x >= 0
        const R t = x - (R)j;
        R c[6];
        kt_load<R>(kt, j, c);
        R d = c[5];
        R p = fma(c[5], t, c[4]);
#pragma unroll
        for (int k = 3; k >= 0; --k) {
            d = fma(d, t, p);
            p = fma(p, t, c[k]);
        }
        // J = p, J' r = (dJ/dt) (1/h) r = d x
        const R ff = fma(-d, x, p) * ir * ir;
        u = p * ir;
        fr_over_r = ff * ir;
        f_r = ff * r;
        return;
    }
    const R ar = al * r;
    const R ec = r_erfc(ar);
    R uu = ec * ir;
    R ff = ec * ir * ir + c2a * r_exp(-ar * ar) * ir;
    if (slater) {
        const R br = be * r;
        const R e2 = r_exp((R)-2 * br);
        uu -= ((R)1 + br) * e2 * ir;
        ff -= ((R)1 + (R)2 * br + (R)2 * br * br) * e2 * ir * ir;
    }
    u = uu;
    fr_over_r = ff * ir;   // multiplies the displacement vector
    f_r = ff * r;          // virial term r f(r)
}

template <typename R> __host__ __device__ constexpr bool real_half() { return sizeof(R) == 8; }

// A lane's sums: the force on its bead (FP32), energy and virial.
template <typename R>
struct RealSum {
    R fx, fy, fz, e, w;
};

// FP32: the pairs (bead pi, noted candidate k of this lane, k < cnt), all lanes in step.
__device__ __forceinline__ void real_drain(const Geo& g, const float4& pi, const int* list, int cnt,
                                           const float4* __restrict__ sq, RealSum<float>& a) {
    const RealK<float>& c = g.rkf;
    const int m = __reduce_max_sync(0xffffffffu, cnt);
    for (int k = 0; k < m; ++k) {
        if (k >= cnt) continue;
        const float4 pj = sq[list[32 * k]];
        const float dx = min_image(pi.x, pj.x, c.L, c.hL);
        const float dy = min_image(pi.y, pj.y, c.L, c.hL);
        const float dz = min_image(pi.z, pj.z, c.L, c.hL);
        float u, fo, fr;
        real_pair<float>(dist2(dx, dy, dz), c.al, c.c2a, c.be, g.slater != 0, u, fo, fr,
                         static_cast<const float*>(g.ktab), g.kn, c.kinv);
        const float qq = c.kap * pi.w * pj.w;
        a.fx += qq * fo * dx;
        a.fy += qq * fo * dy;
        a.fz += qq * fo * dz;
        a.e += 0.5f * qq * u;   // energy and virial per pair and direction
        a.w += 0.5f * qq * fr;
    }
}

// FP64: ring entries (bead i, candidate j) with the image in their upper bits
// (5 bits, 9 z + 3 y + x of 0: -L, 1: none, 2: +L), one per lane. ALL: the
// displacement is the minimum image instead.
__device__ __forceinline__ int2 real_entry(int i, int j, int image) {
    return make_int2(i | (image & 7) << 29, j | (image >> 3) << 29);
}
template <bool ALL>
__device__ __forceinline__ void real_ring(const Geo& g, const int2 e, const double4_32a* __restrict__ sq,
                                          const double4_32a* __restrict__ sw, double* __restrict__ F,
                                          RealSum<double>& a) {
    const RealK<double>& c = g.rkd;
    const int i = e.x & 0x1fffffff, j = e.y & 0x1fffffff;
    const double4_32a pi = sq[i], pj = sq[j];
    double dx, dy, dz;
    if constexpr (ALL) {
        dx = min_image(pi.x, pj.x, c.L, c.hL);
        dy = min_image(pi.y, pj.y, c.L, c.hL);
        dz = min_image(pi.z, pj.z, c.L, c.hL);
    } else {
        dx = pi.x - pj.x;
        dy = pi.y - pj.y;
        dz = pi.z - pj.z;
        const int im = (int)((unsigned)e.x >> 29 | ((unsigned)e.y >> 29) << 3);
        if (im != 13) {   // across a box face
            const int iz = im / 9, iy = (im - 9 * iz) / 3, ix = im % 3;
            if (ix != 1) dx += ix ? c.L : -c.L;
            if (iy != 1) dy += iy ? c.L : -c.L;
            if (iz != 1) dz += iz ? c.L : -c.L;
        }
    }
    const double r2 = dist2(dx, dy, dz);
    if (!(r2 < c.rc2 && r2 > 0.0)) return;
    double u, fo, fr;
    real_pair<double>(r2, c.al, c.c2a, c.be, g.slater != 0, u, fo, fr, static_cast<const double*>(g.ktab), g.kn, c.kinv);
    const double qq = c.kap * pi.w * pj.w;
    const double gf = qq * fo;
    const double gx = gf * dx, gy = gf * dy, gz = gf * dz;
    double* Fi = F + 3 * (size_t)real_as_int(sw[i].w);
    double* Fj = F + 3 * (size_t)real_as_int(sw[j].w);
    atomicAdd(Fi, gx);
    atomicAdd(Fi + 1, gy);
    atomicAdd(Fi + 2, gz);
    atomicAdd(Fj, -gx);
    atomicAdd(Fj + 1, -gy);
    atomicAdd(Fj + 2, -gz);
    a.e = fma(qq, u, a.e);
    a.w = fma(qq, fr, a.w);
}

// Beads of this block's share. ALL: the stencil covers whole rows of tiles
// (few tiles per dimension), every tile is visited once and displacements
// take the minimum image; else the rows and the x run are wrapped tile by
// tile, and a run's image shift is one constant (the displacement within r_c
// is the one of that image: r_c <= rs tiles, 2 rs + 1 <= tiles per dimension).
template <typename R, bool ALL>
__device__ __forceinline__ void real_sweep(const Geo& g, int nq, int S, const int* __restrict__ tstart,
                                           const typename V4<R>::T* __restrict__ sq,
                                           const typename V4<R>::T* __restrict__ sw, const int* __restrict__ sb,
                                           const float4* __restrict__ spf, int* list, int2* ring,
                                           R* __restrict__ F, RealSum<R>& a, Blk blk) {
    using V = typename V4<R>::T;
    constexpr bool HALF = real_half<R>();
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int NW = kRealThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gpw = 32 / S, sub = lane & (S - 1), grp = lane / S;
    // constants formed on the host: a conversion from double is an instruction on
    // the part's few FP64 units (16 cycles of them per warp), as is every double
    // operation of an FP32 kernel
    const float Lf = g.rkf.L, hLf = g.rkf.hL;
    // FP64: candidates above a band that covers the float error are out, the rest
    // are decided in double
    const float r2hi = HALF ? g.r2hi : g.rkf.rc2;
    const float rT = 1.0f / (float)g.T;
    const int ntd = g.ntd, rs = g.rs;
    int cnt = 0, head = 0;   // noted candidates of this lane (FP32); ring fill and head (FP64)
    for (int s0 = (blk.id * NW + warp) * gpw; s0 < nq; s0 += blk.n * NW * gpw) {
        const int s = s0 + grp;
        const bool own = s < nq;
        float4 pf;
        int tx = 0, ty = 0, tz = 0;
        if (own) {
            pf = spf[s];
            const int pb = sb[s];   // grid base of the bead: its tile
            tx = tile_of(pb & 1023, rT);
            ty = tile_of((pb >> 10) & 1023, rT);
            tz = tile_of((pb >> 20) & 1023, rT);
        }
        a.fx = a.fy = a.fz = (R)0;
        // rows of tiles one after the other (uniform over the warp), each as its run
        // inside the box and its run across the box face (if any bead of the warp
        // has one), as long as the warp's longest; one more turn empties the lists
        const int dz0 = ALL ? 0 : (HALF ? 0 : -rs), dz1 = ALL ? ntd - 1 : rs;
        const int dy0 = ALL ? 0 : -rs, dy1 = ALL ? ntd - 1 : rs;
        int dz = dz0, dy = HALF && !ALL ? 0 : dy0;
        bool across = false;   // uniform: the row's part across the box face
        int w0 = 0, wl = 0;
        float hx = 0.0f, hy = 0.0f, hz = 0.0f;
        while (true) {
            const bool last = dz > dz1;
            int j0 = 0, len = 0;
            if (across) {
                j0 = w0;
                len = wl;
            } else if (!last) {
                int zz = dz, yy = dy;
                hx = hy = hz = 0.0f;
                if (!ALL) {
                    zz += tz;
                    yy += ty;
                    if (zz < 0) { zz += ntd; hz = Lf; } else if (zz >= ntd) { zz -= ntd; hz = -Lf; }
                    if (yy < 0) { yy += ntd; hy = Lf; } else if (yy >= ntd) { yy -= ntd; hy = -Lf; }
                }
                const int* ts = tstart + (zz * ntd + yy) * ntd;
                // FP64, each pair once: the rows after the bead's own, and in its own
                // row the beads after it
                const bool home = HALF && !ALL && dz == 0 && dy == 0;
                const int xa = ALL ? 0 : (home ? tx : tx - rs), xb = ALL ? ntd - 1 : tx + rs;
                wl = 0;
                if (own) {
                    j0 = ts[max(xa, 0)];
                    if (HALF && (home || ALL)) j0 = max(j0, s + 1);
                    len = max(0, ts[min(xb, ntd - 1) + 1] - j0);
                    if (!ALL && (xa < 0 || xb >= ntd)) {
                        w0 = ts[xa < 0 ? xa + ntd : 0];
                        wl = ts[xa < 0 ? ntd : xb - ntd + 1] - w0;
                    }
                }
            }
            const int mlen = __reduce_max_sync(FULL, len);
            const int image = (hz > 0.0f ? 18 : (hz < 0.0f ? 0 : 9)) + (hy > 0.0f ? 6 : (hy < 0.0f ? 0 : 3)) +
                              (hx > 0.0f ? 2 : (hx < 0.0f ? 0 : 1));
            for (int t0 = 0;;) {
                if constexpr (HALF) {
                    while (cnt >= 32) {
                        __syncwarp();
                        real_ring<ALL>(g, ring[(head + lane) & (kRealRing - 1)], sq, sw, F, a);
                        __syncwarp();
                        head += 32;
                        cnt -= 32;
                    }
                } else {
                    if (last || __any_sync(FULL, cnt > kRealQ - kRealU)) {
                        real_drain(g, pf, list, cnt, sq, a);
                        cnt = 0;
                    }
                }
                if (t0 >= mlen) break;
                float4 b[kRealU];
#pragma unroll
                for (int u = 0; u < kRealU; ++u) {
                    const int t = t0 + u * S + sub;
                    if (t < len) b[u] = spf[j0 + t];
                }
#pragma unroll
                for (int u = 0; u < kRealU; ++u) {
                    const int t = t0 + u * S + sub;
                    bool hit = false;
                    if (t < len) {
                        float ex, ey, ez;
                        if (ALL) {
                            ex = min_image(pf.x, b[u].x, Lf, hLf);
                            ey = min_image(pf.y, b[u].y, Lf, hLf);
                            ez = min_image(pf.z, b[u].z, Lf, hLf);
                        } else {
                            ex = __fadd_rn(__fsub_rn(pf.x, b[u].x), hx);
                            ey = __fadd_rn(__fsub_rn(pf.y, b[u].y), hy);
                            ez = __fadd_rn(__fsub_rn(pf.z, b[u].z), hz);
                        }
                        const float r2 = dist2(ex, ey, ez);
                        // FP64 decides exactly in the ring; FP32: the bead itself is at r2 = 0
                        hit = HALF ? r2 <= r2hi : (r2 < r2hi && r2 > 0.0f);
                    }
                    if constexpr (HALF) {
                        const unsigned m = __ballot_sync(FULL, hit);
                        const int at = cnt + __popc(m & ((1u << lane) - 1u));
                        if (hit && ENUF_GUARD(g.check, at < kRealRing, 7))
                            ring[(head + at) & (kRealRing - 1)] = real_entry(s, j0 + t, image);
                        cnt += __popc(m);
                    } else if (hit && ENUF_GUARD(g.check, cnt < kRealQ, 7)) {
                        list[32 * cnt] = j0 + t;
                        ++cnt;
                    }
                }
                t0 += kRealU * S;
            }
            if (last) break;
            if (!ALL && !across && __any_sync(FULL, wl > 0)) {
                across = true;
                hx = tx - rs < 0 ? Lf : -Lf;   // read by the lanes with wl > 0
                continue;
            }
            across = false;
            if (++dy > dy1) {
                dy = dy0;
                ++dz;
            }
        }
        if constexpr (!HALF) {
            for (int o = 1; o < S; o <<= 1) {
                a.fx += __shfl_xor_sync(FULL, a.fx, o);
                a.fy += __shfl_xor_sync(FULL, a.fy, o);
                a.fz += __shfl_xor_sync(FULL, a.fz, o);
            }
            if (own && sub == 0) {   // a global reduction: the DPD blocks of a fused pair launch add into F too
                const int i = real_as_int(sw[s].w);
                atomicAdd(&F[3 * i], a.fx);
                atomicAdd(&F[3 * i + 1], a.fy);
                atomicAdd(&F[3 * i + 2], a.fz);
            }
        }
    }
    if constexpr (HALF) {   // what is left in the ring (cnt < 32)
        __syncwarp();
        if (lane < cnt) real_ring<ALL>(g, ring[(head + lane) & (kRealRing - 1)], sq, sw, F, a);
    }
}

// spf: positions of the sorted beads in float (FP32: the sorted array itself).
// LEAVE: a block without beads leaves before the block sum (batches).
template <typename R, bool LEAVE = false>
__device__ __forceinline__ void k_real_body(Geo g, const int* __restrict__ tstart,
                                                       const typename V4<R>::T* __restrict__ sq,
                                                       const typename V4<R>::T* __restrict__ sw,
                                                       const int* __restrict__ sb, const float4* __restrict__ spf,
                                                       R* __restrict__ F, double* __restrict__ rpart, Blk blk) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* list = reinterpret_cast<int*>(smraw) + warp * 32 * kRealQ + lane;   // FP32: entry k at 32 k
    int2* ring = reinterpret_cast<int2*>(smraw) + warp * kRealRing;          // FP64
    const int nq = tstart[g.ntiles];
    // lanes per bead: enough to fill the chip, no more (see the plan's real_lanes). FP32:
    // two at least, one lane alone walks a bead's whole rows and drains its list more
    // often; whole calls at one / two lanes: 81,000 beads all charged 2004 / 1287 us (1958
    // with staged halos), half of 375,000 1229 / 1018, a tenth of 3M 1034 / 1009
    constexpr int SMIN = real_half<R>() ? 1 : 2;
    int S = 32;
    while (S > SMIN && (long long)nq * S > (S > 8 ? g.real_lanes / 3 * 2 : g.real_lanes)) S >>= 1;
    if (LEAVE && (long long)blk.id * (kRealThreads / S) >= nq) {
        if (threadIdx.x == 0) rpart[2 * blk.id] = rpart[2 * blk.id + 1] = 0.0;
        return;
    }
    RealSum<R> a{(R)0, (R)0, (R)0, (R)0, (R)0};
    if (2 * g.rs + 1 >= g.ntd)
        real_sweep<R, true>(g, nq, S, tstart, sq, sw, sb, spf, list, ring, F, a, blk);
    else
        real_sweep<R, false>(g, nq, S, tstart, sq, sw, sb, spf, list, ring, F, a, blk);
    double e, w;
    block_sum2_r<R>(a.e, a.w, e, w);
    if (threadIdx.x == 0) {
        rpart[2 * blk.id] = e;
        rpart[2 * blk.id + 1] = w;
    }
}

template <typename R>
__global__ void __launch_bounds__(kRealThreads, sizeof(R) == 4 ? 4 : 2) k_real(Geo g, const int* __restrict__ tstart,
                                                       const typename V4<R>::T* __restrict__ sq,
                                                       const typename V4<R>::T* __restrict__ sw,
                                                       const int* __restrict__ sb, const float4* __restrict__ spf,
                                                       R* __restrict__ F, double* __restrict__ rpart) {
    k_real_body<R>(g, tstart, sq, sw, sb, spf, F, rpart, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---------------------------------------------------------------------------
// DPD: cell list of all beads (edge >= 1) by a counting sort.
// ---------------------------------------------------------------------------
// Cells of edge L/ncd > 1 (the plan keeps a relative margin so that rounding
// of x * ncd/L cannot separate two beads closer than 1 by two cells).
// The cell of a wrapped coordinate, for the cell list and for the pair sweep that
// reads it: always inside the list (a coordinate that is not a number converts
// to 0 from float, to the smallest int from double: the last cell).
template <typename R>
__device__ __forceinline__ int cell_of(R xw, R rinv, int ncd) {
    return (int)min((unsigned)(int)(xw * rinv), (unsigned)(ncd - 1));
}

template <typename R>
__global__ void k_cell_count(int N, int ncd, double L, R rinv, float xmaxf, float Lhi, float Llo,
                             const R* __restrict__ pos,
                             int* __restrict__ ckey, int* __restrict__ ccount, R* __restrict__ F) {
    pdl_enter();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        F[3 * i] = (R)0;   // the pair kernel adds into F
        F[3 * i + 1] = (R)0;
        F[3 * i + 2] = (R)0;
        int c[3];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            c[t] = cell_of(wrap_r(pos[3 * i + t], L, xmaxf, Lhi, Llo), rinv, ncd);
        }
        const int cell = (c[2] * ncd + c[1]) * ncd + c[0];
        ckey[i] = cell;
        atomicAdd(&ccount[cell], 1);
    }
}

// Also clears the cell counts for the next step's k_cell_count (the scan has
// read them). FP32: clears the force accumulators of the sorted beads (df) and
// leaves every bead's slot in ckey; FP64: a float copy of the positions (spf).
template <typename R>
__global__ void k_cell_scatter(int N, double L, float xmaxf, float Lhi, float Llo, const R* __restrict__ pos,
                               const R* __restrict__ v0, const int* __restrict__ type, int* __restrict__ ckey,
                               int* __restrict__ ccur, typename V4<R>::T* __restrict__ sp,
                               typename V4<R>::T* __restrict__ sv, float4* __restrict__ df, int* __restrict__ ccount,
                               int ncells) {
    pdl_enter();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) ccount[c] = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int slot = atomicAdd(&ccur[ckey[i]], 1);
        typename V4<R>::T a, b;
        a.x = wrap_r(pos[3 * i], L, xmaxf, Lhi, Llo);
        a.y = wrap_r(pos[3 * i + 1], L, xmaxf, Lhi, Llo);
        a.z = wrap_r(pos[3 * i + 2], L, xmaxf, Lhi, Llo);
        a.w = int_as_real(i, (R)0);
        b.x = v0[3 * i];
        b.y = v0[3 * i + 1];
        b.z = v0[3 * i + 2];
        b.w = int_as_real(type[i], (R)0);
        sp[slot] = a;
        sv[slot] = b;
        if constexpr (sizeof(R) == 4) {
            df[slot] = make_float4(0.f, 0.f, 0.f, 0.f);
            ckey[i] = slot;
        } else {
            df[slot] = make_float4((float)a.x, (float)a.y, (float)a.z, 0.f);
        }
    }
}

// Philox4x32-10 (Salmon et al., SC'11): 10 rounds of two 32x32->64 products,
// key bumped by the Weyl constants between rounds. theta_ij draws word 0 of
// the counter (min(i,j), max(i,j), step_lo, step_hi) under key = seed. Within
// a launch the key and the step are fixed: the round keys come from the host
// (DpdDev::rk0/rk1, read as launch constants) and the first round's product
// of the counter word step_lo is formed once per thread (PhiloxStep); a draw
// then costs one wide multiply for word 0 in the first round, two per round
// after it, and one in the last (whose other outputs are not used).
struct PhiloxStep {
    uint32_t lo1, hi1;   // 0xCD9E8D57 * step_lo
    uint32_t x2;         // step_hi ^ round key 1 of round 0
};
__device__ __forceinline__ PhiloxStep philox_step(const DpdDev& d, uint64_t step) {
    const uint64_t p = (uint64_t)0xCD9E8D57u * (uint32_t)step;
    PhiloxStep ps;
    ps.lo1 = (uint32_t)p;
    ps.hi1 = (uint32_t)(p >> 32);
    ps.x2 = (uint32_t)(step >> 32) ^ d.rk1[0];
    return ps;
}
__device__ __forceinline__ uint32_t philox_word0(uint32_t c0, uint32_t c1, const PhiloxStep& ps, const DpdDev& d) {
    // round 0: the product of word 2 is the launch's
    const uint64_t p00 = (uint64_t)0xD2511F53u * c0;
    uint32_t n0 = ps.hi1 ^ c1 ^ d.rk0[0];
    uint32_t n1 = ps.lo1;
    uint32_t n2 = (uint32_t)(p00 >> 32) ^ ps.x2;
    uint32_t n3 = (uint32_t)p00;
#pragma unroll
    for (int r = 1; r < 9; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * n0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * n2;
        const uint32_t m0 = (uint32_t)(p1 >> 32) ^ n1 ^ d.rk0[r];
        const uint32_t m2 = (uint32_t)(p0 >> 32) ^ n3 ^ d.rk1[r];
        n1 = (uint32_t)p1;
        n3 = (uint32_t)p0;
        n0 = m0;
        n2 = m2;
    }
    // round 9: word 0 only
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * n2;
    return (uint32_t)(p1 >> 32) ^ n1 ^ d.rk0[9];
}

// theta_ij of Eq. 5: uniform on [-sqrt3, sqrt3].
template <typename R>
__device__ __forceinline__ R dpd_theta(const PhiloxStep& ps, const DpdDev& d, int i, int j) {
    const uint32_t w = philox_word0((uint32_t)min(i, j), (uint32_t)max(i, j), ps, d);
    // sqrt3 (2 u - 1) with u = (w + 1/2) 2^-32
    return fma((R)w, (R)(2.0 * 1.7320508075688772935 * 2.3283064365386962890625e-10),
               (R)(1.7320508075688772935 * (2.3283064365386962890625e-10 - 1.0)));
}

// DPD pair forces (Eq. 2-7, R_c = 1): F^C + F^D + F^R/sqrt(dt) on every pair
// closer than 1, each pair once (Newton's third law; theta_ij is symmetric),
// and the bonds (Sec. 2), one thread per bond, into F (zeroed by the caller).
//
// S lanes per bead of the cell-sorted order, 32 / S consecutive beads per warp,
// as in the real-space sweep: a bead's partners are the beads of its forward
// half shell -- those after it in its own cell, the next cell along x, the
// cells x-1..x+1 of the row (0, +1) and of the rows (+1, -1..1) -- which are 5
// contiguous runs of sorted beads (and their parts across the box face), read
// straight from the sorted arrays. Cells have an edge > 1 and there are at
// least 3 per dimension, so a run's image shift is one constant.
//   FP32: each lane notes its pairs in a list of its own and evaluates the
//     lists in step; the force on its bead stays in registers, -f goes to bead
//     j's accumulator by one 16-byte reduction (df, sorted order, cleared by
//     k_cell_scatter; the closing kick adds it to F).
//   FP64: the cutoff is tested on a float copy, the pairs go to a ring per warp
//     and are decided and evaluated on full warps (every FP64 instruction costs
//     the whole warp); +f and -f go to F by global reductions.
// The form before staged 4^3-cell blocks with their halo in shared memory: 512
// blocks of uneven size at 81k beads, six 4-byte reductions per pair. The one
// launch of both pair sums at 81k beads 49 -> 39 us (FP32), the step 101 -> 94;
// steps of 3000 beads 56 -> 44; FP64 steps 374 -> 357 (bound by the FP64
// instructions of the pairs in either form).
constexpr int kDpdThreads = 256;
template <typename R>
constexpr int dpd_smem_bytes() { return real_smem_bytes<R>(); }

// Four consecutive floats by one reduction (16-byte aligned).
__device__ __forceinline__ void red_add4(float4* p, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// |F| / r of a pair at squared distance r2 (Eq. 3-5 with w^D = (w^R)^2 = w^2):
// w (a - gamma w (r.v)/r + sigma theta/sqrt(dt)) / r; adds a w^2 to ec.
template <typename R>
__device__ __forceinline__ R dpd_force(const DpdDev& d, const PhiloxStep& ps, R r2, R vd, R a, int i, int j, R& ec) {
    const R ir = r_rsqrt(r2);
    const R w = (R)1 - r2 * ir;
    const R th = dpd_theta<R>(ps, d, i, j);
    const R wi = w * ir;
    ec = fma(a * w, w, ec);   // halved once per block
    return wi * fma(-dpd_k(d, (R)0).gam * wi, vd, fma(dpd_k(d, (R)0).srdt, th, a));
}

// FP32: the noted pairs of this lane's bead (pi, vi), all lanes in step.
__device__ __forceinline__ void dpd_drain(const DpdDev& d, const PhiloxStep& ps, const float4& pi, const float4& vi,
                                          const int* list, int cnt, const float4* __restrict__ sp,
                                          const float4* __restrict__ sv, const float* __restrict__ atab,
                                          float4* __restrict__ df, float& fx, float& fy, float& fz, float& ec) {
    const float L = d.kf.L, hL = d.kf.hL;
    const float* arow = atab + __float_as_int(vi.w) * d.ntypes;
    const int m = __reduce_max_sync(0xffffffffu, cnt);
    for (int k = 0; k < m; ++k) {
        if (k >= cnt) continue;
        const int j = list[32 * k];
        const float4 pj = sp[j], vj = sv[j];
        const float rx = min_image(pi.x, pj.x, L, hL);
        const float ry = min_image(pi.y, pj.y, L, hL);
        const float rz = min_image(pi.z, pj.z, L, hL);
        const float vd = (vi.x - vj.x) * rx + (vi.y - vj.y) * ry + (vi.z - vj.z) * rz;   // r_ij . v_ij
        const float fm = dpd_force<float>(d, ps, dist2(rx, ry, rz), vd, arow[__float_as_int(vj.w)],
                                          __float_as_int(pi.w), __float_as_int(pj.w), ec);
        const float gx = fm * rx, gy = fm * ry, gz = fm * rz;
        fx += gx;
        fy += gy;
        fz += gz;
        red_add4(df + j, -gx, -gy, -gz, 0.f);
    }
}

// FP64: one ring entry (bead i, candidate j, image as in real_entry) per lane.
__device__ __forceinline__ void dpd_ring(const DpdDev& d, const PhiloxStep& ps, const int2 e,
                                         const double4_32a* __restrict__ sp, const double4_32a* __restrict__ sv,
                                         const double* __restrict__ atab, double* __restrict__ F, double& ec) {
    const int i = e.x & 0x1fffffff, j = e.y & 0x1fffffff;
    const double4_32a pi = sp[i], pj = sp[j];
    double rx = pi.x - pj.x, ry = pi.y - pj.y, rz = pi.z - pj.z;
    const int im = (int)((unsigned)e.x >> 29 | ((unsigned)e.y >> 29) << 3);
    if (im != 13) {   // across a box face
        const double L = d.kd.L;
        const int iz = im / 9, iy = (im - 9 * iz) / 3, ix = im % 3;
        if (ix != 1) rx += ix ? L : -L;
        if (iy != 1) ry += iy ? L : -L;
        if (iz != 1) rz += iz ? L : -L;
    }
    const double r2 = dist2(rx, ry, rz);
    if (!(r2 < 1.0 && r2 > 0.0)) return;
    const double4_32a vi = sv[i], vj = sv[j];
    const int oi = real_as_int(pi.w), oj = real_as_int(pj.w);
    const double vd = (vi.x - vj.x) * rx + (vi.y - vj.y) * ry + (vi.z - vj.z) * rz;
    const double fm = dpd_force<double>(d, ps, r2, vd, atab[real_as_int(vi.w) * d.ntypes + real_as_int(vj.w)], oi, oj,
                                        ec);
    const double gx = fm * rx, gy = fm * ry, gz = fm * rz;
    atomicAdd(&F[3 * oi], gx);
    atomicAdd(&F[3 * oi + 1], gy);
    atomicAdd(&F[3 * oi + 2], gz);
    atomicAdd(&F[3 * oj], -gx);
    atomicAdd(&F[3 * oj + 1], -gy);
    atomicAdd(&F[3 * oj + 2], -gz);
}

// spf: float positions of the sorted beads (FP32: sp itself).
template <typename R>
__device__ __forceinline__ void k_dpd_body(const DpdDev& d, const typename V4<R>::T* __restrict__ sp,
                                           const typename V4<R>::T* __restrict__ sv,
                                           const float4* __restrict__ spf, const int* __restrict__ cstart,
                                           const R* __restrict__ atab, const R* __restrict__ pos,
                                           const int* __restrict__ bnd, const uint64_t* __restrict__ stepp,
                                           float4* __restrict__ df, R* __restrict__ F, double* __restrict__ dpart,
                                           Blk bk) {
    pdl_enter();
    using V = typename V4<R>::T;
    constexpr bool F64 = sizeof(R) == 8;
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int NW = kDpdThreads / 32;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int* list = reinterpret_cast<int*>(smraw) + warp * 32 * kRealQ + lane;   // FP32: entry k at 32 k
    int2* ring = reinterpret_cast<int2*>(smraw) + warp * kRealRing;          // FP64
    const PhiloxStep ps = philox_step(d, *stepp);
    const R L = dpd_k(d, (R)0).L;
    R ec = 0, eb = 0;
    // harmonic bonds (Sec. 2): one thread per bond, +f to i and -f to j
    {
        const R Kb = dpd_k(d, (R)0).Kb, r0b = dpd_k(d, (R)0).r0b, iL = dpd_k(d, (R)0).iL;
        for (int k = bk.id * blockDim.x + tid; k < d.nbonds; k += bk.n * blockDim.x) {
            const int i = bnd[2 * k], j = bnd[2 * k + 1];
            R dd[3];
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                // minimum image of the raw (unwrapped) difference; a bond is far
                // shorter than L/2, so d/L is never near a half-integer
                const R dx = pos[3 * i + t] - pos[3 * j + t];
                dd[t] = dx - L * rint(dx * iL);
            }
            const R r2 = dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2];
            const R ir = r2 > (R)0 ? r_rsqrt(r2) : (R)0;
            const R dr = r2 * ir - r0b;   // r - r0
            eb = fma(Kb * dr, dr, eb);    // K (r - r0)^2; halved once per block
            if (r2 > (R)0) {
                const R fm = -Kb * dr * ir;
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    atomicAdd(&F[3 * i + t], fm * dd[t]);
                    atomicAdd(&F[3 * j + t], -fm * dd[t]);
                }
            }
        }
    }
    // FP64: float positions carry at most L 2^-24 each, so for r2 near 1
    // |r2f - r2| <= 7e-7 (L + 1)
    const float Lf = d.kf.L, hi = F64 ? 1.0f + 1e-4f + 4e-6f * Lf : 1.0f;
    const int ncd = d.ncd;
    int S = 32;
    while (S > 1 && (long long)d.N * S > d.lanes) S >>= 1;
    const int gpw = 32 / S, sub = lane & (S - 1), grp = lane / S;
    int cnt = 0, head = 0;   // noted pairs of this lane (FP32); ring fill and head (FP64)
    for (int s0 = (bk.id * NW + warp) * gpw; s0 < d.N; s0 += bk.n * NW * gpw) {
        const int s = s0 + grp;
        const bool own = s < d.N;
        float4 pf;
        V vi;
        int cx = 0, cy = 0, cz = 0;
        if (own) {
            pf = spf[s];
            if constexpr (!F64) vi = sv[s];
            const V pw = sp[s];   // the cell as k_cell_count decided it, in the working precision
            const R ri = dpd_cinv(d, (R)0);
            cx = cell_of(pw.x, ri, ncd);
            cy = cell_of(pw.y, ri, ncd);
            cz = cell_of(pw.z, ri, ncd);
        }
        float fx = 0.f, fy = 0.f, fz = 0.f;
        // the half shell's rows (uniform over the warp), each as its run inside the box
        // and its run across the box face; one more turn empties the lists
        int row = 0;
        bool across = false;
        int w0 = 0, wl = 0;
        float hx = 0.0f, hy = 0.0f, hz = 0.0f;
        while (true) {
            const bool last = row == 5;
            int j0 = 0, len = 0;
            if (across) {
                j0 = w0;
                len = wl;
            } else if (!last) {
                const int dz = row >= 2 ? 1 : 0, dy = row >= 2 ? row - 3 : row;
                int zz = cz + dz, yy = cy + dy;
                hx = hy = hz = 0.0f;
                if (zz >= ncd) { zz -= ncd; hz = -Lf; }
                if (yy < 0) { yy += ncd; hy = Lf; } else if (yy >= ncd) { yy -= ncd; hy = -Lf; }
                const int* cs = cstart + (zz * ncd + yy) * ncd;
                const int xa = row == 0 ? cx : cx - 1, xb = cx + 1;
                wl = 0;
                if (own) {
                    j0 = row == 0 ? s + 1 : cs[max(xa, 0)];
                    len = cs[min(xb, ncd - 1) + 1] - j0;
                    if (xa < 0 || xb >= ncd) {
                        w0 = cs[xa < 0 ? ncd - 1 : 0];
                        wl = cs[xa < 0 ? ncd : 1] - w0;
                    }
                }
            }
            const int mlen = __reduce_max_sync(FULL, len);
            const int image = (hz < 0.0f ? 0 : 9) + (hy > 0.0f ? 6 : (hy < 0.0f ? 0 : 3)) +
                              (hx > 0.0f ? 2 : (hx < 0.0f ? 0 : 1));
            for (int t0 = 0;;) {
                if constexpr (F64) {
                    while (cnt >= 32) {
                        __syncwarp();
                        dpd_ring(d, ps, ring[(head + lane) & (kRealRing - 1)], sp, sv, atab, F, ec);
                        __syncwarp();
                        head += 32;
                        cnt -= 32;
                    }
                } else {
                    if (last || __any_sync(FULL, cnt > kRealQ - kRealU)) {
                        dpd_drain(d, ps, pf, vi, list, cnt, sp, sv, atab, df, fx, fy, fz, ec);
                        cnt = 0;
                    }
                }
                if (t0 >= mlen) break;
                float4 b[kRealU];
#pragma unroll
                for (int u = 0; u < kRealU; ++u) {
                    const int t = t0 + u * S + sub;
                    if (t < len) b[u] = spf[j0 + t];
                }
#pragma unroll
                for (int u = 0; u < kRealU; ++u) {
                    const int t = t0 + u * S + sub;
                    bool hit = false;
                    if (t < len) {
                        const float r2 = dist2(__fadd_rn(__fsub_rn(pf.x, b[u].x), hx),
                                               __fadd_rn(__fsub_rn(pf.y, b[u].y), hy),
                                               __fadd_rn(__fsub_rn(pf.z, b[u].z), hz));
                        hit = F64 ? r2 <= hi : (r2 < hi && r2 > 0.0f);   // FP64 decides in the ring
                    }
                    if constexpr (F64) {
                        const unsigned m = __ballot_sync(FULL, hit);
                        const int at = cnt + __popc(m & ((1u << lane) - 1u));
                        if (hit && ENUF_GUARD(d.check, at < kRealRing, 8))
                            ring[(head + at) & (kRealRing - 1)] = real_entry(s, j0 + t, image);
                        cnt += __popc(m);
                    } else if (hit && ENUF_GUARD(d.check, cnt < kRealQ, 8)) {
                        list[32 * cnt] = j0 + t;
                        ++cnt;
                    }
                }
                t0 += kRealU * S;
            }
            if (last) break;
            if (!across && __any_sync(FULL, wl > 0)) {
                across = true;
                hx = row > 0 && cx == 0 ? Lf : -Lf;   // read by the lanes with wl > 0
                continue;
            }
            across = false;
            ++row;
        }
        if constexpr (!F64) {
            for (int o = 1; o < S; o <<= 1) {
                fx += __shfl_xor_sync(FULL, fx, o);
                fy += __shfl_xor_sync(FULL, fy, o);
                fz += __shfl_xor_sync(FULL, fz, o);
            }
            if (own && sub == 0) red_add4(df + s, fx, fy, fz, 0.f);
        }
    }
    if constexpr (F64) {   // what is left in the ring (cnt < 32)
        __syncwarp();
        if (lane < cnt) dpd_ring(d, ps, ring[(head + lane) & (kRealRing - 1)], sp, sv, atab, F, ec);
    }
    double e1, e2;
    block_sum2_r<R>(ec, eb, e1, e2);
    if (tid == 0) {
        dpart[2 * bk.id] = 0.5 * e1;
        dpart[2 * bk.id + 1] = 0.5 * e2;
    }
}

template <typename R>
__global__ void __launch_bounds__(kDpdThreads, sizeof(R) == 4 ? 4 : 3)
    k_dpd(DpdDev d, const typename V4<R>::T* __restrict__ sp, const typename V4<R>::T* __restrict__ sv,
          const float4* __restrict__ spf, const int* __restrict__ cstart, const R* __restrict__ atab,
          const R* __restrict__ pos, const int* __restrict__ bnd, const uint64_t* __restrict__ stepp,
          float4* __restrict__ df, R* __restrict__ F, double* __restrict__ dpart) {
    k_dpd_body<R>(d, sp, sv, spf, cstart, atab, pos, bnd, stepp, df, F, dpart, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// The DPD pair forces and the real-space electrostatic pairs in one launch
// (horizontal fusion): blocks [0, nd) run the DPD body over the all-bead cell
// list, the others the real-space body over the charged-bead tiles. Both add
// into F (global reductions and per-bead sums) and write their own block
// partials; launched once both cell structures exist.
template <typename R>
__global__ void __launch_bounds__(kDpdThreads, sizeof(R) == 4 ? 4 : 2)
    k_pairs(DpdDev d, const typename V4<R>::T* __restrict__ sp, const typename V4<R>::T* __restrict__ sv,
            const float4* __restrict__ spf, const int* __restrict__ cstart, const R* __restrict__ atab,
            const R* __restrict__ pos, const int* __restrict__ bnd, const uint64_t* __restrict__ stepp,
            float4* __restrict__ df, R* __restrict__ F, double* __restrict__ dpart, int nd, Geo g,
            const int* __restrict__ tstart, const typename V4<R>::T* __restrict__ sq,
            const typename V4<R>::T* __restrict__ sw, const int* __restrict__ sb, const float4* __restrict__ sqf,
            double* __restrict__ rpart) {
    static_assert(kDpdThreads == kRealThreads && kRealThreads <= kSumThreads, "one block size for both roles");
    if ((int)blockIdx.x < nd)
        k_dpd_body<R>(d, sp, sv, spf, cstart, atab, pos, bnd, stepp, df, F, dpart, Blk{(int)blockIdx.x, nd});
    else
        k_real_body<R>(g, tstart, sq, sw, sb, sqf, F, rpart, Blk{(int)blockIdx.x - nd, (int)gridDim.x - nd});
}

// Table 2 steps 0-2 (m = 1): v0 = v + lambda F dt; v += F dt/2; r += v dt; step += 1.
// Four components per thread (the arrays are 32-byte aligned): the loads of
// all three arrays are in flight together.
template <typename R>
__global__ void k_vv_pre(int N, R lam, R dt, R* __restrict__ pos, R* __restrict__ vel, R* __restrict__ v0,
                         const R* __restrict__ F, uint64_t* __restrict__ stepp) {
    pdl_enter();
    using V = typename V4<R>::T;
    if (blockIdx.x == 0 && threadIdx.x == 0) *stepp += 1;
    const int n3 = 3 * N, n4 = n3 / 4;
    auto one = [&](R f, R v, R& x, R& w) {   // returns the new velocity
        w = v + lam * f * dt;
        const R vn = v + (R)0.5 * f * dt;
        x = x + vn * dt;
        return vn;
    };
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n4; k += gridDim.x * blockDim.x) {
        const V f = reinterpret_cast<const V*>(F)[k];
        V v = reinterpret_cast<const V*>(vel)[k], x = reinterpret_cast<const V*>(pos)[k], w;
        v.x = one(f.x, v.x, x.x, w.x);
        v.y = one(f.y, v.y, x.y, w.y);
        v.z = one(f.z, v.z, x.z, w.z);
        v.w = one(f.w, v.w, x.w, w.w);
        reinterpret_cast<V*>(v0)[k] = w;
        reinterpret_cast<V*>(vel)[k] = v;
        reinterpret_cast<V*>(pos)[k] = x;
    }
    const int k = 4 * n4 + (int)threadIdx.x;   // the last n3 mod 4 components
    if (blockIdx.x == 0 && k < n3) {
        R x = pos[k], w;
        const R vn = one(F[k], vel[k], x, w);
        v0[k] = w;
        vel[k] = vn;
        pos[k] = x;
    }
}

// FP32: adds the DPD pair forces (df, in the cell-sorted order; slot: each
// bead's place in it) to F. The closing kick does it in a step; this kernel in
// force evaluations outside one.
static __global__ void __launch_bounds__(256) k_dpd_add(int N, float* __restrict__ F, const float4* __restrict__ df,
                                                        const int* __restrict__ slot) {
    pdl_enter();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const float4 a = df[slot[i]];
        F[3 * i] += a.x;
        F[3 * i + 1] += a.y;
        F[3 * i + 2] += a.z;
    }
}

// Table 2 step 6: v += F dt/2 (FP32: after adding the DPD pair forces to F);
// kinetic energy partials. The last block then reduces all energies of the
// step (totals).
template <typename R>
__global__ void __launch_bounds__(256) k_vv_post(Geo g, int N, R dt, R* __restrict__ vel, R* __restrict__ F,
                                                const float4* __restrict__ df, const int* __restrict__ slot,
                                                double* __restrict__ kpart, TotalsArgs tot) {
    pdl_enter();
    double ke = 0.0, dummy = 0.0;
    auto one = [&](R f, R v) {
        const R vn = v + (R)0.5 * f * dt;
        ke = fma((double)vn, (double)vn, ke);
        return vn;
    };
    if constexpr (sizeof(R) == 4) {
#pragma unroll 2
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
            const float4 a = df[slot[i]];
            const float f0 = F[3 * i] + a.x, f1 = F[3 * i + 1] + a.y, f2 = F[3 * i + 2] + a.z;
            const float v0 = vel[3 * i], v1 = vel[3 * i + 1], v2 = vel[3 * i + 2];
            F[3 * i] = f0;
            F[3 * i + 1] = f1;
            F[3 * i + 2] = f2;
            vel[3 * i] = one(f0, v0);
            vel[3 * i + 1] = one(f1, v1);
            vel[3 * i + 2] = one(f2, v2);
        }
    } else {
        using V = typename V4<R>::T;
        const int n3 = 3 * N, n4 = n3 / 4;
#pragma unroll 2
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n4; k += gridDim.x * blockDim.x) {
            const V f = reinterpret_cast<const V*>(F)[k];
            V v = reinterpret_cast<const V*>(vel)[k];
            v.x = one(f.x, v.x);
            v.y = one(f.y, v.y);
            v.z = one(f.z, v.z);
            v.w = one(f.w, v.w);
            reinterpret_cast<V*>(vel)[k] = v;
        }
        const int k = 4 * n4 + (int)threadIdx.x;
        if (blockIdx.x == 0 && k < n3) vel[k] = one(F[k], vel[k]);
    }
    block_sum2(ke, dummy);
    if (threadIdx.x == 0) kpart[blockIdx.x] = 0.5 * ke;
    if (tot.Edev) totals_if_last(g, tot, (int)gridDim.x);
}

// Standalone totals (one CTA), for evaluations outside a step graph.
static __global__ void __launch_bounds__(1024) k_totals(Geo g, TotalsArgs t) {
    pdl_enter();
    totals_block(g, t);
}

}  // namespace enuf
