// enuf_internal.h -- plan layout shared by the C-ABI layer and the kernel
// translation units (one per precision).
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

#include "enuf_fft.cuh"

namespace enuf {

// Debug builds (-DENUF_CHECK): device-side index checks. ENUF_GUARD(word,
// cond, bit) is cond, and when cond fails sets bit `bit` of the plan's check
// word (read by enuf_check_word); the caller skips the access it guards.
// Release builds compile it to true.
#ifdef ENUF_CHECK
__device__ __forceinline__ bool enuf_guard(unsigned int* word, bool ok, int bit) {
    if (!ok && word != nullptr) atomicOr(word, 1u << bit);
    return ok;
}
#define ENUF_GUARD(word, cond, bit) enuf_guard((word), (cond), (bit))
#else
#define ENUF_GUARD(word, cond, bit) true
#endif

// Tiles up to which the scatter blocks of the binning scan the counters for
// themselves (16 KB of shared memory and 16 counters a thread, ~1 us, less than
// a launch); more go through a scan kernel.
constexpr int kBinScanTiles = 4096;

// Constants of the real-space pair arithmetic in one working precision.
template <typename R>
struct RealK {
    R L, hL, rc2;     // box edge, L / 2, r_c^2
    R al, c2a, be;    // alpha, 2 alpha / sqrt(pi), beta
    R kap, kinv;      // kappa, kernel table intervals per unit length
};

// Window constants in one working precision: 1 / b, (pi b)^{-1/2}, the force prefactor.
template <typename R>
struct WinK {
    R rb, wn, pref;
};

// DPD constants in one working precision: box, dissipation, sigma / sqrt(dt),
// bond constants, 1 / L.
template <typename R>
struct DpdK {
    R L, hL, gam, srdt, Kb, r0b, iL;
};

// Geometry and constants every kernel needs, passed by value. The kernels take
// their constants in the working precision from the host (rkf/rkd, wkf/wkd):
// on this part a conversion from double, like every double operation, takes
// 16 cycles of an SM's FP64 units per warp, in an FP32 kernel too.
struct Geo {
    int n;        // oversampled grid per dimension (sigma_s * M)
    int nc;       // kept modes per side, |k_t| <= nc
    int K;        // 2 nc + 1
    int p;        // window cutoff (2p taps per dimension)
    int T;        // spreading tile edge (grid points)
    int ntd;      // tiles per dimension
    int ntiles;   // ntd^3
    int rs;       // real-space stencil radius in tiles
    int nbin;     // blocks of the charged-bead binning
    int chunk;    // beads per binning block
    int kmask;
    int nf;       // reciprocal force fields: 3 (ik-differentiation) or 1 (window gradient)
    int h4;       // FP32: the fields interleaved, float4 (h_x, h_y, h_z, 0) per point
    int bin_scan; // 1: every scatter block scans the tile counters itself (up to
                  //    kBinScanTiles tiles); 0: a scan kernel between count and scatter
    double L, alpha, beta, kappa, rc;
    double b;      // Gaussian window parameter 2 sigma p / ((2 sigma - 1) pi)
    double wnorm;  // (pi b)^{-1/2}
    double e3[9];  // wnorm e^{-m^2/b}, m = 0 .. p
    double ratio;  // n / L: grid coordinate u = x * ratio (one FP64 product)
    double rb;     // 1 / b
    double pref;   // kappa * 2 / L^2 (Eq. 25 prefactor); gradient mode: -kappa n / (pi L^2)
    double c2a;    // 2 alpha / sqrt(pi)
    float xmaxf;   // largest float below L: float x is inside [0, L) iff 0 <= x <= xmaxf
    float rhi, rlo;  // n/L split into two floats (compensated float grid coordinate)
    double c_self;   // -kappa alpha / sqrt(pi)           (E_self = c_self * sum q^2)
    double c_neut;   // -kappa pi / (2 V alpha^2)         (E_neutral = c_neut * Q^2)
    double c_recip;  // kappa / (2 pi L)                  (E_recip = c_recip * sum D |F|^2)
    int slater_k;    // 1: Slater form factor in k space (real-space kernel J = B1 - I)
    int kn;          // real-space kernel table intervals on [0, r_c] (0: no table)
    double kinv;     // kn / r_c
    double kh;       // r_c / kn
    const void* ktab;  // real [kn][kKtStride]: quintic coefficients of J(r) = r u(r) per interval
    RealK<float> rkf;
    RealK<double> rkd;
    WinK<float> wkf;
    WinK<double> wkd;
    float Lhi, Llo;   // L split into two floats (FP32 wrap)
    int real_lanes;   // real space: lanes per bead S while N_q S stays below this
    int slater;   // beta > 0: the real-space term carries the Slater correction
    // FP64 cutoff pre-test on float positions: r_c^2 plus a band that covers the float
    // error (positions and L rounded to float, |r2f - r2| <= ~1.5e-6 L r_c)
    float r2hi;
    int nmax;          // capacity in beads (sorted charged-bead arrays)
    unsigned int* check;  // debug builds: failure bits of the device index checks
};

// Footprint spreading on bricks (k_spread_brick): staging capacities and the
// shared memory of a brick of T x T rows of BX points (fx_bytes: the fused x
// pass's twiddles and line buffers, which reuse the staging region).
constexpr int kBrickCand = 512;    // candidates staged per round
constexpr int kBrickItems = 64;    // items per weight batch
constexpr int kBrickRanges = 18;   // contiguous runs of sorted beads around a brick
constexpr int kBrickTaps = 16;     // weight row length (2p <= 16)
template <typename R>
__host__ __device__ constexpr int brick_stage_bytes() {
    return kBrickCand * (4 + 4 + (int)sizeof(R) + 4) +
           kBrickItems * (3 * kBrickTaps * (int)sizeof(R) + 4 + (int)sizeof(R));
}
template <typename R>
__host__ __device__ constexpr int brick_smem(int T, int BX, int fx_bytes) {
    return T * T * BX * (int)sizeof(R) + (brick_stage_bytes<R>() > fx_bytes ? brick_stage_bytes<R>() : fx_bytes);
}

// Preferred shared-memory split of the two-factor FFT kernels (percent): the plane
// passes share SMs with the pair kernels, the persistent line passes want three
// CTAs of 72 KB.
constexpr int kSMs = 152;
constexpr int kCarvePlanes = 60, kCarveLines = 100;

// Row length of the real-space kernel table (16-byte aligned rows).
constexpr int kKtStride64 = 6;   // c_0..c_5 in double
constexpr int kKtStride32 = 8;   // c_0..c_5 in float, 2 padding

// Lines per CTA of each FFT pass.
struct FftShape {
    int lx;    // complex lines (pairs of real rows) per CTA, forward x
    int ly;    // lines per CTA, forward y
    int lz;    // lines per CTA, z pass (forward + convolve + 3 inverses)
    int liy;   // lines per CTA, inverse y
    int lix;   // complex lines per CTA, inverse x (two-factor: row pairs, of every field)
    int tx, ty, tz, tiy, tix;   // threads per CTA of each pass
    int smem_x, smem_y, smem_z, smem_iy, smem_ix;   // dynamic smem bytes
    int grid_x, grid_y_z, grid_z, grid_iy, grid_ix; // CTAs (grid_y_z: z-chunks of the y pass)
    // small grids: a whole z-plane per CTA, forward x+y and inverse y+x fused
    // (two kernels instead of four); spec2 is then plane-major [z][kx][ky]
    int fused;
    int t_xy, t_yx, smem_xy, smem_yx;
    int composite;   // the radix plan uses 6, 10, 12, 16 or 20 (FP32): the CR kernel instances
    int two;         // FP32 two-factor kernels (FftPlanDev::f1, f2), same shapes and layouts
    int two_ext;     // their split uses radix 9, 15 or 18 (reported as the Stockham schedule)
    // spreading: 1 tile form, 2 footprint bricks into the grid, 3 bricks fused with
    // the forward x pass (the x pass kernel is then not launched), 4 scatter form
    // over regions of edge sc_E
    int spread;
    // automatic choice of the tile or scatter form's sizes: the reduction form runs
    // (1; plan info keeps reporting `spread`); the grid is cleared by the count kernel
    // (1) or by a memset beside the binning (2)
    int red, red_zero;
    int brick_x, brick_threads, brick_smem, brick_grid, brick_lp;
    int sc_E;
};

// Device workspace of one plan (all pointers device memory, one allocation).
struct Work {
    // charged binning
    int* cnt_blk;    // [nbin] charged beads of each binning block
    int* tcnt;       // [ntiles] tile counters of the binning (0 between evaluations)
    int* tstart;     // [ntiles + 1]
    int* ticket;     // [4] arrival counters of last-block reductions (0 between launches)
    unsigned int* check;  // [1] failure bits of the ENUF_CHECK index checks
    int* crank;      // [nbin * chunk] rank of each compacted charged bead in its tile
    void* cpos;      // real4 [nbin * chunk] wrapped x, y, z, q of each compacted charged bead
    void* cfrac;     // real4 [nbin * chunk] fractional grid coordinates, original index bits
    int* cbase;      // [nbin * chunk] packed base grid index
    void* sq;        // real4 [n_max]  wrapped x, y, z, q (sorted)
    void* sw;        // real4 [n_max]  fractional grid coordinates, original index bits
    int* sb;         // [n_max]  packed base grid index
    float4* spf;     // [n_max]  float copy of the sorted positions (FP64; FP32: sq itself)
    void* wb;        // real [n_max][3][2p]  window weights psi(u - l) of each sorted bead
    // grids and spectra
    void* grid;      // real [n^3]
    void* spec1;     // cplx [n][nc+1][n]      after forward x   ([z][kx][y])
    void* spec2;     // cplx [nc+1][K][n]      after forward y   ([kx][ky][z])
    void* spec3;     // cplx [nf][n][nc+1][K]  after z pass      ([a][z][kx][ky]; three fields: G and kz G)
    void* spec4;     // cplx [3][n][n][nc+1]   after inverse y   ([a][z][y][kx])
    void* h;         // real [3][n^3]          conjugated-NFFT fields (Geo::h4: real [n^3][4])
    double* tab;     // [nc+1][K][K] influence/deconvolution table D(k) (0 outside the mode set)
    double* tabv;    // [nc+1][K][K] D(k) times the virial weight 1 - 2 pi^2 k^2/(alpha L)^2
    void* tabr;      // real copy of tab
    void* tw;        // cplx [n] twiddles e^{-2 pi i t/n}
    void* ktab;      // real [kn][kKtStride] real-space kernel table (FP64, or slater_k = 1)
    double* part;    // per-block partial sums
    double* Edev;    // [16] reduced totals
    // partial-sum segments (offsets into part, in doubles)
    int off_q, off_real, off_recip, off_dpd, off_kin;
    int nblk_real, nblk_conv, nblk_dpd, nblk_kin, nblk_gather;
    // preferred shared-memory split (percent, 0: none) of the pair and spreading kernels,
    // and of the binning, cell list and integrator
    int carve, carve_b;
    int off_pre;   // 8 doubles: the step's quantities 0-7 reduced beside the gather
};

// Arguments of one electrostatics evaluation.
struct EvalArgs {
    int N;
    const void* pos;   // real [N][3] (device)
    const void* q;     // real [N]
    void* F;           // real [N][3]
    bool zeroF;        // overwrite F (pure electrostatics) vs add into it (DPD step)
};

// Where the final FP64 totals read their per-block partials (offsets into
// Work::part, counts) and write Edev; ticket is the arrival counter of the
// kernel whose last block reduces them. Edev == nullptr: no totals.
struct TotalsArgs {
    const double* part;
    int off_q, nq, off_real, nreal, off_recip, nrecip, off_dpd, ndpd, off_kin, nkin;
    double* Edev;
    int* ticket;
    // pre (or nullptr): quantities 0-7 already reduced (k_totals_pre); the
    // closing totals then reduce the kinetic partials only
    double* pre;
};

// DPD device state and cell list (one per system).
struct DpdDev {
    unsigned int* check;   // the plan's check word (debug builds)
    int N, ntypes, ncd, ncells;
    int lanes;         // pair sweep: lanes per bead S while N S stays below this
    double L, gamma, sigma, dt, lambda_vv, K_bond, r0_bond;
    double rdt;    // 1 / sqrt(dt)
    double cinv;   // ncd / L
    float cinvf;
    DpdK<float> kf;
    DpdK<double> kd;
    float Lhi, Llo;   // L split into two floats (FP32 wrap)
    float xmaxf;   // largest float below L
    uint64_t seed;
    // Philox4x32-10 round keys of the seed (key bumped by the Weyl constants
    // each round), formed on the host: the kernel's rounds read them as
    // launch constants
    uint32_t rk0[10], rk1[10];
    void* pos; void* vel; void* v0; void* F; void* q;   // real
    int* type;
    void* atab;        // real [ntypes^2]
    int nbonds;
    int* bnd;                // bond pairs [nbonds][2]
    int* ckey; int* ccount; int* cstart; int* ccur;
    void* sp; void* sv;      // real4 [N] sorted: (x, y, z, orig) and (v0, type)
    // float4 [N], sorted order: FP32 the DPD force accumulators (ckey then holds every
    // bead's slot), FP64 a float copy of the positions
    float4* df;
    uint64_t* step_dev;      // device copy of the step counter
};

constexpr int kStageCount = 8;

// Host-side record of the launches one enqueue made (for the launch count).
struct LaunchLog {
    int kernels = 0;
};

struct Events {
    cudaEvent_t start[kStageCount];
    cudaEvent_t stop[kStageCount];
    bool on = false;
};

// One system of a batched launch sequence (FP32): its plan's geometry,
// shapes, workspace and this evaluation's arrays; Edev receives its totals.
struct BatchSys {
    Geo g;
    FftShape fs;
    FftPlanDev fp;
    Work w;
    int N;
    const void* pos;
    const void* q;
    void* F;
    double* Edev;
};

// Launch parameters of one batched kernel: its argument table and block map
// (device), the blocks of all systems together, threads and shared memory
// (the largest any system needs).
struct BatchKernel {
    void* tab = nullptr;
    int* cmap = nullptr;
    int blocks = 0, threads = 0, smem = 0;
    int T = 0;   // spreading (per group), gather: the common tap count 2p (0: mixed)
};
struct BatchLaunch {
    BatchKernel bin_count, bin_scatter, bin_weights, real, fft_xy, fft_z, fft_yx, gather;
    BatchKernel spread[6];   // one per tile edge present (8, 10, 12, 16, 20, 24)
    int nspread = 0;
};

template <typename R> cudaError_t configure_kernels(int max_smem);
// Attributes of the two-factor FFT kernels a plan runs (those of one length).
cudaError_t configure_fft2(const FftShape& fs, const FftPlanDev& fp, int max_smem);
template <typename R> int spread_smem(const Geo& g);
// dpd (a DPD step with fused pair kernels, or nullptr): the real-space launch
// also runs the DPD pair forces (k_pairs), which enqueue_dpd_forces then leaves out.
// evZ, evT (DPD steps, or nullptr): after the FFT the side stream reduces the
// step's energies other than the kinetic one (k_totals_pre, beside the
// gather) and records evT, on which the closing half kick must wait.
template <typename R>
cudaError_t enqueue_enuf(const Geo& g, const FftShape& fs, const FftPlanDev& fp, const Work& w,
                         const EvalArgs& a, cudaStream_t s0, cudaStream_t s1, cudaEvent_t evFork,
                         cudaEvent_t evJoin, Events* ev, LaunchLog* log, bool fuse_totals,
                         const DpdDev* dpd = nullptr, cudaEvent_t evZ = nullptr, cudaEvent_t evT = nullptr);
template <typename R>
cudaError_t enqueue_totals(const Geo& g, const Work& w, bool dpd, cudaStream_t s, LaunchLog* log, bool pdl);
template <typename R>
cudaError_t enqueue_dpd_forces(const Work& w, const DpdDev& d, cudaStream_t s, Events* ev, LaunchLog* log,
                               bool pair_kernel = true);
template <typename R>
cudaError_t enqueue_vv_pre(const Work& w, const DpdDev& d, cudaStream_t s, LaunchLog* log);
template <typename R>
cudaError_t enqueue_vv_post(const Geo& g, const Work& w, const DpdDev& d, cudaStream_t s, LaunchLog* log, bool pdl,
                            bool pre = false);
template <typename R>
cudaError_t enqueue_dpd_add(const DpdDev& d, cudaStream_t s, LaunchLog* log, bool pdl);
template <typename R>
cudaError_t enqueue_spread_only(const Geo& g, const Work& w, const EvalArgs& a, void* grid_out, cudaStream_t s);
// Batched launch sequence (FP32): a system qualifies when its plan runs the
// fused-plane two-factor FFT, has a tile edge of the column form and forms its tile
// starts in the scatter kernel. batch_bytes: the device tables' size; batch_build writes
// them (argument tables and block maps) into dbuf and fills the launch
// parameters; batch_enqueue launches the sequence (fork/join on s1 for the
// real-space pairs).
template <typename R> cudaError_t configure_batch(int max_smem);
template <typename R> size_t batch_bytes(const BatchSys* sys, int nsys);
template <typename R>
cudaError_t batch_build(void* dbuf, const BatchSys* sys, int nsys, BatchLaunch* out);
template <typename R>
cudaError_t batch_enqueue(const BatchLaunch& L, cudaStream_t s0, cudaStream_t s1, cudaEvent_t evFork, cudaEvent_t evJoin,
                          LaunchLog* log);

}  // namespace enuf
