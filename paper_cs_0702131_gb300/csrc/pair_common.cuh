// What the pair-force translation units share: kernel arguments, the striped
// sums, exact cut-off decisions and the packed words of the cluster kernels.
#pragma once

#include <math.h>

#include "aica_internal.cuh"

namespace aica {

constexpr int kParts = 16;           // accumulator row: U, W[6], counters[8]

struct SpeciesTab {
    float4 f[kMaxSpecies * kMaxSpecies];    // sigma^2, 24 eps, 4 eps, u(rc) for FP32
    double d[kMaxSpecies * kMaxSpecies][4]; // same in FP64
};

struct PairArgs {
    int C;
    const int *cell_off, *work_off;
    const WorkEntry *work;
    const int *run_off;
    const RunEntry *runs;
    const int *orgm;             // molecule-frame origins in units of 2^-10
    float Lhi[3], Llo[3];        // box lengths as float pairs (Lhi + Llo = L to ~1e-14)
    const float4 *xloc;
    const double *xs64;
    const float4 *sph;           // per-cell molecule bounding spheres (local frame)
    float rc2_lo, rc2_hi;
    float rc2_pre;               // cluster kernel: hi-part test threshold (margin above the remainders)
    double rc2_d;
    double L[3];
    int S;
    void *facc;                  // float4 (FP32) or double4 (FP64), binned order
    const void *vs;              // backward: grad_force in binned order (float4 / double4)
    double *acc;                 // [0..6] U, W; [8..15] counters (as unsigned long long); [16..] grads
    unsigned *next_cell;         // FP32 kernel: next unclaimed cell (zero at launch)
    int ghosts;                  // portion mode: xloc.w carries kGhostBit on halo molecules
    int xf;                      // general referring transforms: image field = transform index
    int n_xf;                    // transforms in xft
    const XfDev *xft;            // [n_xf] transforms (identity first)
    const float4 *run_d;         // general transforms: shift of each run in I's molecule frame
    SpeciesTab tab;
};

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

template <class R> struct R3 { R x, y, z; };

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// FP64 re-decision of r^2 < rc^2 with the all-pairs definition's operation order
static __device__ __noinline__ bool band_in(const PairArgs &a, int k, int l, int np) {
    const double *xk = a.xs64 + 3 * (size_t)k, *xl = a.xs64 + 3 * (size_t)l;
    double dx = __dsub_rn(__dsub_rn(xk[0], xl[0]), __dmul_rn(a.L[0], (double)unpack_n(np, 0)));
    double dy = __dsub_rn(__dsub_rn(xk[1], xl[1]), __dmul_rn(a.L[1], (double)unpack_n(np, 1)));
    double dz = __dsub_rn(__dsub_rn(xk[2], xl[2]), __dmul_rn(a.L[2], (double)unpack_n(np, 2)));
    double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return r2 < a.rc2_d;
}

// Sums of the pair kernels.  Every warp adds its totals (FP64 sums identical
// in all lanes; counters per lane) to one of kStripes rows of FP64
// accumulators (row = warp index mod kStripes, so few warps share an
// address); finish_sums adds the rows.  Row layout: [0..6] U and W,
// [7..14] the counters, exactly representable in FP64.
constexpr int kStripes = 64;
constexpr int kAccStripes = 64;        // offset of the rows in acc (doubles)

static __device__ void warp_to_stripe(const PairArgs &a, int gwarp, const double (&dsum)[7], const unsigned (&cv)[8],
                               int lane) {
    double *row = a.acc + kAccStripes + (size_t)(gwarp % kStripes) * kParts;
    for (int i = 0; i < 8; ++i) {
        const unsigned s = __reduce_add_sync(0xffffffffu, cv[i]);
        if (lane == 0 && s) atomicAdd(row + 7 + i, (double)s);
    }
    if (lane < 7) atomicAdd(row + lane, dsum[lane < 7 ? lane : 0]);
}

__device__ __forceinline__ void atomic_add3(double *p, double x, double y, double z) {
    atomicAdd(p, x);
    atomicAdd(p + 1, y);
    atomicAdd(p + 2, z);
}

// r = (x_k - x_l) - n.L with the all-pairs definition's rounding
__device__ __forceinline__ void sep64(const double *xk, const double *xl, const double *L, int np, double &rx,
                                      double &ry, double &rz, double &r2) {
    rx = __dsub_rn(__dsub_rn(xk[0], xl[0]), __dmul_rn(L[0], (double)unpack_n(np, 0)));
    ry = __dsub_rn(__dsub_rn(xk[1], xl[1]), __dmul_rn(L[1], (double)unpack_n(np, 1)));
    rz = __dsub_rn(__dsub_rn(xk[2], xl[2]), __dmul_rn(L[2], (double)unpack_n(np, 2)));
    r2 = __dadd_rn(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)), __dmul_rn(rz, rz));
}

// A binned molecule split at multiples of 2^-q: hi exact on the grid, lo the
// rest (xloc - hi is exact; adding the stored remainder rounds far below
// the separation's own rounding).  Valid for |x| < 2^(22 - q).
__device__ __forceinline__ void grid_split(float4 x, float4 r, float qr, float4 &hi, float4 &lo) {
    hi.x = __fsub_rn(__fadd_rn(x.x, qr), qr);
    hi.y = __fsub_rn(__fadd_rn(x.y, qr), qr);
    hi.z = __fsub_rn(__fadd_rn(x.z, qr), qr);
    hi.w = x.w;
    lo = make_float4(__fsub_rn(x.x, hi.x) + r.x, __fsub_rn(x.y, hi.y) + r.y, __fsub_rn(x.z, hi.z) + r.z, 0.f);
}

// Adjoint: slots [0, 8) of the stripe rows hold dL/d eps_s, [8, 16) dL/d sigma_s.
constexpr int kGradSlots = 2 * kMaxSpecies;
static_assert(kGradSlots <= kParts, "gradient slots must fit a stripe row");

struct BwdTab {
    double eps, sig2, inv_eps, inv_sig, fa, fb;   // fa, fb: d eps_ab / d eps_a, d eps_ab / d eps_b
};

// A warp's species-gradient totals (lane q < kGradSlots holds slot q) into its stripe row.
__device__ __forceinline__ void grads_to_stripe(const PairArgs &a, int gwarp, double g, int lane) {
    double *row = a.acc + kAccStripes + (size_t)(gwarp % kStripes) * kParts;
    if (lane < kGradSlots && g != 0.0) atomicAdd(row + lane, g);
}

// Arguments of the cluster kernels.
struct ClKArgs {
    const int *cl_first, *cl_run_off;
    const ClRun *runs;
    const float4 *xlo;
    float4 *cl_box;              // out: each cluster's box of molecules (lo, hi; hi parts, own frame)
    int ncl;
    float qround;                // 1.5 * 2^(23 - q): x + qround - qround rounds x to a multiple of 2^-q
};

// packed survivor / tile word (.w of the hi position)
constexpr int kSpBits = 7, kSameBit = 1 << 3, kImgBit = 1 << 4, kGhostW = 1 << 21;
__device__ __forceinline__ int cellq_of(int w) { return (w >> 5) & 15; }
__device__ __forceinline__ int32_t n_of(int w) {   // 3 x 4-bit image -> pack_n
    const int c = w >> 9;
    return pack_n((c << 28) >> 28, (c << 24) >> 28, (c << 20) >> 28);
}


// FP64 cluster kernels (pair64.cu): forces, energy, virial and counts, or
// the adjoint (t: pair terms of the species gradients).  False when they do
// not apply (sigma beyond the range of its 12th power); nothing is launched.
bool launch_fwd64c(const PairArgs &a, const ClKArgs &c, const aica_lj *lj, cudaStream_t st);
bool launch_bwd64c(const PairArgs &a, const ClKArgs &c, const aica_lj *lj, const BwdTab *t, cudaStream_t st);

}  // namespace aica
