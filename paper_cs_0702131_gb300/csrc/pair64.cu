// FP64 pair kernels over clusters: the forces (step a8-a9 in FP64) and their
// adjoint (a10) with box periodicity and minimum-distance lists.
//
// What bounds them: the FP64 pipe (GB300: one warp instruction per 16 cycles
// and SM, 1/64 of FP32), so the kernels spend FP32 and integer work to
// spend less FP64: every distance test runs in packed FP32 with margins
// (cluster.cuh), only the pairs within rc reach the FP64 body, and a lane
// always has one of them (the survivors are dealt out by their pair counts).
// A separation is formed as the all-pairs definition rounds it, three FP64
// subtractions (six for periodic images); 1/r^2 starts from the FP32 reciprocal and takes one step
// of the hyperpower iteration of order three (e = 1 - r^2 y; y + y (e + e^2), from a
// relative error below 2^-21 to below 2^-62 before the last rounding); conversions are done on the bit
// patterns, which would otherwise run on the FP64 pipe too; and the virial is
// the sum of x (x) F over the forces a warp hands out (x in the cluster's
// frame; each pair adds f and -f, so the origin cancels) instead of six products
// per pair.  A pair then carries an error of about 2^-53 |x| |f| where its virial is
// r (x) f, so pairs much closer than their coordinates (r < rc / 8; none in a
// fluid, some among overlapping molecules) hand out their force and
// r (x) f directly.
#include <algorithm>

#include "cluster.cuh"

namespace aica {
namespace {

constexpr int kCap64 = 224;          // survivors buffered per warp
constexpr int kW64 = 2;              // warps per block

// Pair parameters: f = (A / r^12 - B / r^6) r / r^2, u = C / r^12 - D / r^6 - ush;
// adjoint: E..H the multiples of A and B in its derivatives, and the chain
// factors of the species gradients.
struct Par64 {
    double A, B, C, D, ush, E, F, G, H, fa, fb, fs;
};
struct Tab64 {
    Par64 p[kMaxSpecies * kMaxSpecies];
};

template <bool BWD>
struct Warp64 : ClShare<kCap64> {
    double xd[3][kCap64];            // survivor: wrapped position of the molecule (without its image
                                     // shift), then its reaction (adjoint: position gradient)
    int sl[kCap64];                  //   its binned index
    double col[3][kTile][kCols];     // tile: forces by accumulator column
    double xi[3][kTile];             //   wrapped positions
    double sh64[3][16];              // n L for the image numbers n = -8 .. 7
    double vd[BWD ? 3 : 1][BWD ? kCap64 : 1];    // adjoint: v = dL/dF of the survivors
    double vi[BWD ? 3 : 1][BWD ? kTile : 1];     //   and of the tile
};

// Per-lane species sums of the adjoint with several species.
struct Slots64 {
    double s[kGradSlots][32];
};

// FP32 bits of a positive FP64 value in FP32's normal range (truncated), and
// back, on the integer units.
__device__ __forceinline__ float f32_of(int hi, int lo) {
    return __int_as_float(__funnelshift_l((unsigned)lo, (unsigned)(hi - 0x38000000), 3));
}
__device__ __forceinline__ double f64_of(float x) {
    const unsigned b = __float_as_uint(x);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// 1 / r2: exact division outside [2^-100, 2^100] (also 0, infinities and NaN)
__device__ __forceinline__ double recip64(double r2) {
    const int hi = __double2hiint(r2);
    if ((unsigned)(hi - ((1023 - 100) << 20)) >= (200u << 20)) return 1.0 / r2;
    const double y = f64_of(rcp_approx(f32_of(hi, __double2loint(r2))));
    double e = fma(-r2, y, 1.0);
    e = fma(e, e, e);
    return fma(y, e, y);
}

// r2 < rc^2 where the leading 20 bits decide it; otherwise the all-pairs
// operation order on the wrapped positions decides.  (r2 here is
// fused and differs from that order's by a few roundings.)
__device__ __forceinline__ bool within64(const PairArgs &a, double r2, int rc_hi, int k, int l, int wj) {
    const int h = __double2hiint(r2) - rc_hi;
    if ((unsigned)(h + 1) <= 2u) return band_in(a, k, l, n_of(wj));
    return h < 0;
}

// x (x) f added to the virial sums v[1..6] (xx, yy, zz, xy, xz, yz)
__device__ __forceinline__ void vir_add64(double (&v)[7], double x, double y, double z, double fx, double fy,
                                          double fz) {
    v[1] = fma(x, fx, v[1]);
    v[2] = fma(y, fy, v[2]);
    v[3] = fma(z, fz, v[3]);
    v[4] = fma(x, fy, v[4]);
    v[5] = fma(x, fz, v[5]);
    v[6] = fma(y, fz, v[6]);
}

// BWD: the adjoint.  acc[0], acc[1] then hold the sums of (r.w) g and
// (r.w) dg/d ln sigma for one species; several species use the lane's column
// of slots.
template <bool MULTI, bool SHIFT, bool BWD>
__global__ void __launch_bounds__(kW64 * 32) pair64c(PairArgs a, ClKArgs c, Tab64 T, int parts) {
    extern __shared__ __align__(16) unsigned char sh_raw[];
    static_assert(alignof(Warp64<BWD>) == 16 && sizeof(Warp64<BWD>) % 16 == 0 && alignof(Slots64) <= 16,
                  "the warps' shares are read with 16-byte loads");
    __shared__ Par64 tab[MULTI ? kMaxSpecies * kMaxSpecies : 1];
    if (MULTI)
        for (int i = threadIdx.x; i < kMaxSpecies * kMaxSpecies; i += blockDim.x) tab[i] = T.p[i];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    Warp64<BWD> &w = reinterpret_cast<Warp64<BWD> *>(sh_raw)[wib];
    double(*slots)[32] = nullptr;
    if (BWD && MULTI) {
        slots = reinterpret_cast<Slots64 *>(reinterpret_cast<Warp64<BWD> *>(sh_raw) + kW64)[wib].s;
        for (int i = 0; i < kGradSlots; ++i) slots[i][lane] = 0.0;
    }
    __syncthreads();
    const float pre2 = a.rc2_pre, rcut = sqrtf(pre2) * 1.00001f, rcut2 = rcut * rcut;
    const int rc_hi = __double2hiint(a.rc2_d);
    const int close_hi = rc_hi - (6 << 20);              // r^2 below about rc^2 / 64
    double *facc = (double *)a.facc;
    const double *vs = (const double *)a.vs;
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    unsigned n0 = 0, n1 = 0, n2 = 0, tests = 0, culls = 0;
    for (;;) {
        int u = lane == 0 ? (int)atomicAdd(a.next_cell, 1u) : 0;
        u = __shfl_sync(FULL, u, 0);
        if (u >= c.ncl * parts) break;
        const int A = u / parts, part = u - A * parts;
        const int c0 = c.cl_first[A], c1 = c.cl_first[A + 1];
        const int s0 = a.cell_off[c0], s1 = a.cell_off[c1], nA = s1 - s0;
        if (nA == 0) continue;
        cl_box_of(a, w, s0, s1, lane);
        for (int i = lane; i < 48; i += 32) {
            const int d = i >> 4, n = (i & 15) - 8;
            w.sh64[d][i & 15] = a.L[d] * (double)n;
        }
        double oA[3];
        for (int d = 0; d < 3; ++d) oA[d] = (double)a.orgm[3 * c0 + d] * (1.0 / 1024.0);
        ClCursor q{s0, s1, c.cl_run_off[A], c.cl_run_off[A + 1], 0, 0, 0, 0, 0u, false};
        const int ntile = (nA + kTile - 1) / kTile, wtile = (nA + ntile - 1) / ntile;
        for (bool more = true; more;) {
            int nq = 0;
            more = cl_fill(a, c, w, q, nq, rcut2, part, parts, lane, [&](int slot, int l, float4 xh) {
                w.sh[slot] = xh;
                w.sl[slot] = l;
            });
            if (nq == 0) break;
            __syncwarp();
            if (BWD)
                for (int j = lane; j < nq; j += 32)
#pragma unroll
                    for (int d = 0; d < 3; ++d) w.vd[d][j] = vs[4 * (size_t)w.sl[j] + d];
            for (int i0 = 0; i0 < nA; i0 += wtile) {
                const int ni = min(wtile, nA - i0), k0 = s0 + i0;
                const int ne = cl_load_tile(a, c, w, k0, ni, lane);
                for (int j = lane; j < nq; j += 32)
#pragma unroll
                    for (int d = 0; d < 3; ++d) w.xd[d][j] = a.xs64[3 * (size_t)w.sl[j] + d];
                if (lane < ni) {
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        w.xi[d][lane] = a.xs64[3 * (size_t)(k0 + lane) + d];
                        if (BWD) w.vi[d][lane] = vs[4 * (size_t)(k0 + lane) + d];
                    }
                }
                for (int i = lane; i < ni * kCols; i += 32)
#pragma unroll
                    for (int d = 0; d < 3; ++d) (&w.col[d][0][0])[i] = 0.0;
                cl_masks(w, nq, k0, ne, pre2, lane, [&](int j) { return w.sl[j]; }, n0, n1, n2);
                tests += (unsigned)(nq * ni);
                const int live = cl_balance(w, nq, lane);
                int next = 0, j = -1, l = 0, wj = 0;
                unsigned m = 0;
                double x = 0, y = 0, z = 0, fx = 0, fy = 0, fz = 0, vx = 0, vy = 0, vz = 0;
                for (;;) {
                    // idle lanes take the next survivors (those with most pairs come first)
                    const unsigned idle = __ballot_sync(FULL, m == 0);
                    if (idle == FULL && next >= live) break;
                    if (m == 0 && j >= 0) {
                        w.xd[0][j] = fx; w.xd[1][j] = fy; w.xd[2][j] = fz;
                        j = -1;
                    }
                    if (m == 0) {
                        const int slot = next + __popc(idle & lt);
                        if (slot < live) {
                            j = w.ord[slot];
                            m = w.mask[j];
                            l = w.sl[j];
                            wj = __float_as_int(w.sh[j].w);
                            x = w.xd[0][j]; y = w.xd[1][j]; z = w.xd[2][j];
                            fx = fy = fz = 0.0;
                            if (BWD) {
                                vx = w.vd[0][j]; vy = w.vd[1][j]; vz = w.vd[2][j];
                            }
                        }
                    }
                    next += __popc(idle);
                    __syncwarp();
                    const unsigned bit = cl_pick(m, lane);
                    m ^= bit;
                    if (bit) {
                        const int t = ne - 1 - (31 - __clz(bit));
                        double rx = w.xi[0][t] - x, ry = w.xi[1][t] - y, rz = w.xi[2][t] - z;
                        if (wj & kImgBit) {              // (x_k - x_l) - n L, as the all-pairs definition rounds it
                            rx -= w.sh64[0][((wj >> 9) + 8) & 15];
                            ry -= w.sh64[1][((wj >> 13) + 8) & 15];
                            rz -= w.sh64[2][((wj >> 17) + 8) & 15];
                        }
                        const double r2 = fma(rz, rz, fma(ry, ry, rx * rx));
                        if (within64(a, r2, rc_hi, k0 + t, l, wj)) {
                            const int spi = w.tw[t] & kSpBits, spj = wj & kSpBits;
                            const Par64 &P = MULTI ? tab[spi * kMaxSpecies + spj] : T.p[0];
                            const double inv = recip64(r2);
                            const double i6 = inv * inv * inv, i8 = i6 * inv;
                            const double t1 = fma(P.A, i6, -P.B), fs = i8 * t1;
                            double gx, gy, gz;           // force, or J w
                            if (BWD) {
                                const double wx = w.vi[0][t] - vx, wy = w.vi[1][t] - vy, wz = w.vi[2][t] - vz;
                                const double rw = fma(rz, wz, fma(ry, wy, rx * wx)), p = i8 * rw;
                                const double cc = (p * inv) * fma(P.E, i6, P.F);
                                const double t2 = fma(P.G, i6, P.H);
                                if (MULTI) {
                                    const double ea = t1 * p, sa = t2 * p * P.fs;
                                    slots[spi][lane] = fma(ea, P.fa, slots[spi][lane]);
                                    slots[spj][lane] = fma(ea, P.fb, slots[spj][lane]);
                                    slots[kMaxSpecies + spi][lane] += sa;
                                    slots[kMaxSpecies + spj][lane] += sa;
                                } else {
                                    acc[0] = fma(t1, p, acc[0]);
                                    acc[1] = fma(t2, p, acc[1]);
                                }
                                gx = fma(fs, wx, cc * rx);
                                gy = fma(fs, wy, cc * ry);
                                gz = fma(fs, wz, cc * rz);
                                fx -= gx;
                                fy -= gy;
                                fz -= gz;
                            } else {
                                acc[0] = fma(i6, fma(P.C, i6, -P.D), acc[0]);
                                if (SHIFT) acc[0] -= P.ush;
                            }
                            double *f = &w.col[0][t][lane & (kCols - 1)];
                            if (BWD) {
                                f[0] += gx;
                                f[kTile * kCols] += gy;
                                f[2 * kTile * kCols] += gz;
                            } else if (__double2hiint(r2) < close_hi) {
                                gx = fs * rx;
                                gy = fs * ry;
                                gz = fs * rz;
                                atomic_add3(facc + 4 * (size_t)(k0 + t), gx, gy, gz);
                                atomic_add3(facc + 4 * (size_t)l, -gx, -gy, -gz);
                                vir_add64(acc, rx, ry, rz, gx, gy, gz);
                            } else {
                                fx = fma(-fs, rx, fx);
                                fy = fma(-fs, ry, fy);
                                fz = fma(-fs, rz, fz);
                                f[0] = fma(fs, rx, f[0]);
                                f[kTile * kCols] = fma(fs, ry, f[kTile * kCols]);
                                f[2 * kTile * kCols] = fma(fs, rz, f[2 * kTile * kCols]);
                            }
                        } else {                         // inside the margin of the test, beyond rc
                            --n1;
                            if (wj & kImgBit) --n2;
                            if ((wj & kSameBit) && cellq_of(w.tw[t]) == cellq_of(wj)) --n0;
                        }
                    }
                    __syncwarp();
                }
                if (j >= 0) {
                    w.xd[0][j] = fx; w.xd[1][j] = fy; w.xd[2][j] = fz;
                }
                __syncwarp();
                // the tile's forces: sum the columns, then one molecule per lane
                for (int i = lane; i < 3 * ni; i += 32) {
                    double *f = &w.col[i % 3][i / 3][0];
                    double s = 0.0;
#pragma unroll
                    for (int e = 0; e < kCols; ++e) s += f[(e + lane) & (kCols - 1)];
                    f[0] = s;
                }
                __syncwarp();
                if (lane < ni) {
                    const double gx = w.col[0][lane][0], gy = w.col[1][lane][0], gz = w.col[2][lane][0];
                    atomic_add3(facc + 4 * (size_t)(k0 + lane), gx, gy, gz);
                    if (!BWD)
                        vir_add64(acc, w.xi[0][lane] - oA[0], w.xi[1][lane] - oA[1], w.xi[2][lane] - oA[2], gx, gy, gz);
                }
                // the survivors' reactions
                for (int j = lane; j < nq; j += 32) {
                    if (w.mask[j]) {
                        const double gx = w.xd[0][j], gy = w.xd[1][j], gz = w.xd[2][j];
                        atomic_add3(facc + 4 * (size_t)w.sl[j], gx, gy, gz);
                        if (!BWD) {
                            const int wj = __float_as_int(w.sh[j].w);
                            const double *x = a.xs64 + 3 * (size_t)w.sl[j];
                            double p[3] = {x[0] - oA[0], x[1] - oA[1], x[2] - oA[2]};
                            if (wj & kImgBit)
#pragma unroll
                                for (int d = 0; d < 3; ++d) p[d] += w.sh64[d][((wj >> (9 + 4 * d)) + 8) & 15];
                            vir_add64(acc, p[0], p[1], p[2], gx, gy, gz);
                        }
                    }
                }
                __syncwarp();
            }
            __syncwarp();
        }
        culls += q.culls;
    }
    const int gwarp = blockIdx.x * kW64 + wib;
    if constexpr (BWD) {
        double dg = 0.0;
        if (MULTI) {
            __syncwarp();
            if (lane < kGradSlots)
                for (int e = 0; e < 32; ++e) dg += slots[lane][(e + lane) & 31];
        } else {
            const double e = warp_sum(acc[0]) * T.p[0].fa, s = warp_sum(acc[1]) * T.p[0].fs;
            dg = lane == 0 ? e : lane == kMaxSpecies ? s : 0.0;
        }
        grads_to_stripe(a, gwarp, dg, lane);
    } else {
        double dsum[7];
        for (int i = 0; i < 7; ++i) dsum[i] = warp_sum(acc[i]);
        unsigned cv[8] = {0u, 0u, 0u, n0, n1 - n0 - n2, n2, lane == 0 ? tests : 0u, lane == 0 ? culls : 0u};
        warp_to_stripe(a, gwarp, dsum, cv, lane);
    }
}

// A persistent grid, every SM filled to its occupancy.  A cluster is shared
// between warps only when there are fewer clusters than resident warps: each
// share repeats the box, the tile and the column sums (256 000 molecules,
// 13 824 clusters: 0.50 ms whole, 0.64 in two shares, 1.02 in four).
template <bool MULTI, bool SHIFT, bool BWD>
void launch64c(const PairArgs &a, const ClKArgs &c, const Tab64 &T, cudaStream_t st) {
    static int cache[64] = {0};
    const size_t shm = (sizeof(Warp64<BWD>) + (BWD && MULTI ? sizeof(Slots64) : 0)) * kW64;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    if (!cache[dev]) {
        cudaFuncSetAttribute(pair64c<MULTI, SHIFT, BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pair64c<MULTI, SHIFT, BWD>, kW64 * 32, shm);
        cache[dev] = std::max(1, sms * std::max(1, per));
    }
    const int warps = cache[dev] * kW64;
    const int parts = std::max(1, std::min(8, warps / std::max(1, c.ncl)));
    const int grid = std::min(cache[dev], std::max(1, (c.ncl * parts + kW64 - 1) / kW64));
    pair64c<MULTI, SHIFT, BWD><<<grid, kW64 * 32, shm, st>>>(a, c, T, parts);
}

// The pair parameters; false when a 12th power of sigma leaves FP64's range.
bool fill_tab64(const PairArgs &a, const aica_lj *lj, Tab64 &T) {
    for (int i = 0; i < a.S; ++i)
        for (int j = 0; j < a.S; ++j) {
            const double e = sqrt(lj->eps[i] * lj->eps[j]), sg = 0.5 * (lj->sigma[i] + lj->sigma[j]);
            const double s6 = (sg * sg) * (sg * sg) * (sg * sg);
            Par64 &p = T.p[i * kMaxSpecies + j];
            p = Par64{};
            p.A = 48.0 * e * s6 * s6;
            p.B = 24.0 * e * s6;
            p.C = 4.0 * e * s6 * s6;
            p.D = 4.0 * e * s6;
            p.E = -14.0 * p.A;
            p.F = 8.0 * p.B;
            p.G = 12.0 * p.A;
            p.H = -6.0 * p.B;
            p.ush = a.tab.d[i * kMaxSpecies + j][3];
            if (!(sg > 1e-16 && sg < 1e16 && e < 1e60 && (e == 0.0 || e > 1e-60))) return false;
        }
    return true;
}

}  // namespace

bool launch_fwd64c(const PairArgs &a, const ClKArgs &c, const aica_lj *lj, cudaStream_t st) {
    Tab64 T{};       // zero where a species has no parameters: such pairs carry nothing
    if (!fill_tab64(a, lj, T)) return false;
    if (a.S > 1) {
        if (lj->shift) launch64c<true, true, false>(a, c, T, st);
        else launch64c<true, false, false>(a, c, T, st);
    } else {
        if (lj->shift) launch64c<false, true, false>(a, c, T, st);
        else launch64c<false, false, false>(a, c, T, st);
    }
    return true;
}

bool launch_bwd64c(const PairArgs &a, const ClKArgs &c, const aica_lj *lj, const BwdTab *t, cudaStream_t st) {
    Tab64 T{};       // zero where a species has no parameters: such pairs carry nothing
    if (!fill_tab64(a, lj, T)) return false;
    for (int i = 0; i < a.S; ++i)
        for (int j = 0; j < a.S; ++j) {
            const BwdTab &b = t[i * kMaxSpecies + j];
            Par64 &p = T.p[i * kMaxSpecies + j];
            p.fa = b.fa * b.inv_eps;
            p.fb = b.fb * b.inv_eps;
            p.fs = 0.5 * b.inv_sig;
        }
    if (a.S == 1) {                  // one species: both molecules of a pair count
        T.p[0].fa = t[0].inv_eps;
        T.p[0].fs = t[0].inv_sig;
    }
    if (a.S > 1) launch64c<true, false, true>(a, c, T, st);
    else launch64c<false, false, true>(a, c, T, st);
    return true;
}

}  // namespace aica
