// Building blocks of the FP64 cluster kernels (pair64.cu): a warp takes one cluster of
// cells (or one of `parts` shares of its candidates), collects the partner
// molecules that survive the cull against the cluster's box into a buffer in
// shared memory (cl_fill), tests them against the cluster's molecules with
// packed FP32 arithmetic into bit masks (cl_masks), orders them by their
// numbers of pairs (cl_balance), and lets each lane walk the mask of one
// survivor at a time, taking the next one when it is done (cl_pick).
//
// Why: of the distance tests that the cull leaves, 17 to 25 % are within the
// cut-off (a cell's box grown by rc against the sphere of radius rc).  A test
// here costs 4 issue slots (two tests per packed instruction, one funnel
// shift per test collects the sign of r^2 - rc^2), so the pair body runs only
// for the pairs within the cut-off, and with nearly all lanes busy.
#pragma once

#include "pair_common.cuh"

namespace aica {

// two FP32 values in one 64-bit register (sm_100 and later: one issue slot
// for two operations)
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

constexpr int kTile = 32;                 // molecules of the cluster per tile (bits of a mask; at most 32)

// Per-warp shared memory of the fill and test stages.
template <int CAP>
struct ClShare {
    float4 sh[CAP];           // survivor: position in A's frame (FP32), .w packed word
    float4 txy[kTile / 2];    // tile molecules 2p, 2p + 1: x, x', y, y'
    float2 tz[kTile / 2];     //   z, z'
    int tw[kTile];            //   packed word (species, cell label within the cluster) of molecule t
    float4 ed[32];            // live partner runs of the batch: shift (multiple of 2^-q), image code << 12
    int eb[32];               //   first molecule minus candidate position
    unsigned mask[CAP];       // tile molecules within reach of the survivor (bit order: cl_bit)
    unsigned cellm[16];       // tile molecules of each cell label (same bit order)
    int hist[33];               // survivors by number of pairs, then first position of each number
    float box[6];             // joint box of A's molecules (lo, hi)
    unsigned char ord[CAP];   // survivors by decreasing number of pairs
};

// Where the candidates of a cluster stand.
struct ClCursor {
    int own, s1;              // next own molecule, end of the own molecules
    int eb, e1;               // next batch of 32 partner runs, end of the runs
    int p0, total, inc;       // candidate position in the loaded runs
    int g;                    // share of the next group of 32 candidates
    unsigned culls;           // candidates tested
    bool live;
};

// Bounding box of A's molecules s0 .. s1 - 1 (FP32 positions) into w.box.
template <int CAP>
__device__ __forceinline__ void cl_box_of(const PairArgs &a, ClShare<CAP> &w, int s0, int s1, int lane) {
    const unsigned FULL = 0xffffffffu;
    float bl[3] = {1e30f, 1e30f, 1e30f}, bh[3] = {-1e30f, -1e30f, -1e30f};
    for (int k = s0 + lane; k < s1; k += 32) {
        const float4 x = a.xloc[k];
        bl[0] = fminf(bl[0], x.x); bl[1] = fminf(bl[1], x.y); bl[2] = fminf(bl[2], x.z);
        bh[0] = fmaxf(bh[0], x.x); bh[1] = fmaxf(bh[1], x.y); bh[2] = fmaxf(bh[2], x.z);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            bl[d] = fminf(bl[d], __shfl_xor_sync(FULL, bl[d], o));
            bh[d] = fmaxf(bh[d], __shfl_xor_sync(FULL, bh[d], o));
        }
    if (lane < 3) {
        w.box[lane] = lane == 0 ? bl[0] : lane == 1 ? bl[1] : bl[2];
        w.box[3 + lane] = lane == 0 ? bh[0] : lane == 1 ? bh[1] : bh[2];
    }
    __syncwarp();
}

// Append survivors until the buffer cannot take 32 more (returns true) or
// the cluster's candidates are used up (false): A's own molecules (their
// packed words carry kSameBit and the cell label), then the molecules of its
// partner runs, moved into A's frame and culled against A's box.  Group g of
// 32 candidates belongs to share g mod parts.  store(slot, l, xh): l the
// binned index, xh position and word.  Halo molecules (portion mode) are not marked.
template <int CAP, class Store>
__device__ __forceinline__ bool cl_fill(const PairArgs &a, const ClKArgs &c, ClShare<CAP> &w, ClCursor &q, int &nq,
                                        float rcut2, int part, int parts, int lane, Store store) {
    const unsigned FULL = 0xffffffffu, lt = (1u << lane) - 1u, le = FULL >> (31 - lane);
    while (nq <= CAP - 32) {
        if (q.own < q.s1) {
            if (q.g == part) {
                const int k = q.own + lane;
                const bool alive = k < q.s1;
                if (alive) {
                    float4 x = a.xloc[k];
                    const int w0 = __float_as_int(x.w), lab = __float_as_int(c.xlo[k].w) & 15;
                    x.w = __int_as_float((w0 & kSpBits) | kSameBit | (lab << 5));
                    store(nq + lane, k, x);
                }
                nq += min(32, q.s1 - q.own);
            }
            q.own += 32;
            if (++q.g == parts) q.g = 0;
        } else if (q.p0 < q.total) {
            if (q.g == part) {
                const int b = q.inc - q.p0;
                const int base = __popc(__ballot_sync(FULL, q.live && b <= 0));
                const unsigned M = __reduce_or_sync(FULL, (q.live && b > 0 && b < 32) ? (1u << b) : 0u);
                const int p = q.p0 + lane;
                bool alive = false;
                float4 xh = make_float4(0.f, 0.f, 0.f, 0.f);
                int l = 0;
                if (p < q.total) {
                    const int o = base + __popc(M & le);
                    l = p + w.eb[o];
                    const float4 dh = w.ed[o], x = a.xloc[l];
                    xh = make_float4(x.x + dh.x, x.y + dh.y, x.z + dh.z, 0.f);
                    const float dx = fmaxf(fmaxf(w.box[0] - xh.x, xh.x - w.box[3]), 0.f);
                    const float dy = fmaxf(fmaxf(w.box[1] - xh.y, xh.y - w.box[4]), 0.f);
                    const float dz = fmaxf(fmaxf(w.box[2] - xh.z, xh.z - w.box[5]), 0.f);
                    alive = dx * dx + dy * dy + dz * dz <= rcut2;
                    const int code = __float_as_int(dh.w) >> 12;
                    const int w0 = __float_as_int(x.w);
                    xh.w = __int_as_float((w0 & kSpBits) | (code != 0 ? kImgBit : 0) | (code << 9));
                }
                const unsigned bal = __ballot_sync(FULL, alive);
                if (alive) store(nq + __popc(bal & lt), l, xh);
                nq += __popc(bal);
                q.culls += (unsigned)min(32, q.total - q.p0);
            }
            q.p0 += 32;
            if (++q.g == parts) q.g = 0;
        } else if (q.eb < q.e1) {
            // the next 32 partner runs: candidate counts prefix-summed, live runs compacted
            int js = 0, n = 0;
            float4 dh = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q.eb + lane < q.e1) {
                const ClRun r = c.runs[q.eb + lane];
                const int cf = __float_as_int(r.dh.w), code = __float_as_int(r.dl.w);
                js = a.cell_off[cf];
                n = a.cell_off[cf + (code & 4095)] - js;
                dh = make_float4(r.dh.x, r.dh.y, r.dh.z, r.dl.w);
            }
            q.inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, q.inc, o);
                if (lane >= o) q.inc += y;
            }
            q.total = __shfl_sync(FULL, q.inc, 31);
            q.live = n > 0;
            const unsigned lbal = __ballot_sync(FULL, q.live);
            __syncwarp();                       // the previous runs' readers are done
            if (q.live) {
                const int sl = __popc(lbal & lt);
                w.ed[sl] = dh;
                w.eb[sl] = js - (q.inc - n);
            }
            __syncwarp();
            q.eb += 32;
            q.p0 = 0;
        } else {
            return false;
        }
    }
    return true;
}

// Load the tile's molecules k0 .. k0 + ni - 1 for the tests.  An odd tile is
// padded with a far-away molecule; bit cl_bit(t) of a mask stands for
// molecule t.  Returns the padded size.
template <int CAP>
__device__ __forceinline__ int cl_load_tile(const PairArgs &a, const ClKArgs &c, ClShare<CAP> &w, int k0, int ni,
                                            int lane) {
    const int ne = (ni + 1) & ~1;
    if (lane < 16) w.cellm[lane] = 0u;
    __syncwarp();
    if (lane < ne) {
        float4 x = make_float4(1e18f, 1e18f, 1e18f, 0.f);
        if (lane < ni) {
            x = a.xloc[k0 + lane];
            const int w0 = __float_as_int(x.w), lab = __float_as_int(c.xlo[k0 + lane].w) & 15;
            w.tw[lane] = (w0 & kSpBits) | (lab << 5);
            atomicOr(&w.cellm[lab], 1u << (ne - 1 - lane));
        }
        float *xy = (float *)&w.txy[lane >> 1];
        xy[lane & 1] = x.x;
        xy[2 + (lane & 1)] = x.y;
        ((float *)&w.tz[lane >> 1])[lane & 1] = x.z;
    }
    __syncwarp();
    return ne;
}

// Masks of the survivors 0 .. nq - 1 over the tile (ne molecules, padded):
// the tile molecules within reach, r^2 < pre2 on FP32 positions (a superset
// of the pairs within rc: pre2 covers the rounding of the positions).  Own
// molecules pair with tile molecules of lower binned index only (limit(j):
// binned index of an own survivor).  The per-lane counts of the pairs
// {same cell, all, images} go to n0, n1, n2.
template <int CAP, class Index>
__device__ __forceinline__ void cl_masks(ClShare<CAP> &w, int nq, int k0, int ne, float pre2, int lane, Index index,
                                         unsigned &n0, unsigned &n1, unsigned &n2) {
    const f32x2 neg = pack2(-pre2, -pre2);
    w.hist[lane] = 0;
    if (lane == 0) w.hist[32] = 0;
    __syncwarp();
    for (int jb = 0; jb < nq; jb += 32) {
        const int j = jb + lane;
        const float4 x = w.sh[min(j, nq - 1)];
        const f32x2 mx = pack2(-x.x, -x.x), my = pack2(-x.y, -x.y), mz = pack2(-x.z, -x.z);
        unsigned m = 0;
#pragma unroll 4
        for (int p = 0; p < (ne >> 1); ++p) {
            const float4 xy = w.txy[p];
            const float2 z = w.tz[p];
            const f32x2 rx = add2(pack2(xy.x, xy.y), mx), ry = add2(pack2(xy.z, xy.w), my),
                        rz = add2(pack2(z.x, z.y), mz);
            const f32x2 d = fma2(rz, rz, fma2(ry, ry, fma2(rx, rx, neg)));
            m = __funnelshift_l((unsigned)d, m, 1);                 // sign bits: r^2 < pre2
            m = __funnelshift_l((unsigned)(d >> 32), m, 1);
        }
        if (j < nq) {
            const int wj = __float_as_int(x.w);
            if (wj & kSameBit) {
                const int lim = min(max(index(j) - k0, 0), ne);     // tile molecules below the survivor
                m = lim > 0 ? m & (0xffffffffu << (ne - lim)) : 0u;
                n0 += __popc(m & w.cellm[cellq_of(wj)]);
            }
            const int n = __popc(m);
            n1 += n;
            if (wj & kImgBit) n2 += n;
            w.mask[j] = m;
            atomicAdd(&w.hist[n], 1);
        }
    }
    __syncwarp();
}

// Order the survivors with at least one pair by decreasing number of pairs
// (into w.ord); returns how many they are.
template <int CAP>
__device__ __forceinline__ int cl_balance(ClShare<CAP> &w, int nq, int lane) {
    const unsigned FULL = 0xffffffffu;
    // position of the first survivor with n pairs: survivors with more pairs
    const int h = w.hist[32 - lane];                       // lane i: survivors with 32 - i pairs
    int inc = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += y;
    }
    const int live = __shfl_sync(FULL, inc, 31);
    __syncwarp();
    w.hist[32 - lane] = inc - h;
    __syncwarp();
    for (int j = lane; j < nq; j += 32) {
        const int n = __popc(w.mask[j]);
        if (n) w.ord[atomicAdd(&w.hist[n], 1)] = (unsigned char)j;
    }
    __syncwarp();
    return live;
}

// One pair of the lane's mask m: the bit taken, 0 if none.  Lanes that are
// equal modulo kCols add to the same column of the tile's accumulators, so
// they take different molecules: each leaves alone what the lanes before it
// took.
constexpr int kCols = 8;                  // accumulator columns of a tile
__device__ __forceinline__ unsigned cl_pick(unsigned m, int lane) {
    unsigned bit = 0, used = 0;
#pragma unroll
    for (int g = 0; g < 32 / kCols; ++g) {
        const unsigned r = m & ~used, b = r & (0u - r);
        if (lane / kCols == g) bit = b;
        if (g + 1 < 32 / kCols) used |= __shfl_sync(0xffffffffu, b, (lane & (kCols - 1)) + kCols * g);
    }
    return bit;
}

}  // namespace aica
