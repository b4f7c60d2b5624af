// Short-range particle-particle force (paper Sec. 2.2.3 and Eq. PP):
//   F_i += V_p / (4 pi) (R(r, b_pp) - R(r, b_range)) (x_j - x_i) / r,   0 < r < b_range,
// with R(r, b) of Eq. (refforce).  The IOS order is the cell list (Sec. 2.3): the
// IOS cell is at least b_range wide, so the 27 cells around a particle's cell
// hold all its partners.  The cells of one (dz, dy) row are adjacent in memory,
// so a run of cells along x is one contiguous particle range.
//
// The plain and the persistent kernel (and the counting ones) give the same bits:
// products and sums that could be contracted are written as fmaf or kept apart.
//
// Arithmetic is carried out in IOS-cell units.  A particle's in-cell offset
// off/2^16 is exact in FP32 (prep kernel, once per force evaluation) and so is
// (cell step + offset) and the separation of two such values: the pair term is
// bitwise antisymmetric.  Each ordered pair is evaluated from both sides (gather
// form, no atomics, deterministic).
//
// One thread per target.  Targets are taken in pencil order (pp_pencil_kernel),
// so that the 32 of a warp lie in a compact block of cells at any density; the
// particles of dense cells (64 or more) are reordered by a 4x4x4 sub-cell key
// inside their cell (PP's own position array and slot -> particle map; results
// are written back to the particle's index).  A warp shares one source stream:
// the particles of the cells within one of its block, staged by one lane each
// and dropped where they are out of reach of the targets' bounding box.
// Compact warps evaluate every pair of target and kept source; others test all
// of them (packed arithmetic) and evaluate the ones found in range from a queue
// per lane.  The few warps spread along x (nearly empty regions) walk each
// lane's own 27 cells.  Long streams of small boxes are shared by eight warps in a
// second kernel.  The adjoint's Jacobian product (pp_vjp_kernel) uses the same stream.
//
// 256^3 run, a step's PP at z = 49 / z = 1 / z = 0: 1.35 / 5.0 / 8.7 ms;
// with the targets in IOS order (streams only for warps inside one row, the
// 27-cell walk for all others) 1.39 / 7.4 / 13.4 ms.
// Per-particle sums are compensated: plain FP32 partials per batch are added to
// the running total with Kahan's scheme.  The path a warp takes depends only
// on the cell layout and every sum has a fixed order, so results are bitwise
// reproducible.
#include "common.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>

namespace cube2 {
namespace {

// Counters of one PP evaluation (zeroed before it).
struct PPWork {
    int dense;          // cells reordered by sub-cell
    unsigned places;    // target places in use
    int crowd;          // targets with long streams, by the cells around them
    int n;              // warps with long streams, listed
};

struct PPParams {
    const float4 *pos;          // [N] (off_x, off_y, off_z)/2^16, .w = cell id bits, in PP slot order
    const int32_t *perm;        // [N] particle index of each slot
    const int32_t *tgt;         // slot of each target, pencil by pencil, padded to whole warps with -1
    PPWork *work;
    const int32_t *count, *start;
    float *acc0, *acc1, *acc2;
    float *vel0, *vel1, *vel2;
    unsigned long long *stats;  // [4]: in-range ordered pairs, candidates; the same of per-lane walks
    int n_ios, accumulate;
    unsigned div_mul;           // c / n_ios = umulhi(c, div_mul) >> div_shift for 0 <= c < 2^31
    int div_shift;
    float inv_bpp, inv_bcut, bcut2, bpp2;   // IOS-cell units
    float ratio2;                     // 1 / b_pp^2, IOS-cell units
    float coef;                       // V_p / (4 pi s_ios^2)
    float kick;                       // 0: no kick; else v += kick * acc after the sum
    int *status;
    // adaptive third level: targets in a refined subtile (pm3_slot >= 0) use
    // the range b_3 (bcut2_3, inv_bcut_3) instead of b_cut; null when off
    const int32_t *pm3_slot;
    int pm3_T, pm3_ns;
    float bcut2_3, inv_bcut_3;
    bool even;                        // dense throughout (pp_compact)
    int long_min;                     // longer streams go to the list and are shared by PP_PARTS warps
    int32_t *long_list;               // target places / 32 of those warps
    int long_crowd;                   // most targets with long streams with which that is done
};

// R(r, b) of Eq. (refforce) times b^2, as a function of u = r / b < 1.
__device__ __forceinline__ float ref_force_scaled(float u) {
    if (u < 0.5f) {
        // 64/5 u - 256/5 u^3 + 32 u^4 + 1536/35 u^5 - 192/5 u^6
        return u * (64.0f / 5.0f + u * u * (-256.0f / 5.0f + u * (32.0f + u * (1536.0f / 35.0f - 192.0f / 5.0f * u))));
    }
    // 3/(35 u^2) - 32/5 + 256/5 u - 96 u^2 + 256/5 u^3 + 32 u^4 - 1536/35 u^5 + 64/5 u^6
    const float poly = -32.0f / 5.0f + u * (256.0f / 5.0f + u * (-96.0f + u * (256.0f / 5.0f + u * (32.0f + u * (-1536.0f / 35.0f + 64.0f / 5.0f * u)))));
    return 3.0f / (35.0f * u * u) + poly;
}

__device__ __forceinline__ void kahan_add(float &sum, float &comp, float v) {
    const float y = __fsub_rn(v, comp);   // v is never contracted into the difference
    const float t = __fadd_rn(sum, y);
    comp = __fsub_rn(__fsub_rn(t, sum), y);
    sum = t;
}

__device__ __forceinline__ void finish(const PPParams &P, int64_t i, float a0, float a1, float a2) {
    if (P.accumulate) {
        a0 += P.acc0[i];
        a1 += P.acc1[i];
        a2 += P.acc2[i];
    }
    P.acc0[i] = a0;
    P.acc1[i] = a1;
    P.acc2[i] = a2;
    if (P.kick != 0.0f) {
        const float v0 = fmaf(P.kick, a0, P.vel0[i]);
        const float v1 = fmaf(P.kick, a1, P.vel1[i]);
        const float v2 = fmaf(P.kick, a2, P.vel2[i]);
        P.vel0[i] = v0;
        P.vel1[i] = v1;
        P.vel2[i] = v2;
        if (!isfinite(v0) || !isfinite(v1) || !isfinite(v2)) set_status(P.status, ST_NONFINITE);
    } else if (!isfinite(a0) || !isfinite(a1) || !isfinite(a2)) {
        set_status(P.status, ST_NONFINITE);
    }
}

__device__ __forceinline__ void add_stats(unsigned long long *stats, unsigned long long pairs,
                                          unsigned long long cands) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        cands += __shfl_xor_sync(0xffffffffu, cands, o);
    }
    if ((threadIdx.x & 31) == 0 && (pairs | cands)) {
        atomicAdd(&stats[0], pairs);
        atomicAdd(&stats[1], cands);
    }
}


// The particles of the three cells (x-1, x, x+1) of row r as at most two
// contiguous ranges; dx of particle j in range k is base[k] + (j >= b1[k]) + (j >= b2[k]).
struct RowRanges {
    int beg[2], end[2], b1[2], b2[2], base[2];
    int nseg;
    __device__ __forceinline__ RowRanges(const PPParams &P, int64_t r, int cx, int n) {
        const int BIG = 0x7fffffff;
        if (cx > 0 && cx < n - 1) {
            nseg = 1;
            beg[0] = P.start[r + cx - 1];
            b1[0] = P.start[r + cx];
            b2[0] = P.start[r + cx + 1];
            end[0] = b2[0] + P.count[r + cx + 1];
            base[0] = -1;
        } else if (cx == 0) {
            nseg = 2;
            beg[0] = P.start[r];
            b1[0] = P.start[r + 1];
            b2[0] = BIG;
            end[0] = b1[0] + P.count[r + 1];
            base[0] = 0;
            beg[1] = P.start[r + n - 1];
            end[1] = beg[1] + P.count[r + n - 1];
            b1[1] = b2[1] = BIG;
            base[1] = -1;
        } else {
            nseg = 2;
            beg[0] = P.start[r + n - 2];
            b1[0] = P.start[r + n - 1];
            b2[0] = BIG;
            end[0] = b1[0] + P.count[r + n - 1];
            base[0] = -1;
            beg[1] = P.start[r];
            end[1] = beg[1] + P.count[r];
            b1[1] = b2[1] = BIG;
            base[1] = 1;
        }
    }
    __device__ __forceinline__ int size() const { return (end[0] - beg[0]) + (nseg > 1 ? end[1] - beg[1] : 0); }
};

constexpr int PP_ITEM = 128;                                // target places of a persistent work item
constexpr int PREP_WARPS = 4, PREP_CTA = PREP_WARPS * 32;   // input kernels

// Targets are taken in pencil order: the cells of a pencil (PEN_Y x PEN_Z cells
// in y and z, all of x) slab by slab along x, so that 32 consecutive targets
// lie in a compact block at any density (8 x 2 x 2 cells at one particle per
// cell, one cell where it holds 32) and one source stream per warp is short: 98
// sources in reach of the block at one particle per cell.  2 x 2 against 4 x 2
// cells: 1.35 against 1.68 ms at z = 49 (the block's eight x cells in a row make
// its loads and stores whole sectors), equal late; 2 x 1: 1.50.  Each pencil
// starts on a whole warp (its tail is padded with -1): a warp never spans two.
constexpr int PEN_Y = 2, PEN_Z = 2, PEN = PEN_Y * PEN_Z;

constexpr int PP_ROWS = (PEN_Y + 2) * (PEN_Z + 2);   // rows of cells that a warp's targets see

// A warp in a halo has a stream of thousands of sources and works on it long after
// the rest of a small box is done.  Streams longer than PPParams.long_min are put on a
// list and shared by the PP_PARTS warps of a CTA in a second kernel; the partial sums
// are added in their order, so the result does not depend on which path (the
// ensemble's persistent kernel works on the parts one after another) computed them.
//
// Splitting repeats the staging in every part and starts after the first kernel: it
// pays while a few long warps outlive the others, that is in small boxes and where the
// long warps would not fill the chip by themselves.  PP with / without, 64^3 particles
// 20 % or 40 % in haloes (600 and 1300 long warps): 0.23 / 0.30 and 0.34 / 0.44 ms;
// 500000 in 32^3 cells, 262144 in 24^3 or a tenth of 64^3 cells, all evenly (8000 to
// 16000): 0.63 / 0.39, 0.40 / 0.27 and 0.27 / 0.19 ms.  96^3 particles, 20 % or 55 %
// in haloes: 0.49 / 0.50 and 0.87 / 0.82 ms, larger boxes less.  The limit of 512
// against 1024 and 2048: 0.22 / 0.25 / 0.33 ms (64^3, 20 % in haloes).  The adjoint's
// pairs cost several times more: two products of 128^3 particles, 10 % or 40 % in
// haloes, 2.07 / 2.20 and 4.06 / 3.82 ms.  4 or 16 parts are no better than 8.
// What decides is counted from the cells before the first warp runs (pp_pencil_kernel),
// so that every launch of a state decides the same.
constexpr int PP_PARTS = 8;
constexpr int PP_UNSPLIT = 0x7fffffff;
constexpr int64_t PP_LONG_N = 65536;    // smaller boxes: the second launch costs more than it gives

constexpr int LONG_SLAB = 8;            // targets of a pencil's slab of cells from which its streams are looked at

inline int pp_long_min(int64_t N) { return N < PP_LONG_N || N >= (1 << 19) ? PP_UNSPLIT : 512; }
inline int vjp_long_min(int64_t N) { return N < PP_LONG_N || N >= (1 << 22) ? PP_UNSPLIT : N < (1 << 20) ? 512 : (int)(N / 2048); }

__host__ __device__ __forceinline__ int pencils_y(int n) { return (n + PEN_Y - 1) / PEN_Y; }
__host__ __device__ __forceinline__ int pencils_z(int n) { return (n + PEN_Z - 1) / PEN_Z; }

// One CTA per pencil: the target places of its cells (cells of sort_min
// particles or more are listed with their first place for pp_dense_sort_kernel,
// which writes them with a warp each) and the padding of the pencil's tail.
// Pencils take their places in tgt by an atomic on their number: their order varies,
// the warps of a pencil and so the results do not.  LONG: counts the targets whose
// streams are longer than long_min, about.
template <bool LONG>
__global__ void __launch_bounds__(PREP_CTA) pp_pencil_kernel(const int32_t *__restrict__ count,
                                                             const int32_t *__restrict__ start, int n, int sort_min,
                                                             int long_min, int32_t *__restrict__ tgt,
                                                             int2 *__restrict__ list, PPWork *work) {
    __shared__ unsigned s_base;   // places are unsigned: N plus the padding may pass 2^31
    __shared__ int s_warp[PREP_WARPS];
    const int npy = pencils_y(n);
    const int y0 = (int)(blockIdx.x % npy) * PEN_Y, z0 = (int)(blockIdx.x / npy) * PEN_Z;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // cell k of a slab: y forwards in the first z plane, backwards in the second
    auto row_of = [&](int k) -> int64_t {
        const int z = z0 + k / PEN_Y, y = y0 + (k < PEN_Y ? k : PEN - 1 - k);
        return (y < n && z < n) ? ((int64_t)z * n + y) * n : -1;
    };
    if (w == 0) {   // a row's particles are contiguous
        const int64_t r = lane < PEN ? row_of(lane) : -1;
        int total = r >= 0 ? start[r + n - 1] + count[r + n - 1] - start[r] : 0;
        total = __reduce_add_sync(0xffffffffu, total);
        const int padded = (total + 31) & ~31;
        unsigned base = 0;
        if (lane == 0 && padded) base = atomicAdd(&work->places, (unsigned)padded);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (lane < padded - total) tgt[base + total + lane] = -1;
        if (lane == 0) s_base = base;
    }
    __syncthreads();
    unsigned run = s_base;
    for (int xb = 0; xb < n; xb += PREP_CTA) {
        const int x = xb + threadIdx.x;
        int cnt[PEN], sum = 0;
#pragma unroll
        for (int k = 0; k < PEN; ++k) {
            const int64_t r = row_of(k);
            cnt[k] = (x < n && r >= 0) ? count[r + x] : 0;
            sum += cnt[k];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_warp[w] = incl;
        __syncthreads();
        unsigned at = run + incl - sum;
#pragma unroll
        for (int k = 0; k < PREP_WARPS; ++k) {
            if (k < w) at += s_warp[k];
            run += s_warp[k];
        }
        __syncthreads();
        if (LONG) {   // a stream: the rows around the pencil's, over the slabs of 32 targets and one on each side
            // thinner slabs hold few of the targets with long streams, and a nearly empty box hundreds of slabs
            // for each particle (10^5 evenly in 192^3 cells with them counted: PP 0.094 ms instead of 0.07)
            int near = 0;
            if (sum >= LONG_SLAB) {
#pragma unroll 4
                for (int k = 0; k < PP_ROWS; ++k) {
                    const int64_t r = ((int64_t)wrap(z0 - 1 + k / (PEN_Y + 2), n) * n + wrap(y0 - 1 + k % (PEN_Y + 2), n)) * n;
                    near += count[r + wrap(x - 1, n)] + count[r + x] + count[r + wrap(x + 1, n)];
                }
                near += (int)((int64_t)near * 32 / (3 * sum));
            }
            const int crowd = __reduce_add_sync(0xffffffffu, near > long_min ? sum : 0);
            if (lane == 0 && crowd) atomicAdd(&work->crowd, crowd);
        }
#pragma unroll
        for (int k = 0; k < PEN; ++k) {
            const int64_t r = row_of(k);
            if (x < n && r >= 0) {
                if (cnt[k] >= sort_min) {
                    list[atomicAdd(&work->dense, 1)] = make_int2((int)(r + x), (int)at);
                } else if (cnt[k]) {
                    const int st = start[r + x];
                    for (int j = 0; j < cnt[k]; ++j) tgt[at + j] = st + j;
                }
                at += cnt[k];
            }
        }
    }
}

// Float offsets (and the cell id bits) for the PP kernel.
__global__ void __launch_bounds__(PREP_CTA) prep_positions_kernel(const uint16_t *off0, const uint16_t *off1,
                                                                const uint16_t *off2, const int32_t *cellid,
                                                                float4 *pos, int32_t *perm, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float s = 1.0f / FIX;
    pos[i] = make_float4((float)off0[i] * s, (float)off1[i] * s, (float)off2[i] * s, __int_as_float(cellid[i]));
    perm[i] = (int32_t)i;
}

// Dense cells are reordered for PP by a 4x4x4 sub-cell key (Morton order of
// the top two offset bits per axis), stably: a warp's targets then lie close
// together and have similar neighbour counts, so set-bit evaluation wastes
// fewer lanes (measured 5 % off PP at z ~ 0).  Only PP's own arrays are
// reordered (pos4 and the slot -> particle map); the particle arrays are not.
constexpr int PP_SORT_MIN = 64;   // cells with fewer particles keep their order

__device__ __forceinline__ int subcell_key(unsigned ox, unsigned oy, unsigned oz) {
    const unsigned x = ox >> 14, y = oy >> 14, z = oz >> 14;   // two bits each
    return (int)((((x >> 1) | ((y >> 1) << 1) | ((z >> 1) << 2)) << 3) | ((x & 1) | ((y & 1) << 1) | ((z & 1) << 2)));
}

// One warp per listed cell: histogram of the 64 keys, exclusive scan, then a
// stable scatter 32 particles at a time (rank among equal keys of the chunk
// by match masks, chunks in order).
__global__ void __launch_bounds__(256) pp_dense_sort_kernel(const uint16_t *off0, const uint16_t *off1,
                                                            const uint16_t *off2, const int32_t *count,
                                                            const int32_t *start, const int2 *list, const int *list_n,
                                                            float4 *pos, int32_t *perm, int32_t *tgt) {
    chain();
    __shared__ int hist[8][64], run[8][64];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nwarps_total = gridDim.x * (blockDim.x >> 5);
    const int nl = *list_n;
    const float s = 1.0f / FIX;
    for (int li = blockIdx.x * (blockDim.x >> 5) + w; li < nl; li += nwarps_total) {
        const int c = list[li].x;
        const unsigned place = (unsigned)list[li].y;
        const int st = start[c], cnt = count[c];
        for (int j = lane; j < cnt; j += 32) tgt[place + j] = st + j;
        hist[w][lane] = 0;
        hist[w][lane + 32] = 0;
        __syncwarp();
        for (int j = lane; j < cnt; j += 32)
            atomicAdd(&hist[w][subcell_key(off0[st + j], off1[st + j], off2[st + j])], 1);
        __syncwarp();
        // exclusive scan of 64 bins: lane holds bins 2 lane, 2 lane + 1
        const int h0 = hist[w][2 * lane], h1 = hist[w][2 * lane + 1];
        int incl = h0 + h1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int ex = incl - h0 - h1;
        run[w][2 * lane] = ex;
        run[w][2 * lane + 1] = ex + h0;
        __syncwarp();
        for (int j0 = 0; j0 < cnt; j0 += 32) {
            const int j = j0 + lane;
            const bool ok = j < cnt;
            const unsigned act = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const unsigned o0 = off0[st + j], o1 = off1[st + j], o2 = off2[st + j];
                const int k = subcell_key(o0, o1, o2);
                const unsigned peers = __match_any_sync(act, k);
                const int rank = __popc(peers & ((1u << lane) - 1u));
                const int slot = run[w][k] + rank;
                __syncwarp(act);
                if (rank == 0) run[w][k] += __popc(peers);
                pos[st + slot] = make_float4((float)o0 * s, (float)o1 * s, (float)o2 * s, __int_as_float(c));
                perm[st + slot] = st + j;
            }
            __syncwarp();
        }
    }
}

// Compensated sum of three components: terms are added plainly into a block
// partial (a tile or a row of candidates), and each block partial is added to
// the running total with Kahan compensation.
struct Sum3 {
    float x = 0.f, y = 0.f, z = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    __device__ __forceinline__ void add_block(float bx, float by, float bz) {
        kahan_add(x, cx, bx);
        kahan_add(y, cy, by);
        kahan_add(z, cz, bz);
    }
};

// Sources of a warp whose targets lie in cells [xa, xb] x [ya, yb] x [za, zb] of
// one pencil: for each row of the block one cell larger on every side, the
// cells xa-1 .. xb+1 as a main range and, at the box's faces, the wrapped cell
// on the left and on the right, flattened into one stream of the non-empty
// ranges.  Positions p from begin[s] on are slots p + seg[s].x; a source's
// coordinates in the warp's frame (cell (xa, ya - 1, za - 1) at 0) are (cell id
// - seg[s].y) + off_x, row_y + off_y, row_z + off_z with the row's offsets as
// floats in seg[s].z and .w: exact in FP32, and so are their differences, while they
// are below 256 cells.
constexpr int PP_SEGS = 3 * PP_ROWS;

// A warp is on the shared stream when it spans at most PP_WIDEST + 1 cells along x, as
// far as its frame is exact; the few wider ones (fewer than 32 particles in that many
// slabs) walk each lane's own 27 cells.  A lane of a halo at the end of a wide warp
// walks alone: 70000 particles in 96^3 cells, half of them in 64 clumps, 0.21 ms with
// streams of up to 65 cells, now 0.16; 10^6 evenly in 256^3 cells 0.24 -> 0.22.  The line
// is the same for every launch: the two paths add in different orders, and an ensemble
// gives its boxes the bits of their own steps.
constexpr int PP_WIDEST = 250;

struct PPBlock {
    int xa, xb, ya, yb, za, zb;
};

// Staged sources by component, so that a 16-byte load brings two packed pairs.
template <int N>
struct Soa {
    float x[N], y[N], z[N];
    __device__ __forceinline__ void put(int i, float4 q) {
        x[i] = q.x;
        y[i] = q.y;
        z[i] = q.z;
    }
};

constexpr int OUTER_N = 64;             // sources evaluated at a time, no pair of them closer than half the range
constexpr int MIXED_N = 32;             // sources evaluated at a time, any distance
constexpr int SPARSE_N = 128;           // sources tested before the pairs found are evaluated
constexpr int QUEUE_N = 32;             // pairs a lane can hold

struct alignas(16) PPWarpShared {
    union {
        struct {
            Soa<OUTER_N + 32> outer;
            Soa<MIXED_N + 32> mixed;
        } d;
        struct {
            Soa<SPARSE_N + 4> src;
            unsigned char queue[QUEUE_N][32];
        } s;
    } u;
    int4 seg[PP_SEGS];
    int begin[PP_SEGS];
    // bounding box of the warp's targets: (lo x, y, z, largest squared range), (hi x, y, z, where the outer half begins)
    float4 box[2];
};

__device__ __forceinline__ float4 frame_position(float4 q, int4 g) {
    return make_float4((float)(__float_as_int(q.w) - g.y) + q.x, q.y + __int_as_float(g.z), q.z + __int_as_float(g.w),
                       0.0f);
}

// padding sources: out of range of every target, and no overflow in the pair formula
constexpr float PP_FAR = 4096.0f;

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// Build the warp's segment table; returns the stream length.
__device__ __forceinline__ int build_segments(const PPParams &P, int4 *seg, int *begin, const PPBlock &B, int &nseg) {
    const int lane = threadIdx.x & 31;
    const int n = P.n_ios;
    const int ny = B.yb - B.ya + 3, rows = ny * (B.zb - B.za + 3);
    const int rz = lane / ny, ry = lane - rz * ny;
    const int rb = lane < rows ? (wrap(B.za - 1 + rz, n) * n + wrap(B.ya - 1 + ry, n)) * n : 0;
    int run = 0;
    nseg = 0;
#pragma unroll 1
    for (int g = 0; g < 3; ++g) {
        if ((g == 1 && B.xa > 0) || (g == 2 && B.xb < n - 1)) continue;
        int beg = 0, len = 0, adj = rb + B.xa;
        if (lane < rows) {
            if (g == 0) {
                const int lo = max(B.xa - 1, 0), hi = min(B.xb + 1, n - 1);
                beg = P.start[rb + lo];
                len = P.start[rb + hi] + P.count[rb + hi] - beg;
            } else {
                const int c = g == 1 ? rb + n - 1 : rb;
                beg = P.start[c];
                len = P.count[c];
                adj += g == 1 ? n : -n;
            }
        }
        if (len > 0) {   // its first sources on their way before the stream comes to them
            prefetch_l1(&P.pos[beg]);
            if (len > 1) prefetch_l1(&P.pos[beg + min(len, 16) - 1]);
        }
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const unsigned full = __ballot_sync(0xffffffffu, len > 0);
        const int at = run + incl - len;
        if (len > 0) {
            const int k = nseg + __popc(full & ((1u << lane) - 1u));
            begin[k] = at;
            seg[k] = make_int4(beg - at, adj, __float_as_int((float)ry), __float_as_int((float)rz));
        }
        run += __shfl_sync(0xffffffffu, incl, 31);
        nseg += __popc(full);
    }
    __syncwarp();
    return run;
}

// ------------------------------------------------------------ pair factor
// R_PP(r)/r of a pair with b_pp <= r < b_cut (Eq. PP) in units of 1/b_cut^3, as
// a function of u^2 = (r / b_cut)^2.  Where r >= b_pp the first term of R_PP is
// 1/r^2 and R_PP(r)/r = m(u)/u^3: the outer shell of Eq. (refforce) gives
//   u >= 1/2: m = (1-u)^5 q(u), q = 32/35 + 32/7 u + 704/35 u^2 + 64/5 u^3
//             (an exact polynomial shift, free of cancellation near the cutoff),
//             so m/u^3 = t^5 u^2 q(u) with t = 1/u - 1, zero beyond the cutoff
//             where t is clamped at 0;
//   u < 1/2:  m = 1 - 64/5 u^3 + 256/5 u^5 - 32 u^6 - 1536/35 u^7 + 192/5 u^8.
// u^2 is 0 or at least 2^-32, so the flush of denormals never acts.
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr float Q0 = 32.0f / 35.0f, Q1 = 32.0f / 7.0f, Q2 = 704.0f / 35.0f, Q3 = 64.0f / 5.0f;
constexpr float I0 = -64.0f / 5.0f, I2 = 256.0f / 5.0f, I3 = -32.0f, I4 = -1536.0f / 35.0f, I5 = 192.0f / 5.0f;

// R(r, b)/r of Eq. (refforce) in units of 1/b^3 at x = r/b <= 1.
__device__ __forceinline__ float soft_factor(float x2) {
    const float xinv = rsqrt_ftz(x2);
    const float x = x2 * xinv;
    if (x2 < 0.25f) return -fmaf(fmaf(fmaf(fmaf(I5, x, I4), x, I3), x, I2), x2, I0);
    const float t = __saturatef(xinv - 1.0f);
    const float a = t * t * x;
    return fmaf(-(a * a * t), fmaf(fmaf(fmaf(Q3, x, Q2), x, Q1), x, Q0), xinv * xinv * xinv);
}

// R_PP(r)/r for 0 < r < b_pp, same units as the far factor: both terms of Eq.
// PP are softened.  ratio2 = (b_cut/b_pp)^2.
__device__ __forceinline__ float close_factor(float u2, float ratio2) {
    return fmaf(ratio2 * sqrtf(ratio2), soft_factor(u2 * ratio2), -soft_factor(u2));
}

// Two FP32 values in one 64-bit register pair (packed FP32 arithmetic: the rate
// of the FMA pipe is that of two scalar instructions, the issue slots are
// those of one).
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack(f2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 twice(float a) { return pack(a, a); }

// A target as the pair loops see it.
struct PPLane {
    float mx, my, mz;        // position in the warp's frame
    float bcut2, ib2;        // range^2, 1/range^2 [IOS cells]
    float coef;              // of the sums: V_p/(4 pi s^2) / range^3
    bool has;
};

// The far factor of two pairs (OUTER: both at u >= 1/2 or out of range).
template <bool OUTER>
__device__ __forceinline__ f2 far_factor2(f2 u2) {
    float ua, ub;
    unpack(u2, ua, ub);
    const float ia = rsqrt_ftz(ua), ib = rsqrt_ftz(ub);
    const f2 uinv = pack(ia, ib), u = mul2(u2, uinv);
    const f2 t = pack(__saturatef(ia - 1.0f), __saturatef(ib - 1.0f));   // at most 1 where it is used
    const f2 c = mul2(mul2(t, t), u);
    const f2 q = fma2(fma2(fma2(twice(Q3), u, twice(Q2)), u, twice(Q1)), u, twice(Q0));
    const f2 g = mul2(mul2(mul2(c, c), t), q);
    if constexpr (OUTER) return g;
    const f2 m = fma2(fma2(fma2(fma2(fma2(twice(I5), u, twice(I4)), u, twice(I3)), u, twice(I2)), u2, twice(I0)),
                      mul2(u2, u), twice(1.0f));
    const f2 gi = mul2(m, mul2(mul2(uinv, uinv), uinv));
    float oa, ob, na, nb;
    unpack(g, oa, ob);
    unpack(gi, na, nb);
    return pack(ua < 0.25f ? na : oa, ub < 0.25f ? nb : ob);
}

// Bounding box of the warp's targets and the largest squared range, kept in the
// warp's shared memory (fewer live registers in the stream loops); returns the
// expected candidates per pair.  Frame coordinates are not negative, so their
// bit patterns order like the values (padding lanes repeat lane 0's target).
__device__ __forceinline__ float warp_box(float4 *box, float mx, float my, float mz, float bcut2, float bpp2) {
    const unsigned all = 0xffffffffu;
    const float lx = __uint_as_float(__reduce_min_sync(all, __float_as_uint(mx)));
    const float ly = __uint_as_float(__reduce_min_sync(all, __float_as_uint(my)));
    const float lz = __uint_as_float(__reduce_min_sync(all, __float_as_uint(mz)));
    const float hx = __uint_as_float(__reduce_max_sync(all, __float_as_uint(mx)));
    const float hy = __uint_as_float(__reduce_max_sync(all, __float_as_uint(my)));
    const float hz = __uint_as_float(__reduce_max_sync(all, __float_as_uint(mz)));
    const float reach2 = __uint_as_float(__reduce_max_sync(all, __float_as_uint(bcut2)));
    if ((threadIdx.x & 31) == 0) {
        box[0] = make_float4(lx, ly, lz, reach2);
        // beyond it every pair is in the outer half of its range and no close one
        box[1] = make_float4(hx, hy, hz, 1.00001f * fmaxf(0.25f * reach2, bpp2));
    }
    __syncwarp();
    const float ex = hx - lx, ey = hy - ly, ez = hz - lz, r = sqrtf(reach2);
    // volume within reach of the box over that of one sphere: candidates per pair at even density
    const float area = fmaf(ex, ey, fmaf(ey, ez, __fmul_rn(ez, ex)));
    const float beyond = fmaf(ex * ey, ez, fmaf(2.0f * r, area, __fmul_rn(3.1416f * reach2, ex + ey + ez)));
    return __fadd_rn(beyond / (4.1888f * reach2 * r), 1.0f);
}

// Squared distance of a source from the box [lo, hi] of the warp's targets.
__device__ __forceinline__ float box_distance2(float4 lo, float4 hi, float4 q) {
    const float dx = fmaxf(fmaxf(lo.x - q.x, q.x - hi.x), 0.0f);
    const float dy = fmaxf(fmaxf(lo.y - q.y, q.y - hi.y), 0.0f);
    const float dz = fmaxf(fmaxf(lo.z - q.z, q.z - hi.z), 0.0f);
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// The sources of a warp's stream, 32 positions at a time, the next ones loaded
// while the current ones are worked on.  The segment of position b0 + lane: the
// segments that begin inside the window [b0, b0 + 32) as one bit mask; before:
// those begun ahead of it.
struct PPStream {
    int nseg, first, total, before, mine;   // this warp's part [first, total); mine: where segment `lane` begins
    int4 g;
    float4 raw = make_float4(0.f, 0.f, 0.f, 0.f);
    int slot;
    __device__ __forceinline__ void init(const PPParams &P, const PPWarpShared &W) {
        const int lane = threadIdx.x & 31;
        first = before = 0;
        mine = lane < nseg ? W.begin[lane] : 0x7fffffff;
        load(P, W, 0);   // the target itself is in the stream: never empty
    }
    // part p of PP_PARTS of the stream of `all` sources (never empty: all > PP_PARTS * 32)
    __device__ __forceinline__ void init_part(const PPParams &P, const PPWarpShared &W, int all, int p) {
        const int lane = threadIdx.x & 31, windows = (all + 31) / 32;
        first = (int)((int64_t)windows * p / PP_PARTS) * 32;
        total = min(all, (int)((int64_t)windows * (p + 1) / PP_PARTS) * 32);
        mine = lane < nseg ? W.begin[lane] : 0x7fffffff;
        int n = mine < first;
        for (int k = lane + 32; k < nseg; k += 32) n += W.begin[k] < first;
        before = __reduce_add_sync(0xffffffffu, n);
        load(P, W, first);
    }
    __device__ __forceinline__ void load(const PPParams &P, const PPWarpShared &W, int b0) {
        const int lane = threadIdx.x & 31;
        unsigned d = (unsigned)(mine - b0), bit = d < 32u ? 1u << d : 0u;
        for (int k = lane + 32; k < nseg; k += 32) {   // warps at the box's x faces only
            d = (unsigned)(W.begin[k] - b0);
            if (d < 32u) bit |= 1u << d;
        }
        const unsigned mask = __reduce_or_sync(0xffffffffu, bit);
        g = W.seg[before + __popc(mask & (0xffffffffu >> (31 - lane))) - 1];
        before += __popc(mask);
        slot = b0 + lane + g.x;
        if (b0 + lane < total) raw = P.pos[slot];
    }
    // the source at b0 + lane in the warp's frame (of no meaning past the end)
    __device__ __forceinline__ float4 next(const PPParams &P, const PPWarpShared &W, int b0) {
        const float4 q = frame_position(raw, g);
        if (b0 + 32 < total) load(P, W, b0 + 32);
        return q;
    }
};

// Pairs of every lane's target with n staged sources (n a multiple of 4), all
// of them, no test.  OUTER: no pair closer than half the range.  Out-of-range
// pairs get 0 from the clamped t; pairs closer than b_pp (the target itself
// among them) get 0 here and their bit in close (source k of 32: bit 31 - k).
template <bool OUTER, bool COUNT, int N>
__device__ __forceinline__ void eval_all(const Soa<N> &S, int n, const PPLane &L, float bpp2, f2 sum[3], unsigned &pairs,
                                         unsigned &close) {
    const f2 nx = twice(-L.mx), ny = twice(-L.my), nz = twice(-L.mz), ib2 = twice(L.ib2);
    f2 px = 0ull, py = 0ull, pz = 0ull;
#pragma unroll 1
    for (int k = 0; k < n; k += 4) {
        const ulonglong2 X = *reinterpret_cast<const ulonglong2 *>(&S.x[k]);
        const ulonglong2 Y = *reinterpret_cast<const ulonglong2 *>(&S.y[k]);
        const ulonglong2 Z = *reinterpret_cast<const ulonglong2 *>(&S.z[k]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const f2 rx = add2(h ? X.y : X.x, nx), ry = add2(h ? Y.y : Y.x, ny), rz = add2(h ? Z.y : Z.x, nz);
            const f2 r2 = fma2(rz, rz, fma2(ry, ry, mul2(rx, rx)));
            f2 g = far_factor2<OUTER>(mul2(r2, ib2));
            if constexpr (!OUTER || COUNT) {
                float ra, rb;
                unpack(r2, ra, rb);
                if constexpr (!OUTER) {
                    float ga, gb;
                    unpack(g, ga, gb);
                    const float ca = ra - bpp2, cb = rb - bpp2;
                    g = pack(ca < 0.0f ? 0.0f : ga, cb < 0.0f ? 0.0f : gb);
                    close = __funnelshift_l(__float_as_uint(ca), close, 1);
                    close = __funnelshift_l(__float_as_uint(cb), close, 1);
                }
                if constexpr (COUNT)
                    if (L.has) pairs += (ra > 0.0f && ra < L.bcut2) + (rb > 0.0f && rb < L.bcut2);
            }
            px = fma2(g, rx, px);
            py = fma2(g, ry, py);
            pz = fma2(g, rz, pz);
        }
    }
    sum[0] = px;
    sum[1] = py;
    sum[2] = pz;
}

__device__ __forceinline__ void add_pairs(Sum3 &a, const PPLane &L, f2 x, f2 y, f2 z) {
    float x0, x1, y0, y1, z0, z1;
    unpack(x, x0, x1);
    unpack(y, y0, y1);
    unpack(z, z0, z1);
    a.add_block(__fmul_rn(L.coef, x0 + x1), __fmul_rn(L.coef, y0 + y1), __fmul_rn(L.coef, z0 + z1));
}

// A warp's targets share one source stream.  Each source is staged once by one
// lane and kept only if it lies within the warp's largest PP range of the
// bounding box of the warp's targets (no pair of it can be in range otherwise).
//
// Compact warps (targets within about a cell): most kept sources are in range
// of most targets, and evaluating every pair costs less than finding those in
// range (20 FMA-pipe cycles a pair without a test, no idle lanes, against 6 a
// test and about 80 a pair found).  Sources at least half a range from the box
// are evaluated without the inner branch of the pair factor.
template <bool COUNT>
__device__ __forceinline__ void stream_compact(const PPParams &P, PPWarpShared &W, PPStream &T, const PPLane &L, Sum3 &a,
                                               unsigned &pairs, unsigned &cands) {
    const int lane = threadIdx.x & 31;
    auto &O = W.u.d.outer;
    auto &M = W.u.d.mixed;
    int fo = 0, fm = 0;
#pragma unroll 1
    for (int b0 = T.first; b0 < T.total || fo || fm; b0 += 32) {
        if (b0 < T.total) {
            const float4 q = T.next(P, W, b0);
            const float4 lo = W.box[0], hi = W.box[1];
            const float d2 = box_distance2(lo, hi, q);
            const bool keep = b0 + lane < T.total && d2 < lo.w, far = d2 > hi.w;
            const unsigned ko = __ballot_sync(0xffffffffu, keep && far), km = __ballot_sync(0xffffffffu, keep && !far);
            const unsigned lt = (1u << lane) - 1u;
            if (keep) {
                if (far) O.put(fo + __popc(ko & lt), q);
                else M.put(fm + __popc(km & lt), q);
            }
            fo += __popc(ko);
            fm += __popc(km);
            if (COUNT && L.has) cands += __popc(ko | km);
        }
        const bool last = b0 + 32 >= T.total;   // from here on only what is staged
        f2 sum[3];
        if (fo >= OUTER_N || (last && fo)) {
            const int n = min(OUTER_N, (fo + 3) & ~3);
            if (lane < n - fo) O.put(fo + lane, make_float4(PP_FAR, PP_FAR, PP_FAR, 0.f));
            __syncwarp();
            unsigned none = 0u;
            eval_all<true, COUNT>(O, n, L, 0.0f, sum, pairs, none);
            add_pairs(a, L, sum[0], sum[1], sum[2]);
            __syncwarp();
            fo = max(0, fo - OUTER_N);
            if (lane < fo) O.put(lane, make_float4(O.x[OUTER_N + lane], O.y[OUTER_N + lane], O.z[OUTER_N + lane], 0.f));
        }
        if (fm >= MIXED_N || (last && fm)) {
            const int n = min(MIXED_N, (fm + 3) & ~3);
            if (lane < n - fm) M.put(fm + lane, make_float4(PP_FAR, PP_FAR, PP_FAR, 0.f));
            __syncwarp();
            unsigned close = 0u;
            eval_all<false, COUNT>(M, n, L, P.bpp2, sum, pairs, close);
            close <<= 32 - n;
            if (__any_sync(0xffffffffu, close != 0u)) {
                float px = 0.f, py = 0.f, pz = 0.f;
#pragma unroll 1
                while (close) {
                    const int k = __clz(close);
                    close ^= 0x80000000u >> k;
                    const float rx = M.x[k] - L.mx, ry = M.y[k] - L.my, rz = M.z[k] - L.mz;
                    const float r2 = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
                    if (r2 > 0.0f) {   // not the target itself, nor a coincident particle
                        const float g = close_factor(r2 * L.ib2, P.ratio2 * L.bcut2);
                        px = fmaf(g, rx, px);
                        py = fmaf(g, ry, py);
                        pz = fmaf(g, rz, pz);
                    }
                }
                a.add_block(__fmul_rn(L.coef, px), __fmul_rn(L.coef, py), __fmul_rn(L.coef, pz));
            }
            add_pairs(a, L, sum[0], sum[1], sum[2]);
            __syncwarp();
            fm = max(0, fm - MIXED_N);
            if (lane < fm) M.put(lane, make_float4(M.x[MIXED_N + lane], M.y[MIXED_N + lane], M.z[MIXED_N + lane], 0.f));
        }
        __syncwarp();
    }
}

// Other warps (few of the sources are in range of any one target): every lane
// tests all kept sources, 32 to a mask (sign of r^2 - b_cut^2 shifted in, packed
// arithmetic: 6 FMA-pipe cycles a test), notes the sources in range in its own
// queue, and the queues are evaluated together, two pairs at a time, once up to
// SPARSE_N sources are through: the lanes then idle by the spread of their
// totals, not of every mask (about 7 pair evaluations a warp instead of 12 at
// one particle per cell).
__device__ __forceinline__ void eval_queue(const PPParams &P, const PPWarpShared &W, int held, const PPLane &L, Sum3 &a,
                                           unsigned &pairs) {
    const int lane = threadIdx.x & 31;
    const auto &S = W.u.s.src;
    const f2 nx = twice(-L.mx), ny = twice(-L.my), nz = twice(-L.mz), ib2 = twice(L.ib2);
    f2 px = 0ull, py = 0ull, pz = 0ull;
#pragma unroll 1
    for (int i = 0; i < held; i += 2) {
        const int ka = W.u.s.queue[i][lane];
        const int kb = i + 1 < held ? W.u.s.queue[i + 1][lane] : SPARSE_N;   // slot SPARSE_N: PP_FAR
        const f2 rx = add2(pack(S.x[ka], S.x[kb]), nx), ry = add2(pack(S.y[ka], S.y[kb]), ny),
                 rz = add2(pack(S.z[ka], S.z[kb]), nz);
        const f2 r2 = fma2(rz, rz, fma2(ry, ry, mul2(rx, rx)));
        const f2 u2 = mul2(r2, ib2);
        f2 g = far_factor2<false>(u2);
        float ra, rb;
        unpack(r2, ra, rb);
        if (__builtin_expect(fminf(ra, rb) < P.bpp2, 0)) {   // rare: a close pair; the target itself gets 0
            float ga, gb, ua, ub;
            unpack(g, ga, gb);
            unpack(u2, ua, ub);
#pragma unroll 1
            for (int e = 0; e < 2; ++e) {
                const float r = e ? rb : ra;
                if (r < P.bpp2) {
                    const float c = r > 0.0f ? close_factor(e ? ub : ua, P.ratio2 * L.bcut2) : 0.0f;
                    pairs -= r == 0.0f;
                    if (e) gb = c;
                    else ga = c;
                }
            }
            g = pack(ga, gb);
        }
        px = fma2(g, rx, px);
        py = fma2(g, ry, py);
        pz = fma2(g, rz, pz);
    }
    if (held) add_pairs(a, L, px, py, pz);
}

// stage(place, slot) and drain(held): what the caller keeps of a staged source and
// does with the queues.
template <class Stage, class Drain>
__device__ __forceinline__ void stream_sparse(const PPParams &P, PPWarpShared &W, PPStream &T, const PPLane &L,
                                              unsigned &pairs, unsigned &cands, const Stage &stage, const Drain &drain) {
    const int lane = threadIdx.x & 31;
    auto &S = W.u.s.src;
    int fill = 0;
    if (lane == 0) S.put(SPARSE_N, make_float4(PP_FAR, PP_FAR, PP_FAR, 0.f));
#pragma unroll 1
    for (int b0 = T.first; b0 < T.total; b0 += 32) {
        const int slot = T.slot;
        const float4 q = T.next(P, W, b0);
        const float4 lo = W.box[0], hi = W.box[1];
        const bool keep = b0 + lane < T.total && box_distance2(lo, hi, q) < lo.w;
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            const int at = fill + __popc(km & ((1u << lane) - 1u));
            S.put(at, q);
            stage(at, slot);
        }
        fill += __popc(km);
        if (fill <= SPARSE_N - 32 && b0 + 32 < T.total) continue;
        // pad to whole groups of 8, test, queue
        const int n8 = (fill + 7) & ~7;
        if (lane < n8 - fill) S.put(fill + lane, make_float4(PP_FAR, PP_FAR, PP_FAR, 0.f));
        __syncwarp();
        if (L.has) cands += (unsigned)fill;
        const f2 nx = twice(-L.mx), ny = twice(-L.my), nz = twice(-L.mz), nb = twice(L.has ? -L.bcut2 : 1.0f);
        int held = 0;
#pragma unroll 1
        for (int w0 = 0;; w0 += 32) {
            unsigned m = 0u;
            const int kn = min(32, n8 - w0);
#pragma unroll 1
            for (int k = 0; k < kn; k += 8) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const ulonglong2 X = *reinterpret_cast<const ulonglong2 *>(&S.x[w0 + k + 4 * h]);
                    const ulonglong2 Y = *reinterpret_cast<const ulonglong2 *>(&S.y[w0 + k + 4 * h]);
                    const ulonglong2 Z = *reinterpret_cast<const ulonglong2 *>(&S.z[w0 + k + 4 * h]);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const f2 rx = add2(e ? X.y : X.x, nx), ry = add2(e ? Y.y : Y.x, ny), rz = add2(e ? Z.y : Z.x, nz);
                        const f2 d = fma2(rx, rx, fma2(ry, ry, fma2(rz, rz, nb)));
                        float da, db;
                        unpack(d, da, db);
                        m = __funnelshift_l(__float_as_uint(da), m, 1);
                        m = __funnelshift_l(__float_as_uint(db), m, 1);
                    }
                }
            }
            const bool done = kn <= 0;   // nothing left to test: the queues' last evaluation
            if (!done) m <<= 32 - kn;
            const int more = __popc(m);
            pairs += more;
            if (done || __any_sync(0xffffffffu, held + more > QUEUE_N)) {
                __syncwarp();
                drain(held);
                held = 0;
                if (done) break;
            }
#pragma unroll 1
            while (m) {
                const int k = __clz(m);
                m ^= 0x80000000u >> k;
                W.u.s.queue[held++][lane] = (unsigned char)(w0 + k);
            }
        }
        fill = 0;
        __syncwarp();
    }
}

// Warps whose targets span a wide x range (nearly empty regions):
// each lane walks its own 27 cells as 9 row ranges and evaluates the pairs in
// range as it meets them.  Plain nested loops keep the loads pipelined.  (A
// per-lane queue of the pairs in range, evaluated when full, measured 2x
// slower over the 256^3 run: lanes of warps straddling two rows of a dense
// region fill their queues at different steps and evaluate them one at a
// time; skipping the rows and end cells beyond the range saved 6 % of the
// candidates at z = 49 and cost more than that.)
__device__ void lane_path(const PPParams &P, int c, float4 me, const PPLane &L, Sum3 &a, unsigned &pairs,
                          unsigned &cands) {
    if (!L.has) return;
    const int n = P.n_ios;
    const int cx = c % n, cy = (c / n) % n, cz = c / (n * n);
    const float bpp2 = P.bpp2;
#pragma unroll 1
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll 1
        for (int dy = -1; dy <= 1; ++dy) {
            const int64_t r = ((int64_t)wrap(cz + dz, n) * n + wrap(cy + dy, n)) * n;
            const RowRanges rr(P, r, cx, n);
            cands += rr.size();
            const float fdy = (float)dy, fdz = (float)dz;
            float px = 0.f, py = 0.f, pz = 0.f;
            for (int sgi = 0; sgi < rr.nseg; ++sgi) {
#pragma unroll 1
                for (int j = rr.beg[sgi]; j < rr.end[sgi]; ++j) {
                    const float4 q = P.pos[j];
                    const float fdx = (float)(rr.base[sgi] + (j >= rr.b1[sgi]) + (j >= rr.b2[sgi]));
                    const float rx = (fdx + q.x) - me.x;
                    const float ry = (fdy + q.y) - me.y;
                    const float rz = (fdz + q.z) - me.z;
                    const float r2 = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
                    if (r2 < L.bcut2 && r2 > 0.0f) {
                        float g, unused;
                        if (r2 >= bpp2) unpack(far_factor2<false>(twice(r2 * L.ib2)), g, unused);
                        else g = close_factor(r2 * L.ib2, P.ratio2 * L.bcut2);
                        px = fmaf(g, rx, px);
                        py = fmaf(g, ry, py);
                        pz = fmaf(g, rz, pz);
                        ++pairs;
                    }
                }
            }
            a.add_block(__fmul_rn(L.coef, px), __fmul_rn(L.coef, py), __fmul_rn(L.coef, pz));
        }
}

// ---------------------------------------------------------------- adjoint
// d(R(r, b) b^2)/du of Eq. (refforce), u = r/b < 1 (derivative of each branch).
__device__ __forceinline__ float ref_force_deriv_scaled(float u) {
    if (u < 0.5f)
        return 64.0f / 5.0f + u * u * (-768.0f / 5.0f + u * (128.0f + u * (1536.0f / 7.0f - 1152.0f / 5.0f * u)));
    return -6.0f / (35.0f * u * u * u) +
           (256.0f / 5.0f + u * (-192.0f + u * (768.0f / 5.0f + u * (128.0f + u * (-1536.0f / 7.0f + 384.0f / 5.0f * u)))));
}

// For the pair term g(r) d of the PP force (g = R_PP(r)/r, IOS-cell units):
// gc = g(r) and gp = g'(r)/r, so that the pair's Jacobian block is
// gc I + gp d d^T.  Far pairs (r >= b_pp), two at a time: with u = r/b_cut and the
// shell polynomial m(u), gc = m r^-3 and gp = h r^-5, h = u m' - 3 m; on [0, 1/2)
// both are polynomials in u, on [1/2, 1] in v = 1 - u, zero beyond.  Both branches
// are evaluated and one is chosen: the lanes of a warp need both all the time.
__device__ __forceinline__ void far_jacobian2(f2 r2, float inv_bcut, f2 &gc, f2 &gp) {
    float ra, rb, ua, ub;
    unpack(r2, ra, rb);
    const f2 rinv = pack(rsqrtf(ra), rsqrtf(rb));
    unpack(mul2(mul2(r2, rinv), twice(inv_bcut)), ua, ub);
    ua = fminf(ua, 1.0f);
    ub = fminf(ub, 1.0f);
    const f2 u = pack(ua, ub), v = fma2(u, twice(-1.0f), twice(1.0f));
    const f2 v2 = mul2(v, v), v4 = mul2(v2, v2);
    f2 mh = fma2(v, twice(-64.0f / 5.0f), twice(2048.0f / 35.0f));
    mh = fma2(v, mh, twice(-416.0f / 5.0f));
    mh = mul2(mul2(v4, v), fma2(v, mh, twice(192.0f / 5.0f)));
    f2 hh = fma2(v, twice(-64.0f), twice(11776.0f / 35.0f));
    hh = fma2(v, hh, twice(-3296.0f / 5.0f));
    hh = fma2(v, hh, twice(576.0f));
    hh = mul2(v4, fma2(v, hh, twice(-192.0f)));
    const f2 u2 = mul2(u, u), u3 = mul2(u2, u);
    f2 ml = fma2(u, twice(192.0f / 5.0f), twice(-1536.0f / 35.0f));
    ml = fma2(u, ml, twice(-32.0f));
    ml = fma2(u, ml, twice(256.0f / 5.0f));
    ml = fma2(u3, fma2(u2, ml, twice(-64.0f / 5.0f)), twice(1.0f));
    f2 hl = fma2(u, twice(192.0f), twice(-6144.0f / 35.0f));
    hl = fma2(u, hl, twice(-96.0f));
    hl = fma2(u, hl, twice(512.0f / 5.0f));
    hl = fma2(mul2(u3, u2), hl, twice(-3.0f));
    float mha, mhb, mla, mlb, hha, hhb, hla, hlb;
    unpack(mh, mha, mhb);
    unpack(ml, mla, mlb);
    unpack(hh, hha, hhb);
    unpack(hl, hla, hlb);
    const f2 i2 = mul2(rinv, rinv), i3 = mul2(i2, rinv);
    gc = mul2(pack(ua >= 0.5f ? mha : mla, ub >= 0.5f ? mhb : mlb), i3);
    gp = mul2(pack(ua >= 0.5f ? hha : hla, ub >= 0.5f ? hhb : hlb), mul2(i3, i2));
}

// Pairs closer than b_pp: the two-term formula and its derivative; the target itself: 0.
__device__ __noinline__ float2 close_jacobian(float r2, float inv_bpp, float inv_bcut) {
    if (!(r2 > 0.0f)) return make_float2(0.0f, 0.0f);
    const float rinv = rsqrtf(r2), r = r2 * rinv;
    const float gc = (ref_force_scaled(r * inv_bpp) * inv_bpp * inv_bpp -
                      ref_force_scaled(r * inv_bcut) * inv_bcut * inv_bcut) *
                     rinv;
    const float dr = ref_force_deriv_scaled(r * inv_bpp) * inv_bpp * inv_bpp * inv_bpp -
                     ref_force_deriv_scaled(r * inv_bcut) * inv_bcut * inv_bcut * inv_bcut;
    return make_float2(gc, (dr - gc) * rinv * rinv);
}

struct VjpIO {
    const float *v0, *v1, *v2;
    float *w0, *w1, *w2;
    float scale;   // coef / s_ios: Jacobian in cell units to d/dx in Mpc/h
};

// PP part of the vector-Jacobian product: w_i += sum_j A_ij (v_j - v_i) with
// A_ij = g I + (g'/r) d d^T (the force's Jacobian blocks are symmetric).
// Warps are dispatched as in the force: targets in pencil order, one source stream per
// warp (v_j staged with the positions; the force's test, queues and packed evaluation
// in compact warps too), long streams shared by eight warps, and each lane's 27 cells for
// the few warps wider than a stream.  The two products of a gradient
// over 128^3 particles at z = 1: 2.43 ms with a pair at a time, both branches of the
// polynomials taken in turn and every warp on its own, now 2.09.
__device__ __forceinline__ void jacobian_term(float rx, float ry, float rz, float r2, float4 vj, float vix, float viy,
                                              float viz, const PPParams &P, float &px, float &py, float &pz) {
    float gc, gp, unused;
    if (r2 >= P.bpp2) {
        f2 c2, p2;
        far_jacobian2(twice(r2), P.inv_bcut, c2, p2);
        unpack(c2, gc, unused);
        unpack(p2, gp, unused);
    } else {
        const float2 g = close_jacobian(r2, P.inv_bpp, P.inv_bcut);
        gc = g.x;
        gp = g.y;
    }
    const float dvx = vj.x - vix, dvy = vj.y - viy, dvz = vj.z - viz;
    const float dd = gp * (rx * dvx + ry * dvy + rz * dvz);
    px += gc * dvx + dd * rx;
    py += gc * dvy + dd * ry;
    pz += gc * dvz + dd * rz;
}

__device__ void lane_vjp(const PPParams &P, const VjpIO &V, bool has, int c, float4 me, float vix, float viy,
                         float viz, Sum3 &a) {
    if (!has) return;
    const int n = P.n_ios;
    const int cx = c % n, cy = (c / n) % n, cz = c / (n * n);
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy) {
            const int64_t r = ((int64_t)wrap(cz + dz, n) * n + wrap(cy + dy, n)) * n;
            const RowRanges rr(P, r, cx, n);
            const float fdy = (float)dy, fdz = (float)dz;
            float px = 0.f, py = 0.f, pz = 0.f;
            for (int sgi = 0; sgi < rr.nseg; ++sgi) {
                for (int j = rr.beg[sgi]; j < rr.end[sgi]; ++j) {
                    const float4 q = P.pos[j];
                    const float fdx = (float)(rr.base[sgi] + (j >= rr.b1[sgi]) + (j >= rr.b2[sgi]));
                    const float rx = (fdx + q.x) - me.x;
                    const float ry = (fdy + q.y) - me.y;
                    const float rz = (fdz + q.z) - me.z;
                    const float r2 = rx * rx + ry * ry + rz * rz;
                    if (r2 < P.bcut2 && r2 > 0.0f) {
                        const int pj = P.perm[j];
                        const float4 vj = make_float4(V.v0[pj], V.v1[pj], V.v2[pj], 0.f);
                        jacobian_term(rx, ry, rz, r2, vj, vix, viy, viz, P, px, py, pz);
                    }
                }
            }
            a.add_block(px, py, pz);
        }
}

struct PPVjpWarpShared : PPWarpShared {
    Soa<SPARSE_N + 4> vel;  // v_j of the staged sources
};

// Product terms of the pairs in the lanes' queues, two at a time.
__device__ __forceinline__ void vjp_queue(const PPParams &P, const PPVjpWarpShared &W, int held, const PPLane &L, float vix,
                                          float viy, float viz, Sum3 &a) {
    const int lane = threadIdx.x & 31;
    const auto &S = W.u.s.src;
    const auto &V = W.vel;
    const f2 nx = twice(-L.mx), ny = twice(-L.my), nz = twice(-L.mz);
    const f2 nvx = twice(-vix), nvy = twice(-viy), nvz = twice(-viz);
    f2 px = 0ull, py = 0ull, pz = 0ull;
#pragma unroll 1
    for (int i = 0; i < held; i += 2) {
        const int ka = W.u.s.queue[i][lane];
        const int kb = i + 1 < held ? W.u.s.queue[i + 1][lane] : SPARSE_N;   // slot SPARSE_N: PP_FAR
        const f2 rx = add2(pack(S.x[ka], S.x[kb]), nx), ry = add2(pack(S.y[ka], S.y[kb]), ny),
                 rz = add2(pack(S.z[ka], S.z[kb]), nz);
        const f2 r2 = fma2(rz, rz, fma2(ry, ry, mul2(rx, rx)));
        f2 gc, gp;
        far_jacobian2(r2, P.inv_bcut, gc, gp);
        float ra, rb;
        unpack(r2, ra, rb);
        if (__builtin_expect(fminf(ra, rb) < P.bpp2, 0)) {   // rare: a close pair, or the target itself
            float ca, cb, pa, pb;
            unpack(gc, ca, cb);
            unpack(gp, pa, pb);
#pragma unroll 1
            for (int e = 0; e < 2; ++e) {
                const float r = e ? rb : ra;
                if (r < P.bpp2) {
                    const float2 g = close_jacobian(r, P.inv_bpp, P.inv_bcut);
                    if (e) cb = g.x, pb = g.y;
                    else ca = g.x, pa = g.y;
                }
            }
            gc = pack(ca, cb);
            gp = pack(pa, pb);
        }
        const f2 dx = add2(pack(V.x[ka], V.x[kb]), nvx), dy = add2(pack(V.y[ka], V.y[kb]), nvy),
                 dz = add2(pack(V.z[ka], V.z[kb]), nvz);
        const f2 dd = mul2(gp, fma2(rz, dz, fma2(ry, dy, mul2(rx, dx))));
        px = fma2(gc, dx, fma2(dd, rx, px));
        py = fma2(gc, dy, fma2(dd, ry, py));
        pz = fma2(gc, dz, fma2(dd, rz, pz));
    }
    float xa, xb, ya, yb, za, zb;
    unpack(px, xa, xb);
    unpack(py, ya, yb);
    unpack(pz, za, zb);
    if (held) a.add_block(xa + xb, ya + yb, za + zb);
}

// The warp's target of each lane: its slot (lane 0's in padding lanes), cell
// coordinates and the block of cells that the warp's targets span.
struct PPTarget {
    float4 me;
    int slot, cx, cy, cz;
    bool has;
};

__device__ __forceinline__ PPTarget warp_target(const PPParams &P, int j, PPBlock &B) {
    PPTarget t;
    t.has = j >= 0;
    const int j0 = __shfl_sync(0xffffffffu, j, 0);   // a warp's first target is never padding
    t.slot = t.has ? j : j0;
    t.me = P.pos[t.slot];
    const int n = P.n_ios, c = __float_as_int(t.me.w);
    const int row = (int)(__umulhi((unsigned)c, P.div_mul) >> P.div_shift);
    t.cx = c - row * n;
    t.cz = (int)(__umulhi((unsigned)row, P.div_mul) >> P.div_shift);
    t.cy = row - t.cz * n;
    B.xa = __reduce_min_sync(0xffffffffu, t.cx);
    B.xb = __reduce_max_sync(0xffffffffu, t.cx);
    B.ya = __reduce_min_sync(0xffffffffu, t.cy);
    B.yb = __reduce_max_sync(0xffffffffu, t.cy);
    B.za = __reduce_min_sync(0xffffffffu, t.cz);
    B.zb = __reduce_max_sync(0xffffffffu, t.cz);
    return t;
}

// Warps with fewer expected candidates per pair than this evaluate every pair.
// The estimate takes the sources as evenly spread; around haloes more of them
// are in range.  PP at z = 0 of the 256^3 run with 6 / 9 / 14 / 20: 9.8 / 9.0 /
// 8.7 / 8.7 ms; 512^3 particles at z = 1 with 6 / 9 / 14: 25.0 / 23.4 / 22.9 ms.
//
// Where the sources are as even as the estimate has them, 9 is the better line, which
// matters in boxes that are dense throughout: 8 / 9 / 11 particles a cell, evenly, in
// 64^3, 48^3 and 64^3 cells 0.82 / 0.50 / 1.60 ms with 14, 0.71 / 0.44 / 1.48 with 9.
// Even: the density of the whole stream is PP_EVEN_LO to PP_EVEN_HI times the targets' own (32 in
// their box).  With about one particle a cell the dense places are haloes, where the
// rule costs more than it gives (the 256^3 run at z = 0 9.27 -> 9.36 ms): it is for
// boxes of PP_EVEN_MEAN particles a cell or more.
constexpr float PP_COMPACT = 14.0f, PP_COMPACT_EVEN = 9.0f;
constexpr float PP_EVEN_LO = 1.3f, PP_EVEN_HI = 3.0f;
constexpr int PP_EVEN_MEAN = 4;

__device__ __forceinline__ bool pp_compact(const PPParams &P, const float4 *box, float candidates, int total, const PPBlock &B) {
    if (!P.even || candidates < PP_COMPACT_EVEN) return candidates < PP_COMPACT;
    const float4 lo = box[0], hi = box[1];
    const float own = (hi.x - lo.x) * (hi.y - lo.y) * (hi.z - lo.z) * (1.0f / 32.0f);   // cells a target
    const float around = (float)((B.xb - B.xa + 3) * (B.yb - B.ya + 3) * (B.zb - B.za + 3));
    const float ratio = (float)total * own / around;
    return candidates < (ratio > PP_EVEN_LO && ratio < PP_EVEN_HI ? PP_COMPACT_EVEN : PP_COMPACT);
}

// The targets as the pair loops see them.
template <bool PM3>
__device__ __forceinline__ PPLane pp_lane(const PPParams &P, const PPTarget &t, const PPBlock &B) {
    PPLane L;
    L.has = t.has;
    // PP range of this target: b_3 inside a refined subtile of the third level
    float ibc = P.inv_bcut;
    L.bcut2 = P.bcut2;
    if (PM3) {
        const int T = P.pm3_T;
        const int s = (t.cz / T * P.pm3_ns + t.cy / T) * P.pm3_ns + t.cx / T;
        if (P.pm3_slot[s] >= 0) {
            L.bcut2 = P.bcut2_3;
            ibc = P.inv_bcut_3;
        }
    }
    L.ib2 = ibc * ibc;
    L.coef = P.coef * (L.ib2 * ibc);
    L.mx = (float)(t.cx - B.xa) + t.me.x;
    L.my = (float)(t.cy - B.ya + 1) + t.me.y;
    L.mz = (float)(t.cz - B.za + 1) + t.me.z;
    return L;
}

// Part of the warp's stream, by the loop that suits it.
template <bool COUNT>
__device__ __forceinline__ void pp_stream(const PPParams &P, PPWarpShared &W, PPStream &T, const PPLane &L, bool compact,
                                          Sum3 &a, unsigned &pairs, unsigned &cands) {
    if (compact)
        stream_compact<COUNT>(P, W, T, L, a, pairs, cands);
    else
        stream_sparse(P, W, T, L, pairs, cands, [](int, int) {}, [&](int held) { eval_queue(P, W, held, L, a, pairs); });
}

// The warp's 32 target places from i on.  COUNT: accumulate the work counters
// (off unless asked for: they live through the whole stream).  LIST: long streams
// go to the list (otherwise their parts are worked on here).
template <bool PM3, bool COUNT, bool LIST>
__device__ __forceinline__ void pp_warp(const PPParams &P, int64_t i, PPWarpShared &W) {
    const int j = P.tgt[i];   // with the length's load under way
    if ((i & ~(int64_t)31) >= P.work->places) return;   // whole warps: places past the last pencil's end
    PPBlock B;
    const PPTarget t = warp_target(P, j, B);
    const bool stream = B.xb - B.xa <= PP_WIDEST;
    // the sums' destinations on their way while the pairs are worked on (perm
    // stays inside the cell; both prefetches: 1.38 -> 1.35 ms at z = 49)
    if (P.accumulate) {
        prefetch_l1(&P.acc0[t.slot]);
        prefetch_l1(&P.acc1[t.slot]);
        prefetch_l1(&P.acc2[t.slot]);
    }
    if (P.kick != 0.0f) {
        prefetch_l1(&P.vel0[t.slot]);
        prefetch_l1(&P.vel1[t.slot]);
        prefetch_l1(&P.vel2[t.slot]);
    }
    const PPLane L = pp_lane<PM3>(P, t, B);
    Sum3 a;
    unsigned pairs = 0, cands = 0;
    if (stream) {
        PPStream T;
        T.total = build_segments(P, W.seg, W.begin, B, T.nseg);
        const bool split = T.total > P.long_min && P.work->crowd <= P.long_crowd;
        if (LIST && split) {
            if ((threadIdx.x & 31) == 0) P.long_list[atomicAdd(&P.work->n, 1)] = (int32_t)(i >> 5);
            return;
        }
        const bool compact = pp_compact(P, W.box, warp_box(W.box, L.mx, L.my, L.mz, L.bcut2, P.bpp2), T.total, B);
        if constexpr (LIST) {
            T.init(P, W);
            pp_stream<COUNT>(P, W, T, L, compact, a, pairs, cands);
        } else {
            const int all = T.total, parts = split ? PP_PARTS : 1;
#pragma unroll 1
            for (int p = 0; p < parts; ++p) {
                if (split) T.init_part(P, W, all, p);
                else T.init(P, W);
                Sum3 b;
                pp_stream<COUNT>(P, W, T, L, compact, b, pairs, cands);
                a.add_block(b.x - b.cx, b.y - b.cy, b.z - b.cz);
            }
        }
    } else {
        lane_path(P, __float_as_int(t.me.w), t.me, L, a, pairs, cands);
    }
    if (t.has) finish(P, P.perm[t.slot], a.x - a.cx, a.y - a.cy, a.z - a.cz);
    if constexpr (COUNT) {
        add_stats(P.stats, pairs, cands);
        if (!stream) add_stats(P.stats + 2, pairs, cands);   // warp-uniform
    }
}

// 64 registers, 32 warps per SM: the stream loops' packed constants and sums fit;
// more warps with 48 registers or fewer with 80 measured slower (z = 49 / z = 0:
// 1.56 / 9.4 and 1.59 / 9.0 ms against 1.38 / 8.7), and so did a kernel of its own
// for the compact warps (1.40 / 9.3).  Two warps per CTA: one is 2 % faster late
// (long warps hold no place of a finished one) and 6 % slower early.
constexpr int PP_WARPS = 2;
template <bool PM3, bool COUNT>
__global__ void __launch_bounds__(PP_WARPS * 32, 32 / PP_WARPS) pp_kernel(PPParams P) {
    chain();
    __shared__ PPWarpShared sh[PP_WARPS];
    pp_warp<PM3, COUNT, true>(P, (int64_t)blockIdx.x * (PP_WARPS * 32) + threadIdx.x, sh[threadIdx.x >> 5]);
}

// Partial sums of the parts of one warp's targets, added in their order by warp 0.
struct PPPartSums {
    float v[PP_PARTS][3][32];
    __device__ __forceinline__ void put(const Sum3 &a) {
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        v[w][0][lane] = a.x - a.cx;
        v[w][1][lane] = a.y - a.cy;
        v[w][2][lane] = a.z - a.cz;
    }
    __device__ __forceinline__ Sum3 sum() const {
        const int lane = threadIdx.x & 31;
        Sum3 a;
        for (int p = 0; p < PP_PARTS; ++p) a.add_block(v[p][0][lane], v[p][1][lane], v[p][2][lane]);
        return a;
    }
};

// The listed warps, a CTA each.
template <bool PM3, bool COUNT>
__global__ void __launch_bounds__(PP_PARTS * 32, 32 / PP_PARTS) pp_long_kernel(PPParams P) {
    chain();
    __shared__ PPWarpShared sh[PP_PARTS];
    __shared__ PPPartSums part;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, n = P.work->n;
    PPWarpShared &W = sh[w];
    for (int item = blockIdx.x; item < n; item += gridDim.x) {
        PPBlock B;
        const PPTarget t = warp_target(P, P.tgt[(int64_t)P.long_list[item] * 32 + lane], B);
        const PPLane L = pp_lane<PM3>(P, t, B);
        PPStream T;
        const int all = build_segments(P, W.seg, W.begin, B, T.nseg);
        const bool compact = pp_compact(P, W.box, warp_box(W.box, L.mx, L.my, L.mz, L.bcut2, P.bpp2), all, B);
        T.init_part(P, W, all, w);
        Sum3 a;
        unsigned pairs = 0, cands = 0;
        pp_stream<COUNT>(P, W, T, L, compact, a, pairs, cands);
        part.put(a);
        __syncthreads();
        if (w == 0 && t.has) {
            const Sum3 b = part.sum();
            finish(P, P.perm[t.slot], b.x - b.cx, b.y - b.cy, b.z - b.cz);
        }
        if constexpr (COUNT) add_stats(P.stats, pairs, cands);
        __syncthreads();
    }
}

// The product over one part of the warp's stream.
__device__ __forceinline__ void vjp_stream(const PPParams &P, const VjpIO &V, PPVjpWarpShared &W, PPStream &T, const PPLane &L,
                                           float vix, float viy, float viz, Sum3 &a) {
    if ((threadIdx.x & 31) == 0) W.vel.put(SPARSE_N, make_float4(0.f, 0.f, 0.f, 0.f));
    unsigned pairs = 0, cands = 0;   // not asked for
    stream_sparse(P, W, T, L, pairs, cands,
                  [&](int at, int slot) {
                      const int k = P.perm[slot];
                      W.vel.put(at, make_float4(V.v0[k], V.v1[k], V.v2[k], 0.f));
                  },
                  [&](int held) { vjp_queue(P, W, held, L, vix, viy, viz, a); });
}

__device__ __forceinline__ void vjp_finish(const VjpIO &V, int pi, const Sum3 &a) {
    V.w0[pi] += V.scale * (a.x - a.cx);
    V.w1[pi] += V.scale * (a.y - a.cy);
    V.w2[pi] += V.scale * (a.z - a.cz);
}

// 28 warps per SM (72 registers): 82 registers and 24 warps took 2.35 ms for the two
// products of 128^3 particles at z = 1, 64 and 32 2.30, this 2.29 (an unevolved state:
// 0.52, 0.45, 0.43).
constexpr int VJP_BLOCKS = 28;
__global__ void __launch_bounds__(32, VJP_BLOCKS) pp_vjp_kernel(PPParams P, VjpIO V) {
    chain();
    __shared__ PPVjpWarpShared sh;
    const int64_t i = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const int j = P.tgt[i];   // with the length's load under way
    if ((int64_t)blockIdx.x * 32 >= P.work->places) return;
    PPBlock B;
    const PPTarget t = warp_target(P, j, B);
    const int pi = P.perm[t.slot];
    const float vix = V.v0[pi], viy = V.v1[pi], viz = V.v2[pi];
    Sum3 a;
    if (B.xb - B.xa <= PP_WIDEST) {
        PPStream T;
        T.total = build_segments(P, sh.seg, sh.begin, B, T.nseg);
        if (T.total > P.long_min && P.work->crowd <= P.long_crowd) {
            if (threadIdx.x == 0) P.long_list[atomicAdd(&P.work->n, 1)] = blockIdx.x;
            return;
        }
        const PPLane L = pp_lane<false>(P, t, B);
        warp_box(sh.box, L.mx, L.my, L.mz, P.bcut2, P.bpp2);
        T.init(P, sh);
        vjp_stream(P, V, sh, T, L, vix, viy, viz, a);
    } else {
        lane_vjp(P, V, t.has, __float_as_int(t.me.w), t.me, vix, viy, viz, a);
    }
    if (t.has) vjp_finish(V, pi, a);
}

__global__ void __launch_bounds__(PP_PARTS * 32, VJP_BLOCKS / PP_PARTS) pp_vjp_long_kernel(PPParams P, VjpIO V) {
    chain();
    __shared__ PPVjpWarpShared sh[PP_PARTS];
    __shared__ PPPartSums part;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, n = P.work->n;
    PPVjpWarpShared &W = sh[w];
    for (int item = blockIdx.x; item < n; item += gridDim.x) {
        PPBlock B;
        const PPTarget t = warp_target(P, P.tgt[(int64_t)P.long_list[item] * 32 + lane], B);
        const int pi = P.perm[t.slot];
        const PPLane L = pp_lane<false>(P, t, B);
        PPStream T;
        const int all = build_segments(P, W.seg, W.begin, B, T.nseg);
        warp_box(W.box, L.mx, L.my, L.mz, P.bcut2, P.bpp2);
        T.init_part(P, W, all, w);
        Sum3 a;
        vjp_stream(P, V, W, T, L, V.v0[pi], V.v1[pi], V.v2[pi], a);
        part.put(a);
        __syncthreads();
        if (w == 0 && t.has) vjp_finish(V, pi, part.sum());
        __syncthreads();
    }
}

// ------------------------------------------------- ensemble: one persistent PP
// kernel over many boxes.  Work items are (box, block) pairs; a per-step cost
// estimate orders them largest first (the load balancing of Sec. 2.2.3: work
// sorted by its density, taken in that order by whoever is free), and
// persistent CTAs take the next item from a device counter.  The host
// publishes each step's queue with a stream-ordered write of the step's epoch;
// the kernel waits for that epoch for at most timeout_ns (%globaltimer), then
// records CUBE2_ERR_TIMEOUT in the queue's status word and returns.
struct PPQueueDev {
    int head;        // next item to take
    int count;       // items of this step
    int ready;       // epoch published by the host
    int status;      // sticky ST_TIMEOUT
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// cost[k] of item k (box b = item_box[k], block j = k - base[b]): the number of
// particles in the IOS cells of its targets, a proxy of the block's pair count
__global__ void __launch_bounds__(256) pp_item_cost_kernel(const PPParams *__restrict__ boxes,
                                                            const int32_t *__restrict__ item_box,
                                                            const int32_t *__restrict__ base, int n_items,
                                                            unsigned *__restrict__ cost) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_items) return;
    const int b = item_box[k];
    const PPParams &P = boxes[b];
    const int64_t i0 = (int64_t)(k - base[b]) * PP_ITEM;
    const int64_t i1 = min(i0 + PP_ITEM, (int64_t)P.work->places);
    unsigned s = 0;
    for (int64_t i = i0; i < i1; ++i) {
        const int j = P.tgt[i];
        if (j >= 0) s += (unsigned)P.count[__float_as_int(P.pos[j].w)];
    }
    cost[k] = s;
}

// One CTA: items bucketed by floor(log2(cost + 1)), largest bucket first,
// written to order[]; the queue's counters are reset for the step.
__global__ void __launch_bounds__(1024) pp_item_order_kernel(const unsigned *__restrict__ cost, int n_items,
                                                             int32_t *__restrict__ order, PPQueueDev *q) {
    __shared__ int hist[33], offs[33];
    if (threadIdx.x < 33) hist[threadIdx.x] = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < n_items; k += blockDim.x) atomicAdd(&hist[32 - __clz(cost[k] + 1u)], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int b = 32; b >= 0; --b) {
            offs[b] = run;
            run += hist[b];
        }
        q->head = 0;
        q->count = n_items;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n_items; k += blockDim.x) order[atomicAdd(&offs[32 - __clz(cost[k] + 1u)], 1)] = k;
}

__global__ void __launch_bounds__(PP_ITEM, 8) pp_persistent_kernel(const PPParams *__restrict__ boxes,
                                                                       const int32_t *__restrict__ item_box,
                                                                       const int32_t *__restrict__ base,
                                                                       const int32_t *__restrict__ order,
                                                                       PPQueueDev *q, int epoch,
                                                                       unsigned long long timeout_ns) {
    __shared__ PPWarpShared sh[PP_ITEM / 32];
    __shared__ int s_item, s_ok;
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned long long t0 = global_ns();
        while (atomicAdd(&q->ready, 0) != epoch) {
            if (atomicAdd(&q->status, 0) != 0 || global_ns() - t0 > timeout_ns) {
                atomicOr(&q->status, ST_TIMEOUT);
                ok = 0;
                break;
            }
            __nanosleep(2000);
        }
        s_ok = ok;
    }
    __syncthreads();
    if (!s_ok) return;
    const int count = *((volatile int *)&q->count);
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(&q->head, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= count) break;
        const int k = order[item];
        const int b = item_box[k];
        pp_warp<false, false, false>(boxes[b], (int64_t)(k - base[b]) * PP_ITEM + threadIdx.x, sh[threadIdx.x >> 5]);
    }
}

}  // namespace

// Target places, a whole number of items: every pencil's tail padded to a whole
// warp (a pencil with targets is at most 31 places longer than they are).
int64_t pp_target_items(int64_t N, int n_ios) {
    const int64_t pencils = (int64_t)pencils_y(n_ios) * pencils_z(n_ios);
    return (N + 31 * (pencils < N ? pencils : N) + PP_ITEM - 1) / PP_ITEM;
}

int64_t pp_target_slots(int64_t N, int n_ios) { return pp_target_items(N, n_ios) * PP_ITEM; }

size_t pp_work_bytes() { return sizeof(PPWork); }

// Cells that can hold PP_SORT_MIN particles.
int64_t pp_dense_cells(int64_t N) { return N / PP_SORT_MIN; }

static PPParams pp_params(cube2_ctx *ctx, const cube2_particles *p, int accumulate, float kick);

// PP inputs: target order, float positions, dense cells sorted by sub-cell.
static void launch_pp_inputs(cube2_ctx *ctx, const cube2_particles *p, const PPParams &P) {
    const int n = ctx->n_ios;
    {
        ProfScope prof(ctx, P_PP_ORDER, 0);
        cudaMemsetAsync(P.work, 0, sizeof(PPWork), ctx->stream);
        auto *pencils = P.long_min < PP_UNSPLIT ? pp_pencil_kernel<true> : pp_pencil_kernel<false>;
        pencils<<<(unsigned)(pencils_y(n) * pencils_z(n)), PREP_CTA, 0, ctx->stream>>>(
            p->count, p->start, n, PP_SORT_MIN, P.long_min, ctx->pp_tgt, ctx->pp_dense, P.work);
    }
    {
        ProfScope prof(ctx, P_PREP, 0);
        prep_positions_kernel<<<(unsigned)((ctx->N + PREP_CTA - 1) / PREP_CTA), PREP_CTA, 0, ctx->stream>>>(
            p->off[0], p->off[1], p->off[2], ctx->cellid, ctx->pos4, ctx->pp_perm, ctx->N);
    }
    {
        ProfScope prof(ctx, P_PP_ORDER, 0);
        launch_chained(ctx->chained, pp_dense_sort_kernel, (unsigned)(ctx->num_sms * 8), 256, 0, ctx->stream,
            p->off[0], p->off[1], p->off[2], p->count, p->start, ctx->pp_dense, &P.work->dense, ctx->pos4, ctx->pp_perm,
            ctx->pp_tgt);
    }
    ctx->launches += 3;
}

cudaError_t launch_pp_vjp(cube2_ctx *ctx, const cube2_particles *p, const float *const v[3], float *const w[3]) {
    if (ctx->N == 0) return cudaSuccess;
    PPParams P = pp_params(ctx, p, 1, 0.0f);
    P.long_min = vjp_long_min(ctx->N);
    VjpIO V{};
    V.v0 = v[0]; V.v1 = v[1]; V.v2 = v[2];
    V.w0 = w[0]; V.w1 = w[1]; V.w2 = w[2];
    V.scale = (float)((double)P.coef / ctx->s_ios);
    launch_pp_inputs(ctx, p, P);
    ProfScope prof(ctx, P_PP_VJP, 0);
    launch_chained(ctx->chained, pp_vjp_kernel, (unsigned)(pp_target_slots(ctx->N, ctx->n_ios) / 32), 32, 0, ctx->stream, P, V);
    ctx->launches += 1;
    if (P.long_min < PP_UNSPLIT) {
        launch_chained(ctx->chained, pp_vjp_long_kernel, (unsigned)(ctx->num_sms * (VJP_BLOCKS / PP_PARTS)), PP_PARTS * 32, 0, ctx->stream, P, V);
        ctx->launches += 1;
    }
    return cudaGetLastError();
}

static PPParams pp_params(cube2_ctx *ctx, const cube2_particles *p, int accumulate, float kick) {
    PPParams P{};
    P.pos = ctx->pos4;
    P.perm = ctx->pp_perm;
    P.tgt = ctx->pp_tgt;
    P.work = reinterpret_cast<PPWork *>(ctx->pp_work);
    P.count = p->count; P.start = p->start;
    P.acc0 = p->acc[0]; P.acc1 = p->acc[1]; P.acc2 = p->acc[2];
    if (ctx->vel32) {   // FP16 storage: the second kick updates the step's FP32 working copy
        P.vel0 = ctx->vel32; P.vel1 = ctx->vel32 + ctx->N; P.vel2 = ctx->vel32 + 2 * ctx->N;
    } else {
        P.vel0 = p->vel[0]; P.vel1 = p->vel[1]; P.vel2 = p->vel[2];
    }
    P.stats = ctx->pp_stats;
    P.n_ios = ctx->n_ios;
    {   // ceil(2^(31 + l) / n) with 2^(l-1) < n <= 2^l: exact quotients below 2^31
        int l = 1;
        while ((1 << l) < ctx->n_ios) ++l;
        P.div_mul = (unsigned)(((1ull << (31 + l)) + (unsigned)ctx->n_ios - 1) / (unsigned)ctx->n_ios);
        P.div_shift = l - 1;
    }
    P.accumulate = accumulate;
    P.even = ctx->N >= PP_EVEN_MEAN * ctx->n_cells;
    const double s = ctx->s_ios;
    // Separations are 0 or at least 2^-16 cells: shorter lengths all act like these, whose
    // powers stay within FP32 (the square of a softening that underflowed to 0 would no
    // longer tell the target itself from a far pair).
    const double b_cut = std::max(ctx->b_range, ldexp(s, -17)), b_pp = std::max(ctx->cfg.b_pp, ldexp(s, -18));
    P.inv_bpp = (float)(s / b_pp);
    P.inv_bcut = (float)(s / b_cut);
    P.bcut2 = (float)((b_cut / s) * (b_cut / s));
    P.bpp2 = (float)((b_pp / s) * (b_pp / s));
    P.ratio2 = (float)((s / b_pp) * (s / b_pp));
    const double vp = ctx->cfg.box * ctx->cfg.box * ctx->cfg.box / (double)ctx->N;
    P.coef = (float)(vp / (4.0 * 3.14159265358979323846) / (s * s));
    P.kick = kick;
    P.status = ctx->dev_status;
    P.long_min = pp_long_min(ctx->N);
    P.long_list = ctx->pp_long;
    P.long_crowd = ctx->num_sms * 32 * 32 * 3 / 5;   // 0.6 of the resident warps' targets
    if (ctx->pm3.on) {
        P.pm3_slot = ctx->pm3.slot;
        P.pm3_T = ctx->pm3.T;
        P.pm3_ns = ctx->pm3.ns;
        const double b3 = std::max(ctx->pm3.b3, ldexp(s, -17));
        P.bcut2_3 = (float)((b3 / s) * (b3 / s));
        P.inv_bcut_3 = (float)(s / b3);
    }
    return P;
}

cudaError_t launch_pp(cube2_ctx *ctx, const cube2_particles *p, int accumulate, float kick) {
    PPParams P = pp_params(ctx, p, accumulate, kick);
    if (ctx->N == 0) return cudaSuccess;
    const unsigned ctas = (unsigned)(pp_target_slots(ctx->N, ctx->n_ios) / (PP_WARPS * 32));
    launch_pp_inputs(ctx, p, P);
    if (ctx->defer_pp) {   // an ensemble's persistent kernel runs this box's PP later
        static_assert(sizeof(PPParams) <= sizeof(ctx->pp_deferred), "deferred PP parameters");
        memcpy(ctx->pp_deferred, &P, sizeof P);
        return cudaGetLastError();
    }
    {
        ProfScope prof(ctx, P_PP, 0);
        const bool pm3 = P.pm3_slot != nullptr, count = ctx->pp_count;
        launch_chained(ctx->chained, pm3 ? (count ? pp_kernel<true, true> : pp_kernel<true, false>)
                           : (count ? pp_kernel<false, true> : pp_kernel<false, false>),
                       ctas, PP_WARPS * 32, 0, ctx->stream, P);
        ctx->launches += 1;
        if (P.long_min < PP_UNSPLIT) {
            launch_chained(ctx->chained, pm3 ? (count ? pp_long_kernel<true, true> : pp_long_kernel<true, false>)
                               : (count ? pp_long_kernel<false, true> : pp_long_kernel<false, false>),
                           (unsigned)(ctx->num_sms * (32 / PP_PARTS)), PP_PARTS * 32, 0, ctx->stream, P);
            ctx->launches += 1;
        }
    }
    return cudaGetLastError();
}

size_t pp_params_bytes() { return sizeof(PPParams); }

cudaError_t launch_pp_persistent_step(cudaStream_t st, const void *boxes, const int32_t *item_box,
                                      const int32_t *base, int n_items, unsigned *cost, int32_t *order, void *queue,
                                      const int *publish_host, int epoch, unsigned long long timeout_ns, int grid) {
    const PPParams *B = static_cast<const PPParams *>(boxes);
    PPQueueDev *q = static_cast<PPQueueDev *>(queue);
    pp_item_cost_kernel<<<(unsigned)((n_items + 255) / 256), 256, 0, st>>>(B, item_box, base, n_items, cost);
    pp_item_order_kernel<<<1, 1024, 0, st>>>(cost, n_items, order, q);
    // the host's publication of this step's work count
    cudaError_t e = cudaMemcpyAsync(&q->ready, publish_host, sizeof(int), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    pp_persistent_kernel<<<(unsigned)grid, PP_ITEM, 0, st>>>(B, item_box, base, order, q, epoch, timeout_ns);
    return cudaGetLastError();
}

size_t pp_queue_bytes() { return sizeof(PPQueueDev); }

}  // namespace cube2
