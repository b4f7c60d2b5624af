// CIC mass assignment onto the PM levels (paper Sec. 2.1.2, Eq. filter with the
// CIC reading; IOS input of Sec. 2.3), one launch per level.
//
// Design: one CTA owns a brick of mesh cells and holds their 64-bit accumulators
// in shared memory as split words (low, high).  The tile has one more cell on
// each side, so that every cloud that touches an owned cell lies in it whole and
// no corner is tested (the border is not read back).  A corner weight is added
// with two 32-bit shared-memory atomics, low word first, the high word with its
// carry.  The CTA then converts each owned cell once and writes it with
// coalesced stores.  No global atomics and no 64-bit mesh in HBM.
//
// A level as fine as the IOS cells or finer (deposit_kernel): the brick is BI^3
// IOS cells; the CTA walks their particles and those of a one-cell IOS halo (a
// set of x-rows whose particles are contiguous in IOS order, two segments where
// a row wraps around the box; items map to particles through a short search over
// the row prefix), drops the ones whose cloud misses the owned cells and adds 8
// corners for each of the others.
//
// The level of half the IOS resolution (deposit_coarse_kernel): all particles of
// the 2 x 2 x 2 IOS cells around a mesh corner have that lower corner.  A thread
// takes such a block (a warp, where it holds many), sums the moments of its
// particles' fractions (number, x, y, z, xy, xz, yz, xyz, exact) and adds the 8
// corner sums, linear in the moments, once.
//
// Integer CIC: X = c 2^16 + off is the IOS fixed-point coordinate; the mesh
// coordinate floored to 2^-16 cell is X >> s (s >= 0) or X << -s.  With
// T = Xm - 2^15 the lower corner is T >> 16 and the 1-D weights are
// 2^16 - (T & 0xffff) and (T & 0xffff); the 3-D weight is their exact product.
// Sums are exact, so they do not depend on their order.  A cell of fewer than
// 2^16 particles cannot overflow; bricks with more watch the high word wrap.
//
// Bound: the latency of the phases (rows, particles, atomics, write-out) with the
// four CTAs that the tiles leave on an SM; the shared-memory pipe is 58 % busy.
// 256^3 run, 512^3 + 128^3 meshes, z = 49 / z = 0: 0.75 / 1.11 ms, against 0.96 /
// 1.18 with one pass over both levels and every corner tested against the owned
// cells; 64^3 particles 41 against 60 us, 512^3 6.8 against 8.2 ms.
#include "common.cuh"

namespace cube2 {
namespace {

struct DepParams {
    const uint16_t *off0, *off1, *off2;
    const int32_t *count, *start, *cellid;
    int n_ios, nbx;       // IOS cells per axis, bricks per axis
    int n;                // mesh cells per axis
    float *out_f32;       // FP32 overdensity grid (or null)
    uint64_t *out_u64;    // raw accumulator (or null)
    uint64_t mean_int;
    float scale;
    int *status;
};

__device__ __forceinline__ float u64_delta_to_f32(uint64_t acc, uint64_t m, float scale) {
    // RN32(acc - M) exactly (the magnitude is formed in uint64), then one FP32 multiply
    const float mag = acc >= m ? __ull2float_rn(acc - m) : -__ull2float_rn(m - acc);
    return __fmul_rn(mag, scale);
}

constexpr int DEP_THREADS = 384;       // four CTAs per SM with 40 registers (256: 0.79 ms, 512: 0.80 against 0.75)
constexpr int COARSE = 8;              // owned mesh cells per axis of a coarse brick
// Coarse blocks of COARSE_WARP particles get a warp, if they are few.  Of more than
// COARSE_FEW in a brick the warps take only those of COARSE_MEANS times the average, and
// threads the others: a warp does its share one after another, about 1.5 us each (16
// particles a cell, evenly, in 64^3 cells: 0.213 ms with all of them by warps, 0.08 by
// threads; 64^3 particles, half in clumps, 0.044 against 0.105).  Warps from 96 / 128 /
// 160 particles on: 12 a cell in 32^3 cells 0.091 / 0.056 / 0.054 ms, 64^3 particles,
// half in clumps, 0.045 / 0.047 / 0.048, the 256^3 run at z = 0 1.178 / 1.186 / 1.194.
constexpr int COARSE_WARP = 128, COARSE_FEW = 96, COARSE_MEANS = 4;
constexpr int COARSE_TOP = 4096;       // always a warp from here on: eight smaller blocks cannot overflow a cell
// Mean particles per cell from which a brick's lanes take DENSE_RUN particles in a row
// (always: 0.96 ms at z = 49 instead of 0.81).  Longer runs than that have a line of
// every array in use per lane, more than the L1 holds beside four CTAs' tiles: 16
// particles a cell in 96^3 cells, 192^3 mesh, with runs of 4 / 8 / 16 / 32 / a 32nd of
// the warp's 0.27 / 0.33 / 0.43 / 0.64 / 0.73 ms, 64 a cell in 32^3 0.23 / 0.27 / 0.34 /
// 0.52 / 0.86; the 256^3 run at z = 0 1.185 to 1.20 ms.
constexpr int DENSE_RUN = 4;            // a power of two
constexpr int DENSE_ITEMS = 3;

// The high word of a weight, with the carry of its low word's addition to old.
// CHECK: watch the high word wrap.
template <bool CHECK>
__device__ __forceinline__ void add_high(unsigned int *hi, unsigned int old, uint64_t w, int *status) {
    unsigned int add, sum;
    asm("add.cc.u32 %1, %2, %3;\n\taddc.u32 %0, %4, 0;"
        : "=r"(add), "=r"(sum)
        : "r"(old), "r"((unsigned int)w), "r"((unsigned int)(w >> 32)));
    if (!add) return;
    if (CHECK) {
        const unsigned int oldh = atomicAdd(hi, add);
        if (oldh + add < oldh) set_status(status, ST_CAPACITY);
    } else {
        atomicAdd(hi, add);
    }
}
template <bool CHECK>
__device__ __forceinline__ void add_weight(unsigned int *lo, unsigned int *hi, int c, uint64_t w, int *status) {
    add_high<CHECK>(&hi[c], atomicAdd(&lo[c], (unsigned int)w), w, status);
}

// Eight weights at the corners of the cloud at base (x fastest): the low words'
// atomics first, so that their returns overlap.
template <int W, bool CHECK>
__device__ __forceinline__ void add_corners(unsigned int *lo, unsigned int *hi, int base, const uint64_t (&w)[8], int *status) {
    unsigned int old[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) old[k] = atomicAdd(&lo[base + (k >> 2) * W * W + (k >> 1 & 1) * W + (k & 1)], (unsigned int)w[k]);
#pragma unroll
    for (int k = 0; k < 8; ++k) add_high<CHECK>(&hi[base + (k >> 2) * W * W + (k >> 1 & 1) * W + (k & 1)], old[k], w[k], status);
}

// The corner weights of one particle: f the fractions (weights of the upper corners).
template <int W, bool CHECK>
__device__ __forceinline__ void add_particle(unsigned int *lo, unsigned int *hi, int base, const int (&f)[3], int *status) {
    uint64_t w[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint64_t wyz = (uint64_t)(unsigned int)(k >> 1 ? f[2] : FIX - f[2]) *
                             (unsigned int)(k & 1 ? f[1] : FIX - f[1]);   // up to 2^32
        w[2 * k + 1] = wyz * (unsigned int)f[0];
        w[2 * k] = (wyz << FIX_BITS) - w[2 * k + 1];
    }
    add_corners<W, CHECK>(lo, hi, base, w, status);
}

// A lane's run of particles with one lower corner, as moments of the fractions.
struct Moments {
    uint64_t n, x, y, z, xy, xz, yz, xyz;
    __device__ __forceinline__ void clear() { n = x = y = z = xy = xz = yz = xyz = 0; }
    __device__ __forceinline__ void add(unsigned int fx, unsigned int fy, unsigned int fz) {
        const unsigned int p = fx * fy;   // fractions are below 2^16
        n += 1;
        x += fx;
        y += fy;
        z += fz;
        xy += p;
        xz += (uint64_t)fx * fz;
        yz += (uint64_t)fy * fz;
        xyz += (uint64_t)p * fz;
    }
};

// Corner sums from the moments: sum of products of f or 2^16 - f, modulo 2^64.
template <int W, bool CHECK>
__device__ __forceinline__ void add_moments(unsigned int *lo, unsigned int *hi, int base, const Moments &m, int *status) {
    const uint64_t c111 = m.xyz;
    const uint64_t c110 = (m.xy << 16) - c111, c101 = (m.xz << 16) - c111, c011 = (m.yz << 16) - c111;   // digits x y z
    const uint64_t c100 = (m.x << 32) - c110 - c101 - c111, c010 = (m.y << 32) - c110 - c011 - c111,
                   c001 = (m.z << 32) - c101 - c011 - c111;
    const uint64_t c000 = (m.n << 48) - c100 - c010 - c001 - c110 - c101 - c011 - c111;
    const uint64_t w[8] = {c000, c100, c010, c110, c001, c101, c011, c111};
    add_corners<W, CHECK>(lo, hi, base, w, status);
}

template <int BI>
struct Segments {
    static constexpr int MAX = 3 * (BI + 2) * (BI + 2);
    int pre[MAX + 1];    // item prefix over the halo-row segments
    int first[MAX];      // first particle of each segment minus its prefix
    int info[MAX];       // hy | hz << 8
    int c0[MAX];         // cell id of the halo's x = 0 in the segment's row
};

// The tile: own + 2 rows and planes; rows are own + 2 words apart and the owned
// cells begin at an even word (pairs of cells are read back 8 bytes at a time),
// so the cell right of a row is the unused first word of the next.
template <int OWN>
struct DepTile {
    static constexpr int W = OWN + 2;
    static constexpr int CELLS = (W * W * W + 4) & ~3;
    static constexpr size_t SMEM = (size_t)CELLS * 8;
    __device__ static int at(int x, int y, int z) { return ((z + 1) * W + y + 1) * W + x + 2; }   // owned-local
    __device__ static void zero(unsigned int *words) {
        for (int i = threadIdx.x; i < CELLS / 2; i += DEP_THREADS)
            reinterpret_cast<uint4 *>(words)[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // each owned cell converted and written once
    __device__ static void write(const DepParams &P, const unsigned int *lo, const unsigned int *hi, int ox, int oy, int oz,
                                 int ex, int ey, int ez) {
        if (!P.out_u64 && ex == OWN && ey == OWN && ez == OWN) {   // a whole brick: two cells of a row per thread
            constexpr int PAIRS = OWN / 2;
            float *out = P.out_f32 + ((int64_t)oz * P.n + oy) * P.n + ox;
#pragma unroll 4
            for (int i = threadIdx.x; i < PAIRS * OWN * OWN; i += DEP_THREADS) {
                const int x = 2 * (i % PAIRS), y = i / PAIRS % OWN, z = i / (PAIRS * OWN), c = at(x, y, z);
                const uint2 l = *reinterpret_cast<const uint2 *>(&lo[c]), h = *reinterpret_cast<const uint2 *>(&hi[c]);
                float2 f;
                f.x = u64_delta_to_f32(((uint64_t)h.x << 32) | l.x, P.mean_int, P.scale);
                f.y = u64_delta_to_f32(((uint64_t)h.y << 32) | l.y, P.mean_int, P.scale);
                *reinterpret_cast<float2 *>(&out[((int64_t)z * P.n + y) * P.n + x]) = f;   // n and ox are even
            }
            return;
        }
        for (int i = threadIdx.x; i < ex * ey * ez; i += DEP_THREADS) {
            const int x = i % ex, y = i / ex % ey, z = i / (ex * ey), c = at(x, y, z);
            const uint64_t v = ((uint64_t)hi[c] << 32) | (uint64_t)lo[c];
            const int64_t g = ((int64_t)(oz + z) * P.n + (oy + y)) * P.n + ox + x;
            if (P.out_u64) P.out_u64[g] = v;
            else P.out_f32[g] = u64_delta_to_f32(v, P.mean_int, P.scale);
        }
    }
};

// ------------------------------------- levels as fine as the IOS cells or finer
template <int UP, int BI, bool CHECK>
__device__ __forceinline__ void deposit_items(const DepParams &P, const Segments<BI> &G, int nseg, int total,
                                              unsigned int *lo, unsigned int *hi, int ext0, int ext1, int ext2) {
    using Tile = DepTile<(BI << UP)>;
    // Even bricks: lanes on consecutive particles (their loads share lines).
    // Dense ones: each lane DENSE_RUN in a row, so that the lanes sit in different
    // cells or parts of one and fewer of their corners hit the same words.
    const int nwarps = DEP_THREADS / 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per_w = ((total + nwarps - 1) / nwarps + 31) & ~31;
    const int last = total > DENSE_ITEMS * (BI + 2) * (BI + 2) * (BI + 2) ? DENSE_RUN - 1 : 0;   // of a run, per_w % 32 == 0
    const int it0 = w * per_w + lane * (last + 1), it1 = min(total, (w + 1) * per_w);
    if (it0 >= it1) return;
    int sg = 0, hi_s = nseg - 1;   // last segment with pre <= it0
    while (sg < hi_s) {
        const int mid = (sg + hi_s + 1) >> 1;
        if (G.pre[mid] <= it0) sg = mid;
        else hi_s = mid - 1;
    }
    int next = G.pre[sg + 1];
    for (int t = it0; t < it1; t += (t & last) == last ? 32 + 31 * last : 1) {
        while (next <= t) next = G.pre[++sg + 1];
        const int p = G.first[sg] + t, info = G.info[sg];
        const int hx = P.cellid[p] - G.c0[sg], hy = info & 0xff, hz = info >> 8;
        // fixed-point coordinates relative to the brick's origin, in mesh cells
        const int X[3] = {(hx - 1) * FIX + (int)P.off0[p], (hy - 1) * FIX + (int)P.off1[p],
                          (hz - 1) * FIX + (int)P.off2[p]};
        int i0[3], f[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int tt = X[a] * (1 << UP) - (FIX >> 1);
            i0[a] = tt >> FIX_BITS;   // lower corner, owned-local: -1 .. own - 1 where the cloud touches
            f[a] = tt & (FIX - 1);
        }
        if ((unsigned)(i0[0] + 1) > (unsigned)ext0 || (unsigned)(i0[1] + 1) > (unsigned)ext1 ||
            (unsigned)(i0[2] + 1) > (unsigned)ext2)
            continue;
        add_particle<Tile::W, CHECK>(lo, hi, Tile::at(i0[0], i0[1], i0[2]), f, P.status);
    }
}

// UP: log2(n / n_ios).
template <int UP, int BI>
__device__ __forceinline__ void fine_brick(const DepParams &P, int brick, unsigned int *words) {
    using Tile = DepTile<(BI << UP)>;
    __shared__ Segments<BI> G;
    unsigned int *lo = words, *hi = words + Tile::CELLS;   // [CELLS] low words, [CELLS] high words
    const int n = P.n_ios;
    const int bx = brick % P.nbx, by = (brick / P.nbx) % P.nbx, bz = brick / (P.nbx * P.nbx);
    const int c0x = bx * BI, c0y = by * BI, c0z = bz * BI;
    const int ex = min(BI, n - c0x), ey = min(BI, n - c0y), ez = min(BI, n - c0z);
    // segment (row, part): part 0 the cells inside [0, n) of a halo row's x in
    // [c0x-1, c0x+ex], parts 1 and 2 (bricks at the box's x faces only) the
    // cells that wrap on the left and right
    const int nrows = (ey + 2) * (ez + 2);
    const int parts = c0x == 0 || c0x + ex == n ? 3 : 1, nseg = parts * nrows;
    Tile::zero(words);
    for (int sg = threadIdx.x; sg < nseg; sg += DEP_THREADS) {
        const int row = sg / parts, part = sg - row * parts;
        const int hz = row / (ey + 2), hy = row - hz * (ey + 2);
        const int cy = wrap(c0y - 1 + hy, n), cz = wrap(c0z - 1 + hz, n);
        const int rbase = (cz * n + cy) * n;
        int xa = 0, xb = -1, hx0 = 0;      // empty
        if (part == 0) {
            xa = max(c0x - 1, 0);
            xb = min(c0x + ex, n - 1);
            hx0 = xa - (c0x - 1);
        } else if (part == 1 && c0x == 0) {
            xa = xb = n - 1;                // the halo cell left of x = 0
        } else if (part == 2 && c0x + ex == n) {
            xa = xb = 0;                    // the halo cell right of x = n - 1
            hx0 = ex + 1;
        }
        int st = 0, cnt = 0;
        if (xb >= xa) {
            st = P.start[rbase + xa];
            cnt = P.start[rbase + xb] + P.count[rbase + xb] - st;
        }
        G.pre[sg] = cnt;
        G.first[sg] = st;
        G.info[sg] = hy | (hz << 8);
        G.c0[sg] = rbase + xa - hx0;
    }
    __syncthreads();
    if (threadIdx.x < 32) {            // exclusive scan of the segment sizes
        const int lane = threadIdx.x;
        const int per = (nseg + 31) / 32;
        const int b0 = min(nseg, lane * per), b1 = min(nseg, b0 + per);
        int acc = 0;
        for (int i = b0; i < b1; ++i) acc += G.pre[i];
        int incl = acc;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int run = incl - acc;
        for (int i = b0; i < b1; ++i) {
            const int v = G.pre[i];
            G.pre[i] = run;
            G.first[i] -= run;
            run += v;
        }
        if (lane == 31) G.pre[nseg] = incl;
    }
    __syncthreads();
    const int total = G.pre[nseg];
    if (total < FIX) deposit_items<UP, BI, false>(P, G, nseg, total, lo, hi, ex << UP, ey << UP, ez << UP);
    else deposit_items<UP, BI, true>(P, G, nseg, total, lo, hi, ex << UP, ey << UP, ez << UP);
    __syncthreads();
    Tile::write(P, lo, hi, c0x << UP, c0y << UP, c0z << UP, ex << UP, ey << UP, ez << UP);
}

// ------------------------------------------- the level of half the IOS resolution
// One row (dy, dz) of a block: the particles of its two cells along x, at most
// two contiguous ranges (one, except across the box's face).
struct CoarseRow {
    int beg, mid, end, beg2, end2;     // [beg, end) with the second cell from mid on; [beg2, end2) the second cell
    __device__ CoarseRow(const DepParams &P, int r, int xa, int xb) {
        beg = P.start[r + xa];
        mid = P.start[r + xb];
        if (xb > xa) {
            end = mid + P.count[r + xb];
            beg2 = end2 = 0;
        } else {
            end = beg + P.count[r + xa];
            beg2 = mid;
            end2 = mid + P.count[r + xb];
            mid = 0x7fffffff;
        }
    }
    __device__ int size() const { return end - beg + end2 - beg2; }
};

constexpr size_t COARSE_SMEM = DepTile<COARSE>::SMEM + 2 * sizeof(int) * (COARSE + 1) * (COARSE + 1) * (COARSE + 1);

__device__ __forceinline__ void coarse_brick(const DepParams &P, int brick, unsigned int *words) {
    using Tile = DepTile<COARSE>;
    __shared__ int s_n;
    __shared__ unsigned long long s_sum;
    unsigned int *lo = words, *hi = words + Tile::CELLS;
    int *s_list = reinterpret_cast<int *>(words + 2 * Tile::CELLS);   // large blocks
    int *s_size = s_list + (COARSE + 1) * (COARSE + 1) * (COARSE + 1);
    const int n = P.n_ios;
    const int ox = brick % P.nbx * COARSE, oy = brick / P.nbx % P.nbx * COARSE, oz = brick / (P.nbx * P.nbx) * COARSE;
    const int ex = min(COARSE, P.n - ox), ey = min(COARSE, P.n - oy), ez = min(COARSE, P.n - oz);
    Tile::zero(words);
    if (threadIdx.x == 0) s_n = 0, s_sum = 0;
    __syncthreads();
    // block (bx, by, bz): lower corner b - 1 (owned-local), IOS cells 2 (o + b) - 1 and 2 (o + b) per axis
    auto rows = [&](int b, int (&r)[4], int &xa, int &xb, int &base) {
        const int bx = b % (ex + 1), by = b / (ex + 1) % (ey + 1), bz = b / ((ex + 1) * (ey + 1));
        xa = wrap(2 * (ox + bx) - 1, n);
        xb = wrap(2 * (ox + bx), n);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            r[k] = (wrap(2 * (oz + bz) - 1 + (k >> 1), n) * n + wrap(2 * (oy + by) - 1 + (k & 1), n)) * n;
        base = Tile::at(bx - 1, by - 1, bz - 1);
    };
    auto take = [&](Moments &m, int j, int dx, int k) {   // fraction: half a cell for the second one, plus half the offset
        m.add((dx << 15) + (P.off0[j] >> 1), ((k & 1) << 15) + (P.off1[j] >> 1), ((k >> 1) << 15) + (P.off2[j] >> 1));
    };
    auto by_thread = [&](const int (&r)[4], int xa, int xb, int base) {
        Moments m;
        m.clear();
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            const CoarseRow R(P, r[k], xa, xb);
            for (int j = R.beg; j < R.end; ++j) take(m, j, j >= R.mid, k);
            for (int j = R.beg2; j < R.end2; ++j) take(m, j, 1, k);
        }
        add_moments<Tile::W, false>(lo, hi, base, m, P.status);
    };
    const int nblocks = (ex + 1) * (ey + 1) * (ez + 1);
    for (int b = threadIdx.x; b < nblocks; b += DEP_THREADS) {
        int r[4], xa, xb, base;
        rows(b, r, xa, xb, base);
        int many = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) many += CoarseRow(P, r[k], xa, xb).size();
        if (many == 0) continue;
        if (many >= COARSE_WARP) {
            const int at = atomicAdd(&s_n, 1);
            s_list[at] = b;
            s_size[at] = many;
            atomicAdd(&s_sum, (unsigned long long)many);
            continue;
        }
        by_thread(r, xa, xb, base);
    }
    __syncthreads();
    int warp_from = 0;
    if (s_n > COARSE_FEW) {
        static_assert(8 * COARSE_TOP < FIX, "no watch on the blocks that threads take");
        warp_from = (int)min((unsigned long long)COARSE_TOP, COARSE_MEANS * s_sum / s_n);
        for (int i = threadIdx.x; i < s_n; i += DEP_THREADS) {
            if (s_size[i] >= warp_from) continue;
            int r[4], xa, xb, base;
            rows(s_list[i], r, xa, xb, base);
            by_thread(r, xa, xb, base);
        }
        __syncthreads();   // before the watched additions
    }
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < s_n; i += DEP_THREADS / 32) {
        if (s_size[i] < warp_from) continue;
        int r[4], xa, xb, base, many = 0;
        rows(s_list[i], r, xa, xb, base);
        Moments m;
        m.clear();
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            const CoarseRow R(P, r[k], xa, xb);
            many += R.size();
            const int len = R.end - R.beg;
            for (int q = lane; q < R.size(); q += 32) {
                const int j = q < len ? R.beg + q : R.beg2 + q - len;
                take(m, j, q < len ? j >= R.mid : 1, k);
                if (m.n == 32768) {   // far from a wrap of a lane's own sums
                    add_moments<Tile::W, true>(lo, hi, base, m, P.status);
                    m.clear();
                }
            }
        }
        if (many < 32768) {
            uint64_t *v = &m.n;
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
            if (lane == 0) add_moments<Tile::W, true>(lo, hi, base, m, P.status);
        } else {
            add_moments<Tile::W, true>(lo, hi, base, m, P.status);
        }
    }
    __syncthreads();
    Tile::write(P, lo, hi, ox, oy, oz, ex, ey, ez);
}

template <int UP, int BI>
__global__ void __launch_bounds__(DEP_THREADS, 4) deposit_kernel(DepParams fine) {
    chain();
    extern __shared__ __align__(16) unsigned int dep_words[];
    fine_brick<UP, BI>(fine, blockIdx.x, dep_words);
}

// A fine level and, in the first blocks of the grid, the coarse level of the same
// particles: for boxes of few bricks, where two launches would each leave the
// chip half empty (128^3 particles at z = 1: 0.144 against 0.213 ms; at 256^3 the
// launches apart are faster, 0.79 against 0.88: the coarse bricks would hold the
// fine ones' shared memory).  Figures with 256 threads.
template <int UP, int BI>
__global__ void __launch_bounds__(DEP_THREADS) deposit_both_kernel(DepParams fine, DepParams coarse, int n_coarse) {
    chain();
    extern __shared__ __align__(16) unsigned int dep_words[];
    if ((int)blockIdx.x < n_coarse) coarse_brick(coarse, blockIdx.x, dep_words);
    else fine_brick<UP, BI>(fine, (int)blockIdx.x - n_coarse, dep_words);
}

__global__ void __launch_bounds__(DEP_THREADS) deposit_coarse_kernel(DepParams coarse) {
    chain();
    extern __shared__ __align__(16) unsigned int dep_words[];
    coarse_brick(coarse, blockIdx.x, dep_words);
}

int64_t bricks(const DepParams &P) { return (int64_t)P.nbx * P.nbx * P.nbx; }

cudaError_t launch_coarse(cube2_ctx *ctx, const DepParams &coarse) {
    launch_chained(ctx->chained, deposit_coarse_kernel, (unsigned)bricks(coarse), DEP_THREADS, COARSE_SMEM, ctx->stream, coarse);
    ctx->launches++;
    return cudaGetLastError();
}

constexpr int64_t BOTH_BRICKS = 8192;   // most fine bricks with which the coarse level shares a launch

template <int UP, int BI>
cudaError_t launch_fine(cube2_ctx *ctx, DepParams fine, const DepParams *coarse) {
    constexpr size_t SMEM = DepTile<(BI << UP)>::SMEM, BOTH = SMEM > COARSE_SMEM ? SMEM : COARSE_SMEM;
    static PerDevice made;
    const cudaError_t opt = once_per_device(made, [] {
        return first_error({allow_shared(deposit_kernel<UP, BI>, SMEM), allow_shared(deposit_both_kernel<UP, BI>, BOTH)});
    });
    if (opt != cudaSuccess) return opt;
    fine.nbx = (fine.n_ios + BI - 1) / BI;
    if (coarse && bricks(fine) <= BOTH_BRICKS) {
        launch_chained(ctx->chained, deposit_both_kernel<UP, BI>, (unsigned)(bricks(*coarse) + bricks(fine)), DEP_THREADS, BOTH, ctx->stream,
            fine, *coarse, (int)bricks(*coarse));
    } else {
        const cudaError_t e = coarse ? launch_coarse(ctx, *coarse) : cudaSuccess;
        if (e != cudaSuccess) return e;
        launch_chained(ctx->chained, deposit_kernel<UP, BI>, (unsigned)bricks(fine), DEP_THREADS, SMEM, ctx->stream, fine);
    }
    ctx->launches++;
    return cudaGetLastError();
}

}  // namespace

// level >= 0: that level only; level = -1: every level.
// out_u64 (level >= 0 only): write the raw accumulator instead of the FP32 grid.
cudaError_t launch_deposit(cube2_ctx *ctx, int level, const cube2_particles *p, uint64_t *out_u64) {
    DepParams P{};
    P.off0 = p->off[0]; P.off1 = p->off[1]; P.off2 = p->off[2];
    P.count = p->count; P.start = p->start; P.cellid = ctx->cellid;
    P.n_ios = ctx->n_ios;
    P.status = ctx->dev_status;
    ProfScope prof(ctx, P_DEPOSIT, 0);
    cudaError_t e = cudaSuccess;
    DepParams coarse{};
    bool have_coarse = false;   // the coarse level rides along with the next one
    const int hi = level < 0 ? ctx->nl : level + 1;
    for (int l = level < 0 ? 0 : level; l < hi && e == cudaSuccess; ++l) {
        const Level &L = ctx->lev[l];
        P.n = L.n;
        P.out_u64 = out_u64;
        P.out_f32 = out_u64 ? nullptr : L.real;
        P.mean_int = L.mean_int;
        P.scale = L.dens_scale;
        if (L.shift == 1) {
            coarse = P;
            coarse.nbx = (L.n + COARSE - 1) / COARSE;
            have_coarse = l + 1 < hi;
            if (have_coarse) continue;
            e = launch_coarse(ctx, coarse);
            continue;
        }
        const DepParams *c = have_coarse ? &coarse : nullptr;
        have_coarse = false;
        switch (L.shift) {
            case 0: e = launch_fine<0, 8>(ctx, P, c); break;
            case -1: e = launch_fine<1, 8>(ctx, P, c); break;
            case -2: e = launch_fine<2, 4>(ctx, P, c); break;
            default: e = cudaErrorInvalidValue;
        }
    }
    return e;
}

}  // namespace cube2
