// Kick, fixed-point drift and IOS re-binning of the kick-drift-kick step (paper
// Secs. 2.2.3 and 2.3; constant Delta a, Sec. 3.2).
//
// Drift: X_d <- (X_d + rint(p_d Dr 2^16 / s_ios)) mod n_ios 2^16 (round half to
// even), X_d = c_d 2^16 + off_d.  Re-bin: a stable counting sort by the new
// cell id (ties keep the previous order) rebuilds count/start and permutes the
// offsets and momenta, so the IOS order stays the cell list.
//   1. kick_drift : new coordinates into scratch records; slot = count[new cell]++
//                   (atomic: a provisional, order-dependent rank in the cell)
//   2. scan       : start = exclusive prefix sum of count (multi-level)
//   3. scatter    : slots[start[cell] + slot] = old index
//   4. sort       : cells of more than RANK_MAX particles get their segment of
//                   slots sorted by old index: up to WARP_SORT by a warp, larger
//                   ones by a CTA (bitonic in shared memory up to 8192, beyond that
//                   sorted 8192-runs merged through global scratch)
//   5. gather     : off, vel, cellid and the map of each new index from its old
//                   one.  In a cell of up to RANK_MAX particles the new index is
//                   the start plus the number of smaller old indices in the
//                   segment, which makes the result stable and independent of
//                   the atomics' order without sorting it first.
// The histogram and its scan are made in the caller's count and start, which the
// step no longer reads once cellid is known.
#include "common.cuh"

#include <cuda_fp16.h>

namespace cube2 {
namespace {

// A place in each lane's cell.  Particles come in cell order and most stay in
// their cell or move with their neighbours: one atomic per run of lanes with the
// same cell (256^3 run's kick and drift at z = 0 / 1 / 49: 0.31 / 0.27 / 0.19 -> 0.23 / 0.22
// / 0.20 ms; one per distinct cell by __match_any_sync: 0.21 / 0.23 / 0.35).  mask: the
// warp's lanes with a particle, from lane 0 on.
__device__ __forceinline__ int take_slot(int32_t *count, int cell, unsigned mask) {
    const int lane = threadIdx.x & 31;
    const int before = __shfl_up_sync(mask, cell, 1);
    const unsigned heads = __ballot_sync(mask, lane == 0 || before != cell);
    const int head = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
    const unsigned later = heads & ~(0xffffffffu >> (31 - head));   // heads after this run's
    const int end = later ? __ffs(later) - 1 : __popc(mask);
    int base = 0;
    if (lane == head) base = atomicAdd(&count[cell], end - head);
    return __shfl_sync(mask, base, head) + lane - head;
}

constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_CHUNK = SCAN_THREADS * SCAN_ITEMS;   // 4096 elements per block

__global__ void kick_kernel(float *v0, float *v1, float *v2, const float *a0, const float *a1,
                            const float *a2, int64_t n, float kick, int *status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = v0[i] + kick * a0[i], y = v1[i] + kick * a1[i], z = v2[i] + kick * a2[i];
    v0[i] = x;
    v1[i] = y;
    v2[i] = z;
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) set_status(status, ST_NONFINITE);
}

// A particle between its old place and its new one, by old index: two records, so
// that the gather's scattered reads touch two or three sectors and not seven (256^3
// run at z = 49 / 0: gather 0.29 / 0.34 -> 0.18 / 0.23 ms; 512^3 2.63 -> 1.67).
struct Moved {
    float4 *vel_off;   // three velocities, the first two offsets in 16 bits each
    int2 *cell_off;    // new cell, third offset
    int32_t *slot;     // provisional slot within the cell

    __device__ __forceinline__ void put(int64_t i, float vx, float vy, float vz, const uint16_t off[3], int cell, int s) const {
        vel_off[i] = make_float4(vx, vy, vz, __uint_as_float((unsigned)off[0] | (unsigned)off[1] << 16));
        cell_off[i] = make_int2(cell, off[2]);
        slot[i] = s;
    }
};

struct DriftParams {
    const uint16_t *off0, *off1, *off2;
    const float *vel0, *vel1, *vel2;
    const uint16_t *v16_0, *v16_1, *v16_2;   // FP16 storage (null: FP32 vel)
    const float *vscale;                     // its per-cell scale
    const float *acc0, *acc1, *acc2;
    const int32_t *cellid;
    int32_t *count;           // zeroed before the launch, receives the new histogram
    Moved to;
    int64_t N;
    int n_ios;
    float kick, drift_fix;    // drift_fix = Dr 2^16 / s_ios
    int *status;
};

__global__ void __launch_bounds__(256) kick_drift_kernel(DriftParams P) {
    chain();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, i < P.N);
    if (i >= P.N) return;
    const int n = P.n_ios;
    const int c = P.cellid[i];
    const int cc[3] = {c % n, (c / n) % n, c / (n * n)};
    const uint16_t off[3] = {P.off0[i], P.off1[i], P.off2[i]};
    float v0[3];
    if (P.v16_0) {
        const float sc = P.vscale[c];
        v0[0] = __half2float(__ushort_as_half(P.v16_0[i])) * sc;
        v0[1] = __half2float(__ushort_as_half(P.v16_1[i])) * sc;
        v0[2] = __half2float(__ushort_as_half(P.v16_2[i])) * sc;
    } else {
        v0[0] = P.vel0[i];
        v0[1] = P.vel1[i];
        v0[2] = P.vel2[i];
    }
    const float v[3] = {v0[0] + P.kick * P.acc0[i], v0[1] + P.kick * P.acc1[i], v0[2] + P.kick * P.acc2[i]};
    const int period = n * FIX;
    int nc[3];
    uint16_t no[3];
    bool bad = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float d = v[a] * P.drift_fix;
        if (!(fabsf(d) < 0.5f * (float)period)) bad = true;   // also catches NaN
        const int disp = bad ? 0 : __float2int_rn(d);
        int X = cc[a] * FIX + (int)off[a] + disp;
        X = X < 0 ? X + period : (X >= period ? X - period : X);
        nc[a] = X >> FIX_BITS;
        no[a] = (uint16_t)(X & (FIX - 1));
    }
    if (bad) set_status(P.status, isfinite(v[0] + v[1] + v[2]) ? ST_DISPLACEMENT : ST_NONFINITE);
    const int cell = (nc[2] * n + nc[1]) * n + nc[0];
    const int slot = take_slot(P.count, cell, mask);
    P.to.put(i, v[0], v[1], v[2], no, cell, slot);
}

// Placement of arbitrary positions into IOS (the entry of a differentiable
// run): X_d = rint(x_d / s_ios * 2^16) mod n_ios 2^16 in FP64 (round half to
// even), then the same stable counting sort as the re-bin, ties in input order.
//
// The chip has two FP64 lanes an SM, and dividing, rounding and reducing there took
// a third of the call (319 us for 128^3 positions, now 226).  So the quotient is
// formed in integers: the mantissa times a 64-bit reciprocal of s_ios / 2^16, whose
// top 64 bits hold whole part and fraction with an error below 2^-62 of the value.
// Below 2^31 the FP64 quotient is within 2^-22 of it: where the fraction is further
// than 2^-20 from a half both round to the same integer, and only the rest (one in
// half a million, non-finite and huge values) goes through FP64.
struct PlaceParams {
    const double *pos0, *pos1, *pos2;
    const float *mom0, *mom1, *mom2;   // may be null: zero momenta
    int32_t *count;
    Moved to;
    int64_t N;
    int n_ios;
    double s_ios;
    uint64_t recip;                    // see reciprocal()
    int recip_shift;
    int *status;
};

// 1 / s in 64 bits: for x = m 2^(e - 1075) > 0, m the 53-bit mantissa and e the
// biased exponent, x 2^16 / s = ((m << 11) recip >> 64) 2^-(shift - e).
void reciprocal(double s, uint64_t &recip, int &shift) {
    int ex;
    const double f = frexp(s, &ex);                        // s = f 2^ex, f in [1/2, 1)
    const uint64_t ms = (uint64_t)ldexp(f, 53);            // s = ms 2^(ex - 53)
    const unsigned __int128 top = ~(unsigned __int128)0 >> 12;   // 2^116 - 1
    recip = (uint64_t)(top / ms);                          // in [2^63, 2^64)
    shift = 1122 + ex - 53;
    if (!(s >= 1e-30 && s <= 1e30)) shift = -100000;       // every position through FP64
}

// rint(x / s_ios 2^16) mod period as FP64 gives it
__device__ __forceinline__ int place_coord(double x, const PlaceParams &P, unsigned period, bool &bad) {
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    const int sh = P.recip_shift - (int)((bits >> 52) & 0x7ff);
    if (sh >= 33) {
        const uint64_t m = (bits << 11) | 0x8000000000000000ull;
        const uint64_t w = sh < 96 ? __umul64hi(m, P.recip) >> (sh - 32) : 0;   // whole part, 32 bits of fraction
        const unsigned frac = (unsigned)w;
        if (frac - 0x7ffff000u > 0x2000u) {
            unsigned q = (unsigned)(w >> 32) + (frac >> 31);
            if (q >= period) q %= period;
            return (int)((int64_t)bits < 0 && q ? period - q : q);
        }
    }
    const double u = rint(x / P.s_ios * (double)FIX);
    if (!(fabs(u) < 4.0e18)) {   // also catches NaN
        bad = true;
        return 0;
    }
    const int64_t X = (int64_t)u % (int64_t)period;
    return (int)(X < 0 ? X + period : X);
}

__global__ void __launch_bounds__(256) place_kernel(PlaceParams P) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    const int n = P.n_ios;
    const double x[3] = {P.pos0[i], P.pos1[i], P.pos2[i]};
    int nc[3];
    uint16_t no[3];
    bool bad = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int X = place_coord(x[a], P, (unsigned)n * (unsigned)FIX, bad);
        nc[a] = X >> FIX_BITS;
        no[a] = (uint16_t)(X & (FIX - 1));
    }
    if (bad) set_status(P.status, ST_NONFINITE);
    const int cell = (nc[2] * n + nc[1]) * n + nc[0];
    const int slot = atomicAdd(&P.count[cell], 1);
    P.to.put(i, P.mom0 ? P.mom0[i] : 0.0f, P.mom1 ? P.mom1[i] : 0.0f, P.mom2 ? P.mom2[i] : 0.0f, no, cell, slot);
}

// -------------------------------------------------------------- scan
__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        int w = lane < nw ? warp_sums[lane] : 0;
        int wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < nw) warp_sums[lane] = wi - w;
        if (lane == nw - 1) warp_sums[32] = wi;
    }
    __syncthreads();
    const int out = warp_sums[warp] + incl - v;
    total = warp_sums[32];
    __syncthreads();
    return out;
}

// A thread's SCAN_ITEMS elements; wide: both arrays on 16-byte boundaries (256^3
// cells: 0.095 -> 0.049 ms against single words, 512^3 0.65 -> 0.28)
__device__ __forceinline__ void scan_load(const int32_t *in, int64_t base, int64_t n, bool wide, int v[SCAN_ITEMS]) {
    if (wide && base + SCAN_ITEMS <= n) {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; k += 4) {
            const int4 q = *reinterpret_cast<const int4 *>(in + base + k);
            v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) v[k] = base + k < n ? in[base + k] : 0;
    }
}

__global__ void __launch_bounds__(SCAN_THREADS) scan_reduce_kernel(const int32_t *in, int32_t *sums, int64_t n, bool wide) {
    chain();
    __shared__ int ws[33];
    const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS], s = 0;
    scan_load(in, base, n, wide, v);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) s += v[k];
    int total;
    block_exclusive_scan(s, ws, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// exclusive scan of in[0, n) into out, adding offsets[blockIdx] (if non-null)
__global__ void __launch_bounds__(SCAN_THREADS) scan_apply_kernel(const int32_t *in, int32_t *out, int64_t n,
                                                                  const int32_t *offsets, bool wide) {
    chain();
    __shared__ int ws[33];
    const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS], s = 0;
    scan_load(in, base, n, wide, v);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) s += v[k];
    int total;
    int run = block_exclusive_scan(s, ws, total) + (offsets ? offsets[blockIdx.x] : 0);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        const int t = v[k];
        v[k] = run;
        run += t;
    }
    if (wide && base + SCAN_ITEMS <= n) {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; k += 4)
            *reinterpret_cast<int4 *>(out + base + k) = make_int4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k)
            if (base + k < n) out[base + k] = v[k];
    }
}

// ------------------------------------------------------------- rebin
__global__ void __launch_bounds__(256) scatter_kernel(Moved from, const int32_t *start, int32_t *perm,
                                                      int64_t n) {
    chain();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    perm[start[from.cell_off[i].x] + from.slot[i]] = (int32_t)i;
}

// Cells of more than RANK_MAX particles, whose segments are sorted ascending
// (old index = stable order): up to WARP_SORT from the front of `big` (one warp
// per cell), larger ones from the back (one CTA per cell: a warp takes 80 us for a
// cell of 1000, which the whole step of a small box waits for).  Ranking in the
// gather costs reads of cached slots and scales with a cell's square; at 160 the
// 256^3 run at z = 0 takes 0.34 ms there and 0.124 here, at 96 0.33 and 0.153, at
// 48 0.33 and 0.195.  512 threads: one cell of some thousands costs a 64^3 box
// 0.033 ms (256: 0.052, 1024: 0.025), the many of the 256^3 run 0.124 (0.128, 0.197).
constexpr int RANK_MAX = 160;
constexpr int WARP_SORT = 256;
constexpr int SORT_THREADS = 512, SORT_WARPS = SORT_THREADS / 32;
constexpr int BIG_SORT_SMEM = 8192;

__global__ void __launch_bounds__(256) sort_list_kernel(const int32_t *__restrict__ count, int64_t n_cells, int32_t *big,
                                                        int *big_n, bool wide) {
    const int64_t c0 = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    int4 v = make_int4(0, 0, 0, 0);
    if (wide && c0 + 3 < n_cells) v = *reinterpret_cast<const int4 *>(count + c0);
    else
        for (int k = 0; c0 + k < n_cells && k < 4; ++k) (&v.x)[k] = count[c0 + k];
    if (max(max(v.x, v.y), max(v.z, v.w)) <= RANK_MAX) return;
    for (int k = 0; k < 4; ++k) {
        const int cnt = (&v.x)[k];
        if (cnt <= RANK_MAX) continue;
        if (cnt <= WARP_SORT) big[atomicAdd(&big_n[0], 1)] = (int32_t)(c0 + k);
        else big[n_cells - 1 - atomicAdd(&big_n[1], 1)] = (int32_t)(c0 + k);
    }
}

__device__ void bitonic_smem(int32_t *s, int np2) {
    for (int k = 2; k <= np2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < np2; i += blockDim.x) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const bool up = (i & k) == 0;
                    const int32_t a = s[i], b = s[ixj];
                    if ((a > b) == up) { s[i] = b; s[ixj] = a; }
                }
            }
            __syncthreads();
        }
    }
}

// sort keys[0, n) (n <= BIG_SORT_SMEM) in place through shared memory
__device__ void sort_run_smem(int32_t *keys, int n, int32_t *s) {
    int np2 = 1;
    while (np2 < n) np2 <<= 1;
    for (int i = threadIdx.x; i < np2; i += blockDim.x) s[i] = i < n ? keys[i] : 0x7fffffff;
    __syncthreads();
    bitonic_smem(s, np2);
    for (int i = threadIdx.x; i < n; i += blockDim.x) keys[i] = s[i];
    __syncthreads();
}

// merge sorted a[0, la) and b[0, lb) into out (keys unique), CTA-cooperative
__device__ void merge_runs(const int32_t *a, int la, const int32_t *b, int lb, int32_t *out) {
    const int total = la + lb;
    const int per = (total + blockDim.x - 1) / blockDim.x;
    const int d0 = min(total, (int)threadIdx.x * per), d1 = min(total, d0 + per);
    if (d0 >= d1) return;
    int lo = max(0, d0 - lb), hi = min(d0, la);
    while (lo < hi) {                      // merge-path split of diagonal d0
        const int mid = (lo + hi) >> 1;
        if (a[mid] <= b[d0 - mid - 1]) lo = mid + 1; else hi = mid;
    }
    int i = lo, j = d0 - lo;
    for (int d = d0; d < d1; ++d) {
        if (j >= lb || (i < la && a[i] <= b[j])) out[d] = a[i++];
        else out[d] = b[j++];
    }
}

// One cell of up to WARP_SORT particles by a warp: a bitonic sort of the segment
// (padded to a power of two) in the warp's own shared buffer, every lane
// exchanging pairs at each stage, with warp barriers only.
__device__ void sort_warp(int32_t *seg, int n, int32_t *s) {
    const int lane = threadIdx.x & 31;
    int np2 = 64;
    while (np2 < n) np2 <<= 1;
    for (int i = lane; i < np2; i += 32) s[i] = i < n ? seg[i] : 0x7fffffff;
    __syncwarp();
    for (int k = 2; k <= np2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int q = lane; q < (np2 >> 1); q += 32) {
                const int i = ((q & ~(j - 1)) << 1) | (q & (j - 1));   // lower index of pair q
                const int ixj = i | j;
                const bool up = (i & k) == 0;
                const int32_t a = s[i], b = s[ixj];
                if ((a > b) == up) {
                    s[i] = b;
                    s[ixj] = a;
                }
            }
            __syncwarp();
        }
    for (int i = lane; i < n; i += 32) seg[i] = s[i];
    __syncwarp();
}

__global__ void __launch_bounds__(SORT_THREADS) sort_cells_kernel(const int32_t *count, const int32_t *start,
                                                                  int32_t *perm, int32_t *scratch, const int32_t *big,
                                                                  const int *big_n, int64_t n_cells) {
    chain();
    __shared__ int32_t s[BIG_SORT_SMEM];
    static_assert(SORT_WARPS * WARP_SORT <= BIG_SORT_SMEM, "a buffer per warp");
    const int n_cta = big_n[1];
    for (int item = blockIdx.x; item < n_cta; item += gridDim.x) {
        const int64_t c = big[n_cells - 1 - item];
        const int n = count[c];
        int32_t *seg = perm + start[c];
        if (n <= BIG_SORT_SMEM) {
            sort_run_smem(seg, n, s);
            continue;
        }
        for (int r = 0; r < n; r += BIG_SORT_SMEM) sort_run_smem(seg + r, min(BIG_SORT_SMEM, n - r), s);
        int32_t *src = seg, *dst = scratch + start[c];
        for (int w = BIG_SORT_SMEM; w < n; w <<= 1) {
            for (int lo = 0; lo < n; lo += 2 * w) {
                const int la = min(w, n - lo), lb = max(0, min(w, n - lo - w));
                merge_runs(src + lo, la, src + lo + la, lb, dst + lo);
            }
            __syncthreads();
            int32_t *t = src; src = dst; dst = t;
        }
        if (src != seg)
            for (int i = threadIdx.x; i < n; i += blockDim.x) seg[i] = src[i];
        __syncthreads();
    }
    const int w = threadIdx.x >> 5, n_warp = big_n[0];
    for (int item = blockIdx.x * SORT_WARPS + w; item < n_warp; item += gridDim.x * SORT_WARPS) {
        const int64_t c = big[item];
        sort_warp(perm + start[c], count[c], s + w * WARP_SORT);
    }
}

struct GatherParams {
    const int32_t *slots;          // old index by provisional slot (scatter_kernel)
    int32_t *perm;                 // old index by new index
    const int32_t *count, *start;
    Moved from;
    uint16_t *off0, *off1, *off2;
    float *vel0, *vel1, *vel2;
    int32_t *cellid;
    int64_t N;
};

// One thread per provisional slot: its place is its rank in the cell.  Bound by
// the scattered reads of a particle's 24 bytes.  A pass of its own that sorted the
// small segments, a thread per cell, took 0.28 ms and the gather 0.25 on the 256^3
// run at z = 0 (512^3 at z = 1: 1.91 and 2.01); together they took 0.34
// (2.63), with the packed records 0.23 (1.67).
__global__ void __launch_bounds__(256) gather_kernel(GatherParams P) {
    chain();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= P.N) return;
    const int j = P.slots[s];
    const int2 co = P.from.cell_off[j];
    const float4 vo = P.from.vel_off[j];
    const int c = co.x;
    const int cnt = P.count[c];
    int64_t i = s;
    if (cnt > 1 && cnt <= RANK_MAX) {
        const int st = P.start[c];
        int rank = 0;
        for (int k = 0; k < cnt; ++k) rank += P.slots[st + k] < j;
        i = st + rank;
    }
    const unsigned off01 = __float_as_uint(vo.w);
    P.perm[i] = j;
    P.off0[i] = (uint16_t)off01;
    P.off1[i] = (uint16_t)(off01 >> 16);
    P.off2[i] = (uint16_t)co.y;
    P.vel0[i] = vo.x;
    P.vel1[i] = vo.y;
    P.vel2[i] = vo.z;
    P.cellid[i] = c;
}

// FP16 velocity codec: per IOS cell the FP32 scale max_p,d |v_d| (an atomic
// max on the bit patterns, which order like the values for v >= 0, so the
// result does not depend on order), then code = RN_half(RN32(v / scale)).
//
// One pass, a CTA per 1024 cells: their particles lie in a row, the maxima stay in
// shared memory, the first ENCODE_HELD rounds of velocities in registers (more, in a
// dense state, are read again from the caches).  As two kernels with the maxima in
// global memory it took 1.81 ms for 512^3 particles, now 0.86 (256 cells
// and one round, waiting for its loads: 1.73; 512 cells: 1.07).
constexpr int ENCODE_CELLS = 1024, ENCODE_HELD = 4, ENCODE_THREADS = 256;

__device__ __forceinline__ uint16_t velocity_code(float v, float s) {
    return s > 0.0f ? __half_as_ushort(__float2half_rn(__fdiv_rn(v, s))) : (uint16_t)0;
}

__global__ void __launch_bounds__(ENCODE_THREADS)
vel_encode_kernel(const float *v0, const float *v1, const float *v2, const int32_t *cellid, const int32_t *count,
                  const int32_t *start, float *__restrict__ vscale, uint16_t *__restrict__ c0, uint16_t *__restrict__ c1,
                  uint16_t *__restrict__ c2, int64_t n_cells) {
    chain();
    __shared__ int top[ENCODE_CELLS];
    const int64_t first = (int64_t)blockIdx.x * ENCODE_CELLS;
    const int cells = (int)min((int64_t)ENCODE_CELLS, n_cells - first);
    const int lane = threadIdx.x & 31;
    const int64_t b = start[first], e = (int64_t)start[first + cells - 1] + count[first + cells - 1];
    for (int k = threadIdx.x; k < ENCODE_CELLS; k += ENCODE_THREADS) top[k] = 0;
    auto largest = [&](int c, float x, float y, float z) {
        int m = c >= 0 ? __float_as_int(fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)))) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {   // a run of lanes in one cell: its maximum, at its last lane
            const int cu = __shfl_up_sync(0xffffffffu, c, o), mu = __shfl_up_sync(0xffffffffu, m, o);
            if (lane >= o && cu == c) m = max(m, mu);
        }
        const int next = __shfl_down_sync(0xffffffffu, c, 1);
        if (c >= 0 && (lane == 31 || next != c)) atomicMax(&top[c], m);
    };
    int c[ENCODE_HELD];
    float x[ENCODE_HELD], y[ENCODE_HELD], z[ENCODE_HELD];
#pragma unroll
    for (int k = 0; k < ENCODE_HELD; ++k) {
        const int64_t i = b + k * ENCODE_THREADS + threadIdx.x;
        c[k] = -1;
        x[k] = y[k] = z[k] = 0.0f;
        if (i < e) {
            c[k] = cellid[i] - (int)first;
            x[k] = v0[i]; y[k] = v1[i]; z[k] = v2[i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ENCODE_HELD; ++k)
        if (b + k * ENCODE_THREADS < e) largest(c[k], x[k], y[k], z[k]);
    const int64_t rest = b + ENCODE_HELD * ENCODE_THREADS;
    for (int64_t w = rest + (threadIdx.x & ~31); w < e; w += ENCODE_THREADS) {   // a warp at a time
        const int64_t i = w + lane;
        const bool in = i < e;
        largest(in ? cellid[i] - (int)first : -1, in ? v0[i] : 0.0f, in ? v1[i] : 0.0f, in ? v2[i] : 0.0f);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < cells; k += ENCODE_THREADS) vscale[first + k] = __int_as_float(top[k]);
#pragma unroll
    for (int k = 0; k < ENCODE_HELD; ++k) {
        const int64_t i = b + k * ENCODE_THREADS + threadIdx.x;
        if (i < e) {
            const float s = __int_as_float(top[c[k]]);
            c0[i] = velocity_code(x[k], s);
            c1[i] = velocity_code(y[k], s);
            c2[i] = velocity_code(z[k], s);
        }
    }
    for (int64_t i = rest + threadIdx.x; i < e; i += ENCODE_THREADS) {
        const float s = __int_as_float(top[cellid[i] - (int)first]), vx = v0[i], vy = v1[i], vz = v2[i];
        c0[i] = velocity_code(vx, s);
        c1[i] = velocity_code(vy, s);
        c2[i] = velocity_code(vz, s);
    }
}

__global__ void vel_decode_kernel(const uint16_t *__restrict__ c0, const uint16_t *__restrict__ c1,
                                  const uint16_t *__restrict__ c2, const int32_t *__restrict__ cellid,
                                  const float *__restrict__ vscale, float *__restrict__ v0, float *__restrict__ v1,
                                  float *__restrict__ v2, int64_t N) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const float s = vscale[cellid[i]];
    v0[i] = __half2float(__ushort_as_half(c0[i])) * s;
    v1[i] = __half2float(__ushort_as_half(c1[i])) * s;
    v2[i] = __half2float(__ushort_as_half(c2[i])) * s;
}

}  // namespace

// p->vel16 / p->vscale from FP32 momenta v (ctx->cellid must hold p's cells).
cudaError_t launch_vel_encode(cube2_ctx *ctx, const cube2_particles *p, const float *const v[3]) {
    if (ctx->N == 0) return cudaMemsetAsync(p->vscale, 0, sizeof(float) * ctx->n_cells, ctx->stream);
    ProfScope prof(ctx, P_KICK, 0);
    launch_chained(ctx->chained, vel_encode_kernel, (unsigned)((ctx->n_cells + ENCODE_CELLS - 1) / ENCODE_CELLS), ENCODE_THREADS, 0, ctx->stream,
        v[0], v[1], v[2], ctx->cellid, p->count, p->start, p->vscale, p->vel16[0], p->vel16[1], p->vel16[2],
        ctx->n_cells);
    ctx->launches++;
    return cudaGetLastError();
}

cudaError_t launch_vel_decode(cube2_ctx *ctx, const cube2_particles *p, float *const v[3]) {
    const int64_t blocks = (ctx->N + 255) / 256;
    if (blocks == 0) return cudaSuccess;
    vel_decode_kernel<<<(unsigned)blocks, 256, 0, ctx->stream>>>(p->vel16[0], p->vel16[1], p->vel16[2], ctx->cellid,
                                                                p->vscale, v[0], v[1], v[2], ctx->N);
    ctx->launches++;
    return cudaGetLastError();
}

int64_t scan_scratch_len(int64_t n) {
    int64_t total = 0;
    while (n > SCAN_CHUNK) {
        n = (n + SCAN_CHUNK - 1) / SCAN_CHUNK;
        total += n;
    }
    return total + 1;
}

cudaError_t launch_scan(cube2_ctx *ctx, const int32_t *in, int32_t *out, int64_t n) {
    // the callers' arrays may lie anywhere (4-byte words): wide loads only where both allow them
    const bool wide = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    if (n <= SCAN_CHUNK) {
        launch_chained(ctx->chained, scan_apply_kernel, 1, SCAN_THREADS, 0, ctx->stream, in, out, n, nullptr, wide);
        ctx->launches++;
        return cudaGetLastError();
    }
    // level sums live in ctx->scan_tmp, consumed recursively
    const int64_t nb = (n + SCAN_CHUNK - 1) / SCAN_CHUNK;
    int32_t *sums = ctx->scan_tmp;
    // reserve this level's sums, recurse on the remainder of the scratch
    launch_chained(ctx->chained, scan_reduce_kernel, (unsigned)nb, SCAN_THREADS, 0, ctx->stream, in, sums, n, wide);
    ctx->launches++;
    int32_t *saved = ctx->scan_tmp;
    ctx->scan_tmp = saved + nb;
    cudaError_t e = launch_scan(ctx, sums, sums, nb);
    ctx->scan_tmp = saved;
    if (e != cudaSuccess) return e;
    launch_chained(ctx->chained, scan_apply_kernel, (unsigned)nb, SCAN_THREADS, 0, ctx->stream, in, out, n, sums, wide);
    ctx->launches++;
    return cudaGetLastError();
}

cudaError_t launch_kick(cube2_ctx *ctx, const cube2_particles *p, float kick) {
    const int64_t blocks = (ctx->N + 255) / 256;
    if (blocks == 0) return cudaSuccess;
    ProfScope prof(ctx, P_KICK, 0);
    kick_kernel<<<(unsigned)blocks, 256, 0, ctx->stream>>>(p->vel[0], p->vel[1], p->vel[2], p->acc[0], p->acc[1],
                                                          p->acc[2], ctx->N, kick, ctx->dev_status);
    ctx->launches++;
    return cudaGetLastError();
}

static Moved moved(const cube2_ctx *ctx) {
    return {reinterpret_cast<float4 *>(ctx->moved16), reinterpret_cast<int2 *>(ctx->moved8), ctx->tslot};
}

cudaError_t launch_kick_drift(cube2_ctx *ctx, const cube2_particles *p, float kick, float drift_fix) {
    DriftParams P{};
    P.off0 = p->off[0]; P.off1 = p->off[1]; P.off2 = p->off[2];
    P.vel0 = p->vel[0]; P.vel1 = p->vel[1]; P.vel2 = p->vel[2];
    if (ctx->vel32) {
        P.v16_0 = p->vel16[0]; P.v16_1 = p->vel16[1]; P.v16_2 = p->vel16[2];
        P.vscale = p->vscale;
    }
    P.acc0 = p->acc[0]; P.acc1 = p->acc[1]; P.acc2 = p->acc[2];
    P.cellid = ctx->cellid;
    P.count = p->count;
    P.to = moved(ctx);
    P.N = ctx->N;
    P.n_ios = ctx->n_ios;
    P.kick = kick;
    P.drift_fix = drift_fix;
    P.status = ctx->dev_status;
    ProfScope prof(ctx, P_KICK_DRIFT, 0);
    cudaError_t e = cudaMemsetAsync(p->count, 0, sizeof(int32_t) * ctx->n_cells, ctx->stream);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (ctx->N + 255) / 256;
    if (blocks == 0) return cudaSuccess;
    launch_chained(ctx->chained, kick_drift_kernel, (unsigned)blocks, 256, 0, ctx->stream, P);
    ctx->launches++;
    return cudaGetLastError();
}

cudaError_t launch_place(cube2_ctx *ctx, const double *const pos[3], const float *const mom[3],
                         const cube2_particles *p) {
    PlaceParams P{};
    P.pos0 = pos[0]; P.pos1 = pos[1]; P.pos2 = pos[2];
    if (mom) { P.mom0 = mom[0]; P.mom1 = mom[1]; P.mom2 = mom[2]; }
    P.count = p->count;
    P.to = moved(ctx);
    P.N = ctx->N;
    P.n_ios = ctx->n_ios;
    P.s_ios = ctx->s_ios;
    reciprocal(ctx->s_ios, P.recip, P.recip_shift);
    P.status = ctx->dev_status;
    cudaError_t e = cudaMemsetAsync(p->count, 0, sizeof(int32_t) * ctx->n_cells, ctx->stream);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (ctx->N + 255) / 256;
    if (blocks == 0) return cudaSuccess;
    place_kernel<<<(unsigned)blocks, 256, 0, ctx->stream>>>(P);
    ctx->launches++;
    return cudaGetLastError();
}

cudaError_t launch_rebin(cube2_ctx *ctx, const cube2_particles *p) {
    cudaError_t e;
    {
        ProfScope prof(ctx, P_SCAN, 0);
        e = launch_scan(ctx, p->count, p->start, ctx->n_cells);
    }
    if (e != cudaSuccess) return e;
    const int64_t pb = (ctx->N + 255) / 256, cb = (ctx->n_cells + 255) / 256;
    if (pb > 0) {
        {
            ProfScope prof(ctx, P_SCATTER, 0);
            launch_chained(ctx->chained, scatter_kernel, (unsigned)pb, 256, 0, ctx->stream, moved(ctx), p->start, ctx->perm2, ctx->N);
        }
        e = cudaMemsetAsync(ctx->big_n, 0, 2 * sizeof(int), ctx->stream);
        if (e != cudaSuccess) return e;
        {
            ProfScope prof(ctx, P_SORT, 0);
            sort_list_kernel<<<(unsigned)((cb + 3) / 4), 256, 0, ctx->stream>>>(
                p->count, ctx->n_cells, ctx->big, ctx->big_n, (reinterpret_cast<uintptr_t>(p->count) & 15) == 0);
        }
        {
            ProfScope prof(ctx, P_SORT_BIG, 0);
            launch_chained(ctx->chained, sort_cells_kernel, (unsigned)(ctx->num_sms * (1536 / SORT_THREADS)), SORT_THREADS, 0, ctx->stream,
                p->count, p->start, ctx->perm2, ctx->perm, ctx->big, ctx->big_n, ctx->n_cells);
        }
        GatherParams G{};
        G.slots = ctx->perm2;
        G.perm = ctx->perm;
        G.count = p->count;
        G.start = p->start;
        G.from = moved(ctx);
        G.off0 = p->off[0]; G.off1 = p->off[1]; G.off2 = p->off[2];
        if (ctx->vel32) {   // FP16 storage: the step's FP32 working copy
            G.vel0 = ctx->vel32; G.vel1 = ctx->vel32 + ctx->N; G.vel2 = ctx->vel32 + 2 * ctx->N;
        } else {
            G.vel0 = p->vel[0]; G.vel1 = p->vel[1]; G.vel2 = p->vel[2];
        }
        G.cellid = ctx->cellid;
        G.N = ctx->N;
        {
            ProfScope prof(ctx, P_GATHER, 0);
            launch_chained(ctx->chained, gather_kernel, (unsigned)pb, 256, 0, ctx->stream, G);
        }
        ctx->launches += 4;
    }
    return cudaGetLastError();
}

}  // namespace cube2
