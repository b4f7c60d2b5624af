// 3-D real FFT Poisson solve of one PM level (paper Sec. 2.1.2: phi(k) = rho(k) G(k);
// Sec. 2.2.2: batches of 1-D line FFTs along each axis).
//
// Layout: real grid [z][y][x] (x fastest, n^3 FP32); half spectrum
// [kz][ky][kx] complex64 with kx in [0, n/2] stored in rows of kxp >= n/2+1
// (multiple of 16, so every row starts on a 128-byte boundary).
//
// Passes (each one read + one write of the grid, in place where possible):
//   X  r2c : two real rows packed as one complex line a + ib, one complex FFT per
//            line, split into the two half spectra.
//   Y      : L consecutive kx columns x n rows of one kz plane per CTA.
//   Z+G    : L consecutive kx columns x n planes of one ky row per CTA: forward
//            FFT along z, multiply by G(k) (1/n^3 folded in), inverse FFT along z.
//   Y^-1, X^-1 c2r : mirror images of Y and X.
// A line is transformed by a Stockham autosort sequence of radix-16/8/4/3/2 stages
// (natural order in and out): a stage takes R values with stride n/R, applies
// the twiddles exp(-2 pi i r (j mod Ns) / (Ns R)), does an R-point DFT in
// registers and puts them with stride Ns to position (j / Ns) Ns R + (j mod Ns).
// The first stage takes its values straight from global memory and the last one
// writes them there, so a line of three stages crosses shared memory twice; the
// passes are bound by that crossing, not by DRAM.  In the z pass the forward
// transform's last stage leaves each thread the values that the inverse's first
// stage wants (the inverse runs the radices in reverse), with G applied between
// them in registers.  In the x passes the threads of a line take the last
// (first) stage's butterflies in pairs j, n/R - j, which hold both members of
// every conjugate pair k, n - k: the two half spectra are split (joined) in
// registers.  512^3: x 0.35 -> 0.18 ms each (0.165 at the copy rate), z + G 0.41 -> 0.38, y
// 0.23 -> 0.24 (the rate of its strided rows); all five 1.58 -> 1.23 ms, at 1024^3
// 15.5 -> 10.3 ms, at 128^3 59 -> 44 us, against every stage through shared memory.
// Twiddles are FP32 tables built from FP64 sincospi, one row of n/R entries per
// stage and factor r, so that a stage's reads are consecutive.
#include "common.cuh"
#include "fft_plan.cuh"

#include <algorithm>
#include <string>

namespace cube2 {
namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// multiply by -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 rot90(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <int R, bool INV>
struct Dft;

template <bool INV>
struct Dft<2, INV> {
    __device__ __forceinline__ static void run(float2 *v) {
        const float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};

template <bool INV>
struct Dft<4, INV> {
    __device__ __forceinline__ static void run(float2 *v) {
        const float2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        const float2 s13 = cadd(v[1], v[3]), d13 = rot90<INV>(csub(v[1], v[3]));
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd(d02, d13);
        v[3] = csub(d02, d13);
    }
};

template <bool INV>
struct Dft<8, INV> {
    __device__ __forceinline__ static void run(float2 *v) {
        const float h = 0.70710678118654752440f;
        // radix-2 split: even/odd halves
        float2 a[4] = {v[0], v[2], v[4], v[6]};
        float2 b[4] = {v[1], v[3], v[5], v[7]};
        Dft<4, INV>::run(a);
        Dft<4, INV>::run(b);
        // twiddle b[k] by w8^k, w8 = exp(-+ i pi/4)
        const float2 b1 = b[1], b3 = b[3];
        b[1] = INV ? make_float2(h * (b1.x - b1.y), h * (b1.x + b1.y))
                   : make_float2(h * (b1.x + b1.y), h * (b1.y - b1.x));
        b[2] = rot90<INV>(b[2]);
        b[3] = INV ? make_float2(-h * (b3.x + b3.y), h * (b3.x - b3.y))
                   : make_float2(h * (b3.y - b3.x), -h * (b3.x + b3.y));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = cadd(a[k], b[k]);
            v[k + 4] = csub(a[k], b[k]);
        }
    }
};

template <bool INV>
struct Dft<16, INV> {   // 4 x 4
    __device__ __forceinline__ static void run(float2 *v) {
        constexpr float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f, h = 0.70710678118654752440f;
        // w16^m, m = n2 k1 (forward: exp(-i pi m / 8))
        constexpr float C[10] = {1.0f, c1, h, s1, 0.0f, 0.0f, -h, 0.0f, 0.0f, -c1};
        constexpr float D[10] = {0.0f, s1, h, c1, 1.0f, 0.0f, h, 0.0f, 0.0f, -s1};
        float2 a[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
            for (int n1 = 0; n1 < 4; ++n1) a[n2][n1] = v[4 * n1 + n2];
            Dft<4, INV>::run(a[n2]);
        }
#pragma unroll
        for (int n2 = 1; n2 < 4; ++n2)
#pragma unroll
            for (int k1 = 1; k1 < 4; ++k1) {
                const int m = n2 * k1;
                const float2 b = a[n2][k1];
                if (m == 4) a[n2][k1] = rot90<INV>(b);
                else a[n2][k1] = cmul(b, make_float2(C[m], INV ? D[m] : -D[m]));
            }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            float2 b[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
            Dft<4, INV>::run(b);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = b[k2];
        }
    }
};

template <bool INV>
struct Dft<3, INV> {
    __device__ __forceinline__ static void run(float2 *v) {
        const float c = -0.5f;
        const float s = INV ? 0.86602540378443864676f : -0.86602540378443864676f;
        const float2 t = cadd(v[1], v[2]);
        const float2 d = csub(v[1], v[2]);
        const float2 m = make_float2(v[0].x + c * t.x, v[0].y + c * t.y);
        const float2 r = make_float2(-s * d.y, s * d.x);   // i s d
        v[0] = cadd(v[0], t);
        v[1] = cadd(m, r);
        v[2] = csub(m, r);
    }
};

template <int N, bool INV, bool XP>
struct Plan {
    static constexpr int S = stages_of(N, XP);
    __host__ __device__ static constexpr int radix(int s) { return radix_at(N, INV ? S - 1 - s : s, XP); }
    __host__ __device__ static constexpr int span(int s) {   // Ns: product of the earlier radices
        int v = 1;
        for (int i = 0; i < s; ++i) v *= radix(i);
        return v;
    }
};

// The fraction of a turn of entry idx, if it lies in one of a line's rows from stage s on.
template <int N, bool XP, bool INV, int s>
__device__ __forceinline__ void twiddle_turn(int idx, int &num, int &den) {
    if constexpr (s < stages_of(N, XP)) {
        constexpr int R = Plan<N, INV, XP>::radix(s), NB = N / R, NS = Plan<N, INV, XP>::span(s), at = twiddle_row(N, XP, INV, s);
        if (idx >= at && idx < at + (R - 1) * NB) {
            num = (INV ? 1 : -1) * (((idx - at) / NB + 1) * ((idx - at) % NB % NS));
            den = NS * R;
        }
        twiddle_turn<N, XP, INV, s + 1>(idx, num, den);
    }
}

// Sizes are template parameters: with the rows looked up at run time the kernel took
// longer than the five passes of a small mesh, whose allocation-free solve makes its
// twiddles in each call (64^3 81 us a call, 96^3 172).
constexpr int TWIDDLE_THREADS = 64;
template <int N>
__global__ void __launch_bounds__(TWIDDLE_THREADS) twiddle_rows_kernel(float2 *tw) {
    const int idx = blockIdx.x * TWIDDLE_THREADS + threadIdx.x;
    if (idx >= twiddle_entries(N)) return;
    int num = 0, den = 1;
    twiddle_turn<N, false, false, 1>(idx, num, den);
    twiddle_turn<N, false, true, 1>(idx, num, den);
    twiddle_turn<N, true, false, 1>(idx, num, den);
    twiddle_turn<N, true, true, 1>(idx, num, den);
    double si, co;
    sincospi(2.0 * (double)num / (double)den, &si, &co);
    tw[idx] = make_float2((float)co, (float)si);
}
template <int N>
cudaError_t make_twiddles(float2 *tw, cudaStream_t st) {
    twiddle_rows_kernel<N><<<(twiddle_entries(N) + TWIDDLE_THREADS - 1) / TWIDDLE_THREADS, TWIDDLE_THREADS, 0, st>>>(tw);
    return cudaGetLastError();
}

// Values of stage s's butterflies j twiddled and transformed; nothing to twiddle in stage 0.
template <int N, bool INV, bool XP, int s, int R>
__device__ __forceinline__ void butterfly(float2 (&v)[R], int j, const float2 *__restrict__ tw) {
    if constexpr (s > 0) {
        constexpr int row = twiddle_row(N, XP, INV, s);
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(&tw[row + (r - 1) * (N / R) + j]));
    }
    Dft<R, INV>::run(v);
}

// ------------------------------------------------------- tiles of y and z
// L lines (columns) per tile, position-major in shared memory: a row of a tile
// is 16 consecutive complex values (128 bytes) in shared memory as in global.
// Thread b takes butterflies b, b + T, ... of every stage: line b % L, j = b / L.
// About 16 values (24 with a radix 3) per thread: at 512 two CTAs of 512 threads
// per SM with 64 registers.  A 1024-point tile of 16 lines leaves one CTA per SM:
// its y passes take 8 lines (2.34 -> 1.83 ms), the z pass, with the strides of
// whole planes, stays at 16 (3.85 against 4.26 ms).  Up to 128 points the grids
// are small and registers are left to the compiler (z at 64: 8.9 -> 6.7 us).
template <int N, bool Z>
struct Tile {
    static constexpr int L = N >= 2048 || (N == 1024 && !Z) ? 8 : FFT_LINES;
    static constexpr int V = (N % 3 == 0 ? 3 : 2) * (N <= 96 ? 4 : 8);
    static constexpr int T0 = N * L / V;
    static constexpr int T = T0 < 32 ? 32 : (T0 > 1024 ? 1024 : T0);
    static constexpr size_t SMEM = (size_t)N * L * sizeof(float2);
    static constexpr int MINB = (N > 128 && T <= 512 && 2 * SMEM <= 200 * 1024) ? (N % 3 == 0 ? 768 : 1024) / T : 1;
    template <int R>
    static constexpr int per() { return (N / R * L + T - 1) / T; }
};

// Tiles are read and written once a pass: streaming loads and stores (512^3: z
// 0.41 -> 0.38 ms); past 512 the plain L2 ones (z at 1024: 3.85 against 4.00 ms).
// volatile: not moved above chain().
template <int N>
__device__ __forceinline__ float2 tile_load(const float2 *p) {
    float2 v;
    if constexpr (N <= 512)
        asm volatile("ld.global.cs.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(__cvta_generic_to_global(p)) : "memory");
    else
        asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(__cvta_generic_to_global(p)) : "memory");
    return v;
}
template <int N>
__device__ __forceinline__ void tile_store(float2 *p, float2 v) {
    if constexpr (N <= 512) __stcs(p, v);
    else __stcg(p, v);
}

// Stages s .. of the tile's lines.  In stage 0 the values come from load(pos,
// line); the last stage hands its values to store(pos, line, v) or, with KEEP,
// leaves them in out.
template <int N, bool Z, bool INV, int s, class Load, class Store>
__device__ __forceinline__ void tile_stages(float2 *S, const float2 *__restrict__ tw, Load load, Store store) {
    using TL = Tile<N, Z>;
    constexpr int R = Plan<N, INV, false>::radix(s), NB = N / R, NS = Plan<N, INV, false>::span(s), L = TL::L, T = TL::T;
    constexpr int PER = TL::template per<R>();
    constexpr bool LAST = s + 1 == Plan<N, INV, false>::S;
    float2 v[PER][R];
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int b = threadIdx.x + p * T;
        if (NB * L % T == 0 || b < NB * L) {
            const int line = b % L, j = b / L;
#pragma unroll
            for (int r = 0; r < R; ++r) v[p][r] = s == 0 ? load(j + r * NB, line, p, r) : S[(j + r * NB) * L + line];
        }
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int b = threadIdx.x + p * T;
        if (NB * L % T == 0 || b < NB * L) butterfly<N, INV, false, s>(v[p], b / L, tw);
    }
    if constexpr (!LAST) {
        if (s > 0) __syncthreads();   // all have read what is overwritten now
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int b = threadIdx.x + p * T;
            if (NB * L % T == 0 || b < NB * L) {
                const int line = b % L, j = b / L, base = (j / NS) * NS * R + j % NS;
#pragma unroll
                for (int r = 0; r < R; ++r) S[(base + r * NS) * L + line] = v[p][r];
            }
        }
        __syncthreads();
        tile_stages<N, Z, INV, s + 1>(S, tw, load, store);
    } else {
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int b = threadIdx.x + p * T;
            if (NB * L % T == 0 || b < NB * L) {
                const int line = b % L, j = b / L;
#pragma unroll
                for (int r = 0; r < R; ++r) store(j + r * NS, line, p, r, v[p][r]);   // NS = NB: base is j
            }
        }
    }
}

// ---------------------------------------------------------------- X passes
// Each pass is a per-block body with two entry kernels: one block per tile for
// a single mesh (BATCH = false), or, for the batched meshes of the adaptive
// third level (BATCH = true), a resident-sized grid whose blocks loop over the
// tiles of the meshes in use (*active, on the device).
//
// TL threads per line (a warp or a part of one up to 1024 / 3 * 2 points: the
// stages then meet at warp barriers only; beyond that 64 or 128 threads at a
// named barrier), lanes along the line: global rows are read and written in
// full sectors.  In shared memory position p of a line lies at p + p / 8.
template <int N>
struct XLine {
    static constexpr int V = N % 3 == 0 ? (N == 48 || N == 12 ? 12 : 24) : (N == 32 || N == 16 ? 8 : N == 8 ? 4 : 16);
    static constexpr int TL0 = N / V;
    static constexpr int TL = N == 12 ? 2 : N == 24 ? 4 : TL0;
    static constexpr int CTA = 256;
    static constexpr int MINB = N % 3 == 0 ? 3 : 4;   // 64 registers; 80 with a radix 3
    static constexpr int LINES = CTA / TL;
    static constexpr int PITCH = N + N / 8;
    static constexpr size_t SMEM = (size_t)LINES * PITCH * sizeof(float2);
    static constexpr int R1 = radix_at(N, stages_of(N, true) - 1, true);   // radix of the paired stage
    static constexpr int NB1 = N / R1, PAIRS = NB1 / 2 / TL;
    static_assert(NB1 % 2 == 0 && NB1 / 2 % TL == 0, "paired butterflies deal out evenly");
    __device__ __forceinline__ static void sync(int line) {
        if constexpr (TL <= 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(line + 1), "r"(TL) : "memory");
    }
};

__device__ __forceinline__ int pad8(int p) { return p + (p >> 3); }

// One plain stage (not the paired one) of a line: values from load or shared
// memory, to shared memory or store.
template <int N, bool INV, int s, class Load, class Store>
__device__ __forceinline__ void line_stage(float2 *S, int t, int line, const float2 *__restrict__ tw, Load load,
                                           Store store) {
    using X = XLine<N>;
    constexpr int R = Plan<N, INV, true>::radix(s), NB = N / R, NS = Plan<N, INV, true>::span(s), TL = X::TL;
    constexpr int PER = (NB + TL - 1) / TL;
    constexpr bool LAST = s + 1 == Plan<N, INV, true>::S;
    float2 v[PER][R];
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int j = t + p * TL;
        if (NB % TL == 0 || j < NB) {
#pragma unroll
            for (int r = 0; r < R; ++r) v[p][r] = s == 0 ? load(j + r * NB) : S[pad8(j + r * NB)];
        }
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int j = t + p * TL;
        if (NB % TL == 0 || j < NB) butterfly<N, INV, true, s>(v[p], j, tw);
    }
    if (!LAST && s > 0) X::sync(line);
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int j = t + p * TL;
        if (NB % TL == 0 || j < NB) {
            const int base = (j / NS) * NS * R + j % NS;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if constexpr (LAST) store(base + r * NS, v[p][r]);
                else S[pad8(base + r * NS)] = v[p][r];
            }
        }
    }
    if (!LAST) X::sync(line);
}

template <int N, bool INV, int s, int END, class Load, class Store>
__device__ __forceinline__ void line_stages(float2 *S, int t, int line, const float2 *__restrict__ tw, Load load,
                                            Store store) {
    if constexpr (s < END) {
        line_stage<N, INV, s>(S, t, line, tw, load, store);
        line_stages<N, INV, s + 1, END>(S, t, line, tw, load, store);
    }
}

template <int N>
__device__ __forceinline__ void x_r2c_block(float2 *smem, const float *in, float2 *__restrict__ out,
                                            int64_t nlines, int kxp, const float2 *__restrict__ tw, int64_t vb) {
    using X = XLine<N>;
    constexpr int R = X::R1, NB = X::NB1, TL = X::TL, LAST = Plan<N, false, true>::S - 1;
    const int line = threadIdx.x / TL, t = threadIdx.x % TL;
    const int64_t want = vb * X::LINES + line, l = want < nlines ? want : nlines - 1;   // spare threads repeat the last
    const float *a = in + 2 * l * N, *b = a + N;
    float2 *S = smem + line * X::PITCH;
    line_stages<N, false, 0, LAST>(S, t, line, tw, [&](int x) { return make_float2(a[x], b[x]); },
                                   [](int, float2) {});
    float2 *A = out + 2 * l * kxp, *B = A + kxp;
#pragma unroll
    for (int i = 0; i < X::PAIRS; ++i) {
        // butterflies q and NB - q (0 and NB / 2): outputs k = q + r NB and their conjugates' n - k
        const int q = t + i * TL, jb = q ? NB - q : NB / 2;
        float2 va[R], vb2[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            va[r] = S[pad8(q + r * NB)];
            vb2[r] = S[pad8(jb + r * NB)];
        }
        butterfly<N, false, true, LAST>(va, q, tw);
        butterfly<N, false, true, LAST>(vb2, jb, tw);
        auto split = [&](int k, float2 z, float2 zc) {
            A[k] = make_float2(0.5f * (z.x + zc.x), 0.5f * (z.y - zc.y));
            B[k] = make_float2(0.5f * (z.y + zc.y), -0.5f * (z.x - zc.x));
        };
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 ca = q ? vb2[R - 1 - r] : va[(R - r) % R], cb = q ? va[R - 1 - r] : vb2[R - 1 - r];
            if (q + r * NB <= N / 2) split(q + r * NB, va[r], ca);
            if (jb + r * NB <= N / 2) split(jb + r * NB, vb2[r], cb);
        }
    }
}

template <int N>
__device__ __forceinline__ void x_c2r_block(float2 *smem, const float2 *in, float *__restrict__ out,
                                            int64_t nlines, int kxp, const float2 *__restrict__ tw, int64_t vb) {
    using X = XLine<N>;
    constexpr int R = X::R1, NB = X::NB1, TL = X::TL;
    const int line = threadIdx.x / TL, t = threadIdx.x % TL;
    const int64_t want = vb * X::LINES + line, l = want < nlines ? want : nlines - 1;
    const float2 *A = in + 2 * l * kxp, *B = A + kxp;
    float2 *S = smem + line * X::PITCH;
#pragma unroll
    for (int i = 0; i < X::PAIRS; ++i) {
        const int q = t + i * TL, jb = q ? NB - q : NB / 2;
        float2 va[R], vb2[R];
        // Z[k] = A + iB and Z[n - k] = conj(A) + i conj(B) of every k <= n/2 that q or NB - q holds
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int ka = q + r * NB, kb = jb + r * NB;
            if (ka <= N / 2) {
                float2 x = A[ka], y = B[ka];
                if (ka == 0 || ka == N / 2) x.y = y.y = 0.0f;
                const float2 z = make_float2(x.x - y.y, x.y + y.x), zc = make_float2(x.x + y.y, y.x - x.y);
                va[r] = z;
                if (q) vb2[R - 1 - r] = zc;
                else if (ka != 0 && ka != N / 2) va[(R - r) % R] = zc;
            }
            if (kb <= N / 2) {
                float2 x = A[kb], y = B[kb];
                if (kb == N / 2) x.y = y.y = 0.0f;
                const float2 z = make_float2(x.x - y.y, x.y + y.x), zc = make_float2(x.x + y.y, y.x - x.y);
                vb2[r] = z;
                if (q) va[R - 1 - r] = zc;
                else if (kb != N / 2) vb2[R - 1 - r] = zc;
            }
        }
        Dft<R, true>::run(va);
        Dft<R, true>::run(vb2);
#pragma unroll
        for (int r = 0; r < R; ++r) {   // the first stage of the inverse: span 1
            S[pad8(q * R + r)] = va[r];
            S[pad8(jb * R + r)] = vb2[r];
        }
    }
    X::sync(line);
    float *a = out + 2 * l * N, *b = a + N;
    line_stages<N, true, 1, Plan<N, true, true>::S>(S, t, line, tw, [](int) { return make_float2(0.f, 0.f); },
                                              [&](int x, float2 v) {
                                                  a[x] = v.x;
                                                  b[x] = v.y;
                                              });
}

template <int N, bool BATCH>
__global__ void __launch_bounds__(XLine<N>::CTA, XLine<N>::MINB) fft_x_r2c(const float *in, float2 *__restrict__ out,
                                                              int64_t nlines, int kxp, const float2 *__restrict__ tw,
                                                              const int *active) {
    chain();
    extern __shared__ __align__(16) float2 S[];
    if constexpr (BATCH) {
        nlines = (int64_t)*active * N * N / 2;
        for (int64_t vb = blockIdx.x; vb * XLine<N>::LINES < nlines; vb += gridDim.x) {
            x_r2c_block<N>(S, in, out, nlines, kxp, tw, vb);
            __syncthreads();
        }
    } else {
        x_r2c_block<N>(S, in, out, nlines, kxp, tw, blockIdx.x);
    }
}

template <int N, bool BATCH>
__global__ void __launch_bounds__(XLine<N>::CTA, XLine<N>::MINB) fft_x_c2r(const float2 *in, float *__restrict__ out,
                                                              int64_t nlines, int kxp, const float2 *__restrict__ tw,
                                                              const int *active) {
    chain();
    extern __shared__ __align__(16) float2 S[];
    if constexpr (BATCH) {
        nlines = (int64_t)*active * N * N / 2;
        for (int64_t vb = blockIdx.x; vb * XLine<N>::LINES < nlines; vb += gridDim.x) {
            x_c2r_block<N>(S, in, out, nlines, kxp, tw, vb);
            __syncthreads();
        }
    } else {
        x_c2r_block<N>(S, in, out, nlines, kxp, tw, blockIdx.x);
    }
}

// ---------------------------------------------------------------- Y passes
template <int N, bool INV>
__device__ __forceinline__ void y_block(float2 *S, float2 *__restrict__ data, int kxp, const float2 *__restrict__ tw,
                                        int64_t vb) {
    using TL = Tile<N, false>;
    const int tiles_x = kxp / TL::L;
    const int tx = (int)(vb % tiles_x);
    const int64_t z = vb / tiles_x;                    // plane over all batched meshes
    float2 *base = data + z * N * kxp + tx * TL::L;
    tile_stages<N, false, INV, 0>(
        S, tw, [&](int y, int line, int, int) { return tile_load<N>(&base[(int64_t)y * kxp + line]); },
        [&](int y, int line, int, int, float2 v) { tile_store<N>(&base[(int64_t)y * kxp + line], v); });
}

template <int N, bool INV, bool BATCH>
__global__ void __launch_bounds__(Tile<N, false>::T, Tile<N, false>::MINB) fft_y(float2 *__restrict__ data, int kxp,
                                                                   const float2 *__restrict__ tw,
                                                                   const int *active) {
    chain();
    extern __shared__ __align__(16) float2 S[];
    if constexpr (BATCH) {
        const int64_t nvb = (int64_t)*active * N * (kxp / Tile<N, false>::L);
        for (int64_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
            y_block<N, INV>(S, data, kxp, tw, vb);
            __syncthreads();
        }
    } else {
        y_block<N, INV>(S, data, kxp, tw, blockIdx.x);
    }
}

// ------------------------------------------------------------ Z (+ Green)
// GMODE 0: forward z FFT only; 1: G from a full [kz][ky][kxp] table; 2: G
// from the symmetry-reduced table (green_index); 3: G from the table folded in
// ky and kz ([kz <= N/2][ky <= N/2][kxp], the reduced table's entries).
template <int N, int GMODE>
__device__ __forceinline__ void z_block(float2 *S, float2 *__restrict__ data, const float *__restrict__ green,
                                        int kxp, const float2 *__restrict__ tw, int64_t vb) {
    using TL = Tile<N, true>;
    constexpr int L = TL::L;
    const int tiles_x = kxp / L;
    const int tx = (int)(vb % tiles_x);
    const int64_t row = vb / tiles_x;                     // (mesh, ky) over all batched meshes
    const int64_t mesh = row / N;
    const int ky = (int)(row - mesh * N);
    const int64_t zstride = (int64_t)N * kxp;
    float2 *base = data + mesh * N * zstride + (int64_t)ky * kxp + tx * L;
    auto load = [&](int z, int line, int, int) { return tile_load<N>(&base[z * zstride + line]); };
    auto store = [&](int z, int line, int, int, float2 v) { tile_store<N>(&base[z * zstride + line], v); };
    if constexpr (GMODE == 0) {
        tile_stages<N, true, false, 0>(S, tw, load, store);
    } else {
        // the forward's last stage and the inverse's first have the same radix
        // and positions: the values stay with their thread
        constexpr int R = Plan<N, false, false>::radix(Plan<N, false, false>::S - 1);
        static_assert(R == Plan<N, true, false>::radix(0), "radices reversed");
        float2 keep[TL::template per<R>()][R];
        tile_stages<N, true, false, 0>(S, tw, load, [&](int z, int line, int p, int r, float2 v) {
            const int kx = tx * L + line;
            float g;
            if (GMODE == 1) {
                g = __ldg(&green[(int64_t)z * zstride + (int64_t)ky * kxp + kx]);
            } else if (GMODE == 3) {
                const int zf = z <= N / 2 ? z : N - z, kyf = ky <= N / 2 ? ky : N - ky;
                g = __ldg(&green[((int64_t)zf * (N / 2 + 1) + kyf) * kxp + kx]);
            } else {   // padding columns (kx > N/2) hold zeros
                g = kx <= N / 2 ? __ldg(&green[green_index(kx, ky, z, N)]) : 0.0f;
            }
            keep[p][r] = make_float2(v.x * g, v.y * g);
        });
        __syncthreads();   // the inverse's first exchange overwrites what the forward's last stage has read
        tile_stages<N, true, true, 0>(S, tw, [&](int, int, int p, int r) { return keep[p][r]; }, store);
    }
}

template <int N, int GMODE, bool BATCH>
__global__ void __launch_bounds__(Tile<N, true>::T, Tile<N, true>::MINB) fft_z(float2 *__restrict__ data, const float *__restrict__ green,
                                                   int kxp, const float2 *__restrict__ tw, const int *active) {
    chain();
    extern __shared__ __align__(16) float2 S[];
    if constexpr (BATCH) {
        const int64_t nvb = (int64_t)*active * N * (kxp / Tile<N, true>::L);
        for (int64_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
            z_block<N, GMODE>(S, data, green, kxp, tw, vb);
            __syncthreads();
        }
    } else {
        z_block<N, GMODE>(S, data, green, kxp, tw, blockIdx.x);
    }
}

// Grid of a pass: every block for a single mesh; for batched meshes a
// resident-sized grid that loops over the blocks of the meshes in use.
inline unsigned pass_grid(const cube2_ctx *ctx, const Level &Lv, int64_t blocks) {
    return (unsigned)(Lv.active ? std::min<int64_t>(blocks, (int64_t)ctx->num_sms * 16) : blocks);
}

// the batched variants exist for the local meshes of the adaptive third level
constexpr int BATCH_MAX_N = 256;

template <int N>
struct Launcher {
    template <bool B>
    static cudaError_t forward_v(cube2_ctx *ctx, Level &Lv) {
        const int64_t nlines = (int64_t)Lv.batch * N * N / 2;
        const unsigned bx = pass_grid(ctx, Lv, (nlines + XLine<N>::LINES - 1) / XLine<N>::LINES);
        {
            ProfScope prof(ctx, B ? -1 : P_FFT_X_FWD, Lv.index);   // batched meshes: profiled as one group by the caller
            launch_chained(ctx->chained, fft_x_r2c<N, B>, bx, XLine<N>::CTA, XLine<N>::SMEM, ctx->stream, Lv.real, Lv.spec, nlines, Lv.kxp, Lv.tw,
                                                                            Lv.active);
        }
        const unsigned by = pass_grid(ctx, Lv, (int64_t)Lv.batch * N * (Lv.kxp / Tile<N, false>::L));
        {
            ProfScope prof(ctx, B ? -1 : P_FFT_Y_FWD, Lv.index);
            launch_chained(ctx->chained, fft_y<N, false, B>, by, Tile<N, false>::T, Tile<N, false>::SMEM, ctx->stream, Lv.spec, Lv.kxp, Lv.tw, Lv.active);
        }
        ctx->launches += 2;
        return cudaGetLastError();
    }
    template <bool B>
    static cudaError_t z_pass_v(cube2_ctx *ctx, Level &Lv, bool green) {
        const unsigned bz = pass_grid(ctx, Lv, (int64_t)Lv.batch * N * (Lv.kxp / Tile<N, true>::L));
        ProfScope prof(ctx, B ? -1 : P_FFT_Z_GREEN, Lv.index);
        if (green && !B && Lv.green2)
            launch_chained(ctx->chained, fft_z<N, 3, false>, bz, Tile<N, true>::T, Tile<N, true>::SMEM, ctx->stream, Lv.spec, Lv.green2, Lv.kxp, Lv.tw,
                                                                              Lv.active);
        else if (green)
            launch_chained(ctx->chained, fft_z<N, 2, B>, bz, Tile<N, true>::T, Tile<N, true>::SMEM, ctx->stream, Lv.spec, Lv.green, Lv.kxp, Lv.tw, Lv.active);
        else
            launch_chained(ctx->chained, fft_z<N, 0, B>, bz, Tile<N, true>::T, Tile<N, true>::SMEM, ctx->stream, Lv.spec, nullptr, Lv.kxp, Lv.tw, Lv.active);
        ctx->launches += 1;
        return cudaGetLastError();
    }
    template <bool B>
    static cudaError_t inverse_v(cube2_ctx *ctx, Level &Lv) {
        const unsigned by = pass_grid(ctx, Lv, (int64_t)Lv.batch * N * (Lv.kxp / Tile<N, false>::L));
        {
            ProfScope prof(ctx, B ? -1 : P_FFT_Y_INV, Lv.index);
            launch_chained(ctx->chained, fft_y<N, true, B>, by, Tile<N, false>::T, Tile<N, false>::SMEM, ctx->stream, Lv.spec, Lv.kxp, Lv.tw, Lv.active);
        }
        const int64_t nlines = (int64_t)Lv.batch * N * N / 2;
        const unsigned bx = pass_grid(ctx, Lv, (nlines + XLine<N>::LINES - 1) / XLine<N>::LINES);
        {
            ProfScope prof(ctx, B ? -1 : P_FFT_X_INV, Lv.index);
            launch_chained(ctx->chained, fft_x_c2r<N, B>, bx, XLine<N>::CTA, XLine<N>::SMEM, ctx->stream, Lv.spec, Lv.real, nlines, Lv.kxp, Lv.tw,
                                                                            Lv.active);
        }
        ctx->launches += 2;
        return cudaGetLastError();
    }
    static cudaError_t forward(cube2_ctx *ctx, Level &Lv) {
        const cudaError_t e = setup();
        if (e != cudaSuccess) return e;
        if constexpr (N <= BATCH_MAX_N)
            if (Lv.active) return forward_v<true>(ctx, Lv);
        if (Lv.active) return cudaErrorInvalidValue;
        return forward_v<false>(ctx, Lv);
    }
    static cudaError_t z_pass(cube2_ctx *ctx, Level &Lv, bool green) {
        const cudaError_t e = setup();
        if (e != cudaSuccess) return e;
        if constexpr (N <= BATCH_MAX_N)
            if (Lv.active) return z_pass_v<true>(ctx, Lv, green);
        if (Lv.active) return cudaErrorInvalidValue;
        return z_pass_v<false>(ctx, Lv, green);
    }
    static cudaError_t inverse(cube2_ctx *ctx, Level &Lv) {
        const cudaError_t e = setup();
        if (e != cudaSuccess) return e;
        if constexpr (N <= BATCH_MAX_N)
            if (Lv.active) return inverse_v<true>(ctx, Lv);
        if (Lv.active) return cudaErrorInvalidValue;
        return inverse_v<false>(ctx, Lv);
    }
    template <bool B>
    static cudaError_t setup_v() {
        constexpr size_t y = Tile<N, false>::SMEM, z = Tile<N, true>::SMEM, x = XLine<N>::SMEM;
        return first_error({allow_shared(fft_x_r2c<N, B>, x), allow_shared(fft_x_c2r<N, B>, x),
                            allow_shared(fft_y<N, false, B>, y), allow_shared(fft_y<N, true, B>, y),
                            allow_shared(fft_z<N, 0, B>, z), allow_shared(fft_z<N, 2, B>, z)});
    }
    static cudaError_t setup() {
        static PerDevice made;
        return once_per_device(made, [] {
            cudaError_t e = first_error({setup_v<false>(), allow_shared(fft_z<N, 1, false>, Tile<N, true>::SMEM),
                                         allow_shared(fft_z<N, 3, false>, Tile<N, true>::SMEM)});
            if constexpr (N <= BATCH_MAX_N)
                if (e == cudaSuccess) e = setup_v<true>();
            return e;
        });
    }
};

enum class Op { Twiddles, Forward, ZGreen, ZForward, Inverse };

template <int N>
cudaError_t run_op(cube2_ctx *ctx, Level &Lv, Op op) {
    switch (op) {
        case Op::Twiddles: return make_twiddles<N>(Lv.tw, ctx->stream);
        case Op::Forward: return Launcher<N>::forward(ctx, Lv);
        case Op::ZGreen: return Launcher<N>::z_pass(ctx, Lv, true);
        case Op::ZForward: return Launcher<N>::z_pass(ctx, Lv, false);
        case Op::Inverse: return Launcher<N>::inverse(ctx, Lv);
    }
    return cudaErrorInvalidValue;
}

cudaError_t dispatch(cube2_ctx *ctx, Level &Lv, Op op) {
    switch (Lv.n) {
        case 8: return run_op<8>(ctx, Lv, op);
        case 12: return run_op<12>(ctx, Lv, op);
        case 16: return run_op<16>(ctx, Lv, op);
        case 24: return run_op<24>(ctx, Lv, op);
        case 32: return run_op<32>(ctx, Lv, op);
        case 48: return run_op<48>(ctx, Lv, op);
        case 64: return run_op<64>(ctx, Lv, op);
        case 96: return run_op<96>(ctx, Lv, op);
        case 128: return run_op<128>(ctx, Lv, op);
        case 192: return run_op<192>(ctx, Lv, op);
        case 256: return run_op<256>(ctx, Lv, op);
        case 384: return run_op<384>(ctx, Lv, op);
        case 512: return run_op<512>(ctx, Lv, op);
        case 768: return run_op<768>(ctx, Lv, op);
        case 1024: return run_op<1024>(ctx, Lv, op);
        case 1536: return run_op<1536>(ctx, Lv, op);
        case 2048: return run_op<2048>(ctx, Lv, op);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int64_t fft_twiddle_entries(int n) { return twiddle_entries(n); }

cudaError_t launch_init_twiddles(cube2_ctx *ctx, Level &L) {
    ctx->launches++;
    return dispatch(ctx, L, Op::Twiddles);
}

bool fft_size_supported(int n) {
    switch (n) {
        case 8: case 12: case 16: case 24: case 32: case 48: case 64: case 96: case 128: case 192:
        case 256: case 384: case 512: case 768: case 1024: case 1536: case 2048: return true;
        default: return false;
    }
}

cudaError_t launch_fft_forward(cube2_ctx *ctx, Level &L) { return dispatch(ctx, L, Op::Forward); }
cudaError_t launch_fft_z_green(cube2_ctx *ctx, Level &L) { return dispatch(ctx, L, Op::ZGreen); }
cudaError_t launch_fft_z_forward(cube2_ctx *ctx, Level &L) { return dispatch(ctx, L, Op::ZForward); }
cudaError_t launch_fft_inverse(cube2_ctx *ctx, Level &L) { return dispatch(ctx, L, Op::Inverse); }

cudaError_t launch_fft_batched_solve(cube2_ctx *ctx, Level &L) {
    cudaError_t e = dispatch(ctx, L, Op::Forward);
    if (e == cudaSuccess) e = dispatch(ctx, L, Op::ZGreen);
    if (e == cudaSuccess) e = dispatch(ctx, L, Op::Inverse);
    return e;
}

}  // namespace cube2

// ---------------------------------------------------------------------------
// Allocation-free Poisson solve (cube2_solve_pm_noalloc).
//
// Some callers cannot allocate device memory at the point where they need a
// solve: code that runs under a fixed device-memory budget handed out by its
// host application, or that must not let cudaMalloc/cudaFree synchronise the
// device in the middle of its own work.  For them this variant of solve_pm
// takes the density, the Green's table and the output from the caller and keeps
// its own working memory (spectrum, padded Green's table, twiddles) in one
// file-scope device array, resolved once per device with cudaGetSymbolAddress.
// It calls no allocating CUDA or library routine.
#include <mutex>

namespace cube2 {
namespace {

constexpr int NOALLOC_KXP = ((NOALLOC_MAX_N / 2 + 1) + 15) / 16 * 16;
constexpr size_t NOALLOC_HALF = (size_t)NOALLOC_MAX_N * NOALLOC_MAX_N * NOALLOC_KXP;
constexpr size_t NOALLOC_SPEC_BYTES = NOALLOC_HALF * sizeof(float2);
constexpr size_t NOALLOC_GREEN_BYTES = NOALLOC_HALF * sizeof(float);
constexpr size_t NOALLOC_BYTES = NOALLOC_SPEC_BYTES + NOALLOC_GREEN_BYTES + NOALLOC_TWIDDLES * sizeof(float2);

// Working memory of every cube2_solve_pm_noalloc call on a device (15.7 MB).
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;
void *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

template <int N>
cudaError_t noalloc_passes(const float *rho, float2 *spec, const float *gpad, float *phi, float2 *tw, int kxp,
                           cudaStream_t st) {
    cudaError_t e = Launcher<N>::setup();
    if (e == cudaSuccess) e = make_twiddles<N>(tw, st);
    if (e != cudaSuccess) return e;
    constexpr int L = Tile<N, true>::L;
    static_assert(L == Tile<N, false>::L, "one grid for y and z");
    static_assert(twiddle_entries(N) <= NOALLOC_TWIDDLES && (size_t)N * N * ((N / 2 + 16) / 16 * 16) <= NOALLOC_HALF,
                  "the fixed array holds this size");
    const int64_t nlines = (int64_t)N * N / 2;
    const unsigned bx = (unsigned)((nlines + XLine<N>::LINES - 1) / XLine<N>::LINES);
    const unsigned by = (unsigned)((int64_t)N * (kxp / L));
    fft_x_r2c<N, false><<<bx, XLine<N>::CTA, XLine<N>::SMEM, st>>>(rho, spec, nlines, kxp, tw, nullptr);
    fft_y<N, false, false><<<by, Tile<N, false>::T, Tile<N, false>::SMEM, st>>>(spec, kxp, tw, nullptr);
    fft_z<N, 1, false><<<by, Tile<N, true>::T, Tile<N, true>::SMEM, st>>>(spec, gpad, kxp, tw, nullptr);
    fft_y<N, true, false><<<by, Tile<N, false>::T, Tile<N, false>::SMEM, st>>>(spec, kxp, tw, nullptr);
    fft_x_c2r<N, false><<<bx, XLine<N>::CTA, XLine<N>::SMEM, st>>>(spec, phi, nlines, kxp, tw, nullptr);
    return cudaGetLastError();
}

}  // namespace

void set_context_free_error(const std::string &msg);

}  // namespace cube2

extern "C" int cube2_solve_pm_noalloc(const float *rho, const float *green, float *phi, int32_t n, void *stream) {
    using namespace cube2;
    if (!rho || !green || !phi) {
        set_context_free_error("cube2_solve_pm_noalloc: null pointer");
        return CUBE2_ERR_BAD_ARG;
    }
    if (n > NOALLOC_MAX_N || !fft_size_supported(n)) {
        set_context_free_error("cube2_solve_pm_noalloc: mesh size " + std::to_string(n) +
                               " not supported (2^a 3^b from 8 to " + std::to_string(NOALLOC_MAX_N) + ")");
        return CUBE2_ERR_UNSUPPORTED_SIZE;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        set_context_free_error(std::string("cube2_solve_pm_noalloc: no usable device: ") + cudaGetErrorString(e));
        return CUBE2_ERR_CUDA;
    }
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
        set_context_free_error("cube2_solve_pm_noalloc: device index " + std::to_string(dev) + " beyond the " +
                               std::to_string(NOALLOC_MAX_DEVICES) + " devices this entry point serves");
        return CUBE2_ERR_CUDA;
    }
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_ptr[dev]) {
            e = cudaGetSymbolAddress(&g_noalloc_ptr[dev], g_noalloc_scratch);
            if (e != cudaSuccess) {
                g_noalloc_ptr[dev] = nullptr;
                set_context_free_error(std::string("cube2_solve_pm_noalloc: cudaGetSymbolAddress failed: ") +
                                       cudaGetErrorString(e));
                return CUBE2_ERR_CUDA;
            }
        }
        base = g_noalloc_ptr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char *b = static_cast<unsigned char *>(base);
    float2 *spec = reinterpret_cast<float2 *>(b);
    float *gpad = reinterpret_cast<float *>(b + NOALLOC_SPEC_BYTES);
    float2 *tw = reinterpret_cast<float2 *>(b + NOALLOC_SPEC_BYTES + NOALLOC_GREEN_BYTES);
    const size_t nh = (size_t)(n / 2 + 1);
    // rows of the half spectrum padded to a multiple of 16 columns, as in a
    // context; the array holds the 128^3 layout, so every smaller mesh fits
    const int kxp = (int)((nh + 15) / 16 * 16);
    // the caller's compact [n][n][n/2+1] table into the padded layout; the
    // padding columns, left from earlier calls, are cleared
    e = cudaMemcpy2DAsync(gpad, kxp * sizeof(float), green, nh * sizeof(float), nh * sizeof(float),
                          (size_t)n * n, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && (size_t)kxp > nh)
        e = cudaMemset2DAsync(gpad + nh, kxp * sizeof(float), 0, (kxp - nh) * sizeof(float), (size_t)n * n, st);
    if (e == cudaSuccess) {
        switch (n) {
            case 8: e = noalloc_passes<8>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 12: e = noalloc_passes<12>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 16: e = noalloc_passes<16>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 24: e = noalloc_passes<24>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 32: e = noalloc_passes<32>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 48: e = noalloc_passes<48>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 64: e = noalloc_passes<64>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 96: e = noalloc_passes<96>(rho, spec, gpad, phi, tw, kxp, st); break;
            case 128: e = noalloc_passes<128>(rho, spec, gpad, phi, tw, kxp, st); break;
            default: e = cudaErrorInvalidValue; break;
        }
    }
    if (e != cudaSuccess) {
        set_context_free_error(std::string("cube2_solve_pm_noalloc: ") + cudaGetErrorString(e));
        return CUBE2_ERR_CUDA;
    }
    return CUBE2_OK;
}
