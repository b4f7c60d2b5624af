// Stages and twiddle rows of the line transforms (fft.cu): the arithmetic that sizes
// and indexes the tables, without device code, so that it also compiles for the host.
#pragma once

namespace cube2 {

// Radix of stage s of an n-point line (0 past the last): as few stages as radices
// up to 16 allow with the values per thread below (fewer exchanges, fewer
// rounded twiddles), a 3 last, which leaves the last stage an even number of
// butterflies.  The x passes (xp) hold two butterflies of the last radix at once
// and take 128 as 16 8.  (256 as 16 16 is no faster and its low modes come out
// less exact: relative error of the potential 9.4e-7 against 5.8e-7.)
__host__ __device__ constexpr int radix_at(int n, int s, bool xp) {
    constexpr int P[17][6] = {{8, 4, 2}, {12, 4, 3}, {16, 4, 4}, {24, 8, 3}, {32, 8, 4}, {48, 4, 4, 3}, {64, 8, 8},
                              {96, 8, 4, 3}, {128, 8, 16}, {192, 8, 8, 3}, {256, 8, 8, 4}, {384, 8, 4, 4, 3}, {512, 8, 8, 8},
                              {768, 8, 8, 4, 3}, {1024, 16, 8, 8}, {1536, 8, 8, 8, 3}, {2048, 16, 16, 8}};
    if (xp && n == 128) return s == 0 ? 16 : s == 1 ? 8 : 0;
    for (int i = 0; i < 17; ++i)
        if (P[i][0] == n) return s < 5 ? P[i][s + 1] : 0;
    return 0;
}
__host__ __device__ constexpr int stages_of(int n, bool xp) {
    int s = 0;
    while (radix_at(n, s, xp) != 0) ++s;
    return s;
}
// Twiddle rows: for the tile passes and the x passes, forward and inverse (which
// runs the radices in reverse), stage by stage from the second on, entry
// (r - 1) n/R + j of a stage is exp(-+ 2 pi i r (j mod Ns) / (Ns R)).
__host__ __device__ constexpr int twiddle_row(int n, bool xp, bool inv, int stage) {
    int v = 0;
    for (int k = 0; k < 4; ++k) {
        const bool kx = k >= 2, ki = k % 2 == 1;
        const int S = stages_of(n, kx);
        for (int i = 1; i < S; ++i) {
            if (kx == xp && ki == inv && i == stage) return v;
            const int R = radix_at(n, ki ? S - 1 - i : i, kx);
            v += (R - 1) * (n / R);
        }
        if (kx == xp && ki == inv) return v;   // stage past the last: the end of these rows
    }
    return v;
}
__host__ __device__ constexpr int twiddle_entries(int n) { return twiddle_row(n, true, true, 99); }

// Meshes that the allocation-free solve takes, and the twiddles its fixed array holds:
// the most that any of them needs (96 points, with a stage more, take 584, 128 points 464).
constexpr int NOALLOC_MAX_N = 128;
constexpr int most_twiddles(int max_n) {
    int most = 0;
    for (int n = 1; n <= max_n; ++n)
        if (stages_of(n, false) > 0 && twiddle_entries(n) > most) most = twiddle_entries(n);
    return most;
}
constexpr int NOALLOC_TWIDDLES = most_twiddles(NOALLOC_MAX_N);

}  // namespace cube2
