// The Winograd transforms' matrices: the Cook-Toom construction with points {0, +-1, +-2, +-1/2, inf} (the published F(m,3)
// minimal-filtering matrices).
#pragma once

namespace nnv {

// G: row j belongs to point j, the last row to infinity.
template <int M_> struct WinoG;
template <> struct WinoG<2> {
    static constexpr int A = 4;
    __host__ __device__ static constexpr float g(int r, int c) {
        constexpr float t[4][3] = {{1.f, 0.f, 0.f}, {.5f, .5f, .5f}, {.5f, -.5f, .5f}, {0.f, 0.f, 1.f}};
        return t[r][c];
    }
};
template <> struct WinoG<4> {
    static constexpr int A = 6;
    __host__ __device__ static constexpr float g(int r, int c) {
        constexpr float t[6][3] = {{1.f / 4.f, 0.f, 0.f},
                                   {-1.f / 6.f, -1.f / 6.f, -1.f / 6.f},
                                   {-1.f / 6.f, 1.f / 6.f, -1.f / 6.f},
                                   {1.f / 24.f, 1.f / 12.f, 1.f / 6.f},
                                   {1.f / 24.f, -1.f / 12.f, 1.f / 6.f},
                                   {0.f, 0.f, 1.f}};
        return t[r][c];
    }
};
template <> struct WinoG<6> {
    static constexpr int A = 8;
    __host__ __device__ static constexpr float g(int r, int c) {
        constexpr float t[8][3] = {{1.f, 0.f, 0.f},
                                   {-2.f / 9.f, -2.f / 9.f, -2.f / 9.f},
                                   {-2.f / 9.f, 2.f / 9.f, -2.f / 9.f},
                                   {1.f / 90.f, 1.f / 45.f, 2.f / 45.f},
                                   {1.f / 90.f, -1.f / 45.f, 2.f / 45.f},
                                   {32.f / 45.f, 16.f / 45.f, 8.f / 45.f},
                                   {32.f / 45.f, -16.f / 45.f, 8.f / 45.f},
                                   {0.f, 0.f, 1.f}};
        return t[r][c];
    }
};

// A row of G times three values; for F(4,3) and F(6,3) in one order everywhere, so that every kernel that transforms filters gets the same bits.  F(6,3)
// takes the outer taps last, the largest of them at the end: with the part that the points +-p share added first a pair would need a multiply-add less
// (384 -> 384 @12 in one launch 18.0 us a layer against 18.6), but the result is 5 % further from exact (64 -> 64 4.49e-8 / 4.26e-8).  F(4,3) is as exact
// either way, and in F(6,3)'s order the registers of its filter transform spill (all of a ResNet-18-shaped model 34.5 us against 33.5).
template <int M_> __device__ __forceinline__ float wino_filter(int r, float a, float b, float c) {
    using G = WinoG<M_>;
    if (M_ == 2) return a * G::g(r, 0) + b * G::g(r, 1) + c * G::g(r, 2);
    if (r == 0) return G::g(0, 0) * a;
    if (r == G::A - 1) return c;
    return fmaf(G::g(r, 2), c, M_ == 4 ? fmaf(G::g(r, 1), b, G::g(r, 0) * a) : fmaf(G::g(r, 0), a, G::g(r, 1) * b));
}

// B^T (alpha x alpha) and A^T (m x alpha) of the same construction as G: finite points {0, 1, -1, 2, -2, 1/2, -1/2} in that order, then infinity.
template <int M_> struct WinoBA;
template <> struct WinoBA<2> {
    static constexpr int A = 4;
    __host__ __device__ static constexpr float bt(int r, int c) {
        constexpr float t[4][4] = {{1, 0, -1, 0}, {0, 1, 1, 0}, {0, -1, 1, 0}, {0, -1, 0, 1}};
        return t[r][c];
    }
    __host__ __device__ static constexpr float at(int r, int c) {
        constexpr float t[2][4] = {{1, 1, 1, 0}, {0, 1, -1, 1}};
        return t[r][c];
    }
};
template <> struct WinoBA<4> {
    static constexpr int A = 6;
    __host__ __device__ static constexpr float bt(int r, int c) {
        constexpr float t[6][6] = {{4, 0, -5, 0, 1, 0},  {0, -4, -4, 1, 1, 0}, {0, 4, -4, -1, 1, 0},
                                   {0, -2, -1, 2, 1, 0}, {0, 2, -1, -2, 1, 0}, {0, 4, 0, -5, 0, 1}};
        return t[r][c];
    }
    __host__ __device__ static constexpr float at(int r, int c) {
        constexpr float t[4][6] = {{1, 1, 1, 1, 1, 0}, {0, 1, -1, 2, -2, 0}, {0, 1, 1, 4, 4, 0}, {0, 1, -1, 8, -8, 1}};
        return t[r][c];
    }
};
template <> struct WinoBA<6> {
    static constexpr int A = 8;
    __host__ __device__ static constexpr float bt(int r, int c) {
        constexpr float t[8][8] = {{1, 0, -5.25f, 0, 5.25f, 0, -1, 0},
                                   {0, 1, 1, -4.25f, -4.25f, 1, 1, 0},
                                   {0, -1, 1, 4.25f, -4.25f, -1, 1, 0},
                                   {0, .5f, .25f, -2.5f, -1.25f, 2, 1, 0},
                                   {0, -.5f, .25f, 2.5f, -1.25f, -2, 1, 0},
                                   {0, 2, 4, -2.5f, -5, .5f, 1, 0},
                                   {0, -2, 4, 2.5f, -5, -.5f, 1, 0},
                                   {0, -1, 0, 5.25f, 0, -5.25f, 0, 1}};
        return t[r][c];
    }
    __host__ __device__ static constexpr float at(int r, int c) {
        constexpr float t[6][8] = {{1, 1, 1, 1, 1, 1, 1, 0},
                                   {0, 1, -1, 2, -2, .5f, -.5f, 0},
                                   {0, 1, 1, 4, 4, .25f, .25f, 0},
                                   {0, 1, -1, 8, -8, .125f, -.125f, 0},
                                   {0, 1, 1, 16, 16, .0625f, .0625f, 0},
                                   {0, 1, -1, 32, -32, .03125f, -.03125f, 1}};
        return t[r][c];
    }
};


// B^T times A values (d B for a row), the pairs of points sharing their even and odd parts; one order for every kernel that transforms images.
__device__ __forceinline__ void wino_input(const float (&d)[6], float (&v)[6]) {
    const float p = fmaf(-4.f, d[2], d[4]), q = fmaf(-4.f, d[1], d[3]), s = d[4] - d[2], u = d[3] - d[1];
    v[0] = fmaf(4.f, d[0], fmaf(-5.f, d[2], d[4]));
    v[1] = p + q; v[2] = p - q;
    v[3] = fmaf(2.f, u, s); v[4] = fmaf(-2.f, u, s);
    v[5] = fmaf(4.f, d[1], fmaf(-5.f, d[3], d[5]));
}
__device__ __forceinline__ void wino_input(const float (&d)[8], float (&v)[8]) {
    const float p1 = fmaf(-4.25f, d[4], d[2] + d[6]), q1 = fmaf(-4.25f, d[3], d[1] + d[5]);
    const float p2 = fmaf(.25f, d[2], fmaf(-1.25f, d[4], d[6])), q2 = fmaf(.5f, d[1], fmaf(-2.5f, d[3], 2.f * d[5]));
    const float p3 = fmaf(4.f, d[2], fmaf(-5.f, d[4], d[6])), q3 = fmaf(2.f, d[1], fmaf(-2.5f, d[3], .5f * d[5]));
    v[0] = fmaf(5.25f, d[4] - d[2], d[0] - d[6]);
    v[1] = p1 + q1; v[2] = p1 - q1;
    v[3] = p2 + q2; v[4] = p2 - q2;
    v[5] = p3 + q3; v[6] = p3 - q3;
    v[7] = fmaf(5.25f, d[3] - d[5], d[7] - d[1]);
}
__device__ __forceinline__ void wino_input(const float (&d)[4], float (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = 0.f;
#pragma unroll
        for (int l = 0; l < 4; ++l)
            if (WinoBA<2>::bt(i, l) != 0.f) v[i] += WinoBA<2>::bt(i, l) * d[l];
    }
}

}  // namespace nnv
