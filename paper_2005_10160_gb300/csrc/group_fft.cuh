// FP32 transforms of N = 64 .. 1024 points by groups of L lanes, V values a
// lane in registers (V = 16 up to N = 256, else 32; L = N / V), in the
// four-step form N = V x L:
//   x[q + L n2] (lane q) -> V-point DFT over n2 -> twiddle W_N^(q k2)
//   -> transpose through the group's shared area (q <-> k2)
//   -> V / L DFTs of L points over q: lane q then holds the bins k2 + V k1
//   for k2 = q + L i.
// A warp runs 32 / L transforms at once with warp-level syncs only.
//
// The library transforms rows and columns of at most N values zero-padded to
// P = 2N.  Their even and odd bins are two N-point transforms,
//   Z(2k + p) = sum_x (z[x] W_P^(p x)) W_N^(x k),   p = 0, 1,
// and the first N outputs of an inverse are
//   z[m] = IDFT_N(Z(2k))[m] + W_P^(-m) IDFT_N(Z(2k + 1))[m].
// With x = q + L n2 the fold factor W_P^x is W_2V^n2 (a constant of register
// n2) times W_P^q, which is constant over n2 and so rides in the transpose
// twiddles W_P^(q (2 k2 + p)).
#pragma once
#include "fft_block.cuh"
#include "warp_fft.cuh"

namespace grav {

template <int N> struct GroupFft {
    static_assert(N >= 64 && N <= 1024 && (N & (N - 1)) == 0, "64 .. 1024 points");
    static constexpr int V = N <= 256 ? 16 : 32;  // values a lane
    static constexpr int L = N / V;               // lanes of a transform
    static constexpr int GPW = 32 / L;            // transforms of a warp
    static constexpr int ROW = L + 1;             // row pitch of the transpose area
    static constexpr int TR = V * ROW;            // complex values of the transpose area
};

template <int M> __host__ __device__ constexpr int bitrev_m(int j) {
    int r = 0;
    for (int b = 1; b < M; b <<= 1) {
        r = (r << 1) | (j & 1);
        j >>= 1;
    }
    return r;
}

// M-point DFT in registers (M = 2 .. 32), radix-2 decimation in frequency:
// natural order in, u[j] = X[bitrev_m<M>(j)] out.
template <int M, bool INV> __device__ __forceinline__ void dft_regs(float2* u) {
#pragma unroll
    for (int h = M / 2; h >= 1; h >>= 1) {
#pragma unroll
        for (int b = 0; b < M; b += 2 * h) {
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float2 a = u[b + i], c = u[b + i + h];
                u[b + i] = cadd(a, c);
                u[b + i + h] = tw32<INV>(csub(a, c), i * (16 / h));
            }
        }
    }
}

// N-point transform of the group.  In: u[n2] = x[q + L n2].  Out: register
// i L + j holds bin group_bin<N>(q, i L + j).  tr: the group's transpose area
// (TR values, free for the caller afterwards); t2[k2 L + q]: the transpose
// twiddles of the forward sign, conjugated here for the inverse.  Every lane
// of the warp calls this.
template <int N, bool INV>
__device__ __forceinline__ void group_fft(float2 (&u)[GroupFft<N>::V], float2* tr, const float2* t2, int q) {
    using G = GroupFft<N>;
    dft_regs<G::V, INV>(u);
#pragma unroll
    for (int j = 0; j < G::V; ++j) {
        const int k2 = bitrev_m<G::V>(j);
        float2 w = t2[k2 * G::L + q];
        if (INV) w.y = -w.y;
        tr[k2 * G::ROW + q] = cmul(u[j], w);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < G::V / G::L; ++i) {
#pragma unroll
        for (int n1 = 0; n1 < G::L; ++n1) u[i * G::L + n1] = tr[(q + G::L * i) * G::ROW + n1];
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < G::V / G::L; ++i) dft_regs<G::L, INV>(u + i * G::L);
}

// Bin (or output index) in register e of lane q after group_fft.
template <int N> __device__ __forceinline__ constexpr int group_bin(int q, int e) {
    using G = GroupFft<N>;
    const int i = e / G::L, j = e - i * G::L;
    return q + G::L * i + G::V * bitrev_m<G::L>(j);
}

// Fold of the odd bins ahead of group_fft with odd-parity twiddles: register
// n2 times W_2V^n2.
template <int N> __device__ __forceinline__ void fold_regs(float2 (&u)[GroupFft<N>::V]) {
#pragma unroll
    for (int n2 = 0; n2 < GroupFft<N>::V; ++n2) u[n2] = tw64(u[n2], n2 * (32 / GroupFft<N>::V));
}

// a times W_P^(-m) for m = group_bin<N>(q, e): wq = W_P^(-q) (lane q), the
// rest, W_2V^(-i) W_2L^(-k1), is a constant of register e.
template <int N> __device__ __forceinline__ float2 unfold_reg(float2 a, float2 wq, int e) {
    using G = GroupFft<N>;
    const int i = e / G::L, j = e - i * G::L;
    return tw64(cmul(a, wq), -(i * (32 / G::V) + bitrev_m<G::L>(j) * (32 / G::L)));
}

// Fill t2[k2 L + q] = W_P^(q (2 k2 + p)) from W_T (T = P << shift_p).
template <int N> __device__ __forceinline__ void build_group_tw(float2* t2, int p, const float2* __restrict__ tw,
                                                                int shift_p, int tid, int nt) {
    using G = GroupFft<N>;
    for (int e = tid; e < N; e += nt) {
        const int k2 = e / G::L, q = e % G::L;
        t2[e] = tw[((q * (2 * k2 + p)) & (2 * N - 1)) << shift_p];
    }
}

}  // namespace grav
