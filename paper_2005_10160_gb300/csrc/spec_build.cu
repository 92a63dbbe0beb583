// Kernel spectra of the plane plans: the two-dimensional FFT of every embedded
// kernel (the stored vector a of Eq. 19, transformed as in Eq. 18), reduced to
// the real numbers the column stage needs, from the quadrant of offsets that
// kernel_gen writes.
//
// The embedded kernel is exactly even or odd in x and in y, so each row's
// transform is purely real (even) or purely imaginary (odd), and so is each
// column's transform of those real numbers.  Two rows, then two layers'
// columns, therefore travel as one complex transform a + i b whose real and
// imaginary parts are the two results: nothing has to be separated.
//   spec_rows   E[o][v][u] (o = slot nzc + layer, u < nx, v < ny) -> T[kx][o][v],
//               R with X = R (even in x) or X = i R (odd), kx <= px / 2
//   spec_cols   per (kx, ky parity r) folds the columns of two layers,
//               a[m] = (x[m] + (-1)^r sign x[N - m]) W_py^(m r), N = py / 2,
//               N-point FFT, and stores the bins ky = 2q + r, q < J (and the
//               Nyquist bin for r = 0) times 1 / (px py): Re S (real spectra)
//               or Im S (imaginary ones).
//
// Plans with FP64 spectra run in FP64; plans that store FP32 in pairs of FP32
// (pair_float.cuh: 47 bits, rounded to 24 at the end), since FP64 runs at 1/64
// of the FP32 rate.  512 x 512 x 64, six components, FP64 transforms of
// embedded rows and of one column at a time: rows 9.1 ms, columns 17.1 ms.
#include "fft_block.cuh"
#include "grav_internal.h"
#include "pair_float.cuh"

namespace grav {

namespace {

template <typename C, int LOGP, int NSEQ, int NT>
__global__ void __launch_bounds__(NT) spec_rows_kernel(const decltype(C::x)* __restrict__ E, int nx, int ny, int nzc,
                                                       unsigned oddu_mask, decltype(C::x)* __restrict__ T, int ny2,
                                                       const C* __restrict__ tw, int tw_shift) {
    using R = decltype(C::x);
    constexpr int P = 1 << LOGP, SSTR = seq_stride<C>(P);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* tab = buf + NSEQ * SSTR;
    const int tid = threadIdx.x;
    const int o = blockIdx.y, O = gridDim.y, i_base = blockIdx.x * 2 * NSEQ;
    const bool odd = (oddu_mask >> (o / nzc)) & 1u;
    const R* rows = E + (size_t)o * ny * nx;
    build_tw_tab<C, LOGP, NT>(tab, tw, tw_shift, tid);
    __syncthreads();
    block_fft_tab_from<C, LOGP, NSEQ, NT, false>(buf, SSTR, tab, tid, [&](int s, int m) {
        // offset -u of the embedded row at u, its mirror at px - u
        const int i0 = i_base + 2 * s, x = m < nx ? m : P - m;
        C v = cmk<C>(0, 0);
        if (x < nx) {
            if (i0 < ny) v.x = rows[(size_t)i0 * nx + x];
            if (i0 + 1 < ny) v.y = rows[(size_t)(i0 + 1) * nx + x];
            if (odd && m >= nx) v = cmk<C>(-v.x, -v.y);
        }
        return v;
    });
    for (int e = tid; e < NSEQ * (P / 2 + 1); e += NT) {
        const int s = e % NSEQ, kx = e / NSEQ, i0 = i_base + 2 * s;
        if (i0 >= ny) continue;
        const C z = buf[s * SSTR + sidx<C>(kx)];
        // z = X0 + i X1 with X = R or X = i R; ny2 is even, so the pair fits
        C v = odd ? cmk<C>(z.y, -z.x) : z;
        *reinterpret_cast<C*>(T + ((size_t)kx * O + o) * ny2 + i0) = v;
    }
}

__device__ __forceinline__ float scaled(pairf v, pairf s, float*) { return (v * s).h; }
__device__ __forceinline__ double scaled(double v, double s, double*) { return v * s; }

template <typename C> struct SpecScale { decltype(C::x) s[kMaxPlanComp]; };

template <typename C, typename RO, int LOGN, int NT, int NSEQ>
__global__ void __launch_bounds__(NT) spec_cols_kernel(const decltype(C::x)* __restrict__ T, int ny, int ny2,
                                                       int kx_count, int nzc, int ncomp, int n0, int nz, int jp,
                                                       unsigned oddu_mask, unsigned oddv_mask, SpecScale<C> scale,
                                                       RO* __restrict__ spec, const C* __restrict__ tw, int tw_shift_n,
                                                       int tw_shift_p) {
    using R = decltype(C::x);
    constexpr int N = 1 << LOGN;
    constexpr int J = N / 2 > 0 ? N / 2 : 1;
    constexpr int SSTR = seq_stride<C>(N);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* tab = buf + NSEQ * SSTR;
    const int tid = threadIdx.x;
    const int kx = blockIdx.x, r = blockIdx.y, pair0 = blockIdx.z * NSEQ;
    const int O = ncomp * nzc, half = (nzc + 1) / 2, pairs = ncomp * half;  // pairs of layers of one slot
    build_tw_tab<C, LOGN, NT>(tab, tw, tw_shift_n, tid);
    __syncthreads();
    block_fft_tab_from<C, LOGN, NSEQ, NT, false>(buf, SSTR, tab, tid, [&](int sq, int m) {
        const int pr = pair0 + sq;
        C v = cmk<C>(0, 0);
        if (pr < pairs) {
            const int slot = pr / half, l = 2 * (pr - slot * half);
            const R* t0 = T + ((size_t)kx * O + slot * nzc + l) * ny2;
            const R* t1 = l + 1 < nzc ? t0 + ny2 : nullptr;
            const bool neg = ((oddv_mask >> slot) & 1u) != (unsigned)r;  // sign of x[N - m] in the fold
            C x1 = cmk<C>(0, 0);
            if (m < ny) v = cmk<C>(t0[m], t1 ? t1[m] : R(0.0));
            if (m > 0 && N - m < ny) x1 = cmk<C>(t0[N - m], t1 ? t1[N - m] : R(0.0));
            v = neg ? csub(v, x1) : cadd(v, x1);
            if (r) v = cmul(v, tw[m << tw_shift_p]);
        }
        return v;
    });
    const int nvals = (r == 0) ? J + 1 : J;
#pragma unroll
    for (int sq = 0; sq < NSEQ; ++sq) {
        const int pr = pair0 + sq;
        if (pr >= pairs) break;
        const int slot = pr / half, l = 2 * (pr - slot * half);
        const bool ov = (oddv_mask >> slot) & 1u, ou = (oddu_mask >> slot) & 1u;
        const size_t row = (size_t)ncomp * jp;  // one layer of spectra
        RO* dst = spec + ((size_t)(r * kx_count + kx) * nz + n0 + l) * row + (size_t)slot * jp;
        const R sc = scale.s[slot];
        for (int q = tid; q < jp; q += NT) {
            RO a = 0, b = 0;
            if (q < nvals) {
                const C z = buf[sq * SSTR + sidx<C>(q == J ? N / 2 : q)];
                // z = C0 + i C1 with C real (even in y) or i times real (odd in y);
                // odd in both axes: S = i i C, the stored number is -C
                C v = ov ? cmk<C>(z.y, -z.x) : z;
                if (ov && ou) v = cmk<C>(-v.x, -v.y);
                a = scaled(v.x, sc, (RO*)nullptr);
                b = scaled(v.y, sc, (RO*)nullptr);
            }
            dst[q] = a;
            if (l + 1 < nzc) dst[row + q] = b;
        }
    }
}

// Sequences per CTA of the row kernel: 4096 points (64 KB) at most.
constexpr int rows_nseq(int logp) { return logp >= 12 ? 1 : (4096 >> logp) > 8 ? 8 : 4096 >> logp; }

template <typename C, int LOGP>
cudaError_t rows_impl(const void* E, int nx, int ny, int nzc, int O, unsigned oddu_mask, void* T, int ny2, const void* tw,
                      int log_t, cudaStream_t s) {
    using R = decltype(C::x);
    constexpr int NSEQ = rows_nseq(LOGP), NT = 512;
    constexpr size_t smem = ((size_t)NSEQ * seq_stride<C>(1 << LOGP) + tw_tab_len(LOGP)) * sizeof(C);
    static_assert(smem <= (size_t)kMaxSmemOptin, "rows and twiddles fit");
    constexpr auto k = spec_rows_kernel<C, LOGP, NSEQ, NT>;
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    k<<<dim3((ny + 2 * NSEQ - 1) / (2 * NSEQ), O), NT, smem, s>>>((const R*)E, nx, ny, nzc, oddu_mask, (R*)T, ny2,
                                                                 (const C*)tw, log_t - LOGP);
    return cudaGetLastError();
}

template <typename C, typename RO, int LOGN>
cudaError_t cols_impl(const SpecBuild& b, const void* T, int nzc, int n0, const double* factor, void* spec,
                      const void* tw, int log_t, cudaStream_t s) {
    using R = decltype(C::x);
    constexpr int NT = 256, NSEQ = 4;
    constexpr size_t smem = ((size_t)NSEQ * seq_stride<C>(1 << LOGN) + tw_tab_len(LOGN)) * sizeof(C);
    constexpr auto k = spec_cols_kernel<C, RO, LOGN, NT, NSEQ>;
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    SpecScale<C> scale;
    for (int c = 0; c < b.ncomp; ++c) scale.s[c] = R(factor[c]);
    const int pairs = b.ncomp * ((nzc + 1) / 2);
    k<<<dim3(b.kx_count, 2, (pairs + NSEQ - 1) / NSEQ), NT, smem, s>>>(
        (const R*)T, b.ny, b.ny2, b.kx_count, nzc, b.ncomp, n0, b.nz, b.jp, b.oddu_mask, b.oddv_mask, scale, (RO*)spec,
        (const C*)tw, log_t - LOGN, log_t - (LOGN + 1));
    return cudaGetLastError();
}

}  // namespace

template <typename C>
cudaError_t launch_spec_rows(const SpecBuild& b, const void* E, int nzc, void* T, const void* tw, int log_t,
                             cudaStream_t s) {
    const int O = b.ncomp * nzc;
    switch (b.log_px) {
#define CASE(L) \
    case L: return rows_impl<C, L>(E, b.nx, b.ny, nzc, O, b.oddu_mask, T, b.ny2, tw, log_t, s);
        CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10) CASE(11) CASE(12)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
}

template <typename C, typename RO>
cudaError_t launch_spec_cols(const SpecBuild& b, const void* T, int nzc, int n0, const double* factor, RO* spec,
                             const void* tw, int log_t, cudaStream_t s) {
    switch (b.log_py - 1) {
#define CASE(L) \
    case L: return cols_impl<C, RO, L>(b, T, nzc, n0, factor, spec, tw, log_t, s);
        CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_spec_build_chunk(const SpecBuild& b, int fp64, const void* E, int nzc, int n0, void* T,
                                    const double* factor, void* spec, const void* tw, int log_t, cudaStream_t s) {
    cudaError_t e;
    if (fp64) {
        if ((e = launch_spec_rows<double2>(b, E, nzc, T, tw, log_t, s)) != cudaSuccess) return e;
        return launch_spec_cols<double2, double>(b, T, nzc, n0, factor, (double*)spec, tw, log_t, s);
    }
    if ((e = launch_spec_rows<pairf2>(b, E, nzc, T, tw, log_t, s)) != cudaSuccess) return e;
    return launch_spec_cols<pairf2, float>(b, T, nzc, n0, factor, (float*)spec, tw, log_t, s);
}

}  // namespace grav
