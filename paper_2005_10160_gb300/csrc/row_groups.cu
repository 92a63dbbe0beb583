// FP32 row transforms (the row stages of Eq. 18) for P = 128 .. 2048 points
// with at most P / 2 nonzero inputs or wanted outputs, which every plan
// has: register transforms by groups of lanes (group_fft.cuh), one for the
// even and one for the odd bins of each packed row pair a + i b.
//
// A tile is 8 row pairs of one layer (4 for P = 2048, but for the forward rows); warps of even index
// run the even bins, warps of odd index the odd ones, so the fold of the odd
// bins is a warp-uniform branch.  Tiles are walked by a grid that fills the
// machine once, so the twiddle tables are built once per CTA, and the next
// tile's loads are issued, into the registers that a finished transform frees,
// before the tile is written.  Rows of any length and alignment are read with
// scalar loads, each element by the two warps that need it (the second read
// hits L1).
//
// The areas of the transforms start 1 complex value apart modulo 16 (2 for
// tiles of 4 pairs) and the pairs of a warp are chosen so that the 16 lanes of each
// shared-memory phase fall in different banks, in the transposes as well as
// in the passes across pairs.
//
// Against the block FFTs through shared memory that they replaced: 256-value
// rows of 32 layers 11.7 -> 8.9 us, 16 requests of 128-value rows 38.9 -> 24.5,
// 301-value rows of 45 layers 35.7 -> 18.2, their inverse 52.4 -> 30.9 (from
// one summed input instead of two).  1024-value rows of 100 layers: 310 us, 4.1
// TB/s (a kernel of one warp a transform, its rows staged by bulk copies, 313;
// tiles of 4 pairs 317; the inverse rows of six planes are the other way round,
// 48 us in tiles of 4 pairs, 51 of 8).  Issue slots are half busy; the rest waits
// on the shared-memory transposes and the two barriers a tile.
#include <climits>
#include <algorithm>

#include "async_copy.cuh"
#include "grav_internal.h"
#include "group_fft.cuh"

namespace grav {

namespace {

template <int N, int PAIRS_ = (N >= 1024 ? 4 : 8)> struct RowGroup {
    using G = GroupFft<N>;
    static constexpr int PAIRS = PAIRS_;                          // row pairs of a tile
    static constexpr int ROWS = 2 * PAIRS;
    static constexpr int WARPS = 2 * PAIRS / G::GPW;
    static constexpr int NT = 32 * WARPS;
    static constexpr int AREA = PAIRS == 4 ? G::TR + 2 : (G::TR + 15) / 16 * 16 + 1;
    static constexpr int KW = 32 / PAIRS;                         // kx values a warp covers
    static constexpr int KSTEP = NT / PAIRS;                      // kx values the CTA covers
    static constexpr size_t tab_off = (size_t)2 * PAIRS * AREA * sizeof(float2);
    static constexpr int MINB = (G::V > 16 ? 512 : 1024) / NT;  // 128 or 64 registers
    static_assert(AREA >= N, "natural-order results fit in the area");

    // pair of group g of the warps 2 h and 2 h + 1: the groups of one 16-lane
    // phase start L complex values apart modulo 16
    static __device__ __forceinline__ int pair_of(int h, int g) {
        if constexpr (G::GPW == 8) return (g & 3) * 2 + (g >> 2);
        else if constexpr (G::GPW == 4) return (g & 1) * 4 + (g >> 1) + 2 * h;
        else return g + G::GPW * h;
    }
    // first kx of a thread in the passes across pairs: a warp takes KW kx
    // values, those of even parity first, so that a phase sees one parity
    static __device__ __forceinline__ int first_kx(int tid) {
        const int i = (tid / PAIRS) % KW, base = tid / PAIRS - i;
        return base + (i < KW / 2 ? 2 * i : 2 * (i - KW / 2) + 1);
    }
};

// Real rows -> half spectra, written transposed (see launch_row_r2c), in tiles
// of 16 rows at every size: 128-byte runs.
template <int N> using ForwardRows = RowGroup<N, 8>;

template <int N>
__global__ void __launch_bounds__(ForwardRows<N>::NT, ForwardRows<N>::MINB)
    row_r2c_group_kernel(const float* __restrict__ in, size_t in_ostride, size_t in_istride, int l_in, int I, int O,
                         float2* __restrict__ out, int i_pad, const float2* __restrict__ tw, int shift_p,
                         size_t in_bstride, size_t out_bstride, unsigned ntiles, unsigned rbs) {
    using S = ForwardRows<N>;
    using G = GroupFft<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* areas = reinterpret_cast<float2*>(smem_raw);                // area of (pair s, parity p): 2 s + p
    float2* tab = reinterpret_cast<float2*>(smem_raw + S::tab_off);  // transpose twiddles, even then odd
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = warp & 1, g = lane / G::L, q = lane % G::L;
    const int s = S::pair_of(warp >> 1, g);
    chain_trigger();
    build_group_tw<N>(tab, 0, tw, shift_p, tid, S::NT);
    build_group_tw<N>(tab + N, 1, tw, shift_p, tid, S::NT);
    __syncthreads();
    float2* area = areas + (2 * s + p) * S::AREA;
    const float2* t2 = tab + p * N;

    float2 u[G::V];
    auto load = [&](unsigned t) {  // this lane's share of tile t's rows
        const unsigned rest = t / rbs;
        const int bz = (int)(rest / (unsigned)O), o = (int)(rest - (unsigned)bz * (unsigned)O);
        const int i0 = (int)(t - rest * rbs) * S::ROWS + 2 * s;
        const bool ha = t < ntiles && i0 < I, hb = ha && i0 + 1 < I;
        const float* ra = in + (ha ? bz * in_bstride + (size_t)o * in_ostride + (size_t)i0 * in_istride : 0);
        const float* rb = hb ? ra + in_istride : ra;
#pragma unroll
        for (int n2 = 0; n2 < G::V; ++n2) {
            const int x = q + G::L * n2;
            u[n2].x = ha && x < l_in ? load_here(ra + x) : 0.f;
            u[n2].y = hb && x < l_in ? load_here(rb + x) : 0.f;
        }
    };
    load(blockIdx.x);
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const unsigned rest = t / rbs;
        const int ib = (int)(t - rest * rbs) * S::ROWS;
        const int bz = (int)(rest / (unsigned)O), o = (int)(rest - (unsigned)bz * (unsigned)O);
        if (p) fold_regs<N>(u);
        group_fft<N, false>(u, area, t2, q);
#pragma unroll
        for (int e = 0; e < G::V; ++e) area[group_bin<N>(q, e)] = u[e];
        if (t + gridDim.x < ntiles) load(t + gridDim.x);  // in flight while this tile is written
        __syncthreads();
        // A(kx) = (Z(kx) + conj Z(P - kx)) / 2, B(kx) = (Z(kx) - conj Z(P - kx)) / (2i);
        // kx = 2k + r and P - kx have the same parity r
        {
            const int s2 = tid % S::PAIRS, kx0 = S::first_kx(tid), r = kx0 & 1;
            const int j0 = ib + 2 * s2;
            if (j0 < I) {
                const float2* zp = areas + (2 * s2 + r) * S::AREA;
                const bool pair = j0 + 1 < I;
                const size_t dstep = (size_t)S::KSTEP * O * i_pad;
                float2* dst = out + bz * out_bstride + ((size_t)kx0 * O + o) * i_pad + j0;
#pragma unroll 4
                for (int kx = kx0; kx <= N; kx += S::KSTEP, dst += dstep) {
                    const int k = kx >> 1;
                    const float2 zk = zp[k & (N - 1)];
                    const float2 zm = cconj(zp[r ? N - 1 - k : (N - k) & (N - 1)]);
                    const float2 A = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y + zm.y));
                    const float2 d = csub(zk, zm);
                    const float2 B = make_float2(0.5f * d.y, -0.5f * d.x);
                    if (pair) *reinterpret_cast<float4*>(dst) = make_float4(A.x, A.y, B.x, B.y);
                    else dst[0] = A;
                }
            }
        }
        __syncthreads();  // the areas are rewritten by the next tile
    }
}

// Half spectra (in0, or in0 + in1) -> real rows, the first l_out values kept
// (see launch_row_c2r): Z = A + i B is gathered into the even- and odd-bin
// areas, two N-point inverse transforms, their unfolded sum stored.  AHEAD
// (one input, N >= 512, where a CTA has several tiles): the next tile is read
// into the registers that the transform has just freed, so that it arrives
// while this tile is stored (512 x 512 x 64 adjoint: 89 -> 72 us).
template <int N, bool AHEAD>
__global__ void __launch_bounds__(RowGroup<N>::NT, RowGroup<N>::MINB)
    row_c2r_group_kernel(const float2* __restrict__ in0, const float2* __restrict__ in1, int I, int O, int i_pad,
                         float* __restrict__ out, size_t out_stride, int l_out, const float2* __restrict__ tw,
                         int shift_p, size_t in_bstride, size_t out_bstride, unsigned ntiles, unsigned rbs) {
    using S = RowGroup<N>;
    using G = GroupFft<N>;
    constexpr int CNT = N / S::KSTEP + 1;  // kx values of a thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* areas = reinterpret_cast<float2*>(smem_raw);
    float2* t2 = reinterpret_cast<float2*>(smem_raw + S::tab_off);  // even-parity transpose twiddles
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = warp & 1, g = lane / G::L, q = lane % G::L;
    const int s = S::pair_of(warp >> 1, g);
    build_group_tw<N>(t2, 0, tw, shift_p, tid, S::NT);
    float2* area = areas + (2 * s + p) * S::AREA;
    const float2 wq = cconj(__ldg(tw + (q << shift_p)));  // W_P^-q
    const int s2 = tid % S::PAIRS, kx0 = S::first_kx(tid), r = kx0 & 1;
    float2* zp = areas + (2 * s2 + r) * S::AREA;
    const size_t step = (size_t)S::KSTEP * O * i_pad;
    chain_wait();  // the half spectra are in place

    // where tile t's rows of this thread start
    auto place = [&](unsigned t, int& i0) {
        const unsigned rest = t / rbs;
        const int bz = (int)(rest / (unsigned)O), o = (int)(rest - (unsigned)bz * (unsigned)O);
        i0 = (int)(t - rest * rbs) * S::ROWS + 2 * s2;
        return bz * in_bstride + ((size_t)kx0 * O + o) * i_pad + (i0 < I ? i0 : 0);
    };
    // A, B at kx into bins kx and P - kx of Z = A + i B
    auto put = [&](int kx, int i0, float4 v) {
        if (i0 >= I) v.x = v.y = 0.f;
        if (i0 + 1 >= I) v.z = v.w = 0.f;
        if (kx == 0 || kx == N) v.y = v.w = 0.f;  // real DC and Nyquist
        const int k = kx >> 1;
        zp[k] = make_float2(v.x - v.w, v.y + v.z);
        if (kx > 0 && kx < N) zp[r ? N - 1 - k : N - k] = make_float2(v.x + v.w, v.z - v.y);
    };
    float4 next[AHEAD ? CNT : 1];
    auto fetch = [&](unsigned t) {
        // every register is set on every path, so that none lives through the transform
        const bool live = t < ntiles;
        int i0;
        const float2* src = in0 + place(live ? t : 0, i0);
#pragma unroll
        for (int i = 0; i < CNT; ++i)
            next[AHEAD ? i : 0] = live && kx0 + i * S::KSTEP <= N ? load_here4_cg(src + i * step)
                                                                : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    if (AHEAD) fetch(blockIdx.x);

    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const unsigned rest = t / rbs;
        const int ib = (int)(t - rest * rbs) * S::ROWS;
        const int bz = (int)(rest / (unsigned)O), o = (int)(rest - (unsigned)bz * (unsigned)O);
        int i0;
        size_t at = place(t, i0);
        if constexpr (AHEAD) {
#pragma unroll
            for (int i = 0; i < CNT; ++i)
                if (kx0 + i * S::KSTEP <= N) put(kx0 + i * S::KSTEP, i0, next[i]);
        } else {
#pragma unroll 4
            for (int kx = kx0; kx <= N; kx += S::KSTEP, at += step) {
                float4 v = __ldcg(reinterpret_cast<const float4*>(in0 + at));
                if (in1) {
                    const float4 w = __ldcg(reinterpret_cast<const float4*>(in1 + at));
                    v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
                }
                put(kx, i0, v);
            }
        }
        __syncthreads();
        {
            float2 u[G::V];
#pragma unroll
            for (int n2 = 0; n2 < G::V; ++n2) u[n2] = area[q + G::L * n2];
            __syncwarp();
            group_fft<N, true>(u, area, t2, q);
            if (p) {
#pragma unroll
                for (int e = 0; e < G::V; ++e) area[group_bin<N>(q, e)] = unfold_reg<N>(u[e], wq, e);
            } else {
#pragma unroll
                for (int e = 0; e < G::V; ++e) area[group_bin<N>(q, e)] = u[e];
            }
        }
        if (AHEAD) fetch(t + gridDim.x);
        __syncthreads();
        // a warp stores 32 values of both rows of one pair at a time
        const int chunks = (l_out + 31) >> 5;
        for (int w = warp; w < S::PAIRS * chunks; w += S::WARPS) {
            const int sp = w / chunks, x = (w - sp * chunks) * 32 + lane;
            const int j0 = ib + 2 * sp;
            if (j0 < I && x < l_out) {
                const float2 z = cadd(areas[2 * sp * S::AREA + x], areas[(2 * sp + 1) * S::AREA + x]);
                float* oa = out + bz * out_bstride + ((size_t)o * I + j0) * out_stride + x;
                oa[0] = z.x;
                if (j0 + 1 < I) oa[out_stride] = z.y;
            }
        }
        __syncthreads();  // the areas are rewritten by the next tile
    }
}

// The y passes of the equal-dimension plans.  384 x 320 x 64 adjoint: forward
// rows 599 -> 428 us (2.1 GB: 0.31 ms at the copy rate; 463 us without the
// next tile's loads in flight during the writes), inverse 95 -> 84 us, against
// block transforms.
//
// Complex rows, l_in <= N values zero-padded to 2N points: row k of `in` to
// row k of `out`, written as (Z(2k), Z(2k + 1)) pairs of 16 bytes.  A tile is
// PAIRS rows.
template <int N>
__global__ void __launch_bounds__(RowGroup<N>::NT, RowGroup<N>::MINB)
    rows_fwd_group_kernel(const float2* __restrict__ in, size_t in_stride, int l_in, float2* __restrict__ out,
                          size_t out_stride, long rows, const float2* __restrict__ tw, int shift_p, unsigned ntiles) {
    using S = RowGroup<N>;
    using G = GroupFft<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* areas = reinterpret_cast<float2*>(smem_raw);
    float2* tab = reinterpret_cast<float2*>(smem_raw + S::tab_off);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = warp & 1, g = lane / G::L, q = lane % G::L;
    const int s = S::pair_of(warp >> 1, g);
    build_group_tw<N>(tab, 0, tw, shift_p, tid, S::NT);
    build_group_tw<N>(tab + N, 1, tw, shift_p, tid, S::NT);
    __syncthreads();
    float2* area = areas + (2 * s + p) * S::AREA;
    float2 u[G::V];
    auto load = [&](unsigned t) {
        const long row = (long)t * S::PAIRS + s;
        const bool ok = row < rows;
        const float2* src = in + (size_t)(ok ? row : 0) * in_stride;
#pragma unroll
        for (int n2 = 0; n2 < G::V; ++n2) {
            const int x = q + G::L * n2;
            u[n2] = ok && x < l_in ? load_here(src + x) : make_float2(0.f, 0.f);
        }
    };
    load(blockIdx.x);
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const long row0 = (long)t * S::PAIRS;
        if (p) fold_regs<N>(u);
        group_fft<N, false>(u, area, tab + p * N, q);
#pragma unroll
        for (int e = 0; e < G::V; ++e) area[group_bin<N>(q, e)] = u[e];
        if (t + gridDim.x < ntiles) load(t + gridDim.x);  // in flight while this tile is written
        __syncthreads();
        for (int e = tid; e < S::PAIRS * N; e += S::NT) {
            const int sr = e / N, k = e % N;
            if (row0 + sr >= rows) break;
            const float2 a = areas[2 * sr * S::AREA + k], b = areas[(2 * sr + 1) * S::AREA + k];
            reinterpret_cast<float4*>(out + (size_t)(row0 + sr) * out_stride)[k] = make_float4(a.x, a.y, b.x, b.y);
        }
        __syncthreads();  // the areas are rewritten by the next tile
    }
}

// The inverse: rows of 2N bins, the first l_out <= N outputs kept.
template <int N>
__global__ void __launch_bounds__(RowGroup<N>::NT, RowGroup<N>::MINB)
    rows_inv_group_kernel(const float2* __restrict__ in, size_t in_stride, float2* __restrict__ out, size_t out_stride,
                          int l_out, long rows, const float2* __restrict__ tw, int shift_p, unsigned ntiles) {
    using S = RowGroup<N>;
    using G = GroupFft<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* areas = reinterpret_cast<float2*>(smem_raw);
    float2* t2 = reinterpret_cast<float2*>(smem_raw + S::tab_off);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = warp & 1, g = lane / G::L, q = lane % G::L;
    const int s = S::pair_of(warp >> 1, g);
    build_group_tw<N>(t2, 0, tw, shift_p, tid, S::NT);
    __syncthreads();
    float2* area = areas + (2 * s + p) * S::AREA;
    const float2 wq = cconj(__ldg(tw + (q << shift_p)));  // W_P^-q
    float2 u[G::V];
    auto load = [&](unsigned t) {
        const long row = (long)t * S::PAIRS + s;
        const bool ok = row < rows;
        const float2* src = in + (size_t)(ok ? row : 0) * in_stride + p;
#pragma unroll
        for (int n2 = 0; n2 < G::V; ++n2) u[n2] = ok ? load_here(src + 2 * (q + G::L * n2)) : make_float2(0.f, 0.f);
    };
    load(blockIdx.x);
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const long row0 = (long)t * S::PAIRS;
        group_fft<N, true>(u, area, t2, q);
        if (p) {
#pragma unroll
            for (int e = 0; e < G::V; ++e) area[group_bin<N>(q, e)] = unfold_reg<N>(u[e], wq, e);
        } else {
#pragma unroll
            for (int e = 0; e < G::V; ++e) area[group_bin<N>(q, e)] = u[e];
        }
        if (t + gridDim.x < ntiles) load(t + gridDim.x);  // in flight while this tile is written
        __syncthreads();
        const int chunks = (l_out + 31) >> 5;
        for (int w = warp; w < S::PAIRS * chunks; w += S::WARPS) {
            const int sr = w / chunks, x = (w - sr * chunks) * 32 + lane;
            if (row0 + sr < rows && x < l_out)
                out[(size_t)(row0 + sr) * out_stride + x] =
                    cadd(areas[2 * sr * S::AREA + x], areas[(2 * sr + 1) * S::AREA + x]);
        }
        __syncthreads();  // the areas are rewritten by the next tile
    }
}

int log2_of(int n) {
    int l = 0;
    while (n > 1) n >>= 1, ++l;
    return l;
}

// CTAs that fill the device, once per kernel and device.
template <auto Kernel>
int resident_ctas(int nt, size_t smem) {
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    int n = cache[dev & 63].load(std::memory_order_relaxed);
    if (n == 0) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, nt, smem) != cudaSuccess)
            return 0;
        n = sms * (per_sm > 0 ? per_sm : 1);
        cache[dev & 63].store(n, std::memory_order_relaxed);
    }
    return n;
}

template <int N>
cudaError_t r2c_launch(const float* in, size_t in_ostride, size_t in_istride, int l_in, int I, int O, void* out,
                       int i_pad, const void* tw, int log_t, cudaStream_t s, Batch b) {
    using S = ForwardRows<N>;
    constexpr auto k = row_r2c_group_kernel<N>;
    constexpr size_t smem = S::tab_off + 2 * N * sizeof(float2);
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    const unsigned rbs = (unsigned)((I + S::ROWS - 1) / S::ROWS);
    const long ntiles = (long)b.count * O * rbs;
    if (ntiles > INT_MAX) return cudaErrorInvalidValue;  // the kernel counts tiles in 32 bits
    const long fill = resident_ctas<k>(S::NT, smem);
    if (fill <= 0) return cudaErrorInvalidConfiguration;
    if (ntiles == 0) return cudaSuccess;
    const int shift_p = log_t - log2_of(2 * N);
    k<<<(unsigned)std::min(ntiles, fill), S::NT, smem, s>>>(in, in_ostride, in_istride, l_in, I, O, (float2*)out, i_pad,
                                                            (const float2*)tw, shift_p, b.in, b.out, (unsigned)ntiles,
                                                            rbs);
    return cudaGetLastError();
}

template <int N, bool AHEAD>
cudaError_t c2r_launch(const void* in0, const void* in1, int I, int O, int i_pad, float* out, size_t out_stride,
                       int l_out, const void* tw, int log_t, cudaStream_t s, Batch b) {
    using S = RowGroup<N>;
    constexpr auto k = row_c2r_group_kernel<N, AHEAD>;
    constexpr size_t smem = S::tab_off + N * sizeof(float2);
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    const unsigned rbs = (unsigned)((I + S::ROWS - 1) / S::ROWS);
    const long ntiles = (long)b.count * O * rbs;
    if (ntiles > INT_MAX) return cudaErrorInvalidValue;
    const long fill = resident_ctas<k>(S::NT, smem);
    if (fill <= 0) return cudaErrorInvalidConfiguration;
    if (ntiles == 0) return cudaSuccess;
    const int shift_p = log_t - log2_of(2 * N);
    return launch_chained(k, dim3((unsigned)std::min(ntiles, fill)), S::NT, smem, s, (const float2*)in0,
                          (const float2*)in1, I, O, i_pad, out, out_stride, l_out, (const float2*)tw, shift_p, b.in,
                          b.out, (unsigned)ntiles, rbs);
}

template <int N>
cudaError_t c2r_either(const void* in0, const void* in1, int I, int O, int i_pad, float* out, size_t out_stride,
                       int l_out, const void* tw, int log_t, cudaStream_t s, Batch b) {
    if constexpr (N >= 512) {
        if (!in1) return c2r_launch<N, true>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
    }
    return c2r_launch<N, false>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
}

template <int N>
cudaError_t rows_fwd_launch(const void* in, size_t in_stride, int l_in, void* out, size_t out_stride, long rows,
                            const void* tw, int log_t, cudaStream_t s) {
    using S = RowGroup<N>;
    constexpr auto k = rows_fwd_group_kernel<N>;
    constexpr size_t smem = S::tab_off + 2 * N * sizeof(float2);
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    const long ntiles = (rows + S::PAIRS - 1) / S::PAIRS;
    if (ntiles > INT_MAX) return cudaErrorInvalidValue;
    const long fill = resident_ctas<k>(S::NT, smem);
    if (fill <= 0) return cudaErrorInvalidConfiguration;
    if (ntiles == 0) return cudaSuccess;
    k<<<(unsigned)std::min(ntiles, fill), S::NT, smem, s>>>((const float2*)in, in_stride, l_in, (float2*)out, out_stride,
                                                            rows, (const float2*)tw, log_t - log2_of(2 * N),
                                                            (unsigned)ntiles);
    return cudaGetLastError();
}

template <int N>
cudaError_t rows_inv_launch(const void* in, size_t in_stride, void* out, size_t out_stride, int l_out, long rows,
                            const void* tw, int log_t, cudaStream_t s) {
    using S = RowGroup<N>;
    constexpr auto k = rows_inv_group_kernel<N>;
    constexpr size_t smem = S::tab_off + N * sizeof(float2);
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    const long ntiles = (rows + S::PAIRS - 1) / S::PAIRS;
    if (ntiles > INT_MAX) return cudaErrorInvalidValue;
    const long fill = resident_ctas<k>(S::NT, smem);
    if (fill <= 0) return cudaErrorInvalidConfiguration;
    if (ntiles == 0) return cudaSuccess;
    k<<<(unsigned)std::min(ntiles, fill), S::NT, smem, s>>>((const float2*)in, in_stride, (float2*)out, out_stride, l_out,
                                                            rows, (const float2*)tw, log_t - log2_of(2 * N),
                                                            (unsigned)ntiles);
    return cudaGetLastError();
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

cudaError_t launch_row_r2c_group(int log_p, const float* in, size_t in_ostride, size_t in_istride, int l_in, int I,
                                 int O, void* out, int i_pad, const void* tw, int log_t, cudaStream_t s, Batch b) {
    if (log_p < 7 || log_p > 11 || l_in > (1 << log_p) / 2 || i_pad % 2 || b.out % 2 || !aligned16(out))
        return cudaErrorInvalidValue;
    switch (log_p) {
        case 7: return r2c_launch<64>(in, in_ostride, in_istride, l_in, I, O, out, i_pad, tw, log_t, s, b);
        case 8: return r2c_launch<128>(in, in_ostride, in_istride, l_in, I, O, out, i_pad, tw, log_t, s, b);
        case 9: return r2c_launch<256>(in, in_ostride, in_istride, l_in, I, O, out, i_pad, tw, log_t, s, b);
        case 10: return r2c_launch<512>(in, in_ostride, in_istride, l_in, I, O, out, i_pad, tw, log_t, s, b);
        default: return r2c_launch<1024>(in, in_ostride, in_istride, l_in, I, O, out, i_pad, tw, log_t, s, b);
    }
}

cudaError_t launch_row_c2r_group(int log_p, const void* in0, const void* in1, int I, int O, int i_pad, float* out,
                                 size_t out_stride, int l_out, const void* tw, int log_t, cudaStream_t s, Batch b) {
    if (log_p < 7 || log_p > 11 || l_out > (1 << log_p) / 2 || i_pad % 2 || b.in % 2 || !aligned16(in0) ||
        !aligned16(in1))
        return cudaErrorInvalidValue;
    switch (log_p) {
        case 7: return c2r_either<64>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
        case 8: return c2r_either<128>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
        case 9: return c2r_either<256>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
        case 10: return c2r_either<512>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
        default: return c2r_either<1024>(in0, in1, I, O, i_pad, out, out_stride, l_out, tw, log_t, s, b);
    }
}

cudaError_t launch_rows_fwd_group(int log_p, const void* in, size_t in_stride, int l_in, void* out, size_t out_stride,
                                  long rows, const void* tw, int log_t, cudaStream_t s) {
    if (log_p < 7 || log_p > 11 || l_in > (1 << log_p) / 2 || out_stride % 2 || !aligned16(out))
        return cudaErrorInvalidValue;
    switch (log_p) {
        case 7: return rows_fwd_launch<64>(in, in_stride, l_in, out, out_stride, rows, tw, log_t, s);
        case 8: return rows_fwd_launch<128>(in, in_stride, l_in, out, out_stride, rows, tw, log_t, s);
        case 9: return rows_fwd_launch<256>(in, in_stride, l_in, out, out_stride, rows, tw, log_t, s);
        case 10: return rows_fwd_launch<512>(in, in_stride, l_in, out, out_stride, rows, tw, log_t, s);
        default: return rows_fwd_launch<1024>(in, in_stride, l_in, out, out_stride, rows, tw, log_t, s);
    }
}

cudaError_t launch_rows_inv_group(int log_p, const void* in, size_t in_stride, void* out, size_t out_stride, int l_out,
                                  long rows, const void* tw, int log_t, cudaStream_t s) {
    if (log_p < 7 || log_p > 11 || l_out > (1 << log_p) / 2) return cudaErrorInvalidValue;
    switch (log_p) {
        case 7: return rows_inv_launch<64>(in, in_stride, out, out_stride, l_out, rows, tw, log_t, s);
        case 8: return rows_inv_launch<128>(in, in_stride, out, out_stride, l_out, rows, tw, log_t, s);
        case 9: return rows_inv_launch<256>(in, in_stride, out, out_stride, l_out, rows, tw, log_t, s);
        case 10: return rows_inv_launch<512>(in, in_stride, out, out_stride, l_out, rows, tw, log_t, s);
        default: return rows_inv_launch<1024>(in, in_stride, out, out_stride, l_out, rows, tw, log_t, s);
    }
}

}  // namespace grav
