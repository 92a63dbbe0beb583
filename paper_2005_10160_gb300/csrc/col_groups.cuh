// Column stage (Eqs. 18-21) for FP32 column transforms of N = Py / 2 = 64,
// 128 or 256 points (33 <= ny <= 256): register transforms by groups of
// lanes (group_fft.cuh), eight layers at a time.
//
// A layer group is the J = N / 2 threads that own the mirror pairs of one ky
// parity.  With V = 16 values a lane the same J threads are exactly eight
// transforms of N / 16 lanes, so a round transforms eight layers and then
// accumulates eight layers, and only a barrier of the group (a warp sync for
// N = 64) stands between.
//
// Forward: one CTA per (kx, ky parity).  128- and 256-point columns run one
// layer group, J threads, through all rounds; a 64-point group is a single warp,
// so a CTA holds up to eight that take the rounds in turn, each with its own
// compensated sums, which the first group adds up.  Then the inverse transforms
// of all components run at once (one per transform slot, at most eight).  The
// next round's rows are read into registers before the accumulation, and the
// spectra one layer ahead.  The sum is plain over the eight layers of a round and
// compensated over the rounds; compensated every four layers it is no closer to
// 64 bits (1.8e-7 of the field at 256 x 256 x 32, 1.4e-7 for the requests below,
// either way) and takes 41.4 against 39.1 and 116 against 105 us for the whole
// calls.
//
// Adjoint: one CTA per kx and chunk of layers, both ky parities (N threads):
// the residual columns of all components are transformed at once, each
// thread keeps its pair's bins, with i for imaginary spectra and the mirror
// sign for odd components already applied, and combines eight layers per
// round; the two parities' inverse transforms are exchanged by halves
// through shared memory and added, so each layer's column is written once,
// Z[kx][n][y] (ColumnArgs::z_summed).
//
// Bound by latency, not by memory: under ncu (caches kept) at 256 x 256 x 32 with
// six components (52 MB of spectra) the forward takes 25 us at 42% of the issue
// slots, the block-FFT kernel it replaced 35; the adjoint 22 us at 40%, 75 before.
// 16 requests of 128 x 128 x 32: forward 74 us at 46%, 129 before.
#pragma once
#include "async_copy.cuh"
#include "grav_internal.h"
#include "group_fft.cuh"
#include "spectral.cuh"

namespace grav {

template <int N> struct ColGroup {
    using G = GroupFft<N>;
    static_assert(N >= 64 && N <= 256, "16 values a lane");
    static constexpr int J = N / 2;      // mirror pairs of one parity
    static constexpr int JP = J + 4;     // spectra row pitch: J + 1 rounded up to 4
    static constexpr int SLOTS = 8;      // transforms of J threads
    // slots of one 16-lane phase start L complex values apart modulo 16
    static constexpr int AREA = (G::TR + 15) / 16 * 16 + G::L % 16;
    static constexpr int MAXG = 256 / J;  // layer groups of a forward CTA
    // forward CTAs of six and more components keep their compensation terms in
    // shared memory, which leaves six without spills at 128 registers a thread;
    // seven still spill 8 to 88 bytes and eight 196 to 244
    static constexpr bool cmp_in_smem(int nc) { return nc >= 6; }
    static constexpr size_t fwd_smem(int groups, int nc) {
        return (size_t)(N + groups * (SLOTS * AREA + (cmp_in_smem(nc) ? 2 * nc * J : 0))) * sizeof(float2);
    }
    static constexpr size_t adj_smem = (size_t)(2 * N + 2 * SLOTS * AREA) * sizeof(float2);
};

template <int N, int NC>
__global__ void __launch_bounds__(256, 2)
    forward_column_group_kernel(ColumnArgs a, int groups, const float2* __restrict__ X, const float* __restrict__ spec,
                                float2* __restrict__ Y, const float2* __restrict__ tw, size_t x_bstride,
                                size_t y_bstride) {
    using C = float2;
    using S = ColGroup<N>;
    using G = GroupFft<N>;
    constexpr int J = S::J, V = G::V, L = G::L, SLOTS = S::SLOTS;
    static_assert(NC <= SLOTS, "one inverse transform per slot");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* t2 = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x, nt = groups * J;
    const int grp = tid / J, lt = tid % J, t = lt / L, q = lt % L;
    C* slots = t2 + N + grp * SLOTS * S::AREA;
    C* slot = slots + t * S::AREA;
    const int r = blockIdx.x & 1, kx = blockIdx.x >> 1;
    const int nz = a.nz, ny = a.ny;
    X += blockIdx.y * x_bstride + (size_t)kx * nz * a.ny_pad;  // request of a batched call
    Y += blockIdx.y * y_bstride;
    constexpr int S_ROW = NC * S::JP;  // floats per layer of spectra
    const float* Sk = request_spec(a, spec, blockIdx.y) + (size_t)(r * a.kx_count + kx) * nz * S_ROW;
    // spectra of the rounds first .. first + groups SLOTS into L2
    auto prefetch = [&](int first) {
        const int cnt = min(groups * SLOTS, nz - first);
        if (tid == 0 && cnt > 0) bulk_prefetch_l2(Sk + (size_t)first * S_ROW, (uint32_t)cnt * S_ROW * sizeof(float));
    };
    auto gsync = [&] {  // the groups of a CTA run the same number of rounds
        if constexpr (J == 32) __syncwarp();
        else __syncthreads();
    };
    C u[V];
    auto load = [&](int n) {  // layer n's rows of this lane (zero beyond nz and ny)
        const C* row = X + (size_t)n * a.ny_pad;
#pragma unroll
        for (int n2 = 0; n2 < V; ++n2) {
            const int m = q + L * n2;
            u[n2] = n < nz && m < ny ? __ldcg(row + m) : make_float2(0.f, 0.f);
        }
    };
    // this thread's spectra values of the next layer it accumulates
    const float* Sq = Sk + lt;
    float sv[NC];
    auto load_spec = [&](int n) {
#pragma unroll
        for (int c = 0; c < NC; ++c) sv[c] = n < nz ? __ldg(Sq + (size_t)n * S_ROW + c * S::JP) : 0.f;
    };
    chain_trigger();
    prefetch(0);
    load_spec(grp * SLOTS);
    prefetch(groups * SLOTS);
    build_group_tw<N>(t2, r, tw, a.tw_shift_p, tid, nt);
    chain_wait();  // X is in place
    load(grp * SLOTS + t);
    __syncthreads();

    int k1, k2;
    pair_pos<N>(lt, r, k1, k2);
    // pair 0 of the even parity holds ky = 0 and the Nyquist row, each with
    // its own stored value; only its warp takes the path that reads both
    const bool nyq = r == 0 && lt == 0, nyq_warp = r == 0 && lt < 32;
    constexpr bool CS = S::cmp_in_smem(NC);
    C acc[NC][2], cmpr[CS ? 1 : NC][2];
    C* cmps = t2 + N + groups * SLOTS * S::AREA + tid;  // [2 c + j][thread]
    auto cmp = [&](int c, int j) -> C& {
        if constexpr (CS) return cmps[(2 * c + j) * nt];
        else return cmpr[c][j];
    };
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[c][j] = cmp(c, j) = make_float2(0.f, 0.f);
    auto add_comp = [&](int c, int j, C v) {  // compensated acc += v
        const C y = csub(v, cmp(c, j));
        const C s = cadd(acc[c][j], y);
        cmp(c, j) = csub(csub(s, acc[c][j]), y);
        acc[c][j] = s;
    };

    for (int base = 0; base < nz; base += groups * SLOTS) {
        const int n0 = base + grp * SLOTS;
        const int cnt = min(SLOTS, nz - n0);  // may be negative for the last groups
        if (r) fold_regs<N>(u);
        group_fft<N, false>(u, slot, t2, q);
#pragma unroll
        for (int e = 0; e < V; ++e) slot[group_bin<N>(q, e)] = u[e];
        gsync();
        load(n0 + groups * SLOTS + t);  // in flight during the accumulation
        prefetch(base + 2 * groups * SLOTS);
        C part[NC][2];
#pragma unroll
        for (int c = 0; c < NC; ++c) part[c][0] = part[c][1] = make_float2(0.f, 0.f);
        const float* row = Sq + (size_t)n0 * S_ROW;
        // one layer; nl: the layer whose spectra are read meanwhile
        auto mac = [&](auto with_nyq, int l, int nl) {
            float s1[NC], s2[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                s1[c] = s2[c] = sv[c];
                if (decltype(with_nyq)::value && nyq) s2[c] = __ldg(row + l * S_ROW + c * S::JP + J);
            }
            load_spec(nl);
            const C v1 = slots[l * S::AREA + k1], v2 = slots[l * S::AREA + k2];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                part[c][0] = __ffma2_rn(make_float2(s1[c], s1[c]), v1, part[c][0]);
                part[c][1] = __ffma2_rn(make_float2(s2[c], s2[c]), v2, part[c][1]);
            }
        };
        const int next = n0 + groups * SLOTS;  // the next round's first layer
        if (cnt == SLOTS) {  // whole rounds without a branch per layer, so that loads move up
            if (nyq_warp) {
#pragma unroll
                for (int l = 0; l < SLOTS; ++l) mac(std::true_type{}, l, l + 1 < SLOTS ? n0 + l + 1 : next);
            } else {
#pragma unroll
                for (int l = 0; l < SLOTS; ++l) mac(std::false_type{}, l, l + 1 < SLOTS ? n0 + l + 1 : next);
            }
        } else {
#pragma unroll 1
            for (int l = 0; l < cnt; ++l) mac(std::true_type{}, l, n0 + l + 1);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int j = 0; j < 2; ++j) add_comp(c, j, part[c][j]);
        gsync();  // the slots are rewritten by the next round
    }

    if (groups > 1) {
        // the other groups hand their sums to the first through their slots
        C* red = slots;
        if (grp) {
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int j = 0; j < 2; ++j) red[(2 * c + j) * J + lt] = csub(acc[c][j], cmp(c, j));
        }
        __syncthreads();
        for (int g = 1; g < groups && grp == 0; ++g) {
            red += SLOTS * S::AREA;
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int j = 0; j < 2; ++j) add_comp(c, j, red[(2 * c + j) * J + lt]);
        }
    }
    // i (imaginary spectra) and the mirror sign (odd in y), constant over the layers
    if (grp == 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C b1 = csub(acc[c][0], cmp(c, 0)), b2 = csub(acc[c][1], cmp(c, 1));
            if (!nyq && ((a.oddv_mask >> c) & 1u)) b2 = make_float2(-b2.x, -b2.y);
            if ((a.imag_mask >> c) & 1u) {
                b1 = make_float2(-b1.y, b1.x);
                b2 = make_float2(-b2.y, b2.x);
            }
            slots[c * S::AREA + k1] = b1;
            slots[c * S::AREA + k2] = b2;
        }
    }
    gsync();
    if (grp) return;  // only warp syncs follow
    // inverse transform of component t; the parity-1 input is scaled by
    // W_P^q to cancel the extra factor of its conjugated twiddles
#pragma unroll
    for (int n2 = 0; n2 < V; ++n2) u[n2] = slot[q + L * n2];
    __syncwarp();
    const C wq = __ldg(tw + (q << a.tw_shift_p));
    if (r) {
#pragma unroll
        for (int n2 = 0; n2 < V; ++n2) u[n2] = cmul(u[n2], wq);
    }
    group_fft<N, true>(u, slot, t2, q);
    if (t < NC) {
        C* dst = Y + ((size_t)(r * a.kx_count + kx) * NC + t) * a.ny_pad;
        const C wc = cconj(wq);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const int y = group_bin<N>(q, e);
            if (y < ny) dst[y] = r ? unfold_reg<N>(u[e], wc, e) : u[e];
        }
    }
}

template <int N, int NC>
__global__ void __launch_bounds__(N, 512 / N)
    adjoint_column_group_kernel(ColumnArgs a, int chunk, const float2* __restrict__ Xr, const float* __restrict__ spec,
                                float2* __restrict__ Z, const float2* __restrict__ tw, size_t x_bstride,
                                size_t z_bstride) {
    using C = float2;
    using S = ColGroup<N>;
    using G = GroupFft<N>;
    constexpr int J = S::J, V = G::V, L = G::L, SLOTS = S::SLOTS;
    static_assert(NC <= SLOTS, "one residual transform per slot");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tab = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x;
    const int p = tid / J, lt = tid % J, t = lt / L, q = lt % L;
    const C* t2 = tab + p * N;
    C* slots = tab + 2 * N + p * SLOTS * S::AREA;  // this parity's
    C* slot = slots + t * S::AREA;
    const C* other = tab + 2 * N + ((1 - p) * SLOTS + t) * S::AREA;
    const int kx = blockIdx.x, nz = a.nz, ny = a.ny;
    const int first = blockIdx.y * chunk, last = min(nz, first + chunk);
    Xr += blockIdx.z * x_bstride + (size_t)kx * NC * a.ny_pad;  // request of a batched call
    Z += blockIdx.z * z_bstride + (size_t)kx * nz * a.ny_pad;
    constexpr int S_ROW = NC * S::JP;  // floats per layer of spectra
    const float* Sq = request_spec(a, spec, blockIdx.z) + (size_t)(p * a.kx_count + kx) * nz * S_ROW + lt;
    // spectra of the layers n .. n + 8 (below last) of both parities into L2
    auto prefetch = [&](int n) {
        const int cnt = min(SLOTS, last - n);
        if (lt == 0 && cnt > 0) bulk_prefetch_l2(Sq + (size_t)n * S_ROW, (uint32_t)cnt * S_ROW * sizeof(float));
    };
    prefetch(first);
    prefetch(first + SLOTS);

    C u[V];
    chain_trigger();
    build_group_tw<N>(tab, 0, tw, a.tw_shift_p, tid, N);
    build_group_tw<N>(tab + N, 1, tw, a.tw_shift_p, tid, N);
    chain_wait();  // Xr is in place
    {
        const C* col = Xr + (size_t)t * a.ny_pad;  // residual column of component t
#pragma unroll
        for (int n2 = 0; n2 < V; ++n2) {
            const int m = q + L * n2;
            u[n2] = t < NC && m < ny ? __ldcg(col + m) : make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    if (p) fold_regs<N>(u);
    group_fft<N, false>(u, slot, t2, q);
#pragma unroll
    for (int e = 0; e < V; ++e) slot[group_bin<N>(q, e)] = u[e];
    __syncthreads();
    int k1, k2;
    pair_pos<N>(lt, p, k1, k2);
    const bool nyq = p == 0 && lt == 0, nyq_warp = tid < 32;
    C rc[NC][2];
    {
        // parity 1: W_P^(k mod L) of the inverse transforms' input (see the forward)
        C w1 = make_float2(1.f, 0.f), w2 = w1;
        if (p) {
            w1 = __ldg(tw + ((k1 % L) << a.tw_shift_p));
            w2 = __ldg(tw + ((k2 % L) << a.tw_shift_p));
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C v1 = slots[c * S::AREA + k1], v2 = slots[c * S::AREA + k2];
            if (p) {
                v1 = cmul(v1, w1);
                v2 = cmul(v2, w2);
            }
            if ((a.imag_mask >> c) & 1u) {  // conj(i s) v = s (-i v)
                v1 = make_float2(v1.y, -v1.x);
                v2 = make_float2(v2.y, -v2.x);
            }
            if (!nyq && ((a.oddv_mask >> c) & 1u)) v2 = make_float2(-v2.x, -v2.y);
            rc[c][0] = v1;
            rc[c][1] = v2;
        }
    }
    const C wc = cconj(__ldg(tw + (q << a.tw_shift_p)));  // W_P^-q

    float sv[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) sv[c] = first < last ? __ldg(Sq + (size_t)first * S_ROW + c * S::JP) : 0.f;
    for (int n0 = first; n0 < last; n0 += SLOTS) {
        __syncthreads();  // every read of the slots is done
        const int cnt = min(SLOTS, last - n0);
        prefetch(n0 + 2 * SLOTS);
        const float* row = Sq + (size_t)n0 * S_ROW;
        auto combine = [&](auto with_nyq, int l) {
            float s1[NC], s2[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                s1[c] = s2[c] = sv[c];
                if (decltype(with_nyq)::value && nyq) s2[c] = __ldg(row + l * S_ROW + c * S::JP + J);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c)  // the next layer's values
                sv[c] = n0 + l + 1 < last ? __ldg(row + (l + 1) * S_ROW + c * S::JP) : 0.f;
            C z1 = make_float2(0.f, 0.f), z2 = z1;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                z1 = __ffma2_rn(make_float2(s1[c], s1[c]), rc[c][0], z1);
                z2 = __ffma2_rn(make_float2(s2[c], s2[c]), rc[c][1], z2);
            }
            slots[l * S::AREA + k1] = z1;
            slots[l * S::AREA + k2] = z2;
        };
        if (cnt == SLOTS) {  // whole rounds without a branch per layer, so that loads move up
            if (nyq_warp) {
#pragma unroll
                for (int l = 0; l < SLOTS; ++l) combine(std::true_type{}, l);
            } else {
#pragma unroll
                for (int l = 0; l < SLOTS; ++l) combine(std::false_type{}, l);
            }
        } else {
#pragma unroll 1
            for (int l = 0; l < cnt; ++l) combine(std::true_type{}, l);
        }
        __syncthreads();
#pragma unroll
        for (int n2 = 0; n2 < V; ++n2) u[n2] = slot[q + L * n2];
        __syncwarp();
        group_fft<N, true>(u, slot, t2, q);
        // parity 0 finishes the first half of the outputs, parity 1 the second
        if (p) {
#pragma unroll
            for (int e = 0; e < V; ++e) u[e] = unfold_reg<N>(u[e], wc, e);
#pragma unroll
            for (int e = 0; e < V / 2; ++e) slot[group_bin<N>(q, e)] = u[e];
        } else {
#pragma unroll
            for (int e = V / 2; e < V; ++e) slot[group_bin<N>(q, e)] = u[e];
        }
        __syncthreads();
        if (t < cnt) {
            C* dst = Z + (size_t)(n0 + t) * a.ny_pad;
#pragma unroll
            for (int e = 0; e < V / 2; ++e) {
                const int y0 = group_bin<N>(q, e), y1 = group_bin<N>(q, e + V / 2);
                const int y = p ? y1 : y0;
                if (y < ny) dst[y] = cadd(p ? u[e + V / 2] : u[e], other[y]);
            }
        }
    }
}

}  // namespace grav
