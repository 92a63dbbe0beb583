// Forward column stage for 1024-point FP32 column transforms (Py = 2048)
// with one warp per layer transform.
//
// 16 warps at 128 registers a thread (the whole register file; six components
// spill 32 bytes of stores and 44 of loads, eight 84 and 144).  Warps 0-7
// accumulate: thread t owns the mirror pairs 2t and 2t + 1 for every component
// (the layer sum of Eq. 20 in the Fourier domain), as two-wide FP32
// operations over the two pairs.  Warps 8-15 transform: each layer's
// 1024-point FFT is done by a single warp in registers, 32 values a lane, as
// 1024 = 32 x 32 (the four-step form):
//   x[32 n1 + n2] -> 32-point DFTs over n1 (lane n2) -> twiddle W_1024^(n2 k1)
//   -> transpose through shared memory -> 32-point DFTs over n2 (lane k1).
// A warp transform needs no block or group barrier, so eight layers are in
// flight at once and the transform costs about a third of the instructions
// of a shared-memory radix-8 transform by a thread group.
//
// The layer sum is plain over blocks of 32 layers and compensated (Kahan)
// over the blocks; the compensated sums and their corrections are touched
// once per block and live in tensor memory (16 columns a component and
// warp), which leaves the registers to the block's sums and to spectra two
// layers ahead.  With one pair a thread and the sums in registers (24 warps
// at 80 registers) the accumulate loop had no register for that, and spent
// 37% of the kernel's instructions on integer work.
//
// 1024 x 1024 x 100, six components: 777 us (3.46 GB: 4.45 TB/s), 813 with the
// older split.  Bound by the latency of the accumulate loop: without its
// spectra loads the kernel takes 687 us, without the transforms 955 in a
// version whose loads the compiler had moved down to their use (1028, hence
// load_here).  Spectra brought into shared memory by bulk copies three layers
// ahead: 1222 us; four layers ahead in registers: 961.
//
// Data movement: FFT warp f handles layers f, f + 8, ...; X slot f is its
// own, so after reading layer n it refills the slot with layer n + 8 itself
// (bulk copy) and prefetches a later layer's spectra into L2.  The
// accumulate threads read their spectra values from global memory two layers
// ahead, in registers.  The spectra value of the Nyquist row (one per
// component, used by one thread of the even-ky CTA) rides in the spare tail
// of the layer's F slot.  Every wait is bounded.
//
// The odd-ky CTA transforms the folded column x[m] W_Py^m (Py = 2N).  With
// m = 32 n1 + n2 the fold factor is W_64^n1 W_2048^n2: the first factor is a
// constant of register n1, the second is constant over n1 and so moves past
// the first 32-point pass into the transpose twiddles, t2 = W_2048^((2 k1 +
// r) n2).  The inverse transform cancels the extra W_2048^-n2 that these
// twiddles carry by scaling its input by W_2048^n2 first, and unfolds its
// output y = n2 + 32 k by W_2048^-n2 W_64^-k.
#pragma once
#include "async_copy.cuh"
#include "fft_block.cuh"
#include "grav_internal.h"
#include "spectral.cuh"
#include "spectral_ws.cuh"
#include "tensor_memory.cuh"
#include "warp_fft.cuh"

namespace grav {

struct WfShape {
    static constexpr int N = 1024;
    static constexpr int J = 512;          // mirror pairs
    static constexpr int MT = J / 2;       // accumulate threads (8 warps), two pairs each
    static constexpr int FWARPS = 8;       // FFT warps
    static constexpr int NT = MT + 32 * FWARPS;
    static constexpr int FSLOT = kWarpFftSlot;  // complex values per F slot (transpose area)
    static constexpr int TCOLS = 256;      // tensor-memory columns: 2 warps per lane quarter x 8 components x 16
    static constexpr int DX = FWARPS;      // one X slot per FFT warp
    static constexpr int PF = 5;           // spectra prefetch distance (layers; with 8 the stage takes 812 us)
    static constexpr int JP = 516;         // spectra row pitch: J + 1 rounded up to 4
    static constexpr int BLOCK = 32;       // layers per compensated block
};

struct WfSmem {
    int df;
    uint32_t x_bytes, s_bytes, f_bytes;
    uint32_t f_off, t2_off, bar_off, flag_off, total;
};

template <int NC>
__global__ void __launch_bounds__(WfShape::NT, 1)
    forward_column_wf_kernel(ColumnArgs a, WfSmem L, const float2* __restrict__ X, const float* __restrict__ spec,
                             float2* __restrict__ Y, const float2* __restrict__ tw, int* __restrict__ err,
                             size_t x_bstride, size_t y_bstride) {
    using C = float2;
    constexpr int N = WfShape::N, J = WfShape::J, MT = WfShape::MT, FW = WfShape::FWARPS, NT = WfShape::NT;
    constexpr int FS = WfShape::FSLOT, DX = WfShape::DX, PF = WfShape::PF, JP = WfShape::JP;
    constexpr int S_ROW = NC * JP;  // floats per layer of spectra
    static_assert(NC <= FW, "one inverse transform per FFT warp");
    static_assert(NC <= FS - N, "Nyquist spectra values fit in the F slot tail");
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* xring = smem;
    C* fring = reinterpret_cast<C*>(smem + L.f_off);
    C* t2 = reinterpret_cast<C*>(smem + L.t2_off);  // W_2048^((2 k1 + r) n2) at [k1][n2]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bar_off);
    uint64_t* xfull = bars;
    uint64_t* ffull = xfull + DX;
    uint64_t* fempty = ffull + L.df;
    volatile int* abort = reinterpret_cast<volatile int*>(smem + L.flag_off);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L.flag_off) + 1;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r = blockIdx.x & 1, kx = blockIdx.x >> 1;
    const int nz = a.nz, ny = a.ny;
    X += blockIdx.y * x_bstride;  // request of a batched call
    Y += blockIdx.y * y_bstride;
    const C* Xk = X + (size_t)kx * nz * a.ny_pad;
    const float* Sk = request_spec(a, spec, blockIdx.y) + (size_t)(r * a.kx_count + kx) * nz * S_ROW;

    if (tid == 0) {
        for (int s = 0; s < DX; ++s) mbar_init(&xfull[s], 1);
        for (int s = 0; s < L.df; ++s) {
            mbar_init(&ffull[s], 32);
            mbar_init(&fempty[s], MT);
        }
        *abort = 0;
        fence_mbar_init();
        // first layer of every X slot, and the first PF layers' spectra into L2,
        // while the tables are built
        for (int n = 0; n < DX && n < nz; ++n) {
            mbar_arrive_expect_tx(&xfull[n], L.x_bytes);
            bulk_g2s(xring + (size_t)n * L.x_bytes, Xk + (size_t)n * a.ny_pad, L.x_bytes, &xfull[n]);
        }
        for (int n = 0; n < PF && n < nz; ++n) bulk_prefetch_l2(Sk + (size_t)n * S_ROW, L.s_bytes);
    }
    for (int e = tid; e < N; e += NT) {
        const int k1 = e >> 5, n2 = e & 31;
        t2[e] = tw[(((2 * k1 + r) * n2) & (2 * N - 1)) << a.tw_shift_p];
    }
    if (warp == 1) tmem_alloc<WfShape::TCOLS>(tmem_slot);  // the register file admits one such CTA per SM
    __syncthreads();

    bool failed = false;
    const bool is_mac = tid < MT;

    if (!is_mac) {
        // ---------------- FFT warp f: layers f, f + FW, ... ----------------
        const int f = warp - (MT >> 5);
        unsigned char* xslot = xring + (size_t)f * L.x_bytes;
        const C* xs = reinterpret_cast<const C*>(xslot);
        int pending = f < nz ? f : -1;  // layer of the copy in flight into X slot f
        // Nyquist-row spectra value of component `lane` (even-ky CTA), loaded
        // one iteration ahead so that its latency is never waited on
        const bool has_nyq = r == 0 && lane < NC;
        float snyq_next = (has_nyq && f < nz) ? __ldg(Sk + (size_t)f * S_ROW + lane * JP + J) : 0.f;
        for (int n = f; n < nz; n += FW) {
            const int sf = n % L.df;
            int ok = 1;
            if (lane == 0) {
                ok = ws_wait(&xfull[f], (uint32_t)((n / DX) & 1), abort);
                if (ok) pending = -1;
                if (ok && n >= L.df) ok = ws_wait(&fempty[sf], (uint32_t)((n / L.df - 1) & 1), abort);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                failed = true;
                break;
            }
            const float snyq = snyq_next;
            if (has_nyq && n + FW < nz) snyq_next = __ldg(Sk + (size_t)(n + FW) * S_ROW + lane * JP + J);
            float2 u[32];
#pragma unroll
            for (int n1 = 0; n1 < 32; ++n1) {
                const int m = 32 * n1 + lane;
                C v = make_float2(0.f, 0.f);
                if (m < ny) v = xs[m];
                u[n1] = v;
            }
            __syncwarp();  // every lane's reads of X slot f are done
            if (lane == 0) {
                if (n + FW < nz) {
                    fence_proxy_async_smem();
                    mbar_arrive_expect_tx(&xfull[f], L.x_bytes);
                    bulk_g2s(xslot, Xk + (size_t)(n + FW) * a.ny_pad, L.x_bytes, &xfull[f]);
                    pending = n + FW;
                }
                if (n + PF < nz) bulk_prefetch_l2(Sk + (size_t)(n + PF) * S_ROW, L.s_bytes);
            }
            if (r) {
#pragma unroll
                for (int n1 = 0; n1 < 32; ++n1) u[n1] = tw64(u[n1], n1);  // fold factor W_64^n1
            }
            C* fb = fring + sf * FS;
            warp_fft1024<false>(u, fb, t2, lane);
#pragma unroll
            for (int j = 0; j < 32; ++j) fb[lane + 32 * bitrev5(j)] = u[j];
            if (lane < NC) fb[N + lane] = make_float2(snyq, 0.f);
            mbar_arrive(&ffull[sf]);  // this lane's writes of the F slot are done
        }
        if (lane == 0 && pending >= 0) {
            // a copy that will not be consumed (failure path): let it land
            // (bounded) before the CTA's shared memory is released
            mbar_wait_bounded(&xfull[f], (uint32_t)((pending / DX) & 1), kWaitLimitNs);
        }
        if (cta_sync_or(failed || *abort)) return;
        cta_sync();  // the accumulate threads have written the sums
        // inverse column transform of component f (F slot f)
        const int c = f;
        if (c < NC) {
            C* fb = fring + c * FS;
            float2 u[32];
#pragma unroll
            for (int n1 = 0; n1 < 32; ++n1) u[n1] = fb[32 * n1 + lane];
            __syncwarp();
            if (r) {
                const C w = __ldg(tw + (lane << a.tw_shift_p));  // W_2048^n2, n2 = lane
#pragma unroll
                for (int n1 = 0; n1 < 32; ++n1) u[n1] = cmul(u[n1], w);
            }
            warp_fft1024<true>(u, fb, t2, lane);
            C* dst = Y + ((size_t)(r * a.kx_count + kx) * a.ncomp + c) * a.ny_pad;
            if (r) {
                // unfold: W_2048^-y with y = lane + 32 k is W_2048^-lane W_64^-k
                const C w = cconj(__ldg(tw + (lane << a.tw_shift_p)));
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int y = lane + 32 * bitrev5(j);
                    if (y < ny) dst[y] = tw64(cmul(u[j], w), 64 - bitrev5(j));
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int y = lane + 32 * bitrev5(j);
                    if (y < ny) dst[y] = u[j];
                }
            }
        }
    } else {
        // ---------------- accumulate: thread t owns mirror pairs 2t, 2t + 1 ----------------
        const int q = 2 * tid;
        const uint32_t tm = tmem_addr(*tmem_slot, warp, (warp >> 2) * 128);
        // bins of the two pairs: k1 = q, q + 1; k2 = N - q, N - q - 1 (even ky;
        // pair 0: the Nyquist bin N / 2) or N - 1 - q, N - 2 - q (odd ky)
        const int k2a = r ? N - 1 - q : q ? N - q : N / 2, k2b = r ? N - 2 - q : N - 1 - q;
        // sums of the block, two-wide over the pairs: re and im of bin 1, of bin 2
        float2 part[NC][4];
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int j = 0; j < 4; ++j) part[c][j] = make_float2(0.f, 0.f);
        // this thread's spectra values Sk[n][c][q], [q + 1], two layers ahead
        const float* Sq = Sk + q;
        float2 sv[2][NC];
        auto load_spec = [&](int n, float2 (&s)[NC]) {
            if (n >= nz) return;
            const float* row = Sq + (size_t)n * S_ROW;
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c] = load_here2(row + c * JP);
        };
        load_spec(0, sv[0]);
        load_spec(1, sv[1]);
        int sf = 0, wrap = 0;  // F slot of layer n (n % df) and n / df, stepped with n
        auto layer = [&](int n, float2 (&s)[NC]) {
            // the warp leaves its loop together (the tensor-memory accesses need whole warps)
            if (!__all_sync(0xffffffffu, ws_wait(&ffull[sf], (uint32_t)(wrap & 1), abort))) return false;
            const C* fb = fring + sf * FS;
            const float4 a = *reinterpret_cast<const float4*>(fb + q);
            const C b0 = fb[k2a], b1 = fb[k2b];
            const float2 x1 = make_float2(a.x, a.z), y1 = make_float2(a.y, a.w);
            const float2 x2 = make_float2(b0.x, b1.x), y2 = make_float2(b0.y, b1.y);
            if (r == 0 && warp == 0) {
                // lane 0 holds the Nyquist bin, which has spectra values of its own
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float2 s2 = make_float2(lane ? s[c].x : fb[N + c].x, s[c].y);
                    part[c][0] = __ffma2_rn(s[c], x1, part[c][0]);
                    part[c][1] = __ffma2_rn(s[c], y1, part[c][1]);
                    part[c][2] = __ffma2_rn(s2, x2, part[c][2]);
                    part[c][3] = __ffma2_rn(s2, y2, part[c][3]);
                }
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    part[c][0] = __ffma2_rn(s[c], x1, part[c][0]);
                    part[c][1] = __ffma2_rn(s[c], y1, part[c][1]);
                    part[c][2] = __ffma2_rn(s[c], x2, part[c][2]);
                    part[c][3] = __ffma2_rn(s[c], y2, part[c][3]);
                }
            }
            mbar_arrive(&fempty[sf]);
            if (++sf == L.df) {
                sf = 0;
                ++wrap;
            }
            load_spec(n + 2, s);
            return true;
        };
        // part into the compensated sums (tensor memory: 8 sums, 8 corrections a
        // component); keep: leave the corrected sums in part instead
        auto flush = [&](bool first, bool keep) {
            __syncwarp();
            if (!first) tmem_wait_st();
#pragma unroll
            for (int c = 0; c < NC; ++c) {
#pragma unroll
                for (int h = 0; h < 4; h += 2) {  // bin 1, bin 2
                    float v[8];
                    if (first) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = 0.f;
                    } else {
                        tmem_ld8(tm + 16 * c + 4 * h, v);
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        float2& p = part[c][h + j];
                        kahan_add(v[2 * j], v[4 + 2 * j], p.x);
                        kahan_add(v[2 * j + 1], v[5 + 2 * j], p.y);
                        p = keep ? make_float2(v[2 * j] - v[4 + 2 * j], v[2 * j + 1] - v[5 + 2 * j])
                                 : make_float2(0.f, 0.f);
                    }
                    if (!keep) tmem_st8(tm + 16 * c + 4 * h, v);
                }
            }
        };
        for (int n = 0; n < nz; n += 2) {
            if (!layer(n, sv[0]) || (n + 1 < nz && !layer(n + 1, sv[1]))) {
                failed = true;
                break;
            }
            const int done = n + 2;  // blocks end after an even number of layers
            if (done >= nz || done % WfShape::BLOCK == 0) flush(done <= WfShape::BLOCK, done >= nz);
        }
        __syncwarp();
        tmem_wait_st();  // (a failed loop may have left one in flight)
        if (cta_sync_or(failed || *abort)) {
            if (tid == 0) atomicExch(err, 1);
            __syncwarp();
            if (warp == 1) tmem_free<WfShape::TCOLS>(*tmem_slot);
            return;
        }
        // the compensated sums (times i for imaginary spectra, with the
        // mirror sign for odd components) into F slot c, natural order
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C* fb = fring + c * FS;
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // pair q + h
                C b1 = h ? make_float2(part[c][0].y, part[c][1].y) : make_float2(part[c][0].x, part[c][1].x);
                C b2 = h ? make_float2(part[c][2].y, part[c][3].y) : make_float2(part[c][2].x, part[c][3].x);
                const bool nyq = r == 0 && tid == 0 && h == 0;
                if (!nyq && ((a.oddv_mask >> c) & 1u)) b2 = make_float2(-b2.x, -b2.y);
                if ((a.imag_mask >> c) & 1u) {
                    b1 = make_float2(-b1.y, b1.x);
                    b2 = make_float2(-b2.y, b2.x);
                }
                fb[q + h] = b1;
                fb[h ? k2b : k2a] = b2;
            }
        }
        cta_sync();  // also: every warp has read its tensor memory
        if (warp == 1) tmem_free<WfShape::TCOLS>(*tmem_slot);
    }
}

// Shared-memory layout; df == 0 when it does not fit.  The F ring holds
// one slot per FFT warp plus the accumulate threads' lag.
inline WfSmem wf_smem(int ny_pad, int ncomp, int jp, int nc_inst, int max_bytes) {
    WfSmem L{};
    L.x_bytes = (uint32_t)(ny_pad * sizeof(float2));
    L.s_bytes = (uint32_t)(ncomp * jp * sizeof(float));
    L.f_bytes = (uint32_t)(WfShape::FSLOT * sizeof(float2));
    if (ny_pad > WfShape::N || nc_inst > WfShape::FWARPS || ncomp != nc_inst || jp != WfShape::JP ||
        (L.x_bytes & 15u) || (L.s_bytes & 15u))
        return WfSmem{};
    for (int df = 18; df >= WfShape::FWARPS + 1; --df) {
        WfSmem l = L;
        l.df = df;
        l.f_off = (uint32_t)(WfShape::DX * L.x_bytes + 127) & ~127u;
        l.t2_off = l.f_off + df * L.f_bytes;
        l.bar_off = l.t2_off + WfShape::N * sizeof(float2);
        l.flag_off = l.bar_off + (WfShape::DX + 2 * df) * 8;
        l.total = l.flag_off + 16;
        if ((int)l.total <= max_bytes) return l;
    }
    return WfSmem{};
}

}  // namespace grav
