// Adjoint column stage for 1024-point FP32 column transforms (Py = 2048),
// the transpose of Eq. 21: for every layer n,
//   Z_n = IFFT_y( sum_c conj(S_c,n) . FFT_y(R_c) )
// on one kx column and one ky parity (the same parity split as the forward).
//
// 16 warps at 128 registers a thread.  Warps 8-15 first transform the
// residual's row-transform columns (component f in warp f), one warp each,
// in registers (warp_fft1024); thread t of warps 0-7 keeps both bins of the
// mirror pairs 2t and 2t + 1 of every component in registers, with -i for
// imaginary spectra and the mirror sign for odd components applied.  Then,
// layer by layer, the combine threads form the layer's spectrum from their
// bins and the layer's spectra values, as two-wide FP32 operations over the
// two pairs (spectra read from global memory two layers ahead, after a bulk L2
// prefetch eight layers ahead: the combine threads run ahead of the
// transforms, so a load from DRAM would stall every layer) and write it
// into a ring slot; FFT warp f inverse-transforms layers f, f + 8, ... from
// the slot (which is also its transpose area) and writes the rows y < ny.
// The combine threads run up to (ring depth - 8) layers ahead of the
// transforms.  The FFT warps form the Nyquist bin themselves.  Every wait is
// bounded.
//
// 1024 x 1024 x 100, six components: 760 us (4.2 GB: 5.5 TB/s); 993 with one
// pair a thread (24 warps at 80 registers, spectra one layer ahead), 949 with
// two pairs while the compiler moved the spectra loads down to their use and
// the residual columns were read after the tables.
#pragma once
#include "async_copy.cuh"
#include "grav_internal.h"
#include "spectral.cuh"
#include "spectral_ws.cuh"
#include "warp_fft.cuh"

namespace grav {

struct AwShape {
    static constexpr int N = 1024;
    static constexpr int J = 512;     // mirror pairs
    static constexpr int MT = J / 2;  // combine threads (8 warps), two pairs each
    static constexpr int FWARPS = 8;  // FFT warps
    static constexpr int NT = MT + 32 * FWARPS;
    static constexpr int SLOT = kWarpFftSlot;
    static constexpr int JP = 516;    // spectra row pitch: J + 1 rounded up to 4
    static constexpr int PF = 8;      // spectra prefetch distance into L2 (layers)
};

struct AwSmem {
    int dz;
    uint32_t slot_off, tw_off, t2_off, stage_off, bar_off, flag_off, total;
};

template <int NC>
__global__ void __launch_bounds__(AwShape::NT, 1)
    adjoint_column_wf_kernel(ColumnArgs a, AwSmem L, const float2* __restrict__ Xr, const float* __restrict__ spec,
                             float2* __restrict__ Z, const float2* __restrict__ tw, int* __restrict__ err,
                             size_t x_bstride, size_t z_bstride, const __grid_constant__ CUtensorMap zmap) {
    using C = float2;
    constexpr int N = AwShape::N, J = AwShape::J, MT = AwShape::MT, FW = AwShape::FWARPS, NT = AwShape::NT;
    constexpr int FS = AwShape::SLOT, JP = AwShape::JP, S_ROW = NC * JP;
    static_assert(NC <= FW, "one residual transform per FFT warp");
    extern __shared__ __align__(128) unsigned char smem[];
    C* ring = reinterpret_cast<C*>(smem + L.slot_off);
    C* tws = reinterpret_cast<C*>(smem + L.tw_off);  // fold twiddles W_Py^m, m < N
    C* t2 = reinterpret_cast<C*>(smem + L.t2_off);   // W_1024^(n2 k1) at [k1][n2]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bar_off);
    uint64_t* zfull = bars;
    uint64_t* zempty = zfull + L.dz;
    volatile int* abort = reinterpret_cast<volatile int*>(smem + L.flag_off);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r = blockIdx.x & 1, kx = blockIdx.x >> 1;
    const int nz = a.nz, ny = a.ny;
    Xr += blockIdx.y * x_bstride;  // request of a batched call
    Z += blockIdx.y * z_bstride;
    const float* Sk = request_spec(a, spec, blockIdx.y) + (size_t)(r * a.kx_count + kx) * nz * S_ROW;

    // FFT warp c reads component c's residual column while the tables are built
    const bool transforms = warp >= MT / 32 && warp - MT / 32 < NC;
    float2 u[32];
    if (transforms) {
        const C* col = Xr + ((size_t)kx * a.ncomp + (warp - MT / 32)) * a.ny_pad;
#pragma unroll
        for (int n1 = 0; n1 < 32; ++n1) {
            const int m = 32 * n1 + lane;
            u[n1] = m < ny ? col[m] : make_float2(0.f, 0.f);
        }
    }
    if (tid == 0) {
        // spectra of the first PF layers into L2, later one layer more each
        // iteration, so that the loads ahead hit L2
        for (int n = 0; n < AwShape::PF && n < nz; ++n)
            bulk_prefetch_l2(Sk + (size_t)n * S_ROW, S_ROW * sizeof(float));
        for (int s = 0; s < L.dz; ++s) {
            mbar_init(&zfull[s], MT);
            mbar_init(&zempty[s], 32);
        }
        *abort = 0;
        fence_mbar_init();
    }
    for (int e = tid; e < N; e += NT) {
        tws[e] = tw[e << a.tw_shift_p];
        const int k1 = e >> 5, n2 = e & 31;
        t2[e] = tw[((k1 * n2) & (N - 1)) << a.tw_shift_n];
    }
    __syncthreads();

    // FFT_y of every component's residual column, into slots 0 .. NC-1
    if (transforms) {
        const int c = warp - MT / 32;
        if (r) {
#pragma unroll
            for (int n1 = 0; n1 < 32; ++n1) u[n1] = cmul(u[n1], tws[32 * n1 + lane]);  // fold for ky parity r
        }
        C* fb = ring + c * FS;
        warp_fft1024<false>(u, fb, t2, lane);
#pragma unroll
        for (int j = 0; j < 32; ++j) fb[lane + 32 * bitrev5(j)] = u[j];
    }
    __syncthreads();

    bool failed = false;
    if (tid < MT) {
        // ---------------- combine: thread t owns mirror pairs 2t, 2t + 1 ----------------
        const int q = 2 * tid;
        // bins of the two pairs: k1 = q, q + 1; k2 = N - q, N - q - 1 (even ky;
        // pair 0: the Nyquist bin N / 2) or N - 1 - q, N - 2 - q (odd ky)
        const int k2a = r ? N - 1 - q : q ? N - q : N / 2, k2b = r ? N - 2 - q : N - 1 - q;
        // (the FFT warps form the Nyquist bin, which has spectra values of its own)
        // bins, two-wide over the pairs: re and im of bin 1, of bin 2; conj(S) v
        // with S = s or i s: -i and the mirror sign are applied here
        float2 rc[NC][4];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const C* fb = ring + c * FS;
            C a1 = fb[q], b1 = fb[q + 1], a2 = fb[k2a], b2 = fb[k2b];
            if ((a.imag_mask >> c) & 1u) {
                a1 = make_float2(a1.y, -a1.x);
                b1 = make_float2(b1.y, -b1.x);
                a2 = make_float2(a2.y, -a2.x);
                b2 = make_float2(b2.y, -b2.x);
            }
            if ((a.oddv_mask >> c) & 1u) {
                a2 = make_float2(-a2.x, -a2.y);
                b2 = make_float2(-b2.x, -b2.y);
            }
            rc[c][0] = make_float2(a1.x, b1.x);
            rc[c][1] = make_float2(a1.y, b1.y);
            rc[c][2] = make_float2(a2.x, b2.x);
            rc[c][3] = make_float2(a2.y, b2.y);
        }
        cta_sync();  // every combine thread has its bins: the slots become the ring
        const float* Sq = Sk + q;
        float2 sv[2][NC];
        auto load = [&](int n, float2 (&s)[NC]) {
            if (n >= nz) return;
            const float* row = Sq + (size_t)n * S_ROW;
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c] = load_here2(row + c * JP);
        };
        constexpr int PF = AwShape::PF;
        load(0, sv[0]);
        load(1, sv[1]);
        int sz = 0, wrap = 0;  // ring slot of layer n (n % dz) and n / dz, stepped with n
        auto layer = [&](int n, float2 (&s)[NC]) {
            if (tid == 0 && n + PF < nz) bulk_prefetch_l2(Sk + (size_t)(n + PF) * S_ROW, S_ROW * sizeof(float));
            if (n >= L.dz && !ws_wait(&zempty[sz], (uint32_t)((wrap - 1) & 1), abort)) return false;
            float2 z[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) z[j] = make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int j = 0; j < 4; ++j) z[j] = __ffma2_rn(s[c], rc[c][j], z[j]);
            load(n + 2, s);
            C* zb = ring + sz * FS;
            *reinterpret_cast<float4*>(zb + q) = make_float4(z[0].x, z[1].x, z[0].y, z[1].y);
            zb[k2a] = make_float2(z[2].x, z[3].x);
            zb[k2b] = make_float2(z[2].y, z[3].y);
            mbar_arrive(&zfull[sz]);
            if (++sz == L.dz) {
                sz = 0;
                ++wrap;
            }
            return true;
        };
        for (int n = 0; n < nz; n += 2) {
            if (!layer(n, sv[0]) || (n + 1 < nz && !layer(n + 1, sv[1]))) {
                failed = true;
                break;
            }
        }
        if (cta_sync_or(failed || *abort)) {
            if (tid == 0) atomicExch(err, 1);
        }
    } else {
        // ---------------- FFT warp f: inverse transforms of layers f, f + 8, ... ----------------
        const int f = warp - MT / 32;
        // even ky: lane c holds the Nyquist bin of component c and reads its
        // spectra values, one of its layers ahead; their products add up to
        // bin N / 2 = 32 x 16 of the layer (register 16 of lane 0)
        const bool nyq = r == 0 && lane < NC;
        C rn = make_float2(0.f, 0.f);
        if (nyq) {
            rn = ring[lane * FS + N / 2];
            if ((a.imag_mask >> lane) & 1u) rn = make_float2(rn.y, -rn.x);
        }
        const float* Sn = Sk + (nyq ? lane : 0) * JP + J;
        float sn = nyq && f < nz ? __ldg(Sn + (size_t)f * S_ROW) : 0.f;
        cta_sync();
        // ring slot of layer n (n % dz) and the parity of n / dz, stepped with
        // n (n advances by FW < dz)
        int sz = f, wrap = 0;
        for (int n = f; n < nz; n += FW) {
            int ok = 1;
            if (lane == 0) ok = ws_wait(&zfull[sz], (uint32_t)(wrap & 1), abort);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                failed = true;
                break;
            }
            C* zb = ring + sz * FS;
            float2 u[32];
#pragma unroll
            for (int n1 = 0; n1 < 32; ++n1) u[n1] = zb[32 * n1 + lane];
            if (r == 0) {
                C v = cscale(rn, sn);
                sn = nyq && n + FW < nz ? __ldg(Sn + (size_t)(n + FW) * S_ROW) : 0.f;
#pragma unroll
                for (int o = 4; o; o >>= 1) {
                    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
                    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
                }
                if (lane == 0) u[16] = v;
            }
            __syncwarp();
            warp_fft1024<true>(u, zb, t2, lane);
            if (a.z_tiled) {
                // The slot was only the transform's transpose area: free it now.  Stage the
                // layer in this warp's own buffer in the order of its tiles, Z[.][.][y / 8][kx][8]
                // with row pair (y % 8) / 2 at 16-byte position ((y % 8) / 2 + kx / 2) % 4,
                // and write it with one tensor store (zmap: 8 x kx x y/8 x (r, n) x request)
                // that is not waited for: the next layer waits, before it restages, until
                // this store has read the buffer.
                mbar_arrive(&zempty[sz]);
                C* stg = reinterpret_cast<C*>(smem + L.stage_off) + f * N;
                if (lane == 0) bulk_wait_read_all();  // the previous layer's store has read the buffer
                __syncwarp();
                const int pos = 2 * ((((lane & 7) >> 1) + (kx >> 1)) & 3) + (lane & 1);  // y % 8 = lane % 8
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int y = lane + 32 * bitrev5(j);
                    C v = u[j];
                    if (r) v = cmul(v, cconj(tws[y]));
                    stg[(y & ~7) + pos] = v;
                }
                fence_proxy_async_smem();  // these writes before the tensor store's reads
                __syncwarp();
                if (lane == 0) {
                    tma_store_5d(&zmap, stg, 0, kx, 0, r * nz + n, blockIdx.y);
                    bulk_commit();
                }
            } else {
                mbar_arrive(&zempty[sz]);  // this lane is done with the slot (transposes included)
                C* dst = Z + ((size_t)(r * a.kx_count + kx) * nz + n) * a.ny_pad;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int y = lane + 32 * bitrev5(j);
                    if (y < ny) {
                        C v = u[j];
                        if (r) v = cmul(v, cconj(tws[y]));
                        dst[y] = v;
                    }
                }
            }
            sz += FW;
            if (sz >= L.dz) {
                sz -= L.dz;
                ++wrap;
            }
        }
        if (a.z_tiled && lane == 0) bulk_wait_read_all();  // every tensor store has read its buffer
        cta_sync_or(failed || *abort);
    }
}

// Ring depth and offsets; dz == 0 when the kernel does not apply.
inline AwSmem aw_smem(int ny_pad, int ncomp, int jp, int nc_inst, int max_bytes) {
    if (ny_pad > AwShape::N || nc_inst > AwShape::FWARPS || ncomp != nc_inst || jp != AwShape::JP) return AwSmem{};
    for (int dz = 16; dz >= AwShape::FWARPS + 2; --dz) {
        AwSmem l{};
        l.dz = dz;
        l.slot_off = 0;
        l.tw_off = (uint32_t)(dz * AwShape::SLOT * sizeof(float2));
        l.t2_off = l.tw_off + AwShape::N * sizeof(float2);
        l.stage_off = (l.t2_off + AwShape::N * sizeof(float2) + 127) & ~127u;  // tensor-store sources: 128-byte aligned
        l.bar_off = l.stage_off + AwShape::FWARPS * AwShape::N * sizeof(float2);
        l.flag_off = l.bar_off + 2 * dz * 8;
        l.total = l.flag_off + 16;
        if ((int)l.total <= max_bytes) return l;
    }
    return AwSmem{};
}

}  // namespace grav
