// Adjoint column stage for 64-, 128- and 256-point FP32 columns: launches of
// the kernel in col_groups.cuh.
#include <type_traits>

#include "col_groups.cuh"

namespace grav {

namespace {

// Layers per CTA: all of them, halved (to whole rounds of 8, at least 8)
// until the launch gives every SM 8 warps; each CTA repeats the residual
// transforms, about one round's work, so chunks only pay where SMs would idle
// (256 x 256 x 32, six components, whole adjoint: 37.6 us, with 16 warps an SM
// as the goal 40.0, with 32 41.0).
template <int N> int chunk_layers(const ColumnArgs& a, int batch) {
    constexpr int R = ColGroup<N>::SLOTS;
    int chunk = (a.nz + R - 1) / R * R;
    while (chunk > R && (long)a.kx_count * batch * (N / 32) * ((a.nz + chunk - 1) / chunk) < 152 * 8)
        chunk = (chunk / 2 + R - 1) / R * R;
    return chunk;
}

template <int N, int NC>
cudaError_t launch_nc(const ColumnArgs& a, const void* Xr, const float* spec, void* Z, const void* tw, cudaStream_t s,
                      Batch b) {
    using S = ColGroup<N>;
    constexpr auto k = adjoint_column_group_kernel<N, NC>;
    const int chunk = chunk_layers<N>(a, b.count);
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    return launch_chained(k, dim3(a.kx_count, (a.nz + chunk - 1) / chunk, b.count), N, S::adj_smem, s, a, chunk,
                          (const float2*)Xr, spec, (float2*)Z, (const float2*)tw, b.in, b.out);
}

template <int N>
cudaError_t launch_n(const ColumnArgs& a, const void* Xr, const float* spec, void* Z, const void* tw, cudaStream_t s,
                     Batch b) {
    switch (a.ncomp) {
        case 1: return launch_nc<N, 1>(a, Xr, spec, Z, tw, s, b);
        case 2: return launch_nc<N, 2>(a, Xr, spec, Z, tw, s, b);
        case 3: return launch_nc<N, 3>(a, Xr, spec, Z, tw, s, b);
        case 4: return launch_nc<N, 4>(a, Xr, spec, Z, tw, s, b);
        case 5: return launch_nc<N, 5>(a, Xr, spec, Z, tw, s, b);
        case 6: return launch_nc<N, 6>(a, Xr, spec, Z, tw, s, b);
        case 7: return launch_nc<N, 7>(a, Xr, spec, Z, tw, s, b);
        case 8: return launch_nc<N, 8>(a, Xr, spec, Z, tw, s, b);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_adjoint_groups(int log_n, const ColumnArgs& a, const void* Xr, const float* spec, void* Z,
                                  const void* tw, cudaStream_t s, Batch b) {
    switch (log_n) {
        case 6: return launch_n<64>(a, Xr, spec, Z, tw, s, b);
        case 7: return launch_n<128>(a, Xr, spec, Z, tw, s, b);
        case 8: return launch_n<256>(a, Xr, spec, Z, tw, s, b);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace grav
