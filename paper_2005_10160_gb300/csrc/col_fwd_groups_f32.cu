// Forward column stage for 64-, 128- and 256-point FP32 columns: launches of
// the kernel in col_groups.cuh.
#include <type_traits>

#include "col_groups.cuh"

namespace grav {

namespace {

// Layer groups per CTA: one, except for 64-point columns, whose group is a
// single warp: those take the layers in one go (up to 8 groups).  Measured in an
// earlier form of the kernel, whole calls at 256 x 256 x 32 and 16 requests of
// 128 x 128 x 32, six components (39 and 105 us now): one group 49 and 112 us,
// two and four groups 51 and 152 us (the final sum over the groups costs more
// than the shorter chain gains).  The rule looks at the plan
// only: the order of the layer sum, and so the result, must not depend on how
// many requests share a launch.
template <int N> int layer_groups(const ColumnArgs& a) {
    int g = 1;
    while (N == 64 && g < ColGroup<N>::MAXG && g * ColGroup<N>::SLOTS < a.nz) g *= 2;
    return g;
}

template <int N, int NC>
cudaError_t launch_nc(const ColumnArgs& a, const void* X, const float* spec, void* Y, const void* tw, cudaStream_t s,
                      Batch b) {
    using S = ColGroup<N>;
    constexpr auto k = forward_column_group_kernel<N, NC>;
    const int g = layer_groups<N>(a);
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    return launch_chained(k, dim3(2 * a.kx_count, b.count), g * S::J, S::fwd_smem(g, NC), s, a, g, (const float2*)X,
                          spec, (float2*)Y, (const float2*)tw, b.in, b.out);
}

template <int N>
cudaError_t launch_n(const ColumnArgs& a, const void* X, const float* spec, void* Y, const void* tw, cudaStream_t s,
                     Batch b) {
    switch (a.ncomp) {
        case 1: return launch_nc<N, 1>(a, X, spec, Y, tw, s, b);
        case 2: return launch_nc<N, 2>(a, X, spec, Y, tw, s, b);
        case 3: return launch_nc<N, 3>(a, X, spec, Y, tw, s, b);
        case 4: return launch_nc<N, 4>(a, X, spec, Y, tw, s, b);
        case 5: return launch_nc<N, 5>(a, X, spec, Y, tw, s, b);
        case 6: return launch_nc<N, 6>(a, X, spec, Y, tw, s, b);
        case 7: return launch_nc<N, 7>(a, X, spec, Y, tw, s, b);
        case 8: return launch_nc<N, 8>(a, X, spec, Y, tw, s, b);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_forward_groups(int log_n, const ColumnArgs& a, const void* X, const float* spec, void* Y,
                                  const void* tw, cudaStream_t s, Batch b) {
    switch (log_n) {
        case 6: return launch_n<64>(a, X, spec, Y, tw, s, b);
        case 7: return launch_n<128>(a, X, spec, Y, tw, s, b);
        case 8: return launch_n<256>(a, X, spec, Y, tw, s, b);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace grav
