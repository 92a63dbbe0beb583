// FP64 kernel generation: the translation-equivalent geometric kernel
// K_c(u, v, n) of every component c over the offset grid (Eq. 10), i.e. the
// first row and column of every Toeplitz block of G (Eqs. 17, 19).
//
// K_c(u, v, n) is the field at a station due to a unit-density cell offset
// by (u, v) columns in layer n.  With the station at the origin the cell has
// corners x_i = (1/2 - u) dx, -(1/2 + u) dx, y_j likewise, z_k = -h - zeta_k
// with zeta in {n dz, (n+1) dz}, and
//     K_c = upsilon * sum_{ijk} mu_ijk F_c(x_i, y_j, z_k),  mu_ijk = (-1)^(i+j+k)
// (Eq. 2).  F_c is the closed form of Eq. 2 for gz (its logarithms written
// as asinh, which is the same function and keeps far offsets accurate) and
// the standard prism forms for the gradient components:
//     gxx: atan(yz/(xr))   gyy: atan(xz/(yr))   gzz: atan(xy/(zr))
//     gxy: -asinh(z/sqrt(x^2+y^2))   gxz: -asinh(y/sqrt(x^2+z^2))
//     gyz: -asinh(x/sqrt(y^2+z^2))
// and for the horizontal first derivatives the gz form with x (resp. y) as
// the distinguished axis:
//     gx: -[y asinh(z/sqrt(x^2+y^2)) + z asinh(y/sqrt(x^2+z^2)) - x atan(yz/(xr))]
//     gy: -[z asinh(x/sqrt(y^2+z^2)) + x asinh(z/sqrt(x^2+y^2)) - y atan(xz/(yr))]
// FP64 throughout: the eight corner terms cancel to a few parts in 1e7 at
// the far offsets of a 1024-cell mesh, so FP32 generation is unusable.
//
// One thread per offset (u, v) of the quadrant u, v >= 0, in tiles that
// share their corner terms (see kernel_gen below).  Walking down the layers,
// each thread writes its quadrant value, or the four mirrored offsets
// (+-u, +-v) using the component's parity under reflection (Sec. 2.2), so the
// kernel is exactly even or odd.
#include <algorithm>

#include "corner_terms.cuh"
#include "grav_internal.h"

namespace grav {

namespace {

// asinh(v / rho), inv = 1 / rho > 0, s = rho + sqrt(rho^2 + v^2), by
// asinh(q) = log1p(q + q^2 / (1 + sqrt(1 + q^2))), which keeps the relative
// accuracy of small q.
__device__ __forceinline__ double asinh_ratio(double v, double inv, double s, const CornerTables& t) {
    const double a = fabs(v), q = a * inv;
    return copysign(log1p_pos(fma(q, a / s, q), t), v);
}

// A distance and its inverse.
struct Dist { double d, inv; };
__device__ __forceinline__ Dist distance(double a, double b) {
    const double d = sqrt(a * a + b * b);
    return Dist{d, 1.0 / d};
}

// NC: components kept per corner, 7 (gz ... gzz) or 9 (with gx, gy); plans
// without gx, gy use 7 so that the kernel keeps fewer registers.  rxy, rxz,
// ryz: distances in the coordinate planes.
//
// TABLES: corner_terms.cuh and the shared distances, for plans that store FP32
// spectra (see corner_tables_fit).  Otherwise CUDA's asinh and atan, 2.3 times
// the FP64 instructions.
template <int NC, bool TABLES>
__device__ __forceinline__ void corner_terms(double x, double y, double z, const Dist* rxy, const Dist* rxz,
                                             const Dist* ryz, unsigned comps, const CornerTables& t,
                                             double (&F)[NC]) {
    const bool want_ay = comps & (GRAV_GZ | GRAV_GXZ | GRAV_GX), want_ax = comps & (GRAV_GZ | GRAV_GYZ | GRAV_GY),
               want_az = comps & (GRAV_GXY | GRAV_GX | GRAV_GY), want_tz = comps & (GRAV_GZ | GRAV_GZZ),
               want_tx = comps & (GRAV_GXX | GRAV_GX), want_ty = comps & (GRAV_GYY | GRAV_GY);
    const double x2 = x * x, y2 = y * y, z2 = z * z, r = sqrt(x2 + y2 + z2);
    double ay = 0.0, ax = 0.0, az = 0.0, tz = 0.0, tx = 0.0, ty = 0.0;
    if constexpr (TABLES) {
        const double xa = fabs(x), ya = fabs(y), za = fabs(z);
        if (want_ay) ay = asinh_ratio(y, rxz->inv, r + rxz->d, t);
        if (want_ax) ax = asinh_ratio(x, ryz->inv, r + ryz->d, t);
        if (want_az) az = asinh_ratio(z, rxy->inv, r + rxy->d, t);
        if (want_tz) tz = copysign(atan_ratio(xa * ya, za * r, t), x * y * z);
        if (want_tx) tx = copysign(atan_ratio(ya * za, xa * r, t), x * y * z);
        if (want_ty) ty = copysign(atan_ratio(xa * za, ya * r, t), x * y * z);
    } else {
        if (want_ay) ay = asinh(y / sqrt(x2 + z2));
        if (want_ax) ax = asinh(x / sqrt(y2 + z2));
        if (want_az) az = asinh(z / sqrt(x2 + y2));
        if (want_tz) tz = atan(x * y / (z * r));
        if (want_tx) tx = atan(y * z / (x * r));
        if (want_ty) ty = atan(x * z / (y * r));
    }
    F[0] = -(x * ay + y * ax - z * tz);
    F[1] = tx;
    F[2] = -az;
    F[3] = -ay;
    F[4] = ty;
    F[5] = -ax;
    F[6] = tz;
    if constexpr (NC > 7) {
        F[7] = -(y * az + z * ay - x * tx);  // gx: the gz form with x as the distinguished axis
        F[8] = -(z * ax + x * az - y * ty);  // gy: the same with y
    }
}

// v as an unevaluated FP32 pair; the high part truncates v by integer
// arithmetic (conversions run at the FP64 rate), 0 below FP32's range.
__device__ __forceinline__ float2 split_pair(double v) {
    const uint64_t b = bits_of(v);
    const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
    const bool ok = e > 0 && e < 255;
    const uint32_t hb = (uint32_t)(b >> 63) << 31 | (uint32_t)(e & 255) << 23 | (uint32_t)((b >> 29) & 0x7fffffu);
    const double hd = of_bits(b & ~0x1fffffffull);
    return ok ? make_float2(__uint_as_float(hb), (float)(v - hd)) : make_float2((float)v, 0.f);
}

// Offsets per CTA: a kGenTX x TY tile of the quadrant.  Neighbouring
// offsets share prism corners (the far x-corner of offset u is the near one
// of u + 1), so the CTA evaluates the corner terms of its (kGenTX + 1) x
// (TY + 1) corners once per z-level, keeps the difference to the level
// above in shared memory, and every thread forms its offsets' kernel values
// from four differences.  blockIdx.z takes a run of `per` layers.
//
// Bound by the FP64 pipe, 86% active with the tables (four layers of 1024 x
// 1024).  1024 x 1024 x 100, six components: 65 ms with the tables, 92 ms with the library's
// asinh and atan and tiles of 32 x 8.
constexpr int kGenTX = 32, kGenThreads = 256;
template <int TY> struct GenTile {
    static constexpr int CX = kGenTX + 1, CY = TY + 1, COR = CX * CY;
    static constexpr size_t smem(int nc) {
        return sizeof(CornerTables) + (size_t)COR * 2 * nc * sizeof(double) + (size_t)(COR + CX + CY) * sizeof(Dist);
    }
};

template <int NC, bool TABLES, int TY>
__global__ void __launch_bounds__(kGenThreads)
    kernel_gen(Geometry g, GenOut o, unsigned comps, int n0, int n1, int per, void* __restrict__ out) {
    constexpr int CX = GenTile<TY>::CX, CY = GenTile<TY>::CY, COR = GenTile<TY>::COR, NT = kGenThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CornerTables& tab = *reinterpret_cast<CornerTables*>(smem_raw);
    double* F = reinterpret_cast<double*>(smem_raw + sizeof(CornerTables));  // corner terms of the level above
    double* D = F + COR * NC;   // level minus the level above
    Dist* rxy = reinterpret_cast<Dist*>(D + COR * NC);  // sqrt(x^2 + y^2) per corner
    Dist* rxz = rxy + COR;                              // sqrt(x^2 + z^2), sqrt(y^2 + z^2) of the level
    Dist* ryz = rxz + CX;
    const int tid = threadIdx.x, tx = tid % kGenTX, ty0 = tid / kGenTX;
    const int u0 = blockIdx.x * kGenTX, v0 = blockIdx.y * TY;
    const int u = u0 + tx;
    const int first = n0 + blockIdx.z * per, last = min(n1, first + per);

    // corner (cx, cy) sits at x = (1/2 - u0 - cx) dx, y = (1/2 - v0 - cy) dy (station at the origin)
    auto cx_of = [&](int cx) { return (0.5 - (u0 + cx)) * g.dx; };
    auto cy_of = [&](int cy) { return (0.5 - (v0 + cy)) * g.dy; };
    if constexpr (TABLES) {
        for (int e = tid; e < CornerTables::LOGS; e += NT) corner_table_entry(tab, e);
        for (int e = tid; e < COR; e += NT) rxy[e] = distance(cx_of(e % CX), cy_of(e / CX));
    }
    // corner terms of z-level z into F and, but for the first level, their change into D
    auto level = [&](double z, bool difference) {
        if constexpr (TABLES) {
            if (tid < CX) rxz[tid] = distance(cx_of(tid), z);
            else if (tid >= 64 && tid < 64 + CY) ryz[tid - 64] = distance(cy_of(tid - 64), z);
        }
        __syncthreads();  // distances in place; D and the tables free or in place
        for (int e = tid; e < COR; e += NT) {
            const int cy = e / CX, cx = e - cy * CX;
            if (u0 + cx > g.nx || v0 + cy > g.ny) continue;
            double t[NC];
            corner_terms<NC, TABLES>(cx_of(cx), cy_of(cy), z, rxy + e, rxz + cx, ryz + cy, comps, tab, t);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (!(comps & (1u << c))) continue;
                if (difference) D[e * NC + c] = t[c] - F[e * NC + c];
                F[e * NC + c] = t[c];
            }
        }
        __syncthreads();
    };

    const int nzc = n1 - n0;
    const int wx = 2 * g.nx - 1, wy = 2 * g.ny - 1;
    level(-g.h - first * g.dz, false);
    for (int n = first; n < last; ++n) {
        level(-g.h - (n + 1) * g.dz, true);
        for (int ty = ty0; ty < TY; ty += NT / kGenTX) {
            const int v = v0 + ty;
            if (u >= g.nx || v >= g.ny) continue;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (!(comps & (1u << c))) continue;
                const int s = __popc(comps & ((1u << c) - 1u));  // output slot of component c
                // mu_ijk: +1 for the bottom z-level when i + j is even; corners
                // (u + i, v + j)
                const double* d = D + (ty * CX + tx) * NC + c;
                const double K = o.factor[c] * ((d[0] - d[CX * NC]) - (d[NC] - d[CX * NC + NC]));
                const bool zero = (u == 0 && odd_u(c)) || (v == 0 && odd_v(c));
                if (o.mode == GenOut::kQuadrant || o.mode == GenOut::kQuadrantPairs) {
                    // the offset (-u, -v)
                    const double val = zero ? 0.0 : odd_u(c) != odd_v(c) ? -K : K;
                    const size_t idx = (((size_t)s * nzc + (n - n0)) * g.ny + v) * g.nx + u;
                    if (o.mode == GenOut::kQuadrant) static_cast<double*>(out)[idx] = val;
                    else static_cast<float2*>(out)[idx] = split_pair(val);
                    continue;
                }
                double* dst = static_cast<double*>(out);
                for (int mu = 0; mu < (u > 0 ? 2 : 1); ++mu) {
                    for (int mv = 0; mv < (v > 0 ? 2 : 1); ++mv) {
                        double val = K;
                        if (mu && odd_u(c)) val = -val;
                        if (mv && odd_v(c)) val = -val;
                        if (zero) val = 0.0;
                        const int U = mu ? -u : u, V = mv ? -v : v;
                        if (o.mode == GenOut::kHalfRows) {
                            // rows b = -V < py / 2 only (V <= 0): the rest mirror them
                            if (V > 0) continue;
                            const int a = (o.px - U) & (o.px - 1), b = -V;
                            dst[(((size_t)s * nzc + (n - n0)) * (o.py / 2) + b) * o.px + a] = val;
                        } else {
                            dst[(((size_t)s * g.nz + n) * wy + (V + g.ny - 1)) * wx + (U + g.nx - 1)] = val;
                        }
                    }
                }
            }
        }
    }
}

// Tiles of TY rows, and the runs of layers that they are cut into: each run
// costs one level more, so at least 8 layers, and no more runs than give every
// SM 12 CTAs.
dim3 gen_grid(const Geometry& g, int nz, int ty, int* per) {
    dim3 grid((g.nx + kGenTX - 1) / kGenTX, (g.ny + ty - 1) / ty);
    const int tiles = (int)(grid.x * grid.y);
    const int want = std::max(1, std::min((12 * 152 + tiles - 1) / tiles, nz / 8));
    *per = (nz + want - 1) / want;
    grid.z = (nz + *per - 1) / *per;
    return grid;
}

template <int NC, bool TABLES, int TY>
cudaError_t gen_launch(const Geometry& g, const GenOut& o, unsigned comps, int n0, int n1, void* out, cudaStream_t s) {
    constexpr auto k = kernel_gen<NC, TABLES, TY>;
    cudaError_t e = ensure_smem_limit<k>();
    if (e != cudaSuccess) return e;
    int per;
    const dim3 grid = gen_grid(g, n1 - n0, TY, &per);
    k<<<grid, kGenThreads, GenTile<TY>::smem(NC), s>>>(g, o, comps, n0, n1, per, out);
    return cudaGetLastError();
}

template <int NC>
cudaError_t gen_either(const Geometry& g, const GenOut& o, unsigned comps, int n0, int n1, void* out, cudaStream_t s) {
    if (o.tables) return gen_launch<NC, true, 16>(g, o, comps, n0, n1, out, s);
    // the library functions' corners take long enough that a mesh of fewer
    // tiles than SMs waits for the trips of one tile: two of 256 corners a level
    // with 8 rows, three with 16 (16 x 16 x 4 FP64 plan, six components: 370 us
    // with 8, 510 with 16; where the SMs are full 16 rows share more corners)
    int per;
    const dim3 grid = gen_grid(g, n1 - n0, 16, &per);
    if (grid.x * grid.y * grid.z < 152) return gen_launch<NC, false, 8>(g, o, comps, n0, n1, out, s);
    return gen_launch<NC, false, 16>(g, o, comps, n0, n1, out, s);
}

}  // namespace

cudaError_t launch_kernel_gen(const Geometry& g, const GenOut& o, unsigned comps, int n0, int n1, void* out,
                              cudaStream_t s) {
    comps &= kCompBits;
    return comps & (GRAV_GX | GRAV_GY) ? gen_either<9>(g, o, comps, n0, n1, out, s)
                                       : gen_either<7>(g, o, comps, n0, n1, out, s);
}

// The eight corner terms cancel, so a kernel value carries their rounding
// enlarged.  Over meshes wider than they are deep that stays below FP32's
// rounding in the field, and the tables' is 0.7 .. 1.2 times the library
// functions'.  For a narrow mesh far below its stations it does not: with z the
// deepest level, V a cell's volume and X, Y the mesh's width it is about 2^-53
// z^3 / V, times z / X and z / Y for the components odd in x and y, and the
// tables' rounding of those is up to 2.3 times the functions' (7 x 3 x 5 cells
// of 84 x 40 x 65 m at 6800 m: gxy 4.3e-7 of the field with the functions, 1e-6
// with the tables).  Measured on 220 meshes of 3 .. 1024 cells a side, both
// layers' ends and nine components against 113-bit arithmetic: what the tables
// add to a field error of 2e-7 is below 3e-4 of it up to a factor of 2^22, and
// below 2e-4 of it on every mesh no deeper than wide.  (Equal-dimension plans
// transform all depths together, where the offsets near a station set the
// size: they always take the tables for FP32 spectra.)
bool corner_tables_fit(const Geometry& g) {
    const double z = g.h + g.nz * g.dz, X = std::max(g.nx - 1, 1) * g.dx, Y = std::max(g.ny - 1, 1) * g.dy;
    if (z <= X && z <= Y) return true;
    return z / g.dx * (z / g.dy) * (z / g.dz) * std::max(1.0, z / X) * std::max(1.0, z / Y) <= 0x1p22;
}

GenOut gen_out(GenOut::Mode mode, bool tables, int px, int py) {
    GenOut o{};
    o.mode = mode;
    o.tables = tables;
    o.px = px;
    o.py = py;
    for (double& f : o.factor) f = kUpsilon;
    return o;
}

}  // namespace grav
