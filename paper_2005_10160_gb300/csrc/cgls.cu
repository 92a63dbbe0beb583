// The damped CGLS loop (least-squares density inversion, Sec. 1 and Sec. 4)
// enqueued whole on one stream: forward and adjoint products plus the vector
// updates between them, with every scalar of the recurrence on the device, so
// the host neither waits nor launches per dot product.
//
// In x = W_m m with s = A^T r - lam x, A = W_d G W_m^-1:
//   q = A p;  alpha = (s, s) / ((q, q) + lam (p, p));  x += alpha p;  r -= alpha q
//   s' = A^T r - lam x;  beta = (s', s') / (s, s);  p = s' + beta p
// The model-size vectors are touched twice per iteration:
//   step_model   x += alpha p, s = g / w_n - lam x (in place of g = G^T w r), (s, s), (x, x)
//   next_dir     p = s + beta p, t = p / w_n (the next forward's input), (p, p)
// i.e. nine passes over a vector in all, where separate operations took
// about forty.  A dot product is one FP64 partial per block; the last block to
// finish adds them in a fixed order, so the kernels that use it read one number.
//
// 512 x 512 x 64, two components: 0.57 GB per iteration in 0.15 ms (step_model
// 68 us, next_dir 55, the three data-size kernels 10 each); three iterations
// from 4.68 to 2.30 ms, 1.9 ms of vector operations before.
//
// FP64 instructions run at 1/64 of the FP32 rate here, and two products and
// two widenings per element in FP64 took longer than the memory traffic
// (step_model 174 us at 512 x 512 x 64 for 0.34 GB).  A thread therefore keeps
// an FP32 plan's sum as an unevaluated pair of floats: the product's rounding
// error by fused multiply-add, the sum's by the two-sum of Knuth (TAOCP 2,
// 4.2.2), both added to the low part; the sum is good to about 2^-45, more than
// that of separately rounded FP32 products.  A pair has FP32's range: a thread
// whose sum leaves it adds FP32 products in FP64 over the values it has stored
// (a test for it in the loop, with FP64 instructions behind it, took the three
// iterations below from 2.08 to 3.06 ms), and the rounding error of a square
// below about 1e-32 is lost, as in an FP32 product.
#include <algorithm>

#include "grav_internal.h"

namespace grav {

namespace {

constexpr int kVecThreads = 256;
constexpr int kMaxParts = 1216;  // most blocks (partial sums) of a vector kernel: 8 per SM

// Sum over the block, valid in thread 0.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double part[kVecThreads / 32];
    __syncthreads();  // an earlier sum's values are read
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kVecThreads / 32; ++w) s += part[w];
    return s;
}

// A dot product: the result, and the number of blocks that have handed in
// their share (0 before and after each use).
struct Dot {
    double value;
    unsigned done, pad;
};
// A dot product in the making and where the blocks' partials go: one array per
// dot product of a kernel, free again when the kernel ends.
struct Making {
    Dot* dot;
    double* parts;
};

// Every block of the grid hands in its share (all threads call this); the last
// one adds the partials up in block order.
__device__ __forceinline__ void put_dot(Making m, double share) {
    Dot* d = m.dot;
    __shared__ bool last;
    const unsigned nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x;
    const double s = block_sum(share);
    if (threadIdx.x == 0) {
        m.parts[b] = s;
        __threadfence();
        last = atomicInc(&d->done, nb - 1) == nb - 1;  // wraps to 0 for the next use
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double v = 0.0;
    for (unsigned i = threadIdx.x; i < nb; i += kVecThreads) v += __ldcg(&m.parts[i]);
    v = block_sum(v);
    if (threadIdx.x == 0) d->value = v;
}

// Sum of squares of one thread's values.
template <typename R> struct Squares;
template <> struct Squares<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s += v * v; }
    template <typename F> __device__ __forceinline__ double get(F&&) const { return s; }
};
template <> struct Squares<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float p = __fmul_rn(v, v), pe = __fmaf_rn(v, v, -p);
        const float t = __fadd_rn(hi, p), z = __fsub_rn(t, hi);
        const float te = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(p, z));
        hi = t;
        lo = __fadd_rn(lo, __fadd_rn(pe, te));
    }
    // again(f) calls f with every value once more
    template <typename F> __device__ __forceinline__ double get(F&& again) const {
        if (isfinite(hi)) return (double)hi + (double)lo;
        double s = 0.0;
        again([&](float v) { s += (double)__fmul_rn(v, v); });
        return s;
    }
};

template <typename R, int VEC> struct alignas(sizeof(R) * VEC) Pack { R v[VEC]; };

// f(v) for every value of a data-size vector that this thread wrote.
template <typename R, typename F> __device__ __forceinline__ void each_data(const R* v, size_t n, F&& f) {
    for (size_t i = (size_t)blockIdx.x * kVecThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kVecThreads) f(v[i]);
}
// The same for a model-size vector.
template <int VEC, typename R, typename F>
__device__ __forceinline__ void each_model(const R* v, size_t plane, int nz, F&& f) {
    for (int n = blockIdx.y; n < nz; n += gridDim.y)
        for (size_t i = ((size_t)blockIdx.x * kVecThreads + threadIdx.x) * VEC; i < plane; i += (size_t)gridDim.x * kVecThreads * VEC)
            for (int j = 0; j < VEC; ++j) f(v[(size_t)n * plane + i + j]);
}

// What the steps found, the first int of the workspace.
enum { kStepsDone = 0, kNoStepLength = 1, kStepLengthRange = 2 };

// (s, s) before the step, (p, p), (q, q)
struct Scalars {
    const Dot *gamma, *pp, *qq;
    double lam;
    int* status;
};
// alpha, the same value in every thread.  A vanished gradient ends the
// recurrence: nothing moves any more.  RECORD: one thread of the grid notes a
// step without a length (a gradient, but (q, q) + lam (p, p) = 0) or with one
// past R's range.
template <typename R, bool RECORD> __device__ __forceinline__ double step_length(const Scalars& k) {
    __shared__ double alpha;
    if (threadIdx.x == 0) {
        const double gamma = k.gamma->value, curv = k.qq->value + k.lam * k.pp->value;
        const double a = gamma == 0.0 ? 0.0 : gamma / curv;
        alpha = a;
        if (RECORD && blockIdx.x == 0 && gamma != 0.0 && !isfinite((R)a) && *k.status == kStepsDone) {
            if (curv == 0.0) *k.status = kNoStepLength;
            else if (isfinite(a)) *k.status = kStepLengthRange;
        }
    }
    __syncthreads();
    return alpha;
}

// r = w d, wr = w r, (r, r); clears the status
template <typename R>
__global__ void __launch_bounds__(kVecThreads) cgls_first_data(const R* __restrict__ d, const R* __restrict__ w, R* __restrict__ r,
                                                               R* __restrict__ wr, size_t n, Making rr, int* status) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *status = kStepsDone;
    Squares<R> s;
    for (size_t i = (size_t)blockIdx.x * kVecThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kVecThreads) {
        const R v = w[i] * d[i];
        r[i] = v;
        wr[i] = w[i] * v;
        s.add(v);
    }
    put_dot(rr, s.get([&](auto f) { each_data(r, n, f); }));
}

// q = w y in place, (q, q)
template <typename R>
__global__ void __launch_bounds__(kVecThreads) cgls_weigh(const R* __restrict__ w, R* __restrict__ q, size_t n, Making qq) {
    Squares<R> s;
    for (size_t i = (size_t)blockIdx.x * kVecThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kVecThreads) {
        const R v = w[i] * q[i];
        q[i] = v;
        s.add(v);
    }
    put_dot(qq, s.get([&](auto f) { each_data(q, n, f); }));
}

// r -= alpha q, wr = w r, (r, r)
template <typename R>
__global__ void __launch_bounds__(kVecThreads) cgls_step_data(Scalars k, const R* __restrict__ w, const R* __restrict__ q, R* __restrict__ r,
                                                              R* __restrict__ wr, size_t n, Making rr) {
    const R alpha = (R)step_length<R, true>(k);
    Squares<R> s;
    for (size_t i = (size_t)blockIdx.x * kVecThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kVecThreads) {
        const R v = r[i] - alpha * q[i];
        r[i] = v;
        wr[i] = w[i] * v;
        s.add(v);
    }
    put_dot(rr, s.get([&](auto f) { each_data(r, n, f); }));
}

// Model-size kernels: block rows take layers blockIdx.y, blockIdx.y + gridDim.y,
// ..., so that the depth weight is constant over a block's inner loop.
#define GRAV_FOR_LAYERS                                        \
    for (int n = blockIdx.y; n < nz; n += gridDim.y) {         \
        const R wn = wm[n];                                    \
        const size_t base = (size_t)n * plane;                 \
        for (size_t i = ((size_t)blockIdx.x * kVecThreads + threadIdx.x) * VEC; i < plane; i += (size_t)gridDim.x * kVecThreads * VEC) {

// s = g / w_n in place, p = s, t = p / w_n, (s, s)
template <typename R, int VEC>
__global__ void __launch_bounds__(kVecThreads) cgls_first_model(const R* __restrict__ wm, R* __restrict__ g, R* __restrict__ p,
                                                                R* __restrict__ t, size_t plane, int nz, Making ss, Making pp) {
    using P = Pack<R, VEC>;
    Squares<R> sum;
    GRAV_FOR_LAYERS
            P gv = *reinterpret_cast<const P*>(g + base + i), tv;
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                const R s = gv.v[j] / wn;
                gv.v[j] = s;
                tv.v[j] = s / wn;
                sum.add(s);
            }
            *reinterpret_cast<P*>(p + base + i) = gv;
            *reinterpret_cast<P*>(t + base + i) = tv;
        }
    }
    const double share = sum.get([&](auto f) { each_model<VEC>(p, plane, nz, f); });
    put_dot(ss, share);
    put_dot(pp, share);
}

// x += alpha p (x = alpha p in the first step), s = g / w_n - lam x in place
// of g, (s, s), (x, x); m = x / w_n if wanted
template <typename R, int VEC>
__global__ void __launch_bounds__(kVecThreads) cgls_step_model(Scalars k, bool first, const R* __restrict__ wm, const R* __restrict__ p, R* __restrict__ x,
                                                               R* __restrict__ g, R* __restrict__ m, size_t plane, int nz,
                                                               Making ss, Making xx) {
    using P = Pack<R, VEC>;
    const R alpha = (R)step_length<R, false>(k), lam = (R)k.lam;
    Squares<R> s2, x2;
    GRAV_FOR_LAYERS
            const P pv = *reinterpret_cast<const P*>(p + base + i);
            P gv = *reinterpret_cast<const P*>(g + base + i), xv, mv;
            if (first) {
#pragma unroll
                for (int j = 0; j < VEC; ++j) xv.v[j] = 0;
            } else {
                xv = *reinterpret_cast<const P*>(x + base + i);
            }
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                xv.v[j] += alpha * pv.v[j];
                const R s = gv.v[j] / wn - lam * xv.v[j];
                gv.v[j] = s;
                mv.v[j] = xv.v[j] / wn;
                s2.add(s);
                x2.add(xv.v[j]);
            }
            *reinterpret_cast<P*>(x + base + i) = xv;
            *reinterpret_cast<P*>(g + base + i) = gv;
            if (m) *reinterpret_cast<P*>(m + base + i) = mv;
        }
    }
    put_dot(ss, s2.get([&](auto f) { each_model<VEC>(g, plane, nz, f); }));
    put_dot(xx, x2.get([&](auto f) { each_model<VEC>(x, plane, nz, f); }));
}

// p = s + beta p, t = p / w_n, (p, p)
template <typename R, int VEC>
__global__ void __launch_bounds__(kVecThreads) cgls_next_dir(const Dot* gamma, const Dot* gamma_new, const R* __restrict__ wm,
                                                             const R* __restrict__ s, R* __restrict__ p, R* __restrict__ t,
                                                             size_t plane, int nz, Making pp) {
    using P = Pack<R, VEC>;
    __shared__ double beta_sh;
    if (threadIdx.x == 0) beta_sh = gamma->value == 0.0 ? 0.0 : gamma_new->value / gamma->value;
    __syncthreads();
    const R beta = (R)beta_sh;
    Squares<R> p2;
    GRAV_FOR_LAYERS
            const P sv = *reinterpret_cast<const P*>(s + base + i);
            P pv = *reinterpret_cast<const P*>(p + base + i), tv;
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                pv.v[j] = sv.v[j] + beta * pv.v[j];
                tv.v[j] = pv.v[j] / wn;
                p2.add(pv.v[j]);
            }
            *reinterpret_cast<P*>(p + base + i) = pv;
            *reinterpret_cast<P*>(t + base + i) = tv;
        }
    }
    put_dot(pp, p2.get([&](auto f) { each_model<VEC>(p, plane, nz, f); }));
}
#undef GRAV_FOR_LAYERS

// objectives[k] = (r, r) + lam (x, x) after k steps; dots: (r, r), (x, x), (s, s) per step
__global__ void __launch_bounds__(kVecThreads) cgls_objectives(const Dot* dots, int n, double lam, double* __restrict__ obj) {
    for (int k = threadIdx.x; k < n; k += kVecThreads) obj[k] = dots[3 * k].value + (k ? lam * dots[3 * k + 1].value : 0.0);
}

size_t pad256(size_t v) { return (v + 255) / 256 * 256; }

// The caller's workspace: the status; data vectors r, q, wr; model vectors p, t,
// g, x; two arrays of partials; then the dot products: (p, p), (q, q) and, per
// step, (r, r), (x, x), (s, s).
struct Work {
    static constexpr size_t kHead = 256;  // the status
    size_t nd, plane, data, model;
    int nz, iters;
    size_t dots() const { return 2 + 3 * ((size_t)iters + 1); }
    static constexpr size_t kParts = kMaxParts * sizeof(double);
    size_t bytes() const { return kHead + 3 * data + 4 * model + 2 * kParts + dots() * sizeof(Dot); }
};
Work work_of(const grav_plan* p, int iters) {
    Work w{};
    const size_t real = p->fp64 ? 8 : 4;
    w.plane = (size_t)p->ny * p->nx;
    w.nd = w.plane * p->ncomp;
    w.nz = p->nz;
    w.iters = iters;
    w.data = pad256(w.nd * real);
    w.model = pad256(w.plane * p->nz * real);
    return w;
}

template <typename R> struct Loop {
    Work k;
    int* status;
    R *r, *q, *wr, *p, *t, *g, *x;
    double* parts;
    Dot *pp, *qq, *step;
    unsigned gd;      // blocks of the data-size kernels
    dim3 gm;          // blocks of the model-size kernels
    bool vec;
    Loop(const grav_plan* plan, int iters, void* work) : k(work_of(plan, iters)) {
        unsigned char* b = (unsigned char*)work + Work::kHead;
        status = (int*)work;
        auto take = [&](size_t n) {
            R* v = (R*)b;
            b += n;
            return v;
        };
        r = take(k.data), q = take(k.data), wr = take(k.data);
        p = take(k.model), t = take(k.model), g = take(k.model), x = take(k.model);
        parts = (double*)b;
        pp = (Dot*)(b + 2 * Work::kParts);
        qq = pp + 1;
        step = pp + 2;
        gd = (unsigned)std::min<size_t>((k.nd + kVecThreads - 1) / kVecThreads, kMaxParts / 2);
        constexpr int V = 16 / sizeof(R);
        vec = k.plane % V == 0;
        const unsigned gy = (unsigned)std::min(k.nz, kMaxParts);
        const size_t per = (size_t)kVecThreads * (vec ? V : 1);
        const unsigned gx = (unsigned)std::min<size_t>((k.plane + per - 1) / per, kMaxParts / gy);
        gm = dim3(gx, gy);
    }
    Making first(Dot* d) const { return {d, parts}; }
    Making second(Dot* d) const { return {d, parts + kMaxParts}; }
    Dot* rr(int it) const { return step + (size_t)3 * it; }
    Dot* xx(int it) const { return rr(it) + 1; }
    Dot* ss(int it) const { return rr(it) + 2; }
};

// Where the steps leave models: one buffer per step (host array of device
// pointers), the steps' models in one block, or the last step's model only.
template <typename R> struct Models {
    void* const* each;
    R *block, *last;
};

template <typename R>
int run_start(grav_plan* plan, const R* d, const R* w, const R* wm, int iters, void* work, cudaStream_t s) {
    const Loop<R> L(plan, iters, work);
    constexpr int V = 16 / sizeof(R);
    cudaError_t e = cudaMemsetAsync(L.pp, 0, L.k.dots() * sizeof(Dot), s);  // no block done yet
    if (e != cudaSuccess) return cuda_fail(e, "grav_cgls_start");
    cgls_first_data<R><<<L.gd, kVecThreads, 0, s>>>(d, w, L.r, L.wr, L.k.nd, L.first(L.rr(0)), L.status);
    const int rc = grav_adjoint(plan, L.wr, L.g, s);
    if (rc != GRAV_OK) return rc;
    if (L.vec) cgls_first_model<R, V><<<L.gm, kVecThreads, 0, s>>>(wm, L.g, L.p, L.t, L.k.plane, L.k.nz, L.first(L.ss(0)), L.second(L.pp));
    else cgls_first_model<R, 1><<<L.gm, kVecThreads, 0, s>>>(wm, L.g, L.p, L.t, L.k.plane, L.k.nz, L.first(L.ss(0)), L.second(L.pp));
    e = cudaGetLastError();
    return e == cudaSuccess ? GRAV_OK : cuda_fail(e, "grav_cgls_start");
}

template <typename R>
int run_steps(grav_plan* plan, const R* w, const R* wm, double lam, int iters, const Models<R>& models, double* obj,
              void* work, cudaStream_t s) {
    const Loop<R> L(plan, iters, work);
    constexpr int V = 16 / sizeof(R);
    const size_t cells = L.k.plane * L.k.nz;
    if (iters == 0 && models.last) {
        const cudaError_t e = cudaMemsetAsync(models.last, 0, cells * sizeof(R), s);
        if (e != cudaSuccess) return cuda_fail(e, "grav_cgls_steps");
    }
    for (int it = 0; it < iters; ++it) {
        int rc = grav_forward(plan, L.t, L.q, s);
        if (rc != GRAV_OK) return rc;
        cgls_weigh<R><<<L.gd, kVecThreads, 0, s>>>(w, L.q, L.k.nd, L.first(L.qq));
        const Scalars k{L.ss(it), L.pp, L.qq, lam, L.status};
        cgls_step_data<R><<<L.gd, kVecThreads, 0, s>>>(k, w, L.q, L.r, L.wr, L.k.nd, L.first(L.rr(it + 1)));
        rc = grav_adjoint(plan, L.wr, L.g, s);
        if (rc != GRAV_OK) return rc;
        R* m = models.each ? (R*)models.each[it] : models.block ? models.block + it * cells : it + 1 == iters ? models.last : nullptr;
        if (L.vec) cgls_step_model<R, V><<<L.gm, kVecThreads, 0, s>>>(k, it == 0, wm, L.p, L.x, L.g, m, L.k.plane, L.k.nz, L.first(L.ss(it + 1)), L.second(L.xx(it + 1)));
        else cgls_step_model<R, 1><<<L.gm, kVecThreads, 0, s>>>(k, it == 0, wm, L.p, L.x, L.g, m, L.k.plane, L.k.nz, L.first(L.ss(it + 1)), L.second(L.xx(it + 1)));
        if (it + 1 < iters) {
            if (L.vec) cgls_next_dir<R, V><<<L.gm, kVecThreads, 0, s>>>(L.ss(it), L.ss(it + 1), wm, L.g, L.p, L.t, L.k.plane, L.k.nz, L.first(L.pp));
            else cgls_next_dir<R, 1><<<L.gm, kVecThreads, 0, s>>>(L.ss(it), L.ss(it + 1), wm, L.g, L.p, L.t, L.k.plane, L.k.nz, L.first(L.pp));
        }
    }
    cgls_objectives<<<1, kVecThreads, 0, s>>>(L.step, iters + 1, lam, obj);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GRAV_OK : cuda_fail(e, "grav_cgls_steps");
}

int check_cgls(const grav_plan* plan, bool pointers, int iters, const void* work, const char* name) {
    if (!plan || !pointers || !work || iters < 0) {
        set_error("%s: null plan or buffer, or a negative number of steps", name);
        return GRAV_EINVAL;
    }
    if (plan->kind != 0) {
        set_error("%s: the plan was made by grav_plan_create3d", name);
        return GRAV_EINVAL;
    }
    if (reinterpret_cast<uintptr_t>(work) & 255) {
        set_error("%s: workspace must be 256-byte aligned", name);
        return GRAV_EINVAL;
    }
    return GRAV_OK;
}

int steps(grav_plan* plan, const void* w, const void* wm, double lam, int iters, void* const* each, void* block,
          void* last, double* obj, void* work, cudaStream_t s, const char* name) {
    uintptr_t bits = reinterpret_cast<uintptr_t>(block) | reinterpret_cast<uintptr_t>(last);
    for (int it = 0; each && it < iters; ++it) {
        if (!each[it]) {
            set_error("%s: null model buffer", name);
            return GRAV_EINVAL;
        }
        bits |= reinterpret_cast<uintptr_t>(each[it]);
    }
    if (bits & 15) {
        set_error("%s: models must be 16-byte aligned", name);
        return GRAV_EINVAL;
    }
    if (plan->fp64)
        return run_steps<double>(plan, (const double*)w, (const double*)wm, lam, iters,
                                 Models<double>{each, (double*)block, (double*)last}, obj, work, s);
    return run_steps<float>(plan, (const float*)w, (const float*)wm, lam, iters,
                            Models<float>{each, (float*)block, (float*)last}, obj, work, s);
}

}  // namespace

}  // namespace grav

using namespace grav;

extern "C" {

size_t grav_cgls_work_bytes(const grav_plan* plan, int iters) {
    return plan && plan->kind == 0 && iters >= 0 ? work_of(plan, iters).bytes() : 0;
}

int grav_cgls_start(grav_plan* plan, const void* d_dev, const void* w_dev, const void* wm_dev, int iters, void* work_dev,
                    void* stream) {
    const int rc = check_cgls(plan, d_dev && w_dev && wm_dev, iters, work_dev, "grav_cgls_start");
    if (rc != GRAV_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    return plan->fp64 ? run_start<double>(plan, (const double*)d_dev, (const double*)w_dev, (const double*)wm_dev, iters, work_dev, s)
                      : run_start<float>(plan, (const float*)d_dev, (const float*)w_dev, (const float*)wm_dev, iters, work_dev, s);
}

int grav_cgls_steps(grav_plan* plan, const void* w_dev, const void* wm_dev, double lam, int iters, int keep_models,
                    void* models_dev, double* objectives_dev, void* work_dev, void* stream) {
    const int rc = check_cgls(plan, w_dev && wm_dev && objectives_dev && (models_dev || (keep_models && iters == 0)), iters,
                              work_dev, "grav_cgls_steps");
    if (rc != GRAV_OK) return rc;
    return steps(plan, w_dev, wm_dev, lam, iters, nullptr, keep_models ? models_dev : nullptr,
                 keep_models ? nullptr : models_dev, objectives_dev, work_dev, (cudaStream_t)stream, "grav_cgls_steps");
}

int grav_cgls_steps_kept(grav_plan* plan, const void* w_dev, const void* wm_dev, double lam, int iters,
                         void* const* models_dev, double* objectives_dev, void* work_dev, void* stream) {
    const int rc = check_cgls(plan, w_dev && wm_dev && objectives_dev && (models_dev || iters == 0), iters, work_dev,
                              "grav_cgls_steps_kept");
    if (rc != GRAV_OK) return rc;
    return steps(plan, w_dev, wm_dev, lam, iters, models_dev, nullptr, nullptr, objectives_dev, work_dev,
                 (cudaStream_t)stream, "grav_cgls_steps_kept");
}

}  // extern "C"
