// Small kernels around the time loop: receiver sampling, residual and FP64
// misfit (Sec. 6: phi = 1/2 ||d_sim - d_obs||^2), model setup (m = 1/c^2 ->
// w = dt^2 c^2), gradient output and checkpoint up-casts.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace ckfwi {

namespace {

__global__ void sample_kernel(const float* __restrict__ u, Sample smp)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= smp.n) return;
    float acc = 0.0f;
    for (int i = 0; i < smp.nst; ++i)
        acc = __fmaf_rn(smp.wt[r * smp.nst + i], __ldg(u + smp.idx[r * smp.nst + i]), acc);
    smp.out[r] = acc;
}

constexpr int RED_THREADS = 256;

// r = d - dobs for rows 1..rows-1 (row 0 zero); per-CTA FP64 partial sums
// of r^2 over a fixed contiguous range, reduced by a fixed tree.
__global__ void residual_kernel(const float* __restrict__ d, const float* __restrict__ dobs,
                                float* __restrict__ r, long long n, long long first,
                                double* __restrict__ partials, long long per_cta)
{
    __shared__ double sh[RED_THREADS];
    const long long lo = (long long)blockIdx.x * per_cta;
    const long long hi = min(lo + per_cta, n);
    double acc = 0.0;
    // eight values' loads in flight; the sum keeps its order
    for (long long i0 = lo + threadIdx.x; i0 < hi; i0 += 8 * RED_THREADS) {
        float a[8], b[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const long long i = i0 + k * RED_THREADS;
            const bool on = i < hi && i >= first;
            a[k] = on ? d[i] : 0.0f;
            b[k] = on ? dobs[i] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const long long i = i0 + k * RED_THREADS;
            if (i >= hi) break;
            const double dv = (double)a[k] - (double)b[k];
            r[i] = (float)dv;
            acc += dv * dv;
        }
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

__global__ void final_sum_kernel(const double* __restrict__ partials, int n, double* phi)
{
    __shared__ double sh[RED_THREADS];
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += RED_THREADS) acc += partials[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s = RED_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *phi = 0.5 * sh[0];
}

// The dense <-> padded kernels below are streams of 12 - 40 B/pt.  A thread
// takes four consecutive points of a row: one division (32-bit where the grid
// allows it) finds the row of four points instead of two 64-bit ones for
// every point, and rows that start 16-byte aligned move as vectors.  (One
// point a thread, 64-bit divisions: 217 us for the medium of 208^3 and 2580 us
// for 300 x 600 x 600, 13 times the memory's time.)
struct Quad {
    bool on, vec;
    int n;               // points of the quad inside the row
    long long z, y, x0;
    long long dense;     // of its first point
};
__device__ __forceinline__ Quad quad_at(const FieldGeom& g, bool dense_aligned)
{
    Quad q;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned nvx = (unsigned)(g.nx + 3) / 4;
    const long long rows = (long long)g.nz * g.ny;
    q.on = t < rows * nvx;
    if (!q.on) return q;
    long long row;
    if (rows * nvx <= 0xffffffffLL) {
        row = (unsigned)t / nvx;
        q.z = (unsigned)row / (unsigned)g.ny;
    } else {
        row = t / nvx;
        q.z = row / g.ny;
    }
    q.x0 = 4 * (t - row * nvx);
    q.y = row - q.z * g.ny;
    q.n = (int)min(4LL, g.nx - q.x0);
    q.dense = row * g.nx + q.x0;
    q.vec = dense_aligned && q.n == 4;
    return q;
}
__device__ __forceinline__ void load4(float (&v)[4], const float* p, bool vec, int n)
{
    if (vec) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = i < n ? p[i] : 1.0f;
    }
}
__device__ __forceinline__ void store4(float* p, const float (&v)[4], bool vec, int n)
{
    if (vec) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < n) p[i] = v[i];
    }
}

// kind 0: velocity c, kind 1: m = 1/c^2.  w = dt^2 c^2 (FP64, rounded once);
// c_dense keeps c in float for the gradient output.  (The square of a float is
// exact in FP64 and its root is that float, so kind 0 needs no root.)
__global__ void model_kernel(const float* __restrict__ in, int kind, double dt2, FieldGeom g, bool aligned,
                             float* __restrict__ w, float* __restrict__ c_dense, int* err)
{
    const Quad q = quad_at(g, aligned);
    if (!q.on) return;
    float v[4], wv[4], cv[4];
    load4(v, in + q.dense, q.vec, q.n);
    int bad = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (!isfinite(v[i])) bad |= 2;
        else if (!(v[i] > 0.0f)) bad |= 1;
        const double c2 = (kind == 0) ? (double)v[i] * (double)v[i] : 1.0 / (double)v[i];
        wv[i] = (float)(dt2 * c2);
        cv[i] = kind == 0 ? v[i] : (float)sqrt(c2);
    }
    if (bad) atomicOr(err, bad);
    store4(w + q.z * g.pxy + q.y * g.px + q.x0, wv, q.n == 4, q.n);      // padded rows are aligned
    store4(c_dense + q.dense, cv, q.vec, q.n);
}

// dphi/dm = gacc c^2 ; dphi/dc = dphi/dm dm/dc = -2 gacc / c
__device__ __forceinline__ float grad_value(float ga, float c, int kind)
{
    return (kind == 1) ? __fmul_rn(ga, __fmul_rn(c, c)) : __fdiv_rn(__fmul_rn(-2.0f, ga), c);
}

__global__ void grad_out_kernel(const float* __restrict__ gacc, const float* __restrict__ c, int kind, float scale,
                                FieldGeom g, bool aligned, float* __restrict__ out)
{
    const Quad q = quad_at(g, aligned);
    if (!q.on) return;
    float ga[4], cv[4], r[4];
    load4(ga, gacc + q.z * g.pxy + q.y * g.px + q.x0, q.n == 4, q.n);
    load4(cv, c + q.dense, q.vec, q.n);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float v = grad_value(ga[i], cv[i], kind);
        r[i] = scale == 1.0f ? v : __fmul_rn(scale, v);
    }
    store4(out + q.dense, r, q.vec, q.n);
}

// Neumaier-compensated FP64 accumulation of one shot's gradient into a
// dense array that may be larger than the shot's grid: point (z, y, x) of
// the grid adds into q = o0 + z * gsz + y * gsy + x.
__global__ void grad_sum_kernel(const float* __restrict__ gacc, const float* __restrict__ c, int kind, FieldGeom g,
                                bool aligned, long long o0, long long gsy, long long gsz, double* __restrict__ sum,
                                double* __restrict__ comp)
{
    const Quad q = quad_at(g, aligned);
    if (!q.on) return;
    float ga[4], cv[4];
    load4(ga, gacc + q.z * g.pxy + q.y * g.px + q.x0, q.n == 4, q.n);
    load4(cv, c + q.dense, q.vec, q.n);
    const long long o = o0 + q.z * gsz + q.y * gsy + q.x0;
    double s[4], k[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        s[i] = i < q.n ? sum[o + i] : 0.0;
        k[i] = i < q.n ? comp[o + i] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i >= q.n) break;
        const double v = (double)grad_value(ga[i], cv[i], kind);
        const double t = s[i] + v;
        comp[o + i] = k[i] + ((fabs(s[i]) >= fabs(v)) ? (s[i] - t) + v : (v - t) + s[i]);
        sum[o + i] = t;
    }
}

// Up-cast of a checkpoint field into an FP32 working field: one thread per
// four consecutive x points of a row (one 8- or 16-byte load and one 16-byte
// store; rows start 16-byte aligned in both layouts), the ragged end of a
// row value by value.  Halo cells are not touched.
template <class T>
__device__ __forceinline__ float up1(T v);
template <> __device__ __forceinline__ float up1<float>(float v) { return v; }
template <> __device__ __forceinline__ float up1<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float up1<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <class T>
__global__ void upcast_kernel(const T* __restrict__ src, FieldGeom g, float* __restrict__ dst)
{
    const Quad q = quad_at(g, true);
    if (!q.on) return;
    const long long o = q.z * g.pxy + q.y * g.px + q.x0;
    if (q.n == 4) {
        float4 r;
        if constexpr (sizeof(T) == 4) {
            r = __ldg(reinterpret_cast<const float4*>(src + o));
        } else {
            const uint2 w = __ldg(reinterpret_cast<const uint2*>(src + o));
            const T* h = reinterpret_cast<const T*>(&w);
            r = make_float4(up1<T>(h[0]), up1<T>(h[1]), up1<T>(h[2]), up1<T>(h[3]));
        }
        *reinterpret_cast<float4*>(dst + o) = r;
    } else {
        for (int i = 0; i < q.n; ++i) dst[o + i] = up1<T>(src[o + i]);
    }
}

__global__ void copy_f64_kernel(const double* __restrict__ a, double* __restrict__ b, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = a[i];
}

__global__ void add_f64_kernel(const double* __restrict__ a, const double* __restrict__ b, double scale,
                               double* __restrict__ out, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = scale * (a[i] + b[i]);
}

__global__ void f64_to_f32_kernel(const double* __restrict__ a, float* __restrict__ out, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)a[i];
}

// max |u| over the total grid of a padded field (the wavefield's scale, for
// stating a codec tolerance relative to it): the cells outside the grid are
// zero, so whole padded planes are read, as vectors, four in flight a thread;
// the magnitudes' bit patterns order like the values, so one unsigned
// atomicMax per warp.  (Row by row, one value at a time: 28 us at 208^3.)
__global__ void absmax_kernel(const float4* __restrict__ u, long long n, unsigned* __restrict__ out)
{
    unsigned m = 0u;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += 4 * step) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = i0 + k * step < n ? __ldg(u + i0 + k * step) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            m = max(max(m, max(__float_as_uint(fabsf(v[k].x)), __float_as_uint(fabsf(v[k].y)))),
                    max(__float_as_uint(fabsf(v[k].z)), __float_as_uint(fabsf(v[k].w))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

inline unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }
// CTAs of 256 threads, a quad of a row each; whether dense rows start 16-byte
// aligned (the library's own dense arrays are allocations, hence aligned)
inline unsigned quad_blocks(const FieldGeom& g) { return blocks_for((long long)((g.nx + 3) / 4) * g.ny * g.nz, 256); }
inline bool dense_aligned(const FieldGeom& g, const void* p)
{
    return g.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

}  // namespace

cudaError_t launch_sample(const float* u, const Sample& smp, cudaStream_t s)
{
    if (smp.n <= 0) return cudaSuccess;
    sample_kernel<<<blocks_for(smp.n, 128), 128, 0, s>>>(u, smp);
    return cudaGetLastError();
}

cudaError_t launch_absmax(const float* u_origin, const FieldGeom& g, unsigned* out, cudaStream_t s)
{
    // the grid's planes, from the start of the first one's first (padded) row:
    // 128-byte aligned rows of a multiple of 32 values
    const float* base = u_origin - g.X0;
    const long long n = ((long long)(g.nz - 1) * g.pxy + (long long)g.ny * g.px) / 4;
    const unsigned nb = (unsigned)std::min<long long>((n + 1023) / 1024, 8LL * 152);
    absmax_kernel<<<nb, 256, 0, s>>>(reinterpret_cast<const float4*>(base), n, out);
    return cudaGetLastError();
}

cudaError_t launch_residual(const float* d, const float* dobs, float* r, int rows, int nrec,
                            double* partials, int nparts, double* phi, cudaStream_t s)
{
    const long long n = (long long)rows * nrec;
    const long long per = (n + nparts - 1) / nparts;
    residual_kernel<<<nparts, RED_THREADS, 0, s>>>(d, dobs, r, n, (long long)nrec, partials, per);
    final_sum_kernel<<<1, RED_THREADS, 0, s>>>(partials, nparts, phi);
    return cudaGetLastError();
}

cudaError_t launch_to_padded_w(const float* dense, int kind, float dt, const FieldGeom& g,
                               float* w_origin, float* c_dense, int* err, cudaStream_t s)
{
    model_kernel<<<quad_blocks(g), 256, 0, s>>>(dense, kind, (double)dt * (double)dt, g, dense_aligned(g, dense),
                                                w_origin, c_dense, err);
    return cudaGetLastError();
}

cudaError_t launch_grad_out(const float* gacc_origin, const float* c_dense, int kind, float scale,
                            const FieldGeom& g, float* out_dense, cudaStream_t s)
{
    grad_out_kernel<<<quad_blocks(g), 256, 0, s>>>(gacc_origin, c_dense, kind, scale, g, dense_aligned(g, out_dense),
                                                   out_dense);
    return cudaGetLastError();
}

cudaError_t launch_grad_out_f64(const float* gacc_origin, const float* c_dense, int kind,
                                const FieldGeom& g, long long o0, long long gsy, long long gsz,
                                double* sum, double* comp, cudaStream_t s)
{
    grad_sum_kernel<<<quad_blocks(g), 256, 0, s>>>(gacc_origin, c_dense, kind, g, dense_aligned(g, c_dense), o0, gsy, gsz,
                                                   sum, comp);
    return cudaGetLastError();
}

cudaError_t launch_cast_restore(const void* src, int utype, const FieldGeom& g, float* dst_origin,
                                cudaStream_t s)
{
    const unsigned nb = blocks_for((long long)((g.nx + 3) / 4) * g.ny * g.nz, 256);
    if (utype == U_BF16)
        upcast_kernel<__nv_bfloat16><<<nb, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(src), g, dst_origin);
    else if (utype == U_FP16)
        upcast_kernel<__half><<<nb, 256, 0, s>>>(static_cast<const __half*>(src), g, dst_origin);
    else
        upcast_kernel<float><<<nb, 256, 0, s>>>(static_cast<const float*>(src), g, dst_origin);
    return cudaGetLastError();
}

cudaError_t launch_copy_f64(const double* a, double* b, long long n, cudaStream_t s)
{
    copy_f64_kernel<<<blocks_for(n, 256), 256, 0, s>>>(a, b, n);
    return cudaGetLastError();
}

}  // namespace ckfwi

namespace ckfwi {
cudaError_t launch_add_f64(const double* a, const double* b, double scale, double* out, long long n, cudaStream_t s)
{
    add_f64_kernel<<<blocks_for(n, 256), 256, 0, s>>>(a, b, scale, out, n);
    return cudaGetLastError();
}

cudaError_t launch_f64_to_f32(const double* a, float* out, long long n, cudaStream_t s)
{
    f64_to_f32_kernel<<<blocks_for(n, 256), 256, 0, s>>>(a, out, n);
    return cudaGetLastError();
}
}  // namespace ckfwi
