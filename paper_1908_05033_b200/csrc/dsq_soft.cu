// Training-side elementwise kernels of DSQ: the soft quantiser Q_S (Eq. 3-8)
// and its back-propagation (Eq. 10-13, Algorithm 1).  HBM-bound streaming
// kernels: 8 bytes per element forward (fp32 in, fp32 out), 12 bytes per
// element backward (x and dL/dy in, dL/dx out) plus three scalar reductions.
#include "dsq_common.cuh"
#include "dsq_launch.h"
#include "dsq_ptx.cuh"

using dsq_ptx::grid_dependency_wait;
using dsq_ptx::grid_launch_dependents;

namespace {

// Everything that depends on (b, l, u, alpha) only, formed on the host in
// binary64 and rounded once to binary32.
struct SoftP {
    float lo, hi, delta, inv_delta, k, s;
    float half_ds;        // Delta/2 * s
    float half_dsk;       // Delta/2 * s * k
    float half_s;         // s / 2
    float da_t, da_x;     // Delta/2 ds/dalpha, Delta/2 s dk/dalpha
    double inv_n;         // 1/(2^b-1)
    float imax;           // 2^b - 2
};

// eight consecutive values, used once (32-byte aligned)
struct V8 { float v[8]; };
__device__ __forceinline__ V8 ld_stream(const float *p)
{
    V8 r;
    asm volatile("ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]),
                   "=f"(r.v[6]), "=f"(r.v[7])
                 : "l"(p));
    return r;
}
__device__ __forceinline__ void st_stream(float *p, const V8 &r)
{
    asm volatile("st.global.L1::no_allocate.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p),
                 "f"(r.v[0]), "f"(r.v[1]), "f"(r.v[2]), "f"(r.v[3]), "f"(r.v[4]), "f"(r.v[5]),
                 "f"(r.v[6]), "f"(r.v[7])
                 : "memory");
}

// interval index i, tanh(k (x - m_i)) and x - m_i of a value inside [l, u]
__device__ __forceinline__ void soft_core(float x, const SoftP &p, float &fi, float &t, float &xm)
{
    const float xc = fminf(fmaxf(x, p.lo), p.hi);
    fi = fminf(fmaxf(floorf((xc - p.lo) * p.inv_delta), 0.0f), p.imax);
    const float m = fmaf(fi + 0.5f, p.delta, p.lo);
    xm = xc - m;
    t = tanhf(p.k * xm);
}

__device__ __forceinline__ float soft_fwd_one(float x, const SoftP &p)
{
    float fi, t, xm;
    soft_core(x, p, fi, t, xm);
    // l + Delta (i + (phi + 1)/2) = l + Delta i + Delta/2 + (Delta/2) s tanh
    float y = fmaf(p.half_ds, t, fmaf(fi + 0.5f, p.delta, p.lo));
    y = x < p.lo ? p.lo : y;
    y = x > p.hi ? p.hi : y;
    return x != x ? x : y;        // NaN stays NaN
}

// Both kernels are bound by memory (8 and 12 bytes an element).  Eight elements a thread
// in 32-byte accesses keep twice the bytes in flight of 16-byte ones; forward at 12.8M
// elements 19.9 -> 18.0 us.  What the vector loop leaves: `head` elements in front of the
// first 32-byte boundary that the arrays share (they are 16-byte aligned: 0 or 4; all
// elements when they share none), and what is behind the last group of eight.
__global__ void __launch_bounds__(256) soft_fwd_kernel(const float *__restrict__ x,
                                                       float *__restrict__ y, int64_t n,
                                                       int64_t head, SoftP p)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const int64_t n8 = (n - head) >> 3;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = tid; i < n8; i += stride) {
        const V8 v = ld_stream(x + head + 8 * i);
        V8 o;
#pragma unroll
        for (int k = 0; k < 8; ++k) o.v[k] = soft_fwd_one(v.v[k], p);
        st_stream(y + head + 8 * i, o);
    }
    const int64_t rest = n - 8 * n8;
    for (int64_t i = tid; i < rest; i += stride) {
        const int64_t at = i < head ? i : i + 8 * n8;
        y[at] = soft_fwd_one(x[at], p);
    }
}

// tanh(z) and sech^2(z) from one exponential and one reciprocal (the special
// function unit's ex2 and rcp, each good to about 2^-22 relative):
//   e = exp(2 z), r = 1/(e + 1):  tanh = 1 - 2 r,  sech^2 = 4 e r^2
// sech^2 has no cancellation (relative error ~1e-6); tanh is good to ~1e-6
// absolute, and it only enters sums next to terms of order one.  z -> +inf:
// e = inf, r = 0, tanh = 1 and sech^2 is forced to 0; z -> -inf: e = 0.
__device__ __forceinline__ void tanh_sech2(float z, float &t, float &sech2)
{
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(z * 2.885390081777927f));   // 2 log2(e)
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(e + 1.0f));
    t = fmaf(-2.0f, r, 1.0f);
    sech2 = r == 0.0f ? 0.0f : 4.0f * e * r * r;
}

// One element of the backward pass: returns dL/dx and adds the element's terms
// (binary32 partial sums of four elements; the caller folds them into binary64).
// With v = (x - l)/Delta, q = i + (phi + 1)/2 (Eq. 13) and dx = dQ/dx inside [l, u]:
//   dQ/du = (q - dx v) / n            (Eq. 12; n = 2^b - 1)
//   dQ/dl = 1 - dx - dQ/du            (Eq. 11; a shift of x, l and u together moves Q
//                                      by the same amount)
//   dQ/dalpha = Delta/2 (ds/da tanh + s dk/da sech^2 (x - m))     (Eq. 10)
// so the three sums are made of sum g da, sum g (q - dx v), sum dL/dx, and the sums of
// g up to u and above it: fewer operations than adding the three derivatives, and no
// branches (a warp used to take all three of below, inside and above).
struct SoftSums { float a, u, in, x, above; };
__device__ __forceinline__ float soft_bwd_one(float x, float g, const SoftP &p, SoftSums &s)
{
    const bool inside = x >= p.lo && x <= p.hi;
    const float xc = inside ? x : p.lo, gi = inside ? g : 0.0f;
    const float v = (xc - p.lo) * p.inv_delta;
    // floor by the 2^23 trick (0 <= v <= 2^8)
    const float fi = fminf(__fsub_rn(__fadd_rd(v, 8388608.0f), 8388608.0f), p.imax) + 0.5f;
    const float xm = xc - fmaf(fi, p.delta, p.lo);
    float t, sech2;
    tanh_sech2(p.k * xm, t, sech2);
    const float dx = p.half_dsk * sech2;
    const float gx = gi * dx;
    s.a = fmaf(gi, fmaf(p.da_t, t, p.da_x * (sech2 * xm)), s.a);
    s.u = fmaf(gi, fmaf(-dx, v, fmaf(p.half_s, t, fi)), s.u);
    s.x += gx;
    s.in += x <= p.hi ? g : 0.0f;                  // inside and below
    s.above += x > p.hi ? g : 0.0f;
    return x != x ? x : gx;
}

// Calls of fewer elements have their sums cleared by a memset, outside graphs: the GPU is through
// with them before the host has enqueued the next, so that the launch that costs the host least is the
// better one.  Forward and backward one after the other, memset / kernel, us: 21758 elements 10.4 / 11.3,
// 600000 10.7 / 11.3, 1000000 12.2 / 11.4 (with the hosts of these GPUs; a slower one moves the line up).
constexpr int64_t SOFT_SMALL = 3 << 18;

// Clears the three sums.  The backward kernel, launched dependently behind it, starts when
// everything ahead of this one has completed (it waits for that before it lets the next one start) and
// waits for it only before it adds to the sums: until then it reads x and dL/dy and writes dL/dx.
// With a memset in front, 16384 / 1M / 12.8M elements took 6.2 / 7.7 / 29.2 us in a graph, so 2.7 / 4.5 / 26.7
// (forward and backward 8.4 / 10.7 / 48.8 -> 4.3 / 7.0 / 44.4).
__global__ void soft_clear_kernel(double *sums)
{
    grid_dependency_wait();
    grid_launch_dependents();
    if (threadIdx.x < 3) sums[threadIdx.x] = 0.0;
}

// 12.8M elements 41.9 -> 28.9 us, 67M 182 -> 126 us (the sums' binary64 additions and the
// conversions in front of them run beside the loads).
__global__ void __launch_bounds__(256) soft_bwd_kernel(const float *__restrict__ x,
                                                       const float *__restrict__ gy,
                                                       float *__restrict__ gx, int64_t n,
                                                       int64_t head, SoftP p,
                                                       double *__restrict__ sums)
{
    double da = 0.0, du = 0.0, din = 0.0, dx = 0.0, dab = 0.0;
    auto fold = [&](const SoftSums &s) {
        da += (double)s.a;
        du += (double)s.u;
        din += (double)s.in;
        dx += (double)s.x;
        dab += (double)s.above;
    };
    const int64_t n8 = (n - head) >> 3;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = tid; i < n8; i += stride) {
        const V8 v = ld_stream(x + head + 8 * i), g = ld_stream(gy + head + 8 * i);
        V8 o;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            SoftSums s = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int k = 4 * h; k < 4 * h + 4; ++k) o.v[k] = soft_bwd_one(v.v[k], g.v[k], p, s);
            fold(s);
        }
        st_stream(gx + head + 8 * i, o);
    }
    const int64_t rest = n - 8 * n8;
    for (int64_t i = tid; i < rest; i += stride) {
        const int64_t at = i < head ? i : i + 8 * n8;
        SoftSums s = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        gx[at] = soft_bwd_one(x[at], gy[at], p, s);
        fold(s);
    }
    double aa = da, au = du * p.inv_n, al = (din - dx) - au;
    au += dab;
    // the three sums: warp shuffles, one shared-memory pass per block, one
    // double-precision atomic add per block and sum
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        aa += __shfl_xor_sync(0xffffffffu, aa, o);
        al += __shfl_xor_sync(0xffffffffu, al, o);
        au += __shfl_xor_sync(0xffffffffu, au, o);
    }
    __shared__ double part[3][8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { part[0][warp] = aa; part[1][warp] = al; part[2][warp] = au; }
    grid_dependency_wait();                        // the sums are clear
    grid_launch_dependents();
    __syncthreads();
    if (threadIdx.x < 3) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += part[threadIdx.x][w];
        atomicAdd(sums + threadIdx.x, s);
    }
}

int make_soft_params(const dsq_quant_t *q, float alpha, SoftP *out)
{
    if (!q) return DSQ_ERR_NULL;
    if (q->bits < 1 || q->bits > 8) return DSQ_ERR_BITS;
    if (!dsq_finite(q->lo) || !dsq_finite(q->hi) || !(q->hi > q->lo)) return DSQ_ERR_RANGE;
    if (!(alpha > 0.0f && alpha < 1.0f)) return DSQ_ERR_RANGE;
    const double lo = q->lo, hi = q->hi, a = alpha;
    const double n = (double)((1 << q->bits) - 1);
    const double delta = (hi - lo) / n;
    const double k = log(2.0 / a - 1.0) / delta;          // Eq. 8
    const double s = 1.0 / (1.0 - a);                     // Eq. 7
    SoftP p;
    p.lo = q->lo; p.hi = q->hi;
    p.delta = (float)delta; p.inv_delta = (float)(1.0 / delta);
    p.k = (float)k; p.s = (float)s;
    p.half_ds = (float)(0.5 * delta * s);
    p.half_dsk = (float)(0.5 * delta * s * k);
    p.half_s = (float)(0.5 * s);
    p.da_t = (float)(0.5 * delta / ((1.0 - a) * (1.0 - a)));        // ds/dalpha = 1/(1-alpha)^2
    p.da_x = (float)(-s / (a * (2.0 - a)));                          // dk/dalpha = -2/(Delta alpha (2-alpha))
    p.inv_n = 1.0 / n;
    p.imax = (float)((1 << q->bits) - 2);
    *out = p;
    return DSQ_OK;
}

// Blocks per SM: whole sets of all that are resident together (forward 8, backward 4: 32 and
// 57 registers a thread), since every block walks the array at the same step and the last set
// should not be a partial one.  Backward, us after an L2 flush with 3 / 4 / 5 / 6 / 8 / 16 blocks:
// 12.8M elements 36.9 / 32.8 / 41.0 / 37.0 / 34.8 / 36.0, 33.5M 77.8 / 71.7 / 88.0 / 81.9 / 72.7 / 73.8, 67M
// 141 / 133 / 160 / 146 / 133 / 133; below 4M the counts do not differ.  Forward with 4 / 8 / 16 / 32:
// 12.8M 26.6 / 24.6 / 22.6 / 24.6, 67M 102 / 100 / 96 / 88.
int soft_grid(int64_t n, int per_sm)
{
    const int sms = dsq_sm_count() > 0 ? dsq_sm_count() : 148;
    int64_t g = (n / 8 + 255) / 256;
    if (g > (int64_t)sms * per_sm) g = (int64_t)sms * per_sm;
    return g < 1 ? 1 : (int)g;
}

// elements in front of the arrays' common 32-byte boundary (n: they have none)
int64_t soft_head(const void *a, const void *b, const void *c, int64_t n)
{
    const uintptr_t x = (uintptr_t)a & 31u;
    if (((uintptr_t)b & 31u) != x || ((uintptr_t)c & 31u) != x) return n;
    const int64_t head = x ? 4 : 0;
    return head < n ? head : n;
}

}  // namespace

extern "C" int dsq_soft_quantize_fwd(const float *x, int64_t n, const dsq_quant_t *q, float alpha,
                                     float *y, void *stream)
{
    if (!x || !y) return DSQ_ERR_NULL;
    SoftP p;
    const int st = make_soft_params(q, alpha, &p);
    if (st) return st;
    if (n <= 0) return DSQ_ERR_SHAPE;
    if (!dsq_aligned16(x) || !dsq_aligned16(y)) return DSQ_ERR_ALIGN;
    return dsq_launch(soft_fwd_kernel, dim3(soft_grid(n, 16)), dim3(256), 0, (cudaStream_t)stream,
                      dsq_launch_hooks().pdl, 0, x, y, n, soft_head(x, y, y, n), p);
}

extern "C" int dsq_soft_quantize_bwd(const float *x, const float *grad_y, int64_t n,
                                     const dsq_quant_t *q, float alpha, float *grad_x,
                                     double *grad_params, void *stream)
{
    if (!x || !grad_y || !grad_x || !grad_params) return DSQ_ERR_NULL;
    SoftP p;
    const int st = make_soft_params(q, alpha, &p);
    if (st) return st;
    if (n <= 0) return DSQ_ERR_SHAPE;
    if (!dsq_aligned16(x) || !dsq_aligned16(grad_y) || !dsq_aligned16(grad_x) ||
        (reinterpret_cast<uintptr_t>(grad_params) & 7u))
        return DSQ_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    const int pdl = dsq_launch_hooks().pdl;
    // (a memset takes 0.7 us less of the host than a launch; in a graph the host does not matter)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (n < SOFT_SMALL && !dsq_recording_plan() && cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
        DSQ_CUDA_TRY(cudaMemsetAsync(grad_params, 0, 3 * sizeof(double), s));
    } else {
        const int st2 = dsq_launch(soft_clear_kernel, dim3(1), dim3(32), 0, s, pdl, 0, grad_params);
        if (st2) return st2;
    }
    return dsq_launch(soft_bwd_kernel, dim3(soft_grid(n, 4)), dim3(256), 0, s, pdl, 0, x, grad_y, grad_x,
                      n, soft_head(x, grad_y, grad_x, n), p, grad_params);
}
