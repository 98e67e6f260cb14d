// tt_reg.cu -- regularisers of the loss (Section "Optimization": L2Norm and
// TotalVariation, the Huber norm of the spatial gradient of every basis mode)
// on a volume c [nx][ny][nz][K], with FP64 value reduction.
#include <cmath>

#include "tt_kernels.cuh"

namespace tt {

// Four elements as 16-byte accesses (two for double), and their number.
__device__ __forceinline__ void reg_load(const float *p, float (&v)[4])
{
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void reg_load(const double *p, double (&v)[4])
{
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p)), b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void reg_store(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void reg_store(double *p, const double (&v)[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}

// Sum of a value per element: compensated FP32 per thread and across the CTA
// for float, FP64 for double.
template <typename T>
struct RegSum {
    Dot2 a = {0.f, 0.f};
    double v = 0.0;
    __device__ __forceinline__ void add(T x)
    {
        if constexpr (std::is_same<T, float>::value) dot2_add1(a, x);
        else v += x;
    }
    __device__ __forceinline__ void square(T x)
    {
        if constexpr (std::is_same<T, float>::value) dot2_add(a, x, x);
        else v = fma(x, x, v);
    }
    __device__ __forceinline__ double total(double *red) const
    {
        if constexpr (std::is_same<T, float>::value) return dot2_block_sum(a, reinterpret_cast<Dot2 *>(red));
        else return block_sum(v, red);
    }
};

// value = sum c^2, grad = 2 c.  Grid-stride over quads (the entry points take
// 16-byte aligned c and grad only), the last n % 4 elements by themselves;
// per-block FP64 partials.  Bound by its reads and writes (100^3, 28 channels:
// 86 -> 80 us in the whole call), in FP64 by its arithmetic, so the value alone
// has a kernel without the gradient's products (100^3, 45 channels: 197 -> 107 us).
template <typename T, bool GRAD>
__global__ void k_l2(const T *__restrict__ c, long long n, T *__restrict__ grad, double *__restrict__ partials)
{
    __shared__ double red[32];
    RegSum<T> sum;
    const long long n4 = n / 4, stride = (long long)gridDim.x * blockDim.x;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
#pragma unroll 4
    for (long long q = t0; q < n4; q += stride) {
        T x[4];
        reg_load(c + 4 * q, x);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sum.square(x[k]);
            if (GRAD) x[k] *= T(2);
        }
        if (GRAD) reg_store(grad + 4 * q, x);
    }
    for (long long i = 4 * n4 + t0; i < n; i += stride) {
        const T x = c[i];
        sum.square(x);
        if (GRAD) grad[i] = T(2) * x;
    }
    const double v = sum.total(red);
    if (threadIdx.x == 0) partials[blockIdx.x] = v;
}

// Huber total variation of every channel i:
//   g_i(x)_d = c_i(x + e_d) - c_i(x) if x_d + 1 < N_d else 0,  t = |g_i(x)|,
//   value = sum H(t), H(t) = t^2/(2 delta) (t <= delta) or t - delta/2,
//   grad_i(y) = sum_{d: y_d >= 1} w(y - e_d) g_i(y - e_d)_d - w(y) sum_d g_i(y)_d,
//   w = H'(t)/t = 1/delta (t <= delta) or 1/t.
template <typename T>
__device__ __forceinline__ void tv_point(T g0, T g1, T g2, T inv_delta, T delta, T &w, T &H)
{
    const T t = sqrt(g0 * g0 + g1 * g1 + g2 * g2);
    if (t <= delta) {
        w = inv_delta;
        H = T(0.5) * t * t * inv_delta;
    } else {
        w = T(1) / t;
        H = t - T(0.5) * delta;
    }
}

// A thread walks x through a run of up to kTvRun planes for one (y, z, channel); the
// plane behind it stays in registers, so an element takes seven loads and three
// weights (its own and its y and z predecessors') where taking every weight by
// itself took sixteen and four, with three index divisions.  An item is a run
// of 256 consecutive (y, z, channel) of a plane: all loads are contiguous.
// 100^3, 28 channels: 460 -> 279 us in the whole call (c read and grad written
// once: 33).
constexpr int kTvRun = 10;
template <typename T, bool GRAD>
__global__ void __launch_bounds__(256)
k_tv_huber(const T *__restrict__ c, int nx, int ny, int nz, int K, int run_len, T delta, T *__restrict__ grad,
           double *__restrict__ partials)
{
    __shared__ double red[32];
    const T inv_delta = T(1) / delta;
    const int row = nz * K;
    const long long plane = (long long)ny * row, segs = (plane + 255) / 256;
    const long long items = segs * ((nx + run_len - 1) / run_len);
    RegSum<T> sum;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const int run = (int)(it / segs);
        const long long e = (it - run * segs) * 256 + threadIdx.x;
        if (e >= plane) continue;
        const int y = (int)(e / row), zk = (int)(e - (long long)y * row);
        const bool y0 = y >= 1, y1 = y + 1 < ny, z0 = zk >= K, z1 = zk + K < row;
        const int x0 = run * run_len, x1 = min(nx, x0 + run_len);
        const T *p = c + x0 * plane + e;
        T cc = __ldg(p), cy = GRAD && y0 ? __ldg(p - row) : T(0), cz = GRAD && z0 ? __ldg(p - K) : T(0);   // here, y - 1, z - 1
        T back = T(0);                                     // w g_x of the plane behind
        if (GRAD && x0 > 0) {
            const T *q = p - plane;
            const T b = __ldg(q);
            T w, H;
            tv_point<T>(cc - b, y1 ? __ldg(q + row) - b : T(0), z1 ? __ldg(q + K) - b : T(0), inv_delta, delta, w, H);
            back = w * (cc - b);
        }
        for (int x = x0; x < x1; ++x, p += plane) {
            const bool on = x + 1 < nx;
            const T nc = on ? __ldg(p + plane) : T(0);
            const T py = y1 ? __ldg(p + row) : T(0), pz = z1 ? __ldg(p + K) : T(0);
            const T gx = on ? nc - cc : T(0), gy = y1 ? py - cc : T(0), gz = z1 ? pz - cc : T(0);
            T w, H;
            tv_point<T>(gx, gy, gz, inv_delta, delta, w, H);
            sum.add(H);
            if (GRAD) {
                T gr = -w * (gx + gy + gz) + back;
                back = w * gx;
                T wm, Hm;
                if (y0) {
                    const T ny1 = on ? __ldg(p + plane - row) : T(0);
                    tv_point<T>(on ? ny1 - cy : T(0), cc - cy, z1 ? __ldg(p - row + K) - cy : T(0), inv_delta, delta, wm, Hm);
                    gr += wm * (cc - cy);
                    cy = ny1;
                }
                if (z0) {
                    const T nz1 = on ? __ldg(p + plane - K) : T(0);
                    tv_point<T>(on ? nz1 - cz : T(0), y1 ? __ldg(p + row - K) - cz : T(0), cc - cz, inv_delta, delta, wm, Hm);
                    gr += wm * (cc - cz);
                    cz = nz1;
                }
                grad[x * plane + e] = gr;
            }
            cc = nc;
        }
    }
    const double v = sum.total(red);
    if (threadIdx.x == 0) partials[blockIdx.x] = v;
}

static unsigned reg_grid(const tt_handle *h, long long n)
{
    long long b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > dot_blocks(h) ? dot_blocks(h) : b));
}

template <typename T>
static tt_status reg_finish(tt_handle *h, unsigned blocks, double *value_host)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "regulariser launch");
    e = launch_reduce(h, h->red, blocks, h->loss_dev + 1, nullptr, 1.0);
    if (e != cudaSuccess) return cuda_fail(e, "regulariser reduce");
    e = cudaMemcpyAsync(h->loss_pinned + 1, h->loss_dev + 1, sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(e, "regulariser value copy");
    *value_host = h->loss_pinned[1];
    if (!std::isfinite(*value_host)) {
        set_error("regulariser value is not finite");
        return TT_NONFINITE;
    }
    return TT_OK;
}

template <typename T>
static tt_status l2_impl(tt_handle *h, const T *c, T *grad, double *value_host)
{
    const long long n = h->nvox() * h->K;
    const unsigned blocks = reg_grid(h, n);
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_VECTOR, &ev);
    (grad ? k_l2<T, true> : k_l2<T, false>)<<<blocks, 256, 0, h->stream>>>(c, n, grad, h->red);
    prof_end(h, TT_KSLOT_VECTOR, ev);
    return reg_finish<T>(h, blocks, value_host);
}

// Planes of a run.  Float: ten, fewer while the runs do not give every SM two
// blocks (small volumes are bound by the planes a thread takes one after the
// other).
static int tv_run_f32(const tt_handle *h, long long segs)
{
    int run = kTvRun;
    while (run > 1 && segs * ((h->N[0] + run - 1) / run) < 2 * h->n_sm) run = (run + 1) / 2;
    return run;
}
// Double is bound by its arithmetic, so by the SM with the most of it: a run
// takes 3 run + 1 weights with the gradient and run without (the same runs for
// both, so that the value is the same), and the blocks, four per SM at most, go
// round the SMs in turn.  55 x 65 x 55, 6 channels, the value alone: 105 us in tens,
// 86 in threes; 27 x 22 x 25, 15 channels, with the gradient 83 in twos, 79 in threes.
static int tv_run_f64(const tt_handle *h, long long segs)
{
    const long long grid = dot_blocks(h), sms = h->n_sm;
    int best = 1;
    long long least = -1;
    for (int run = 1; run <= kTvRun; ++run) {
        const long long items = segs * ((h->N[0] + run - 1) / run);
        const long long most = items / grid * (grid / sms) + (items % grid + sms - 1) / sms;
        if (least < 0 || most * (4 * run + 1) < least) {
            least = most * (4 * run + 1);
            best = run;
        }
    }
    return best;
}

template <typename T>
static tt_status tv_impl(tt_handle *h, const T *c, double delta, T *grad, double *value_host)
{
    const long long plane = (long long)h->N[1] * h->N[2] * h->K;
    const long long segs = (plane + 255) / 256;
    const int run = std::is_same<T, double>::value ? tv_run_f64(h, segs) : tv_run_f32(h, segs);
    const unsigned blocks = reg_grid(h, segs * 256 * ((h->N[0] + run - 1) / run));
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_VECTOR, &ev);
    (grad ? k_tv_huber<T, true> : k_tv_huber<T, false>)<<<blocks, 256, 0, h->stream>>>(c, h->N[0], h->N[1], h->N[2], h->K, run, (T)delta, grad, h->red);
    prof_end(h, TT_KSLOT_VECTOR, ev);
    return reg_finish<T>(h, blocks, value_host);
}

static tt_status reg_check(const tt_handle *h, tt_precision want, const void *c, const void *grad, const double *value)
{
    if (!h) { set_error("null handle"); return TT_INVALID_ARG; }
    if ((h->prec == TT_F64) != (want == TT_F64)) {
        set_error("handle precision does not match the entry point");
        return TT_INVALID_ARG;
    }
    if (!c || !value || (reinterpret_cast<uintptr_t>(c) & 15u) || (grad && (reinterpret_cast<uintptr_t>(grad) & 15u))) {
        set_error("regulariser: c and value must be non-null, device pointers 16-byte aligned");
        return TT_INVALID_ARG;
    }
    return TT_OK;
}

}  // namespace tt

using namespace tt;

extern "C" {

tt_status tt_l2_norm(tt_handle *h, const float *c, float *grad, double *value_host)
{
    tt_status st = reg_check(h, TT_F32, c, grad, value_host);
    return st != TT_OK ? st : l2_impl<float>(h, c, grad, value_host);
}

tt_status tt_l2_norm_f64(tt_handle *h, const double *c, double *grad, double *value_host)
{
    tt_status st = reg_check(h, TT_F64, c, grad, value_host);
    return st != TT_OK ? st : l2_impl<double>(h, c, grad, value_host);
}

tt_status tt_tv_huber(tt_handle *h, const float *c, double delta, float *grad, double *value_host)
{
    tt_status st = reg_check(h, TT_F32, c, grad, value_host);
    if (st == TT_OK && !(delta > 0.0 && std::isfinite(delta))) { set_error("delta must be positive"); st = TT_INVALID_ARG; }
    return st != TT_OK ? st : tv_impl<float>(h, c, delta, grad, value_host);
}

tt_status tt_tv_huber_f64(tt_handle *h, const double *c, double delta, double *grad, double *value_host)
{
    tt_status st = reg_check(h, TT_F64, c, grad, value_host);
    if (st == TT_OK && !(delta > 0.0 && std::isfinite(delta))) { set_error("delta must be positive"); st = TT_INVALID_ARG; }
    return st != TT_OK ? st : tv_impl<double>(h, c, delta, grad, value_host);
}

}  // extern "C"
