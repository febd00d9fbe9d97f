// power.cu -- the power method of arXiv 2010.16114, Section 4.4, on the 2-bit
// genotype tiles: ||X_c||_2^2 for the Section 5.3 step, as X_c^T (X_c v) on the
// tensor-core products.
//
// Each vector enters the product kernel as LIMBS_W e2m1 digits per entry (the
// wide form, one column): with max |x| 2^-s in [1, 2), x 2^(28-s) rounded to an
// integer and written in balanced radix 8, so an entry is held to 2^(s-29),
// exactly where |x| >= 2^-5 max |x|, and the products' window sums are exact.  The
// estimate is 1.6e-9 to 4.1e-9 from FP64 (root mean square, four sizes; ~1e-8 with the
// FP32 product before): ||v|| after its rounding to FP32, and a's roundings, which have
// the offset mu^T v in common.
// One iteration is six kernels and one 8-byte copy:
//   k_pow_v      v = b / ||b||, its digits, mu^T v
//   (product)    X v, partial slots
//   k_pow_a      a = X v - mu^T v, sum a, max |a|
//   k_pow_alimbs digits of a in the K order of the SNP-major copy
//   (product)    X^T a, partial slots
//   k_pow_b      b = X^T a - mu sum a, ||b||^2, max |b|
// Reductions leave one FP64 partial per block; the block that finishes last adds
// them in block order, so a result does not depend on timing.
// Bound: HBM (each copy of X once per iteration).  20 iterations at n = 100,000,
// p = 50,000 take 9.4 ms (5.3 TB/s over both copies, reductions and the host's
// look at ||b|| included), against 174 ms (0.3 TB/s) for a product of one thread
// per row and one multiply-add per code with one-block reductions.
#include <algorithm>
#include <cmath>

#include "internal.h"

namespace coxgb {
namespace {

constexpr int PT = 256;          // threads per block
constexpr int POW_BLOCKS = 256;  // most blocks of a reducing kernel

// Scalars and block partials of the reductions (device).
struct PowScal {
    double nb2;        // ||b||^2
    double muv;        // mu^T v
    double suma;       // sum a
    float maxb, maxa;  // max |b|, max |a|
    int s1, s4;        // scale exponents of the two digit matrices
    int err;           // device error bits of the products
    unsigned count;    // blocks done
    double part[POW_BLOCKS];
    float maxp[POW_BLOCKS];
};

__device__ __forceinline__ double block_sum(double x, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < PT / 32; ++w) t += sh[w];
    __syncthreads();
    return t;
}

__device__ __forceinline__ float block_max(float x, float *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < PT / 32; ++w) t = fmaxf(t, sh[w]);
    __syncthreads();
    return t;
}

// Leave this block's sum and maximum; true in every thread of the block that
// finishes last, with the totals over all blocks (in block order).
__device__ __forceinline__ bool reduce_last(PowScal *S, double &sum, float &mx)
{
    __shared__ double shd[PT / 32];
    __shared__ float shf[PT / 32];
    __shared__ bool last;
    sum = block_sum(sum, shd);
    mx = block_max(mx, shf);
    if (threadIdx.x == 0) {
        S->part[blockIdx.x] = sum;
        S->maxp[blockIdx.x] = mx;
        __threadfence();
        last = atomicAdd(&S->count, 1u) == gridDim.x - 1;
        if (last) S->count = 0;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    const int t = threadIdx.x;
    static_assert(POW_BLOCKS <= PT, "one partial per thread");
    sum = block_sum(t < static_cast<int>(gridDim.x) ? __ldcg(&S->part[t]) : 0.0, shd);
    mx = block_max(t < static_cast<int>(gridDim.x) ? __ldcg(&S->maxp[t]) : 0.f, shf);
    return true;
}

// Scale exponent s (max |x| 2^-s in [1, 2)) and the digits of x.
__device__ __forceinline__ int pow_scale(float mx) { return mx > 0.f && isfinite(mx) ? ilogbf(mx) : 0; }

__device__ __forceinline__ void digits(float x, int s, uint8_t *d)
{
    const float r = ldexpf(x, 28 - s);  // |r| < 2^29; a NaN has no digits (it reaches the sums instead)
    split_wide(isfinite(r) ? __float2int_rn(r) : 0, d);
}

// b = start / ||start|| (start null: all entries 1/sqrt(p)) with ||b||^2 taken as 1; one block.
__global__ void __launch_bounds__(PT) k_pow_start(const double *__restrict__ start, int64_t p, float *__restrict__ b,
                                                  PowScal *S)
{
    __shared__ double sh[PT / 32];
    __shared__ float shf[PT / 32];
    double s = 0.0;
    for (int64_t j = threadIdx.x; j < p; j += PT) s += start ? start[j] * start[j] : 1.0;
    const double inv = 1.0 / sqrt(block_sum(s, sh));
    float mx = 0.f;
    for (int64_t j = threadIdx.x; j < p; j += PT) {
        const float v = static_cast<float>((start ? start[j] : 1.0) * inv);
        b[j] = v;
        mx = fmaxf(mx, fabsf(v));
    }
    mx = block_max(mx, shf);
    if (threadIdx.x == 0) {
        S->nb2 = 1.0;
        S->maxb = mx;
        S->count = 0;
        S->err = 0;
    }
}

// v = b / ||b|| (FP32), its digits (byte t holds SNPs 16 (t / 8) + t mod 8 and that + 8), mu^T v
__global__ void __launch_bounds__(PT) k_pow_v(const float *__restrict__ b, const double *__restrict__ mu, int64_t p,
                                              int64_t p_pad, uint8_t *__restrict__ Bq, PowScal *S)
{
    const double inv = 1.0 / sqrt(S->nb2);
    const int s = pow_scale(static_cast<float>(static_cast<double>(S->maxb) * inv));
    const int64_t rb = p_pad / 2;
    double dot = 0.0;
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * PT + threadIdx.x; t < rb; t += static_cast<int64_t>(gridDim.x) * PT) {
        const int64_t j = ((t >> 3) << 4) + (t & 7);
        if (j >= p) continue;
        uint8_t d0[LIMBS_W], d1[LIMBS_W] = {};
        const float v0 = static_cast<float>(static_cast<double>(b[j]) * inv);
        dot += mu[j] * static_cast<double>(v0);
        digits(v0, s, d0);
        if (j + 8 < p) {
            const float v1 = static_cast<float>(static_cast<double>(b[j + 8]) * inv);
            dot += mu[j + 8] * static_cast<double>(v1);
            digits(v1, s, d1);
        }
#pragma unroll
        for (int l = 0; l < LIMBS_W; ++l) Bq[l * rb + t] = static_cast<uint8_t>(d0[l] | (d1[l] << 4));
    }
    float mx = 0.f;
    if (reduce_last(S, dot, mx) && threadIdx.x == 0) {
        S->muv = dot;
        S->s1 = s - 7;  // the product's wide limbs are worth 2^(scale + 7)
    }
}

// Sum of a product's partial slots at row i.
__device__ __forceinline__ double slots(const float *__restrict__ part, int64_t stride, int64_t i, int group_rows, int KC,
                                        int64_t L)
{
    const int64_t g = i / group_rows;
    const int cnt = static_cast<int>((g * KC + KC - 1) / L - (g * KC) / L + 1);
    double v = 0.0;
    for (int sl = 0; sl < cnt; ++sl) v += static_cast<double>(part[sl * stride + i]);
    return v;
}

// a = X v - mu^T v for the n subjects, in FP32; sum a, max |a|
__global__ void __launch_bounds__(PT) k_pow_a(const float *__restrict__ part, int64_t stride, int group_rows, int KC,
                                              int64_t L, int64_t n, float *__restrict__ a, PowScal *S)
{
    const double muv = S->muv;
    double sum = 0.0;
    float mx = 0.f;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * PT + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * PT) {
        const float v = static_cast<float>(slots(part, stride, i, group_rows, KC, L) - muv);
        a[i] = v;
        sum += static_cast<double>(v);
        mx = fmaxf(mx, fabsf(v));
    }
    if (reduce_last(S, sum, mx) && threadIdx.x == 0) {
        S->suma = sum;
        S->maxa = mx;
        S->s4 = pow_scale(mx) - 7;
    }
}

// digits of a at the A4 K positions (byte order as k_pow_v's, in sorted blocks of 16)
__global__ void __launch_bounds__(PT) k_pow_alimbs(const float *__restrict__ a, int64_t n, int64_t n_pad, int64_t pa,
                                                   int64_t pnb, uint8_t *__restrict__ Vq, const PowScal *S)
{
    const int s = S->s4 + 7;
    const int64_t rb = n_pad / 2;
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * PT + threadIdx.x; t < rb; t += static_cast<int64_t>(gridDim.x) * PT) {
        const int64_t i = ((t >> 3) << 4) + (t & 7);
        if (i >= n) continue;
        uint8_t d0[LIMBS_W], d1[LIMBS_W] = {};
        digits(a[i], s, d0);
        if (i + 8 < n) digits(a[i + 8], s, d1);
        const int64_t byte = e2m1_byte(a4_pos(i, pa, pnb));
#pragma unroll
        for (int l = 0; l < LIMBS_W; ++l) Vq[l * rb + byte] = static_cast<uint8_t>(d0[l] | (d1[l] << 4));
    }
}

// b = X^T a - mu sum a, in FP32; ||b||^2, max |b|
__global__ void __launch_bounds__(PT) k_pow_b(const float *__restrict__ part, int64_t stride, int group_rows, int KC,
                                              int64_t L, int64_t p, const double *__restrict__ mu, float *__restrict__ b,
                                              PowScal *S)
{
    const double suma = S->suma;
    double sum = 0.0;
    float mx = 0.f;
    for (int64_t j = static_cast<int64_t>(blockIdx.x) * PT + threadIdx.x; j < p; j += static_cast<int64_t>(gridDim.x) * PT) {
        const double v = slots(part, stride, j, group_rows, KC, L) - mu[j] * suma;
        b[j] = static_cast<float>(v);
        sum += v * v;
        mx = fmaxf(mx, fabsf(static_cast<float>(v)));
    }
    if (reduce_last(S, sum, mx) && threadIdx.x == 0) {
        S->nb2 = sum;
        S->maxb = mx;
    }
}

int64_t up256(int64_t b) { return (b + 255) / 256 * 256; }

} // namespace

// The work memory and the two plans, made with the handle so that a call needs
// no device allocation: digits of both vectors (8 bytes per padded entry), the
// vectors, one product's partial slots and the start vector.
int power_setup(cox_handle *h)
{
    PowerWork &w = h->pow;
    w = PowerWork();
    const int64_t n_pad = h->n_pad, p_pad = h->p_pad, NP = limb_cols_wide(1);
    const int64_t bq = up256(NP * p_pad / 2), vq = up256(NP * n_pad / 2);
    // the plans' slot counts do not depend on the buffers' addresses: plan on
    // the genotype copies first, allocate, then plan on the digit matrices
    COX_TRY(plan_gemm(h, w.g1, h->d_A1, n_pad, p_pad, reinterpret_cast<const uint8_t *>(h->d_A1), 1, FORM_WIDE, 0, 0, 0, 0));
    COX_TRY(plan_gemm(h, w.g4, h->d_A4, p_pad, n_pad, reinterpret_cast<const uint8_t *>(h->d_A4), 1, FORM_WIDE, 0, 0, 0, 0));
    const int64_t part = up256(4 * std::max(w.g1.max_slots * n_pad, w.g4.max_slots * p_pad));
    const int64_t fb = up256(4 * p_pad), fa = up256(4 * n_pad), st = up256(8 * h->p), sc = up256(sizeof(PowScal));
    uint8_t *base = nullptr;
    COX_TRY(dmalloc(h, reinterpret_cast<void **>(&base), static_cast<size_t>(bq + vq + part + fb + fa + st + sc)));
    w.base = base;
    w.Bq = base;
    w.Vq = w.Bq + bq;
    w.part = reinterpret_cast<float *>(w.Vq + vq);
    w.b = reinterpret_cast<float *>(w.Vq + vq + part);
    w.a = reinterpret_cast<float *>(w.Vq + vq + part + fb);
    w.start = reinterpret_cast<double *>(w.Vq + vq + part + fb + fa);
    w.scal = w.Vq + vq + part + fb + fa + st;
    // digit rows past LIMBS_W and K positions of padding stay zero
    COX_CUDA(cudaMemset(w.Bq, 0, static_cast<size_t>(bq + vq)));
    COX_TRY(plan_gemm(h, w.g1, h->d_A1, n_pad, p_pad, w.Bq, 1, FORM_WIDE, 0, 0, 0, 0));
    COX_TRY(plan_gemm(h, w.g4, h->d_A4, p_pad, n_pad, w.Vq, 1, FORM_WIDE, 0, 0, 0, 0));
    return COX_OK;
}

// L = 2 ||X_c||_2^2 / n of a genotype handle: from `start` (host, p doubles) or
// all ones, until the estimate changes by at most tol relative or after maxiter
// iterations.  Legacy stream; synchronous.
int power_method_tiles(cox_handle *h, const double *start, double tol, int maxiter, double *L_out)
{
    PowerWork &w = h->pow;
    const int64_t n = h->n, p = h->p;
    PowScal *S = reinterpret_cast<PowScal *>(w.scal);
    cudaStream_t st = 0;
    if (start) COX_CUDA(cudaMemcpyAsync(w.start, start, p * sizeof(double), cudaMemcpyHostToDevice, st));
    k_pow_start<<<1, PT, 0, st>>>(start ? w.start : nullptr, p, w.b, S);
    auto blocks = [](int64_t items) { return static_cast<unsigned>(std::min<int64_t>(POW_BLOCKS, (items + PT - 1) / PT)); };
    auto product = [&](const GemmPlan &g, const int *bscale) -> int {
        EpiArgs e;
        e.part = w.part;
        e.bscale = bscale;
        e.err = &S->err;
        e.wait = std::max(h->wait_cycles, MIN_WAIT_CYCLES);
        return launch_gemm(h, g, e, 1, st);
    };
    double s = 0.0, s_prev = 0.0;
    for (int it = 1; it <= maxiter; ++it) {
        k_pow_v<<<blocks(h->p_pad / 2), PT, 0, st>>>(w.b, h->d_mu, p, h->p_pad, w.Bq, S);
        COX_TRY(product(w.g1, &S->s1));
        k_pow_a<<<blocks(n), PT, 0, st>>>(w.part, h->n_pad, w.g1.T * TILE, w.g1.KC, w.g1.L, n, w.a, S);
        k_pow_alimbs<<<static_cast<unsigned>(std::min<int64_t>(8LL * h->sm_count, (h->n_pad / 2 + PT - 1) / PT)), PT, 0, st>>>(
            w.a, n, h->n_pad, h->kperm_a, h->kperm_nb, w.Vq, S);
        COX_TRY(product(w.g4, &S->s4));
        k_pow_b<<<blocks(p), PT, 0, st>>>(w.part, h->p_pad, w.g4.T * TILE, w.g4.KC, w.g4.L, p, h->d_mu, w.b, S);
        COX_CUDA(cudaGetLastError());
        double nb2 = 0.0;
        COX_CUDA(cudaMemcpy(&nb2, &S->nb2, sizeof(double), cudaMemcpyDeviceToHost));
        if (!(nb2 > 0.0) || !std::isfinite(nb2)) {
            s = 0.0;
            break;
        }
        s = std::sqrt(nb2);  // ||X_c^T X_c v|| -> largest eigenvalue of X_c^T X_c
        if (it > 1 && std::fabs(s - s_prev) <= tol * s) break;
        s_prev = s;
    }
    int e = 0;
    COX_CUDA(cudaMemcpy(&e, &S->err, sizeof(int), cudaMemcpyDeviceToHost));
    if (e & DEVERR_TIMEOUT) return COX_ERR_TIMEOUT;
    *L_out = 2.0 * s / static_cast<double>(n);
    return COX_OK;
}

} // namespace coxgb
