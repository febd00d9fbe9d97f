// scans.cu -- Breslow risk-set sums of the Cox iteration (arXiv 2010.16114,
// Section 5.3: w = exp(eta), W_j = sum_{y_i >= y_j} w_i, u = P delta; the
// paper's remark that sorting by time turns W into a cumulative sum; Section 6:
// Breslow ties).
//
// Subjects are stored in ascending time order, so with R_r = sum_{s >= r} w_s
// (a reverse inclusive scan), and the tie groups that hold events numbered
// g = 0, 1, ... in time order (head h_g, e_g events):
//   W_g = R_{h_g}                       the risk-set sum of group g
//   F_g = sum_{g' <= g} e_g' / W_g'     a forward scan over event groups
//   u_r = w_r F_{G(r) - 1}              G(r) = event groups with head <= r's
//                                       tie tail (u_r = 0 when G(r) = 0)
//   V_r = delta_r - u_r                 (the vector X^T multiplies)
//   f   = (1/n) [sum_g e_g log W_g - sum_r delta_r (eta_r - c)],  c = max eta.
// delta / W is nonzero only at events, and tied events share W, so the
// forward scan runs over the event groups (a few thousand with times in whole
// days) instead of the n subjects.
//
// One cooperative kernel, k_scans, runs all of it in five phases with a grid
// barrier between them, over chunks of subjects (1, 2, 4, 5; a warp each) or tiles
// of 256 event groups (3; a block each) of every column:
//   1  eta from the product's partial slots (+ Z gamma); chunk maxima, sums of
//      delta eta
//   2  w = exp(eta - c); reverse scans inside the chunks, kept at the heads of
//      event groups; chunk totals                        -> suffix sums
//   3  W_g, e_g / W_g, scans inside the tiles; sum e_g log W_g
//                                                        -> prefix sums of the tiles
//   4  V; chunk maxima of |V|; sums of Z^T V
//   5  limbs of V; sums of the values they hold          -> sum V, f, F, gamma
// The block that is the last to finish a column's part of a phase does the work
// on the right, in a fixed order, so results never depend on timing.
//
// What bounds it.  GB300 has two FP64 lanes per SM, so one warp-wide FP64
// instruction holds the pipe for 16 cycles: per-subject arithmetic in the FP32-exp
// modes therefore runs in pairs of floats (TwoSum and FMA error terms, ~2^-47
// relative; the summands are FP32 values themselves), and FP64 is left to
// per-group and per-column work.  A chunk belongs to one warp, so nothing inside a
// phase waits for another warp: the same phases with a block per chunk and a
// counter per chunk took twice as long (latency: 541 us against 264 at n = 400,000,
// k = 32).  At small n the five phases are latency alone (~3-5 us each with their
// barriers).  Measured against seven FP64 kernels (eta, scan, chunk totals, groups,
// V, limbs, sums): 264 us against 590 (n = 400,000, k = 32), 152 against 345 (k = 16),
// 37 against ~95 (n = 100,000, k = 1); a whole FP64 step at n = 1,000, p = 2,000 took 67 us
// against 86 (49 to 53 now).  The steps' errors against FP64 are those of the FP64 kernels:
// 20 seeds and sizes of iterations in the e2m1 form gave the same bits, or the same error.
#include <algorithm>

#include "internal.h"
#include "pairs.cuh"
#include "ptx.cuh"

namespace coxgb {
namespace {

constexpr int NT = 256;
constexpr int NW = NT / 32;
constexpr int MAXQ = 16;
constexpr int GT = NT;  // event groups per tile

__device__ __forceinline__ tf plus(tf a, tf b) { return tf_add(a, b); }
__device__ __forceinline__ double plus(double a, double b) { return a + b; }
__device__ __forceinline__ bool less(tf a, tf b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }
__device__ __forceinline__ bool less(double a, double b) { return a < b; }
__device__ __forceinline__ double as_double(tf a) { return tf_double(a); }
__device__ __forceinline__ double as_double(double a) { return a; }

// ---- block reductions and scans (every thread gets the result) --------------------

template <typename T>
__device__ __forceinline__ T block_sum(T x, T *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = plus(x, shfl_xor(x, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    static_assert(NW == 8, "three levels");
    const T t = plus(plus(plus(sh[0], sh[1]), plus(sh[2], sh[3])), plus(plus(sh[4], sh[5]), plus(sh[6], sh[7])));
    __syncthreads();
    return t;
}

// Inclusive scan in thread order; total = the whole block's sum.
template <typename T>
__device__ __forceinline__ T block_incl_scan(T x, T *sh, T &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = shfl_up(x, o);
        if (lane >= o) x = plus(y, x);
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    T p = sh[lane & (NW - 1)];  // every warp scans the warp sums
#pragma unroll
    for (int o = 1; o < NW; o <<= 1) {
        const T y = shfl_up(p, o);
        if ((lane & (NW - 1)) >= o) p = plus(y, p);
    }
    total = shfl_at(p, NW - 1);
    const T pre = shfl_at(p, warp > 0 ? warp - 1 : 0);
    __syncthreads();
    return warp > 0 ? plus(pre, x) : x;
}

__device__ __forceinline__ float block_max(float x, float *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    float t = sh[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) t = fmaxf(t, sh[w]);
    __syncthreads();
    return t;
}

// m (positive, normal) -> m 2^-e in [1, 2); returns e.  Lets a product of
// many positive factors be carried as (mantissa, exponent) without overflow.
__device__ __forceinline__ int renorm(double &m)
{
    const long long b = __double_as_longlong(m);
    m = __longlong_as_double((b & 0x000FFFFFFFFFFFFFLL) | 0x3FF0000000000000LL);
    return static_cast<int>(b >> 52) - 1023;
}

struct SP {
    int64_t n, n_pad;
    int nch, k, ntile;
    int64_t per;            // chunks per block
    int64_t G;              // event groups
    const uint8_t *delta, *evflag;   // evflag padded with zeros to whole chunks
    const int32_t *evhead, *evcnt, *evidx;
    const int32_t *a4blk;   // 16-subject block -> its block in the K order of the SNP-major copy
    // eta source
    int src, group_rows, KC;
    const void *eta_in;
    int64_t slot_stride, col_stride, L;
    // workspace (per column: chunks, tiles, groups)
    void *eta, *w;          // tf and float, or double and double
    float *V32;
    double *Wg, *Fg, *csw, *suf, *lossp, *tot, *tbase, *lgp, *vsp, *zvp;
    void *cmaxp;            // chunk maxima of eta (tf or double)
    float *vmaxp;
    double *colc;           // per column: c
    unsigned *cnt;          // [0] barrier arrivals, [1] blocks done, then 3 per column
    // covariates
    int q;
    const double *Z;
    double *gamma, *gz;
    bool gamma_step;
    const int *active;
    double step;
    // output
    int vo, form;
    void *V;
    int *bs;
    int l1_blocks;
    const double *l1p, *lam;
    double *sumV, *f, *l1, *F, *F_out;
    bool need_loss;
    int *err;
    long long wait_limit;
};

// All blocks of the (cooperative) grid reach barrier `b` (1, 2, ...) before any
// goes on.  Bounded like every wait: past the limit the block reports a timeout
// and goes on (all indexes below come from the handle's static arrays).
__device__ __forceinline__ void grid_barrier(const SP &s, unsigned b)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(s.cnt, 1u);
        const unsigned want = b * gridDim.x;
        const long long t0 = clock64();
        unsigned v;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(s.cnt) : "memory");
            if (v >= want) break;
            if (clock64() - t0 > s.wait_limit) {
                atomicOr(s.err, DEVERR_TIMEOUT);
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
}

// Called by every block that took part in column kk in a phase (or once per tile):
// true in the one whose call is the last of `total`.
__device__ __forceinline__ bool last_of_column(const SP &s, int kk, int phase, unsigned total)
{
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned *c = s.cnt + 2 + 3 * kk + phase;
        last = atomicAdd(c, 1u) == total - 1u;
        if (last) *c = 0;
        __threadfence();
    }
    __syncthreads();
    return last;
}

// Blocks whose range of `per` tasks meets column kk (its nch tasks follow those of column kk - 1).
__device__ __forceinline__ unsigned column_blocks(const SP &s, int kk)
{
    const int64_t a = static_cast<int64_t>(kk) * s.nch, b = a + s.nch - 1;
    return static_cast<unsigned>(b / s.per - a / s.per + 1);
}

// sum V, f, ||beta||_1, F = f + lambda ||beta||_1, and for covariates g_Z =
// Z^T (delta - u) / n and, for a step, gamma <- gamma + step g_Z (Section 6: the
// covariates take a plain gradient step; a frozen column keeps its gamma); flags
// non-finite values.
__device__ __forceinline__ void finalize_column(const SP &s, int kk)
{
    const double n = static_cast<double>(s.n);
    const int lane = threadIdx.x & 31;
    for (int cq = threadIdx.x >> 5; cq < s.q; cq += NW) {  // a warp per covariate
        const double *zp = s.zvp + (static_cast<int64_t>(kk) * s.q + cq) * s.nch;
        double z4[4] = {0.0, 0.0, 0.0, 0.0};
        int c = lane;
        for (; c + 224 < s.nch; c += 256) {
            double u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) u[e] = zp[c + 32 * e];
#pragma unroll
            for (int e = 0; e < 8; ++e) z4[e & 3] += u[e];
        }
        for (; c < s.nch; c += 32) z4[0] += zp[c];
        double z = (z4[0] + z4[1]) + (z4[2] + z4[3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        z /= n;
        if (lane == 0) {
            s.gz[kk * s.q + cq] = z;
            if (s.gamma_step && (!s.active || s.active[kk])) s.gamma[kk * s.q + cq] += s.step * z;
            if (!isfinite(z)) atomicOr(s.err, DEVERR_NONFINITE);
        }
    }
    // f = (sum_g e_g log W_g + (events) c - sum_r delta_r eta_r) / n
    double x[4] = {0.0, 0.0, 0.0, 0.0};  // sum V, sum delta eta, ||beta||_1, sum e log W
    for (int c = threadIdx.x; c < s.nch; c += NT) {
        x[0] += s.vsp[static_cast<int64_t>(kk) * s.nch + c];
        if (s.need_loss) x[1] += s.lossp[static_cast<int64_t>(kk) * s.nch + c];
    }
    if (s.need_loss) {
        if (s.l1p)
            for (int c = threadIdx.x; c < s.l1_blocks; c += NT) x[2] += s.l1p[kk * s.l1_blocks + c];
        for (int t = threadIdx.x; t < s.ntile; t += NT) x[3] += s.lgp[static_cast<int64_t>(kk) * s.ntile + t];
    }
    __shared__ double sh4[4][NW];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] += __shfl_xor_sync(0xffffffffu, x[e], o);
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int e = 0; e < 4; ++e) sh4[e][threadIdx.x >> 5] = x[e];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            x[e] = ((sh4[e][0] + sh4[e][1]) + (sh4[e][2] + sh4[e][3])) + ((sh4[e][4] + sh4[e][5]) + (sh4[e][6] + sh4[e][7]));
    }
    __syncthreads();
    const double v = x[0], b1 = x[2];
    if (threadIdx.x != 0) return;
    s.sumV[kk] = v;
    if (s.need_loss) {
        const double lo = (x[3] - x[1]) / n;
        s.f[kk] = lo;
        s.l1[kk] = b1;
        const double F = lo + (s.lam ? s.lam[kk] * b1 : 0.0);
        s.F[kk] = F;
        if (s.F_out) s.F_out[kk] = F;
        if (!isfinite(lo)) atomicOr(s.err, DEVERR_NONFINITE);
    }
    if (!isfinite(v)) atomicOr(s.err, DEVERR_NONFINITE);
}

// Exclusive prefix (of `in`, this thread's run in thread order) from the block's
// inclusive scan.
template <typename T>
__device__ __forceinline__ T block_excl(T run, T *sh, T zero)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T total;
    const T in = block_incl_scan(run, sh, total);
    T ex = shfl_up(in, 1);
    if (lane == 31) sh[warp] = in;
    __syncthreads();
    if (lane == 0) ex = warp > 0 ? sh[warp - 1] : zero;
    __syncthreads();
    return ex;
}

// Partial slots of row group g: the CTAs whose unit ranges meet it.
__device__ __forceinline__ int slot_count(const SP &s, int64_t g)
{
    const int64_t a = g * s.KC, b = a + s.KC - 1;
    if (b < (int64_t(1) << 31) && s.L < (int64_t(1) << 31))
        return static_cast<int>(static_cast<uint32_t>(b) / static_cast<uint32_t>(s.L) -
                                static_cast<uint32_t>(a) / static_cast<uint32_t>(s.L)) + 1;
    return static_cast<int>(b / s.L - a / s.L + 1);
}

// Padded shared-memory index of element e of a chunk (the scan reads runs of
// EPT elements per lane: without the padding 8-way bank conflicts).
__device__ __forceinline__ int padded(int e) { return e + (e >> 5); }

// EPT: subjects per lane (a chunk is the 32 EPT subjects of one warp); F64: FP64
// throughout (COX_FP64); Q: the most unpenalised covariates (0, 4, 8 or 16; FP64 handles
// have no 8).  A covariate costs two FP64 multiply-adds per subject and column whether a
// call has it or not, and two registers, so a call takes the smallest variant that holds
// its q: a step at n = 400,000, p = 5,000, k = 16 takes 736 us with q <= 4 (four blocks
// per SM), 845 with q <= 8 (three), 970 with q <= 12 and 1,066 with 16 (two), where one
// variant of 16 took 1,040-1,060 for any q, more than the separate kernels before the
// fused scans for q < 8 (898 at q = 1, 24 more per covariate).
// Block b takes the chunks [b per, (b + 1) per) of the column-major
// list, its warps in turn; nothing inside a chunk waits for another warp.
template <int EPT, bool F64, int Q>
__global__ void __launch_bounds__(NT, Q > 8 ? 2 : Q > 4 ? 3 : 4) k_scans(const SP s)
{
    constexpr int CW = 32 * EPT;
    constexpr int SURE = F64 ? 0 : Q > 4 ? Q / 2 : 0;  // covariates that every call of this variant has
    constexpr int BW = CW + CW / 32;  // doubles of a warp's buffer
    using acc_t = typename std::conditional<F64, double, tf>::type;
    using w_t = typename std::conditional<F64, double, float>::type;
    acc_t zero, low;  // 0 and minus infinity
    if constexpr (F64) {
        zero = 0.0;
        low = -INFINITY;
    } else {
        zero = tf{0.f, 0.f};
        low = tf{-INFINITY, 0.f};
    }
    __shared__ __align__(16) double buf_all[NW * BW];  // per warp: w of a chunk (2), C of its event groups (4)
    __shared__ double shd[NW];
    __shared__ acc_t sha[NW];
    __shared__ float shf[NW];
    __shared__ long long shl[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *const buf = buf_all + warp * BW;
    pdl_trigger();  // the product behind may set up as soon as this grid runs
    const int64_t nch = s.nch, tasks = nch * s.k;
    const int64_t lo = min(tasks, blockIdx.x * s.per), hi = min(tasks, lo + s.per);

    // ---- phase 1: eta, chunk maxima, chunk sums of delta eta ----
    for (int64_t t = lo + warp; t < hi; t += NW) {
        const int kk = static_cast<int>(t / nch);
        const int64_t c = t - kk * nch, i0 = c * CW;
        int cnt0 = 1, cnt1 = 1;
        if (s.src == ETA_PARTIAL_F32) {  // a chunk meets at most two row groups (of 128 or 256)
            cnt0 = slot_count(s, i0 / s.group_rows);
            cnt1 = EPT == 8 ? slot_count(s, (i0 + 128) / s.group_rows) : cnt0;
        }
        acc_t v[EPT];
        uint8_t ev[EPT];
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
            const int64_t i = min(i0 + lane + 32 * j, s.n - 1);
            ev[j] = s.delta[i];
            if (s.src == ETA_PARTIAL_F32 || s.src == ETA_DENSE_F32) {
                const float a = static_cast<const float *>(s.eta_in)[kk * s.col_stride + i];
                if constexpr (F64) v[j] = static_cast<double>(a);
                else v[j] = tf{a, 0.f};
            } else {
                const double a = static_cast<const double *>(s.eta_in)[kk * s.col_stride + i];
                if constexpr (F64) v[j] = a;
                else v[j] = tf_of(a);
            }
        }
        if (cnt0 > 1 || cnt1 > 1) {  // a row group cut between CTAs
#pragma unroll
            for (int j = 0; j < EPT; ++j) {
                const int64_t i = min(i0 + lane + 32 * j, s.n - 1);
                const float *part = static_cast<const float *>(s.eta_in) + kk * s.col_stride + i;
                const int cnt = EPT == 8 && j >= 4 ? cnt1 : cnt0;
                for (int sl = 1; sl < cnt; ++sl) {
                    const float b = part[sl * s.slot_stride];
                    if constexpr (F64) v[j] += static_cast<double>(b);
                    else v[j] = tf_add(v[j], tf{b, 0.f});
                }
            }
        }
        acc_t mx = low, de = zero;
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
            const int64_t i = i0 + lane + 32 * j;
            if (i >= s.n) break;
            if (Q) {  // eta += Z gamma (Section 6 unpenalised covariates), in FP64
                double zg[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
                for (int cq = 0; cq < Q; ++cq) {  // unrolled: every load in flight at once
                    if (cq == 12 && s.q <= 12) break;
                    if (cq < SURE || cq < s.q) zg[cq & 3] += s.Z[cq * s.n + i] * s.gamma[kk * s.q + cq];
                }
                const double vd = as_double(v[j]) + ((zg[0] + zg[1]) + (zg[2] + zg[3]));
                if constexpr (F64) v[j] = vd;
                else v[j] = tf_of(vd);
            }
            static_cast<acc_t *>(s.eta)[kk * s.n + i] = v[j];
            if (less(mx, v[j])) mx = v[j];
            if (ev[j]) de = plus(de, v[j]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const acc_t y = shfl_xor(mx, o);
            if (less(mx, y)) mx = y;
            de = plus(de, shfl_xor(de, o));
        }
        if (lane == 0) {
            static_cast<acc_t *>(s.cmaxp)[t] = mx;
            s.lossp[t] = as_double(de);
        }
    }
    grid_barrier(s, 1);

    // ---- phase 2: w = exp(eta - c); chunk-local reverse scan of w, kept at the
    // heads of the tie groups that hold events (the only places W is read) ----
    for (int64_t t0 = lo; t0 < hi;) {
        const int kk = static_cast<int>(t0 / nch);
        const int64_t t1 = min(hi, (kk + 1) * nch);
        acc_t cm = low;  // c: the column's largest eta (every block for itself)
#pragma unroll 4
        for (int64_t q = tid; q < nch; q += NT) {
            const acc_t y = static_cast<const acc_t *>(s.cmaxp)[kk * nch + q];
            if (less(cm, y)) cm = y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const acc_t y = shfl_xor(cm, o);
            if (less(cm, y)) cm = y;
        }
        if (lane == 0) sha[warp] = cm;
        __syncthreads();
        cm = sha[0];
#pragma unroll
        for (int w = 1; w < NW; ++w)
            if (less(cm, sha[w])) cm = sha[w];
        __syncthreads();
        if (tid == 0 && t0 == kk * nch) s.colc[kk] = as_double(cm);
        for (int64_t t = t0 + warp; t < t1; t += NW) {
            const int64_t c = t - kk * nch, i0 = c * CW;
            w_t *wb = reinterpret_cast<w_t *>(buf);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < EPT; ++j) {
                const int64_t i = i0 + lane + 32 * j;
                w_t wv = 0;
                if (i < s.n) {
                    const acc_t v = static_cast<const acc_t *>(s.eta)[kk * s.n + i];
                    if constexpr (F64) {
                        wv = exp(v - cm);
                    } else {
                        const tf d = two_sum(v.h, -cm.h);
                        wv = expf(d.h + (d.l + (v.l - cm.l)));  // the FP32 rounding of eta - c
                    }
                    static_cast<w_t *>(s.w)[kk * s.n + i] = wv;
                }
                wb[padded(lane + 32 * j)] = wv;
            }
            const int64_t ib = i0 + CW - EPT * (lane + 1);  // this lane's subjects: ib .. ib + EPT - 1
            uint64_t fl;  // their event-group flags, a byte each
            if constexpr (EPT == 8) fl = *reinterpret_cast<const uint64_t *>(s.evflag + ib);
            else if constexpr (EPT == 4) fl = *reinterpret_cast<const uint32_t *>(s.evflag + ib);
            else if constexpr (EPT == 2) fl = *reinterpret_cast<const uint16_t *>(s.evflag + ib);
            else fl = s.evflag[ib];
            __syncwarp();
            // lane l owns reversed positions [EPT l, EPT l + EPT): elements CW-1-(EPT l + j)
            acc_t loc[EPT], run = zero;
#pragma unroll
            for (int j = 0; j < EPT; ++j) {
                const w_t wv = wb[padded(CW - 1 - (EPT * lane + j))];
                if constexpr (F64) run += wv;
                else run = tf_add(run, tf{wv, 0.f});
                loc[j] = run;
            }
            acc_t incl = run;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const acc_t y = shfl_up(incl, o);
                if (lane >= o) incl = plus(y, incl);
            }
            acc_t excl = shfl_up(incl, 1);
            if (lane == 0) excl = zero;
            if (fl) {
#pragma unroll
                for (int j = 0; j < EPT; ++j)
                    if ((fl >> (8 * (EPT - 1 - j))) & 0xff)
                        s.Wg[kk * s.G + s.evidx[ib + EPT - 1 - j] - 1] = as_double(plus(excl, loc[j]));
            }
            if (lane == 31) s.csw[t] = as_double(incl);
        }
        if (last_of_column(s, kk, 0, column_blocks(s, kk))) {
            // exclusive suffix sums of the chunk totals; thread t owns a contiguous run
            // of chunks in scan order
            const double *src = s.csw + kk * nch;
            double *dst = s.suf + kk * nch;
            const int64_t per = (nch + NT - 1) / NT;
            double tot = 0.0;
#pragma unroll 8
            for (int64_t j = 0; j < per; ++j)
                if (tid * per + j < nch) tot += src[nch - 1 - (tid * per + j)];
            double acc = block_excl(tot, shd, 0.0);
#pragma unroll 8
            for (int64_t j = 0; j < per; ++j) {
                const int64_t q = tid * per + j;
                if (q < nch) {
                    dst[nch - 1 - q] = acc;
                    acc += src[nch - 1 - q];
                }
            }
        }
        t0 = t1;
    }
    grid_barrier(s, 2);

    // ---- phase 3: W_g = the chunk-local reverse sum at the group's head plus the
    // suffix of later chunks; D_g = e_g / W_g (one FP64 division per event time:
    // tied events share W, Breslow); scans of D inside tiles of GT groups ----
    const int64_t tiles = static_cast<int64_t>(s.ntile) * s.k;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int kk = static_cast<int>(t / s.ntile);
        const int64_t g = (t - static_cast<int64_t>(kk) * s.ntile) * GT + tid;
        double D = 0.0;
        if (g < s.G) {
            const double W = s.Wg[kk * s.G + g] + s.suf[kk * nch + s.evhead[g] / CW];
            D = static_cast<double>(s.evcnt[g]) / W;
        }
        double total;
        const double incl = block_incl_scan(D, shd, total);
        if (g < s.G) s.Fg[kk * s.G + g] = incl;  // within the tile; the tile's base is added in phase 4
        if (tid == 0) s.tot[t] = total;
        if (last_of_column(s, kk, 1, s.ntile)) {
            const double *src = s.tot + static_cast<int64_t>(kk) * s.ntile;
            double *dst = s.tbase + static_cast<int64_t>(kk) * s.ntile;
            const int per = (s.ntile + NT - 1) / NT;
            double run = 0.0;
            for (int j = 0; j < per; ++j)
                if (tid * per + j < s.ntile) run += src[tid * per + j];
            double acc = block_excl(run, shd, 0.0);
            for (int j = 0; j < per; ++j)
                if (tid * per + j < s.ntile) {
                    dst[tid * per + j] = acc;
                    acc += src[tid * per + j];
                }
        }
    }
    // ---- beside phase 3, on the last blocks: the loss term sum_g e_g log W_g +
    // (events) c of the tiles, of products carried as (mantissa, exponent), one log
    // per tile (FP64 log is costly) ----
    for (int64_t t = gridDim.x - 1 - blockIdx.x; s.need_loss && t < tiles; t += gridDim.x) {
        const int kk = static_cast<int>(t / s.ntile);
        const int64_t g = (t - static_cast<int64_t>(kk) * s.ntile) * GT + tid;
        double pm = 1.0, lsum = 0.0;
        int pe = 0, ev = 0;
        if (g < s.G) {
            const double W = s.Wg[kk * s.G + g] + s.suf[kk * nch + s.evhead[g] / CW];
            ev = s.evcnt[g];
            if (ev <= 64 && W >= 0x1p-1000 && W <= 0x1p+1000) {
                double b = W;  // W^ev by squaring, both factors renormalised at every step
                int be = renorm(b);
                for (int x = ev; x > 0; x >>= 1) {
                    if (x & 1) {
                        pm *= b;
                        pe += be + renorm(pm);
                    }
                    b *= b;
                    be = 2 * be + renorm(b);
                }
            } else {
                lsum = static_cast<double>(ev) * log(W);  // many tied events, or W zero, huge, subnormal, NaN
            }
        }
        lsum = block_sum(lsum, shd);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {  // 32 factors in [1, 2): no overflow
            pm *= __shfl_xor_sync(0xffffffffu, pm, o);
            pe += __shfl_xor_sync(0xffffffffu, pe, o);
            ev += __shfl_xor_sync(0xffffffffu, ev, o);
        }
        if (lane == 0) {
            shd[warp] = pm;
            shl[warp] = (static_cast<long long>(pe) << 32) | static_cast<unsigned>(ev);
        }
        __syncthreads();
        if (tid == 0) {
            long long pes = pe, evs = ev;
            for (int w = 1; w < NW; ++w) {
                pes += renorm(pm);
                pm *= shd[w];
                pes += shl[w] >> 32;
                evs += shl[w] & 0xffffffffLL;
            }
            s.lgp[t] = lsum + (log(pm) + static_cast<double>(pes) * 0.6931471805599453 + static_cast<double>(evs) * s.colc[kk]);
        }
        __syncthreads();
    }

    grid_barrier(s, 3);

    // ---- phase 4: C = F of the last event group at or before the tie tail; u = w C;
    // V = delta - u.  The FP32 dense form feeds a product over the SNP-major copy and
    // is written at its K positions; the FP64 form stays in sorted order; for the
    // limbs, V goes to V32 with chunk maxima of |V| ----
    const bool limbs = s.vo == V_LIMBS_E4M3;
    for (int64_t t = lo + warp; t < hi; t += NW) {
        const int kk = static_cast<int>(t / nch);
        const int64_t c = t - kk * nch, i0 = c * CW;
        w_t wv[EPT];
        int gi[EPT];
        uint8_t ev[EPT];
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
            const int64_t i = min(i0 + lane + 32 * j, s.n - 1);
            wv[j] = static_cast<const w_t *>(s.w)[kk * s.n + i];
            gi[j] = s.evidx[i];
            ev[j] = s.delta[i];
        }
        // C at the event groups the chunk reads (at most one more per subject), as
        // pairs of floats unless covariates need V in FP64 or some C leaves FP32's range
        const int glo = __shfl_sync(0xffffffffu, gi[0], 0), ghi = __shfl_sync(0xffffffffu, gi[EPT - 1], 31);
        __syncwarp();
        bool wide = F64 || Q;
        for (int pass = 0; pass < 2; ++pass) {
            bool big = false;
            for (int u = lane; u <= ghi - glo; u += 32) {
                const int g = glo + u;
                const double C = g > 0 ? s.Fg[kk * s.G + g - 1] + s.tbase[static_cast<int64_t>(kk) * s.ntile + (g - 1) / GT] : 0.0;
                if (wide) {
                    buf[u] = C;
                } else {
                    big |= !(C < 1e37);
                    reinterpret_cast<tf *>(buf)[u] = tf_of(C);
                }
            }
            big = __any_sync(0xffffffffu, big);
            if (wide || !big) break;
            wide = true;
        }
        __syncwarp();
        acc_t vs = zero;
        float vm32 = 0.f;
        double zv[Q ? Q : 1] = {};  // Z^T V over this lane's subjects (unpenalised covariates)
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
            const int64_t i = i0 + lane + 32 * j;
            if (i >= s.n) break;
            const int u = gi[j] - glo;
            float v32;
            double V = 0.0;
            if (wide) {
                V = (ev[j] ? 1.0 : 0.0) - static_cast<double>(wv[j]) * buf[u];
                v32 = static_cast<float>(V);
            } else {
                const tf C = reinterpret_cast<const tf *>(buf)[u];
                const float wf = static_cast<float>(wv[j]);
                const float p = wf * C.h;
                const float r = fmaf(wf, C.l, fmaf(wf, C.h, -p));  // w C = p + r
                const tf d = two_sum(ev[j] ? 1.f : 0.f, -p);
                v32 = d.h + (d.l - r);
            }
            if (Q) {
#pragma unroll
                for (int cq = 0; cq < Q; ++cq) {
                    if (cq == 12 && s.q <= 12) break;
                    if (cq < SURE || cq < s.q) zv[cq] += s.Z[cq * s.n + i] * V;
                }
            }
            // sum V in the form the product reads: X^T V - mu sum V is then
            // exactly the centred product of that V.  (Censored subjects between
            // two event times share one V, so their rounding errors do not
            // cancel; with the exact sum, mu times their sum would remain.)
            if (limbs) {
                s.V32[kk * s.n + i] = v32;
                vm32 = fmaxf(vm32, fabsf(v32));
            } else if constexpr (F64) {
                static_cast<double *>(s.V)[kk * s.n + i] = V;
                vs += V;
            } else {
                static_cast<float *>(s.V)[static_cast<int64_t>(s.a4blk[i >> 4]) * 16 + (i & 15) + kk * s.n_pad] = v32;
                vs = tf_add(vs, tf{v32, 0.f});
            }
        }
        if (limbs) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) vm32 = fmaxf(vm32, __shfl_xor_sync(0xffffffffu, vm32, o));
            if (lane == 0) s.vmaxp[t] = vm32;
        } else {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) vs = plus(vs, shfl_xor(vs, o));
            if (lane == 0) s.vsp[t] = as_double(vs);
        }
        if constexpr (Q > 0) {
            // sums over the lanes of all Q values at once: at each of the first log2 Q steps a
            // lane passes half of its values on and keeps the other half (Q = 16: 16 FP64 adds
            // against 80); the 32 / Q lanes from (32 / Q) cq on end with covariate cq's
#pragma unroll
            for (int o = 16, m = Q / 2; m > 0; o >>= 1, m >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int e = 0; e < m; ++e) {
                    const double send = up ? zv[e] : zv[e + m], keep = up ? zv[e + m] : zv[e];
                    zv[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
#pragma unroll
            for (int o = 16 / Q; o > 0; o >>= 1) zv[0] += __shfl_xor_sync(0xffffffffu, zv[0], o);
            const int cq = lane / (32 / Q);
            if (lane % (32 / Q) == 0 && cq < s.q) s.zvp[(static_cast<int64_t>(kk) * s.q + cq) * nch + c] = zv[0];
        }
    }
    if (limbs) grid_barrier(s, 4);

    // ---- phase 5: V (FP32) -> limbs at the A4 K positions under the column's
    // power-of-two scale; chunk sums of the values the limbs hold, exact integers:
    // units of 2^(s-21) (e4m3 values, below 2^30 each) or 2^(s-22) (e2m1) ----
    for (int64_t t0 = lo; t0 < hi;) {
        const int kk = static_cast<int>(t0 / nch);
        const int64_t t1 = min(hi, (kk + 1) * nch);
        if (limbs) {
            float m = 0.f;  // the column's largest |V| (every block for itself)
#pragma unroll 4
            for (int64_t q = tid; q < nch; q += NT) m = fmaxf(m, s.vmaxp[kk * nch + q]);
            m = block_max(m, shf);
            const bool bad = !isfinite(m);
            if (bad) m = 0.f;
            const int sc = s.form == FORM_E2M1 ? limb_scale4(m) : limb_scale(m);
            if (tid == 0 && t0 == kk * nch) {
                s.bs[kk] = sc;
                if (bad) atomicOr(s.err, DEVERR_NONFINITE);
            }
            // V 2^-sc, in two exact factors (sc lies in [-156, 127]; |V| >= 1/n whenever
            // V is not all zero, so nothing the limbs can hold becomes subnormal)
            const float s1 = ldexpf(1.f, -(sc / 2)), s2 = ldexpf(1.f, -(sc - sc / 2));
            uint8_t *Vq = static_cast<uint8_t *>(s.V);
            const float *V32 = s.V32 + kk * s.n;
            for (int64_t t = t0 + warp; t < t1; t += NW) {
                const int64_t i0 = (t - kk * nch) * CW;
                long long q = 0;
                bool finite = true;
                if (s.form == FORM_E4M3) {
#pragma unroll
                    for (int j = 0; j < EPT; ++j) {
                        const int64_t i = i0 + lane + 32 * j;
                        if (i >= s.n) break;
                        uint8_t d[LIMBS];
                        const float r = V32[i] * s1 * s2;
                        finite = finite && isfinite(r);
                        q += split_e4m3_units(r, d);
                        const int64_t pos = static_cast<int64_t>(s.a4blk[i >> 4]) * 16 + (i & 15);
#pragma unroll
                        for (int l = 0; l < LIMBS; ++l) Vq[(LIMBS * kk + l) * s.n_pad + pos] = d[l];
                    }
                } else {
                    // subjects 16 (e / 8) + e mod 8 and that + 8 share one byte per limb row (e2m1_byte)
                    const int64_t rb = s.n_pad / 2;
#pragma unroll
                    for (int j = 0; j < (EPT + 1) / 2; ++j) {
                        const int e = lane + 32 * j;
                        const int64_t ia = i0 + ((e >> 3) << 4) + (e & 7);
                        if (e >= CW / 2 || ia >= s.n) break;
                        const float ra = V32[ia] * s1 * s2;
                        const float rb8 = ia + 8 < s.n ? V32[ia + 8] * s1 * s2 : 0.f;
                        finite = finite && isfinite(ra) && isfinite(rb8);
                        const int64_t byte = static_cast<int64_t>(s.a4blk[ia >> 4]) * 8 + (ia & 7);
                        if (s.form == FORM_E2M1) {
                            uint8_t d0[LIMBS4], d1[LIMBS4];
                            q += split_e2m1_units(ra, d0);
                            q += split_e2m1_units(rb8, d1);
#pragma unroll
                            for (int l = 0; l < LIMBS4; ++l)
                                Vq[(LIMBS4 * kk + l) * rb + byte] = static_cast<uint8_t>(d0[l] | (d1[l] << 4));
                        } else {
                            uint8_t d[LIMBS], d0[LIMBS_W], d1[LIMBS_W];
                            const int qa = split_e4m3_units(ra, d), qb = split_e4m3_units(rb8, d);
                            q += qa;
                            q += qb;
                            split_wide(qa, d0);
                            split_wide(qb, d1);
#pragma unroll
                            for (int l = 0; l < LIMBS_W; ++l)
                                Vq[(LIMBS_W * kk + l) * rb + byte] = static_cast<uint8_t>(d0[l] | (d1[l] << 4));
                        }
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
                finite = __all_sync(0xffffffffu, finite);
                const int unit = s.form == FORM_E2M1 ? 1 + 3 * (LIMBS4 - 1) : 21;
                if (lane == 0) s.vsp[t] = finite ? ldexp(static_cast<double>(q), sc - unit) : NAN;
            }
        }
        if (last_of_column(s, kk, 2, column_blocks(s, kk))) finalize_column(s, kk);
        t0 = t1;
    }

    // the last block to end leaves the barrier's counters at zero for the next launch
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(s.cnt + 1, 1u) == gridDim.x - 1) {
            s.cnt[0] = 0;
            s.cnt[1] = 0;
        }
    }
}

// eta (FP64) from the product's partial slots, for cox_eta.
__global__ void k_eta(const float *__restrict__ part, int64_t n, int64_t slot_stride, int64_t col_stride, int group_rows,
                      int KC, int64_t L, double *__restrict__ eta)
{
    const int kk = blockIdx.y;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * NT + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * NT) {
        const int64_t g = i / group_rows;
        const int cnt = static_cast<int>((g * KC + KC - 1) / L - (g * KC) / L + 1);
        double v = 0.0;
        for (int sl = 0; sl < cnt; ++sl) v += static_cast<double>(part[sl * slot_stride + kk * col_stride + i]);
        eta[kk * n + i] = v;
    }
}

using ScanFn = void (*)(const SP);

template <int EPT, bool F64>
ScanFn pick_scan(int q)
{
    if (q > 8 || (F64 && q > 4)) return k_scans<EPT, F64, MAXQ>;
    if (q > 4) return k_scans<EPT, F64, F64 ? MAXQ : 8>;
    return q > 0 ? k_scans<EPT, F64, 4> : k_scans<EPT, F64, 0>;
}

ScanFn pick_scan(int ept, bool f64, int q)
{
    switch (ept) {
    case 1: return f64 ? pick_scan<1, true>(q) : pick_scan<1, false>(q);
    case 2: return f64 ? pick_scan<2, true>(q) : pick_scan<2, false>(q);
    case 4: return f64 ? pick_scan<4, true>(q) : pick_scan<4, false>(q);
    default: return f64 ? pick_scan<8, true>(q) : pick_scan<8, false>(q);
    }
}

} // namespace

// Subjects per lane: the smallest of 1, 2, 4, 8 that leaves at most 2000 chunks
// (warps) a column, so that one column of a small problem spreads over the SMs.
int scan_ept(int64_t n)
{
    for (int e = 1; e < 8; e *= 2)
        if (n <= static_cast<int64_t>(2000) * 32 * e) return e;
    return 8;
}

int scan_tiles(int64_t n_evhead) { return static_cast<int>((n_evhead + GT - 1) / GT); }

int run_scans(cox_handle *h, const ScanArgs &a, cudaStream_t st)
{
    Workspace &ws = h->ws;
    if (a.eta_only) {
        k_eta<<<dim3(static_cast<unsigned>(std::min<int64_t>((h->n + NT - 1) / NT, 1024)), a.k), NT, 0, st>>>(
            static_cast<const float *>(a.eta), h->n, a.slot_stride, a.col_stride, a.group_rows, a.KC, a.L, ws.eta);
        COX_CUDA(cudaGetLastError());
        return COX_OK;
    }
    SP s;
    s.n = h->n;
    s.n_pad = h->n_pad;
    s.nch = h->n_chunks;
    s.k = a.k;
    s.G = h->n_evhead;
    s.ntile = scan_tiles(s.G);
    s.delta = h->d_delta;
    s.evflag = h->d_evflag;
    s.evhead = h->d_evhead;
    s.evcnt = h->d_evcnt;
    s.evidx = h->d_evidx;
    s.a4blk = h->d_a4blk;
    s.src = a.eta_src;
    s.group_rows = a.group_rows;
    s.KC = a.KC;
    s.eta_in = a.eta;
    s.slot_stride = a.slot_stride;
    s.col_stride = a.col_stride;
    s.L = a.L;
    s.eta = ws.eta;
    s.w = ws.w;
    s.V32 = ws.Vf;
    s.Wg = ws.Wg;
    s.Fg = ws.Fg;
    s.csw = ws.csw;
    s.suf = ws.suf;
    s.lossp = ws.lossp;
    s.tot = ws.tot;
    s.tbase = ws.tbase;
    s.lgp = ws.lgp;
    s.vsp = ws.vsp;
    s.zvp = ws.zvp;
    s.cmaxp = ws.cmax;
    s.vmaxp = ws.vmaxp;
    s.colc = ws.colc;
    s.cnt = ws.scnt;
    s.q = a.gamma ? h->q : 0;
    s.Z = h->d_Z;
    s.gamma = a.gamma;
    s.gz = a.gz;
    s.gamma_step = a.gamma_step;
    s.active = a.active;
    s.step = a.step;
    s.vo = a.v_out;
    s.form = ws.g4.f4;
    s.V = a.V;
    s.bs = ws.bs4;
    s.l1_blocks = h->l1_blocks;
    s.l1p = a.need_loss ? ws.l1p : nullptr;
    s.lam = a.lam;
    s.sumV = ws.sumV;
    s.f = ws.f;
    s.l1 = ws.l1;
    s.F = ws.F;
    s.F_out = a.F_out;
    s.need_loss = a.need_loss;
    s.err = h->d_err;
    s.wait_limit = std::max(h->wait_cycles, MIN_WAIT_CYCLES);  // FP64 and FP32 handles have no other waits to limit
    const ScanFn fn = pick_scan(h->scan_ept, a.exp64, s.q);
    int occ = 0;
    COX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, NT, 0));
    // a warp per chunk, up to what the SMs hold at once (the grid barrier needs every
    // block resident), and a block per tile of event groups while there is room
    const int64_t room = static_cast<int64_t>(occ) * h->sm_count, tasks = static_cast<int64_t>(s.nch) * a.k;
    const int64_t mains = std::min(room, (tasks + NW - 1) / NW);
    s.per = (tasks + mains - 1) / mains;
    const unsigned grid = static_cast<unsigned>(std::min(room, mains + 2 * static_cast<int64_t>(s.ntile) * a.k));
    COX_CUDA(launch_pdl(fn, dim3(grid), NT, 0, st, true, s));
    return COX_OK;
}

} // namespace coxgb
