// internal.h -- handle layout and cross-file entry points of libcoxgb.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <utility>
#include <vector>

#include "../../include/coxgb.h"

namespace coxgb {

// Device-side error bits (OR-ed into handle->d_err by kernels).
enum : int { DEVERR_TIMEOUT = 1, DEVERR_NONFINITE = 2, DEVERR_CODE3 = 4 };

constexpr int TILE = 128;          // rows per tensor-core tile, K per chunk
constexpr int BLOCK_BYTES = 4096;  // one 128 x 128 block of 2-bit codes
constexpr int PAD = 1024;          // n, p padding of the tiled layouts
constexpr int MAX_K_TC = 64;       // largest k of the tensor-core path
constexpr int LIMBS = 4;           // e4m3 limbs per coefficient (4 significant bits each)
constexpr int DEC_GROUPS = 3;      // decoder warp groups of the tensor-core products
constexpr int LIMBS4 = 8;          // e2m1 limbs per coefficient (3 significant bits each)
constexpr int LIMBS_W = 10;         // e2m1 limbs that hold a four-limb e4m3 value exactly (the wide form)
constexpr int SF_COL = 504;        // TMEM columns 504..511: unit block scales of the e2m1 products

// Limb columns of a k-column product: LIMBS k rounded up to an MMA width class.
inline int limb_cols(int k)
{
    const int n = LIMBS * k;
    return n <= 16 ? 16 : n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : 256;
}

// Limb columns of the e2m1 form: LIMBS4 k rounded up to 64 or 128 (k <= MAX_K_E2M1);
// 0 beyond.
constexpr int MAX_K_E2M1 = 16;
inline int limb_cols4(int k)
{
    const int n = LIMBS4 * k;
    return n <= 64 ? 64 : n <= 128 ? 128 : 0;
}

// Operand forms of a product (GemmPlan::f4).
enum Form : int {
    FORM_E4M3 = COX_FORM_E4M3,  // e4m3 codes, LIMBS e4m3 limbs (kind::f8f6f4)
    FORM_E2M1 = COX_FORM_E2M1,  // e2m1 codes, LIMBS4 e2m1 limbs (kind::mxf4)
    FORM_WIDE = COX_FORM_WIDE   // e2m1 codes, the LIMBS e4m3 limbs' value as LIMBS_W e2m1 limbs (kind::mxf4)
};
inline int limbs_of(int form) { return form == FORM_WIDE ? LIMBS_W : form == FORM_E2M1 ? LIMBS4 : LIMBS; }

// Limb columns of the wide form: LIMBS_W k rounded up to an MMA width class, 0 past
// MAX_K_WIDE.  One coefficient per LIMBS_W columns; the rest of a class stays zero.
constexpr int MAX_K_WIDE = 12;
inline int limb_cols_wide(int k)
{
    const int n = LIMBS_W * k;
    return n <= 16 ? 16 : n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : 0;
}

// Limb columns of k coefficients in a form (0: not held).
inline int limb_cols_of(int form, int k)
{
    return form == FORM_WIDE ? limb_cols_wide(k) : form == FORM_E2M1 ? limb_cols4(k) : limb_cols(k);
}

// Position of code K (0..15) of a 16-code word: bit 8 (K mod 4) + 2 (K div 4),
// so that (word >> 2q) & 0x03030303 is the four codes 4q..4q+3, one per byte:
// as e4m3 bytes these are the subnormals c 2^-9, exact tensor-core operands.
__host__ __device__ inline int code_bit(int K) { return 8 * (K & 3) + 2 * (K >> 2); }

// ---- e4m3 limbs -----------------------------------------------------------------
// A coefficient column b is held as LIMBS e4m3 numbers: with a power-of-two
// scale 2^s putting max |b| 2^-s in [128, 256) (e4m3 reaches 448),
// r_0 = b 2^-s, d_l = RN_e4m3(r_l), r_(l+1) = 16 (r_l - d_l); each step keeps
// |r| <= 256, and b = 2^s sum_l d_l 2^-4l with about 4 LIMBS significant bits.

// Value of an e4m3 byte (the hardware's conversion to half is exact).
__device__ inline float e4m3_value(uint8_t q)
{
    return __half2float(__half(__nv_cvt_fp8_to_halfraw(q, __NV_E4M3)));
}

__device__ inline int limb_scale(float mx) { return mx > 0.f ? ilogbf(mx) - 7 : 0; }

// Limbs of r (|r| <= 256) into d[0..LIMBS); returns the value they represent.
__device__ inline float split_e4m3(float r, uint8_t *d)
{
    if (!isfinite(r)) {
        for (int l = 0; l < LIMBS; ++l) d[l] = 0x7F;  // NaN: the products flag it
        return r;
    }
    float rep = 0.f, w = 1.f;
#pragma unroll
    for (int l = 0; l < LIMBS; ++l) {
        const uint8_t q = static_cast<uint8_t>(__nv_cvt_float_to_fp8(r, __NV_SATFINITE, __NV_E4M3));
        const float v = e4m3_value(q);
        d[l] = q;
        rep = fmaf(v, w, rep);
        r = (r - v) * 16.f;
        w *= 0.0625f;
    }
    return rep;
}

// The split of split_e4m3, returning the value the limbs represent times 2^21
// as an exact integer (limb l is a multiple of 2^-9 weighted 16^-l; below
// 2^30 in magnitude for |r| <= 256).  Non-finite r gives NaN limbs and 0.
__device__ inline int split_e4m3_units(float r, uint8_t *d)
{
    if (!isfinite(r)) {
        for (int l = 0; l < LIMBS; ++l) d[l] = 0x7F;
        return 0;
    }
    int q = 0;
#pragma unroll
    for (int l = 0; l < LIMBS; ++l) {
        const uint8_t b = static_cast<uint8_t>(__nv_cvt_float_to_fp8(r, __NV_SATFINITE, __NV_E4M3));
        const float v = e4m3_value(b);
        d[l] = b;
        q = 16 * q + static_cast<int>(v * 512.f);  // limb l in units of 2^-9, an integer
        r = (r - v) * 16.f;
    }
    return q;
}

// ---- e2m1 limbs -----------------------------------------------------------------
// A coefficient column b is held as LIMBS4 e2m1 numbers on the grid of halves in
// [-2, 2]: with a power-of-two scale 2^s putting max |b| 2^-s in [1, 2),
// r_0 = b 2^-s, d_l = RN(2 r_l) / 2, r_(l+1) = 8 (r_l - d_l) (exact; |r| <= 2),
// and b = 2^s sum_l d_l 8^-l to within 2^(1 - 3 LIMBS4) = 2^-23 of max |b|.
// Limb rows hold two K positions per byte, in the order the decoders give the
// codes (decode16_e2m1): positions K and K + 8 of a 16-code group w share byte
// 8 w + (K mod 8), K in the low nibble.
__host__ __device__ inline int64_t e2m1_byte(int64_t K) { return ((K >> 4) << 3) + (K & 7); }

__device__ inline int limb_scale4(float mx) { return mx > 0.f ? ilogbf(mx) : 0; }

// Limbs of r (|r| < 2) as e2m1 nibbles; returns the value they represent in
// units of 2^(-1 - 3 (LIMBS4 - 1)), an exact integer.  Non-finite r gives zero
// limbs (NAN_SCALE, or a NaN sum of V, stands for it).
__device__ inline int split_e2m1_units(float r, uint8_t *nib)
{
    if (!isfinite(r)) {
        for (int l = 0; l < LIMBS4; ++l) nib[l] = 0;
        return 0;
    }
    int q = 0;
#pragma unroll
    for (int l = 0; l < LIMBS4; ++l) {
        // t = rint(2 r) in -4 .. 4, as 1.5 2^23 + t: the FP32 add rounds (to even),
        // its low bits are t (rintf and the conversion share a quarter-rate unit)
        const float m = fmaf(2.f, r, 12582912.f);
        const float t = m - 12582912.f;
        const int ti = __float_as_int(m) - 0x4B400000;
        nib[l] = static_cast<uint8_t>(ti < 0 ? 8 - ti : ti);
        q = 8 * q + ti;
        r = fmaf(-4.f, t, 8.f * r);  // 8 (r - t / 2), exact
    }
    return q;
}

// Scale exponent of a column's limbs, by the first warp of a block, from the column's
// max |beta| partials (k_l1_32, compared as bits: a NaN exceeds every number).  bs:
// where the product finds it (may be null).  An e4m3 limb can be NaN and takes the
// whole column with it; digits cannot, so a column with a non-finite entry has
// NAN_SCALE there, which turns the e2m1 kernels' partial sums into NaN: as with FP64
// and e4m3 operands, eta, the loss and the gradient of that column are NaN.
constexpr int NAN_SCALE = 1 << 20;
__device__ inline int column_scale(const float *__restrict__ maxp, int nb, int form, int *bs, int *err)
{
    unsigned u = 0;
    for (int b = threadIdx.x; b < nb; b += 32) u = max(u, __float_as_uint(maxp[b]));
    u = __reduce_max_sync(0xffffffffu, u);
    const float m = __uint_as_float(u);
    const bool bad = !isfinite(m);
    const int s = bad ? 0 : form == FORM_E2M1 ? limb_scale4(m) : limb_scale(m);
    if (threadIdx.x == 0) {
        if (isinf(m)) atomicOr(err, DEVERR_NONFINITE);  // a NaN is reported by the scans
        if (bs) *bs = form != FORM_E4M3 && bad ? NAN_SCALE : s;
    }
    return s;
}

// ---- wide e2m1 limbs --------------------------------------------------------------
// The value of a column's LIMBS e4m3 limbs, an integer q of 2^(s-21) units with
// |q| <= 2^29 (split_e4m3_units), as LIMBS_W balanced radix-8 digits
//   q = sum_l t_l 8^(LIMBS_W-1-l),  t_l in [-4, 4],
// each the e2m1 value t_l / 2: the same coefficient, bit for bit, as operands
// of kind::mxf4 (2^(s+7) sum_l (t_l / 2) 8^-l).  The digits of l >= 1 lie in
// [-4, 3], so the first one keeps |t_0| <= 4 up to |q| = 2^29 (1 + 3/28).
__device__ inline void split_wide(int q, uint8_t *nib)
{
#pragma unroll
    for (int l = LIMBS_W - 1; l > 0; --l) {
        const int t = ((q + 4) & 7) - 4;
        nib[l] = static_cast<uint8_t>(t < 0 ? 8 - t : t);
        q = (q - t) >> 3;
    }
    nib[0] = static_cast<uint8_t>(q < 0 ? 8 - q : q);
}

// 32-bit word index, in a tiled 2-bit layout of KC chunks per row tile, of the
// 16 codes of row rit (0..127) of row tile mt at K offset `within` (a multiple
// of 16) of chunk kc: row records of 32 bytes, two 16-byte halves (K 0-63 and
// 64-127 of the chunk), stored swapped in rows with bit 2 set.
__host__ __device__ inline int64_t word_offset(int64_t mt, int64_t KC, int64_t kc, int rit, int within)
{
    const int hh = within >> 6, w = (within & 63) >> 4;
    const int phys = hh ^ ((rit >> 2) & 1);
    return ((mt * KC + kc) * BLOCK_BYTES + rit * 32 + phys * 16 + w * 4) >> 2;
}

// K order of the SNP-major copy (A4).  Sorted subjects are kept in blocks of
// 16 (one packed word), and sorted block b is stored at block (a b) mod nb,
// nb = n_pad / 16, a odd and prime to nb, near nb (sqrt 5 - 1) / 2.  Any run
// of consecutive K positions then holds subjects spread evenly over the time
// order, so the running sums of x_ij V_i that the tensor cores accumulate do
// not drift with the time trend of V (V = delta - u sums to zero only over all
// subjects); the positions inside a block, and so the K-slot scales, are kept.
__host__ __device__ inline int64_t a4_pos(int64_t i, int64_t a, int64_t nb)
{
    return ((a * (i >> 4)) % nb) * 16 + (i & 15);
}

// One tensor-core product: a 2-bit A (rows x K, tiled) times limb matrix B.
struct GemmPlan {
    int T = 2;         // 128-row tiles per CTA (one M group)
    int CH = 1;        // K chunks (128 each) per stage
    int alt = 0;       // 1: two issuers on alternate stages (else one per row tile)
    int pair = 0;      // 1: per-tile issuers commit after every second stage
    int G = 3;         // decoder groups
    int NP = 16;       // limb columns (limb_cols_of(f4, k))
    int f4 = 0;        // operand form (Form): 0 e4m3, else e2m1 operands (kind::mxf4)
    int stages = 6;    // shared-memory pipeline depth (e2m1 form: code slots)
    int stages2 = 0;   // e2m1 form: limb slots
    int ring = 4;      // TMEM A buffers
    int nb_period = 6; // stage period of the named barriers: lcm(decoder groups, ring)
    int F = 32;        // K chunks per TMEM accumulation window
    int stream = 0;    // 1: both copies of the codes exceed half of L2: load them evict-first
    int grid = 0;      // CTAs
    int KC = 0;        // stages per M group (K chunks / CH)
    int n_groups = 0;  // M groups
    int64_t units = 0, L = 0;
    int max_slots = 1;
    int64_t rows_pad = 0;  // row stride of the partial buffer
    size_t smem = 0;
    CUtensorMap tmA, tmB;
};

struct Workspace {
    int k = 0;        // columns the workspace is sized for
    void *base = nullptr;       // the allocation that holds everything below but part1 and Bqa
    // split / gemv / fp64 common (sorted subject order)
    double *eta = nullptr;      // k x n
    void *w = nullptr;          // k x n: float, double for FP64 handles
    float *Vf = nullptr;        // k x n: V in FP32, for the limbs
    double *Wg = nullptr;       // k x event groups: chunk-local reverse sum of w at the group's head
    double *Fg = nullptr;       // k x event groups: cumulative sum of (events / W) inside its tile of groups
    double *tot = nullptr, *tbase = nullptr, *lgp = nullptr;  // k x tiles: sums of events / W, of the tiles before, of events log W
    double *colc = nullptr;     // k: max eta
    unsigned *scnt = nullptr;   // 2 + 3 k counters of k_scans (zero between launches)
    double *cmax = nullptr, *csw = nullptr, *suf = nullptr;
    double *lossp = nullptr, *vsp = nullptr;  // k x chunks (lossp: sum of delta eta per chunk)
    double *l1p = nullptr;                    // k x l1 blocks
    double *sumV = nullptr;    // k
    double *F = nullptr, *f = nullptr, *l1 = nullptr, *Fring = nullptr;  // k each, lag x k, in a row
    double *mub = nullptr;     // k: mu^T beta (cox_eta)
    double *lam = nullptr;     // k
    int *active = nullptr;     // k
    double *Fcol = nullptr;    // 3 k: F, f, l1 of the columns done so far (FP32 baseline, one column at a time)
    // split mode
    uint8_t *Bq = nullptr;     // limbs of beta in g1's form: NP x p_pad e4m3 or NP x p_pad / 2 e2m1 pairs
                               // (row c limbs_of(form) + l: limb l of column c)
    uint8_t *Vq = nullptr;     // limbs of V in g4's form, A4 K order
    int *bs1 = nullptr;        // k: power-of-two scale of the beta limbs
    int *bs4 = nullptr;        // k: power-of-two scale of the V limbs
    float *bmaxp = nullptr;    // k x l1 blocks: partial max |beta|
    float *vmaxp = nullptr;    // k x chunks: partial max |V|
    float *part1 = nullptr;    // slots x k x rows_pad (eta partials)
    float *part4 = nullptr;    // slots x k x rows_pad (X^T V partials)
    int *cnt4 = nullptr;       // per M group of the second product
    // fp64 / gemv
    double *V64 = nullptr;     // k x n
    float *V32 = nullptr;      // n_pad, A4 K order
    float *eta32 = nullptr;    // n
    float *G32 = nullptr;      // p
    float *gpart = nullptr;    // partials of the FP32 baseline's product
    // unpenalised covariates (q > 0)
    double *gamma = nullptr;   // k x q coefficients (column kk at kk q)
    double *gz = nullptr;      // k x q: Z^T (delta - u) / n at the last evaluation
    double *zvp = nullptr;     // k x q x chunks partials
    GemmPlan g1, g4;
    bool plans_ready = false;
    int part1_slots = 0;       // partial slots part1 holds
    // active-set first product (cox_options.active_set)
    GemmPlan g1a;
    bool g1a_ready = false;
    int64_t g1a_K = 0;
    uint8_t *Bqa = nullptr;    // limbs of beta at the active SNPs, g1's form
};

// The power method's work memory and plans (power.cu): genotype handles only.
struct PowerWork {
    void *base = nullptr;         // one allocation
    uint8_t *Bq = nullptr, *Vq = nullptr;
    float *part = nullptr, *a = nullptr, *b = nullptr;
    double *start = nullptr;
    void *scal = nullptr;
    GemmPlan g1, g4;
};

} // namespace coxgb

struct cox_handle {
    int dev = 0, sm_count = 0;
    int64_t l2_bytes = 0;
    int64_t n = 0, p = 0, n_pad = 0, p_pad = 0;
    int64_t kperm_a = 1, kperm_nb = 1;  // K order of A4 (a4_pos)
    int64_t kperm_ainv = 1;             // a^-1 mod nb: A4 block B holds sorted block ainv B mod nb
    int scan_ept = 8;             // subjects per lane of the risk-set scans (a chunk is a warp's)
    int n_chunks = 0, l1_blocks = 0;
    cox_options opt;
    int64_t n_groups_tie = 0;
    // sorted order (host copies)
    std::vector<int64_t> h_order;
    std::vector<double> h_mu;
    // device data
    int32_t *d_evhead = nullptr;  // first positions of the tie groups that hold an event
    int32_t *d_evcnt = nullptr;   // events in each of those groups
    int32_t *d_evidx = nullptr;   // n: event groups whose head is at or before the subject's tie tail
    uint8_t *d_evflag = nullptr;  // n, padded to whole chunks: 1 at the head of a tie group that holds an event
    int32_t *d_a4blk = nullptr;   // n_pad / 16: sorted 16-subject block -> its block in the K order of A4
    int64_t n_evhead = 0;
    int q = 0;                    // unpenalised covariates
    double *d_Z = nullptr;        // q x n, sorted order
    // active set of the first product (active.cu)
    uint8_t *d_inA = nullptr, *d_flag = nullptr;  // p: in the active set; in the current support
    uint8_t *d_near = nullptr;    // p: pre-threshold value within a quarter of the threshold
    int32_t *d_Aidx = nullptr;    // active SNPs, ascending
    uint32_t *d_A1act = nullptr;  // subject-major 2-bit copy of the active columns
    unsigned long long *d_actcnt = nullptr;
    int64_t nA = -1, act_cap = 0, act_Kpad = 0, act_rebuilds = 0;
    std::vector<int32_t> h_Aidx;  // the active set (host copy)
    uint8_t *d_delta = nullptr;
    double *d_mu = nullptr;
    uint32_t *d_A1 = nullptr;  // subject-major 2-bit tiles
    uint32_t *d_A4 = nullptr;  // SNP-major 2-bit tiles
    double *d_Xr = nullptr;    // FP64: n x p, sorted rows
    double *d_Xc = nullptr;    // FP64: p x n (columns), sorted subjects
    int *d_err = nullptr;      // error bits: the head of RES_BYTES, small results behind
    int64_t device_bytes = 0;
    long long wait_cycles = 0;
    coxgb::Workspace ws;
    coxgb::PowerWork pow;
    // path / checkpoint state
    int st_k = 0;
    std::vector<float> st_beta32;
    std::vector<double> st_beta64;
    std::vector<int> st_iters;
    std::vector<double> st_F;
    std::vector<int> st_active;
    std::vector<double> st_gamma;  // q x k
    int64_t st_step = 0;
    // autotuned pipeline shapes per k: row tiles, K chunks, stages of each product
    struct TuneChoice {
        int T1, CH1, S1, A1, T4, CH4, S4, A4;  // A: issue mode (1 per tile, 2 alternating)
        int F1, F4;                            // operand form (Form)
    };
    std::map<int, TuneChoice> tuned;
    // launch accounting and optional per-kernel-class event timing
    int64_t launches = 0;
    bool prof = false;
    struct ProfRec {
        int cls;
        cudaEvent_t a, b;
    };
    std::vector<ProfRec> prof_recs;
    std::vector<cudaEvent_t> ev_pool;
    size_t ev_used = 0;
};

// The e2m1 form of the tensor-core products (COX_SPLIT_E2M1).
inline bool is_e2m1(const cox_handle *h) { return h->opt.precision == COX_SPLIT_E2M1; }

namespace coxgb {

// ---- error helpers ----------------------------------------------------------
int cuda_status(cudaError_t e);
#define COX_CUDA(x)                                      \
    do {                                                 \
        cudaError_t e_ = (x);                            \
        if (e_ != cudaSuccess) return coxgb::cuda_status(e_); \
    } while (0)
#define COX_TRY(x)            \
    do {                      \
        int r_ = (x);         \
        if (r_ != COX_OK) return r_; \
    } while (0)

// cox_options.wait_limit_s is for the iteration's products.  The scans' grid barriers and
// the power method's products replaced kernels without any wait, so a handle with a
// shorter limit gives them at least this one (cycles, about two seconds).
constexpr long long MIN_WAIT_CYCLES = 4000000000LL;

// Launch with programmatic stream serialisation: the kernel may be scheduled while
// the one ahead of it in the stream ends, and waits for it (pdl_wait) before it
// touches global memory.  coop: as a cooperative grid instead, which starts when the
// kernel ahead has ended (both attributes at once measured no faster).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, bool coop,
                       Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    if (coop) {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    } else {
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// Penalties passed by value to the first kernel of an iteration, which puts them in ws.lam.
constexpr int MAX_LAM_ARG = 64;
struct LamArg {
    int k = 0;
    double v[MAX_LAM_ARG] = {};
};

int dmalloc(cox_handle *h, void **p, size_t bytes);
void dfree(void *p);

// The handle's error bits (d_err) are the head of a block whose rest holds small
// results.  A copy to pageable memory is a wait of its own (14-16 us), so what a call
// returns is brought back together with the bits: cox_loss_grad at n = 20,000, p = 2,000
// takes 126 us against 144 with two copies.  (A pinned buffer per handle did the same
// and cost every cox_setup 140 us.)
constexpr size_t RES_HEAD = 64, RES_BYTES = 16384;
// Waits for the stream, reports and clears the device-side errors met; with `bytes`,
// also brings that many back from src (device) to out (host).
int device_status(cox_handle *h, cudaStream_t st, void *out = nullptr, const void *src = nullptr, size_t bytes = 0);

// ---- setup (setup.cu) ----------------------------------------------------------
int setup_genotypes(cox_handle *h, const void *X, int x_format, cudaStream_t st);
int setup_dense64(cox_handle *h, const double *X, cudaStream_t st);

// ---- workspace / plans / one iteration (api.cu) ----------------------------------
int ensure_workspace(cox_handle *h, int k);
// lam: the k penalties on the host, passed to the first kernel by value (null: ws.lam
// holds them); F_out: where this iteration's objectives also go (device, may be null)
int iterate(cox_handle *h, void *beta, int k, int epi, void *grad, double step, cudaStream_t st,
            const double *lam = nullptr, double *F_out = nullptr);
int iterate_from_eta(cox_handle *h, void *beta, const double *eta, int k, double step, cudaStream_t st,
                     const double *lam);
struct ScanArgs;
void set_covariate_args(cox_handle *h, ScanArgs &sa, int col, int epi, double step);

// ---- scans (scans.cu) -------------------------------------------------------------
// Risk-set scans on eta (sorted order, k columns).  eta_src kinds:
enum EtaSrc { ETA_PARTIAL_F32 = 0, ETA_DENSE_F64 = 1, ETA_DENSE_F32 = 2 };
enum VOut { V_LIMBS_E4M3 = 0, V_DENSE_F64 = 1, V_DENSE_F32 = 2 };
struct ScanArgs {
    int k;
    int eta_src;
    const void *eta;      // partial f32 [slot][k][rows_pad] or dense [k][n]
    int64_t slot_stride, col_stride;  // partial layout
    int group_rows, KC;   // partial slot counts: group of a row, K chunks, L
    int64_t L;
    int v_out;
    void *V;              // e4m3 limbs [NP][n_pad] (scales in ws.bs4) or dense
    int NP;
    bool exp64;           // exp in FP64 (FP64 mode) or FP32
    const double *lam;    // k (objective); may be null
    bool need_loss;
    bool eta_only = false;  // stop after eta (cox_eta)
    // unpenalised covariates (the handle's q > 0): gamma (k x q, read for eta,
    // updated when gamma_step), gz (k x q out: Z^T (delta - u) / n), active (k)
    double *gamma = nullptr;
    double *gz = nullptr;
    const int *active = nullptr;
    double step = 0.0;
    bool gamma_step = false;
    double *F_out = nullptr;
};
int run_scans(cox_handle *h, const ScanArgs &a, cudaStream_t st);
int scan_ept(int64_t n);              // subjects per lane
int scan_tiles(int64_t n_evhead);     // tiles of event groups

// ---- tensor-core products (gemm_tc.cu) ---------------------------------------------
// Plan one product; T_req / CH_req / stages_req of 0 take the defaults.
// The shape and depth arithmetic of a product plan (host only, no device):
// T, CH, NP, stages, ring, nb_period and smem of g, or COX_ERR_ARG for a shape
// not compiled for k or a depth the pipeline does not allow.
// issue_req: 0 default, 1 one issuer per row tile, 2 two issuers on alternate
// stages, 3 one issuer per row tile committing after every second stage.
int plan_shape(GemmPlan &g, int k, int T_req, int CH_req, int stages_req, int issue_req, int f4);
int plan_gemm(cox_handle *h, GemmPlan &g, const uint32_t *A, int64_t rows_pad, int64_t K_pad,
              const uint8_t *B, int k, int form, int T_req, int CH_req, int stages_req, int issue_req);
// The compiled (row tiles, K chunks, issue mode) shapes for k columns; returns
// their count.
int gemm_shapes(int k, int *T, int *CH, int *issue, int max, int f4);
enum Epi { EPI_PARTIAL = 0, EPI_PROX = 1, EPI_GRAD = 2 };
struct EpiArgs {
    int epi = EPI_PARTIAL;
    float *part = nullptr;
    int *counters = nullptr;
    float *beta = nullptr;   // p x k (prox: in/out)
    float *grad = nullptr;   // p x k (grad output)
    const double *lam = nullptr;
    double step = 0;
    const double *mu = nullptr;
    const double *sumV = nullptr;
    const int *active = nullptr;
    uint8_t *near = nullptr;      // p: set where |z| > 3/4 of the threshold (active set's headroom)
    const int *bscale = nullptr;  // k: power-of-two scale of the B limbs
    int64_t rows_valid = 0;  // p
    double inv_n = 0;
    int *err = nullptr;           // error bits (null: the handle's) and wait limit (0: the handle's)
    long long wait = 0;
};
int launch_gemm(cox_handle *h, const GemmPlan &g, const EpiArgs &e, int k, cudaStream_t st);
int prep_limbs_beta(cox_handle *h, const float *beta, int k, cudaStream_t st);

// ---- power method on the genotype tiles (power.cu) ------------------------------------
int power_setup(cox_handle *h);
int power_method_tiles(cox_handle *h, const double *start, double tol, int maxiter, double *L_out);

// ---- active-set first product (active.cu) -------------------------------------------
int active_prepare(cox_handle *h, const float *beta, int k, cudaStream_t st, int *use);
void active_free(cox_handle *h);

// ---- CUDA-core paths (gemv.cu) -----------------------------------------------------
// ||beta_c||_1 partials into ws.l1p; with maxp, max |beta_c| partials too
int l1_norms32(cox_handle *h, const float *beta, int k, cudaStream_t st, float *maxp = nullptr,
               const LamArg *lam = nullptr);
int l1_norms64(cox_handle *h, const double *beta, int k, cudaStream_t st, const LamArg *lam = nullptr);
// The FP32 baseline's product y = A x (byte tables of x; part: the partials,
// gemv_lut_part_floats(rows, KC) floats).  Two kernels.
int gemv_lut(cox_handle *h, const uint32_t *A, int64_t rows, int64_t KC, const float *x, int64_t K_valid,
             float *part, float *y, cudaStream_t st);
size_t gemv_lut_part_floats(int64_t rows_pad, int64_t KC);
int gemv_lut_plan(int64_t rows_pad, int64_t KC, int sm_count, int *n_ranges, int64_t *tiles_per_split, int *grid);
int prox_or_grad32(cox_handle *h, const float *G, int col, float *beta, float *grad,
                   const double *lam, double step, cudaStream_t st);
int eta64(cox_handle *h, const double *beta, int k, double *eta, cudaStream_t st);
int xtv64(cox_handle *h, const double *V, int k, double *beta, double *grad, const double *lam,
          double step, cudaStream_t st);
int center_fix_vec(cox_handle *h, const float *v_in, float *a_out, int64_t len, double sub,
                   cudaStream_t st);
// out (k x n) = ws.eta - mu^T beta per column: X_c beta from the uncentred eta
int eta_centred_out(cox_handle *h, const void *beta, bool f64, int k, double *out, cudaStream_t st);

} // namespace coxgb
