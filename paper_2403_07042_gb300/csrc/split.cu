// Split-precision step in increment form.
//
// With E_k = H_kk and P = diag(exp(-i E_k dt)), the propagator factors exactly as
// U = P (I + Delta), Delta = P^-1 U - I, so the "unitary evolution" of Sec. 4.2 is
//     V = U rho U^+ = P (rho + W + W^+ + X) P^+,   W = Delta rho,  X = W Delta^+.
// Only the small increments W and X go through the tensor cores: every operand is split
// into power-of-two scaled FP16 pieces (rho and W: hi + lo; the constant Delta: hi + mid +
// lo, because its representation error would otherwise add up coherently step after
// step) and the products that matter at 2^-22 are accumulated in FP32 (GEMM1: four,
// GEMM2: three).  Complex products use the real embedding with the signs folded into the
// constant operands:
//   GEMM1  [W_re; W_im] (2Dp x Dp)  = [[D_re, D_im], [D_im, -D_re]] . [rho_re | rho_im]^T
//   GEMM2  [X_re | X_im] (Dp x 2Dp) = [W_re | W_im] . [[D_re, D_im], [-D_im, D_re]]^T
// (rho^T = conj(rho) for the Hermitian rho, so the row-major rho planes are the K-major
// operand directly.)
//
// The master rho is held as a double-float (an unevaluated sum of two FP32 words, about
// 48 significant bits): GB300 executes FP64 at a small fraction of its FP32 rate, so the
// per-step element work (forming V, the phase, the Lindblad update of Eq. 3, the next
// FP16 planes) runs entirely in FP32 arithmetic with error-free transformations.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "block.h"
#include "checks.h"
#include "gemm_tc.h"
#include "kernels.h"
#include "pdl.h"
#include "split.h"
#include "df.h"

namespace qed {

// Device-side description of one instance (one model) for the grouped kernels.
struct InstDesc {
    int64_t D, Dp;
    float s_rho;            // scale of the rho planes
    float4 *rho, *V, *Y;    // state, V = U rho U^+, stage buffer of the Strang step
    const float4 *phase;
    const float2 *damp;
    const int32_t *in_ptr, *in_jump, *in_src;
    const float2 *coef;
    const uint32_t *mask;   // [D] the jumps with an entry in row k, bit j, or null (use the lists)
    const int4 *jtab;       // [D][kInMax] per jump j < nj: {src or -1, coef hi, coef lo, 0}, or null
    int nj;
    __half *rho_pl;
    uint32_t *err;          // the instance's error word (bounds checks of the QED_CHECKS build)
};

// Models with at most kInMax jumps have per-jump tables for the Lie update (dissipate_jt_kernel).
constexpr int kInMax = 4;
// Models with at most 32 jumps, kMaskEntries of them into one state, match two rows' entries by
// masks of their jumps; others (a lattice's leaks into the vacuum) merge the lists.
constexpr int kMaskEntries = 16;
// Pairs of incoming lists longer than this in total are merged by the whole warp.
constexpr int kLongMerge = 32;

// 32 x (8 kRows) element blocks (the Lindblad kernels) of one instance
struct TileItem {
    int inst, bx, by, pad;
};

// The grouped work of one or many instances: descriptors, GEMM jobs and work lists.
struct Batch {
    void *block = nullptr;  // the allocation of every table
    int n = 0;
    InstDesc *desc = nullptr;
    GemmJob *jobs1 = nullptr, *jobs2 = nullptr;
    int *kblocks = nullptr;       // the products' k-block lists (GemmJob)
    CUtensorMap *maps = nullptr;  // [4 n]: A1, B1, A2, B2 of each instance
    GemmItem *items1 = nullptr, *items2 = nullptr;
    int n_items1 = 0, n_items2 = 0;
    TileItem *etiles = nullptr;  // blocks of the Lindblad kernels
    int n_etiles = 0, erows = 0; // rows of a block of the general one
    TileItem *pairs = nullptr;   // pairs of 32 x 32 tiles (begin_kernel, end_kernel)
    int n_pairs = 0;
    void **rhos = nullptr, **records = nullptr;  // a batch's pointers of the present call
    uint32_t *errors = nullptr;
    bool jt = false;  // every instance has per-jump incoming tables (dissipate_jt_kernel)
    int cs1 = 1, cs2 = 1;  // split-K slices of GEMM1 / GEMM2 = CTAs per cluster
    int scheme = QED_SCHEME_LIE;
    int bn1 = 256, bn2 = 128;  // tile widths (one per grouped launch)
    // one model on its own: its products launch with their tensor maps and jobs as kernel
    // parameters (tc_gemm_single_launch) instead of through the tables above
    bool single = false;
    int64_t D = 0;
    TcGemm g1, g2;
    GemmJob j1, j2;
    void release() {
        if (block) cudaFree(block);
        *this = Batch();
    }
};

struct SplitState {
    void *arrays = nullptr, *tables = nullptr;  // the allocations of what follows
    Batch self;               // this model as a batch of one
    int64_t Dp = 0;           // padded dimension (multiple of 128)
    int num_sms = 148;
    TcGemm g1, g2;
    // constant operands, FP16 [3 (hi, mid, lo)][2Dp][2Dp]
    __half *a1 = nullptr;     // [[Dre, Dim], [Dim, -Dre]]   (GEMM1 A)
    __half *b2 = nullptr;     // [[Dre, Dim], [-Dim, Dre]]   (GEMM2 B), rows in [re | im] groups of 64
    // dynamic operands, FP16 [2 (hi, lo)][Dp][2Dp]
    __half *rho_pl = nullptr; // rows l: [rho_re | rho_im]
    __half *w_pl = nullptr;   // rows k: [W_re | W_im]
    float *w32 = nullptr;     // [2][Dp][Dp]  W (re plane, im plane)
    float4 *rho_df[2] = {nullptr, nullptr};  // D x D {re_hi, re_lo, im_hi, im_lo}: rho, then V
    float4 *y_df = nullptr;                  // D x D stage buffer of the Strang step
    float4 *phase_df = nullptr;              // D: P_k as {re_hi, re_lo, im_hi, im_lo}
    float2 *damp_df = nullptr;               // D: dt/2 * d_k as {hi, lo}
    float2 *coef_df = nullptr;               // incoming jump entries: sqrt(dt) * coefficient
    uint32_t *mask = nullptr;                // jumps of each row's incoming entries, bit by bit
    int4 *jtab = nullptr;                    // per-jump incoming table (at most kInMax jumps)
    int nj = 0;
    double scale_delta = 1.0, scale_rho = 1.0, scale_w = 1.0;
    uint8_t *stats = nullptr;                // scratch of delta_stats_kernel and delta_blocks_kernel
    std::vector<uint8_t> nz;                 // [ceil(D / 64)]^2: blocks of Delta's planes with a nonzero
    int batch_bn1 = 0, batch_bn2 = 0;  // tile widths of the grouped launches (tuned or set), 0 by size
};

namespace {

inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// ------------------------------------------------------------------ set-up kernels
__device__ __forceinline__ void split_half3(double x, __half &hi, __half &mid, __half &lo) {
    hi = __double2half(x);
    double r = x - (double)__half2float(hi);
    mid = __double2half(r);
    lo = __double2half(r - (double)__half2float(mid));
}

// Delta = P_k^-1 U_kl - delta_kl: conj(P_k) U_kl for the unit phases of U = exp(-i H dt)
// (unit != 0), conj(P_k) U_kl / |P_k|^2 for the damped phases of the effective step
__global__ void make_delta_kernel(int64_t D, const double2 *U, const double2 *P, double2 *Dl, int unit) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= D * D) return;
    int64_t k = idx / D, l = idx % D;
    double2 u = U[idx], p = P[k];
    double2 d = make_double2(p.x * u.x + p.y * u.y, p.x * u.y - p.y * u.x);
    if (!unit) {
        const double inv = 1.0 / (p.x * p.x + p.y * p.y);
        d.x *= inv;
        d.y *= inv;
    }
    if (k == l) d.x -= 1.0;
    Dl[idx] = d;
}

// What the planes' scales need of Delta, one block per row: stats = {max |Delta_kl|,
// max_k sum_l |Delta_kl|} (as bits: non-negative doubles order like integers).
__global__ void __launch_bounds__(256) delta_stats_kernel(int64_t D, const double2 *Dl, unsigned long long *stats) {
    __shared__ double part[2][8];
    const int64_t k = blockIdx.x;
    double top = 0.0, sum = 0.0;
    for (int64_t l = threadIdx.x; l < D; l += blockDim.x) {
        const double2 d = Dl[k * D + l];
        double x = hypot(d.x, d.y);
        if (!(x <= HUGE_VAL)) x = HUGE_VAL;  // NaN counts as infinity
        top = fmax(top, x);
        sum += x;
    }
    for (int off = 16; off > 0; off >>= 1) {
        top = fmax(top, __shfl_xor_sync(0xffffffffu, top, off));
        sum += __shfl_xor_sync(0xffffffffu, sum, off);
    }
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x / 32] = top;
        part[1][threadIdx.x / 32] = sum;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 8; ++w) {
        top = fmax(top, part[0][w]);
        sum += part[1][w];
    }
    atomicMax(&stats[0], (unsigned long long)__double_as_longlong(top));
    atomicMax(&stats[1], (unsigned long long)__double_as_longlong(sum));
}

// nz[k / 64][l / 64]: whether the planes of that block of s Delta have a nonzero (one block per row).
// An element whose leading FP16 piece is zero is zero in all three.  Delta reaches as far as the
// couplings do in the series' terms, its planes only to 2^-39 of its largest element: with lists of
// Delta's own nonzeros the 32 x 32 lattice's GEMM1 takes 100 us and GEMM2 88, with the planes' 75 and 76.
__global__ void __launch_bounds__(256) delta_blocks_kernel(int64_t D, const double2 *Dl, double s, uint8_t *nz) {
    const int64_t k = blockIdx.x, nb = (D + 63) / 64;
    for (int64_t l = threadIdx.x; l < D; l += blockDim.x) {
        const double2 d = Dl[k * D + l];
        if (__half2float(__double2half(d.x * s)) != 0.f || __half2float(__double2half(d.y * s)) != 0.f)
            nz[(k / 64) * nb + l / 64] = 1;
    }
}

// a1 = [[Dre, Dim], [Dim, -Dre]] and b2 = [[Dre, Dim], [-Dim, Dre]] (2Dp x 2Dp) as three
// FP16 planes (hi, mid, lo), about 33 significant bits.  b2's rows are GEMM2's output
// columns; they are stored in groups of 128 = [the re rows of 64 consecutive n | the im rows
// of the same n], so that one 128-wide output tile holds X_re and X_im of 64 columns.
__global__ void static_planes_kernel(int64_t D, int64_t Dp, const double2 *Dl, double s, __half *a1, __half *b2) {
    const int64_t W2 = 2 * Dp;
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= W2 * W2) return;
    int64_t r = idx / W2, c = idx % W2;
    int64_t cm = c % Dp;
    bool clo = c >= Dp;
    int64_t rk = r % Dp;                             // a1: row r = plane (r >= Dp), index r % Dp
    bool rlo = r >= Dp;
    int64_t rkb = 64 * (r / 128) + (r % 64);         // b2: column group r / 128, part (r % 128) / 64
    bool rlob = (r % 128) >= 64;
    double va = 0.0, vb = 0.0;
    if (rk < D && cm < D) {
        double2 d = Dl[rk * D + cm];
        if (!rlo && !clo) va = d.x;
        else if (!rlo && clo) va = d.y;
        else if (rlo && !clo) va = d.y;
        else va = -d.x;
    }
    if (rkb < D && cm < D) {
        double2 d = Dl[rkb * D + cm];
        if (!rlob && !clo) vb = d.x;
        else if (!rlob && clo) vb = d.y;
        else if (rlob && !clo) vb = -d.y;
        else vb = d.x;
    }
    __half h, md, l;
    split_half3(va * s, h, md, l);
    a1[idx] = h;
    a1[W2 * W2 + idx] = md;
    a1[2 * W2 * W2 + idx] = l;
    split_half3(vb * s, h, md, l);
    b2[idx] = h;
    b2[W2 * W2 + idx] = md;
    b2[2 * W2 * W2 + idx] = l;
}

// ------------------------------------------------------------------ per-evolve kernels
// FP16 planes of GEMM1's B operand from the double-float state
__global__ void planes_from_state_kernel(int64_t D, int64_t Dp, const float4 *st, float s, __half *pl) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t m = blockIdx.y;
    if (n >= D) return;
    const float4 v = st[m * D + n];
    const int64_t plane = Dp * 2 * Dp;
    __half h, l;
    df_to_half2({v.x, v.y}, s, h, l);
    pl[m * 2 * Dp + n] = h;
    pl[plane + m * 2 * Dp + n] = l;
    df_to_half2({v.z, v.w}, s, h, l);
    pl[m * 2 * Dp + Dp + n] = h;
    pl[plane + m * 2 * Dp + Dp + n] = l;
}

// Start of a run, one block per pair of 32 x 32 tiles (bx <= by) of an instance: the caller's rho
// (FP64) becomes the double-float state and the FP16 planes of GEMM1's operand, and is checked
// against the split path's precondition: Hermitian (GEMM1's operand is the row-major rho read as
// rho^T = conj(rho), and X = W Delta^+ is formed as a Hermitian matrix) and of unit trace (the FP16
// scale assumes |rho_mn| <= 1 and the renormalisation divides by the trace).  A tile meets its
// mirror in shared memory, so rho is read once; the block of the first pair also sums the
// diagonal (whose trace the effective step moves: kAnyTrace asks for 0 < tr rho <= 1).  With separate
// kernels, one per instance, these took 13 us an instance of a batch.
enum { kNoCheck = 0, kUnitTrace = 1, kAnyTrace = 2 };
int density_check(int scheme) { return scheme == QED_SCHEME_EFFECTIVE ? kAnyTrace : kUnitTrace; }
__global__ void __launch_bounds__(256) begin_kernel(const TileItem *__restrict__ tiles,
                                                    const InstDesc *__restrict__ descs,
                                                    const double2 *const *__restrict__ rhos, const double2 *rho_only,
                                                    int check) {
    __shared__ double2 t[2][32][33];
    __shared__ double part[256];
    const TileItem it = tiles[blockIdx.x];
    const InstDesc &a = descs[it.inst];
    const int64_t D = a.D, Dp = a.Dp, plane = Dp * 2 * Dp;
    const double2 *rho = rho_only ? rho_only : rhos[it.inst];
    const int tx = threadIdx.x;
    bool fine = true;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int64_t n = (int64_t)(side ? it.bx : it.by) * 32 + tx;
        for (int r = threadIdx.y; r < 32; r += 8) {
            const int64_t m = (int64_t)(side ? it.by : it.bx) * 32 + r;
            const bool inside = m < D && n < D;
            const double2 v = inside ? rho[m * D + n] : make_double2(0.0, 0.0);
            t[side][r][tx] = v;
            if (!inside || (side && it.bx == it.by)) continue;
            const float rh = (float)v.x, ih = (float)v.y;
            const df re = {rh, (float)(v.x - (double)rh)}, im = {ih, (float)(v.y - (double)ih)};
            a.rho[m * D + n] = make_float4(re.hi, re.lo, im.hi, im.lo);
            __half h, l;
            __half *pl = a.rho_pl + m * 2 * Dp + n;
            df_to_half2(re, a.s_rho, h, l);
            pl[0] = h;
            pl[plane] = l;
            df_to_half2(im, a.s_rho, h, l);
            pl[Dp] = h;
            pl[plane + Dp] = l;
        }
    }
    if (check == kNoCheck) return;
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8) {
        const double2 x = t[0][r][tx], y = t[1][tx][r];
        const double dr = fabs(x.x - y.x), di = fabs(x.y + y.y);
        fine = fine && dr <= kDensityHermTol && di <= kDensityHermTol;  // (false for NaN)
    }
    if (!fine) atomicOr(a.err, kErrNotDensity);
    if (it.bx != 0 || it.by != 0) return;
    const int q = threadIdx.y * 32 + tx;
    double s = 0.0;
    for (int64_t k = q; k < D; k += 256) s += rho[k * D + k].x;
    part[q] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (q < h) part[q] += part[q + h];
        __syncthreads();
    }
    const bool trace_ok = check == kUnitTrace ? fabs(part[0] - 1.0) <= kDensityTraceTol
                                     : (part[0] > 0.0 && part[0] <= 1.0 + kDensityTraceTol);
    if (q == 0 && !trace_ok) atomicOr(a.err, kErrNotDensity);
}

// End of a run, over the same tiles: the state back into the caller's rho.
__global__ void __launch_bounds__(256) end_kernel(const TileItem *__restrict__ tiles,
                                                  const InstDesc *__restrict__ descs, double2 *const *__restrict__ rhos,
                                                  double2 *rho_only) {
    const TileItem it = tiles[blockIdx.x];
    const InstDesc &a = descs[it.inst];
    const int64_t D = a.D;
    double2 *rho = rho_only ? rho_only : rhos[it.inst];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        if (side && it.bx == it.by) return;
        const int64_t n = (int64_t)(side ? it.bx : it.by) * 32 + threadIdx.x;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t m = (int64_t)(side ? it.by : it.bx) * 32 + threadIdx.y + 8 * r;
            if (m >= D || n >= D) continue;
            const float4 v = a.rho[m * D + n];
            rho[m * D + n] = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
        }
    }
}

// out[i] = instance i's error word.
__global__ void read_errors_kernel(int n, const InstDesc *__restrict__ descs, uint32_t *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = *descs[i].err;
}

// One block per instance: its populations into row `row` of its records.
__global__ void __launch_bounds__(256) batch_populations_kernel(const InstDesc *__restrict__ descs,
                                                                double *const *__restrict__ records, int64_t row) {
    const InstDesc &a = descs[blockIdx.x];
    if (!records[blockIdx.x]) return;
    double *out = records[blockIdx.x] + row * a.D;
    for (int64_t k = threadIdx.x; k < a.D; k += blockDim.x) {
        const float4 v = a.rho[k * a.D + k];
        out[k] = (double)v.x + (double)v.y;
    }
}

// The Lindblad term of Eq. (3) as an update of the double-float buffers:
//   out_mn = B_mn + f [ -(dt/2)(d_m + d_n) X_mn + dt sum_j c_j(m) c_j(n) X[src_j(m), src_j(n)] ],
// f a power of two (exact).  The correction (relative size dt gamma) is formed to FP32
// accuracy and added to the double-float B.  With X = B = V, f = 1 and out = rho this is
// the Euler step of the Lie splitting; with f = 1/4 and 1/2 it gives the two stages of the
// explicit midpoint rule of the Strang splitting.  Optionally writes the FP16 planes of out
// (the next GEMM1's operand).  Buffers are chosen by index: 0 rho, 1 V, 2 the stage buffer.
__device__ __forceinline__ float4 *state_buf(const InstDesc &a, int sel) {
    return sel == 0 ? a.rho : (sel == 1 ? a.V : a.Y);
}

// A pair of long incoming lists (many jumps into one state, e.g. every leak into the
// vacuum): the whole warp (blockDim.x == 32, every lane present) shares the merge of each
// such pair.  Lanes take every 32nd entry of the shorter list and find its jump in the
// longer one by bisection; the owner lane gets the sum of c_p c_q X[src_p, src_q] (dt
// included in the coefficients) added to (gr, gi).  Returns whether this lane's own pair
// was handled.  Kept out of line so that the common path keeps its registers.
__device__ __noinline__ bool long_merge_df(uint32_t *err, int64_t D, const int32_t *in_jump, const int32_t *in_src,
                                           const float2 *coef, const float4 *X, int p, int pe, int q, int qe,
                                           float &gr, float &gi) {
    const bool is_long = pe > p && qe > q && (pe - p) + (qe - q) > kLongMerge;
    unsigned longs = __ballot_sync(0xffffffffu, is_long);
    const int lane = threadIdx.x;
    while (longs) {
        const int owner = __ffs(longs) - 1;
        longs &= longs - 1;
        const int op = __shfl_sync(0xffffffffu, p, owner), ope = __shfl_sync(0xffffffffu, pe, owner);
        const int oq = __shfl_sync(0xffffffffu, q, owner), oqe = __shfl_sync(0xffffffffu, qe, owner);
        const bool m_short = ope - op <= oqe - oq;
        const int s0 = m_short ? op : oq, s1 = m_short ? ope : oqe;
        const int l0 = m_short ? oq : op, l1 = m_short ? oqe : ope;
        float sr = 0.f, si = 0.f;
        if (op == oq) {  // a diagonal element: every entry meets itself
#pragma unroll 4
            for (int e = s0 + lane; e < s1; e += 32) {
                const int k = in_src[e];
                if (!qed_check(err, k >= 0 && k < D)) continue;
                const float2 ce = coef[e];
                const df c = df_mul({ce.x, ce.y}, {ce.x, ce.y});
                const float4 u = X[(int64_t)k * D + k];
                const float ur = u.x + u.y, ui = u.z + u.w;
                sr = __fmaf_rn(c.hi, ur, __fmaf_rn(c.lo, ur, sr));
                si = __fmaf_rn(c.hi, ui, __fmaf_rn(c.lo, ui, si));
            }
        } else {
            for (int e = s0 + lane; e < s1; e += 32) {
                const int j = in_jump[e];
                int lo = l0, hi = l1;  // first entry of the longer list with jump >= j
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (in_jump[mid] < j)
                        lo = mid + 1;
                    else
                        hi = mid;
                }
                const int ep = m_short ? e : lo, eq = m_short ? lo : e;  // row m's entry, row n's
                if (lo < l1 && in_jump[lo] == j &&
                    qed_check(err, in_src[ep] >= 0 && in_src[ep] < D && in_src[eq] >= 0 && in_src[eq] < D)) {
                    const float2 cp = coef[ep], cq = coef[eq];
                    const df c = df_mul({cp.x, cp.y}, {cq.x, cq.y});
                    const float4 u = X[(int64_t)in_src[ep] * D + in_src[eq]];
                    const float ur = u.x + u.y, ui = u.z + u.w;
                    sr = __fmaf_rn(c.hi, ur, __fmaf_rn(c.lo, ur, sr));
                    si = __fmaf_rn(c.hi, ui, __fmaf_rn(c.lo, ui, si));
                }
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            sr += __shfl_xor_sync(0xffffffffu, sr, off);
            si += __shfl_xor_sync(0xffffffffu, si, off);
        }
        if (lane == owner) {
            gr += sr;
            gi += si;
        }
    }
    return is_long;
}

// Rows of one element block of the per-jump kernel: 32 x 8 threads update 32 columns and 8 kRows
// rows; thread (x, y) takes the rows 8 r + y, r < kRows, of its column, so the column's jump
// entries are read once for kRows elements and their loads are in flight together.
constexpr int kRows = 2;
// Blocks of the general Lindblad kernel: kWideCols columns, two adjacent ones a thread (it stores
// pairs), and up to kWideRows rows.  kStaged entries of each row and column are staged.
constexpr int kWideCols = 64, kWideRows = 64, kStaged = 8;

// The output of one element, B_mn + (gr, gi), written as a double-float, and its FP16 planes when
// asked for.
__device__ __forceinline__ void lindblad_store(const InstDesc &a, float4 *O, int64_t m, int64_t n, const cdf &b,
                                               float gr, float gi, bool planes) {
    cdf out;
    out.re = df_add_f(b.re, gr);
    out.im = df_add_f(b.im, gi);
    O[m * a.D + n] = store_cdf(out);
    if (!planes) return;
    const int64_t plane = a.Dp * 2 * a.Dp;
    __half h, l;
    df_to_half2(out.re, a.s_rho, h, l);
    a.rho_pl[m * 2 * a.Dp + n] = h;
    a.rho_pl[plane + m * 2 * a.Dp + n] = l;
    df_to_half2(out.im, a.s_rho, h, l);
    a.rho_pl[m * 2 * a.Dp + a.Dp + n] = h;
    a.rho_pl[plane + m * 2 * a.Dp + a.Dp + n] = l;
}

// -(d_m + d_n) dt/2 X_mn in FP32 (d from the double-float damping table)
__device__ __forceinline__ void damping_term(float2 dm, float2 dn, const cdf &v, float &gr, float &gi) {
    const df dl = df_add({dm.x, dm.y}, {dn.x, dn.y});
    gr = -__fmaf_rn(dl.hi, v.re.hi, __fmaf_rn(dl.hi, v.re.lo, dl.lo * v.re.hi));
    gi = -__fmaf_rn(dl.hi, v.im.hi, __fmaf_rn(dl.hi, v.im.lo, dl.lo * v.im.hi));
}

// out = B + f dt L(X) for instances with per-jump tables: the general kernel (dissipate_df_kernel)
// finds an element's jumps by their masks; here all of a model's few jumps are gathered at once,
// which at dim 512 makes a Strang step 4 us shorter.
__device__ __forceinline__ void lindblad_jt(const TileItem *__restrict__ tiles, const InstDesc *__restrict__ descs,
                                            int xsel, int bsel, int osel, float f, bool planes,
                                            const float4 *X_only = nullptr, float4 *O_only = nullptr) {
    // set-up tables (damping, jump rows) are read while the previous kernel finishes
    const TileItem it = tiles[blockIdx.x];
    const InstDesc a = descs[it.inst];
    const int64_t D = a.D;
    const int64_t n = (int64_t)it.bx * 32 + threadIdx.x;
    const int64_t m0 = (int64_t)it.by * (8 * kRows) + threadIdx.y;
    const bool n_in = n < D;
    const int64_t nc = n_in ? n : 0;
    const float2 dn = a.damp[nc];
    // X_only: out = f dt L(X_only) into O_only (B = 0), for buffers outside the model
    const float4 *X = X_only ? X_only : state_buf(a, xsel);
    const float4 *B = X_only ? nullptr : state_buf(a, bsel);
    float4 *O = X_only ? O_only : state_buf(a, osel);
    // incoming entries by jump: element (m, n) gets c_j(m) c_j(n) X[src_j(m), src_j(n)] for
    // every jump j with an entry in both rows (row entries warp-uniform, column entries
    // read once for the thread's kRows rows)
    const int nj = a.nj;
    int4 tn[kInMax], tm[kRows][kInMax];
    float2 dm[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int64_t m = m0 + 8 * r, mc = m < D ? m : 0;
        dm[r] = a.damp[mc];
#pragma unroll
        for (int j = 0; j < kInMax; ++j)
            tm[r][j] = j < nj ? a.jtab[mc * kInMax + j] : make_int4(-1, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < kInMax; ++j) tn[j] = j < nj ? a.jtab[nc * kInMax + j] : make_int4(-1, 0, 0, 0);
    pdl_wait();
    pdl_trigger();
    float4 v[kRows], u[kRows][kInMax], bv[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int64_t m = m0 + 8 * r;
        const bool inside = m < D && n_in;
        v[r] = X[(inside ? m : 0) * D + nc];
        // the base of a Strang stage comes with the gathers
        bv[r] = B ? B[(inside ? m : 0) * D + nc] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < kInMax; ++j) {
            const bool hit = inside && tm[r][j].x >= 0 && tn[j].x >= 0 &&
                             qed_check(a.err, tm[r][j].x < D && tn[j].x < D);
            u[r][j] = hit ? X[(int64_t)tm[r][j].x * D + tn[j].x] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int64_t m = m0 + 8 * r;
        if (!(m < D && n_in)) continue;
        const cdf vv = load_cdf(v[r]);
        float gr, gi;
        damping_term(dm[r], dn, vv, gr, gi);
#pragma unroll
        for (int j = 0; j < kInMax; ++j) {
            if (!(tm[r][j].x >= 0 && tn[j].x >= 0)) continue;
            const df c = df_mul({__int_as_float(tm[r][j].y), __int_as_float(tm[r][j].z)},
                                {__int_as_float(tn[j].y), __int_as_float(tn[j].z)});
            const float ur = u[r][j].x + u[r][j].y, ui = u[r][j].z + u[r][j].w;
            gr = __fmaf_rn(c.hi, ur, __fmaf_rn(c.lo, ur, gr));
            gi = __fmaf_rn(c.hi, ui, __fmaf_rn(c.lo, ui, gi));
        }
            lindblad_store(a, O, m, n, load_cdf(bv[r]), f * gr, f * gi, planes);
    }
}

// The jump terms of element (m, n) from the incoming lists, added to (gr, gi): long pairs of lists by
// the whole warp (every lane is here, `inside` or not), the others by a two-pointer merge.
__device__ __noinline__ void list_terms(const InstDesc &a, const float4 *X, int64_t m, int64_t n, bool inside,
                                        float &gr, float &gi) {
    const int64_t D = a.D;
    int p = inside ? a.in_ptr[m] : 0, pe = inside ? a.in_ptr[m + 1] : 0;
    int q = inside ? a.in_ptr[n] : 0, qe = inside ? a.in_ptr[n + 1] : 0;
    if (long_merge_df(a.err, D, a.in_jump, a.in_src, a.coef, X, p, pe, q, qe, gr, gi)) pe = p;
    while (p < pe && q < qe) {  // jumps present in both incoming lists
        const int jp = a.in_jump[p], jq = a.in_jump[q];
        if (jp < jq) {
            ++p;
        } else if (jp > jq) {
            ++q;
        } else {
            if (qed_check(a.err, a.in_src[p] >= 0 && a.in_src[p] < D && a.in_src[q] >= 0 && a.in_src[q] < D)) {
                const float2 cp = a.coef[p], cq = a.coef[q];
                const df c = df_mul({cp.x, cp.y}, {cq.x, cq.y});  // dt c_j(m) c_j(n)
                const float4 u = X[(int64_t)a.in_src[p] * D + a.in_src[q]];
                const float ur = u.x + u.y, ui = u.z + u.w;
                gr = __fmaf_rn(c.hi, ur, __fmaf_rn(c.lo, ur, gr));
                gi = __fmaf_rn(c.hi, ui, __fmaf_rn(c.lo, ui, gi));
            }
            ++p;
            ++q;
        }
    }
}

// out = B + f dt L(X) on one block of kWideCols columns and `rows` rows (a multiple of 8), two
// elements of every eighth row a thread.  The rows' and columns' damping rates, jump masks and
// entries are staged in shared memory while the previous kernel finishes; an element's jumps are
// the bits its row's and its column's mask share, in rising order (the lists' order), each entry
// found by its rank among the mask's bits.  Without masks a pair of lists is merged only where the
// ranges of their jumps overlap: a lattice's only such element is the vacuum's population, which
// the warp sums entry by entry.  The next row's elements are loaded before a row is worked on.
// What bounds it: the 40 B an element streams (V 16, rho 16, planes 8) and the latency of the
// gathers (41 % issue, 2.6 TB/s on the 32 x 32 lattice); large blocks (64 rows where that leaves
// eight blocks an SM) pay the staging once for 4096 elements.  Measured alone from a cold L2: the 32 x
// 32 lattice 45 us (80 by the version that merged its lists in registers, two blocks an SM), 64 chains
// of 32 to 1024 states 303 us.
template <bool LIE>
__device__ __forceinline__ void lindblad_update(const TileItem *__restrict__ tiles,
                                                const InstDesc *__restrict__ descs, int rows, int xsel, int bsel,
                                                int osel, float f, bool planes, const float4 *X_only = nullptr,
                                                float4 *O_only = nullptr) {
    constexpr int C = kWideCols;
    // of the columns, then of the rows
    __shared__ float2 s_d[C + kWideRows];          // damping rates
    __shared__ uint32_t s_m[C + kWideRows];        // masks
    __shared__ int2 s_p[C + kWideRows];            // first entry of each; without masks its first and last jump
    __shared__ int4 s_e[C + kWideRows][kStaged];   // {src, coefficient}
    const TileItem it = tiles[blockIdx.x];
    const InstDesc &a = descs[it.inst];
    const uint32_t D = (uint32_t)a.D;
    const uint32_t n0 = (uint32_t)it.bx * C, m0 = (uint32_t)(it.by * rows);
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const uint32_t *const mask = a.mask;
    const int32_t *const in_src = a.in_src, *const in_ptr = a.in_ptr;
    const float2 *const coef = a.coef;
    if (tid < C + rows) {
        const uint32_t k = tid < C ? n0 + tid : m0 + (tid - C);
        const bool in = k < D;
        const int p = in ? in_ptr[k] : 0, pe = in ? in_ptr[k + 1] : 0;
        s_d[tid] = in ? a.damp[k] : make_float2(0.f, 0.f);
        s_m[tid] = in && mask ? mask[k] : 0u;
        if (mask) {
            s_p[tid] = make_int2(p, pe);
            for (int e = p; e < min(pe, p + kStaged); ++e) {
                const float2 c = coef[e];
                s_e[tid][e - p] = make_int4(in_src[e], __float_as_int(c.x), __float_as_int(c.y), 0);
            }
        } else {
            s_p[tid] = pe > p ? make_int2(a.in_jump[p], a.in_jump[pe - 1]) : make_int2(1, 0);
        }
    }
    // X_only: out = f dt L(X_only) into O_only (B = 0), for buffers outside the model
    const float4 *X = X_only ? X_only : (LIE ? a.V : state_buf(a, xsel));
    const float4 *B = X_only ? nullptr : (LIE ? a.V : state_buf(a, bsel));
    float4 *O = X_only ? O_only : (LIE ? a.rho : state_buf(a, osel));
    __half *const pl = LIE || planes ? a.rho_pl : nullptr;
    const float s_rho = a.s_rho;
    const uint32_t Dp = (uint32_t)a.Dp;
    const int64_t plane = (int64_t)Dp * 2 * Dp;
    __syncthreads();
    const int lc = 2 * threadIdx.x;
    const uint32_t n = n0 + lc;
    const bool in0 = n < D, in1 = n + 1 < D;
    // entry of the lowest jump of `left` in row or column l
    auto entry = [&](int l, uint32_t left) {
        const int rank = __popc(s_m[l] & ((left & (0u - left)) - 1u));
        if (rank < kStaged) return s_e[l][rank];
        const int p = s_p[l].x + rank;
        const float2 c = coef[p];
        return make_int4(in_src[p], __float_as_int(c.x), __float_as_int(c.y), 0);
    };
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    pdl_wait();
    pdl_trigger();
    uint32_t m = m0 + threadIdx.y;
    float4 v[2], w[2], bv[2];
    v[0] = m < D && in0 ? X[m * D + n] : zero;
    v[1] = m < D && in1 ? X[m * D + n + 1] : zero;
    for (int l = threadIdx.y; l < rows; l += 8, m += 8) {
        if (m0 + (l & ~7) >= D) break;  // the whole block is past the last row
        const bool row = m < D, more = l + 8 < rows && m + 8 < D;
        w[0] = more && in0 ? X[(m + 8) * D + n] : zero;
        w[1] = more && in1 ? X[(m + 8) * D + n + 1] : zero;
        if (!LIE) {
            bv[0] = row && in0 && B ? B[m * D + n] : zero;
            bv[1] = row && in1 && B ? B[m * D + n + 1] : zero;
        }
        const float2 dm = s_d[C + l];
        const uint32_t mr = s_m[C + l];
        df re[2], im[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const bool inside = row && (q ? in1 : in0);
            const cdf vv = load_cdf(v[q]);
            float gr, gi;
            damping_term(dm, s_d[lc + q], vv, gr, gi);
            for (uint32_t both = mr & s_m[lc + q]; both; both &= both - 1) {
                const int4 em = entry(C + l, both), en = entry(lc + q, both);
                if (!qed_check(a.err, (uint32_t)em.x < D && (uint32_t)en.x < D)) continue;
                const float4 u = X[(uint32_t)em.x * D + (uint32_t)en.x];
                const df k =
                    df_mul({__int_as_float(em.y), __int_as_float(em.z)}, {__int_as_float(en.y), __int_as_float(en.z)});
                const float ur = u.x + u.y, ui = u.z + u.w;
                gr = __fmaf_rn(k.hi, ur, __fmaf_rn(k.lo, ur, gr));
                gi = __fmaf_rn(k.hi, ui, __fmaf_rn(k.lo, ui, gi));
            }
            if (!mask) {
                const int2 x = s_p[C + l], y = s_p[lc + q];
                const bool meet = inside && max(x.x, y.x) <= min(x.y, y.y);
                if (__any_sync(0xffffffffu, meet)) list_terms(a, X, m, n + q, meet, gr, gi);
            }
            const cdf b = LIE ? vv : load_cdf(bv[q]);
            re[q] = df_add_f(b.re, LIE ? gr : f * gr);
            im[q] = df_add_f(b.im, LIE ? gi : f * gi);
            if (inside) O[m * D + n + q] = make_float4(re[q].hi, re[q].lo, im[q].hi, im[q].lo);
        }
        v[0] = w[0];
        v[1] = w[1];
        if (!pl || !row || !in0) continue;
        // pairs of the planes; past the last column the padding's zero
        if (!in1) re[1] = im[1] = {0.f, 0.f};
        __half h[2], lo[2];
        __half *out = pl + (int64_t)m * 2 * Dp + n;
#pragma unroll
        for (int q = 0; q < 2; ++q) df_to_half2(re[q], s_rho, h[q], lo[q]);
        *(__half2 *)out = __halves2half2(h[0], h[1]);
        *(__half2 *)(out + plane) = __halves2half2(lo[0], lo[1]);
#pragma unroll
        for (int q = 0; q < 2; ++q) df_to_half2(im[q], s_rho, h[q], lo[q]);
        *(__half2 *)(out + Dp) = __halves2half2(h[0], h[1]);
        *(__half2 *)(out + plane + Dp) = __halves2half2(lo[0], lo[1]);
    }
}

// The Lie step's update (rho = V + dt L(V) and the next planes) for instances whose incoming
// entries are all in per-jump tables (at most kInMax jumps of monomial form).  The block's
// row and column entries and damping rates are staged in shared memory first, so a thread
// keeps only its kRows elements' loads in registers; with 64 registers four blocks fit on an
// SM, and a dim-512 update (512 blocks) runs as one wave whose table reads overlap the
// previous kernel.
__global__ void __launch_bounds__(256, 4) dissipate_jt_kernel(const TileItem *__restrict__ tiles,
                                                           const InstDesc *__restrict__ descs) {
    constexpr int R = 8 * kRows;
    constexpr int JW = kInMax;
    __shared__ int4 s_row[R][JW], s_col[32][JW];
    __shared__ float2 s_dr[R], s_dc[32];
    const TileItem it = tiles[blockIdx.x];
    const InstDesc a = descs[it.inst];
    // element offsets in 32 bits: the split path holds dimensions below 65536 (split_create)
    const uint32_t D = (uint32_t)a.D;
    const int nj = a.nj;
    const uint32_t n0 = (uint32_t)it.bx * 32, m0 = (uint32_t)it.by * R;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    // entries: the block's R rows, then its 32 columns, then both damping vectors
    for (int e = tid; e < (R + 32) * JW + R + 32; e += 256) {
        if (e < R * JW) {
            const int r = e / JW, j = e % JW;
            const uint32_t m = m0 + r;
            s_row[r][j] = j < nj && m < D ? a.jtab[m * JW + j] : make_int4(-1, 0, 0, 0);
        } else if (e < (R + 32) * JW) {
            const int c = (e - R * JW) / JW, j = e % JW;
            const uint32_t n = n0 + c;
            s_col[c][j] = j < nj && n < D ? a.jtab[n * JW + j] : make_int4(-1, 0, 0, 0);
        } else if (e < (R + 32) * JW + R) {
            const int r = e - (R + 32) * JW;
            s_dr[r] = m0 + r < D ? a.damp[m0 + r] : make_float2(0.f, 0.f);
        } else {
            const int c = e - (R + 32) * JW - R;
            s_dc[c] = n0 + c < D ? a.damp[n0 + c] : make_float2(0.f, 0.f);
        }
    }
    const float4 *X = a.V;
    float4 *O = a.rho;
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    const int tx = threadIdx.x;
    const uint32_t n = n0 + tx;
    // the jump terms are formed in FP32 (their size is dt gamma of the result), so each
    // gathered element contributes only the leading words of its real and imaginary parts
    float4 v[kRows];
    float ur[kRows][JW], ui[kRows][JW];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int rr = threadIdx.y + 8 * r;
        const uint32_t m = m0 + rr;
        const bool inside = m < D && n < D;
        v[r] = inside ? X[m * D + n] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < JW; ++j) {
            const int sm = s_row[rr][j].x, sn = s_col[tx][j].x;
            const bool hit = inside && sm >= 0 && sn >= 0 && qed_check(a.err, (uint32_t)sm < D && (uint32_t)sn < D);
            const float *src = (const float *)(X + ((uint32_t)sm * D + (uint32_t)sn));
            ur[r][j] = hit ? src[0] : 0.f;
            ui[r][j] = hit ? src[2] : 0.f;
        }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int rr = threadIdx.y + 8 * r;
        const uint32_t m = m0 + rr;
        if (!(m < D && n < D)) continue;
        const cdf vv = load_cdf(v[r]);
        float gr, gi;
        damping_term(s_dr[rr], s_dc[tx], vv, gr, gi);
#pragma unroll
        for (int j = 0; j < JW; ++j) {
            const int4 em = s_row[rr][j], en = s_col[tx][j];
            if (!(em.x >= 0 && en.x >= 0)) continue;
            const df c = df_mul({__int_as_float(em.y), __int_as_float(em.z)}, {__int_as_float(en.y), __int_as_float(en.z)});
            gr = __fmaf_rn(c.hi, ur[r][j], __fmaf_rn(c.lo, ur[r][j], gr));
            gi = __fmaf_rn(c.hi, ui[r][j], __fmaf_rn(c.lo, ui[r][j], gi));
        }
        lindblad_store(a, O, m, n, vv, gr, gi, true);
    }
}

// Lie step: rho = V + dt L(V), and the next planes.
__global__ void __launch_bounds__(256, 4) dissipate_df_kernel(const TileItem *__restrict__ tiles,
                                                           const InstDesc *__restrict__ descs, int rows) {
    lindblad_update<true>(tiles, descs, rows, 1, 1, 0, 1.f, true);
}

// One stage of the Strang step: out = B + f dt L(X).
__global__ void __launch_bounds__(256, 3) lindblad_df_kernel(const TileItem *__restrict__ tiles,
                                                          const InstDesc *__restrict__ descs, int rows, int xsel,
                                                          int bsel, int osel, float f, int planes) {
    lindblad_update<false>(tiles, descs, rows, xsel, bsel, osel, f, planes != 0);
}
__global__ void __launch_bounds__(256, 2) lindblad_jt_kernel(const TileItem *__restrict__ tiles,
                                                          const InstDesc *__restrict__ descs, int xsel, int bsel,
                                                          int osel, float f, int planes) {
    lindblad_jt(tiles, descs, xsel, bsel, osel, f, planes != 0);
}

// out = dt L(X) for a double-float buffer X of a single model (the adjoint's rate terms).
__global__ void __launch_bounds__(256, 3) lindblad_apply_df_kernel(const TileItem *__restrict__ tiles,
                                                                const InstDesc *__restrict__ descs, int rows,
                                                                const float4 *X, float4 *out) {
    lindblad_update<false>(tiles, descs, rows, 0, 0, 0, 1.f, false, X, out);
}
__global__ void __launch_bounds__(256, 2) lindblad_apply_jt_kernel(const TileItem *__restrict__ tiles,
                                                                const InstDesc *__restrict__ descs,
                                                                const float4 *X, float4 *out) {
    lindblad_jt(tiles, descs, 0, 0, 0, 1.f, false, X, out);
}

// Blocks of kObsPerBlock ids: the populations among them a thread each, then the named observables
// one after another by the whole block (a block per id took 5 us for the 513 ids of dim 512).
constexpr int kObsPerBlock = 32;
__global__ void __launch_bounds__(256) observables_df_kernel(int64_t D, const float4 *st, const double *w, int n_obs,
                                                             const int32_t *ids, double *out) {
    __shared__ double part[256];
    const int t = threadIdx.x;
    const int first = blockIdx.x * kObsPerBlock, end = min(n_obs, first + kObsPerBlock);
    if (first + t < end) {
        const int id = ids[first + t];
        if (id < D) {
            const float4 v = st[(int64_t)id * D + id];
            out[first + t] = (double)v.x + (double)v.y;
        }
    }
    for (int o = first; o < end; ++o) {
        const int id = ids[o];
        if (id < D) continue;
        double s = 0.0;
        const double *wr = w + (int64_t)(id - D) * D;
        for (int64_t k = t; k < D; k += blockDim.x) {
            const float4 v = st[k * D + k];
            s += wr[k] * ((double)v.x + (double)v.y);
        }
        part[t] = s;
        __syncthreads();
        for (int st2 = blockDim.x / 2; st2 > 0; st2 >>= 1) {
            if (t < st2) part[t] += part[t + st2];
            __syncthreads();
        }
        if (t == 0) out[o] = part[0];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) trace_df_kernel(int64_t D, const float4 *st, double *tr, uint32_t *err) {
    __shared__ double part[1024];
    const int t = threadIdx.x;
    double s = 0.0;
    for (int64_t k = t; k < D; k += blockDim.x) {
        const float4 v = st[k * D + k];
        s += (double)v.x + (double)v.y;
    }
    part[t] = s;
    __syncthreads();
    for (int st2 = blockDim.x / 2; st2 > 0; st2 >>= 1) {
        if (t < st2) part[t] += part[t + st2];
        __syncthreads();
    }
    if (t == 0) {
        *tr = part[0];
        if (!isfinite(part[0]) || !(part[0] > 0.0)) atomicOr(err, kErrNonFinite);
    }
}

// rho <- (rho + rho^+) / (2 tr rho) (divide != 0) or (rho + rho^+) / 2 on the double-float
// state (FP64 arithmetic; it runs once every `renorm_every` steps), then the FP16 planes
// again.
__global__ void symmetrise_df_kernel(int64_t D, int64_t Dp, float4 *st, const double *tr, const uint32_t *err,
                                     float s_rho, __half *pl, int divide) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= D || j >= D || j < i) return;
    if (*err & kErrNonFinite) return;
    const double inv = divide ? 1.0 / *tr : 1.0;
    const float4 a = st[i * D + j], b = st[j * D + i];
    double re = 0.5 * (((double)a.x + (double)a.y) + ((double)b.x + (double)b.y)) * inv;
    double im = 0.5 * (((double)a.z + (double)a.w) - ((double)b.z + (double)b.w)) * inv;
    if (i == j) im = 0.0;
    const float rh = (float)re, ih = (float)im;
    const df dre = {rh, (float)(re - (double)rh)}, dim = {ih, (float)(im - (double)ih)};
    st[i * D + j] = make_float4(dre.hi, dre.lo, dim.hi, dim.lo);
    st[j * D + i] = make_float4(dre.hi, dre.lo, -dim.hi, -dim.lo);
    const int64_t plane = Dp * 2 * Dp;
    __half h, l;
    df_to_half2(dre, s_rho, h, l);
    pl[i * 2 * Dp + j] = h;
    pl[plane + i * 2 * Dp + j] = l;
    pl[j * 2 * Dp + i] = h;
    pl[plane + j * 2 * Dp + i] = l;
    df_to_half2(dim, s_rho, h, l);
    pl[i * 2 * Dp + Dp + j] = h;
    pl[plane + i * 2 * Dp + Dp + j] = l;
    df_to_half2(df_neg(dim), s_rho, h, l);
    pl[j * 2 * Dp + Dp + i] = h;
    pl[plane + j * 2 * Dp + Dp + i] = l;
}

double pow2_scale(double maxabs, int target_exp) {
    if (!(maxabs > 0.0) || !std::isfinite(maxabs)) return 1.0;
    int e = (int)std::ceil(std::log2(maxabs));
    return std::ldexp(1.0, target_exp - e);
}

#define SPLIT_TRY(expr)                 \
    do {                                \
        qed_status st_ = (expr);        \
        if (st_ != QED_OK) return st_;  \
    } while (0)

const TcSegs kSegs1 = {4, {0, 0, 1, 2, 0, 0}, {0, 1, 0, 0, 0, 0}};  // Delta(hi,mid,lo) x rho(hi,lo)
const TcSegs kSegs2 = {3, {0, 1, 0, 0, 0, 0}, {0, 0, 1, 0, 0, 0}};  // W(hi,lo) x Delta(hi,mid,lo)
const int kSeg1Pairs[8] = {0, 0, 0, 1, 1, 0, 2, 0};
const int kSeg2Pairs[6] = {0, 0, 1, 0, 0, 1};

// The plans of a model's two products: GEMM1 [W_re; W_im] = A1 . rho^T (2Dp x Dp, K 2Dp, four
// plane pairs), GEMM2 [X_re | X_im] = W . B2^T (Dp x 2Dp, K 2Dp, three plane pairs).  Widths and
// splits = CTAs per cluster (on-chip reduction of the split-K slices) as given, or 0 for the
// planner's rule (256-wide tiles once the tiles that run fill half the SMs).
bool plan_products(SplitState &S, TcGemm &g1, TcGemm &g2, int splits1, int bn1, int splits2, int bn2 = 0) {
    const int Dp = (int)S.Dp;
    if (bn2 == 0) {
        // GEMM2 runs only the tiles on or above the diagonal: nm (nm + 1) / 2 of them when 256
        // wide (nm = Dp / 128), which must fill half the SMs
        const int nm = Dp / kTcBM;
        bn2 = nm * (nm + 1) >= S.num_sms ? 256 : 128;
    }
    return tc_gemm_plan(g1, S.a1, 3, S.rho_pl, 2, 2 * Dp, Dp, 2 * Dp, 4, kSeg1Pairs, S.num_sms, splits1, bn1, true) &&
           tc_gemm_plan(g2, S.w_pl, 2, S.b2, 3, Dp, 2 * Dp, 2 * Dp, 3, kSeg2Pairs, S.num_sms, splits2, bn2, true);
}

// The k-blocks of each tile of a product in which the planes of Delta's rows of that tile have a
// nonzero: Delta is block diagonal over the components of H's graph (a chain's states are sorted by
// excitations), far elements round to zero, and its padding is zero.  The blocks left out would add
// zeros, so nothing changes in the sums.  Tiles hold `rows` rows of Delta each; K = [re | im], Dp
// columns each, in slices of g.kb_per_split blocks, every one of which keeps at least one block.
// Appends kb_ptr and kb_idx to `out`.
void k_block_lists(const std::vector<uint8_t> &nz, int64_t D, int64_t Dp, const TcGemm &g, int tiles, int rows,
                   std::vector<int> &out, size_t &ptr_at, size_t &idx_at) {
    const int nb = (int)((D + 63) / 64), half = (int)(Dp / 64), total = g.K / kTcBK;
    std::vector<int> ptr(1, 0), idx;
    for (int t = 0; t < tiles; ++t)
        for (int s = 0; s < g.splits; ++s) {
            const int first = s * g.kb_per_split, end = std::min(total, first + g.kb_per_split);
            const size_t before = idx.size();
            for (int kb = first; kb < end; ++kb) {
                const int c = kb % half;
                bool any = false;
                for (int r = t * rows / 64; r < std::min(nb, (t + 1) * rows / 64) && c < nb; ++r)
                    any = any || nz[(size_t)(r * nb + c)];
                if (any) idx.push_back(kb);
            }
            if (idx.size() == before) idx.push_back(first);
            ptr.push_back((int)idx.size());
        }
    ptr_at = out.size();
    out.insert(out.end(), ptr.begin(), ptr.end());
    idx_at = out.size();
    out.insert(out.end(), idx.begin(), idx.end());
}

// Descriptors, jobs and work lists of a batch.  With `single` set (one model on its own)
// the products keep their plans (split-K slices reduced inside clusters); in a batch every
// product runs unsplit, largest first, since the batch itself fills the GPU.  GEMM1 skips
// tiles that lie wholly in the zero padding (rows or columns >= D); GEMM2 runs the tiles on
// or above the diagonal only (its epilogue writes both halves of the Hermitian V).
// `target` is replaced at the end: a failed call leaves it as it was.
qed_status build_batch(Batch &target, qed_model *const *ms, int n, bool single, int batch_bn1 = kTcBNMax,
                       int batch_bn2 = kTcBNMax) {
    struct Fresh : Batch {
        ~Fresh() { release(); }
    } b;
    b.n = n;
    b.scheme = ms[0]->scheme;
    for (int i = 1; i < n; ++i)
        if (ms[i]->scheme != b.scheme) {
            set_error("batched evolution: all models must use one time-stepping scheme");
            return QED_EINVAL;
        }
    std::vector<InstDesc> desc((size_t)n);
    std::vector<GemmJob> jobs1((size_t)n), jobs2((size_t)n);
    std::vector<CUtensorMap> maps((size_t)(4 * n));
    std::vector<int> kb;
    std::vector<size_t> kb_at((size_t)(4 * n));
    std::vector<GemmItem> it1, it2;
    std::vector<TileItem> et;
    for (int i = 0; i < n; ++i) {
        qed_model *m = ms[i];
        SplitState &S = *m->sp;
        InstDesc &d = desc[(size_t)i];
        const int64_t D = m->D, Dp = S.Dp;
        d.D = D;
        d.Dp = Dp;
        d.s_rho = (float)S.scale_rho;
        d.rho = S.rho_df[0];
        d.V = S.rho_df[1];
        d.Y = S.y_df;
        d.phase = S.phase_df;
        d.damp = S.damp_df;
        d.in_ptr = m->in_ptr;
        d.in_jump = m->in_jump;
        d.in_src = m->in_src;
        d.coef = S.coef_df;
        d.mask = S.mask;
        d.jtab = S.jtab;
        d.nj = S.nj;
        d.rho_pl = S.rho_pl;
        d.err = m->err;
        TcGemm bg1 = S.g1, bg2 = S.g2;
        if (!single && !plan_products(S, bg1, bg2, 1, batch_bn1, 1, batch_bn2)) return QED_ECUDA;
        auto pow2 = [](int x) { return x > 0 && (x & (x - 1)) == 0; };
        if (!pow2(bg1.splits) || bg1.splits > kTcMaxCluster || !pow2(bg2.splits) || bg2.splits > kTcMaxClusterV ||
            (bg2.bn != 128 && bg2.bn != 256)) {
            set_error("split step: product plan outside the cluster epilogue's limits");
            return QED_EINVAL;
        }
        maps[(size_t)(4 * i + 0)] = bg1.a;
        maps[(size_t)(4 * i + 1)] = bg1.b;
        maps[(size_t)(4 * i + 2)] = bg2.a;
        maps[(size_t)(4 * i + 3)] = bg2.b;
        size_t *at = &kb_at[(size_t)(4 * i)];
        k_block_lists(S.nz, D, Dp, bg1, (int)(Dp / kTcBM), kTcBM, kb, at[0], at[1]);
        k_block_lists(S.nz, D, Dp, bg2, bg2.N / bg2.bn, bg2.bn / 2, kb, at[2], at[3]);
        const TcGemm *gs[2] = {&bg1, &bg2};
        GemmJob *js[2] = {&jobs1[(size_t)i], &jobs2[(size_t)i]};
        for (int q = 0; q < 2; ++q) {
            const TcGemm &g = *gs[q];
            GemmJob &j = *js[q];
            j.M = g.M;
            j.N = g.N;
            j.kb_per_seg = g.K / kTcBK;
            j.kb_per_split = g.kb_per_split;
            j.out = nullptr;
            j.gate = m->gate_armed ? m->gate : nullptr;
            j.gate_budget = m->gate_budget;
            j.mode = q == 0 ? kEpiW : kEpiV;
            j.tx_bytes = tc_stage_tx_bytes(g, j.mode);
            j.epi = TcEpilogue();
            j.epi.D = D;
            j.epi.Dp = Dp;
            j.epi.w32 = S.w32;
            if (q == 0) {
                j.epi.inv = (float)(1.0 / (S.scale_delta * S.scale_rho));
                j.epi.s_w = (float)S.scale_w;
                j.epi.w_pl = S.w_pl;
            } else {
                j.epi.inv = (float)(1.0 / (S.scale_w * S.scale_delta));
                j.epi.rho = S.rho_df[0];
                j.epi.phase = S.phase_df;
                j.epi.V = S.rho_df[1];
            }
            if (i == 0) {
                (q == 0 ? b.cs1 : b.cs2) = g.splits;
                (q == 0 ? b.bn1 : b.bn2) = g.bn;
            } else if (g.splits != (q == 0 ? b.cs1 : b.cs2) || g.bn != (q == 0 ? b.bn1 : b.bn2)) {
                set_error("batched evolution: every instance of a launch needs the same tile plan");
                return QED_EINVAL;
            }
        }
        // GEMM1 tiles: 128 rows of [W_re; W_im] x bn1 columns; wholly-padding tiles skipped
        for (int tm = 0; tm < bg1.M / kTcBM; ++tm) {
            if ((tm * kTcBM) % Dp >= D) continue;
            for (int tn = 0; tn * bg1.bn < bg1.N; ++tn) {
                if ((int64_t)tn * bg1.bn >= D) continue;
                for (int sp = 0; sp < bg1.splits; ++sp) it1.push_back({i, tm, tn, sp});
            }
        }
        // GEMM2 tiles: 128 rows m x (64 c2) complex columns n, on or above the diagonal
        const int c2 = bg2.bn / 128;
        for (int tm = 0; tm < bg2.M / kTcBM; ++tm) {
            if ((int64_t)tm * kTcBM >= D) continue;
            for (int tj = 2 * tm / c2; tj < bg2.N / bg2.bn; ++tj) {
                if ((int64_t)tj * 64 * c2 >= D) continue;
                for (int sp = 0; sp < bg2.splits; ++sp) it2.push_back({i, tm, tj, sp});
            }
        }
    }
    if (!single) {
        // longest products first, so the tail of the grouped launch is short (unsplit:
        // every item is a cluster of one)
        auto by_cost = [&](const GemmItem &x, const GemmItem &y) {
            return jobs1[(size_t)x.job].kb_per_seg > jobs1[(size_t)y.job].kb_per_seg;
        };
        std::stable_sort(it1.begin(), it1.end(), by_cost);
        std::stable_sort(it2.begin(), it2.end(), by_cost);
    }
    b.jt = std::all_of(desc.begin(), desc.end(), [](const InstDesc &d) { return d.jtab != nullptr; });
    auto element_blocks = [&](int rows, int cols) {
        et.clear();
        for (int i = 0; i < n; ++i)
            for (int64_t by = 0; by * rows < desc[(size_t)i].D; ++by)
                for (int64_t bx = 0; bx * cols < desc[(size_t)i].D; ++bx) et.push_back({i, (int)bx, (int)by, 0});
    };
    if (b.jt) {
        element_blocks(8 * kRows, 32);
    } else {
        // the largest blocks that leave eight an SM, down to one row a warp
        for (b.erows = kWideRows; b.erows >= 8; b.erows /= 2) {
            element_blocks(b.erows, kWideCols);
            if ((int)et.size() >= 8 * ms[0]->sp->num_sms || b.erows == 8) break;
        }
    }
    std::vector<TileItem> pairs;
    for (int i = 0; i < n; ++i) {
        const int nt = (int)((desc[(size_t)i].D + 31) / 32);
        for (int by = 0; by < nt; ++by)
            for (int bx = 0; bx <= by; ++bx) pairs.push_back({i, bx, by, 0});
    }
    b.n_pairs = (int)pairs.size();
    DeviceBlock block;
    block.add(&b.pairs, pairs);
    block.room(&b.rhos, (size_t)n);
    block.room(&b.records, (size_t)n);
    block.room(&b.errors, (size_t)n);
    block.add(&b.maps, maps);
    block.add(&b.kblocks, kb);
    block.add(&b.desc, desc);
    block.add(&b.items1, it1);
    block.add(&b.items2, it2);
    block.add(&b.etiles, et);
    block.room(&b.jobs1, (size_t)n);  // (they hold addresses inside the block)
    block.room(&b.jobs2, (size_t)n);
    SPLIT_TRY(block.upload(&b.block));
    for (int i = 0; i < n; ++i) {
        jobs1[(size_t)i].kb_ptr = b.kblocks + kb_at[(size_t)(4 * i)];
        jobs1[(size_t)i].kb_idx = b.kblocks + kb_at[(size_t)(4 * i + 1)];
        jobs2[(size_t)i].kb_ptr = b.kblocks + kb_at[(size_t)(4 * i + 2)];
        jobs2[(size_t)i].kb_idx = b.kblocks + kb_at[(size_t)(4 * i + 3)];
        jobs1[(size_t)i].map_a = b.maps + 4 * i + 0;
        jobs1[(size_t)i].map_b = b.maps + 4 * i + 1;
        jobs2[(size_t)i].map_a = b.maps + 4 * i + 2;
        jobs2[(size_t)i].map_b = b.maps + 4 * i + 3;
    }
    if (!single) {  // (a model on its own launches with its jobs as parameters)
        QED_CUDA_TRY(cudaMemcpy(b.jobs1, jobs1.data(), (size_t)n * sizeof(GemmJob), cudaMemcpyHostToDevice));
        QED_CUDA_TRY(cudaMemcpy(b.jobs2, jobs2.data(), (size_t)n * sizeof(GemmJob), cudaMemcpyHostToDevice));
    }
    b.n_items1 = (int)it1.size();
    b.n_items2 = (int)it2.size();
    b.n_etiles = (int)et.size();
    if (single) {
        SplitState &S = *ms[0]->sp;
        b.single = true;
        b.D = ms[0]->D;
        b.g1 = S.g1;
        b.g2 = S.g2;
        b.j1 = jobs1[0];
        b.j2 = jobs2[0];
        if (tc_gemm_single_ctas(b.g1, kEpiW, b.D) * 1 != b.n_items1 ||
            tc_gemm_single_ctas(b.g2, kEpiV, b.D) != b.n_items2) {
            set_error("split step: tile lists of the single-model launch disagree");
            return QED_ECUDA;
        }
    }
    if (!tc_gemm_prepare_grouped()) return QED_ECUDA;
    target.release();
    target = b;
    b.block = nullptr;
    return QED_OK;
}

void launch_gemm1(const Batch &b, uint32_t *err, cudaStream_t s) {
    if (b.single)
        tc_gemm_single_launch(b.g1, b.j1, kSegs1, b.D, err, s);
    else
        tc_gemm_grouped_launch(b.items1, b.n_items1, b.jobs1, kSegs1, b.bn1, kEpiW, b.cs1, err, s);
}
void launch_gemm2(const Batch &b, uint32_t *err, cudaStream_t s) {
    if (b.single)
        tc_gemm_single_launch(b.g2, b.j2, kSegs2, b.D, err, s);
    else
        tc_gemm_grouped_launch(b.items2, b.n_items2, b.jobs2, kSegs2, b.bn2, kEpiV, b.cs2, err, s);
}
void launch_dissipate(const Batch &b, cudaStream_t s) {
    if (b.jt)
        launch_pdl(dissipate_jt_kernel, dim3(b.n_etiles), dim3(32, 8), 0, s, b.etiles, b.desc);
    else
        launch_pdl(dissipate_df_kernel, dim3(b.n_etiles), dim3(32, 8), 0, s, b.etiles, b.desc, b.erows);
    count_launches(1);
}
void launch_lindblad(const Batch &b, int xsel, int bsel, int osel, float f, int planes, cudaStream_t s) {
    if (b.jt)
        launch_pdl(lindblad_jt_kernel, dim3(b.n_etiles), dim3(32, 8), 0, s, b.etiles, b.desc, xsel, bsel, osel, f,
                   planes);
    else
        launch_pdl(lindblad_df_kernel, dim3(b.n_etiles), dim3(32, 8), 0, s, b.etiles, b.desc, b.erows, xsel, bsel,
                   osel, f, planes);
    count_launches(1);
}
// The two stages of one explicit-midpoint half step of the Lindblad flow (step dt/2):
// Y = X + (dt/4) L(X), then rho = X + (dt/2) L(Y), with its planes when the next kernel is
// GEMM1 (the leading half step; the trailing one is always followed by the next leading
// half step, a renormalisation or the end of the run, none of which read the planes).
void launch_half_lindblad(const Batch &b, int xsel, int planes, cudaStream_t s) {
    launch_lindblad(b, xsel, xsel, 2, 0.25f, 0, s);
    launch_lindblad(b, 2, xsel, 0, 0.5f, planes, s);
}

}  // namespace

qed_status split_prepare(qed_model *m, cudaStream_t s) {
    const int64_t D = m->D;
    const int64_t Dp = (D + kTcBM - 1) / kTcBM * kTcBM;
    const size_t W2 = (size_t)(2 * Dp) * (size_t)(2 * Dp);
    if (D >= 65536) {
        // (its buffers would exceed any device's memory; the Lindblad kernels index in 32 bits)
        set_error("split precision: dimensions up to 65535");
        return QED_EINVAL;
    }
    if (!m->sp) {
        m->sp = new SplitState();
        SplitState &S = *m->sp;
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&S.num_sms, cudaDevAttrMultiProcessorCount, dev);
        S.Dp = Dp;
        const size_t pl = (size_t)Dp * 2 * Dp * 2, DD = (size_t)(D * D);
        DeviceBlock big;
        big.room(&S.a1, W2 * 3);
        big.room(&S.b2, W2 * 3);
        big.room(&S.rho_df[0], DD);
        big.room(&S.rho_df[1], DD);
        big.room(&S.y_df, DD);
        big.room(&S.rho_pl, pl);
        big.room(&S.w_pl, pl);
        big.room(&S.w32, (size_t)2 * Dp * Dp);
        SPLIT_TRY(big.upload(&S.arrays));
        // zero padding: tiles of GEMM1 that lie wholly in it are never written (the planes and W lie
        // one after another)
        QED_CUDA_TRY(cudaMemset(S.rho_pl, 0, (size_t)((char *)(S.w32 + (size_t)2 * Dp * Dp) - (char *)S.rho_pl)));
        // the planner's split-K factors become the cluster sizes of the on-chip reduction
        static_assert(kTcMaxAutoSplits <= kTcMaxCluster, "plans must fit the cluster epilogues");
        if (!plan_products(S, S.g1, S.g2, 0, 0, 0)) return QED_ECUDA;

        DeviceBlock tables;
        tables.room(&S.phase_df, (size_t)D);
        tables.room(&S.damp_df, (size_t)D);
        tables.room(&S.stats, (size_t)(16 + ((D + 63) / 64) * ((D + 63) / 64)));
        // sqrt(dt) * coefficient of the incoming jump entries as double-floats
        auto split_f = [](double x) { const float h = (float)x; return make_float2(h, (float)(x - (double)h)); };
        const std::vector<int32_t> &ptr = m->h_in_ptr, &jmp = m->h_in_jump, &src = m->h_in_src;
        std::vector<float2> cdf_(m->h_in_coef.size());
        for (size_t e = 0; e < cdf_.size(); ++e) cdf_[e] = split_f(std::sqrt(m->dt) * m->h_in_coef[e]);
        tables.add(&S.coef_df, cdf_);
        // masks of the rows' jumps: at most 32 jumps, each once in a row's entries, which are
        // sorted by jump
        {
            std::vector<uint32_t> mask((size_t)D, 0u);
            bool fits = true;
            for (int64_t k = 0; k < D && fits; ++k) {
                fits = ptr[(size_t)k + 1] - ptr[(size_t)k] <= kMaskEntries;
                for (int32_t e = ptr[(size_t)k]; e < ptr[(size_t)k + 1] && fits; ++e) {
                    const int32_t j = jmp[(size_t)e];
                    fits = j < 32 && !(mask[(size_t)k] >> j & 1u);
                    if (fits) mask[(size_t)k] |= 1u << j;
                }
            }
            if (fits) tables.add(&S.mask, mask);
        }
        // with at most kInMax jumps, and (monomial operators) at most one incoming entry per
        // state and jump, the entries indexed by jump: the Lindblad kernels then read the
        // pairs (m, n) of each jump directly instead of matching the two rows' lists
        const int nj = (int)m->host.gamma.size();
        if (nj >= 1 && nj <= kInMax) {
            std::vector<int4> jt((size_t)D * kInMax, make_int4(-1, 0, 0, 0));
            bool unique = true;
            for (int64_t k = 0; k < D && unique; ++k)
                for (int32_t e = ptr[(size_t)k]; e < ptr[(size_t)k + 1]; ++e) {
                    int4 &slot = jt[(size_t)(k * kInMax + jmp[(size_t)e])];
                    if (slot.x >= 0) {
                        unique = false;
                        break;
                    }
                    const float2 c = cdf_[(size_t)e];
                    int f_hi = 0, f_lo = 0;
                    std::memcpy(&f_hi, &c.x, 4);
                    std::memcpy(&f_lo, &c.y, 4);
                    slot = make_int4(src[(size_t)e], f_hi, f_lo, 0);
                }
            if (unique) {
                tables.add(&S.jtab, jt);
                S.nj = nj;
            }
        }
        SPLIT_TRY(tables.upload(&S.tables));
    }
    SplitState &S = *m->sp;
    const bool eff = m->scheme == QED_SCHEME_EFFECTIVE;
    SPLIT_TRY(ensure_propagator(m, s));
    // Delta into work1, its scales from a host copy, then the constant planes
    make_delta_kernel<<<blocks_for(D * D, 256), 256, 0, s>>>(D, m->U, m->phase, m->work1, eff ? 0 : 1);
    count_launches(1);
    const int64_t nb = (D + 63) / 64;
    QED_CUDA_TRY(cudaMemsetAsync(S.stats, 0, (size_t)(16 + nb * nb), s));
    delta_stats_kernel<<<(unsigned)D, 256, 0, s>>>(D, m->work1, (unsigned long long *)S.stats);
    double top[2];  // largest element, largest row sum
    QED_CUDA_TRY(cudaMemcpyAsync(top, S.stats, sizeof(top), cudaMemcpyDeviceToHost, s));
    QED_CUDA_TRY(cudaStreamSynchronize(s));
    // largest scaled magnitude 2^14 (FP16 max 65504); |rho_kl| <= 1, |W_kl| <= max row sum of |Delta|
    const double scale_delta = S.scale_delta, scale_w = S.scale_w;
    S.scale_delta = pow2_scale(top[0], 14);
    S.scale_rho = std::ldexp(1.0, 14);
    S.scale_w = pow2_scale(top[1], 14);
    delta_blocks_kernel<<<(unsigned)D, 256, 0, s>>>(D, m->work1, S.scale_delta, S.stats + 16);
    count_launches(2);
    std::vector<uint8_t> nz((size_t)(nb * nb));
    QED_CUDA_TRY(cudaMemcpyAsync(nz.data(), S.stats + 16, nz.size(), cudaMemcpyDeviceToHost, s));
    QED_CUDA_TRY(cudaStreamSynchronize(s));
    S.nz.swap(nz);
    // the last that may run out of memory; the tables are written once it has not
    qed_model *self[1] = {m};
    const qed_status st = build_batch(S.self, self, 1, true);
    if (st != QED_OK) {
        S.nz.swap(nz);
        S.scale_delta = scale_delta;
        S.scale_w = scale_w;
        return st;
    }
    {
        // per-row phases P_k and dt/2 d_k (zero for the effective step, whose propagator holds
        // the anticommutator) as double-floats
        auto split_f = [](double x) { const float h = (float)x; return make_float2(h, (float)(x - (double)h)); };
        const std::vector<double2> &ph = m->h_phase;
        std::vector<float4> pdf((size_t)D);
        for (int64_t k = 0; k < D; ++k) {
            const float rh = (float)ph[(size_t)k].x, ih = (float)ph[(size_t)k].y;
            pdf[(size_t)k] = make_float4(rh, (float)(ph[(size_t)k].x - rh), ih, (float)(ph[(size_t)k].y - ih));
        }
        QED_CUDA_TRY(cudaMemcpy(S.phase_df, pdf.data(), (size_t)D * sizeof(float4), cudaMemcpyHostToDevice));
        const std::vector<double> &anti = m->h_anti;
        std::vector<float2> damp((size_t)D);
        for (int64_t k = 0; k < D; ++k) damp[(size_t)k] = split_f(eff ? 0.0 : 0.5 * m->dt * anti[(size_t)k]);
        QED_CUDA_TRY(cudaMemcpy(S.damp_df, damp.data(), (size_t)D * sizeof(float2), cudaMemcpyHostToDevice));
    }
    static_planes_kernel<<<blocks_for((int64_t)W2, 256), 256, 0, s>>>(D, Dp, m->work1, S.scale_delta, S.a1, S.b2);
    count_launches(1);
    QED_CUDA_TRY(cudaGetLastError());
    return QED_OK;
}

qed_status split_begin(qed_model *m, const double2 *rho, bool check, cudaStream_t s) {
    const Batch &b = m->sp->self;
    begin_kernel<<<b.n_pairs, dim3(32, 8), 0, s>>>(b.pairs, b.desc, nullptr, rho,
                                                   check ? density_check(m->scheme) : kNoCheck);
    count_launches(1);
    QED_CUDA_TRY(cudaGetLastError());
    return QED_OK;
}

void batch_step(const Batch &b, uint32_t *err, cudaStream_t s) {
    if (b.scheme == QED_SCHEME_STRANG) launch_half_lindblad(b, 0, 1, s);  // rho <- E(dt/2) rho
    launch_gemm1(b, err, s);  // W and its planes (split-K slices summed inside each cluster)
    launch_gemm2(b, err, s);  // X on and above the diagonal; its epilogue writes V = U rho U^+
    if (b.scheme == QED_SCHEME_STRANG)
        launch_half_lindblad(b, 1, 0, s);  // rho <- E(dt/2) V
    else
        launch_dissipate(b, s);
}

void split_step(qed_model *m, cudaStream_t s) { batch_step(m->sp->self, m->err, s); }

// Chooses the tile width and split-K factor (CTAs per cluster) of each of the model's two
// products by timing whole steps: GEMM1's candidates (128- and 256-wide tiles, 1, 2, 4 or 8
// slices) with GEMM2 as planned, then GEMM2's (128- and 256-wide, 1, 2 or 4 slices) with the
// best GEMM1.  Plans whose slices would not be a power of two are skipped.  Overwrites the
// internal state (qed_evolve imports rho again) and replaces the step tables; the caller
// drops its captured graphs.
qed_status split_autotune(qed_model *m, cudaStream_t s, int steps, std::string &choice) {
    SplitState &S = *m->sp;
    qed_model *self[1] = {m};
    auto candidates = [&](int which, std::vector<TcGemm> &out) -> qed_status {
        for (int bn : {128, 256}) {
            for (int sp : {1, 2, 4, 8}) {
                if (which == 2 && sp > kTcMaxClusterV) continue;
                TcGemm g1, g2;
                if (!plan_products(S, g1, g2, which == 1 ? sp : S.g1.splits, which == 1 ? bn : S.g1.bn,
                                   which == 2 ? sp : S.g2.splits, which == 2 ? bn : S.g2.bn))
                    return QED_ECUDA;
                const TcGemm &g = which == 1 ? g1 : g2;
                bool seen = (g.splits & (g.splits - 1)) != 0;
                for (const auto &h : out) seen = seen || (h.bn == g.bn && h.splits == g.splits);
                if (!seen) out.push_back(g);
            }
        }
        return QED_OK;
    };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    QED_CUDA_TRY(cudaEventCreate(&e0));
    QED_CUDA_TRY(cudaEventCreate(&e1));
    auto time_steps = [&](float &ms) -> qed_status {
        QED_CUDA_TRY(cudaStreamSynchronize(s));
        SPLIT_TRY(build_batch(S.self, self, 1, true));
        for (int i = 0; i < 2; ++i) batch_step(S.self, m->err, s);
        QED_CUDA_TRY(cudaEventRecord(e0, s));
        for (int i = 0; i < steps; ++i) batch_step(S.self, m->err, s);
        QED_CUDA_TRY(cudaEventRecord(e1, s));
        QED_CUDA_TRY(cudaEventSynchronize(e1));
        QED_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
        return QED_OK;
    };
    qed_status st = QED_OK;
    float best = 0.f;
    TcGemm g1 = S.g1, g2 = S.g2;
    std::vector<TcGemm> c1, c2;
    if ((st = candidates(1, c1)) == QED_OK && (st = candidates(2, c2)) == QED_OK && (st = time_steps(best)) == QED_OK) {
        for (const auto &g : c1) {
            S.g1 = g;
            S.g2 = g2;
            float t = 0.f;
            if ((st = time_steps(t)) != QED_OK) break;
            if (t < best) best = t, g1 = g;
        }
        for (size_t i = 0; st == QED_OK && i < c2.size(); ++i) {
            S.g1 = g1;
            S.g2 = c2[i];
            float t = 0.f;
            if ((st = time_steps(t)) != QED_OK) break;
            if (t < best) best = t, g2 = c2[i];
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    S.g1 = g1;
    S.g2 = g2;
    if (st != QED_OK) return st;
    QED_CUDA_TRY(cudaStreamSynchronize(s));
    SPLIT_TRY(build_batch(S.self, self, 1, true));
    choice = "gemm1 " + std::to_string(g1.bn) + "-wide x" + std::to_string(g1.splits) + " slices, gemm2 " +
             std::to_string(g2.bn) + "-wide x" + std::to_string(g2.splits) + " slices, " +
             std::to_string(1e3 * best / steps) + " us per step";
    return QED_OK;
}

// The batched counterpart: the grouped launches share one plan, so the candidates are the
// tile widths of the two products (GEMM1 256 or 128, GEMM2 128 or 256; both unsplit), each
// pair timed on `steps` whole batched steps from a zero state.  The winner is kept in every
// model of the batch.
qed_status split_autotune_batched(qed_model *const *ms, int n, cudaStream_t s, int steps, std::string &choice) {
    for (int i = 0; i < n; ++i) {
        SplitState &S = *ms[i]->sp;
        QED_CUDA_TRY(cudaMemsetAsync(S.rho_df[0], 0, (size_t)(ms[i]->D * ms[i]->D) * sizeof(float4), s));
        QED_CUDA_TRY(cudaMemsetAsync(S.rho_pl, 0, (size_t)S.Dp * 2 * S.Dp * 2 * sizeof(__half), s));
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    QED_CUDA_TRY(cudaEventCreate(&e0));
    QED_CUDA_TRY(cudaEventCreate(&e1));
    Batch b;
    qed_status st = QED_OK;
    float best = -1.f;
    int best1 = kTcBNMax, best2 = kTcBNMax;
    std::string times;
    const int plans[4][2] = {{256, 256}, {128, 256}, {256, 128}, {128, 128}};
    for (const auto &pl : plans) {
        if (cudaStreamSynchronize(s) != cudaSuccess) {
            set_error(std::string("autotune (batched): ") + cudaGetErrorString(cudaGetLastError()));
            st = QED_ECUDA;
            break;
        }
        if ((st = build_batch(b, ms, n, false, pl[0], pl[1])) != QED_OK) break;
        for (int i = 0; i < 2; ++i) batch_step(b, ms[0]->err, s);
        float t = 0.f;
        if (cudaEventRecord(e0, s) != cudaSuccess) { st = QED_ECUDA; break; }
        for (int i = 0; i < steps; ++i) batch_step(b, ms[0]->err, s);
        if (cudaEventRecord(e1, s) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
            cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) {
            set_error(std::string("autotune (batched): ") + cudaGetErrorString(cudaGetLastError()));
            st = QED_ECUDA;
            break;
        }
        times += (times.empty() ? "" : ", ") + std::to_string(pl[0]) + "-wide/" + std::to_string(pl[1]) + "-wide " +
                 std::to_string(1e3 * t / steps) + " us";
        if (best < 0.f || t < best) best = t, best1 = pl[0], best2 = pl[1];
    }
    cudaStreamSynchronize(s);
    b.release();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != QED_OK) return st;
    for (int i = 0; i < n; ++i) ms[i]->sp->batch_bn1 = best1, ms[i]->sp->batch_bn2 = best2;
    choice = "gemm1 " + std::to_string(best1) + "-wide, gemm2 " + std::to_string(best2) +
             "-wide (batched step, gemm1/gemm2 widths: " + times + ")";
    return QED_OK;
}

qed_status split_set_plan(qed_model *m, int bn1, int splits1, int bn2, int splits2, cudaStream_t s) {
    SplitState &S = *m->sp;
    auto pow2 = [](int x) { return x > 0 && (x & (x - 1)) == 0; };
    if ((bn1 != 128 && bn1 != 256) || (bn2 != 128 && bn2 != 256) || !pow2(splits1) || splits1 > kTcMaxCluster ||
        !pow2(splits2) || splits2 > kTcMaxClusterV) {
        set_error("qed_set_plan: widths 128 or 256, slices a power of two (GEMM1 <= 8, GEMM2 <= 4)");
        return QED_EINVAL;
    }
    TcGemm g1, g2;
    if (!plan_products(S, g1, g2, splits1, bn1, splits2, bn2)) return QED_ECUDA;
    if (g1.splits != splits1 || g2.splits != splits2) {
        set_error("qed_set_plan: more K slices than the product's 64-wide K blocks allow");
        return QED_EINVAL;
    }
    std::swap(S.g1, g1);
    std::swap(S.g2, g2);
    const qed_status st = split_rebuild(m, s);
    if (st != QED_OK) {
        S.g1 = g1;
        S.g2 = g2;
        return st;
    }
    S.batch_bn1 = bn1;
    S.batch_bn2 = bn2;
    return QED_OK;
}

void split_lindblad_stage(qed_model *m, int xsel, int bsel, int osel, float f, int planes, cudaStream_t s) {
    launch_lindblad(m->sp->self, xsel, bsel, osel, f, planes, s);
}

void split_apply_lindblad(qed_model *m, const float4 *X, float4 *out, cudaStream_t s) {
    const Batch &b = m->sp->self;
    if (b.jt)
        launch_pdl(lindblad_apply_jt_kernel, dim3(b.n_etiles), dim3(32, 8), 0, s, b.etiles, b.desc, X, out);
    else
        launch_pdl(lindblad_apply_df_kernel, dim3(b.n_etiles), dim3(32, 8), 0, s, b.etiles, b.desc, b.erows, X, out);
    count_launches(1);
}

void split_products(qed_model *m, cudaStream_t s) {
    launch_gemm1(m->sp->self, m->err, s);
    launch_gemm2(m->sp->self, m->err, s);
}

float4 *split_ybuf(qed_model *m) { return m->sp->y_df; }

qed_status split_rebuild(qed_model *m, cudaStream_t s) {
    QED_CUDA_TRY(cudaStreamSynchronize(s));
    qed_model *self[1] = {m};
    return build_batch(m->sp->self, self, 1, true);
}

void split_set_scheme(qed_model *m, int scheme) {
    if (m->sp) m->sp->self.scheme = scheme;
}

// Each kernel of the Lie step replayed `reps` times back to back from a CUDA graph (the way
// the step loop runs them: programmatic dependent launch overlapping one launch's set-up
// with the previous one's tail), after one full step so that W, V and the planes hold
// this state's values.  Each kernel only reads what the others write and overwrites its
// own outputs with the same values, so the replay repeats identical work.  ms[c] = mean
// milliseconds per launch.
qed_status split_profile_replay(qed_model *m, cudaStream_t s, int reps, std::vector<double> &ms, std::string &label) {
    const Batch &b = m->sp->self;
    if (b.scheme != QED_SCHEME_LIE) {
        set_error("qed_profile_replay: the Lie step only");
        return QED_EUNSUPPORTED;
    }
    batch_step(b, m->err, s);
    cudaStream_t cap = nullptr;
    QED_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    qed_status st = QED_OK;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) st = QED_ECUDA;
    ms.assign(3, 0.0);
    for (int c = 0; c < 3 && st == QED_OK; ++c) {
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        if (cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            st = QED_ECUDA;
            break;
        }
        const int64_t before = launches();
        for (int r = 0; r < reps; ++r) {
            if (c == 0) launch_gemm1(b, m->err, cap);
            else if (c == 1) launch_gemm2(b, m->err, cap);
            else launch_dissipate(b, cap);
        }
        count_launches(-(launches() - before));
        const cudaError_t e = cudaStreamEndCapture(cap, &graph);
        if (e != cudaSuccess || !graph || cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) st = QED_ECUDA;
        if (graph) cudaGraphDestroy(graph);
        float t = 0.f;
        if (st == QED_OK && (cudaGraphLaunch(exec, s) != cudaSuccess || cudaEventRecord(e0, s) != cudaSuccess ||
                             cudaGraphLaunch(exec, s) != cudaSuccess || cudaEventRecord(e1, s) != cudaSuccess ||
                             cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&t, e0, e1) != cudaSuccess))
            st = QED_ECUDA;
        count_launches(2 * (int64_t)reps);
        ms[(size_t)c] = (double)t / reps;
        if (exec) cudaGraphExecDestroy(exec);
    }
    if (st == QED_ECUDA) set_error(std::string("qed_profile_replay: ") + cudaGetErrorString(cudaGetLastError()));
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaStreamDestroy(cap);
    label = "gemm1_tc,gemm2_tc_v,dissipate";
    return st;
}

int split_step_timed(qed_model *m, cudaStream_t s, std::string &label) {
    const Batch &b = m->sp->self;
    if (b.scheme == QED_SCHEME_STRANG) {
        int e = 0;
        cudaEventRecord(m->ev[e++], s);
        launch_lindblad(b, 0, 0, 2, 0.25f, 0, s);
        cudaEventRecord(m->ev[e++], s);
        launch_lindblad(b, 2, 0, 0, 0.5f, 1, s);
        cudaEventRecord(m->ev[e++], s);
        launch_gemm1(b, m->err, s);
        cudaEventRecord(m->ev[e++], s);
        launch_gemm2(b, m->err, s);
        cudaEventRecord(m->ev[e++], s);
        launch_lindblad(b, 1, 1, 2, 0.25f, 0, s);
        cudaEventRecord(m->ev[e++], s);
        launch_lindblad(b, 2, 1, 0, 0.5f, 0, s);
        cudaEventRecord(m->ev[e++], s);
        label = "lindblad_a,lindblad_b,gemm1_tc,gemm2_tc_v,lindblad_c,lindblad_d";
        return 6;
    }
    cudaEventRecord(m->ev[0], s);
    launch_gemm1(b, m->err, s);
    cudaEventRecord(m->ev[1], s);
    launch_gemm2(b, m->err, s);
    cudaEventRecord(m->ev[2], s);
    launch_dissipate(b, s);
    cudaEventRecord(m->ev[3], s);
    label = "gemm1_tc,gemm2_tc_v,dissipate";
    return 3;
}

void split_renorm(qed_model *m, cudaStream_t s) {
    SplitState &S = *m->sp;
    trace_df_kernel<<<1, 1024, 0, s>>>(m->D, S.rho_df[0], m->scalars, m->err);
    dim3 block(32, 8);
    dim3 grid(blocks_for(m->D, 32), blocks_for(m->D, 8));
    // the effective step's own trace drift is part of its result: symmetrise only
    symmetrise_df_kernel<<<grid, block, 0, s>>>(m->D, S.Dp, S.rho_df[0], m->scalars, m->err,
                                                (float)S.scale_rho, S.rho_pl, m->scheme != QED_SCHEME_EFFECTIVE);
    count_launches(2);
}

void split_observables(qed_model *m, const int32_t *ids, int32_t n_obs, double *out, cudaStream_t s) {
    if (n_obs <= 0) return;
    observables_df_kernel<<<blocks_for(n_obs, kObsPerBlock), 256, 0, s>>>(m->D, m->sp->rho_df[0], m->obs_w, n_obs,
                                                                         ids, out);
    count_launches(1);
}

void split_end(qed_model *m, double2 *rho, cudaStream_t s) {
    const Batch &b = m->sp->self;
    end_kernel<<<b.n_pairs, dim3(32, 8), 0, s>>>(b.pairs, b.desc, nullptr, rho);
    count_launches(1);
}

qed_status split_batch_begin(const Batch *b, void *const *rhos, double *const *records, cudaStream_t s) {
    // (pageable host memory: staged before the calls return)
    QED_CUDA_TRY(cudaMemcpyAsync(b->rhos, rhos, (size_t)b->n * sizeof(void *), cudaMemcpyHostToDevice, s));
    if (records)
        QED_CUDA_TRY(cudaMemcpyAsync(b->records, records, (size_t)b->n * sizeof(void *), cudaMemcpyHostToDevice, s));
    begin_kernel<<<b->n_pairs, dim3(32, 8), 0, s>>>(b->pairs, b->desc, (const double2 *const *)b->rhos, nullptr,
                                                   density_check(b->scheme));
    count_launches(1);
    QED_CUDA_TRY(cudaGetLastError());
    return QED_OK;
}

void split_batch_populations(const Batch *b, int64_t row, cudaStream_t s) {
    batch_populations_kernel<<<b->n, 256, 0, s>>>(b->desc, (double *const *)b->records, row);
    count_launches(1);
}

qed_status split_batch_end(const Batch *b, std::vector<uint32_t> &errors, cudaStream_t s) {
    end_kernel<<<b->n_pairs, dim3(32, 8), 0, s>>>(b->pairs, b->desc, (double2 *const *)b->rhos, nullptr);
    read_errors_kernel<<<blocks_for(b->n, 256), 256, 0, s>>>(b->n, b->desc, b->errors);
    count_launches(2);
    errors.assign((size_t)b->n, 0u);
    QED_CUDA_TRY(cudaMemcpyAsync(errors.data(), b->errors, (size_t)b->n * 4, cudaMemcpyDeviceToHost, s));
    QED_CUDA_TRY(cudaStreamSynchronize(s));
    QED_CUDA_TRY(cudaGetLastError());
    return QED_OK;
}

qed_status split_batch_create(qed_model *const *ms, int n, Batch **out) {
    Batch *b = new Batch();
    // the tuned tile widths when every model of the batch carries the same ones
    int bn1 = ms[0]->sp->batch_bn1, bn2 = ms[0]->sp->batch_bn2;
    for (int i = 1; i < n; ++i)
        if (ms[i]->sp->batch_bn1 != bn1 || ms[i]->sp->batch_bn2 != bn2) bn1 = bn2 = 0;
    if (bn1 == 0) {
        // wide tiles where they are enough for half the SMs (GEMM1) or all of them (GEMM2, whose
        // epilogue is as long as its main loop): a batch of twelve chains of up to 400 states takes
        // 66 us a step in 128-wide tiles and 97 us in 256-wide ones, 64 of up to 1024 states 1216
        // and 1120 us
        int64_t t1 = 0, t2 = 0;
        for (int i = 0; i < n; ++i) {
            const int64_t nm = (ms[i]->D + kTcBM - 1) / kTcBM;
            t1 += 2 * nm * ((ms[i]->D + 255) / 256);
            t2 += nm * (nm + 1) / 2;
        }
        bn1 = 2 * t1 >= ms[0]->sp->num_sms ? 256 : 128;
        bn2 = t2 >= ms[0]->sp->num_sms ? 256 : 128;
    }
    qed_status st = build_batch(*b, ms, n, false, bn1, bn2);
    if (st != QED_OK) {
        b->release();
        delete b;
        return st;
    }
    *out = b;
    return QED_OK;
}

void split_batch_step(const Batch *b, uint32_t *err, cudaStream_t s) { batch_step(*b, err, s); }

void split_batch_destroy(Batch *b) {
    if (!b) return;
    b->release();
    delete b;
}

float4 *split_state(qed_model *m) { return m->sp->rho_df[0]; }
float4 *split_vbuf(qed_model *m) { return m->sp->rho_df[1]; }
void split_dissipate_only(qed_model *m, cudaStream_t s) { launch_dissipate(m->sp->self, s); }
void split_refresh_planes(qed_model *m, cudaStream_t s) {
    SplitState &S = *m->sp;
    dim3 grid(blocks_for(m->D, 256), (unsigned)m->D);
    planes_from_state_kernel<<<grid, 256, 0, s>>>(m->D, S.Dp, S.rho_df[0], (float)S.scale_rho, S.rho_pl);
    count_launches(1);
}

void split_release(qed_model *m) {
    if (!m->sp) return;
    SplitState &S = *m->sp;
    S.self.release();
    if (S.arrays) cudaFree(S.arrays);
    if (S.tables) cudaFree(S.tables);
    delete m->sp;
    m->sp = nullptr;
}

}  // namespace qed
