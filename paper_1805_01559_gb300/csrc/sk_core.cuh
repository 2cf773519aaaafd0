// Sinkhorn solver core shared by the single-instance and the batched persistent kernels
// (Algorithm 1 of the paper, Sec. III-B, in the log2-unit form described in k_sinkhorn.cu):
// constants, FP32-pair helpers, the row-streaming producer and the consumer warps' loop.
#pragma once

#include <cuda_runtime.h>
#include <float.h>
#include <math.h>

#include <type_traits>

#include "ot_common.cuh"
#include "sk_totals.h"

namespace ota {

static constexpr int NT_F = 256;  // threads per CTA of the finalize kernel (row blocks)
static constexpr double LN2 = 0.69314718055994530942;
static constexpr double LOG2E = 1.44269504088896340736;

enum : int { DEV_ENUMERIC = -7 };

struct DevScalars {
    double sp, sq;  // sums of the caller's p and q
    double inv_sp, inv_sq;
    float inv_sp_f;
    int status;
};

// The loop test compares the FP32 residual of the plan with tol (1 - 2^-5).  That residual is
// formed from FP32 cell values (approximate ex2, one rounding at about |G| per exponent) and
// sits within about 1e-8 of the exact FP64 residual of the same potentials at tol = 1e-6 (it
// can be on either side); the 3% margin keeps the returned plan's exact residual <= tol.
__host__ __device__ __forceinline__ double stop_tol(double tol) { return tol * (1.0 - 0.03125); }

struct LoopState {
    unsigned bar;
    int status;
    int iters;
    int converged;
    double err;
};

// Column state of one solve in global memory (Jp a multiple of 4), in doubles:
//   [0, 2 Jp)       G^k (log2 units, FP64) in buffer k & 1 (the returned potentials)
//   [2 Jp, 3 Jp)    log2 q^_j (FP64)
//   [3 Jp, 4 Jp)    log2 q^_j as FP32 pairs
//   [4 Jp, 4.5 Jp)  fixed-point shift S_j of column j (int)
//   then 2 rows of Jp + 4 64-bit words: per-column fixed-point totals of the sweeps' column
//   partials and their row residuals (words Jp and Jp + 2); sweep s adds into row s mod 2.
//   then Jp FP32 pairs: G^0, later G^1, as the sweeps hold them.
// The totals are sums of integers, the same in any order, so every CTA reads the same column
// sums whatever the number of CTAs or the order in which partitions arrive.
//
// How the words are counted and when a row may be added to again: sk_totals.h.
__host__ __device__ constexpr size_t gstate_words(int Jp) { return (size_t)Jp * 15 / 2 + 8; }
__host__ __device__ constexpr size_t gstate_bytes(int Jp) { return 8 * gstate_words(Jp); }
__device__ __forceinline__ float2* gs_lq2(double* G, int Jp) { return reinterpret_cast<float2*>(G + 3 * (size_t)Jp); }
__device__ __forceinline__ int* gs_sx(double* G, int Jp) { return reinterpret_cast<int*>(G + 4 * (size_t)Jp); }
__device__ __forceinline__ unsigned long long* gs_acc(double* G, int Jp) {
    return reinterpret_cast<unsigned long long*>(G + 4 * (size_t)Jp + Jp / 2);
}

__device__ __forceinline__ float2* gs_pairs(double* G, int Jp) {
    return reinterpret_cast<float2*>(G + (size_t)Jp * 13 / 2 + 8);
}
// An FP64 value as an FP32 pair, to about 2^-48 relative.
__device__ __forceinline__ float2 split_pair(double x) {
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
}

template <int TW, int VPT>
__device__ __forceinline__ void load_G(const double* __restrict__ G, int J, int tl, float4 (&g)[VPT]) {
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const int col = 4 * (tl + 32 * TW * v);
#pragma unroll
        for (int c = 0; c < 4; ++c) comp(g[v], c) = (col + c < J) ? (float)G[col + c] : 0.0f;
    }
}

// Cell exponent x = F + G - k C in log2 units, with F = F_hi + F_lo (FP32 pair) and
// k = k_hi + k_lo.  The exact FMA product cancels the large parts F_hi - C k_hi first, so
// the only roundings happen at the magnitude of |G| and |x|, however large k C and F are on
// the support.  k_lo > 0 always (see split_k): a +inf cost (masked column, forbidden link)
// gives -inf and never inf - inf.
__device__ __forceinline__ float expo(float F_hi, float F_lo_plus_G, float c, float k_hi, float k_lo) {
    return fmaf(-c, k_hi, F_hi) + fmaf(-c, k_lo, F_lo_plus_G);
}

// The same with the column potential as an FP32 pair G = G_hi + G_lo: F_hi - C k_hi (one
// rounding at about |G|) meets G_hi first, where the two nearly cancel on the cells that
// carry mass, and the low parts join at the magnitude of |x|.  No rounding of G itself enters
// the plan, so the plan the sweep measures is the plan of the FP64 potentials it returns.
__device__ __forceinline__ float expo2(float F_hi, float F_lo_plus_G_lo, float G_hi, float c, float k_hi,
                                       float k_lo) {
    return (fmaf(-c, k_hi, F_hi) + G_hi) + fmaf(-c, k_lo, F_lo_plus_G_lo);
}

// Error-free sum a + b = s + e (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// (hi, lo) - d as a renormalised FP32 pair.
__device__ __forceinline__ float2 df_sub(float2 f, float d) {
    float s, e;
    two_sum(f.x, -d, s, e);
    e += f.y;
    float h, l;
    two_sum(s, e, h, l);
    return make_float2(h, l);
}

// k = k_hi + k_lo with k_hi rounded down and 0 < k_lo <= ulp(k_hi): the low part is never
// zero or negative, so -inf * k_lo = -inf and no inf - inf can occur for C = +inf.
static inline void split_k(double k, float* hi, float* lo) {
    float h = (float)k;
    if ((double)h >= k) h = nextafterf(h, 0.0f);
    float l = (float)(k - (double)h);
    if (!(l > 0.0f)) l = 1.4e-45f;  // smallest subnormal; adds nothing measurable
    *hi = h;
    *lo = l;
}

// ------------------------------------------------------------------------------------------
// Row streaming: one producer warp copies contiguous blocks of rows of C into a ring of
// shared-memory stages with bulk copies; the consumer warps work on them.
// ------------------------------------------------------------------------------------------
// Consumer warps per CTA.  A sub-partition of the SM holds 16K registers, so a block whose
// busiest sub-partition runs 4 warps gets 128 registers a thread, whether the block has 13
// warps or 16.  One-warp teams take the full 16 (15 consumers + the producer): the sweep is
// latency-bound, and 15 warps instead of 12 at the same 128 registers made the 50,000 x 800
// solves 10% faster.  Other team widths take the largest multiple of the width that still
// fits: 14 for teams of 2 (5% faster than 12 at 200,000 x 1,536), 12 for teams of 4, and 8
// when a row needs a team of 8 warps.
template <int TW>
struct Cons {
    static constexpr int NCW = (TW == 8) ? 8 : (TW == 1 ? 15 : (TW == 2 ? 14 : 12));
    static constexpr int NT = 32 * (NCW + 1);  // + one producer warp
};
static constexpr int MAX_STAGES = 8;
static constexpr int CONS_BAR = 15;          // named barrier of the consumer warps
static constexpr int SMEM_HDR = 256;         // mbarriers at the start of dynamic smem

struct StreamCfg {
    int rows_per_stage;  // NTEAMS * rpt
    int rpt;             // rows per team per stage
    int stages;
    int stage_floats;    // rows_per_stage * ld (elements of the streamed matrix)
    int rmax;            // most rows any CTA owns
    int off_G;           // byte offsets inside dynamic smem
    int off_F;
    int off_P;
    int off_ring;
};

// Column potentials as FP32 pairs in shared memory: high parts Gs[0, Jp), low parts
// Gs[Jp, 2 Jp) with G_j = hi + lo to about 2^-48 relative (padding columns 0).
__device__ __forceinline__ void load_G_smem(const double* __restrict__ G, int J, int Jp, float* Gs, int tid,
                                            int nthreads) {
    for (int j = tid; j < Jp; j += nthreads) {
        const double x = (j < J) ? G[j] : 0.0;
        const float hi = (float)x;
        Gs[j] = hi;
        Gs[Jp + j] = (float)(x - (double)hi);
    }
}

// The same from pairs formed elsewhere (one thread a column of the whole group, instead of
// FP64 conversions of every column in every CTA).
__device__ __forceinline__ void load_G_pairs(const float2* __restrict__ pairs, int J, int Jp, float* Gs, int tid,
                                             int nthreads) {
    for (int j = tid; j < Jp; j += nthreads) {
        const float2 x = j < J ? __ldcg(pairs + j) : make_float2(0.f, 0.f);
        Gs[j] = x.x;
        Gs[Jp + j] = x.y;
    }
}

// log2(r) for the row and column corrections: a short series when r is within 2^-7 of 1
// (|u|^5/5 < 2^-37 relative to the result), the SFU logarithm otherwise.
__device__ __forceinline__ float log2_corr(float r) {
    const float u = r - 1.0f;  // exact for r in [0.5, 2]
    const float series = u * (1.0f + u * (-0.5f + u * (0.33333334f + u * -0.25f))) * 1.44269504f;
    const float sfu = __log2f(r);
    return fabsf(u) < 0.0078125f ? series : sfu;
}

// A lane's chunk v is certainly inside the row when the dispatch chose VPT = ceil(J4 / (32 TW))
// (pick_kernels and the batched forms do; the multi-solve's wide teams, VPT = 4, do not): then
// every chunk but the lane's last ends at or before column J.
template <int TW, int VPT>
__device__ __forceinline__ constexpr bool chunk_inside(int v) {
    return (TW == 1 || VPT > 4) && v < VPT - 1;
}

// Row load from a shared-memory stage; chunks that can leave the row are checked.
template <int TW, int VPT>
__device__ __forceinline__ void load_row_smem(const float* row, int J, int tl, float4 (&x)[VPT]) {
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const int col = 4 * (tl + 32 * TW * v);
        if (chunk_inside<TW, VPT>(v)) {
            x[v] = *reinterpret_cast<const float4*>(row + col);
        } else if (col < J) {
            float4 t = *reinterpret_cast<const float4*>(row + col);
            if (col + 4 > J) {
                if (col + 1 >= J) t.y = INFINITY;
                if (col + 2 >= J) t.z = INFINITY;
                if (col + 3 >= J) t.w = INFINITY;
            }
            x[v] = t;
        } else {
            x[v] = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        }
    }
}

// Euclidean cost of four columns from coordinates: sqrt(dx^2 + dy^2) in FP32 with explicit
// roundings (no contraction), so any IEEE single-precision evaluation of the same formula
// gives the same values; columns at or past J give +inf (no mass).
__device__ __forceinline__ float4 euclid_chunk(float2 d, const float* rx, const float* ry, int col, int J) {
    float4 a = *reinterpret_cast<const float4*>(rx + col);
    float4 b = *reinterpret_cast<const float4*>(ry + col);
    float4 o;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float dx = __fsub_rn(d.x, comp(a, c));
        const float dy = __fsub_rn(d.y, comp(b, c));
        comp(o, c) = col + c < J ? __fsqrt_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy))) : INFINITY;
    }
    return o;
}
template <int TW, int VPT>
__device__ __forceinline__ void euclid_row(float2 d, const float* rx, const float* ry, int J, int tl, float4 (&x)[VPT]) {
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const int col = 4 * (tl + 32 * TW * v);
        x[v] = col < J ? euclid_chunk(d, rx, ry, col, J) : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
    }
}

// The sweeps read a CTA's rows round after round, so a matrix larger than L2 (129 MB) would
// leave nothing of itself there for the next sweep.  The first L2_KEEP bytes of a CTA's rows
// (80 MB over 152 SMs, 5/8 of L2) keep the normal eviction priority and the rest is marked to
// be evicted first, so the kept part survives and is read from L2.  By itself that took 8% off a
// 50,000 x 800 solve (160 MB) and 2% off 48 ragged instances.  Kept parts from 60 to 100 MB and
// the persisting priority (evict_last) instead of the normal one differ by 3% at most; the
// persisting one would hold L2 against whatever runs next.
static constexpr int64_t L2_KEEP = 80000000 / 152;

// Producer: stream the CTA's row blocks sweep after sweep until the consumers raise s_stop,
// then wait for every copy still in flight before leaving.
template <typename T>
__device__ __forceinline__ void stream_rows_producer(const T* C, int64_t ld, int64_t r0, int64_t r1,
                                                     const StreamCfg& S, T* ring, uint64_t* full,
                                                     uint64_t* empty, volatile int* s_stop, int* status,
                                                     long long spin) {
    const int nblk = (int)((r1 - r0 + S.rows_per_stage - 1) / S.rows_per_stage);
    uint32_t seq = 0;
    const uint64_t keep = l2_policy_normal(), pass = l2_policy_first();
    const int64_t keep_rows = L2_KEEP / (ld * (int64_t)sizeof(T));
    bool stop = (nblk <= 0);
    while (!stop) {
        for (int k = 0; k < nblk && !stop; ++k) {
            const int st = (int)(seq % (uint32_t)S.stages);
            const uint32_t use = seq / (uint32_t)S.stages;
            if (use > 0) {  // wait for the consumers to release this stage's previous copy
                long long n = 0;
                while (!mbar_try_wait_sleep(&empty[st], (use - 1) & 1u, 500)) {
                    if (*s_stop) { stop = true; break; }
                    if ((++n & 1023) == 0 && ld_volatile_i32(status) != DEV_OK) { stop = true; break; }
                    if (n > spin) {
                        atomicCAS(status, DEV_OK, DEV_ETIMEOUT);
                        stop = true;
                        break;
                    }
                }
                if (stop) break;
            }
            if (*s_stop) { stop = true; break; }
            const int64_t row0 = r0 + (int64_t)k * S.rows_per_stage;
            const int rows = (int)min((int64_t)S.rows_per_stage, r1 - row0);
            const uint32_t bytes = (uint32_t)(rows * ld * (int64_t)sizeof(T));
            mbar_arrive_expect_tx(&full[st], bytes);
            bulk_g2s(ring + (size_t)st * S.stage_floats, C + row0 * ld, bytes, &full[st],
                     row0 - r0 < keep_rows ? keep : pass);
            ++seq;
        }
    }
    // Leave no copy in flight: wait for the last use of every stage to land.  This wait has
    // its own limit (about a second), independent of the caller's spin limit: a copy that was
    // issued completes on its own, and the CTA must not leave while one can still land.
    const long long drain_limit = spin > (1LL << 20) ? spin : (1LL << 20);
    for (int st = 0; st < S.stages; ++st) {
        if (seq <= (uint32_t)st) continue;
        const uint32_t uses = (seq - (uint32_t)st + S.stages - 1) / (uint32_t)S.stages;
        long long n = 0;
        while (!mbar_try_wait_sleep(&full[st], (uses - 1) & 1u, 1000) && ++n <= drain_limit) {
        }
    }
}

struct SolveParams {
    const float* C;
    int64_t ld;
    int64_t I;
    int J;
    int Jp;
    int V;            // row partitions (see part_row): the unit of every cross-row reduction
    const float* p;
    const float* q;
    const double* g_warm;                 // warm-start g (natural units) or nullptr
    const unsigned long long* input_bad;  // nonzero => invalid rates upstream, or nullptr
    DevScalars* sc;
    LoopState* st;
    double* G;        // gstate_words(Jp): column potentials G^k (log2 units, FP64) in buffer
                      // k & 1, log2 q^_j, the fixed-point column totals (see gstate_words)
    float2* F_out;    // [I] row potentials of the returned plan (hi, lo), or nullptr
    float* colpart;   // [V][2 * Jp]
    double* errpart;  // [V] during setup (sums of p); reused as float2 [V] residual pairs
    double k;
    float k_hi, k_lo;
    double tol;
    int max_iter;
    long long spin;
    // Finalize sweep after the stop (skipped when fpart is null): column partials
    // (sum_i p^_i t_ij, sum_i p^_i C_ij t_ij) per partition in FP64, row residual per
    // partition, and optionally the plan pi_ij = p_i t_ij and the natural-unit row potentials.
    double2* fpart;   // [V][Jp]
    double* epart;    // [V]
    float* pi;        // [I][pi_ld] or nullptr
    int64_t pi_ld;
    double* f_nat;    // [I] f_i = eps ln2 (F'_i + log2 p_i), or nullptr
    double eps_ln2;
    // Finalize only (F_in not null): no iteration; the finalize sweep runs on the caller's
    // potentials F' (pairs) and G (log2 units).
    const float2* F_in;  // [I]
    const double* G_in;  // [Jp]
    // Euclidean cost formed on the fly (Sec. IV cost choice (i)) instead of read from C:
    // device and RRH coordinates; the RRH coordinates are staged in shared memory at the
    // ring's offset (x then y, Jp floats each).
    const float2* dev_xy;  // [I]
    const float2* rrh_xy;  // [J]
    // Iteration 1 only (the stored-kernel form starts from its potentials): F'^1 to F_out and
    // G^1 in G + Jp, no test sweep and no finalize.
    int init_only = 0;
};

// Row partitions.  The I rows form B = ceil(I / rs) stage blocks of rs rows; partition v of V
// is the run of blocks [B v / V, B (v + 1) / V).  Every sum over rows (column partials, row
// residuals, sums of p) is formed per partition, in a fixed order inside it, and partitions
// are combined in partition order, so the result does not depend on how many CTAs share the
// work: a CTA owns a contiguous run of partitions and walks them one after the other.
__host__ __device__ __forceinline__ int64_t part_row(int64_t I, int rs, int V, int v) {
    const int64_t B = (I + rs - 1) / rs;
    const int64_t r = (B * v / V) * rs;
    return r < I ? r : I;
}
// Rows [r0, r1) of CTA b of nb.
__host__ __device__ __forceinline__ void cta_rows(int64_t I, int rs, int V, int b, int nb, int64_t* r0,
                                                  int64_t* r1) {
    int v0, v1;
    cta_parts(V, b, nb, &v0, &v1);
    *r0 = part_row(I, rs, V, v0);
    *r1 = part_row(I, rs, V, v1);
}
// Partitions of an instance: at most VMAX, at least one stage block and 64 rows each.
static constexpr int VMAX = 152;
__host__ __device__ __forceinline__ int parts_for(int64_t I, int rs) {
    const int64_t B = (I + rs - 1) / rs;
    int64_t v = I / 64;
    if (v > B) v = B;
    if (v > VMAX) v = VMAX;
    return v < 1 ? 1 : (int)v;
}

// Stage geometry and shared-memory layout of an instance solved by nb CTAs with teams of
// `nteams` rows (g_words floats per column at off_G: 2 for the FP32 pairs of G; f_bytes per
// row in each of the two row-potential buffers: an FP32 pair, or one float for the stored
// kernel's scalings).  The rows per stage depend only on the stage target and the row length,
// and the partitions only on I and the rows per stage: the arithmetic of a solve is fixed
// by (I, J, ld, stage target) whatever nb is.  Returns false when a CTA's rows do not fit
// next to two stages.
inline bool plan_stage(int nteams, int64_t I, int Jp, int64_t ld, int nb, int stage_target, size_t budget,
                       StreamCfg* S, size_t* smem, int* Vout, int esize = 4, int g_words = 2,
                       int f_bytes = (int)sizeof(float2), int comb_bufs = 0) {
    // comb_bufs: rows of Jp floats for merging the teams' column partials (0: half the teams)
    const size_t comb = (size_t)(comb_bufs > 0 ? comb_bufs : (nteams + 1) / 2) * Jp * sizeof(float);
    const size_t row_bytes = (size_t)ld * esize;
    const int rpt = (int)(stage_target / ((size_t)nteams * row_bytes) > 1 ? stage_target / ((size_t)nteams * row_bytes)
                                                                           : 1);
    const int rs = nteams * rpt;
    const int V = parts_for(I, rs);
    int64_t rmax = 0;
    for (int b = 0; b < nb; ++b) {
        int64_t r0, r1;
        cta_rows(I, rs, V, b, nb, &r0, &r1);
        rmax = r1 - r0 > rmax ? r1 - r0 : rmax;
    }
    auto up = [](size_t x, size_t m) { return (x + m - 1) / m * m; };
    const size_t off_G = up(SMEM_HDR + comb, 16);
    const size_t off_F = up(off_G + (size_t)g_words * Jp * sizeof(float), 16);  // G pairs: hi, then lo
    const size_t off_P = up(off_F + (size_t)2 * rmax * f_bytes, 16);  // two row-potential buffers
    const size_t off_ring = up(off_P + (size_t)rmax * sizeof(float), 128);
    const size_t stage = (size_t)rs * row_bytes;
    const size_t room = off_ring < budget ? (budget - off_ring) / stage : 0;
    const int stages = (int)(room < (size_t)MAX_STAGES ? room : (size_t)MAX_STAGES);
    if (stages < 2) return false;
    S->rpt = rpt;
    S->rows_per_stage = rs;
    S->stages = stages;
    S->stage_floats = (int)(stage / esize);
    S->rmax = (int)(rmax > 0 ? rmax : 1);
    S->off_G = (int)off_G;
    S->off_F = (int)off_F;
    S->off_P = (int)off_P;
    S->off_ring = (int)off_ring;
    *smem = off_ring + (size_t)stages * stage;
    *Vout = V;
    return true;
}

// A consumer's place in the ring of stages: the stage and the parity of its current use.  Once a
// wait for a stage has given up (the launch is ending, and its status says so; bit 1 of ph) a
// lane neither waits for stages nor releases them any more, but it goes through its rows like the
// others, on whatever the ring holds: if it left them out, its warp would be torn at the shuffles
// and its team left waiting at the team's barriers, which have no limit.
struct RingPos {
    int st = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void wait(uint64_t* full, long long spin, int* status) {
        if (ph < 2u && !mbar_try_wait(&full[st], ph) && !mbar_wait_bounded(&full[st], ph, spin, status)) ph |= 2u;
    }
    // by lane 0 of each warp, after the warp's last read of the stage
    __device__ __forceinline__ void release(uint64_t* empty, int stage) const {
        if (ph < 2u) mbar_arrive(&empty[stage]);
    }
    __device__ __forceinline__ void next(int stages) {
        if (++st == stages) {
            st = 0;
            ph ^= 1u;
        }
    }
};

// Sum of (s, e) pairs over a warp with error-free additions.
__device__ __forceinline__ void warp_sum_pair(float& s, float& e) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
        const float e2 = __shfl_xor_sync(0xffffffffu, e, o);
        float t, u;
        two_sum(s, s2, t, u);
        s = t;
        e = e + e2 + u;
    }
}

// Shared-memory words of the consumer warps (and the producer's stop flag).
struct SkShared {
    alignas(16) unsigned zeros[4];  // a chunk of zeros (stored-kernel loop)
    float red[64];          // team reductions: 2 * NTEAMS * TW <= 24 values (float2 pairs: 48 floats)
    float errf[16];         // per-team row residuals
    double sh_sum[24][2];   // per-warp setup sums (up to 24 consumer warps)
    int s_dec, s_ok, s_bad;
    int flags[2];                    // of a sweep, by parity: the SK_ bits below
    unsigned long long s_err;        // total of the row residuals
    unsigned long long err_was[2][2];  // a row's residual words when last complete (thread 0's)
    unsigned long long werr[16];     // per team, of the current partition
    volatile int s_stop;    // consumers -> producer: stop streaming
    uint32_t tmem;          // tensor-memory address of the column potentials (see G_to_tmem)
    int pend[VMAX + 1];     // stage blocks (from the CTA's first row) at which its partitions end
};

enum : int {
    SK_EXACT = 1,  // some column's total has to be summed from the partials
    SK_BAD = 2,    // and one of those lost its mass
    // A wait for the totals gave up: for a thread's first columns, looked at after those, or for
    // further ones, looked at after all.  Two bits: a thread may be waiting for further columns
    // while another has yet to look at the first ones, and the CTA leaves as one.
    SK_LATE = 4,
    SK_LATER = 8,
};

// The CTAs that solve one instance together: nb CTAs, this one is number b.  `bar` counts
// arrivals at the group's barriers (monotonic; every CTA of the group passes the same
// barriers, `gen` of them so far).  A nonzero *abort ends every wait; *status is the
// instance's status word (the same word as *abort for a single-instance launch).
struct GroupCtx {
    int nb, b;
    unsigned* bar;
    unsigned gen;
    int* abort;
    int* status;
};

// Team sum of per-lane FP32 values as an error-free (hi, lo) pair; `red` holds 4 * NTEAMS * TW
// floats, the halves alternating by `par` as in team_reduce.
template <int TW>
__device__ __forceinline__ float2 team_sum_pair(float s, float* red, int nteams, const Team<TW>& tm, int& par) {
    float e = 0.f;
    warp_sum_pair(s, e);
    if constexpr (TW == 1) {
        return make_float2(s, e);
    } else {
        float2* r = reinterpret_cast<float2*>(red) + (par * nteams + tm.team) * TW;
        if (tm.lane == 0) r[tm.wit] = make_float2(s, e);
        bar_named(1 + tm.team, 32 * TW);
        float2 a = r[0];
#pragma unroll
        for (int w = 1; w < TW; ++w) a = df_add2(a, r[w]);
        par ^= 1;
        return a;
    }
}

// Sum of the teams' float4 column partials acc (in team order: the first half of the teams
// stores, the second half adds onto slot team - HALF, then the HALF slots are summed in
// order); f(j, sum) receives column j's total.  Named barriers over the consumer warps; the
// comb buffer (HALF rows of Jp floats) is free again when it returns.
template <int TW, int VPT, typename Fn>
__device__ __forceinline__ void cta_col_sum(float* comb, const float4 (&acc)[VPT], int J, int Jp, const Team<TW>& tm,
                                            Fn f) {
    constexpr int NCW = Cons<TW>::NCW;
    constexpr int TT = 32 * TW, NTEAMS = NCW / TW, NC = NCW * 32;
    constexpr int HALF = (NTEAMS + 1) / 2;
    if (tm.team < HALF) {
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int col = 4 * (tm.tl + TT * v);
            if (col < Jp) *reinterpret_cast<float4*>(comb + tm.team * Jp + col) = acc[v];
        }
    }
    bar_named(CONS_BAR, NC);
    if (tm.team >= HALF) {
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int col = 4 * (tm.tl + TT * v);
            if (col < Jp) {
                float4* d = reinterpret_cast<float4*>(comb + (tm.team - HALF) * Jp + col);
                float4 o = *d;
                o.x += acc[v].x;
                o.y += acc[v].y;
                o.z += acc[v].z;
                o.w += acc[v].w;
                *d = o;
            }
        }
    }
    bar_named(CONS_BAR, NC);
    for (int j = threadIdx.x; j < J; j += NC) {
        float sum = comb[j];
        for (int t = 1; t < HALF; ++t) sum += comb[t * Jp + j];
        f(j, sum);
    }
    bar_named(CONS_BAR, NC);
}

// Column potentials in tensor memory: the eight words of chunk v (four high parts, four low
// parts) of a lane at columns 8 v .. 8 v + 7 of its warp's quarter.  Lane positions repeat
// every TW warps, so one copy per quarter serves every warp of the CTA (two for teams of 8).
// The sweep reads G (eight bytes a column) once per row: from shared memory that was two thirds
// of its shared-memory wavefronts (84 a row of 800 columns, with 25 more for the copy that
// fills the ring), the busiest unit of the sweep.  Out of tensor memory the sweep of a
// 50,000 x 800 solve takes 41,000 cycles a CTA instead of 46,600 (2% of the solve when the sync
// still hid most of it), and a 100,000 x 1,536 solve 17% less.
template <int TW, int VPT>
constexpr int tmem_cols() {
    constexpr int n = 8 * VPT * (TW == 8 ? 2 : 1);
    // lane positions have to repeat with the warp quarters, and the columns to fit what is allocated
    static_assert((TW == 1 || TW == 2 || TW == 4 || TW == 8) && n <= 128, "columns of tensor memory");
    return n <= 32 ? 32 : (n <= 64 ? 64 : 128);
}
template <int TW, int VPT>
__device__ __forceinline__ uint32_t tmem_G(uint32_t base, const Team<TW>& tm) {
    const uint32_t warp = threadIdx.x >> 5;
    return base + ((warp & 3u) << 21) + (TW == 8 ? (uint32_t)(tm.wit >> 2) * (8 * VPT) : 0u);
}
// Copy G from shared memory to tensor memory (all consumer warps call; G complete in Gs before,
// visible to every consumer warp after).
template <int TW, int VPT>
__device__ __forceinline__ void G_to_tmem(uint32_t base, const float* Gs, int Jp, const Team<TW>& tm) {
    constexpr int WRITERS = TW == 8 ? 8 : 4, TT = 32 * TW;
    if ((threadIdx.x >> 5) < WRITERS) {
        const uint32_t a = tmem_G<TW, VPT>(base, tm);
        tmem_fence_after();
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int col = 4 * (tm.tl + TT * v);
            float4 hi = make_float4(0.f, 0.f, 0.f, 0.f), lo = hi;
            if (col < Jp) {
                hi = *reinterpret_cast<const float4*>(Gs + col);
                lo = *reinterpret_cast<const float4*>(Gs + Jp + col);
            }
            __syncwarp();
            tmem_st8(a + 8 * v, hi, lo);
        }
        tmem_wait_st();
        tmem_fence_before();
    }
    bar_named(CONS_BAR, Cons<TW>::NCW * 32);
    tmem_fence_after();
}

// A lane's chunk of G as two packed pairs of high and of low parts: from tensor memory (TM), or
// from shared memory.  The whole warp calls it, converged.
template <bool TM>
__device__ __forceinline__ void load_G_chunk(uint32_t tG, int v, const float* Gs, int Jp, int col, f32x2 (&gh)[2],
                                             f32x2 (&gl)[2]) {
    if constexpr (TM) {
        uint32_t w[8];
        tmem_ld8(tG + 8 * v, w);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            gh[h] = pack2(__uint_as_float(w[2 * h]), __uint_as_float(w[2 * h + 1]));
            gl[h] = pack2(__uint_as_float(w[4 + 2 * h]), __uint_as_float(w[5 + 2 * h]));
        }
    } else {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(Gs + col);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(Gs + Jp + col);
        gh[0] = a.x;
        gh[1] = a.y;
        gl[0] = b.x;
        gl[1] = b.y;
    }
}
// A lane's chunk of a row of C as two packed pairs, formed from coordinates when EUC.
template <bool EUC>
__device__ __forceinline__ void load_C_chunk(const float* row, float2 dxy, const float* rxs, int Jp, int J, int col,
                                             f32x2 (&c)[2]) {
    if constexpr (EUC) {
        const float4 e = euclid_chunk(dxy, rxs, rxs + Jp, col, J);
        c[0] = pack2(e.x, e.y);
        c[1] = pack2(e.z, e.w);
    } else {
        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(row + col);
        c[0] = e.x;
        c[1] = e.y;
    }
}

// Finalize sweep of the consumer warps, run right after the loop stops: the producer has
// already streamed the next pass over the CTA's rows into the ring, so this is one more
// sweep at streaming speed.  Plan of the returned potentials F' (Fold) and G (Gs, still the
// returned plan's column potentials, also in tensor memory when TM): t_ij = 2^(F'_i + G_j - k C_ij).  Each team keeps FP32
// column sums of p^ t and p^ C t over at most FIN_ROWS rows, then the CTA adds the teams'
// sums (in team order) into the partition's FP64 partials P.fpart[v]; the row residual
// sum_i p^_i |sum_j t_ij - 1| uses error-free row sums.
static constexpr int FIN_ROWS = 16;
template <int TW, int VPT, bool EUC = false, bool TM = true>
__device__ __forceinline__ void sk_finalize_sweep(const SolveParams& P, const StreamCfg& S, SkShared* sh,
                                                  unsigned char* dyn, int64_t r0, int nrow, int v0, int v1,
                                                  const float2* Fold, RingPos& pos, int* abort) {
    constexpr int NCW = Cons<TW>::NCW;
    constexpr int TT = 32 * TW, NTEAMS = NCW / TW, NC = NCW * 32;
    uint64_t* full = reinterpret_cast<uint64_t*>(dyn);
    uint64_t* empty = full + MAX_STAGES;
    float* comb = reinterpret_cast<float*>(dyn + SMEM_HDR);
    const float* Gs = reinterpret_cast<const float*>(dyn + S.off_G);
    const float* Ps = reinterpret_cast<const float*>(dyn + S.off_P);
    const float* ring = reinterpret_cast<const float*>(dyn + S.off_ring);
    const float* rx = ring;  // Euclidean cost: RRH x then y coordinates
    const int tid = threadIdx.x, lane = tid & 31;
    const int J = P.J, Jp = P.Jp, rs_ = S.rows_per_stage;
    const Team<TW> tm;
    int par = 0;
    for (int v = v0; v < v1; ++v)
        for (int j = tid; j < J; j += NC) P.fpart[(int64_t)v * Jp + j] = make_double2(0.0, 0.0);
    f32x2 cpi[VPT][2], crho[VPT][2];
#pragma unroll
    for (int v = 0; v < VPT; ++v) cpi[v][0] = cpi[v][1] = crho[v][0] = crho[v][1] = 0ull;
    const uint32_t tG = TM ? tmem_G<TW, VPT>(sh->tmem, tm) : 0u;
    const f32x2 nk_hi = pack2(-P.k_hi, -P.k_hi), nk_lo = pack2(-P.k_lo, -P.k_lo);
    float errt = 0.f;
    const int nblk = (nrow + rs_ - 1) / rs_;
    const bool want_pi = P.pi != nullptr;
    const int every = max(1, FIN_ROWS / S.rpt);  // stages between flushes
    // Multi-warp teams: a row's sum is reduced within each warp (shuffles only) and the warps'
    // pairs wait in the merge buffer with p^_i; one thread per team combines them, row by row
    // in the same order and arithmetic as a per-row team sum, at the next flush (where the CTA
    // synchronises anyway) instead of a team barrier on every row.
    constexpr int HALF = (NTEAMS + 1) / 2;  // rows of Jp floats in the merge buffer
    const int wrows = every * S.rpt;        // rows a team sees between two flushes
    const bool defer = TW > 1 && (int64_t)wrows * NTEAMS * (2 * TW + 1) <= (int64_t)HALF * Jp;
    float2* wpair = reinterpret_cast<float2*>(comb);                       // [NTEAMS][wrows][TW]
    float* wph = comb + 2 * (size_t)NTEAMS * wrows * TW;                   // [NTEAMS][wrows]
    int wr = 0;
    const int* pend = sh->pend - v0;
    int vp = v0, vbeg = 0;
    int vend = v0 < v1 ? pend[v0] : 0;
    for (int kb = 0; kb < nblk; ++kb) {
        const int st = pos.st;
        if (!EUC) pos.wait(full, P.spin, abort);
        const int lr0 = kb * rs_;
        const int rows = min(rs_, nrow - lr0);
        const float* stage = ring + (size_t)st * S.stage_floats;
        for (int jr = 0; jr < S.rpt; ++jr) {
            const int rr = tm.team + NTEAMS * jr;
            if (rr >= rows) break;
            const int lr = lr0 + rr;
            const float* row = stage + (size_t)rr * P.ld;
            const float2 dxy = EUC ? __ldg(P.dev_xy + r0 + lr) : make_float2(0.f, 0.f);
            const float2 F = Fold[lr];
            const float phat = Ps[lr];
            const int64_t i = r0 + lr;
            const float pf = want_pi ? __ldg(P.p + i) : 0.f;
            float rsum = 0.f;
            const f32x2 Fh = pack2(F.x, F.x), Fl = pack2(F.y, F.y), ph2 = pack2(phat, phat);
            __syncwarp();
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                const bool all_in = chunk_inside<TW, VPT>(v);  // lanes past the row: as in sweep_rows
                const int at = 4 * (tm.tl + TT * v);
                const int col = all_in || at < J ? at : 0;
                f32x2 gh[2], gl[2], c[2], t[2];
                load_G_chunk<TM>(tG, v, Gs, Jp, col, gh, gl);
                load_C_chunk<EUC>(row, dxy, rx, Jp, J, col, c);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 x =
                        unpack2(add2(add2(fma2(c[h], nk_hi, Fh), gh[h]), fma2(c[h], nk_lo, add2(Fl, gl[h]))));
                    float2 e = unpack2(c[h]);
                    float t0 = ex2(x.x), t1 = ex2(x.y);
                    // a +inf cost (no link, no mass) counts as a finite one; past the row neither does
                    e.x = fminf(e.x, FLT_MAX);
                    e.y = fminf(e.y, FLT_MAX);
                    if (!all_in) {
                        if (at + 2 * h >= J) t0 = e.x = 0.f;
                        if (at + 2 * h + 1 >= J) t1 = e.y = 0.f;
                    }
                    rsum += t0;
                    rsum += t1;
                    t[h] = pack2(t0, t1);
                    cpi[v][h] = fma2(ph2, t[h], cpi[v][h]);
                    crho[v][h] = fma2(ph2, mul2(pack2(e.x, e.y), t[h]), crho[v][h]);
                }
                if (want_pi) {  // one uniform branch per chunk, not per cell
                    const float2 ta = unpack2(t[0]), tb = unpack2(t[1]);
                    const float tv[4] = {ta.x, ta.y, tb.x, tb.y};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (at + q < J) P.pi[i * P.pi_ld + at + q] = pf * tv[q];
                    __syncwarp();
                }
            }
            if (defer) {
                float e = 0.f;
                warp_sum_pair(rsum, e);
                if (tm.lane == 0) wpair[((size_t)tm.team * wrows + wr) * TW + tm.wit] = make_float2(rsum, e);
                if (tm.tl == 0) wph[tm.team * wrows + wr] = phat;
                ++wr;
            } else {
                const float2 r = team_sum_pair<TW>(rsum, sh->red, NTEAMS, tm, par);
                errt = fmaf(phat, fabsf((r.x - 1.0f) + r.y), errt);
            }
        }
        __syncwarp();
        if (!EUC && lane == 0) pos.release(empty, st);
        pos.next(S.stages);
        const bool at_end = (kb + 1 == vend);
        if ((kb + 1 - vbeg) % every == 0 || at_end) {
            if (defer) {
                bar_named(CONS_BAR, NC);  // every warp's parked row pairs are visible
                if (tm.tl == 0)
                    for (int k = 0; k < wr; ++k) {
                        const float2* r = wpair + ((size_t)tm.team * wrows + k) * TW;
                        float2 a = r[0];
#pragma unroll
                        for (int w = 1; w < TW; ++w) a = df_add2(a, r[w]);
                        errt = fmaf(wph[tm.team * wrows + k], fabsf((a.x - 1.0f) + a.y), errt);
                    }
                wr = 0;
                bar_named(CONS_BAR, NC);  // the merge buffer is free for the column sums
            }
            // Wide rows (multi-warp teams): reductions without a returned value.  The thread that
            // zeroed fp[j] is the one that adds to it, flush after flush, so the sums are the
            // serial ones, bit for bit, but no thread waits on L2 for the old value (at 4,096
            // columns a read-modify-write per column cost 0.2 ms of a 2.2 ms finalize).  One-warp
            // teams keep the read-modify-write: there the flushes are rare, and the reductions
            // changed the register allocation of the whole solver loop (1.5% slower at 800
            // columns).
            double2* fp = P.fpart + (int64_t)vp * Jp;
            float4 sum_pi[VPT], sum_rho[VPT];
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                const float2 a = unpack2(cpi[v][0]), b = unpack2(cpi[v][1]);
                const float2 c = unpack2(crho[v][0]), d = unpack2(crho[v][1]);
                sum_pi[v] = make_float4(a.x, a.y, b.x, b.y);
                sum_rho[v] = make_float4(c.x, c.y, d.x, d.y);
            }
            if constexpr (TW > 1) {
                cta_col_sum<TW, VPT>(comb, sum_pi, J, Jp, tm, [&](int j, float sum) { atomicAdd(&fp[j].x, (double)sum); });
                cta_col_sum<TW, VPT>(comb, sum_rho, J, Jp, tm, [&](int j, float sum) { atomicAdd(&fp[j].y, (double)sum); });
            } else {
                cta_col_sum<TW, VPT>(comb, sum_pi, J, Jp, tm, [&](int j, float sum) { fp[j].x += (double)sum; });
                cta_col_sum<TW, VPT>(comb, sum_rho, J, Jp, tm, [&](int j, float sum) { fp[j].y += (double)sum; });
            }
#pragma unroll
            for (int v = 0; v < VPT; ++v) cpi[v][0] = cpi[v][1] = crho[v][0] = crho[v][1] = 0ull;
        }
        if (at_end) {
            if (tm.tl == 0) sh->errf[tm.team] = errt;
            bar_named(CONS_BAR, NC);
            if (tid == 0) {
                float2 e = make_float2(sh->errf[0], 0.f);
                for (int t = 1; t < NTEAMS; ++t) e = df_add(e, sh->errf[t]);
                P.epart[vp] = (double)e.x + (double)e.y;
            }
            bar_named(CONS_BAR, NC);
            errt = 0.f;
            ++vp;
            vbeg = kb + 1;
            if (vp < v1) vend = pend[vp];
        }
    }
    // natural-unit row potentials, one row per thread (an FP64 log2 each, off the sweep)
    if (P.f_nat)
        for (int r = tid; r < nrow; r += NC) {
            const float2 F = Fold[r];
            P.f_nat[r0 + r] = P.eps_ln2 * ((double)F.x + (double)F.y + log2((double)__ldg(P.p + r0 + r)));
        }
}

// Sums of R rows' per-lane values over the team, each in the order of team_reduce; every lane
// gets all R.  The rows share one butterfly: after the first exchange the lower half-warp
// holds row 0's sums and the upper half row 1's (the same pairs are added), so two rows take
// the shuffles of one plus one exchange, and wider teams one named barrier.
template <int TW, int R>
__device__ __forceinline__ void team_sum_rows(float (&v)[R], float* red, int nteams, const Team<TW>& tm, int& par) {
    if constexpr (R == 1) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        if constexpr (TW > 1) {  // a team's slots are the same ones as for two rows
            float* r = red + (par * nteams + tm.team) * (2 * TW);
            if (tm.lane == 0) r[tm.wit] = v[0];
            bar_named(1 + tm.team, 32 * TW);
            float a = r[0];
#pragma unroll
            for (int w = 1; w < TW; ++w) a += r[w];
            v[0] = a;
            par ^= 1;
        }
    } else {
        static_assert(R == 2, "one or two rows");
        const bool up = tm.lane >= 16;
        float s = (up ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[1], 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if constexpr (TW == 1) {
            const float w = __shfl_xor_sync(0xffffffffu, s, 16);
            v[0] = up ? w : s;
            v[1] = up ? s : w;
        } else {
            float* r = red + (par * nteams + tm.team) * (2 * TW);
            if ((tm.lane & 15) == 0) r[(up ? TW : 0) + tm.wit] = s;
            bar_named(1 + tm.team, 32 * TW);
            float a = r[0], b = r[TW];
#pragma unroll
            for (int w = 1; w < TW; ++w) {
                a += r[w];
                b += r[TW + w];
            }
            v[0] = a;
            v[1] = b;
            par ^= 1;
        }
    }
}

// Rows a team takes at once.  Two rows of up to 6 chunks a lane fit the registers (128 a
// thread); at 7 chunks the second row spills (50,000 x 800: 3% slower with two rows).  Wider
// teams stay at one: their rows come from HBM, not L2, at the sizes that matter (100,000 x 1,536:
// 2% slower with two).  1000 x 50 is 4% faster with two rows.
template <int TW, int VPT, bool EUC>
__host__ __device__ constexpr int rows_per_pass() {
    return EUC || TW > 1 || VPT > 6 ? 1 : 2;
}

// One plan-scale pass of a team over R rows of C at once (row[k]: the staged row, or unused
// when EUC with the device at dxy[k]): t_ij = 2^(F'_i + G_j - k C_ij), the row sums r_i (left
// in Fnew for row_updates) and the column accumulators acc += t p^ / r, row 0 before row 1.
// Bound by instruction issue and by the latency of a row's chain (shared-memory loads, ex2,
// the team sum, the update) once C streams: two rows in flight hide one chain behind the
// other and share the loads of G, and packed arithmetic halves the instructions of the
// exponent and the accumulation (by itself 4% of a 50,000 x 800 solve, and 24% at 100,000 x 1,536
// with the chunk count of a lane fitted to the row for wide teams too).  Every operation
// rounds as for one row at a time, so results are the same bit for bit.
template <int TW, int VPT, bool EUC, int R>
__device__ __forceinline__ void sweep_rows(const float* (&row)[R], const float2 (&dxy)[R], uint32_t tG, int J,
                                           int Jp, const float* rxs, f32x2 nk_hi, f32x2 nk_lo, const float2* Fold,
                                           float2* Fnew, const float* Ps, const int (&lr)[R], float* red, int nteams,
                                           const Team<TW>& tm, int& par, f32x2 (&acc)[VPT][2]) {
    constexpr int TT = 32 * TW;
    __syncwarp();
    f32x2 t[R][VPT][2], Fh[R], Fl[R];
    float rsum[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const float2 F = Fold[lr[k]];
        Fh[k] = pack2(F.x, F.x);
        Fl[k] = pack2(F.y, F.y);
        rsum[k] = 0.f;
    }
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        // lanes past the row (last chunk only) take column 0 and drop what they get: no branch,
        // so the warp stays converged for the tensor-memory loads
        const bool all_in = chunk_inside<TW, VPT>(v);
        const int at = 4 * (tm.tl + TT * v);
        const int col = all_in || at < J ? at : 0;
        f32x2 gh[2], gl[2];
        load_G_chunk<true>(tG, v, nullptr, Jp, col, gh, gl);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            f32x2 c[2];
            load_C_chunk<EUC>(row[k], dxy[k], rxs, Jp, J, col, c);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // the exponent of expo2, two columns at a time
                const float2 x = unpack2(
                    add2(add2(fma2(c[h], nk_hi, Fh[k]), gh[h]), fma2(c[h], nk_lo, add2(Fl[k], gl[h]))));
                float t0 = ex2(x.x), t1 = ex2(x.y);
                if (!all_in) {
                    t0 = at + 2 * h < J ? t0 : 0.f;
                    t1 = at + 2 * h + 1 < J ? t1 : 0.f;
                }
                rsum[k] += t0;
                rsum[k] += t1;
                t[k][v][h] = pack2(t0, t1);
            }
        }
    }
    team_sum_rows<TW, R>(rsum, red, nteams, tm, par);
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (tm.tl == 0) Fnew[lr[k]].x = rsum[k];
        const float d = __fdividef(Ps[lr[k]], rsum[k]);
        const f32x2 dk = pack2(d, d);
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            acc[v][0] = fma2(t[k][v][0], dk, acc[v][0]);
            acc[v][1] = fma2(t[k][v][1], dk, acc[v][1]);
        }
    }
}

// The row updates F'^s = F'^(s-1) - log2 r of a team's rows lr0, lr0 + step, ... below `end`
// (their sums in Fnew), a lane a row, and the team's part of the residual sum p^ |r - 1| in
// units of 2^-FX_ERR, an integer so that its order does not matter.  Called by the warp that
// stored the sums.  Done for every row by a whole warp inside the sweep, this took 270 of the
// 1,370 cycles of a row of 800 columns, and FP64 in the loop test 1,000 cycles of every sync;
// without both 1000 x 50 took 8% less, 5,000 x 128 warm 7%, 48 ragged instances 3%.
__device__ __forceinline__ unsigned long long row_updates(const float2* Fold, float2* Fnew, const float* Ps, int lr0,
                                                          int step, int end, int lane) {
    unsigned long long e = 0ull;
    __syncwarp();
    for (int lr = lr0 + step * lane; lr < end; lr += step * 32) {
        const float r = Fnew[lr].x;
        Fnew[lr] = df_sub(Fold[lr], log2_corr(r));
        const float x = Ps[lr] * fabsf(r - 1.0f) * 0x1p50f;
        e += x < (float)FX_BROKEN ? __float2ull_rn(x) : FX_BROKEN;
    }
    const unsigned m = (1u << 18) - 1;
    const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)e & m);
    const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(e >> 18) & m);
    const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)(e >> 36));
    e = a + ((unsigned long long)b << 18) + ((unsigned long long)c << 36);
    return e < FX_BROKEN ? e : FX_BROKEN;
}

// The consumer warps' part of one solve (Algorithm 1 on the CTA's partitions, rows [r0, r1)):
// setup, the exact first sweep, then plan-scale sweeps until the loop test stops.  Returns
// true when the loop stopped normally (the returned plan's row potentials are then in row
// potential buffer *ret_par of shared memory, and in P.F_out when given), false when the
// instance failed or a wait gave up.  Either way s_stop is raised for the producer.
// Every decision that ends the loop is taken identically by every CTA of the group.
template <int TW, int VPT, bool EUC = false>
__device__ __forceinline__ bool sk_consumers(const SolveParams& P, const StreamCfg& S, GroupCtx& g, SkShared* sh,
                                             unsigned char* dyn, int64_t r0, int64_t r1, int* ret_par) {
    constexpr int NCW = Cons<TW>::NCW;
    constexpr int TT = 32 * TW, NTEAMS = NCW / TW, NC = NCW * 32;
    constexpr int HALF = (NTEAMS + 1) / 2;
    static_assert(4 * NTEAMS * TW <= 64 && NTEAMS <= 16 && NCW <= 16, "SkShared sizes");
    uint64_t* full = reinterpret_cast<uint64_t*>(dyn);
    uint64_t* empty = full + MAX_STAGES;
    float* comb = reinterpret_cast<float*>(dyn + SMEM_HDR);    // [ceil(NTEAMS / 2)][Jp]
    float* Gs = reinterpret_cast<float*>(dyn + S.off_G);       // [2][Jp]: G pairs (hi, lo)
    float2* Fs = reinterpret_cast<float2*>(dyn + S.off_F);     // [2][rmax]
    float* Ps = reinterpret_cast<float*>(dyn + S.off_P);       // [rmax]
    float* ring = reinterpret_cast<float*>(dyn + S.off_ring);  // [stages][stage_floats]
    const float* rxs = ring;  // Euclidean cost: RRH x then y coordinates [2][Jp]
    float* red = sh->red;
    double(*sh_sum)[2] = sh->sh_sum;
    int& s_bad = sh->s_bad;
    volatile int& s_stop = sh->s_stop;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nb = g.nb, b = g.b;
    const int V = P.V, rs_ = S.rows_per_stage;
    int v0, v1;
    cta_parts(V, b, nb, &v0, &v1);
    const int nrow = (int)max((int64_t)0, r1 - r0);
    int* status = g.status;
    const int J = P.J, Jp = P.Jp;
    const int tid = threadIdx.x;
    // stage blocks (from the CTA's first row) at which each of the CTA's partitions ends
    for (int v = v0 + tid; v < v1; v += NC) sh->pend[v - v0] = (int)((part_row(P.I, rs_, V, v + 1) - r0 + rs_ - 1) / rs_);
    const int* pend = sh->pend - v0;
#define OTA_BARRIER()                                                                              \
    do {                                                                                           \
        if (!grid_barrier_named(g.bar, (unsigned)nb * ++g.gen, g.abort, P.spin, CONS_BAR, NC, &sh->s_ok)) { \
            if (tid == 0) s_stop = 1;                                                              \
            return false;                                                                          \
        }                                                                                          \
    } while (0)
// After a barrier, leave when the instance failed before it.  Only needed when a failed instance
// does not also end every wait (batched launches keep the abort word apart from instance status).
// A write after the barrier that a CTA already sees here makes all CTAs leave before the next one.
#define OTA_BARRIER_CHECK()                                                                        \
    do {                                                                                           \
        OTA_BARRIER();                                                                             \
        if (g.abort != status && bar_named_or(CONS_BAR, NC, ld_volatile_i32(status) != DEV_OK)) {  \
            if (tid == 0) s_stop = 1;                                                              \
            return false;                                                                          \
        }                                                                                          \
    } while (0)

    // ---- setup: sums of p (per partition) and q (every CTA), checks, starting G ----------
    // An SM takes an FP64 warp instruction about every 16 cycles, so what all warps do alike in
    // FP64 adds up: the totals below, formed by all 15 of them, took 17,000 cycles, log2 q^ by
    // the warps of a few CTAs 11,000.  Sums are formed by the warps that hold terms (an absent
    // term is a zero), combined by one warp, and columns are dealt to the CTAs one warp each.
    const int swarp = warp * nb + b, nw = nb * NCW;  // this warp among the group's, CTA by CTA
    {
        int bad = 0;
        for (int v = v0; v < v1; ++v) {
            const int a = (int)(part_row(P.I, rs_, V, v) - r0), e = (int)(part_row(P.I, rs_, V, v + 1) - r0);
            double sp = 0.0;
            for (int r = a + tid; r < e; r += NC) {
                const float x = __ldg(P.p + r0 + r);
                bad |= !(x > 0.0f) || !isfinite(x);
                sp += (double)x;
                Ps[r] = x;
            }
            if (warp * 32 < e - a) {
                sp = warp_sum(sp);
                if (lane == 0) sh_sum[warp][0] = sp;
            }
            bar_named(CONS_BAR, NC);
            if (tid == 0) {
                double t = 0.0;
                for (int w = 0; w < NCW && w * 32 < e - a; ++w) t += sh_sum[w][0];
                P.errpart[v] = t;
            }
            bar_named(CONS_BAR, NC);
        }
        for (int j = swarp * 32 + lane; j < J; j += nw * 32) {
            const double g0 = P.g_warm ? P.g_warm[j] * P.k : 0.0;
            bad |= !isfinite(g0);
            P.G[j] = g0;
            gs_pairs(P.G, Jp)[j] = split_pair(g0);
        }
        if (b == 0 && tid == 0 && P.input_bad && *P.input_bad) bad = 1;
        if (bad) atomicOr(&s_bad, 1);
        bar_named(CONS_BAR, NC);
        if (tid == 0 && s_bad) atomicCAS(status, DEV_OK, DEV_EINVAL);
    }
    OTA_BARRIER_CHECK();
    double inv_sq;
    float inv_sp_f;
    {
        // every CTA forms the same totals in the same order
        double a = 0.0, c = 0.0;
        int badq = 0;
        if (warp * 32 < V) {
            for (int bb = tid; bb < V; bb += NC) a += P.errpart[bb];
            a = warp_sum(a);
        }
        if (warp * 32 < J) {
            for (int j = tid; j < J; j += NC) {
                const float x = __ldcg(P.q + j);
                badq |= !(x > 0.0f) || !isfinite(x);
                c += (double)x;
            }
            c = warp_sum(c);
        }
        if (tid == 0) s_bad = 0;
        bar_named(CONS_BAR, NC);
        if (lane == 0) {
            sh_sum[warp][0] = a;
            sh_sum[warp][1] = c;
        }
        if (badq) atomicOr(&s_bad, 1);
        bar_named(CONS_BAR, NC);
        if (warp == 0) {  // lane 0 the sum of p, lane 1 of q
            double t = 0.0;
            for (int w = 0; w < NCW; ++w) t += sh_sum[w][lane & 1];
            const double inv = 1.0 / t;
            const double sp = __shfl_sync(0xffffffffu, t, 0), sq = __shfl_sync(0xffffffffu, t, 1);
            const double inv_p = __shfl_sync(0xffffffffu, inv, 0), inv_q = __shfl_sync(0xffffffffu, inv, 1);
            __syncwarp();
            if (lane == 0) {
                sh->s_dec = s_bad || !(fabs(sp - sq) <= 1e-5 * sp);
                sh_sum[0][0] = inv_q;
                sh_sum[0][1] = inv_p;
                if (b == 0 && !sh->s_dec) {
                    P.sc->sp = sp;
                    P.sc->sq = sq;
                    P.sc->inv_sp = inv_p;
                    P.sc->inv_sq = inv_q;
                    P.sc->inv_sp_f = (float)inv_p;
                    P.sc->status = DEV_OK;
                }
            }
        }
        bar_named(CONS_BAR, NC);
        if (sh->s_dec) {
            if (b == 0 && tid == 0) atomicCAS(status, DEV_OK, DEV_EINVAL);
            if (tid == 0) s_stop = 1;
            return false;  // the same decision in every CTA
        }
        inv_sq = sh_sum[0][0];
        inv_sp_f = (float)sh_sum[0][1];
    }
    double* LQ = P.G + 2 * Jp;  // log2 q^_j, formed once here (read after the next grid barrier)
    float2* LQ2 = gs_lq2(P.G, Jp);
    int* SX = gs_sx(P.G, Jp);
    unsigned long long* ACC = gs_acc(P.G, Jp);
    {
        for (int j = swarp * 32 + lane; j < J; j += nw * 32) {
            const double lq = log2((double)__ldcg(P.q + j) * inv_sq);
            LQ[j] = lq;
            LQ2[j] = split_pair(lq);
            // the total of column j is about 2^FX_BITS when its sum is q^_j; shifts that the
            // FP32 scale cannot carry send the column to the exact path (shift 0 = "never")
            const int sx = FX_BITS - (int)floor(lq);
            SX[j] = sx <= 126 ? sx : 0;
        }
        for (int t = swarp * 32 + lane; t < 2 * (Jp + 4); t += nw * 32) ACC[t] = 0ull;
        for (int r = tid; r < nrow; r += NC) Ps[r] *= inv_sp_f;  // p^_i
        bar_named(CONS_BAR, NC);
    }
    const Team<TW> tm;
    RingPos pos;
    if (P.F_in) {  // finalize only
        for (int r = tid; r < nrow; r += NC) Fs[r] = P.F_in[r0 + r];
        load_G_smem(P.G_in, J, Jp, Gs, tid, NC);
        bar_named(CONS_BAR, NC);
        G_to_tmem<TW, VPT>(sh->tmem, Gs, Jp, tm);
        *ret_par = 0;
        sk_finalize_sweep<TW, VPT, EUC>(P, S, sh, dyn, r0, nrow, v0, v1, Fs, pos, g.abort);
        if (tid == 0) s_stop = 1;
        return true;
    }
    load_G_pairs(gs_pairs(P.G, Jp), J, Jp, Gs, tid, NC);
    bar_named(CONS_BAR, NC);
    G_to_tmem<TW, VPT>(sh->tmem, Gs, Jp, tm);
    const uint32_t tG = tmem_G<TW, VPT>(sh->tmem, tm);
    const f32x2 nk_hi = pack2(-P.k_hi, -P.k_hi), nk_lo = pack2(-P.k_lo, -P.k_lo);
    int par = 0;

    // ---- sweep 1: the log-domain iteration from G^0 with a fixed column scale --------------
    // Every row of the half-step plan is normalised (t_ij = pi_ij / p_i <= 1 after the row
    // shift), so the column sums of p^_i t_ij 2^64 cannot overflow: one ex2 a cell, like the
    // later sweeps.  A column whose scaled sum falls below 2^-60 (a true sum below 2^-124) is
    // marked, and then the whole first iteration is taken again in the exact form below (an
    // online (max, sum) pair per column) on the next pass of the stream.
    unsigned long long* flag1 = ACC + Jp + 1;  // zeroed with the totals in setup
    bool exact1 = false;
    {
        f32x2 acc[VPT][2];
#pragma unroll
        for (int v = 0; v < VPT; ++v) acc[v][0] = acc[v][1] = 0ull;
        float2* F1 = Fs + S.rmax;  // F'^1 lives in buffer 1
        int kb = 0;
        for (int vp = v0; vp < v1; ++vp) {
            const int vend = pend[vp];
            for (; kb < vend; ++kb) {
                const int st = pos.st;
                if (!EUC) pos.wait(full, P.spin, g.abort);
                const int lr0 = kb * rs_;
                const int rows = min(rs_, nrow - lr0);
                const float* stage = ring + (size_t)st * S.stage_floats;
                for (int j = 0; j < S.rpt; ++j) {
                    const int rr = tm.team + NTEAMS * j;
                    if (rr >= rows) break;
                    const float* row = stage + (size_t)rr * P.ld;
                    const float2 dxy = EUC ? __ldg(P.dev_xy + r0 + lr0 + rr) : make_float2(0.f, 0.f);
                    f32x2 x[VPT][2];
                    float m = -INFINITY;  // row maximum of G^0 - k C (approximate: only a shift)
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < VPT; ++v) {  // lanes past the row: as in sweep_rows
                        const bool all_in = chunk_inside<TW, VPT>(v);
                        const int at = 4 * (tm.tl + TT * v);
                        const int col = all_in || at < J ? at : 0;
                        f32x2 gh[2], gl[2];
                        load_G_chunk<true>(tG, v, nullptr, Jp, col, gh, gl);
                        load_C_chunk<EUC>(row, dxy, rxs, Jp, J, col, x[v]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float2 y = unpack2(fma2(x[v][h], nk_hi, gh[h]));
                            if (all_in || at + 2 * h < J) m = fmaxf(m, y.x);
                            if (all_in || at + 2 * h + 1 < J) m = fmaxf(m, y.y);
                        }
                    }
                    m = team_reduce<TW, float, true>(m, red, NTEAMS, tm, par);
                    const f32x2 nm = pack2(-m, -m);
                    float sum = 0.f;
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < VPT; ++v) {
                        const bool all_in = chunk_inside<TW, VPT>(v);
                        const int at = 4 * (tm.tl + TT * v);
                        f32x2 gh[2], gl[2];
                        load_G_chunk<true>(tG, v, nullptr, Jp, at, gh, gl);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float2 y = unpack2(add2(add2(fma2(x[v][h], nk_hi, nm), gh[h]), fma2(x[v][h], nk_lo, gl[h])));
                            float t0 = ex2(y.x), t1 = ex2(y.y);
                            if (!all_in) {
                                t0 = at + 2 * h < J ? t0 : 0.f;
                                t1 = at + 2 * h + 1 < J ? t1 : 0.f;
                            }
                            sum += t0;
                            sum += t1;
                            x[v][h] = pack2(t0, t1);
                        }
                    }
                    sum = team_reduce<TW, float, false>(sum, red, NTEAMS, tm, par);
                    const float ls = log2f(sum);
                    if (tm.tl == 0) {  // F'^1 = -LSE2_j(y) = -(m + log2 sum), exact as an FP32 pair
                        float hi, lo;
                        two_sum(m, ls, hi, lo);
                        F1[lr0 + rr] = make_float2(-hi, -lo);
                    }
                    const float w = __fdividef(Ps[lr0 + rr], sum) * 0x1p64f;  // p^_i 2^64 / sum
                    const f32x2 w2 = pack2(w, w);
#pragma unroll
                    for (int v = 0; v < VPT; ++v) {
                        acc[v][0] = fma2(x[v][0], w2, acc[v][0]);
                        acc[v][1] = fma2(x[v][1], w2, acc[v][1]);
                    }
                }
                __syncwarp();
                if (!EUC && lane == 0) pos.release(empty, st);
                pos.next(S.stages);
            }
            float* cp = P.colpart + (int64_t)vp * Jp;
            float4 part[VPT];
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                const float2 u = unpack2(acc[v][0]), w = unpack2(acc[v][1]);
                part[v] = make_float4(u.x, u.y, w.x, w.y);
                acc[v][0] = acc[v][1] = 0ull;
            }
            cta_col_sum<TW, VPT>(comb, part, J, Jp, tm, [&](int j, float sum) { cp[j] = sum; });
        }
        tmem_fence_before();  // this sweep's reads of G, before the barriers that precede its next copy
        OTA_BARRIER();
        // G^1_j = G^0_j + log2 q^_j - log2(column sum of pi^(1/2)), one warp per column
        {
            for (int j = swarp; j < J; j += nw) {
                float2 sum = make_float2(0.f, 0.f);
                for (int bb = lane; bb < V; bb += 32) sum = df_add(sum, P.colpart[(int64_t)bb * Jp + j]);
                sum = warp_sum_df(sum);
                if (lane == 0) {
                    if (!(sum.x >= 0x1p-60f) || !isfinite(sum.x)) {
                        atomicOr(flag1, 1ull);
                    } else {
                        const float2 ls = df_log2(sum);
                        const double g1 = P.G[j] + LQ[j] - (((double)ls.x - 64.0) + (double)ls.y);
                        P.G[Jp + j] = g1;
                        gs_pairs(P.G, Jp)[j] = split_pair(g1);
                    }
                }
            }
        }
        OTA_BARRIER_CHECK();
        exact1 = __ldcg(flag1) != 0ull;
        if (!exact1) {
            load_G_pairs(gs_pairs(P.G, Jp), J, Jp, Gs, tid, NC);
            bar_named(CONS_BAR, NC);
        }
    }
    // ---- sweep 1 again, exact log-domain form (a column sum below the fixed scale's range) --
    if (exact1) {
        float4 M[VPT], Sm[VPT];
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            M[v] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            Sm[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float2* F1 = Fs + S.rmax;  // F'^1 lives in buffer 1
        float2* part2 = reinterpret_cast<float2*>(P.colpart);
        int kb = 0;
        for (int vp = v0; vp < v1; ++vp) {
          const int vend = pend[vp];
          for (; kb < vend; ++kb) {
            const int st = pos.st;
            if (!EUC) pos.wait(full, P.spin, g.abort);
            const int lr0 = kb * rs_;
            const int rows = min(rs_, nrow - lr0);
            const float* stage = ring + (size_t)st * S.stage_floats;
            for (int j = 0; j < S.rpt; ++j) {
                const int rr = tm.team + NTEAMS * j;
                if (rr >= rows) break;
                float4 x[VPT];
                if constexpr (EUC)
                    euclid_row<TW, VPT>(__ldg(P.dev_xy + r0 + lr0 + rr), rxs, rxs + Jp, J, tm.tl, x);
                else
                    load_row_smem<TW, VPT>(stage + (size_t)rr * P.ld, J, tm.tl, x);
                // row maximum of y = G0 - k C (approximate values suffice for the shift)
                float m = -INFINITY;
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int col = 4 * (tm.tl + TT * v);
                    float4 gv = col < Jp ? *reinterpret_cast<const float4*>(Gs + col) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < 4; ++c) m = fmaxf(m, fmaf(-comp(x[v], c), P.k_hi, comp(gv, c)));
                }
                m = team_reduce<TW, float, true>(m, red, NTEAMS, tm, par);
                // z = y - m with the large parts cancelled by the exact product
                float s = 0.f;
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int col = 4 * (tm.tl + TT * v);
                    float4 gv = col < Jp ? *reinterpret_cast<const float4*>(Gs + col) : make_float4(0.f, 0.f, 0.f, 0.f);
                    float4 gl = col < Jp ? *reinterpret_cast<const float4*>(Gs + Jp + col) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float z = expo2(-m, comp(gl, c), comp(gv, c), comp(x[v], c), P.k_hi, P.k_lo);
                        comp(x[v], c) = z;
                        s += ex2(z);
                    }
                }
                s = team_reduce<TW, float, false>(s, red, NTEAMS, tm, par);
                const float ls = log2f(s);
                if (tm.tl == 0) {  // F'^1 = -LSE2_j(y) = -(m + log2 s), exact as an FP32 pair
                    float hi, lo;
                    two_sum(m, ls, hi, lo);
                    F1[lr0 + rr] = make_float2(-hi, -lo);
                }
                const float cst = log2f(Ps[lr0 + rr]) - ls;
#pragma unroll
                for (int v = 0; v < VPT; ++v)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        // online (max, sum) of log2 pi^(1/2)_ij, without a branch: a divergent
                        // branch per cell costs more than the second ex2.  The floor keeps
                        // -inf - -inf (a column no row reaches yet) out of the exponent.
                        const float u = comp(x[v], c) + cst;
                        float& Mc = comp(M[v], c);
                        float& Sc = comp(Sm[v], c);
                        const float mn = fmaxf(fmaxf(Mc, u), -1e30f);
                        Sc = fmaf(Sc, ex2(Mc - mn), ex2(u - mn));
                        Mc = mn;
                    }
            }
            __syncwarp();
            if (!EUC && lane == 0) pos.release(empty, st);
            pos.next(S.stages);
          }
            // end of partition vp: merge the teams' (max, sum) pairs in two rounds through
            // the float buffer, the column maxima first (held in Gs meanwhile), then the sums
            // rescaled to them; teams in a fixed order.  Gs gets G^0 back afterwards.
            for (int round = 0; round < 2; ++round) {  // the first half stores, the second half merges
                if ((tm.team < HALF) == (round == 0)) {
                    const int slot = round == 0 ? tm.team : tm.team - HALF;
#pragma unroll
                    for (int v = 0; v < VPT; ++v) {
                        const int col = 4 * (tm.tl + TT * v);
                        if (col < Jp) {
                            float4* d = reinterpret_cast<float4*>(comb + slot * Jp + col);
                            if (round == 0) {
                                *d = M[v];
                            } else {
                                float4 o = *d;
                                o.x = fmaxf(o.x, M[v].x);
                                o.y = fmaxf(o.y, M[v].y);
                                o.z = fmaxf(o.z, M[v].z);
                                o.w = fmaxf(o.w, M[v].w);
                                *d = o;
                            }
                        }
                    }
                }
                bar_named(CONS_BAR, NC);
            }
            for (int j = tid; j < Jp; j += NC) {
                float mm = comb[j];
                for (int t = 1; t < HALF; ++t) mm = fmaxf(mm, comb[t * Jp + j]);
                Gs[j] = mm;
            }
            bar_named(CONS_BAR, NC);
            for (int round = 0; round < 2; ++round) {
                if ((tm.team < HALF) == (round == 0)) {
                    const int slot = round == 0 ? tm.team : tm.team - HALF;
#pragma unroll
                    for (int v = 0; v < VPT; ++v) {
                        const int col = 4 * (tm.tl + TT * v);
                        if (col < Jp) {
                            float4 sc;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const float Mc = comp(M[v], c), mm = Gs[col + c];
                                comp(sc, c) = Mc > -INFINITY ? comp(Sm[v], c) * ex2(Mc - mm) : 0.f;
                            }
                            float4* d = reinterpret_cast<float4*>(comb + slot * Jp + col);
                            if (round == 0) {
                                *d = sc;
                            } else {
                                float4 o = *d;
                                o.x += sc.x;
                                o.y += sc.y;
                                o.z += sc.z;
                                o.w += sc.w;
                                *d = o;
                            }
                        }
                    }
                }
                bar_named(CONS_BAR, NC);
            }
            for (int j = tid; j < J; j += NC) {
                float ss = comb[j];
                for (int t = 1; t < HALF; ++t) ss += comb[t * Jp + j];
                part2[(int64_t)vp * Jp + j] = make_float2(Gs[j], ss);
            }
            bar_named(CONS_BAR, NC);
            load_G_smem(P.G, J, Jp, Gs, tid, NC);
            bar_named(CONS_BAR, NC);
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                M[v] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                Sm[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        OTA_BARRIER();
        // G^1_j = G^0_j + log2 q^_j - log2(column sum of pi^(1/2)), one warp per column
        {
            for (int j = swarp; j < J; j += nw) {
                float mm = -INFINITY;
                for (int bb = lane; bb < V; bb += 32) mm = fmaxf(mm, part2[(int64_t)bb * Jp + j].x);
                mm = warp_max(mm);
                double ss = 0.0;
                if (mm > -INFINITY)
                    for (int bb = lane; bb < V; bb += 32) {
                        const float2 o = part2[(int64_t)bb * Jp + j];
                        if (o.x > -INFINITY) ss += (double)o.y * (double)ex2(o.x - mm);
                    }
                ss = warp_sum(ss);
                if (lane == 0) {
                    if (!(ss > 0.0) || !isfinite(ss)) {
                        atomicCAS(status, DEV_OK, DEV_ENUMERIC);
                    } else {
                        P.G[Jp + j] = P.G[j] + LQ[j] - ((double)mm + log2(ss));
                    }
                }
            }
        }
        OTA_BARRIER_CHECK();
        load_G_smem(P.G + Jp, J, Jp, Gs, tid, NC);
        bar_named(CONS_BAR, NC);
    }

    if (P.init_only) {  // iteration 1 is all that was asked for: no sweep to test its plan
        if (P.F_out)
            for (int r = tid; r < nrow; r += NC) P.F_out[r0 + r] = Fs[S.rmax + r];
        if (b == 0 && tid == 0) {
            P.st->iters = 1;
            P.st->err = 0.0;
            P.st->converged = 0;
        }
        *ret_par = 1;
        if (tid == 0) s_stop = 1;
        return true;
    }

    // ---- sweeps 2, 3, ...: one read of C and one ex2 per cell -----------------------------
    // Each partition adds its column partials (and row residual) as fixed-point integers into
    // the row of totals of this sweep; every CTA waits for the totals themselves and forms all
    // column updates in its shared-memory copy of G.
    //
    // The sync bounds small instances (it is half of an iteration up to 20,000 x 400) and idles
    // HBM in large ones.  A grid barrier cost three dependent trips through L2 (the adds have to
    // land before the arrival is released, the arrival, the totals); waiting on the counted
    // totals costs one: by itself 16% of a 1000 x 50 solve, 8% of 5,000 x 128 warm, 4% of
    // 12,347 x 1,021 packed, 2% of 50,000 x 800.
    constexpr int UC = (4 * TT * VPT + NC - 1) / NC;  // columns a thread looks after: tid + NC u
    constexpr int CU = UC < 3 ? UC : 3;               // and how many at a time
    static_assert(UC <= 32, "one mask word");
    unsigned long long prev[2][UC];  // the rows' words when last complete (the residual's: sh->err_was)
#pragma unroll
    for (int u = 0; u < UC; ++u) prev[0][u] = prev[1][u] = 0ull;
    if (tid == 0) {
        sh->flags[0] = sh->flags[1] = 0;  // a barrier follows (G_to_tmem)
        sh->err_was[0][0] = sh->err_was[0][1] = sh->err_was[1][0] = sh->err_was[1][1] = 0ull;
    }
    const unsigned long long stop_units = fx_stop_units(stop_tol(P.tol) * 0x1p50);
    constexpr int RPP = rows_per_pass<TW, VPT, EUC>();
    // a step takes two blocks where a team's rows of one do not fill its passes, if the ring has
    // stages to spare for that
    const int step_blocks = S.rpt % RPP != 0 && S.stages >= 4 ? 2 : 1;
    G_to_tmem<TW, VPT>(sh->tmem, Gs, Jp, tm);
    for (int s = 2;; ++s) {
        unsigned long long* acc_s = ACC + (size_t)(s & 1) * (Jp + 4);
        const float2* Fold = Fs + ((s - 1) & 1) * S.rmax;  // F'^(s-1)
        float2* Fnew = Fs + (s & 1) * S.rmax;
        f32x2 acc[VPT][2];
#pragma unroll
        for (int v = 0; v < VPT; ++v) acc[v][0] = acc[v][1] = 0ull;
        int kb = 0;
        for (int vp = v0; vp < v1; ++vp) {
          const int vend = pend[vp];
          const int kb0 = kb;
          while (kb < vend) {
            // a step: one stage block, or two when a team's rows in a block do not pair up
            const int nblk = min(step_blocks, vend - kb);
            if (!EUC) pos.wait(full, P.spin, g.abort);
            const int st0 = pos.st;
            pos.next(S.stages);
            const int st1 = pos.st;
            if (nblk == 2) {
                if (!EUC) pos.wait(full, P.spin, g.abort);
                pos.next(S.stages);
            }
            const float* stage0 = ring + (size_t)st0 * S.stage_floats + (size_t)tm.team * P.ld;
            const float* stage1 = ring + (size_t)st1 * S.stage_floats + (size_t)tm.team * P.ld;
            const int lr0 = kb * rs_ + tm.team;  // the team's rows are lr0 + NTEAMS q
            const int nq = min(nblk * S.rpt, (nrow - lr0 + NTEAMS - 1) / NTEAMS);
            auto staged = [&](int q) {
                return q < S.rpt ? stage0 + (size_t)(NTEAMS * q) * P.ld : stage1 + (size_t)(NTEAMS * (q - S.rpt)) * P.ld;
            };
            auto pass = [&](auto rows, int q) {
                constexpr int R = decltype(rows)::value;
                int lr[R];
                const float* row[R];
                float2 dxy[R];
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    lr[k] = lr0 + NTEAMS * (q + k);
                    row[k] = staged(q + k);
                    dxy[k] = EUC ? __ldg(P.dev_xy + r0 + lr[k]) : make_float2(0.f, 0.f);
                }
                sweep_rows<TW, VPT, EUC, R>(row, dxy, tG, J, Jp, rxs, nk_hi, nk_lo, Fold, Fnew, Ps, lr, red, NTEAMS, tm, par,
                                            acc);
            };
            for (int q = 0; q < nq;) {
                if constexpr (RPP == 2)
                    if (q + 1 < nq) {
                        pass(std::integral_constant<int, 2>(), q);
                        q += 2;
                        continue;
                    }
                pass(std::integral_constant<int, 1>(), q);
                ++q;
            }
            __syncwarp();
            if (!EUC && lane == 0) {
                pos.release(empty, st0);
                if (nblk == 2) pos.release(empty, st1);
            }
            kb += nblk;
          }
            // end of partition vp: its column partials (teams in order, as cta_col_sum) and row
            // residual.  The FP32 partial is kept for the exact path and added to the column's
            // total as round(partial 2^S_j); one too large for the total adds 2^FX_TOP, which
            // sends the column there.
            if (tm.wit == 0) {
                const unsigned long long e =
                    row_updates(Fold, Fnew, Ps, kb0 * rs_ + tm.team, NTEAMS, min(vend * rs_, nrow), lane);
                if (lane == 0) sh->werr[tm.team] = e;
            }
            int sx[CU];  // of this thread's first columns: on the way while the teams merge
#pragma unroll
            for (int u = 0; u < CU; ++u) sx[u] = tid + u * NC < J ? __ldcg(SX + tid + u * NC) : 0;
            if (tm.team < HALF) {
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int col = 4 * (tm.tl + TT * v);
                    if (col < Jp) *reinterpret_cast<ulonglong2*>(comb + tm.team * Jp + col) = make_ulonglong2(acc[v][0], acc[v][1]);
                }
            }
            bar_named(CONS_BAR, NC);
            if (tid == 0) {  // its team is done; the other half merges meanwhile
                unsigned long long e = 0ull;
#pragma unroll
                for (int t = 0; t < NTEAMS; ++t) e += sh->werr[t];
                atomicAdd(acc_s + Jp, (unsigned long long)(FX_ONE + fx_err_low(e)));
                atomicAdd(acc_s + Jp + 2, (unsigned long long)(FX_ONE + fx_err_high(e)));
            }
            if (tm.team >= HALF) {
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int col = 4 * (tm.tl + TT * v);
                    if (col < Jp) {
                        ulonglong2* d = reinterpret_cast<ulonglong2*>(comb + (tm.team - HALF) * Jp + col);
                        const ulonglong2 o = *d;
                        *d = make_ulonglong2(add2(o.x, acc[v][0]), add2(o.y, acc[v][1]));
                    }
                }
            }
            bar_named(CONS_BAR, NC);
            float* cp = P.colpart + (int64_t)vp * Jp;
            auto add_total = [&](int j, int sxj) {
                float sum = comb[j];
                for (int t = 1; t < HALF; ++t) sum += comb[t * Jp + j];
                cp[j] = sum;
                const float x = sum * __int_as_float((sxj + 127) << 23);  // S_j <= 126; 0 for "never"
                const bool fits = sxj != 0 && x < (float)(1ull << FX_TOP);
                atomicAdd(acc_s + j, FX_ONE + (fits ? __float2ull_rn(x) : 1ull << FX_TOP));
            };
#pragma unroll
            for (int u = 0; u < CU; ++u)
                if (tid + u * NC < J) add_total(tid + u * NC, sx[u]);
            for (int j = tid + CU * NC; j < J; j += NC) add_total(j, __ldcg(SX + j));
#pragma unroll
            for (int v = 0; v < VPT; ++v) acc[v][0] = acc[v][1] = 0ull;
            if (vp + 1 < v1) bar_named(CONS_BAR, NC);  // comb and werr are free again
        }
        // a CTA without a partition counts itself into the residual words: it has read the other row
        if (v0 == v1 && tid == 0) {
            atomicAdd(acc_s + Jp, (unsigned long long)FX_ONE);
            atomicAdd(acc_s + Jp + 2, (unsigned long long)FX_ONE);
        }
        tmem_fence_before();  // this sweep's reads of G, before the barriers that precede its next copy
        // G^s_j = G^(s-1)_j + log2 q^_j - log2 s_j, every column in every CTA (FP32 pairs).  The
        // sum s_j is the fixed-point total T_j 2^-S_j; a column whose total is too large or too
        // small to carry 30 bits is summed exactly from the partitions' FP32 partials instead.
        unsigned exact = 0;  // of this thread's columns
        int* flags = &sh->flags[s & 1];
        for (int u0 = 0; u0 < UC; u0 += CU) {
            unsigned long long A[CU], was[CU];
            float2 lq[CU];
            int sx[CU];
#pragma unroll
            for (int u = 0; u < CU; ++u) {  // constants of the columns, on the way during the wait
                const int j = tid + (u0 + u) * NC;
                const bool in = u0 + u < UC && j < J;
                lq[u] = in ? __ldcg(LQ2 + j) : make_float2(0.f, 0.f);
                sx[u] = in ? __ldcg(SX + j) : 0;
                was[u] = in ? prev[s & 1][u0 + u] : 0ull;
            }
            const bool first = u0 == 0;
            long long n = 0;
            for (;;) {  // until every addition due to this thread's words has arrived
                bool all = true;
                unsigned long long lo = 0ull, hi = 0ull;  // the residual's words
#pragma unroll
                for (int u = 0; u < CU; ++u) {
                    const int j = tid + (u0 + u) * NC;
                    A[u] = u0 + u < UC && j < J ? ld_relaxed_u64(acc_s + j) : was[u] + ((unsigned long long)fx_due_col(V) << FX_COUNT);
                }
                if (first && tid == 0) {
                    lo = ld_relaxed_u64(acc_s + Jp);
                    hi = ld_relaxed_u64(acc_s + Jp + 2);
                }
#pragma unroll
                for (int u = 0; u < CU; ++u) all = all && fx_complete(A[u], was[u], fx_due_col(V));
                if (first && tid == 0) {
                    unsigned long long* ew = sh->err_was[s & 1];
                    all = all && fx_complete(lo, ew[0], fx_due_err(V, nb)) && fx_complete(hi, ew[1], fx_due_err(V, nb));
                    if (all) {
                        sh->s_err = fx_err(fx_value(lo, ew[0]), fx_value(hi, ew[1]));
                        ew[0] = lo;
                        ew[1] = hi;
                    }
                }
                if (all) {
#pragma unroll
                    for (int u = 0; u < CU; ++u)
                        if (u0 + u < UC) prev[s & 1][u0 + u] = A[u];
                    break;
                }
                ++n;
                if ((n & 63) == 0 && ld_volatile_i32(g.abort) != DEV_OK) {
                    atomicOr(flags, first ? SK_LATE : SK_LATER);
                    break;
                }
                if (n > P.spin) {
                    atomicCAS(g.abort, DEV_OK, DEV_ETIMEOUT);
                    atomicOr(flags, first ? SK_LATE : SK_LATER);
                    break;
                }
                if (n > 256) __nanosleep(32);
            }
            if (first) {
                bar_named(CONS_BAR, NC);
                if (*(volatile int*)flags & SK_LATE) {
                    if (tid == 0) s_stop = 1;
                    return false;
                }
                if (tid == 0) sh->flags[(s + 1) & 1] = 0;  // read last before the barrier that ended sweep s - 1
                // Loop test on pi^(s-1): every CTA reads the same total of the row residuals.
                // (in integers: FP64 in every warp would take a thousand cycles of every sync)
                const bool conv = sh->s_err <= stop_units;
                if (conv || s - 1 >= P.max_iter) {
                    if (b == 0 && tid == 0) {
                        P.st->iters = s - 1;
                        P.st->err = (double)sh->s_err * 0x1p-50;
                        P.st->converged = conv;
                    }
                    if (s > 2)  // the FP64 copy of G^(s-1) (G^1 is there already), each column once
                        for (int j = b * NC + tid; j < J; j += nb * NC)
                            P.G[((s - 1) & 1) * Jp + j] = (double)Gs[j] + (double)Gs[Jp + j];
                    if (P.F_out)
                        for (int r = tid; r < nrow; r += NC) P.F_out[r0 + r] = Fold[r];
                    *ret_par = (s - 1) & 1;
                    if (P.fpart) sk_finalize_sweep<TW, VPT, EUC>(P, S, sh, dyn, r0, nrow, v0, v1, Fold, pos, g.abort);
                    if (tid == 0) s_stop = 1;
                    return true;
                }
            }
#pragma unroll
            for (int u = 0; u < CU; ++u) {
                const int j = tid + (u0 + u) * NC;
                const unsigned long long T = fx_value(A[u], was[u]);
                const bool in = u0 + u < UC && j < J;
                const bool ok = T >= (1ull << 30) && T < (1ull << FX_TOP);
                const float th = __ull2float_rn(T);
                const float tl = (float)((long long)T - (long long)__float2ull_rn(th));
                float2 ls = df_log2(make_float2(ok ? th : 1.f, ok ? tl : 0.f));
                ls.x -= (float)sx[u];
                const float2 d = df_add2(lq[u], make_float2(-ls.x, -ls.y));
                const int jr = in ? j : 0;
                const float2 Gn = df_add2(make_float2(Gs[jr], Gs[Jp + jr]), d);
                if (in && ok) {
                    Gs[j] = Gn.x;
                    Gs[Jp + j] = Gn.y;
                }
                if (in && !ok) exact |= 1u << (u0 + u);
            }
        }
        if (exact) atomicOr(flags, SK_EXACT);
        bar_named(CONS_BAR, NC);
        const int fl = *(volatile int*)flags;
        if (fl & SK_LATER) {
            if (tid == 0) s_stop = 1;
            return false;
        }
        if (fl) {  // every CTA sees the same totals and comes here or not; the partials need a barrier
            OTA_BARRIER();
            int bad = 0;
            for (int u = 0; u < UC; ++u) {
                if (!(exact >> u & 1u)) continue;
                const int j = tid + u * NC;
                float2 sum = make_float2(0.f, 0.f);
                for (int v = 0; v < V; ++v) sum = df_add(sum, __ldcg(P.colpart + (int64_t)v * Jp + j));
                if (!(sum.x > 0.f) || !isfinite(sum.x)) {
                    bad = 1;
                    continue;
                }
                const float2 ls = df_log2(sum);
                const float2 d = df_add2(__ldcg(LQ2 + j), make_float2(-ls.x, -ls.y));
                const float2 Gn = df_add2(make_float2(Gs[j], Gs[Jp + j]), d);
                Gs[j] = Gn.x;
                Gs[Jp + j] = Gn.y;
            }
            if (bad) atomicOr(flags, SK_BAD);
            OTA_BARRIER();  // the partials are read before any CTA writes the next sweep's
            if (*(volatile int*)flags & SK_BAD) {  // the same decision in every CTA
                if (tid == 0) atomicCAS(status, DEV_OK, DEV_ENUMERIC);
                if (tid == 0) s_stop = 1;
                return false;
            }
        }
        G_to_tmem<TW, VPT>(sh->tmem, Gs, Jp, tm);
    }
#undef OTA_BARRIER_CHECK
#undef OTA_BARRIER
}

}  // namespace ota
