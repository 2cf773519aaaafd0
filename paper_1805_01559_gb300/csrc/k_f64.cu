// FP64 Sinkhorn in the log domain (Algorithm 1 of the paper, Sec. III-B), every per-cell
// operation in double precision.  A reference-precision path for small instances (the
// 1000 x 50 configuration): GB300 issues FP64 at a small fraction of its FP32 rate (a warp
// instruction about every 16 cycles an SM), so the FP32 persistent solver is the fast path and
// this one is for checking it.
//
// One cooperative launch.  Iteration 1 is the log-sum-exp form,
//   row update     f_i = eps log p^_i - eps LSE_j((g_j - C_ij) / eps)
//   column update  g_j = eps log q^_j - eps LSE_i((f_i - C_ij) / eps)
// (LSE with the maximum factored out), which no start can underflow.  Afterwards every plan
// pi = exp((f + g - C) / eps) has exact columns and rows of at least min q^ of their mass, so
// an iteration forms each pi_ij once: its row sums give f_i += eps log(p^_i / r_i), and the
// column sums of pi_ij p^_i / r_i give g_j += eps log(q^_j / s_j).  Masses that differ by
// hundreds of decades can still take r_i (down to p^_i min q^) or s_j below the range of a
// double: a row or column whose sum is under F64_LOW is formed with its maximum factored out.
//
// What bounds it is the FP64 pipe: an exponential is some twenty instructions.  So a cell's
// exponential is formed once an iteration (tiles of up to 8 rows in shared memory, summed by
// row, then by column), by every SM, and per-row logarithms are taken a tile at a time.  With
// two passes over the row and two over the column (the column's by one warp a column, 50 of
// them on 1000 x 50) an iteration took 97 us and the solve of 26 iterations 2.50 ms; it takes
// 0.46 ms now, with the same error (1e-14) against a plain FP64 reference.
//
// As in the FP32 solver, the row update of iteration s also gives the row residual of the plan
// of iteration s - 1 (p^_i |exp((f_i^(s-1) - f_i^s) / eps) - 1|), the loop test ("while
// accuracy") is taken on it, and a stop returns that plan's potentials.  Masses are normalised
// to 1 while iterating; f is shifted by eps log(sum p) at the end so that
// pi = exp((f + g - C) / eps) carries the caller's mass.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "ot_common.cuh"
#include "ot_internal.h"

namespace ota {

static constexpr int F64_NT = 256;
static constexpr int F64_NW = F64_NT / 32;
enum : int { F64_ENUMERIC = -7 };
// Terms lost below 2^-1022 are under 2^-122 of such a sum.
static constexpr double F64_LOW = 0x1p-900;

struct F64State {
    unsigned bar;
    int status;
    int iters;
    int converged;
    double err;
    double sp, sq;
};

struct F64Params {
    const double* C;
    int64_t ld;
    int64_t I;
    int J;
    const double* p;
    const double* q;
    const double* g_warm;
    double eps, tol;
    int max_iter;
    double* fb;     // [2][I] row potentials, unit mass (buffer s & 1 holds f^s)
    double* gb;     // [2][J] column potentials (buffer s & 1 holds g^s)
    double* part;   // [grid][4] per-CTA partial sums
    double2* colp;  // [min(grid, tiles)][J] column sums of the CTAs with tiles, or null for a grid of one CTA
    int rows;       // rows of a tile: 8, 4, 2 or 1
    F64State* st;
    // outputs
    double* f_out;
    double* g_out;
    double* rrh_load;
    float* pi;
    int64_t pi_ld;
    SolveSummary* summ;
    long long spin;
};

// Block sum of one double per thread, in a fixed order; every thread gets the total.
__device__ __forceinline__ double block_sum(double v, double* sh) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < F64_NW; ++w) t += sh[w];
    return t;
}
__device__ __forceinline__ double block_max(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = sh[0];
    for (int w = 1; w < F64_NW; ++w) t = fmax(t, sh[w]);
    return t;
}

// Sum over the grid's CTAs of word k of their partials: warp 0 reads them, every thread gets the
// total (FP64 adds by all warps would take longer than the reads).
__device__ __forceinline__ double grid_total(const double* part, int nb, int k, double* s_tot) {
    if (threadIdx.x < 32) {
        double t = 0.0;
        for (int bb = threadIdx.x; bb < nb; bb += 32) t += __ldcg(part + 4 * bb + k);
        t = warp_sum(t);
        if (threadIdx.x == 0) *s_tot = t;
    }
    __syncthreads();
    const double t = *s_tot;
    __syncthreads();
    return t;
}

__device__ __forceinline__ double warp_maxd(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__global__ void __launch_bounds__(F64_NT) sk_solve64(F64Params P) {
    extern __shared__ double tile[];  // [rows][J] plan entries, then [2][J] column sums
    __shared__ double sh[F64_NW], s_row[F64_NW], s_w[F64_NW], s_tot;
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nb = gridDim.x, b = blockIdx.x;
    const int64_t I = P.I;
    const int J = P.J;
    const int R = P.rows, WR = F64_NW / R;        // warps of a row's team
    const int r = warp / WR, tl = (warp % WR) * 32 + lane, NTR = 32 * WR;
    const int64_t ntile = (I + R - 1) / R;
    const int nt = (int)min((int64_t)nb, ntile);  // CTAs with tiles; the others help with the columns
    double* T = tile;
    double* acc = tile + (size_t)R * J;
    double* acc2 = acc + J;
    const double eps = P.eps, inv_eps = 1.0 / P.eps;
    int* status = &P.st->status;
    unsigned gen = 0;
#define F64_BARRIER()                                                                                       \
    do {                                                                                                    \
        if (!grid_barrier_named(&P.st->bar, (unsigned)nb * ++gen, status, P.spin, 1, F64_NT, &s_ok)) return; \
    } while (0)

    // ---- setup: sums of p and q (fixed order), checks, starting g -------------------------
    {
        double sp = 0.0, sq = 0.0;
        int bad = 0;
        for (int64_t i = b * (int64_t)F64_NT + tid; i < I; i += (int64_t)nb * F64_NT) {
            const double v = P.p[i];
            bad |= !(v > 0.0) || !isfinite(v);
            sp += v;
        }
        for (int j = b * F64_NT + tid; j < J; j += nb * F64_NT) {
            const double v = P.q[j];
            bad |= !(v > 0.0) || !isfinite(v);
            sq += v;
            const double g0 = P.g_warm ? P.g_warm[j] : 0.0;
            bad |= !isfinite(g0);
            P.gb[j] = g0;  // g^0 in buffer 0
        }
        sp = block_sum(sp, sh);
        sq = block_sum(sq, sh);
        if (__syncthreads_or(bad) && tid == 0) atomicCAS(status, DEV_OK, DEV_EINVAL);
        if (tid == 0) {
            P.part[4 * b + 0] = sp;
            P.part[4 * b + 1] = sq;
        }
    }
    F64_BARRIER();
    // Written by then, if at all: from here on numerical failures are collected in `bad` and
    // published with the residuals, so that every CTA takes the same decision on them.
    if (__syncthreads_or(ld_volatile_i32(status) != DEV_OK)) return;
    const double sp = grid_total(P.part, nb, 0, &s_tot), sq = grid_total(P.part, nb, 1, &s_tot);
    if (!(fabs(sp - sq) <= 1e-5 * sp)) {
        if (b == 0 && tid == 0) atomicCAS(status, DEV_OK, DEV_EINVAL);
        return;  // the same decision in every CTA
    }
    const double inv_sp = 1.0 / sp, inv_sq = 1.0 / sq, lsp = log(sp);
    int bad = 0;  // a potential that this thread formed is not finite

    // One row's sum over its team from the lanes' values (the whole block calls).
    auto row_sums = [&](double v) {
        v = warp_sum(v);
        if (lane == 0) sh[warp] = v;
        __syncthreads();
        if (tid < R) {
            double t = 0.0;
            for (int w = 0; w < WR; ++w) t += sh[tid * WR + w];
            s_row[tid] = t;
        }
    };

    // log sum_i exp((f_i - C_ij) / eps) of column j, by one warp, in every lane
    auto col_lse = [&](const double* f, int j) {
        double m = -INFINITY, s = 0.0;
        for (int64_t i = lane; i < I; i += 32) m = fmax(m, (__ldcg(f + i) - P.C[i * P.ld + j]) * inv_eps);
        m = warp_maxd(m);
        if (m > -INFINITY)
            for (int64_t i = lane; i < I; i += 32) s += exp((__ldcg(f + i) - P.C[i * P.ld + j]) * inv_eps - m);
        return m + log(warp_sum(s));
    };

    // ---- iteration 1: log-sum-exp by rows, then by columns ----------------------------------
    for (int64_t k = b; k < ntile; k += nb) {
        const int64_t i = k * R + r;
        const double* row = P.C + (i < I ? i : 0) * P.ld;
        double m = -INFINITY;
        if (i < I)
            for (int j = tl; j < J; j += NTR) m = fmax(m, (P.gb[j] - row[j]) * inv_eps);
        m = warp_maxd(m);
        if (lane == 0) sh[warp] = m;
        __syncthreads();
        m = sh[r * WR];
        for (int w = 1; w < WR; ++w) m = fmax(m, sh[r * WR + w]);
        __syncthreads();
        double s = 0.0;
        if (i < I && m > -INFINITY)
            for (int j = tl; j < J; j += NTR) s += exp((P.gb[j] - row[j]) * inv_eps - m);
        row_sums(s);
        if (tl == 0) s_w[r] = m;
        __syncthreads();
        if (tid < R && k * R + tid < I) {
            const int64_t ii = k * R + tid;
            const double fi = eps * (log(P.p[ii] * inv_sp) - (s_w[tid] + log(s_row[tid])));
            bad |= !isfinite(fi);
            P.fb[I + ii] = fi;
        }
        __syncthreads();
    }
    F64_BARRIER();
    {
        const double* f1 = P.fb + I;
        // a CTA a column, or a warp where every warp of the grid has one
        const bool by_warp = J >= nb * F64_NW;
        for (int j = b + nb * warp; by_warp && j < J; j += nb * F64_NW) {
            const double v = log(P.q[j] * inv_sq) - col_lse(f1, j);
            bad |= !isfinite(v);
            if (lane == 0) P.gb[J + j] = eps * v;
        }
        for (int j = b; !by_warp && j < J; j += nb) {
            double m = -INFINITY;
            for (int64_t i = tid; i < I; i += F64_NT) m = fmax(m, (__ldcg(f1 + i) - P.C[i * P.ld + j]) * inv_eps);
            m = block_max(m, sh);
            double s = 0.0;
            if (m > -INFINITY)
                for (int64_t i = tid; i < I; i += F64_NT) s += exp((__ldcg(f1 + i) - P.C[i * P.ld + j]) * inv_eps - m);
            s = block_sum(s, sh);
            if (tid == 0) {
                const double v = log(P.q[j] * inv_sq) - (m + log(s));
                bad |= !isfinite(v);
                P.gb[J + j] = eps * v;
            }
        }
    }
    F64_BARRIER();

    // ---- iterations 2, 3, ...: each plan entry once ------------------------------------------
    int ret = 0;  // buffer holding the returned potentials
    for (int s = 2;; ++s) {
        const double* gprev = P.gb + ((s - 1) & 1) * J;
        const double* fprev = P.fb + ((s - 1) & 1) * I;
        double* fcur = P.fb + (s & 1) * I;
        double res = 0.0;
        for (int j = tid; j < J; j += F64_NT) acc[j] = 0.0;
        for (int64_t k = b; k < ntile; k += nb) {
            const int nr = (int)min((int64_t)R, I - k * R);
            const int64_t i = k * R + r;
            double rs = 0.0;
            if (r < nr) {
                const double* row = P.C + i * P.ld;
                const double fi = fprev[i];  // written by this CTA
                for (int j = tl; j < J; j += NTR) {
                    const double t = exp((fi + __ldcg(gprev + j) - row[j]) * inv_eps);
                    T[(size_t)r * J + j] = t;
                    rs += t;
                }
            }
            row_sums(rs);
            // row k R + tid, whose entries in T sum to s_row[tid] and stand for T e^m
            auto update = [&](double m) {
                const int64_t ii = k * R + tid;
                const double ph = P.p[ii] * inv_sp, w = ph / s_row[tid], fi = fprev[ii];
                const double fn = fi + eps * (log(w) - m);
                bad |= !isfinite(fn);
                fcur[ii] = fn;
                res += ph * fabs(expm1((fi - fn) * inv_eps));
                s_w[tid] = w;
            };
            const bool low = tid < nr && !(s_row[tid] >= F64_LOW);
            if (tid < nr && !low) update(0.0);
            if (__syncthreads_or(low)) {
                const bool mine = r < nr && !(s_row[r] >= F64_LOW);  // this team's row
                const double* row = P.C + (r < nr ? i : 0) * P.ld;
                const double fi = r < nr ? fprev[i] : 0.0;
                double m = -INFINITY;
                if (mine)
                    for (int j = tl; j < J; j += NTR) m = fmax(m, (fi + __ldcg(gprev + j) - row[j]) * inv_eps);
                m = warp_maxd(m);
                if (lane == 0) sh[warp] = m;
                __syncthreads();
                m = sh[r * WR];
                for (int w = 1; w < WR; ++w) m = fmax(m, sh[r * WR + w]);
                __syncthreads();
                rs = 0.0;
                if (mine)
                    for (int j = tl; j < J; j += NTR) {
                        const double t = exp((fi + __ldcg(gprev + j) - row[j]) * inv_eps - m);
                        T[(size_t)r * J + j] = t;
                        rs += t;
                    }
                row_sums(rs);
                if (mine && tl == 0) s_w[r] = m;
                __syncthreads();
                if (low) update(s_w[tid]);
                __syncthreads();
            }
            for (int j = tid; j < J; j += F64_NT) {
                double a = acc[j];
                for (int q = 0; q < nr; ++q) a = fma(T[(size_t)q * J + j], s_w[q], a);
                acc[j] = a;
            }
            __syncthreads();
        }
        const int failed = __syncthreads_or(bad);  // the row updates', and the last column updates'
        if (warp == 0) {  // a tile's rows are updated by threads of warp 0
            res = warp_sum(res);
            if (lane == 0) P.part[4 * b + 2] = failed ? NAN : res;
        }
        if (P.colp && b < nt)
            for (int j = tid; j < J; j += F64_NT) P.colp[(int64_t)b * J + j].x = acc[j];
        F64_BARRIER();
        const double e = grid_total(P.part, nb, 2, &s_tot);
        if (isnan(e)) {  // some CTA has failed: every one leaves, and the caller's outputs stay as they are
            if (b == 0 && tid == 0) {
                P.st->iters = s - 1;
                atomicCAS(status, DEV_OK, F64_ENUMERIC);
            }
            return;
        }
        if (e <= P.tol || s - 1 >= P.max_iter) {  // the same sum in every CTA
            if (b == 0 && tid == 0) {
                P.st->iters = s - 1;
                P.st->err = e;
                P.st->converged = (e <= P.tol);
            }
            ret = (s - 1) & 1;
            break;
        }
        // g_j += eps log(q^_j / s_j): columns dealt over the CTAs' warps, one warp a column
        double* gcur = P.gb + (s & 1) * J;
        for (int j = b + nb * warp; j < J; j += nb * F64_NW) {
            double c = 0.0;
            if (P.colp) {
                for (int bb = lane; bb < nt; bb += 32) c += __ldcg(&P.colp[(int64_t)bb * J + j].x);
                c = warp_sum(c);
            } else {
                c = acc[j];
            }
            const bool low = !(c >= F64_LOW);  // the same in the whole warp: as in iteration 1
            const double lse = low ? col_lse(fcur, j) : 0.0;
            if (lane == 0) {
                const double gn = low ? eps * (log(P.q[j] * inv_sq) - lse)
                                      : __ldcg(gprev + j) + eps * log(P.q[j] * inv_sq / c);
                bad |= !isfinite(gn);
                gcur[j] = gn;
            }
        }
        F64_BARRIER();
    }

    // ---- finalize: plan of (f^ret, g^ret), FP64 marginals, loads, cost ------------------------
    const double* fr = P.fb + ret * I;
    const double* gr = P.gb + ret * J;
    double er = 0.0;
    for (int j = tid; j < J; j += F64_NT) acc[j] = acc2[j] = 0.0;
    for (int64_t k = b; k < ntile; k += nb) {
        const int nr = (int)min((int64_t)R, I - k * R);
        const int64_t i = k * R + r;
        double rs = 0.0;
        if (r < nr) {
            const double* row = P.C + i * P.ld;
            const double fi = fr[i];
            for (int j = tl; j < J; j += NTR) {
                const double t = exp((fi + __ldcg(gr + j) - row[j]) * inv_eps);
                T[(size_t)r * J + j] = t;
                rs += t;
                if (P.pi) P.pi[i * P.pi_ld + j] = (float)(t * sp);
            }
        }
        row_sums(rs);
        if (tid < nr) {
            const int64_t ii = k * R + tid;
            er += fabs(s_row[tid] - P.p[ii] / sp);
            P.f_out[ii] = fr[ii] + eps * lsp;
        }
        __syncthreads();
        for (int j = tid; j < J; j += F64_NT) {
            double a = acc[j], h = acc2[j];
            for (int q = 0; q < nr; ++q) {
                const double t = T[(size_t)q * J + j];
                a += t;
                if (t > 0.0) h = fma(P.C[(k * R + q) * P.ld + j], t, h);
            }
            acc[j] = a;
            acc2[j] = h;
        }
        __syncthreads();
    }
    if (warp == 0) {
        er = warp_sum(er);
        if (lane == 0) P.part[4 * b + 0] = er;
    }
    if (P.colp && b < nt)
        for (int j = tid; j < J; j += F64_NT) P.colp[(int64_t)b * J + j] = make_double2(acc[j], acc2[j]);
    F64_BARRIER();
    {
        double ec = 0.0, cost = 0.0;
        for (int j = b + nb * warp; j < J; j += nb * F64_NW) {
            double c = 0.0, h = 0.0;
            if (P.colp) {
                for (int bb = lane; bb < nt; bb += 32) {
                    const double2 v = __ldcg(&P.colp[(int64_t)bb * J + j]);
                    c += v.x;
                    h += v.y;
                }
                c = warp_sum(c);
                h = warp_sum(h);
            } else {
                c = acc[j];
                h = acc2[j];
            }
            if (lane == 0) {
                ec += fabs(c - P.q[j] / sq);
                cost += h;
                if (P.rrh_load) P.rrh_load[j] = h * sp;
                P.g_out[j] = __ldcg(gr + j);
            }
        }
        ec = block_sum(ec, sh);
        cost = block_sum(cost, sh);
        if (tid == 0) {
            P.part[4 * b + 1] = ec;
            P.part[4 * b + 3] = cost;
        }
    }
    F64_BARRIER();
    if (b == 0) {
        const double e = grid_total(P.part, nb, 0, &s_tot), ec = grid_total(P.part, nb, 1, &s_tot);
        const double co = grid_total(P.part, nb, 3, &s_tot);
        if (tid == 0) {
            P.summ->err_row = e;
            P.summ->err_col = ec;
            P.summ->cost = co * sp;
            P.summ->err_loop = P.st->err;
            P.summ->iters = P.st->iters;
            P.summ->converged = P.st->converged;
            P.summ->status = P.st->status;
            P.summ->absorptions = 0;
        }
    }
#undef F64_BARRIER
}

__global__ void sk_summary64(const F64State* st, SolveSummary* summ) {
    // status of a launch that stopped early (invalid input or a wait that gave up)
    if (threadIdx.x == 0 && st->status != DEV_OK) {
        summ->status = st->status;
        summ->iters = st->iters;
        summ->converged = 0;
    }
}

ot_status launch_solve_f64(ot_assoc_ctx* ctx, const SolveArgs64& a, SolveSummary* sum_host) {
    ot_status st = OT_OK;
    const int64_t I = a.I;
    const int J = a.J;
    // rows of a tile: as many as fit with the two rows of column sums (8 up to 2,896 columns), and
    // fewer where that gives more SMs a tile and leaves a lane two columns of its row or more
    int rows = F64_NW;
    const size_t budget = 232448 - 2048;  // 227 KB per block minus static shared memory
    auto tiles = [&](int r) { return (I + r - 1) / r; };
    while (rows > 1 && (sizeof(double) * (size_t)(rows + 2) * J > budget ||
                        (tiles(rows / 2) <= ctx->num_sms && J >= 2 * 32 * (2 * F64_NW / rows))))
        rows /= 2;
    const size_t smem = sizeof(double) * (size_t)(rows + 2) * J;
    if (allow_max_dynamic_smem((const void*)sk_solve64, smem) != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, OT_ECUDA, "FP64 solver: %zu bytes of shared memory refused", smem);
    }
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sk_solve64, F64_NT, smem) != cudaSuccess || occ < 1) {
        cudaGetLastError();
        return set_error(ctx, OT_ECUDA, "FP64 solver cannot be resident");
    }
    // a CTA a tile, and enough for a warp a column: 20 iterations on 1 x 8,192 take 0.32 ms; with the
    // tiles' CTAs alone they took 42 (one CTA, its warps walking 1,024 columns each), and 6 with a
    // warp a row and a warp a column.  64 x 512: 0.39, 1.73 and 1.20 ms.
    int grid = (int)std::min<int64_t>(std::max<int64_t>(tiles(rows), (J + F64_NW - 1) / F64_NW), ctx->num_sms);
    double* fb = (double*)scratch(ctx, SLOT_F, sizeof(double) * 2 * (size_t)I, &st);
    if (st) return st;
    double* gb = (double*)scratch(ctx, SLOT_G, sizeof(double) * 2 * (size_t)round_up(J, 4), &st);
    if (st) return st;
    double* part = (double*)scratch(ctx, SLOT_ERRPART, sizeof(double) * 4 * (size_t)grid, &st);
    if (st) return st;
    char* state = (char*)scratch(ctx, SLOT_STATE, 4096, &st);
    if (st) return st;
    F64State* fst = (F64State*)state;
    SolveSummary* summ = (SolveSummary*)(state + 512);
    // column sums of the CTAs; where a scratch budget leaves no room for them, fewer CTAs (one
    // alone keeps its sums in shared memory)
    double2* colp = nullptr;
    while (grid > 1) {
        colp = (double2*)scratch(ctx, SLOT_COLPART, sizeof(double2) * (size_t)std::min<int64_t>(grid, tiles(rows)) * J, &st);
        if (!st) break;
        if (st != OT_ENOMEM) return st;
        st = OT_OK;
        grid /= 2;
    }
    if (grid == 1) colp = nullptr;
    SolveSummary* hsum = (SolveSummary*)host_staging(ctx, sizeof(SolveSummary), &st);
    if (st) return st;
    cudaStream_t s = a.stream;
    cudaError_t e = cudaMemsetAsync(state, 0, 1024, s);
    if (e != cudaSuccess) return cuda_error(ctx, e, "memset");
    F64Params P;
    P.C = a.C;
    P.ld = a.ld;
    P.I = I;
    P.J = J;
    P.p = a.p;
    P.q = a.q;
    P.g_warm = a.warm_start ? a.out->g : nullptr;
    P.eps = a.eps;
    P.tol = a.tol;
    P.max_iter = a.max_iter;
    P.fb = fb;
    P.gb = gb;
    P.part = part;
    P.colp = colp;
    P.rows = rows;
    P.st = fst;
    P.f_out = a.out->f;
    P.g_out = a.out->g;
    P.rrh_load = a.out->rrh_load;
    P.pi = a.out->pi;
    P.pi_ld = a.out->pi_ld > 0 ? a.out->pi_ld : J;
    P.summ = summ;
    P.spin = ctx->spin_limit;
    void* args[] = {&P};
    e = cudaLaunchCooperativeKernel((const void*)sk_solve64, dim3(grid), dim3(F64_NT), args, smem, s);
    if (e != cudaSuccess) return cuda_error(ctx, e, "FP64 solve launch");
    sk_summary64<<<1, 32, 0, s>>>(fst, summ);
    ctx->launches += 2;
    e = cudaMemcpyAsync(hsum, summ, sizeof(SolveSummary), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_error(ctx, e, "FP64 solve");
    *sum_host = *hsum;
    if (sum_host->status == F64_ENUMERIC) sum_host->status = OT_ENUMERIC_INTERNAL;
    return OT_OK;
}

}  // namespace ota
