// Exact median of FP32 values.
// eps = eps_rel * median(C) is how the benchmark configurations fix the regularization
// strength of Eq. (5); the median of an even count is the mean of the two middle values.
//
// Method, in one cooperative launch:
//   1. (from 2^20 entries on) every CTA takes the same 8192 entries, one at a hashed place of
//      each 1/8192 of the data, and selects, exactly, the sample ranks s/2 -+ 4.5 sd
//      (sd = sqrt(s)/2, the rank spread of a sample median): a bracket [lo, hi];
//   2. one pass over all n entries counts those below lo and compacts those in [lo, hi]
//      into a candidate buffer (about 5% of n);
//   3. if both middle ranks fall inside the bracket and the candidates fit, select them
//      among the candidates; otherwise select over all n entries.
// Selection is a radix select (11 bits per pass) on order-preserving keys that tracks both
// middle ranks at once; among the candidates it starts below the leading bits that lo and
// hi share.  Every CTA picks the digits itself from the grid's histogram, so a pass takes one
// grid barrier.  The result is exact either way and does not depend on the order in which
// candidates were compacted.
//
// What bounds it: the one pass over the data (160 MB on 50,000 x 800, 24 us of HBM), and below
// about a million entries the trips between passes.  As eleven launches (four for the sample,
// four for the candidates, at 7 to 10 us each) the median took 150 us of the 330 us that rates,
// cost and median of 50,000 x 800 take, and half of the 100 us of a 1000 x 50 cell.
// Now one launch of 70 us there (18 us on 1000 x 50).
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "ot_common.cuh"
#include "ot_internal.h"

namespace ota {

static constexpr int RS_NT = 512;                // threads of a CTA (one CTA an SM)
static constexpr int RS_BITS = 11;
static constexpr int RS_BINS = 1 << RS_BITS;
static constexpr int RS_PASSES = (32 + RS_BITS - 1) / RS_BITS;
static constexpr int RS_PER = 16;                // sample entries a thread
static constexpr int64_t SAMPLE = RS_NT * RS_PER;

// Order-preserving map float bits -> unsigned key (negative values reversed).
__device__ __forceinline__ uint32_t fkey(float f) {
    const uint32_t u = __float_as_uint(f);
    return u ^ ((uint32_t)((int)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

struct SelectState {            // zeroed before the launch
    unsigned bar;
    int status;
    unsigned long long n_cand;  // entries found in [lo, hi]
    unsigned long long c_lo;    // entries found below lo
    unsigned long long hist[RS_PASSES][2][RS_BINS];  // a lone CTA keeps its counts to itself and has none of these
};
static constexpr size_t RS_LONE = offsetof(SelectState, hist);

// The data a pass reads: a strided row-major view (rows x cols, leading dimension ld).
// flat: the view is one contiguous run of rows * cols entries.
struct SelSrc {
    const float* x;
    int64_t rows, cols, ld;
    int vec;   // 16-byte aligned rows (or run): float4 loads
    int flat;
};

// Number of 4-entry chunks of the view.
__host__ __device__ __forceinline__ int64_t n_chunks(const SelSrc& src) {
    return src.flat ? (src.rows * src.cols + 3) / 4 : src.rows * ((src.cols + 3) / 4);
}

// Up to four consecutive entries of the view: chunk t of n chunks.
__device__ __forceinline__ void load_chunk(const SelSrc& src, int64_t t, int64_t n, float v[4], bool ok[4]) {
    v[0] = v[1] = v[2] = v[3] = 0.f;
    ok[0] = ok[1] = ok[2] = ok[3] = false;
    if (t >= n) return;
    const float* p;
    int64_t left;  // entries of this row (or run) from p on
    if (src.flat) {
        p = src.x + 4 * t;
        left = src.rows * src.cols - 4 * t;
    } else {
        const int64_t cch = (src.cols + 3) / 4;
        const int64_t r = t / cch;
        const int64_t c = (t - r * cch) * 4;
        p = src.x + r * src.ld + c;
        left = src.cols - c;
    }
    if (src.vec && left >= 4) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
        ok[0] = ok[1] = ok[2] = ok[3] = true;
    } else {
        for (int e = 0; e < 4; ++e)
            if (e < left) { v[e] = __ldg(p + e); ok[e] = true; }
    }
}

struct SelShared {
    unsigned h[2][RS_BINS];
    unsigned long long warp_sum[2][RS_NT / 32];
    int digit[2], ok;
    long long rank[2];
    unsigned long long below[RS_NT / 32];
};

// Digits of two targets in their histograms of RS_BINS counts, count(0, bin) and, where the two
// differ (NH = 2), count(1, bin), in one block scan: the digit d of target t with excl(d) <=
// rank[t] < excl(d) + count(d), and rank[t] - excl(d).  The whole block calls.
template <int NH, typename Count>
__device__ __forceinline__ void block_pick(Count count, long long (&rank)[2], uint32_t (&digit)[2], SelShared* sh) {
    constexpr int PER = RS_BINS / RS_NT, NW = RS_NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    unsigned long long c[NH][PER], sum[NH], incl[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        sum[h] = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            c[h][k] = count(h, tid * PER + k);
            sum[h] += c[h][k];
        }
        incl[h] = sum[h];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl[h], o);
            if (lane >= o) incl[h] += y;
        }
    }
    __syncthreads();  // the shared words may still be read from the last pick
#pragma unroll
    for (int h = 0; h < NH; ++h)
        if (lane == 31) sh->warp_sum[h][w] = incl[h];
    if (tid < 2) {
        sh->digit[tid] = RS_BINS - 1;  // kept only for an out-of-range rank, which cannot occur
        sh->rank[tid] = rank[tid];
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        unsigned long long before = lane < w && lane < NW ? sh->warp_sum[h][lane] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
        long long excl = (long long)(before + incl[h] - sum[h]);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
#pragma unroll
            for (int t = NH == 1 ? 0 : h; t < (NH == 1 ? 2 : h + 1); ++t)
                if (c[h][k] && rank[t] >= excl && rank[t] < excl + (long long)c[h][k]) {
                    sh->digit[t] = tid * PER + k;
                    sh->rank[t] = rank[t] - excl;
                }
            excl += (long long)c[h][k];
        }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        digit[t] = (uint32_t)sh->digit[t];
        rank[t] = sh->rank[t];
    }
}

// The two targets of a radix select, the same in every thread.
struct Targets {
    long long rank[2];
    uint32_t prefix[2];
    int done;  // leading key bits fixed
    __device__ __forceinline__ int width() const { return min(RS_BITS, 32 - done); }
    __device__ __forceinline__ bool same() const { return prefix[0] == prefix[1]; }
    // count key k into the histograms of its prefix (one histogram while the prefixes agree)
    __device__ __forceinline__ void count(SelShared* sh, float f) const {
        const uint32_t k = fkey(f);
        const uint32_t hi = done ? (k >> (32 - done)) : 0u;
        const uint32_t d = (k >> (32 - done - width())) & ((1u << width()) - 1u);
        if (hi == prefix[0]) atomicAdd(&sh->h[0][d], 1u);
        else if (hi == prefix[1]) atomicAdd(&sh->h[1][d], 1u);
    }
    template <typename Count>
    __device__ __forceinline__ void pick(Count c, SelShared* sh) {
        const int w = width();
        uint32_t d[2];
        if (same()) block_pick<1>(c, rank, d, sh);
        else block_pick<2>(c, rank, d, sh);
        prefix[0] = (prefix[0] << w) | d[0];
        prefix[1] = (prefix[1] << w) | d[1];
        done += w;
    }
};

__device__ __forceinline__ void clear_hist(SelShared* sh, int nh) {
    __syncthreads();
    for (int t = threadIdx.x; t < nh * RS_BINS; t += RS_NT) (&sh->h[0][0])[t] = 0u;
    __syncthreads();
}

static constexpr int RS_UNROLL = 8;
static constexpr int RS_GROUP = 32 * RS_UNROLL * 4;  // entries a warp tests per iteration
static constexpr int RS_STAGE = RS_GROUP + 256;      // entries a warp stages before it writes them out
static constexpr size_t RS_SMEM = sizeof(SelShared) + sizeof(float) * (RS_NT / 32) * RS_STAGE;

// out[0] = median, out[1] = 0; out[1] stays 1 when a wait gave up.
__global__ void __launch_bounds__(RS_NT, 1) rs_select(SelSrc src, int64_t n, long long k1, long long k2, int bracket,
                                                      long long s1, long long s2, SelectState* st, float* cand,
                                                      unsigned long long cap, long long spin, double* out) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    SelShared* sh = reinterpret_cast<SelShared*>(rs_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned nb = gridDim.x;
    unsigned gen = 0;
    if (blockIdx.x == 0 && tid == 0) out[1] = 1.0;
// leaves the kernel when the wait gave up
#define RS_BARRIER()                                                                                       \
    do {                                                                                                   \
        if (!grid_barrier_named(&st->bar, nb * ++gen, &st->status, spin, 1, RS_NT, &sh->ok)) return;      \
    } while (0)
    Targets T;
    T.rank[0] = k1;
    T.rank[1] = k2;
    T.prefix[0] = T.prefix[1] = 0u;
    T.done = 0;
    bool use_cand = false;
    const int64_t nch = n_chunks(src);
    if (bracket) {
        // ---- bracket from a sample, by every CTA alike -------------------------------------
        Targets B;
        B.rank[0] = s1;
        B.rank[1] = s2;
        B.prefix[0] = B.prefix[1] = 0u;
        B.done = 0;
        float v[RS_PER];
        const uint64_t step = (uint64_t)n / SAMPLE;
#pragma unroll
        for (int e = 0; e < RS_PER; ++e) {
            const uint32_t k = tid + RS_NT * e;
            // the place inside the k-th part: hashed, so that it does not follow the rows
            const uint64_t t = step * k + (((uint64_t)(k * 2654435761u) * step) >> 32);
            if (src.flat) {
                v[e] = __ldg(src.x + t);
            } else {
                const uint64_t r = t / (uint64_t)src.cols;
                v[e] = __ldg(src.x + r * src.ld + (t - r * src.cols));
            }
        }
        for (int pass = 0; pass < RS_PASSES; ++pass) {
            clear_hist(sh, B.same() ? 1 : 2);
#pragma unroll
            for (int e = 0; e < RS_PER; ++e) B.count(sh, v[e]);
            __syncthreads();
            B.pick([&](int t, int b) { return (unsigned long long)sh->h[t][b]; }, sh);
        }
        const uint32_t kl = B.prefix[0], kh = B.prefix[1];
        // ---- count those below, compact those inside ------------------------------------------
        // Each warp loads RS_UNROLL chunk groups before testing them, stages its candidates in
        // shared memory and reserves room in the buffer once per 256 or more of them.
        float* wb = reinterpret_cast<float*>(rs_smem + sizeof(SelShared)) + warp * RS_STAGE;
        unsigned fill = 0;  // warp-uniform
        unsigned long long below = 0;
        auto flush = [&]() {
            __syncwarp();
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(&st->n_cand, (unsigned long long)fill);
            base = __shfl_sync(0xffffffffu, base, 0);
            for (unsigned i = lane; i < fill; i += 32)
                if (base + i < cap) cand[base + i] = wb[i];
            __syncwarp();
            fill = 0;
        };
        const int64_t gwarp = (int64_t)blockIdx.x * (RS_NT / 32) + warp, nwarps = (int64_t)nb * (RS_NT / 32);
        // whole warps walk the chunk space together (the compaction uses warp ballots)
        int64_t t0 = gwarp * 32 * RS_UNROLL;
        if (src.flat && src.vec) {
            // One aligned run: whole groups without a check per entry.  A lane notes which of its
            // 32 entries are inside, the warp's lanes find their places by one scan, and only the
            // noted entries (one or two a lane) are touched again.
            const int64_t whole = n / RS_GROUP * (RS_GROUP / 4);  // chunks in whole groups
            const float4* p4 = reinterpret_cast<const float4*>(src.x) + lane;
            const uint32_t span = kh - kl;
            const int64_t stride = nwarps * 32 * RS_UNROLL;
            float4 nx[RS_UNROLL];  // the next group, on the way while this one is tested
#pragma unroll
            for (int u = 0; u < RS_UNROLL; ++u)
                nx[u] = t0 < whole ? __ldg(p4 + t0 + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
            for (; t0 < whole; t0 += stride) {
                float x[4 * RS_UNROLL];
#pragma unroll
                for (int u = 0; u < RS_UNROLL; ++u) {
                    x[4 * u] = nx[u].x;
                    x[4 * u + 1] = nx[u].y;
                    x[4 * u + 2] = nx[u].z;
                    x[4 * u + 3] = nx[u].w;
                }
                if (t0 + stride < whole)
#pragma unroll
                    for (int u = 0; u < RS_UNROLL; ++u) nx[u] = __ldg(p4 + t0 + stride + 32 * u);
                unsigned lt = 0, in = 0;
#pragma unroll
                for (int e = 0; e < 4 * RS_UNROLL; ++e) {
                    const uint32_t d = fkey(x[e]) - kl;  // below lo wraps around, and past span
                    if (d <= span) in |= 1u << e;
                    if (fkey(x[e]) < kl) ++lt;
                }
                below += lt;
                unsigned at = __popc(in);
                unsigned incl = at;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
                at = fill + incl - at;
#pragma unroll
                for (int e = 0; e < 4 * RS_UNROLL; ++e)
                    if (in >> e & 1u) wb[at++] = x[e];
                fill += total;
                if (fill > RS_STAGE - RS_GROUP) flush();  // keep room for one more iteration
            }
            // what is left, less than one group, falls to the warp whose turn it is
        }
        for (; t0 < nch; t0 += nwarps * 32 * RS_UNROLL) {
            float x[RS_UNROLL][4];
            bool ok[RS_UNROLL][4];
#pragma unroll
            for (int u = 0; u < RS_UNROLL; ++u) load_chunk(src, t0 + 32 * u + lane, nch, x[u], ok[u]);
            unsigned lt = 0;
#pragma unroll
            for (int u = 0; u < RS_UNROLL; ++u) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t k = fkey(x[u][e]);
                    lt += ok[u][e] && k < kl;
                    const bool in = ok[u][e] && k - kl <= kh - kl;
                    const unsigned m = __ballot_sync(0xffffffffu, in);
                    if (in) wb[fill + __popc(m & ((1u << lane) - 1u))] = x[u][e];
                    fill += __popc(m);
                }
            }
            below += lt;
            if (fill > RS_STAGE - RS_GROUP) flush();  // keep room for one more iteration
        }
        if (fill) flush();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
        if (lane == 0) sh->below[warp] = below;
        __syncthreads();
        if (tid == 0) {
            unsigned long long b = 0;
            for (int w = 0; w < RS_NT / 32; ++w) b += sh->below[w];
            atomicAdd(&st->c_lo, b);
        }
        RS_BARRIER();
        const long long c_lo = (long long)__ldcg(&st->c_lo), nc = (long long)__ldcg(&st->n_cand);
        const long long a = k1 - c_lo, b = k2 - c_lo;
        use_cand = nc <= (long long)cap && a >= 0 && a < nc && b >= 0 && b < nc;
        if (use_cand) {
            src = SelSrc{cand, 1, nc, nc, 1, 1};  // an aligned contiguous run
            T.rank[0] = a;
            T.rank[1] = b;
            T.done = __clz((int)(kl ^ kh));  // 32 when lo == hi
            T.prefix[0] = T.prefix[1] = T.done == 0 ? 0u : (T.done == 32 ? kl : (kl >> (32 - T.done)));
        }
    }
    // ---- radix select over the candidates, or over all entries ----------------------------------
    const int64_t m = n_chunks(src);
    for (int pass = 0; T.done < 32; ++pass) {
        const int nh = T.same() ? 1 : 2;  // histograms in use
        clear_hist(sh, nh);
        for (int64_t t = (int64_t)blockIdx.x * RS_NT + tid; t < m; t += (int64_t)nb * RS_NT) {
            float x[4];
            bool ok[4];
            if (use_cand) {  // written by other SMs in this launch: not through the read-only path
                const int64_t left = src.cols - 4 * t;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    ok[e] = e < left;
                    x[e] = ok[e] ? __ldcg(cand + 4 * t + e) : 0.f;
                }
            } else {
                load_chunk(src, t, m, x, ok);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (ok[e]) T.count(sh, x[e]);
        }
        __syncthreads();
        if (nb == 1) {
            T.pick([&](int t, int b) { return (unsigned long long)sh->h[t][b]; }, sh);
            continue;
        }
        for (int t = tid; t < nh * RS_BINS; t += RS_NT) {
            const unsigned c = (&sh->h[0][0])[t];
            if (c) atomicAdd(&st->hist[pass][0][0] + t, (unsigned long long)c);
        }
        RS_BARRIER();
        T.pick([&](int t, int b) { return __ldcg(&st->hist[pass][t][b]); }, sh);
    }
    if (blockIdx.x == 0 && tid == 0) {
        out[0] = 0.5 * ((double)fkey_inv(T.prefix[0]) + (double)fkey_inv(T.prefix[1]));
        out[1] = 0.0;
    }
#undef RS_BARRIER
}

ot_status launch_median(ot_assoc_ctx* ctx, const float* x, int64_t rows, int64_t cols, int64_t ld, double* out_dev,
                        cudaStream_t s) {
    ot_status st = OT_OK;
    const int64_t n = rows * cols;
    const long long k1 = (n - 1) / 2, k2 = n / 2;  // equal for odd n
    const int flat = (rows == 1 || ld == cols);
    const int vec = !((uintptr_t)x & 15u) && (flat || ld % 4 == 0);
    const SelSrc src{x, rows, cols, ld, vec, flat};
    const int64_t nch = n_chunks(src);
    const int bracket = n >= (1 << 20);  // below that, three passes over the data cost little
    // the bracket spans about 5% of the entries; more than n/16 means heavy ties
    const unsigned long long cap = bracket ? (unsigned long long)(n / 16) : 0ull;
    int grid = (int)std::max<int64_t>(1, std::min<int64_t>((nch + RS_NT - 1) / RS_NT, ctx->num_sms));
    const size_t off_cand = (size_t)round_up(sizeof(SelectState), 256);
    size_t state = grid > 1 ? sizeof(SelectState) : RS_LONE;
    char* ws = (char*)scratch(ctx, SLOT_SELECT, bracket ? off_cand + sizeof(float) * (size_t)cap : state, &st);
    if (st == OT_ENOMEM && !bracket && grid > 1) {
        // no room for the grid's histograms (98 KB) in the context's budget: one CTA, up to 2^20
        // entries, does without
        st = OT_OK;
        grid = 1;
        state = RS_LONE;
        ws = (char*)scratch(ctx, SLOT_SELECT, state, &st);
    }
    if (st) return st;
    SelectState* ss = (SelectState*)ws;
    float* cand = (float*)(ws + off_cand);
    const double sd = 0.5 * std::sqrt((double)SAMPLE);
    const long long s1 = (long long)(SAMPLE / 2 - 4.5 * sd), s2 = (long long)(SAMPLE / 2 + 4.5 * sd);
    if (allow_max_dynamic_smem((const void*)rs_select, RS_SMEM) != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, OT_ECUDA, "median kernel: %zu bytes of shared memory refused", RS_SMEM);
    }
    cudaError_t e = cudaMemsetAsync(ss, 0, state, s);
    if (e != cudaSuccess) return cuda_error(ctx, e, "median memset");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(RS_NT);
    cfg.dynamicSmemBytes = RS_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, rs_select, src, n, k1, k2, bracket, s1, s2, ss, cand, cap, ctx->spin_limit, out_dev);
    if (e != cudaSuccess) return cuda_error(ctx, e, "median launch");
    ctx->launches += 1;
    return OT_OK;
}

}  // namespace ota
