// Probabilistic state cache of the AceSpec edge step (Sec. III-C,
// Algorithm 1 TREE_DRAFT and the O(1) lookup of w = (pi, x_resampled)).
//
//   k_cache_build   per (sequence, depth) row of the draft distribution: the
//                   F_d largest q over ids != x~_d, in (q desc, id asc)
//                   order, with probability q / (1 - q(x~_d)).  The first
//                   loads are a sample of the row; a value a little below
//                   its F_d-th largest is found from them, and the rest of
//                   the one HBM pass only lists the values that reach it
//                   (hundreds).  When the list proves to hold the F_d
//                   largest it is ordered in shared memory; otherwise (the
//                   sample holds more of them than its share: about one row
//                   in 10^4 when ids come in no order; or one slice of a
//                   cluster does) the row is read again, digit by digit of
//                   the F_d-th largest value: twice as a rule, five times at
//                   most.  Small batches split a row over a cluster of CTAs
//                   whose candidates meet in the first one's shared memory.
//   k_cache_lookup  one thread per sequence scanning the F_pi branches.
#include <cooperative_groups.h>

#define ACES_FILE 3  // site numbers of the checked build
#include "qrow.cuh"

namespace aces {

constexpr int NTC = 256;   // threads per CTA
constexpr int CLD = 8;     // 16-byte loads in flight per thread
constexpr int CCAP = 4096; // candidates kept per row
constexpr int CCL = 8;     // CTAs of a row's cluster, at most
constexpr int RANK_MAX = 512;  // candidates ordered by direct ranking (more: bitonic sort)

#ifdef ACES_CHECKED
static __device__ unsigned int g_selects;  // rows that took cache_row_select
#endif

// the smallest order value of a positive q
constexpr unsigned long long LOWEST = 0x80000001ull << 32;

// The candidates of one row by radix selection, whatever its values (one CTA):
// a histogram of one digit a read, from the top, until the values down to the
// digit that holds the Fd-th largest fit in cand (after 11 of their 31 bits as
// a rule; of more than CCAP equal values the lowest ids, by blocks of 512),
// and a read that lists them.  Returns their number, at least Fd unless the
// row has fewer.  (64 x 8 rows of 152064 in the order of their ids' likelihood,
// F = 64, when the sample held
// the likely ids: eight maxima a read took 809 us a call, this 178.)
__device__ __noinline__ int cache_row_select(const float *qr, int V, int xd, int Fd, unsigned long long *cand) {
    constexpr int NB = 2048, PER = NB / NTC, U = 8;
    static_assert(NB * 4 <= CCAP * 8, "the histogram fits in the candidates' place");
    static_assert(ACES_MAX_V <= NB * 512 && ACES_MAX_BRANCH + 512 <= CCAP, "ids in 20 bits; the last digit's block fits");
    __shared__ unsigned long long red[NTC / 32];
    __shared__ uint32_t s_bin, s_above, s_in;
    __shared__ int s_at;
    uint32_t *hist = reinterpret_cast<uint32_t *>(cand);
    const QChunks qc(qr, V);
    const int tid = threadIdx.x;
    // f(bits, id) of every positive value but the draft token's
    auto visit = [&](auto f) {
        for (int c0 = tid; c0 < qc.nch; c0 += NTC * U) {
            uint4 w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = c0 + u * NTC < qc.nch ? qc.load(c0 + u * NTC) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t bits = e == 0 ? w[u].x : e == 1 ? w[u].y : e == 2 ? w[u].z : w[u].w;
                    const int x = (c0 + u * NTC) * 4 + e - qc.head;
                    if (__uint_as_float(bits) > 0.0f && x != xd) f(bits, x);  // (NaN: not > 0)
                }
        }
    };
    unsigned long long lowest = LOWEST;  // the candidates' smallest order value
    uint32_t pre = 0u, need = (uint32_t)Fd, above = 0u;
#pragma unroll 1
    for (int st = 0; st < 4; ++st) {
        const int hi = st == 0 ? 31 : st == 1 ? 20 : st == 2 ? 9 : 0, lo = st == 0 ? 20 : st == 1 ? 9 : 0;
        __syncthreads();
        for (int i = tid; i < NB; i += NTC) hist[i] = 0u;
        __syncthreads();
        visit([&](uint32_t bits, int x) {
            if (bits >> hi != pre) return;
            const uint32_t b = st < 3 ? (bits >> lo) & ((1u << (hi - lo)) - 1u) : (uint32_t)(ACES_MAX_V - 1 - x) >> 9;
            if (ACES_IN(b, NB)) atomicAdd(&hist[b], 1u);
        });
        __syncthreads();
        // the bin, from the top, that holds the need-th value
        uint32_t n = 0u;
#pragma unroll
        for (int i = 0; i < PER; ++i) n += hist[NB - 1 - (tid * PER + i)];
        unsigned long long tot;
        uint32_t at = (uint32_t)block_exscan_n<NTC>((unsigned long long)n, red, &tot);
        if (tot < need) break;  // (first digit only: fewer than Fd positive values, all of them are listed)
        for (int i = 0; i < PER; ++i) {
            const uint32_t b = NB - 1 - (tid * PER + i), c = hist[b];
            if (at < need && at + c >= need) {  // (one bin of one thread)
                s_bin = b;
                s_above = at;
                s_in = c;
            }
            at += c;
        }
        __syncthreads();
        above += s_above;
        need -= s_above;
        const uint32_t b = s_bin;
        if (st < 3) {
            pre = pre << (hi - lo) | b;
            lowest = (unsigned long long)(pre << lo | 0x80000000u) << 32;
        } else {
            lowest |= 0xFFFFFFFFu - (ACES_MAX_V - 1u - (b << 9));
        }
        if (above + s_in <= (uint32_t)CCAP) break;
    }
    __syncthreads();
    if (tid == 0) s_at = 0;
#ifdef ACES_CHECKED
    if (tid == 0) atomicAdd(&g_selects, 1u);
#endif
    __syncthreads();
    visit([&](uint32_t bits, int x) {
        const unsigned long long o = order_val(bits | 0x80000000u, (uint32_t)x);
        if (o < lowest) return;
        const int at = atomicAdd(&s_at, 1);
        if (at < CCAP && ACES_IN(at, CCAP)) cand[at] = o;
    });
    __syncthreads();
    return min(s_at, CCAP);
}

// One row of q by a cluster of 1 to CCL CTAs, each reading a slice.  Bound by
// HBM on large batches: 588 us for 256 x 16 rows of 256000 with a support cut
// and F = 4 (a sorted list of four per thread and no threshold: 583, and 700 on
// wider support, where its insertions diverge), 645 with F = 64 (1000 with lists
// of eight and a 2048-entry sort a row); 64 rows of full support with F = 64 52
// us on clusters of eight.  One sequence of 16 x 128256 takes 9 us on clusters of
// eight (22 with a CTA a row).  Short rows with wide fan-outs, whose slice is
// its own sample: 64 x 8 rows of 8000 with F = 256 24 us (102 with the lists).
__global__ void __launch_bounds__(NTC, 4) k_cache_build(CacheArgs a) {
    namespace cg = cooperative_groups;
    __shared__ unsigned long long cand[CCAP];  // candidates' order values (the first CTA's: the cluster's)
    __shared__ uint32_t smax[NTC];             // sample: per-thread maxima
    __shared__ unsigned long long red[NTC / 32];
    __shared__ uint32_t s_thr, s_low;          // this CTA's threshold: an order value's upper and lower half
    __shared__ unsigned long long s_tops[CCL]; // the cluster's thresholds (the first CTA's)
    __shared__ int s_n, s_tie;                 // candidates (may pass CCAP)
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int row = blockIdx.x / CL, tid = threadIdx.x, lane = tid & 31;
    const int b = row / a.K, d = row % a.K;
    const int Fd = a.F[d];
    if (Fd == 0) return;  // (the whole cluster)
    const float *qr = a.q + (size_t)row * a.V;
    int32_t *bt = a.bt + (size_t)b * a.total + a.off[d];
    float *bp = a.bp + (size_t)b * a.total + a.off[d];
    const int xd = a.xt[row];
    float den = 0.0f;
    if (xd >= 0 && xd < a.V) den = 1.0f - __ldg(qr + xd);
    if (!(den > 0.0f)) {  // (the whole cluster)
        if (rank == 0)
            for (int j = tid; j < Fd; j += NTC) {
                bt[j] = -1;
                bp[j] = 0.0f;
            }
        return;
    }
    if (tid == 0) s_n = 0;
    const QChunks qc(qr, a.V);
    // The slice must keep its `want` largest: all Fd with one CTA, else a share
    // with a margin (checked below against the other slices).
    const float Ff = (float)Fd, want = CL == 1 ? Ff : fminf(Ff, Ff / CL + 4.0f * sqrtf(Ff / CL) + 8.0f);
    // This CTA's chunks [c_lo, c_lo + cn), in blocks of NTC (32 a warp).
    // Iteration 0 is a sample: each warp's part of one block of each of CLD
    // segments of nit blocks.  The others take the remaining blocks in order,
    // which reads faster (a tile of each segment every time: 620 us against 587
    // on 256 x 16 rows of 256000; with bounds and edges tested per chunk 3%
    // slower).
    const int per = (qc.nch + CL - 1) / CL, c_lo = min(qc.nch, rank * per), cn = min(qc.nch, c_lo + per) - c_lo;
    const int nit = (cn + CLD * NTC - 1) / (CLD * NTC);
    // Few branches: a threshold that `want` + 1 of the sample reach cannot be too
    // high (sure; while it lists few values: 64 x 8 rows of 152064, F = 16, 58 us
    // by the sample's share, 81 so), and the sample is the first block of every
    // segment: it holds the first ids, the likely ones in many vocabularies.
    // Many: the threshold rests on the sample holding its share of the largest
    // values, and half the warps take a block from the middle of each segment,
    // which leaves out the slice's first ids.  (Those rows with the likely ids
    // first: F = 4 83 us without the first ids, 47 with them; F = 64 178 with
    // first blocks alone, which raised the threshold too far, 52 now.  Another
    // block for each warp: 84, and 606 us against 587 for the 256 x 16 rows.)
    const bool sure = want < NTC / 4 && (want + 1.0f) * CL * (float)cn <= 0.375f * RANK_MAX * (CLD * NTC);
    auto sample_block = [&](int wr) { return sure || wr >= NTC / 64 ? 0 : nit / 2; };  // of a warp, in each segment
    uint4 w[CLD];
    int cb[CLD];  // the iteration's chunks, less the thread's number
    const int off = sample_block(tid >> 5);
    int at_b = off == 0 ? NTC : 0, at_o = off == 0 ? 1 : nit - off;  // the next block; blocks since a sample's
#pragma unroll
    for (int u = 0; u < CLD; ++u) cb[u] = (u * nit + off) * NTC;
    const bool whole = qc.head == 0 && (a.V & 3) == 0;  // every chunk is whole
    const float *mine = qc.base + (size_t)(c_lo + tid) * 4;
    auto load = [&]() {
        if (whole && cb[CLD - 1] + NTC <= cn) {
#pragma unroll
            for (int u = 0; u < CLD; ++u) w[u] = ldg16(mine + cb[u] * 4);
        } else {
#pragma unroll
            for (int u = 0; u < CLD; ++u)
                w[u] = cb[u] + tid < cn ? qc.load(c_lo + cb[u] + tid) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    load();
    // ---- a threshold from the sample ----
    // Of the `want` largest the sample, a share f of the slice, holds want * f on
    // average; its rank-r value with r four deviations above that is below the
    // want-th largest but for about one row in 10^4 whose ids come in no order,
    // and about r / f values reach it.  Every thread's maximum stands for its 32
    // values: the rank among the NTC maxima is corrected for values that share a
    // thread (and r for how their number varies, which is all of r's variance
    // when the sample is the whole slice).
    int need = 0;      // (warp 0, while its loads are under way)
    float room = 0.0f;
    if (tid < 32) {
        int ns = 0;  // chunks of the sample, two of its tiles a lane
#pragma unroll
        for (int h = lane; h < CLD * NTC / 32; h += 32) {
            const int wr = h % (NTC / 32), u = h / (NTC / 32);
            ns += max(0, min(32, cn - (u * nit + sample_block(wr)) * NTC - wr * 32));
        }
        ns = __reduce_add_sync(0xffffffffu, ns);
        const float f = cn > 0 ? (float)ns / (float)cn : 1.0f;
        const float wf = want * f, x = wf / NTC;
        const float var = wf * (1.0f - f) + NTC * (exp2f(1.4427f * x) - 1.0f - x);
        const float r = wf + 4.0f * sqrtf(fmaxf(var, 0.0f)) + (f < 1.0f ? 4.0f : 1.0f);
        const auto maxima = [](float values) { return NTC * (1.0f - exp2f(-1.4427f * values / NTC)); };
        need = min((int)ceilf(maxima(r)), NTC);
        if (sure) need = (int)ceilf(want) + 1;
        // the most maxima that may reach the threshold: those of many more values
        // than asked for and than direct ranking takes, or than the list holds
        room = maxima(f * fminf(0.75f * CCAP / CL, fmaxf(0.75f * RANK_MAX / CL, 1.5f * r / f)));
    }
    // Positive floats order like their bits; negative q (and the padding) are
    // at most 0 as integers.
    int mx = 0;
#pragma unroll
    for (int u = 0; u < CLD; ++u) mx = max(mx, max(max((int)w[u].x, (int)w[u].y), max((int)w[u].z, (int)w[u].w)));
    smax[tid] = (uint32_t)mx;
    if (CL > 1) cl.sync();  // (the first CTA's counter is set before another adds to it)
    else __syncthreads();
    if (tid < 32) {
        uint32_t v[NTC / 32], thr = 0u;
        int cnt = NTC, bit = 30;
#pragma unroll
        for (int i = 0; i < NTC / 32; ++i) v[i] = smax[i * 32 + lane];
        auto try_bit = [&]() {
            const uint32_t t = thr | 1u << bit;
            uint32_t n = 0u;
#pragma unroll
            for (int i = 0; i < NTC / 32; ++i) n += v[i] >= t;
            n = __reduce_add_sync(0xffffffffu, n);
            if (n >= (uint32_t)need) {
                thr = t;
                cnt = (int)n;
            }
        };
        // the largest threshold (its exponent and four bits) that `need` maxima reach
        for (; bit >= 19; --bit) try_bit();
        // more bits while too many do (values alike: 64 x 8 uniform rows of 256000, F
        // = 8: 425 us without, 109)
        if (thr > 0u)
            for (; bit >= 0 && (float)cnt > room; --bit) try_bit();
        if (tid == 0) {
            s_thr = thr > 1u ? thr : 1u;  // (at least 1: q > 0)
            s_low = 0u;
            s_tie = thr > 0u && bit < 0 && (float)cnt > room;
        }
    }
    __syncthreads();
    const int tie = s_tie;
    // (the values equal to the threshold are listed by themselves then, below)
    const int thr = (int)s_thr + tie;
    if (tie) {
        // Too many values equal the threshold: of those only the first ids, up to
        // where, at their density in the sample, there are twice the number asked for.
        unsigned long long eq = 0ull;  // of this thread's sampled values; in the upper half, those looked at
#pragma unroll
        for (int u = 0; u < CLD; ++u) {
            eq += ((int)w[u].x == thr - 1) + ((int)w[u].y == thr - 1) + ((int)w[u].z == thr - 1) + ((int)w[u].w == thr - 1);
            eq += (unsigned long long)(cb[u] + tid < cn ? 4 : 0) << 32;
        }
        eq = block_reduce_n<NTC>(eq, red, SumU64());
        const float ids = 2.0f * (Ff + 16.0f) * (float)(eq >> 32) / (float)(uint32_t)eq;  // (eq: at least one)
        const float last = (float)(c_lo * 4) + ids;
        s_low = last < (float)a.V ? 0xFFFFFFFFu - (uint32_t)last : 0u;  // (the same from every thread)
        __syncthreads();
    }
    if (tid == 0) *cl.map_shared_rank(&s_tops[rank], 0) = (unsigned long long)(s_thr | 0x80000000u) << 32 | s_low;
    // ---- every value of the slice that reaches it ----
    unsigned long long *dst = CL > 1 ? cl.map_shared_rank(cand, 0) : cand;
    int *ctr = CL > 1 ? cl.map_shared_rank(&s_n, 0) : &s_n;
    auto consider = [&](uint32_t bits, int x) {
        if ((int)bits < thr || x == xd || !(__uint_as_float(bits) > 0.0f)) return;  // (NaN: not > 0)
        const int at = atomicAdd(ctr, 1);
        if (at < CCAP && ACES_IN(at, CCAP)) dst[at] = order_val(bits | 0x80000000u, (uint32_t)x);
    };
    for (int it = 0; it < nit; ++it) {
        if (it > 0) {
#pragma unroll
            for (int u = 0; u < CLD; ++u) {
                cb[u] = at_b;
                at_b += NTC;
                if (++at_o == nit) {  // (past a segment's sample)
                    at_o = 1;
                    at_b += NTC;
                }
            }
            load();
        }
#pragma unroll
        for (int u = 0; u < CLD; ++u) {
            // one test per four values: the largest
            if (max(max((int)w[u].x, (int)w[u].y), max((int)w[u].z, (int)w[u].w)) >= thr) {
                const int x0 = (c_lo + cb[u] + tid) * 4 - qc.head;
                consider(w[u].x, x0);
                consider(w[u].y, x0 + 1);
                consider(w[u].z, x0 + 2);
                consider(w[u].w, x0 + 3);
            }
        }
    }
    if (tie && __uint_as_float(s_thr) > 0.0f) {  // the first ids of the threshold's value (not a NaN's)
        const uint32_t bits0 = s_thr, last = 0xFFFFFFFFu - s_low;
        for (int c = c_lo + tid; c < c_lo + cn && (long long)c * 4 - qc.head <= (long long)last; c += NTC) {
            const uint4 v = qc.load(c);
            const uint32_t b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int x = c * 4 - qc.head + e;
                if (b[e] != bits0 || x == xd || (uint32_t)x > last) continue;
                const int at = atomicAdd(ctr, 1);
                if (at < CCAP && ACES_IN(at, CCAP)) dst[at] = order_val(bits0 | 0x80000000u, (uint32_t)x);
            }
        }
    }
    if (CL > 1) cl.sync();
    else __syncthreads();
    if (rank != 0) return;  // (nobody reads another CTA's shared memory any more)
    // ---- the first Fd of them ----
    // A value dropped lies below its slice's threshold, so the candidates hold
    // the row's Fd largest when Fd of them reach the largest threshold (or
    // when nothing positive was dropped).
    int n = s_n;
    unsigned long long top = s_tops[0];  // the largest threshold
    for (int c = 1; c < CL; ++c) top = s_tops[c] > top ? s_tops[c] : top;
    bool enough = n <= CCAP;
    if (enough && top > LOWEST) {
        int nr = 0, reach;
        for (int i = tid; i < n; i += NTC) nr += cand[i] >= top;
        if (n <= 2 * NTC) reach = __syncthreads_count(nr >= 1) + __syncthreads_count(nr >= 2);
        else reach = (int)block_reduce_n<NTC>((unsigned long long)nr, red, SumU64());
        enough = reach >= Fd;
    }
    if (!enough) n = cache_row_select(qr, a.V, xd, Fd, cand);
    const int got = min(n, Fd);
    if (n <= RANK_MAX) {
        for (int i = tid; i < n; i += NTC) {
            const unsigned long long key = cand[i];
            int rk = 0;
#pragma unroll 4
            for (int t = 0; t < n; ++t) rk += cand[t] > key;
            if (rk < Fd) {
                bt[rk] = (int32_t)order_id(key);
                bp[rk] = order_value(key) / den;
            }
        }
    } else {
        const int np = next_pow2(n);
        for (int i = n + tid; i < np; i += NTC) cand[i] = 0ull;
        __syncthreads();
        bitonic_sort_desc(cand, np);
        for (int j = tid; j < got; j += NTC) {
            bt[j] = (int32_t)order_id(cand[j]);
            bp[j] = order_value(cand[j]) / den;
        }
    }
    for (int j = got + tid; j < Fd; j += NTC) {
        bt[j] = -1;
        bp[j] = 0.0f;
    }
}

__global__ void k_cache_lookup(const int32_t *bt, CacheArgs a, const int32_t *accept_len,
                               const int32_t *token, int32_t *slot) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.B) return;
    const int pi = accept_len[b];
    if (pi == a.K) {
        slot[b] = -2;
        return;
    }
    int s = -1;
    const int tok = token[b];
    if (pi >= 0 && pi < a.K && tok >= 0) {
        const int32_t *row = bt + (size_t)b * a.total + a.off[pi];
        for (int j = 0; j < a.F[pi]; ++j)
            if (row[j] == tok) {
                s = a.off[pi] + j;
                break;
            }
    }
    slot[b] = s;
}

// One cluster per row: as many CTAs (up to CCL) as fit four an SM at once.
cudaError_t launch_cache_build(const CacheArgs &a, int nsm, cudaStream_t s) {
    const long long rows = (long long)a.B * a.K;
    int cl = CCL;
    while (cl > 1 && (rows * cl > 4LL * nsm || a.V < cl * 1024)) cl >>= 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(rows * cl));
    cfg.blockDim = dim3(NTC);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_cache_build, a);
}

cudaError_t launch_cache_lookup(const int32_t *bt, const CacheArgs &a, const int32_t *accept_len,
                                const int32_t *token, int32_t *slot, cudaStream_t s) {
    k_cache_lookup<<<(a.B + 255) / 256, 256, 0, s>>>(bt, a, accept_len, token, slot);
    return cudaGetLastError();
}

#ifdef ACES_CHECKED
cudaError_t check_take_cache(unsigned long long out[3]) { return check_take(out); }
cudaError_t check_take_selects(unsigned int *n) {
    const unsigned int zero = 0u;
    const cudaError_t e = cudaMemcpyFromSymbol(n, g_selects, sizeof(*n));
    return e != cudaSuccess ? e : cudaMemcpyToSymbol(g_selects, &zero, sizeof(zero));
}
#endif

}  // namespace aces
