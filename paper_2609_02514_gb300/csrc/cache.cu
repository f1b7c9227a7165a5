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
//                   largest it is ordered in shared memory; otherwise (about
//                   one row in 10^4, or more equal values than fit) the row
//                   is read again, TOPL maxima at a time.  Small batches
//                   split a row over a cluster of CTAs whose candidates meet
//                   in the first one's shared memory.
//   k_cache_lookup  one thread per sequence scanning the F_pi branches.
#include <cooperative_groups.h>

#define ACES_FILE 3  // site numbers of the checked build
#include "qrow.cuh"

namespace aces {


constexpr int NTC = 256;   // threads per CTA
constexpr int CLD = 8;     // 16-byte loads in flight per thread
constexpr int CCAP = 4096; // candidates kept per row
constexpr int CCL = 8;     // CTAs of a row's cluster, at most
constexpr int TOPL = 8;    // per-thread list of the repeated passes
constexpr int RANK_MAX = 512;  // candidates ordered by direct ranking (more: bitonic sort)

__device__ __forceinline__ void list_insert(unsigned long long (&Lst)[TOPL], unsigned long long o) {
    Lst[TOPL - 1] = o;
#pragma unroll
    for (int i = TOPL - 1; i > 0; --i) {
        if (Lst[i] > Lst[i - 1]) {
            const unsigned long long t = Lst[i];
            Lst[i] = Lst[i - 1];
            Lst[i - 1] = t;
        }
    }
}

// Repeated passes over the row, TOPL maxima at a time below the last extracted
// order value: exact on any row (one CTA; the row's Fd outputs, padding aside).
// Returns the number of branches written.
__device__ __noinline__ int cache_row_passes(const float *qr, int V, int xd, float den, int Fd, int32_t *bt, float *bp) {
    __shared__ unsigned long long redu[NTC / 32];
    const QChunks qc(qr, V);
    const int tid = threadIdx.x;
    int got = 0;
    unsigned long long ub = ~0ull;  // exclusive upper bound of this pass
    while (got < Fd) {
        unsigned long long Lst[TOPL];
#pragma unroll
        for (int i = 0; i < TOPL; ++i) Lst[i] = 0ull;
        for (int c = tid; c < qc.nch; c += NTC) {
            const uint4 w = qc.load(c);
            const int thr = max(1, (int)((uint32_t)(Lst[TOPL - 1] >> 32) & 0x7FFFFFFFu));
            if (max(max((int)w.x, (int)w.y), max((int)w.z, (int)w.w)) < thr) continue;
#pragma unroll 1
            for (int e = 0; e < 4; ++e) {
                const uint32_t bits = e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w;
                const int x = c * 4 - qc.head + e;
                if ((int)bits < thr || !(__uint_as_float(bits) > 0.0f) || x == xd) continue;
                const unsigned long long o = order_val(bits | 0x80000000u, (uint32_t)x);
                if (o < ub && o > Lst[TOPL - 1]) list_insert(Lst, o);
            }
        }
        const int take = min(TOPL, Fd - got);
        for (int t = 0; t < take; ++t) {
            const unsigned long long best = block_reduce_n<NTC>(Lst[0], redu, MaxU64());
            if (best == 0ull) return got;
            if (Lst[0] == best) {  // order values are unique: one owner
#pragma unroll
                for (int i = 0; i < TOPL - 1; ++i) Lst[i] = Lst[i + 1];
                Lst[TOPL - 1] = 0ull;
            }
            if (tid == 0) {
                bt[got] = (int32_t)order_id(best);
                bp[got] = order_value(best) / den;
            }
            ++got;
            ub = best;
        }
    }
    return got;
}

// One row of q by a cluster of 1 to CCL CTAs, each reading a slice.  Bound by
// HBM on large batches: 579 us for 256 x 16 rows of 256000 with a support cut
// and F = 4 (583 with a sorted list of four per thread and no threshold, 700
// on wider support, where its insertions diverge: 595 here), 640 with F = 64
// (1000 with lists of eight and a 2048-entry sort a row); 64 rows of full
// support with F = 64 195 us (383).  One sequence of 16 x 128256 takes 13 us on
// clusters of eight (22 with a CTA a row).
__global__ void __launch_bounds__(NTC, 4) k_cache_build(CacheArgs a) {
    namespace cg = cooperative_groups;
    __shared__ unsigned long long cand[CCAP];  // candidates' order values (the first CTA's: the cluster's)
    __shared__ uint32_t smax[NTC];             // sample: per-thread maxima
    __shared__ uint32_t s_thr, s_top;          // this CTA's threshold; the cluster's largest
    __shared__ int s_n;                        // candidates (may pass CCAP)
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
    if (tid == 0) {
        s_n = 0;
        s_top = 0u;
    }
    const QChunks qc(qr, a.V);
    // This CTA's chunks [c_lo, c_lo + cn), in blocks of NTC.  Iteration 0 is a
    // sample: the first block of each of eight segments of nit blocks.  The
    // others take the remaining blocks in order, which reads a little faster
    // (one block of each segment every time: 583 us against 579 on 256 x 16
    // rows of 256000; with bounds and edges tested per chunk 595).
    const int per = (qc.nch + CL - 1) / CL, c_lo = min(qc.nch, rank * per), cn = min(qc.nch, c_lo + per) - c_lo;
    const int nit = (cn + CLD * NTC - 1) / (CLD * NTC);
    uint4 w[CLD];
    int cb[CLD];                // the iteration's blocks (their first chunk)
    int at_b = NTC, at_o = 1;   // the next block, its number in its segment
#pragma unroll
    for (int u = 0; u < CLD; ++u) cb[u] = u * nit * NTC;
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
    // Positive floats order like their bits; negative q (and the padding) are
    // at most 0 as integers.
    int mx = 0;
#pragma unroll
    for (int u = 0; u < CLD; ++u) mx = max(mx, max(max((int)w[u].x, (int)w[u].y), max((int)w[u].z, (int)w[u].w)));
    smax[tid] = (uint32_t)mx;
    if (CL > 1) cl.sync();  // (every CTA's counters are set before another adds to them)
    else __syncthreads();
    if (tid < 32) {
        // The slice must keep its `want` largest: all Fd with one CTA, else a
        // share with a margin (checked below against the other slices).  Of
        // those the sample holds want * f on average; its rank-r value with r
        // four deviations above that is below the want-th largest but for
        // about one row in 10^4 (then the passes above take the row), and
        // about r / f values reach it.  Every thread's maximum stands for its
        // 32 values: the rank among the NTC maxima is corrected for values
        // that share a thread.
        const float Ff = (float)Fd, want = CL == 1 ? Ff : fminf(Ff, Ff / CL + 4.0f * sqrtf(Ff / CL) + 8.0f);
        const float f = cn > 0 ? fminf(1.0f, (float)(CLD * NTC) / (float)cn) : 1.0f;
        const float wf = want * f;
        const float r = f < 1.0f ? wf + 4.0f * sqrtf(wf) + 4.0f : want + 1.0f;
        const float rm = f < 1.0f ? (float)NTC * (1.0f - exp2f(-1.4427f * r / (float)NTC)) : r;
        const int need = (int)ceilf(rm);
        uint32_t v[NTC / 32], thr = 0u;
#pragma unroll
        for (int i = 0; i < NTC / 32; ++i) v[i] = smax[i * 32 + lane];
        // the largest threshold (its exponent and four bits) that `need` maxima reach
        if (need <= NTC)
            for (int bit = 30; bit >= 19; --bit) {
                const uint32_t t = thr | 1u << bit;
                uint32_t n = 0u;
#pragma unroll
                for (int i = 0; i < NTC / 32; ++i) n += v[i] >= t;
                if (__reduce_add_sync(0xffffffffu, n) >= (uint32_t)need) thr = t;
            }
        if (tid == 0) {
            s_thr = thr > 1u ? thr : 1u;  // (at least 1: q > 0)
            if (CL > 1) atomicMax(cl.map_shared_rank(&s_top, 0), s_thr);
        }
    }
    __syncthreads();
    const int thr = (int)s_thr;
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
                if (++at_o == nit) {  // (past the next segment's sample)
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
    if (CL > 1) cl.sync();
    else __syncthreads();
    if (rank != 0) return;  // (nobody reads another CTA's shared memory any more)
    // ---- the first Fd of them ----
    // A value dropped lies below its slice's threshold, so the candidates hold
    // the row's Fd largest when Fd of them reach the largest threshold (or
    // when nothing positive was dropped).
    const int n = s_n;
    const uint32_t top = CL > 1 ? s_top : s_thr;
    int got = -1;
    if (n <= CCAP) {
        const unsigned long long *ord = cand;
        if (n <= RANK_MAX) {
            // (rank Fd - 1 settles whether the candidates are enough)
            uint32_t nr = 0u;
            for (int i = tid; i < n; i += NTC) nr += (uint32_t)(cand[i] >> 32) >= (top | 0x80000000u);
            const int reach = __syncthreads_count(nr >= 1u) + __syncthreads_count(nr >= 2u);
            if (reach >= Fd || top <= 1u) {
                got = min(n, Fd);
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
            }
        } else {
            const int np = next_pow2(n);
            for (int i = n + tid; i < np; i += NTC) cand[i] = 0ull;
            __syncthreads();
            bitonic_sort_desc(cand, np);
            if (top <= 1u || (n >= Fd && (uint32_t)(ord[Fd - 1] >> 32) >= (top | 0x80000000u))) {
                got = min(n, Fd);
                for (int j = tid; j < got; j += NTC) {
                    bt[j] = (int32_t)order_id(ord[j]);
                    bp[j] = order_value(ord[j]) / den;
                }
            }
        }
    }
    if (got < 0) got = cache_row_passes(qr, a.V, xd, den, Fd, bt, bp);
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
#endif

}  // namespace aces
