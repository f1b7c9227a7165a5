// Edge-side resample from the sparse downlink payload (Alg. 1
// RESAMPLE(P^_target, Q); Sec. III-B): the cloud returns the rejection index
// pi and the partial target distribution of row pi, and the edge draws the
// corrected token itself from that payload and its own draft row q_pi.
//
// The edge knows the target p only on the payload ids I (probs p^_I) and the
// mass tau = tail outside them.  For pi < K the tail is spread like the
// draft: p^(x) = tau * q(x) / q_rest outside I, with q_rest the draft mass
// outside I, so the residual r^ = max(0, p^ - q) is max(0, p^_x - q(x)) on I
// and q(x) * max(0, tau / q_rest - 1) outside.  For pi = K (bonus) the draw
// uses p^_I alone.  When the nucleus of row pi fits in the payload, tau = 0
// and the draw is the exact residual draw of aces_verify.
//
// One thread-block cluster of 8 CTAs (512 threads each) per sequence:
//   1. the payload of row pi is ordered by id in shared memory (direct rank
//      counting), and its weights (p^ - q on I) are gathered;
//   2. only when tau > 0, the 8 CTAs split q_pi's 16-byte chunks: one pass
//      gives each CTA's share of q_rest (compensated fp32), combined through
//      distributed shared memory; once the spread factor is known a second
//      pass (from L2) gives the weight of every task of whole warp steps, and
//      the CTA holding the draw scans its task with one warp.  A bit per
//      chunk says whether it holds payload ids: nearly none does, and the
//      others need no look at the payload (a merge of every id with the
//      sorted payload took 45 us on 32 rows of 152064 with k = 32).
//      Otherwise the first CTA draws alone and the others exit at once;
//   3. the draw: smallest id j whose prefix sum exceeds floor(u * R), with
//      every weight an integer in units of 2^-52 (exact, order independent).
#include <cooperative_groups.h>

#define ACES_FILE 7  // site numbers of the checked build
#include "qrow.cuh"

namespace aces {

constexpr int NTS = 512;
constexpr int NWS = NTS / 32;
constexpr int SPAY = ACES_MAX_TOPK;    // payload entries
constexpr int SCL = 8;                 // CTAs per sequence: one thread-block cluster
constexpr int SU = 4;                  // warp steps (32 chunks) in flight
constexpr int SSTEPS = (ACES_MAX_V / 4 + 1 + 32 * SCL - 1) / (32 * SCL);  // warp steps of a CTA, at most
constexpr int STASKS = NTS;            // tasks of a CTA, at most

// floor(x * 2^52) of a float x in [0, 2^11) from its bits (0 for x <= 0 or NaN)
__device__ __forceinline__ unsigned long long to_fx52(float x) {
    if (!(x > 0.0f)) return 0ull;
    const uint32_t u = __float_as_uint(x);
    const uint32_t be = u >> 23;
    const unsigned long long mant = (unsigned long long)((u & 0x7FFFFFu) | 0x800000u);
    const int sh = (int)be - 98;  // x * 2^52 = mant * 2^(be - 127 - 23 + 52)
    if (sh >= 40) return ~0ull >> 1;
    return sh >= 0 ? (mant << sh) : (sh > -64 ? (mant >> (-sh)) : 0ull);
}

struct SparseArgs {
    const int32_t *accept_len, *ids, *row_status;
    const float *probs, *tail, *q, *u;
    int B, K, V, k;
    int32_t *token, *status;
};

// first index i in sid[0, n) with sid[i] >= x
__device__ __forceinline__ int lower_bound_id(const int *sid, int n, int x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (sid[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// What a CTA shares with its cluster.
struct SparsePart {
    unsigned long long w;  // weight of its slice
    float ph, pl;          // its share of q_rest
    int bad;
};

__global__ void __cluster_dims__(SCL, 1, 1) __launch_bounds__(NTS) k_resample_sparse(SparseArgs a) {
    namespace cg = cooperative_groups;
    __shared__ unsigned long long skey[SPAY];  // id << 32 | entry (all ones: invalid id)
    __shared__ int sid[SPAY];                  // valid payload ids, ascending
    __shared__ int sidx[SPAY];                 // their payload entries
    __shared__ unsigned long long sw[SPAY];    // their weights (2^-52 units)
    __shared__ uint32_t held[SSTEPS];          // bit l of word k: chunk l of warp step k holds a payload id
    __shared__ unsigned long long tsum[STASKS];  // this CTA's tasks
    __shared__ unsigned long long red[NWS];
    __shared__ float redh[NWS], redl[NWS];
    __shared__ SparsePart part, parts[SCL];
    __shared__ int s_n, s_bad, s_tok, s_task;
    __shared__ float s_gam;
    __shared__ unsigned long long s_base;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int b = blockIdx.x / SCL, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int R1 = a.K + 1;
    const int pi = a.accept_len[b];
    const bool bad_row = pi < 0 || pi > a.K || (a.row_status[(size_t)b * R1 + pi] & ACES_ROW_NONFINITE);
    const size_t row = (size_t)b * R1 + (bad_row ? 0 : pi);
    const float tau = a.tail[row];
    const float *qr = (!bad_row && pi < a.K) ? a.q + ((size_t)b * a.K + pi) * a.V : nullptr;
    // The whole cluster takes part only when the tail may be spread (pi < K,
    // tau > 0): every CTA then decides the same way from the same inputs, so
    // all of them reach every cluster barrier.  Otherwise rank 0 works alone.
    const bool cluster_work = qr != nullptr && tau > 0.0f;
    if (!cluster_work && rank != 0) return;
    if (bad_row) {
        if (tid == 0) {
            a.token[b] = -1;
            a.status[b] = ACES_ROW_NONFINITE;
        }
        return;
    }
    const int32_t *I = a.ids + row * a.k;
    const float *P = a.probs + row * a.k;
    const int V = a.V;
    // this CTA's chunks of q_pi: nstep warp steps of 32 from chunk c_lo
    const QChunks qc(qr != nullptr ? qr : a.q, V);
    const int nws = (qc.nch + 31) / 32, pw = (nws + SCL - 1) / SCL;
    const int w_lo = min(nws, rank * pw), nstep = min(nws, w_lo + pw) - w_lo;
    const int c_lo = w_lo * 32;

    // ---- 1. payload sorted by id, weights on it ----
    // The valid entries (0 <= id < V) are ordered by (id, entry) by direct
    // rank counting: one pass, no barrier stages.
    if (tid == 0) {
        s_n = 0;
        s_bad = 0;
        s_tok = -1;
        s_task = -1;
        s_gam = 0.0f;
    }
    for (int j = tid; j < a.k; j += NTS) {
        unsigned long long key = ~0ull;  // invalid: after every valid key
        const int x = I[j];
        if (x >= 0 && x < V) key = ((unsigned long long)x << 32) | (unsigned long long)j;
        skey[j] = key;
    }
    if (cluster_work)
        for (int i = tid; i < nstep; i += NTS)
            if (ACES_IN(i, SSTEPS)) held[i] = 0u;
    __syncthreads();
    for (int j = tid; j < a.k; j += NTS) {
        const unsigned long long key = skey[j];
        if (key == ~0ull) continue;
        int rk = 0;
#pragma unroll 8
        for (int i = 0; i < a.k; ++i) rk += skey[i] < key;
        const int x = (int)(key >> 32), e = (int)(key & 0xFFFFFFFFull);
        float w = fmaxf(P[e], 0.0f);
        if (qr && ACES_IN(x, V)) {
            const float qx = __ldg(qr + x);
            if (!(qx >= 0.0f)) s_bad = 1;
            w = fmaxf(P[e] - qx, 0.0f);
        }
        if (ACES_IN(rk, SPAY)) {
            sid[rk] = x;
            sidx[rk] = e;
            sw[rk] = to_fx52(w);
        }
        atomicAdd(&s_n, 1);
        const int c = ((x + qc.head) >> 2) - c_lo;
        if (cluster_work && c >= 0 && c < nstep * 32 && ACES_IN(c >> 5, SSTEPS)) atomicOr(&held[c >> 5], 1u << (c & 31));
    }
    __syncthreads();
    const int n = s_n;
    const int bad_pay = s_bad;
    __syncthreads();  // (the pass below sets s_bad: every thread has read it)
    if (bad_pay || n == 0) {  // the same in every CTA of the cluster
        if (rank == 0 && tid == 0) {
            a.token[b] = -1;
            a.status[b] = bad_pay ? ACES_ROW_BAD_Q : 0;
        }
        return;
    }
    // the chunk of this lane in warp step k (0 outside the row)
    auto load = [&](int k) {
        const int c = c_lo + k * 32 + lane;
        return k < nstep && c < qc.nch ? qc.load(c) : make_uint4(0u, 0u, 0u, 0u);
    };
    auto first_id = [&](int k) { return (c_lo + k * 32 + lane) * 4 - qc.head; };
    // the payload entry of id x, -1 when there is none
    auto entry_of = [&](int x) {
        const int j = lower_bound_id(sid, n, x);
        return j < n && sid[j] == x ? j : -1;
    };

    // ---- 2. the tail, spread like the draft (pi < K, tau > 0): the cluster ----
    const int spt = (pw + STASKS - 1) / STASKS;  // warp steps per task
    const int ntask = (nstep + spt - 1) / spt;
    bool spread = false;
    float gam = 0.0f;
    unsigned long long thr = 0ull;
    if (cluster_work) {
        float hi = 0.0f, lo = 0.0f;  // compensated sum of q outside the payload
        int bad = 0;
        for (int k0 = wid; k0 < nstep; k0 += NWS * SU) {
            uint4 v[SU];
#pragma unroll
            for (int i = 0; i < SU; ++i) v[i] = load(k0 + i * NWS);
#pragma unroll
            for (int i = 0; i < SU; ++i) {
                const int k = k0 + i * NWS;
                if (k >= nstep) break;
                float q[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    q[e] = Elem<ACES_F32>::get(v[i], e);
                    if (!(q[e] >= 0.0f)) bad = 1;
                }
                if ((held[k] >> lane) & 1u) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (entry_of(first_id(k) + e) >= 0) q[e] = 0.0f;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {  // two-sum
                    const float t = hi + q[e], bb = t - hi;
                    lo += (hi - (t - bb)) + (q[e] - bb);
                    hi = t;
                }
            }
        }
        if (bad) s_bad = 1;
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
            const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
            const float sm = hi + h2;
            const float bb = sm - hi;
            lo = lo + l2 + ((hi - (sm - bb)) + (h2 - bb));
            hi = sm;
        }
        if (lane == 0) {
            redh[wid] = hi;
            redl[wid] = lo;
        }
        for (int i = tid; i < ntask; i += NTS) tsum[i] = 0ull;
        __syncthreads();
        if (tid == 0) {
            float h = 0.0f, l = 0.0f;
            for (int i = 0; i < NWS; ++i) {
                const float sm = h + redh[i];
                const float bb = sm - h;
                l = l + redl[i] + ((h - (sm - bb)) + (redh[i] - bb));
                h = sm;
            }
            part.ph = h;
            part.pl = l;
            part.bad = s_bad;
        }
        cl.sync();  // every CTA's share is written
        if (tid < SCL) parts[tid] = *cl.map_shared_rank(&part, tid);
        __syncthreads();
        if (tid == 0) {  // every CTA sums the shares in rank order: the same value everywhere
            double qrest = 0.0;
            int anybad = 0;
            for (int j = 0; j < SCL; ++j) {
                qrest += (double)parts[j].ph + (double)parts[j].pl;
                anybad |= parts[j].bad;
            }
            const double g = qrest > 0.0 ? (double)tau / qrest - 1.0 : 0.0;
            s_gam = g > 0.0 ? (float)g : 0.0f;
            s_bad = anybad;
        }
        cl.sync();  // the shares are read before any CTA moves on or exits
        if (s_bad) {
            if (rank == 0 && tid == 0) {
                a.token[b] = -1;
                a.status[b] = ACES_ROW_BAD_Q;
            }
            return;
        }
        gam = s_gam;
        spread = gam > 0.0f;
        if (!spread && rank != 0) return;
    }
    // the weights of a chunk's ids: q * gam outside the payload, sw on it
    auto weights = [&](int k, const uint4 &v, unsigned long long (&w)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = to_fx52(Elem<ACES_F32>::get(v, e) * gam);
        if ((held[k] >> lane) & 1u) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = entry_of(first_id(k) + e);
                if (j >= 0) w[e] = sw[j];
            }
        }
    };

    // ---- 3. the draw ----
    if (spread) {
        for (int k0 = wid; k0 < nstep; k0 += NWS * SU) {
            uint4 v[SU];
#pragma unroll
            for (int i = 0; i < SU; ++i) v[i] = load(k0 + i * NWS);
#pragma unroll
            for (int i = 0; i < SU; ++i) {
                const int k = k0 + i * NWS;
                if (k >= nstep) break;  // (warp-uniform)
                unsigned long long w[4];
                weights(k, v[i], w);
                const unsigned long long ws = warp_sum((w[0] + w[1]) + (w[2] + w[3]));
                if (lane == 0 && ACES_IN(k / spt, STASKS)) atomicAdd(&tsum[k / spt], ws);
            }
        }
        __syncthreads();
        const unsigned long long own = tid < ntask ? tsum[tid] : 0ull;
        unsigned long long tot;
        const unsigned long long ex = block_exscan_n<NTS>(own, red, &tot);
        if (tid == 0) part.w = tot;
        cl.sync();  // every CTA's weight is written
        if (tid < SCL) parts[tid].w = cl.map_shared_rank(&part, tid)->w;
        __syncthreads();
        unsigned long long R = 0ull, before = 0ull;
        for (int j = 0; j < SCL; ++j) {
            if (j == rank) before = R;
            R += parts[j].w;
        }
        cl.sync();  // the weights are read before any CTA exits
        if (R == 0ull) {  // nothing above 2^-52: rank 0 draws on the payload
            spread = false;
            if (rank != 0) return;
        } else {
            thr = floor_u_times(a.u[(size_t)b * R1 + a.K], R);
            if (!(before <= thr && thr < before + tot)) return;  // another CTA holds the draw
            if (before + ex <= thr && thr < before + ex + own) {  // (one thread)
                s_task = tid;
                s_base = before + ex;
            }
            __syncthreads();
        }
    }
    if (spread) {
        // one warp scans the task holding the draw
        if (wid == 0) {
            unsigned long long base = s_base;
            for (int k = s_task * spt; k < min(nstep, (s_task + 1) * spt); ++k) {
                unsigned long long w[4];
                weights(k, load(k), w);
                const unsigned long long loc = (w[0] + w[1]) + (w[2] + w[3]);
                unsigned long long inc = loc;
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += t;
                }
                unsigned long long c = base + inc - loc;
                const bool mine = c <= thr && thr < c + loc;
                if (mine) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        c += w[e];
                        if (c > thr) {
                            s_tok = first_id(k) + e;
                            break;
                        }
                    }
                }
                if (__any_sync(0xffffffffu, mine)) break;
                base += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        __syncthreads();
    } else {
        // weights on the payload only (ascending id): one entry per thread
        unsigned long long w = tid < n ? sw[tid] : 0ull;
        unsigned long long tot;
        unsigned long long ex = block_exscan_n<NTS>(w, red, &tot);
        if (tot == 0ull) {  // p^ <= q wherever it is known: draw from p^ on the payload
            __syncthreads();
            if (tid < n) sw[tid] = to_fx52(fmaxf(P[sidx[tid]], 0.0f));
            __syncthreads();
            w = tid < n ? sw[tid] : 0ull;
            ex = block_exscan_n<NTS>(w, red, &tot);
        }
        if (tot > 0ull) {
            const unsigned long long t2 = floor_u_times(a.u[(size_t)b * R1 + a.K], tot);
            if (ex <= t2 && t2 < ex + w) s_tok = sid[tid];
        }
        __syncthreads();
    }
    if (tid == 0) {
        a.token[b] = s_tok;
        a.status[b] = 0;
    }
}

cudaError_t launch_resample_sparse(const int32_t *accept_len, const int32_t *ids, const float *probs,
                                   const float *tail, const int32_t *row_status, const float *q,
                                   const float *u, int B, int K, int V, int k, int32_t *token,
                                   int32_t *status, cudaStream_t s) {
    SparseArgs a;
    a.accept_len = accept_len;
    a.ids = ids;
    a.row_status = row_status;
    a.probs = probs;
    a.tail = tail;
    a.q = q;
    a.u = u;
    a.B = B;
    a.K = K;
    a.V = V;
    a.k = k;
    a.token = token;
    a.status = status;
    k_resample_sparse<<<B * SCL, NTS, 0, s>>>(a);
    return cudaGetLastError();
}

#ifdef ACES_CHECKED
cudaError_t check_take_resample(unsigned long long out[3]) { return check_take(out); }
#endif

}  // namespace aces
