// Sequence step of AceSpec verification (Sec. III-B, Algorithm 1): the first
// rejection index pi of a drafted chain and the token emitted at pi, drawn
// from norm(max(0, p_pi - q_pi)) when pi < K (from p_pi itself when that is
// all zero) or from p_K when the whole chain was accepted.
//
// The draw is the smallest id j whose prefix sum over ids 0..j exceeds
// u[b, K] times the total.  Every probability enters as an integer in units
// of 2^-40, so all partial sums are exact and independent of the order in
// which threads add them: the three forms below give the same token.
//
//   draw_list     row pi's nucleus was kept (top_p < 1, at most NUC_CAP ids):
//                 the residual max(0, p - q) is zero outside it, so q is read
//                 at those ids only, they are ordered by id, and the draw is
//                 taken from their prefix sums.  Run by the CTA that finishes
//                 the sequence's last row.
//   draw_cluster  the other sequences: a cluster of CTAs sums the residual of 32-chunk
//                 tasks of row pi (q is read where a chunk holds a nucleus
//                 id), then one warp scans the task holding the draw.  Run by
//                 the general kernel once its rows are done, and for the
//                 sequences that they complete.
//   draw_scan     sequences whose residual is zero everywhere: one CTA, the
//                 same with more sums (p as well) and a loop over the members.
// When row pi kept its cut as (value v, count j) (RS_LAZY: the nucleus ends
// among the ids of one bfloat16 value, which the row kernel did not list), the
// ids of value v are summed and counted apart, and the task holding the j-th
// of them (in id order) is scanned first.
#pragma once
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "common.cuh"

namespace aces {

constexpr int DRAW_TASKS = 512;
constexpr int DRAW_CL = 8;  // CTAs of a draw's cluster, at most
constexpr int DRAW_CH = 4;  // 16-byte chunks per lane and step of a task
constexpr int DRAW_SCRATCH = 4 * NUC_CAP * 8;  // bytes of shared memory the draws use, on a 16-byte boundary
static_assert(DRAW_TASKS * (3 * 8 + 4) <= DRAW_SCRATCH, "the tasks' sums fit");
static_assert(2 * NUC_CAP * 8 % 16 == 0, "the list's 32-bit keys are read 16 bytes at a time");

// A row of V logits in 16-byte chunks.  A row that does not start on a
// 16-byte boundary begins `head` elements into chunk 0: element e of chunk c
// is id c * EPC + e - head, and the first and last chunk are read element by
// element (-inf outside the row).  RAGGED = false: the row is whole chunks.
template <int DT, bool RAGGED = true>
struct RowChunks {
    static constexpr int EPC = Elem<DT>::EPC;
    const char *base;  // chunk 0
    int head, V, nch;
    __device__ __forceinline__ RowChunks(const char *row, int V_) : V(V_) {
        head = RAGGED ? (int)((uintptr_t)row & 15u) / Elem<DT>::SIZE : 0;
        base = row - head * Elem<DT>::SIZE;
        nch = (V + head + EPC - 1) / EPC;
    }
    __device__ __forceinline__ const char *row() const { return base + head * Elem<DT>::SIZE; }
    __device__ __forceinline__ bool whole(int c) const { return !RAGGED || (c * EPC >= head && (c + 1) * EPC <= V + head); }
    // the elements from id x0 on, one by one (V: the row's length)
    static __device__ __noinline__ uint4 edge(const char *row, int V, int x0) {
        uint32_t wd[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            wd[q] = Elem<DT>::NEG_INF_WORD;
#pragma unroll
            for (int h = 0; h < EPC / 4; ++h) {
                const int x = x0 + q * (EPC / 4) + h;
                if (x >= 0 && x < V) {
                    const uint32_t bits = __float_as_uint(Elem<DT>::load1(row, x));
                    if (DT == ACES_BF16) wd[q] = h ? ((wd[q] & 0xFFFFu) | bits) : ((wd[q] & 0xFFFF0000u) | bits >> 16);
                    else wd[q] = bits;
                }
            }
        }
        return make_uint4(wd[0], wd[1], wd[2], wd[3]);
    }
    __device__ __forceinline__ uint4 load(int c) const {
        return whole(c) ? ldg16(base + (size_t)c * 16) : edge(base + head * Elem<DT>::SIZE, V, c * EPC - head);
    }
};

// What the scan needs of a sequence and its row pi.
struct ScanRow {
    const char *z;       // logits
    const float *q;      // draft row (null: the bonus position)
    int V, flags;
    float c, kref, inv_S, u;
    unsigned long long cut;
};

// a row's state, perhaps written by another CTA of this kernel
__device__ __forceinline__ RowStat row_stat(const Workspace &ws, int r) {
    union {
        uint4 w[2];
        RowStat rs;
    } v;
    const uint4 *p = reinterpret_cast<const uint4 *>(ws.stats + r);
    v.w[0] = __ldcg(p);
    v.w[1] = __ldcg(p + 1);
    return v.rs;
}

template <int DT>
__device__ __forceinline__ ScanRow scan_row(const RowArgs &a, int b, int pi, const RowStat &rs) {
    ScanRow s;
    s.z = reinterpret_cast<const char *>(a.logits) + (size_t)(b * (a.K + 1) + pi) * a.V * Elem<DT>::SIZE;
    s.q = pi < a.K ? a.q + ((size_t)b * a.K + pi) * a.V : nullptr;
    s.V = a.V;
    s.flags = rs.flags;
    s.c = rs.c;
    s.kref = rs.kref;
    s.inv_S = inv_mass(rs.S_nuc);
    s.u = a.u[(size_t)b * (a.K + 1) + a.K];
    s.cut = rs.cut;
    return s;
}

// the outputs of sequence b (tok: -1 none, -2 an invalid q); one thread
__device__ __forceinline__ void write_draw(const RowArgs &a, int b, int pi, int tok) {
    if (tok == -2) a.row_status[b * (a.K + 1) + pi] |= ACES_ROW_BAD_Q;
    a.accept_len[b] = pi;
    a.out_token[b] = tok < 0 ? -1 : tok;
}

// membership of a chunk's ids: bit e of the result when element e is in the
// nucleus (or holds a lazy cut's value: also in *tie); x0: the id of element 0
template <int DT>
__device__ __forceinline__ uint32_t member_bits(const uint4 &w, int x0, const ScanRow &s, uint32_t *tie) {
    uint32_t in = 0u, tm = 0u;
    const uint32_t vkey = (uint32_t)(s.cut >> 32);
    if (DT == ACES_BF16 && (s.flags & (RS_LAZY | RS_ALL_IN))) {
        // two ids per compare: lazily cut, members are the ids >= the cut's
        // value, ties those == it (IEEE order: +0 and -0 are one value); with
        // every id in, those above -inf
        const float vv = fkey_inv(vkey);
        const __nv_bfloat162 t2 = __floats2bfloat162_rn(vv, vv);
        const uint32_t wd[4] = {w.x, w.y, w.z, w.w};
        const bool all = (s.flags & RS_ALL_IN) != 0;
        const uint32_t ni = Elem<ACES_BF16>::NEG_INF_WORD;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162 *>(&wd[q]);
            const uint32_t ge = all ? __hgt2_mask(h, *reinterpret_cast<const __nv_bfloat162 *>(&ni)) : __hge2_mask(h, t2);
            const uint32_t eq = all ? 0u : __heq2_mask(h, t2);
            in |= ((ge & 1u) | ((ge >> 15) & 2u)) << (2 * q);
            tm |= ((eq & 1u) | ((eq >> 15) & 2u)) << (2 * q);
        }
    } else {
#pragma unroll
        for (int e = 0; e < Elem<DT>::EPC; ++e) {
            const float v = Elem<DT>::get(w, e);
            bool i, t = false;
            if (s.flags & RS_ALL_IN) {
                i = v > -INFINITY;
            } else if (s.flags & RS_LAZY) {
                const uint32_t k = fkey(v);
                t = k == vkey;
                i = k >= vkey;
            } else {
                // (padding of a partial chunk is -inf, below every cut)
                i = order_val(fkey(v), (uint32_t)(x0 + e)) >= s.cut;
            }
            in |= (uint32_t)i << e;
            tm |= (uint32_t)t << e;
        }
    }
    *tie = tm;
    return in;
}

// q of a chunk's ids (x0: the id of element 0; 0 outside the row).  vec: the
// chunk's q values are 16-byte aligned
template <int DT>
__device__ __forceinline__ void chunk_q(const ScanRow &s, int x0, bool whole, bool vec, float (&qv)[Elem<DT>::EPC]) {
    if (vec && whole) {
#pragma unroll
        for (int h = 0; h < Elem<DT>::EPC / 4; ++h) {
            const uint4 w = ldg16(s.q + x0 + 4 * h);
#pragma unroll
            for (int e = 0; e < 4; ++e) qv[4 * h + e] = Elem<ACES_F32>::get(w, e);
        }
    } else {
#pragma unroll
        for (int e = 0; e < Elem<DT>::EPC; ++e) qv[e] = x0 + e >= 0 && x0 + e < s.V ? __ldg(s.q + x0 + e) : 0.0f;
    }
}

// entry e (a run-time index) of a chunk's values
template <int N>
__device__ __forceinline__ float sel_entry(const float (&v)[N], int e) {
    const float a = (e & 1) ? v[1] : v[0], b = (e & 1) ? v[3] : v[2];
    const float lo = (e & 2) ? b : a;
    if (N == 4) return lo;
    const float c = (e & 1) ? v[N - 3] : v[N - 4], d = (e & 1) ? v[N - 1] : v[N - 2];
    return (e & 4) ? ((e & 2) ? d : c) : lo;
}
template <int DT>
__device__ __forceinline__ float chunk_at(const uint4 &w, int e) {
    if (DT == ACES_BF16) {
        const uint32_t lo = (e & 4) ? w.z : w.x, hi = (e & 4) ? w.w : w.y;
        const uint32_t wd = (e & 2) ? hi : lo;
        return __uint_as_float((e & 1) ? (wd & 0xFFFF0000u) : (wd << 16));
    }
    const uint32_t lo = (e & 2) ? w.z : w.x, hi = (e & 2) ? w.w : w.y;
    return __uint_as_float((e & 1) ? hi : lo);
}

// the mass of one member id with logit v: p in units of 2^-40 (*pf) and the
// residual max(0, p - q) likewise (return value); *bad on a NaN / negative q
// (q is read where p > 0 only: r = 0 elsewhere)
__device__ __forceinline__ unsigned long long member_mass(float v, float qx, bool has_q, const ScanRow &s,
                                                          unsigned long long *pf, int *bad) {
    const float p = ex2(fmaf(v, s.c, -s.kref)) * s.inv_S;
    float rr = p;
    if (has_q) {
        if (!(qx >= 0.0f)) *bad = 1;
        rr = fmaxf(p - qx, 0.0f);
    }
    *pf = to_fx(p);
    return to_fx(rr);
}

// The draw from a whole row by the CTA (all NTH threads; scratch: DRAW_SCRATCH
// bytes).  Returns the token, -1 when there is none, -2 on an invalid q.
template <int DT, int NTH>
__device__ __noinline__ int draw_scan(ScanRow s, unsigned char *scratch) {
    constexpr int EPC = Elem<DT>::EPC;
    constexpr int TPT = (DRAW_TASKS + NTH - 1) / NTH;  // consecutive tasks per thread (prefix sums)
    __shared__ unsigned long long red[NTH / 32];
    __shared__ unsigned long long s_need, s_base, s_tbd;
    __shared__ int s_sp, s_sd, s_tok, s_hit, s_bad;
    unsigned long long *sum_r = reinterpret_cast<unsigned long long *>(scratch);
    unsigned long long *sum_p = sum_r + DRAW_TASKS, *sum_t = sum_p + DRAW_TASKS;
    uint32_t *cnt_t = reinterpret_cast<uint32_t *>(sum_t + DRAW_TASKS);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const RowChunks<DT> rc(s.z, s.V);
    const bool qvec = s.q != nullptr && ((uintptr_t)(s.q - rc.head) & 15u) == 0;
    const bool has_q = s.q != nullptr, lazy = (s.flags & RS_LAZY) != 0;
    const int nstep = (rc.nch + 32 * DRAW_CH - 1) / (32 * DRAW_CH);
    const int spt = (nstep + DRAW_TASKS - 1) / DRAW_TASKS;  // steps per task
    const int ntask = (nstep + spt - 1) / spt;
    const int cpt = spt * 32 * DRAW_CH;                     // chunks per task
    if (tid == 0) {
        s_sp = -1;
        s_sd = -1;
        s_tok = -1;
        s_bad = 0;
        s_need = 0ull;
    }
    __syncthreads();  // (the scratch is free, the words above are set)
    // ---- sums of every task ----
    {
        const uint32_t ni = Elem<DT>::NEG_INF_WORD;
        uint4 nx[DRAW_CH];
        auto load = [&](int c0) {
#pragma unroll
            for (int i = 0; i < DRAW_CH; ++i) {
                const int c = c0 + i * 32 + lane;
                nx[i] = c < rc.nch ? rc.load(c) : make_uint4(ni, ni, ni, ni);
            }
        };
        int bad = 0;
        if (wid < ntask) load(wid * cpt);
        for (int t = wid; t < ntask; t += NTH / 32) {
            unsigned long long ar = 0ull, ap = 0ull, at = 0ull;
            uint32_t an = 0u;
            for (int st = 0; st < spt; ++st) {
                const int c0 = t * cpt + st * 32 * DRAW_CH;
                uint4 w[DRAW_CH];
#pragma unroll
                for (int i = 0; i < DRAW_CH; ++i) w[i] = nx[i];
                // (the warp's next step is loaded before this one is used)
                if (st + 1 < spt) load(c0 + 32 * DRAW_CH);
                else if (t + NTH / 32 < ntask) load((t + NTH / 32) * cpt);
#pragma unroll
                for (int g = 0; g < DRAW_CH; g += 2) {
                    uint32_t in[2], tb[2];
                    float qv[2][EPC];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int c = c0 + (g + i) * 32 + lane, x0 = c * EPC - rc.head;
                        in[i] = member_bits<DT>(w[g + i], x0, s, &tb[i]);
#pragma unroll
                        for (int e = 0; e < EPC; ++e) qv[i][e] = 0.0f;
                        if (has_q && in[i]) chunk_q<DT>(s, x0, rc.whole(c), qvec, qv[i]);
                    }
                    // the members, one per lane and step (the steps of a chunk
                    // are the most members any lane holds in it)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        uint32_t mk = in[i];
                        while (__any_sync(0xffffffffu, mk != 0u)) {
                            if (mk) {
                                const int e = __ffs(mk) - 1;
                                mk &= mk - 1u;
                                unsigned long long pf;
                                const unsigned long long rf = member_mass(
                                    chunk_at<DT>(w[g + i], e), sel_entry<EPC>(qv[i], e), has_q, s, &pf, &bad);
                                if ((tb[i] >> e) & 1u) {
                                    at += rf;
                                    ++an;
                                } else {
                                    ar += rf;
                                    ap += pf;
                                }
                            }
                        }
                    }
                }
            }
            ar = warp_sum(ar);
            ap = warp_sum(ap);
            if (lazy) {
                at = warp_sum(at);
                an = __reduce_add_sync(0xffffffffu, an);
            }
            if (lane == 0 && ACES_IN(t, DRAW_TASKS)) {
                sum_r[t] = ar;
                sum_p[t] = ap;
                sum_t[t] = at;
                cnt_t[t] = an;
            }
        }
        if (bad) s_bad = 1;
    }
    __syncthreads();
    if (s_bad) return -2;
    // one round of the id-by-id scans: this thread's chunk c (in ids)
    auto round_chunk = [&](int c, int c_hi, uint4 &w, uint32_t &in, uint32_t &tb) {
        const uint32_t ni = Elem<DT>::NEG_INF_WORD;
        w = c < c_hi ? rc.load(c) : make_uint4(ni, ni, ni, ni);
        in = member_bits<DT>(w, c * EPC - rc.head, s, &tb);
    };
    // ---- a lazy cut: the task holding the j-th id of its value, and the
    // residual of that value's first ids in it ----
    const unsigned long long j = lazy ? (unsigned long long)(uint32_t)s.cut : 0ull;
    unsigned long long tie_before = 0ull;  // ids of the cut's value before this thread's tasks
    unsigned long long partR = 0ull;
    if (lazy) {
        unsigned long long loc = 0ull, tot;
#pragma unroll
        for (int i = 0; i < TPT; ++i)
            if (tid * TPT + i < ntask) loc += cnt_t[tid * TPT + i];
        tie_before = block_exscan_n<NTH>(loc, red, &tot);
        if (tie_before < j && tie_before + loc >= j) {  // (one thread)
            unsigned long long c = tie_before;
            for (int i = 0; i < TPT && s_sp < 0; ++i) {
                const int t = tid * TPT + i;
                if (t >= ntask) break;
                if (c + cnt_t[t] >= j) {
                    s_sp = t;
                    s_need = j - c;
                }
                c += cnt_t[t];
            }
        }
        __syncthreads();
        const int sp = s_sp;
        if (sp < 0) return -1;  // (fewer ids of the cut's value than j: cannot happen)
        const unsigned long long need = s_need;
        const int c_lo = sp * cpt, c_hi = min(rc.nch, c_lo + cpt);
        unsigned long long seen = 0ull;
        for (int c0 = c_lo; c0 < c_hi && seen < need; c0 += NTH) {
            uint4 w;
            uint32_t in, tb;
            const int c = c0 + tid, x0 = c * EPC - rc.head;
            round_chunk(c, c_hi, w, in, tb);
            unsigned long long ttot;
            unsigned long long rk = seen + block_exscan_n<NTH>((unsigned long long)__popc(tb), red, &ttot);
            unsigned long long part = 0ull;
            if (tb && rk < need) {
                float qv[EPC];
#pragma unroll
                for (int e = 0; e < EPC; ++e) qv[e] = 0.0f;
                if (has_q) chunk_q<DT>(s, x0, rc.whole(c), qvec, qv);
                int bad = 0;
#pragma unroll
                for (int e = 0; e < EPC; ++e)
                    if ((tb >> e) & 1u) {
                        unsigned long long pf;
                        const unsigned long long rf = member_mass(Elem<DT>::get(w, e), qv[e], has_q, s, &pf, &bad);
                        if (rk < need) part += rf;
                        ++rk;
                    }
            }
            partR += block_reduce_n<NTH>(part, red, SumU64());
            seen += ttot;
        }
    }
    // ---- the totals and the task holding the draw ----
    const int sp = s_sp;
    const unsigned long long need = s_need;
    const unsigned long long pstar =  // the mass of one id of the cut's value (the same formula as member_mass)
        lazy ? to_fx(ex2(fmaf(fkey_inv((uint32_t)(s.cut >> 32)), s.c, -s.kref)) * s.inv_S) : 0ull;
    auto weight_r = [&](int t) {
        return sum_r[t] + (!lazy ? 0ull : (t < sp ? sum_t[t] : (t == sp ? partR : 0ull)));
    };
    auto weight_p = [&](int t) {
        return sum_p[t] + (!lazy ? 0ull : (t < sp ? cnt_t[t] : (t == sp ? need : 0ull)) * pstar);
    };
    unsigned long long lr = 0ull, lp = 0ull, R, P;
#pragma unroll
    for (int i = 0; i < TPT; ++i)
        if (tid * TPT + i < ntask) {
            lr += weight_r(tid * TPT + i);
            lp += weight_p(tid * TPT + i);
        }
    unsigned long long ex = block_exscan_n<NTH>(lr, red, &R);
    const bool mode = R == 0ull;  // p <= q everywhere: draw from p itself
    if (mode) {
        ex = block_exscan_n<NTH>(lp, red, &P);
        R = P;
        lr = lp;
    }
    if (R == 0ull) return -1;
    const unsigned long long thr = floor_u_times(s.u, R);
    if (ex <= thr && thr < ex + lr) {  // (one thread)
        unsigned long long tb = tie_before;
        for (int i = 0; i < TPT; ++i) {
            const int t = tid * TPT + i;
            if (t >= ntask) break;
            const unsigned long long wt = mode ? weight_p(t) : weight_r(t);
            if (ex + wt > thr) {
                s_sd = t;
                s_base = ex;
                s_tbd = tb;  // ids of the cut's value before this task
                break;
            }
            ex += wt;
            if (lazy) tb += cnt_t[t];
        }
    }
    if (tid == 0) s_hit = 0;
    __syncthreads();
    // ---- the draw: the smallest id whose prefix sum passes thr ----
    const int sd = s_sd;
    if (sd < 0) return -1;  // (cannot happen)
    unsigned long long base = s_base, rb = s_tbd;
    const int d_lo = sd * cpt, d_hi = min(rc.nch, d_lo + cpt);
    for (int c0 = d_lo; c0 < d_hi; c0 += NTH) {
        uint4 w;
        uint32_t in, tb;
        const int c = c0 + tid, x0 = c * EPC - rc.head;
        round_chunk(c, d_hi, w, in, tb);
        unsigned long long ttot = 0ull;
        unsigned long long rk = lazy ? rb + block_exscan_n<NTH>((unsigned long long)__popc(tb), red, &ttot) : 0ull;
        // the cut's ids of rank < j are in the nucleus
#pragma unroll
        for (int e = 0; e < EPC; ++e)
            if ((tb >> e) & 1u) {
                if (!(rk < j)) in &= ~(1u << e);
                ++rk;
            }
        float qv[EPC];
#pragma unroll
        for (int e = 0; e < EPC; ++e) qv[e] = 0.0f;
        if (has_q && !mode && in) chunk_q<DT>(s, x0, rc.whole(c), qvec, qv);
        unsigned long long wv[EPC], loc = 0ull;
        int bad = 0;
#pragma unroll
        for (int e = 0; e < EPC; ++e) {
            wv[e] = 0ull;
            if ((in >> e) & 1u) {
                unsigned long long pf;
                const unsigned long long rf = member_mass(Elem<DT>::get(w, e), qv[e], has_q && !mode, s, &pf, &bad);
                wv[e] = mode ? pf : rf;
            }
            loc += wv[e];
        }
        unsigned long long tot;
        unsigned long long cum = base + block_exscan_n<NTH>(loc, red, &tot);
        if (cum <= thr && thr < cum + loc) {
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
                cum += wv[e];
                if (cum > thr) {
                    s_tok = x0 + e;
                    break;
                }
            }
            s_hit = 1;
        }
        __syncthreads();
        if (s_hit) break;
        base += tot;
        rb += ttot;
    }
    return s_tok;
}

// floor(x * 2^40) of 0 <= x <= 1 as hi * 2^20 + lo, each in the low bits of a
// float of [2^23, 2^24): the exact value of to_fx without 64-bit shifts
__device__ __forceinline__ void to_fx_parts(float x, uint32_t &hi, uint32_t &lo) {
    const float y = __fmaf_rz(x, 1048576.0f, 8388608.0f);             // 2^23 + floor(x 2^20)
    const float f = fmaf(x, 1048576.0f, -(y - 8388608.0f));           // the rest of x 2^20, exact
    hi = __float_as_uint(y) & 0x7FFFFFu;
    lo = __float_as_uint(__fmaf_rz(f, 1048576.0f, 8388608.0f)) & 0x7FFFFFu;
}

// What a CTA of a draw's cluster shares with the others.
struct DrawPart {
    unsigned long long r, t;  // residual of its nucleus ids (a lazy cut's value aside); of that value's ids
    unsigned long long tcut;  // of that value's ids inside the nucleus (the CTA holding the cut)
    uint32_t nt;              // ids of that value
    int bad;                  // an invalid q was seen
    int pend;                 // (general kernel) a sequence this CTA completed, left to the cluster
};

// The draw of sequence b from row pi by a cluster of up to DRAW_CL CTAs (all
// threads of all of them call it; sh: this CTA's, scratch: DRAW_SCRATCH
// bytes).  Every logit of a chunk is taken whether it is a member or not,
// about 15 instructions each: the chain of loads, barriers and cluster
// exchanges is what it costs.  128 sequences of 128256 bfloat16 logits with
// nuclei of thousands of ids, the whole call: 218 us with the sums and the
// pick as two kernels of their own, 205 here; 222 with the member loops
// unrolled (first use of so much code), 294 with eight CTAs whatever the
// batch, 314 with one CTA a sequence.
template <int DT, int NTH>
__device__ __noinline__ void draw_cluster(const RowArgs &a, int b, int pi, DrawPart *sh, unsigned char *scratch) {
    namespace cg = cooperative_groups;
    constexpr int EPC = Elem<DT>::EPC, NW = NTH / 32;
    __shared__ unsigned long long red[NW], red_t[NW];
    __shared__ uint32_t red_n[NW];
    __shared__ unsigned long long s_base, s_tbase;
    __shared__ int s_task, s_ties;
    __shared__ DrawPart parts[DRAW_CL];  // every CTA's, read once
    unsigned long long *sum_r = reinterpret_cast<unsigned long long *>(scratch), *sum_t = sum_r + DRAW_TASKS;
    uint32_t *cnt_t = reinterpret_cast<uint32_t *>(sum_t + DRAW_TASKS);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), CL = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < DRAW_TASKS; i += NTH) {
        sum_r[i] = 0ull;
        sum_t[i] = 0ull;
        cnt_t[i] = 0u;
    }
    if (tid == 0) sh->bad = 0;
    __syncthreads();
    const int rp = b * (a.K + 1) + pi;
    const RowStat rs = row_stat(a.ws, rp);  // (finite: rows that are not are drawn where they finish)
    const ScanRow s = scan_row<DT>(a, b, pi, rs);
    const RowChunks<DT> rc(s.z, s.V);
    const bool qvec = s.q != nullptr && ((uintptr_t)(s.q - rc.head) & 15u) == 0;
    const bool has_q = s.q != nullptr, lazy = (s.flags & RS_LAZY) != 0;
    // this CTA's chunks: whole warp steps of 32, spt of them to a task
    const int nws = (rc.nch + 31) / 32, pw = (nws + CL - 1) / CL;
    const int spt = (pw + DRAW_TASKS - 1) / DRAW_TASKS;
    const int w_lo = min(nws, rank * pw), w_n = min(nws, w_lo + pw) - w_lo;
    const uint32_t ni = Elem<DT>::NEG_INF_WORD;
    int bad = 0;
    // One warp step of 32 chunks at a time, its logits loaded two steps and
    // its q one step ahead, in one rolled loop: a CTA visits few steps, and
    // with four of them unrolled side by side the cold instruction cache was
    // most of the sum's time (6.8 us for one step of four chunks a lane).
    auto load_z = [&](int k) {
        const int c = (w_lo + k) * 32 + lane;
        return k < w_n && c < rc.nch ? rc.load(c) : make_uint4(ni, ni, ni, ni);
    };
    auto load_q = [&](int k, uint32_t in, float (&qv)[EPC]) {
        const int c = (w_lo + k) * 32 + lane;
#pragma unroll
        for (int e = 0; e < EPC; ++e) qv[e] = 0.0f;
        if (has_q && in) chunk_q<DT>(s, c * EPC - rc.head, rc.whole(c), qvec, qv);
    };
    auto first_id = [&](int k) { return ((w_lo + k) * 32 + lane) * EPC - rc.head; };
    unsigned long long wr = 0ull, wt = 0ull;  // this warp's sums
    uint32_t wn = 0u;
    {
        uint4 z0 = load_z(wid), z1 = load_z(wid + NW);
        uint32_t tb0, in0 = member_bits<DT>(z0, first_id(wid), s, &tb0);
        float q0[EPC];
        load_q(wid, in0, q0);
#pragma unroll 1
        for (int k = wid; k < w_n; k += NW) {
            const uint4 z2 = load_z(k + 2 * NW);
            uint32_t tb1;
            const uint32_t in1 = member_bits<DT>(z1, first_id(k + NW), s, &tb1);
            float q1[EPC];
            load_q(k + NW, in1, q1);
            const uint32_t mk = in0 & ~tb0;
            uint32_t hi = 0u, lo = 0u, qmax = 0u;
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
                const float p = ex2(fmaf(Elem<DT>::get(z0, e), s.c, -s.kref)) * s.inv_S;
                const float r = (mk >> e) & 1u ? fmaxf(p - q0[e], 0.0f) : 0.0f;
                uint32_t h, l;
                to_fx_parts(r, h, l);
                hi += h;
                lo += l;
                qmax = max(qmax, __float_as_uint(q0[e]));
            }
            if (qmax > 0x7F800000u) {  // a negative or NaN q in the chunk: at a member?
                uint32_t m = in0;
                while (m) {
                    if (!(sel_entry<EPC>(q0, __ffs(m) - 1) >= 0.0f)) bad = 1;
                    m &= m - 1u;
                }
            }
            hi = __reduce_add_sync(0xffffffffu, hi);
            lo = __reduce_add_sync(0xffffffffu, lo);
            const int t = k / spt;
            const unsigned long long sum = ((unsigned long long)hi << 20) + lo;
            wr += sum;
            if (lane == 0 && ACES_IN(t, DRAW_TASKS)) {
                if (spt == 1) sum_r[t] = sum;
                else atomicAdd(&sum_r[t], sum);
            }
            if (__any_sync(0xffffffffu, tb0 != 0u)) {  // ids of a lazy cut's value
                unsigned long long at = 0ull;
                uint32_t m = tb0;
                while (m) {
                    const int e = __ffs(m) - 1;
                    m &= m - 1u;
                    unsigned long long pf;
                    at += member_mass(chunk_at<DT>(z0, e), sel_entry<EPC>(q0, e), has_q, s, &pf, &bad);
                }
                __syncwarp();
                at = warp_sum(at);
                const uint32_t nt = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(tb0));
                wt += at;
                wn += nt;
                if (lane == 0 && ACES_IN(t, DRAW_TASKS)) {
                    atomicAdd(&sum_t[t], at);
                    atomicAdd(&cnt_t[t], nt);
                }
            }
            z0 = z1;
            z1 = z2;
            in0 = in1;
            tb0 = tb1;
#pragma unroll
            for (int e = 0; e < EPC; ++e) q0[e] = q1[e];
        }
    }
    if (bad) sh->bad = 1;
    if (lane == 0) {
        red[wid] = wr;
        red_t[wid] = wt;
        red_n[wid] = wn;
    }
    __syncthreads();
    // ---- this CTA's totals; then the cluster's ----
    constexpr int TPT = (DRAW_TASKS + NTH - 1) / NTH;  // consecutive tasks per thread
    const int ntask = (w_n + spt - 1) / spt;
    if (wid == 0) {
        const unsigned long long r_ = warp_sum(lane < NW ? red[lane] : 0ull), t_ = warp_sum(lane < NW ? red_t[lane] : 0ull);
        const uint32_t n_ = __reduce_add_sync(0xffffffffu, lane < NW ? red_n[lane] : 0u);
        if (lane == 0) {
            sh->r = r_;
            sh->t = t_;
            sh->nt = n_;
            s_task = -1;
        }
    }
    // sums of this thread's tasks, and of those before them
    unsigned long long lr = 0ull, lt = 0ull, ln = 0ull, ex_r = 0ull, ex_t = 0ull, ex_n = 0ull, tot_;
#pragma unroll
    for (int i = 0; i < TPT; ++i)
        if (tid * TPT + i < ntask) {
            lr += sum_r[tid * TPT + i];
            lt += sum_t[tid * TPT + i];
            ln += cnt_t[tid * TPT + i];
        }
    cl.sync();
    // scans the task's chunks with the first warp: visits its warp steps in
    // order until f returns true (warp-uniform)
    auto scan_task = [&](int task, auto f) {
        for (int k = task * spt; k < min(w_n, (task + 1) * spt); ++k) {
            const int c = (w_lo + k) * 32 + lane, x0 = c * EPC - rc.head;
            const uint4 w = c < rc.nch ? rc.load(c) : make_uint4(ni, ni, ni, ni);
            uint32_t tb;
            const uint32_t in = member_bits<DT>(w, x0, s, &tb);
            float qv[EPC];
#pragma unroll
            for (int e = 0; e < EPC; ++e) qv[e] = 0.0f;
            if (has_q && in) chunk_q<DT>(s, x0, rc.whole(c), qvec, qv);
            if (f(w, x0, in, tb, qv)) return;
        }
    };
    auto warp_exscan = [&](unsigned long long v, unsigned long long *tot) {
        unsigned long long inc = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        *tot = __shfl_sync(0xffffffffu, inc, 31);
        return inc - v;
    };
    // ---- a lazy cut: the CTA and task holding the j-th id of its value, the
    // residual of that value's first ids ----
    const uint32_t j = lazy ? (uint32_t)s.cut : 0u;
    int cs = CL;               // the CTA holding the cut
    uint32_t nt_before = 0u;   // ids of the value in the CTAs before this one
    if (lazy) {
        uint32_t n = 0u;
        if (tid < CL) parts[tid] = *cl.map_shared_rank(sh, tid);
        __syncthreads();
        for (int c = 0; c < CL; ++c) {
            if (c == rank) nt_before = n;
            const uint32_t nt = parts[c].nt;
            if (n < j && n + nt >= j) cs = c;
            n += nt;
        }
        if (rank == cs) {
            ex_t = block_exscan_n<NTH>(lt, red, &tot_);
            ex_n = block_exscan_n<NTH>(ln, red, &tot_);
            const unsigned long long before = nt_before + ex_n;
            if (before < j && before + ln >= j) {  // (one thread)
                unsigned long long n2 = before, t2 = ex_t;
                for (int i = 0; i < TPT; ++i) {
                    const int t = tid * TPT + i;
                    if (t >= ntask) break;
                    if (n2 + cnt_t[t] >= j) {
                        s_task = t;
                        s_ties = (int)(j - n2);
                        s_tbase = t2;
                        break;
                    }
                    n2 += cnt_t[t];
                    t2 += sum_t[t];
                }
            }
            __syncthreads();
            if (wid == 0 && s_task >= 0) {
                unsigned long long seen = 0ull, acc = 0ull;
                const unsigned long long need = (unsigned long long)s_ties;
                scan_task(s_task, [&](const uint4 &w, int, uint32_t, uint32_t tb, const float (&qv)[EPC]) {
                    unsigned long long tot;
                    unsigned long long rk = seen + warp_exscan((unsigned long long)__popc(tb), &tot);
                    int bd = 0;
#pragma unroll
                    for (int e = 0; e < EPC; ++e)
                        if ((tb >> e) & 1u) {
                            unsigned long long pf;
                            const unsigned long long rf = member_mass(Elem<DT>::get(w, e), qv[e], has_q, s, &pf, &bd);
                            if (rk < need) acc += rf;
                            ++rk;
                        }
                    seen += tot;
                    return seen >= need;
                });
                acc = warp_sum(acc);
                if (lane == 0) sh->tcut = s_tbase + acc;
            }
        }
        cl.sync();
    }
    // ---- the total, and the CTA holding the draw ----
    unsigned long long R = 0ull, before_r = 0ull, own = 0ull;
    int any_bad = 0;
    if (tid < CL) parts[tid] = *cl.map_shared_rank(sh, tid);
    __syncthreads();
    for (int c = 0; c < CL; ++c) {
        const DrawPart *o = &parts[c];
        const unsigned long long wc = o->r + (!lazy ? 0ull : (c < cs ? o->t : (c == cs ? o->tcut : 0ull)));
        any_bad |= o->bad;
        if (c == rank) {
            before_r = R;
            own = wc;
        }
        R += wc;
    }
    const int cut_task = rank == cs ? s_task : -1;
    const unsigned long long cut_t = rank == cs ? sh->tcut : 0ull;
    cl.sync();  // every CTA has read the others' shares
    if (any_bad || (lazy && cs == CL)) {  // (cs == CL: fewer ids of the value than j, cannot happen)
        if (rank == 0 && tid == 0) write_draw(a, b, pi, any_bad ? -2 : -1);
        return;
    }
    if (R == 0ull) {  // p <= q everywhere: drawn from p itself
        if (rank == 0) {
            const int tok = draw_scan<DT, NTH>(s, scratch);
            if (tid == 0) write_draw(a, b, pi, tok);
        }
        return;
    }
    const unsigned long long thr = floor_u_times(s.u, R);
    if (!(before_r <= thr && thr < before_r + own)) return;  // another CTA holds it
    // weight of the ids before this thread's tasks: their residual, and that
    // of the cut's value's ids where they are in the nucleus
    const auto ties_upto = [&](int t, unsigned long long t2) -> unsigned long long {  // t2: sum_t of the tasks before t
        if (!lazy || rank > cs) return 0ull;
        if (rank < cs || t <= cut_task) return t2;
        return cut_t;
    };
    if (tid == 0) s_task = -1;
    ex_r = block_exscan_n<NTH>(lr, red, &tot_);  // (its barriers order s_task)
    if (lazy && rank != cs) {
        ex_t = block_exscan_n<NTH>(lt, red, &tot_);
        ex_n = block_exscan_n<NTH>(ln, red, &tot_);
    }
    {
        unsigned long long r2 = before_r + ex_r, t2 = ex_t;
        uint32_t n2 = nt_before + (uint32_t)ex_n;
        for (int i = 0; i < TPT; ++i) {
            const int t = tid * TPT + i;
            if (t >= ntask) break;
            const unsigned long long lo_w = r2 + ties_upto(t, t2);
            const unsigned long long hi_w = r2 + sum_r[t] + ties_upto(t + 1, t2 + sum_t[t]);
            if (lo_w <= thr && thr < hi_w) {  // (one task of one thread)
                s_task = t;
                s_base = lo_w;
                s_ties = (int)n2;
            }
            r2 += sum_r[t];
            t2 += sum_t[t];
            n2 += cnt_t[t];
        }
    }
    __syncthreads();
    // ---- the draw: the smallest id whose prefix sum passes thr ----
    if (wid == 0) {
        int tok = -1;
        unsigned long long base = s_base, seen = (unsigned long long)s_ties;
        if (s_task >= 0)
            scan_task(s_task, [&](const uint4 &w, int x0, uint32_t in, uint32_t tb, const float (&qv)[EPC]) {
                unsigned long long ttot;
                unsigned long long rk = seen + warp_exscan((unsigned long long)__popc(tb), &ttot);
                unsigned long long wv[EPC], loc = 0ull, tot;
                int bd = 0;
#pragma unroll
                for (int e = 0; e < EPC; ++e) {
                    // (the cut's ids of rank < j are in the nucleus)
                    bool is = (in >> e) & 1u;
                    if ((tb >> e) & 1u) is = rk++ < j;
                    unsigned long long pf;
                    wv[e] = is ? member_mass(Elem<DT>::get(w, e), qv[e], has_q, s, &pf, &bd) : 0ull;
                    loc += wv[e];
                }
                unsigned long long cum = base + warp_exscan(loc, &tot);
                int mine = -1;
                if (cum <= thr && thr < cum + loc) {
#pragma unroll
                    for (int e = 0; e < EPC; ++e) {
                        cum += wv[e];
                        if (mine < 0 && cum > thr) mine = x0 + e;
                    }
                }
                const unsigned bal = __ballot_sync(0xffffffffu, mine >= 0);
                if (bal) tok = __shfl_sync(0xffffffffu, mine, __ffs(bal) - 1);
                base += tot;
                seen += ttot;
                return bal != 0u;
            });
        if (lane == 0) write_draw(a, b, pi, tok);
    }
}

// The draw from row pi's stored nucleus lst (n ids in nucleus order); the ids
// are ordered by direct rank counting (one pass, no barrier stages).  All NTH
// threads call it, NTH * 2 >= NUC_CAP; scratch: DRAW_SCRATCH bytes.  Returns
// as draw_scan.
template <int NTH>
__device__ int draw_list(const ScanRow &s, const unsigned long long *lst, int n, unsigned char *scratch) {
    static_assert(2 * NTH >= NUC_CAP, "two nucleus entries per thread");
    __shared__ unsigned long long red[NTH / 32];
    __shared__ int s_tok, s_bad;
    unsigned long long *rfx = reinterpret_cast<unsigned long long *>(scratch), *pfx = rfx + NUC_CAP;
    uint32_t *inv = reinterpret_cast<uint32_t *>(pfx + NUC_CAP);  // 2^32 - 1 - id (0: none), to be counted from above
    uint32_t *srt = inv + NUC_CAP;                               // entries in ascending id order
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_bad = 0;
        s_tok = -1;
    }
    __syncthreads();
    for (int i = tid; i < ((n + 3) & ~3); i += NTH) {
        if (i >= n) {
            inv[i] = 0u;
            continue;
        }
        const unsigned long long o = lst[i];
        const uint32_t id = order_id(o);
        int bad = 0;
        const bool has_q = s.q != nullptr && ACES_IN(id, s.V);
        rfx[i] = member_mass(order_value(o), has_q ? __ldg(s.q + id) : 0.0f, has_q, s, &pfx[i], &bad);
        if (bad) s_bad = 1;
        inv[i] = 0xFFFFFFFFu - id;
    }
    __syncthreads();
    if (s_bad) return -2;
    for (int i = tid; i < n; i += NTH) {  // ascending id (ids are distinct)
        const int rank = count_above<false>(inv, n, inv[i], nullptr);
        if (ACES_IN(rank, NUC_CAP)) srt[rank] = (uint32_t)i;
    }
    __syncthreads();
    // two consecutive entries (in id order) per thread
    const int e0 = 2 * tid, e1 = 2 * tid + 1;
    int i0 = e0 < n ? (int)srt[e0] : -1;
    int i1 = e1 < n ? (int)srt[e1] : -1;
    if (i0 >= 0 && !ACES_IN(i0, NUC_CAP)) i0 = -1;
    if (i1 >= 0 && !ACES_IN(i1, NUC_CAP)) i1 = -1;
    unsigned long long w0 = i0 >= 0 ? rfx[i0] : 0ull, w1 = i1 >= 0 ? rfx[i1] : 0ull, tot;
    unsigned long long ex = block_exscan_n<NTH>(w0 + w1, red, &tot);
    if (tot == 0ull) {  // p <= q everywhere: draw from p itself
        w0 = i0 >= 0 ? pfx[i0] : 0ull;
        w1 = i1 >= 0 ? pfx[i1] : 0ull;
        ex = block_exscan_n<NTH>(w0 + w1, red, &tot);
    }
    if (tot > 0ull) {
        const unsigned long long thr = floor_u_times(s.u, tot);
        if (ex <= thr && thr < ex + w0) s_tok = (int)(0xFFFFFFFFu - inv[i0]);
        else if (ex + w0 <= thr && thr < ex + w0 + w1) s_tok = (int)(0xFFFFFFFFu - inv[i1]);
    }
    __syncthreads();
    return s_tok;
}

// Called by all threads when this CTA has written row r's outputs and state.
// The CTA that finishes the last row of a sequence draws its token when row
// pi kept its nucleus; otherwise it gets b * 32 + pi, for draw_cluster (the
// others, and those that have drawn, get -1).
template <int DT, int NTH>
__device__ int row_finished(const RowArgs &a, int r, unsigned char *scratch) {
    if (a.ws.seqcnt == nullptr) return -1;  // sparsify
    __shared__ int s_last, s_pi;
    const int b = r / (a.K + 1);
    __syncthreads();  // every thread's writes of this row are issued
    // releases this row's writes; the last row acquires the others'
    if (threadIdx.x == 0) s_last = atomic_add_acq_rel(&a.ws.seqcnt[b], 1) == a.K;
    __syncthreads();
    if (!s_last) return -1;
    if (threadIdx.x < 32) {
        const int pi0 = first_reject_warp(a.ws, b, a.K);
        if (threadIdx.x == 0) s_pi = pi0;
    }
    __syncthreads();
    const int pi = s_pi, rp = b * (a.K + 1) + pi;
    const RowStat rs = row_stat(a.ws, rp);
    int tok = -1;
    if (!(rs.flags & RS_NONFINITE)) {
        if (rs.nnuc < 0) return b * 32 + pi;
        const ScanRow s = scan_row<DT>(a, b, pi, rs);
        tok = draw_list<NTH>(s, a.ws.nuc + (size_t)rp * NUC_CAP, ACES_IN(rs.nnuc - 1, NUC_CAP) ? rs.nnuc : 0, scratch);
    }
    if (threadIdx.x == 0) write_draw(a, b, pi, tok);
    return -1;
}

}  // namespace aces
