// Exact general row kernel of the AceSpec cloud step (Sec. III-B; Sec. II-A
// modified rejection sampling; Sec. V-C payload).  It takes every row that
// the single-pass kernel hands over, and then draws the sequences whose draw
// needs a whole row.  Masses are in 2^-40 fixed point, so every partial sum
// is exact and order-independent.  One CTA of 512 threads per row; a
// persistent grid walks the list of rows handed over.
//   value histogram  (bfloat16 rows) ids counted per bfloat16 value
//                below the max, the crossing and payload values found by a
//                prefix scan, their ids collected and ranked: two row reads;
//   depth histogram  (handed float32 rows, then bfloat16) ids counted in fine
//                bins of depth, exact masses only above the crossing's range:
//                two row reads;
//   binned path  exact per-bin masses over bins of distance below the max
//                (warp-aggregated shared-memory atomics, farther elements
//                summed in registers), then the crossing bin and the payload
//                bins are collected and ordered: three to four row reads;
//   radix path   when a needed bin is too full or too far: exact radix
//                selection over the 64-bit order value
//                O = key(z) << 32 | (2^32 - 1 - id), 8 bits per pass.
#include <climits>
#include <cstddef>
#include <type_traits>

#include <cuda_bf16.h>

#define ACES_FILE 10  // site numbers of the checked build
#include "draw.cuh"

namespace aces {

// ---------------------------------------------------------------------------
// Row epilogue shared by both row kernels: payload, tail, accept test, stats.
// `sorted` holds the first L ids of the nucleus in order (descending order
// values).  Called by all threads of the CTA.
template <int DT>
__device__ void finish_row(const RowArgs &a, int r, const char *row, float kref, double S_nuc,
                           unsigned long long cut, int flags, const unsigned long long *sorted,
                           int L, double *redd) {
    const int tid = threadIdx.x;
    // same formulas as the single-pass row kernel, so a cut and a nucleus mass
    // give the same bits in both: p = e * inv_mass(S_nuc), and the tail from
    // the exact fixed-point sum of the payload masses
    const float inv_S = inv_mass(S_nuc);
    unsigned long long loc = 0ull;
    if (a.k > 0) {
        for (int j = tid; j < a.k; j += NT) {
            size_t o = (size_t)r * a.k + j;
            if (j < L) {
                unsigned long long ov = sorted[j];
                float e = ex2(fmaf(order_value(ov), a.c, -kref));
                loc += to_fx(e);
                a.topk_ids[o] = (int32_t)order_id(ov);
                a.topk_probs[o] = e * inv_S;
            } else {
                a.topk_ids[o] = -1;
                a.topk_probs[o] = 0.0f;
            }
        }
    }
    __shared__ unsigned long long s_redl[NWARP];
    const unsigned long long tot = block_reduce(loc, s_redl, SumU64());
    if (tid != 0) return;
    if (a.k > 0) a.tail[r] = (float)(S_nuc - (double)tot * FX_INV) * inv_S;
    int st = 0;
    if (a.K > 0) {
        int b = r / (a.K + 1), i = r % (a.K + 1);
        if (i < a.K) {
            int x = a.xt[(size_t)b * a.K + i];
            int accept = 0;
            if (x < 0 || x >= a.V) {
                st |= ACES_ROW_BAD_Q;
            } else {
                float v = Elem<DT>::load1(row, x);
                bool in = (flags & RS_ALL_IN) ? (v > -INFINITY) : (order_val(fkey(v), (uint32_t)x) >= cut);
                const float e = in ? ex2(fmaf(v, a.c, -kref)) : 0.0f;
                float qx = a.q[((size_t)b * a.K + i) * a.V + x];
                if (!(qx > 0.0f)) st |= ACES_ROW_BAD_Q;
                else accept = accept_test(a.u[(size_t)b * (a.K + 1) + i], qx, e, S_nuc);
            }
            a.ws.acc[(size_t)b * a.K + i] = accept;
        }
    }
    a.row_status[r] = st;
    RowStat s;
    s.kref = kref;
    s.c = a.c;
    s.S_nuc = S_nuc;
    s.cut = cut;
    s.flags = flags;
    s.nnuc = -1;  // the residual step scans the row
    a.ws.stats[r] = s;
}

// ---------------------------------------------------------------------------
// General path: exact radix selection over the 64-bit order value
// O = key(z) << 32 | (2^32 - 1 - id), 8 bits per pass, masses in 2^-40
// fixed point so that every partial sum is exact and order-independent.
template <int DT, class F>
__device__ __forceinline__ void for_each_elem(const RowChunks<DT> &rc, F f) {
    constexpr int EPC = Elem<DT>::EPC;
#pragma unroll 2
    for (int c = threadIdx.x; c < rc.nch; c += NT) {
        const uint4 w = rc.load(c);
#pragma unroll
        for (int e = 0; e < EPC; ++e) f(c * EPC + e - rc.head, Elem<DT>::get(w, e));  // (-inf outside the row)
    }
}

// Warp-uniform walk over the row: every lane of a warp takes part in every
// round (f gets valid = false outside the row), so f may use warp collectives.
template <int DT, class F>
__device__ __forceinline__ void for_each_elem_warp(const RowChunks<DT> &rc, F f) {
    constexpr int EPC = Elem<DT>::EPC;
    for (int c0 = threadIdx.x & ~31; c0 < rc.nch; c0 += NT) {
        const int c = c0 + (threadIdx.x & 31);
        const bool in = c < rc.nch;
        const uint4 w = in ? rc.load(c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int e = 0; e < EPC; ++e) {
            const int x = c * EPC + e - rc.head;
            f(in && x >= 0 && x < rc.V, x, Elem<DT>::get(w, e));
        }
    }
}

// cnt[d] += 1 and mass[d] += m for every lane with ok; a warp whose lanes
// all hit one bin (the common case in the first digits, where the logits
// share their leading key bits) adds its totals with one atomic each
__device__ __forceinline__ void hist_add(uint32_t *cnt, unsigned long long *mass, bool ok, int d,
                                         unsigned long long m, bool with_mass) {
    const unsigned act = __ballot_sync(0xffffffffu, ok);
    if (act == 0u) return;
    const int d0 = __shfl_sync(0xffffffffu, d, __ffs(act) - 1);
    if (__all_sync(0xffffffffu, !ok || d == d0)) {
        const unsigned long long ms = with_mass ? warp_sum(ok ? m : 0ull) : 0ull;
        if ((threadIdx.x & 31) == 0 && ACES_IN(d0, 256)) {
            atomicAdd(&cnt[d0], (uint32_t)__popc(act));
            if (with_mass) atomicAdd(&mass[d0], ms);
        }
    } else if (ok && ACES_IN(d, 256)) {
        atomicAdd(&cnt[d], 1u);
        if (with_mass) atomicAdd(&mass[d], m);
    }
}

struct SelState {
    uint32_t cnt[256];
    unsigned long long mass[256];
    unsigned long long prefix;
    unsigned long long above;
    unsigned long long S_fx;
    unsigned long long found;
    unsigned above_cnt;
    int sel;
    unsigned sel_cnt;
    int done;
};

// One radix selection.  mode 0: first id where the cumulative mass reaches
// ceil(top_p * S); mode 1: the kk-th id (1-based) by count.
// Returns the order value of the selected id; st->above / above_cnt hold the
// mass / count strictly before it; when want_S, st->S_fx gets the total mass.
template <int DT>
__device__ unsigned long long radix_select(const RowChunks<DT> &rc, float kref, float c, int mode,
                                           double top_p, unsigned kk, bool want_S, SelState *st) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        st->prefix = 0ull;
        st->above = 0ull;
        st->above_cnt = 0u;
        st->done = 0;
        st->S_fx = 0ull;
    }
    unsigned long long target = 0ull;  // (thread 0)
    int nbits = 0;
    for (int s = 56; s >= 0; s -= 8) {
        // digits known in advance: the low 16 key bits of a bf16 value are 0,
        // and ids below 2^24 give 0xFF in bits 31..24 of (2^32 - 1 - id)
        int known = -1;
        if (DT == ACES_BF16 && (s == 40 || s == 32)) known = 0;
        if (s == 24) known = 0xFF;
        if (known >= 0) {
            if (tid == 0) st->prefix = (st->prefix << 8) | (unsigned long long)known;
            nbits += 8;
            __syncthreads();
            continue;
        }
        for (int i = tid; i < 256; i += NT) {
            st->cnt[i] = 0u;
            st->mass[i] = 0ull;
        }
        __syncthreads();
        const unsigned long long prefix = st->prefix;
        const int sh = 64 - nbits;
        const bool with_mass = mode == 0 || want_S;
        for_each_elem_warp<DT>(rc, [&](bool in, int x, float v) {
            const unsigned long long o = order_val(fkey(v), (uint32_t)x);
            const bool ok = in && v > -INFINITY && (nbits == 0 || (o >> sh) == prefix);
            const int d = (int)((o >> s) & 255ull);
            const unsigned long long m = (ok && with_mass) ? to_fx(ex2(fmaf(v, c, -kref))) : 0ull;
            hist_add(st->cnt, st->mass, ok, d, m, with_mass);
        });
        __syncthreads();
        if (tid == 0) {
            if (nbits == 0) {
                unsigned long long S = 0ull;
                for (int d = 0; d < 256; ++d) S += st->mass[d];
                st->S_fx = S;
                if (mode == 0) target = (unsigned long long)ceil(top_p * (double)S);
            }
            int sel = -1;
            int lowest = -1;
            for (int d = 255; d >= 0; --d) {
                if (st->cnt[d] == 0u) continue;
                lowest = d;
                bool hit = mode == 0 ? (st->above + st->mass[d] >= target)
                                     : (st->above_cnt + st->cnt[d] >= kk);
                if (hit) {
                    sel = d;
                    break;
                }
                st->above += st->mass[d];
                st->above_cnt += st->cnt[d];
            }
            if (sel < 0) {  // target not reached (rounding at top_p ~ 1): take the last id
                sel = lowest;
                st->above -= st->mass[sel];
                st->above_cnt -= st->cnt[sel];
            }
            st->sel = sel;
            st->sel_cnt = st->cnt[sel];
            st->prefix = (st->prefix << 8) | (unsigned long long)sel;
            if (mode == 0) st->found = st->mass[sel];  // mass of the bin (of the id when unique)
        }
        __syncthreads();
        nbits += 8;
        if (st->sel_cnt == 1u && s > 0) {
            // a single id carries this prefix: fetch its full order value
            const unsigned long long pf = st->prefix;
            const int sh2 = 64 - nbits;
            for_each_elem<DT>(rc, [&](int x, float v) {
                if (!(v > -INFINITY)) return;
                unsigned long long o = order_val(fkey(v), (uint32_t)x);
                if ((o >> sh2) == pf) st->prefix = o;
            });
            __syncthreads();
            break;
        }
    }
    return st->prefix;
}

// ---------------------------------------------------------------------------
// Binned exact selection.  Elements are binned by their distance below the
// row max, d = (m - z) * inv_w (width T/8, bin 255 = everything farther),
// with exact fixed-point masses per bin.  Bins are ordered by value, so the
// nucleus crossing lies in the first bin whose cumulative mass reaches the
// target, and the first k nucleus ids in the bins up to the one where the
// cumulative count reaches k.  Those bins' elements are collected (at most
// GB_CAP each) and ordered in shared memory.  Returns false, having
// written nothing, when a needed bin is the far bin or too full; the radix
// selection then finishes the row.
constexpr int GB_CAP = 2048;

constexpr int GB_WIN = 96;  // bins of the first pass (12 temperatures below the max)

struct BinState {
    uint32_t cnt[NBIN];              // counts of every bin seen so far
    unsigned long long mass[NBIN];   // masses of the current window's bins
    unsigned long long S_fx;         // total mass of the row
    unsigned long long xs[GB_CAP];  // order values of the crossing bin
    unsigned long long ps[GB_CAP];  // order values of the payload bins
    int nx, np_, bx, bk, ok, nbelow;
    unsigned long long above;       // mass of the bins before the crossing bin
    unsigned long long target;      // the nucleus target, ceil(top_p * S_fx)
};

// appends o to arr[*n] for every lane with take (one atomic per warp)
__device__ __forceinline__ void warp_append(unsigned long long *arr, int *n, bool take, unsigned long long o) {
    const unsigned bal = __ballot_sync(0xffffffffu, take);
    if (bal == 0u) return;
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == __ffs(bal) - 1) base = atomicAdd(n, __popc(bal));
    base = __shfl_sync(0xffffffffu, base, __ffs(bal) - 1);
    const int pos = base + __popc(bal & ((1u << lane) - 1u));
    if (take && pos < GB_CAP) arr[pos] = o;
}

template <int DT>
__device__ bool binned_row(const RowArgs &a, int r, const RowChunks<DT> &rc, float m, float kref,
                           unsigned long long n_fin, BinState *bs, unsigned long long *buf, double *redd,
                           unsigned long long *redu) {
    const int tid = threadIdx.x;
    const char *row = rc.row();
    const bool all_in = a.top_p >= 1.0f;
    // Two windows: the first pass histograms the GB_WIN bins nearest the max
    // with shared-memory atomics and only sums the farther elements in
    // registers, so most elements of a peaked row cost no atomic; a second
    // pass over the remaining bins runs only when the crossing (or the k-th
    // id) lies farther out.
    if (tid == 0) {
        bs->nx = 0;
        bs->np_ = 0;
        bs->above = 0ull;
        bs->nbelow = 0;
        bs->bx = -2;  // crossing bin, -2 while unknown
        bs->bk = -2;  // last payload bin, -2 while unknown
        bs->ok = 1;
    }
    for (int i = tid; i < NBIN; i += NT) bs->cnt[i] = 0u;
    for (int W = 0; W < NBIN - 1; W = W == 0 ? GB_WIN : NBIN - 1) {
        const int WN = W == 0 ? GB_WIN : NBIN - 1 - W;  // bins of this window
        for (int i = tid; i < WN; i += NT) bs->mass[i] = 0ull;
        __syncthreads();
        unsigned long long far_cnt = 0ull, far_mass = 0ull;
        for_each_elem_warp<DT>(rc, [&](bool in, int, float v) {
            const bool fin = in && v > -INFINITY;
            const float dd = (m - v) * a.inv_w;
            const int d = dd < (float)(NBIN - 1) ? (int)dd : NBIN - 1;
            const bool near = fin && d >= W && d < W + WN && d < NBIN - 1;
            unsigned long long mf = 0ull;
            if (fin && d >= W) mf = to_fx(ex2(fmaf(v, a.c, -kref)));
            if (fin && d >= W && !near) {
                far_cnt += 1ull;
                far_mass += mf;
            }
            hist_add(bs->cnt + W, bs->mass, near, d - W, mf, true);
        });
        far_cnt = block_reduce(far_cnt, redu, SumU64());
        far_mass = block_reduce(far_mass, redu, SumU64());
        if (tid == 0) {
            if (W == 0) {  // the first window sees every element: the total
                unsigned long long S = far_mass;
                for (int j = 0; j < WN; ++j) S += bs->mass[j];
                bs->target = (unsigned long long)ceil((double)a.top_p * (double)S);
                bs->S_fx = S;
            }
            unsigned long long above = bs->above;
            int nbelow = bs->nbelow;
            const int wend = W + WN;
            if (!all_in && bs->bx == -2) {
                for (int d = W; d < wend; ++d) {
                    if (above + bs->mass[d - W] >= bs->target) {
                        bs->bx = d;
                        break;
                    }
                    above += bs->mass[d - W];
                    nbelow += (int)bs->cnt[d];
                }
                bs->above = above;
                bs->nbelow = nbelow;
            }
            // once the nucleus size is bounded, the payload needs min(k, it) ids
            const bool bx_known = all_in || bs->bx >= 0;
            if (bx_known && bs->bk == -2) {
                const long long nnuc_max = all_in ? (long long)n_fin : (long long)bs->nbelow + bs->cnt[bs->bx];
                const long long want = a.k < nnuc_max ? a.k : nnuc_max;
                long long c = 0;
                bs->bk = -1;  // k = 0: no payload
                for (int d = 0; d < wend && want > 0; ++d) {
                    c += bs->cnt[d];
                    if (c >= want) {
                        bs->bk = d;
                        break;
                    }
                }
                if (want > 0 && bs->bk < 0) bs->bk = -2;  // farther than this window
                if (bs->bk >= 0 && c > GB_CAP) bs->ok = 0;
            }
            if (bs->bx >= 0 && bs->cnt[bs->bx] > (uint32_t)GB_CAP) bs->ok = 0;
        }
        __syncthreads();
        if (!bs->ok) return false;
        if ((all_in || bs->bx >= 0) && bs->bk != -2) break;
    }
    if ((!all_in && bs->bx < 0) || bs->bk == -2) return false;  // beyond the binned range
    if (tid == 0 && all_in) bs->bx = -1;
    __syncthreads();
    const int bx = bs->bx, bk = bs->bk;
    // collect the crossing bin and the payload bins
    for_each_elem_warp<DT>(rc, [&](bool in, int x, float v) {
        const bool fin = in && v > -INFINITY;
        const float dd = (m - v) * a.inv_w;
        const int d = dd < (float)(NBIN - 1) ? (int)dd : NBIN - 1;
        const unsigned long long o = order_val(fkey(v), (uint32_t)x);
        warp_append(bs->xs, &bs->nx, fin && d == bx, o);
        warp_append(bs->ps, &bs->np_, fin && d <= bk, o);
    });
    __syncthreads();
    const int nx = bs->nx, npl = bs->np_;
    // the payload bins' ids ranked by direct counting (order values are
    // distinct): the first min(npl, k) ranks go straight to buf
    const int lp = npl < a.k ? npl : a.k;
    for (int i = tid; i < npl; i += NT) {
        const unsigned long long key = bs->ps[i];
        int rank = 0;
#pragma unroll 4
        for (int t = 0; t < npl; ++t) rank += bs->ps[t] > key;
        if (rank < lp && ACES_IN(rank, ACES_MAX_TOPK)) buf[rank] = key;
    }
    // the crossing bin in order (descending order value)
    {
        const int p2 = next_pow2(nx < 2 ? 2 : nx);
        for (int i = nx + tid; i < p2; i += NT) bs->xs[i] = 0ull;
        __syncthreads();
        if (bx >= 0) bitonic_sort_desc(bs->xs, p2);
    }
    // the crossing id: the first id of the crossing bin where the cumulative
    // mass reaches the target (the bin's last id if rounding keeps it short);
    // its masses go to ps (free now) and a block scan finds it
    double S_nuc;
    unsigned long long cut = 0ull;
    long long n_nuc;
    if (bx >= 0) {
        for (int i = tid; i < nx; i += NT) bs->ps[i] = to_fx(ex2(fmaf(order_value(bs->xs[i]), a.c, -kref)));
        if (tid == 0) bs->bk = -1;  // reuse: the crossing position, -1 until found
        __syncthreads();
        const int per = (nx + NT - 1) / NT;
        const int lo = tid * per < nx ? tid * per : nx, hi = lo + per < nx ? lo + per : nx;
        unsigned long long loc = 0ull;
        for (int i = lo; i < hi; ++i) loc += bs->ps[i];
        unsigned long long tot;
        unsigned long long cum = bs->above + block_exscan_n<NT>(loc, redu, &tot);
        for (int i = lo; i < hi; ++i) {
            const unsigned long long prev = cum;
            cum += bs->ps[i];
            if (prev < bs->target && cum >= bs->target) {  // one id crosses
                bs->bk = i;
                redd[0] = (double)cum * FX_INV;
            }
        }
        __syncthreads();
        int ix = bs->bk;
        if (ix < 0) {  // rounding: the bin's last id
            ix = nx - 1;
            if (tid == 0) redd[1] = (double)(bs->above + tot) * FX_INV;
            __syncthreads();
            S_nuc = redd[1];
        } else {
            S_nuc = redd[0];
        }
        cut = ACES_IN(ix, GB_CAP) ? bs->xs[ix] : 0ull;
        n_nuc = (long long)bs->nbelow + ix + 1;
    } else {
        S_nuc = (double)bs->S_fx * FX_INV;
        n_nuc = (long long)n_fin;
    }
    int L = (int)(n_nuc < (long long)a.k ? n_nuc : (long long)a.k);
    if (L > lp) L = lp;
    __syncthreads();
    finish_row<DT>(a, r, row, kref, S_nuc, cut, all_in ? RS_ALL_IN : 0, buf, L, redd);
    return true;
}

// ---------------------------------------------------------------------------
// Value-histogram path for bfloat16 rows.  A bfloat16 logit takes one of
// 65536 values, and equal values have equal masses, so counting the elements
// of each value is enough: the values of a window below the row max (at most
// VH_W of them) get a count, one shared-memory atomic per element and no
// per-element mass.  The exp-sum S of the whole row comes with the row, from
// the row kernel.  A prefix scan over the values then gives,
// exactly in 2^-40 fixed point (count x the value's mass), the value holding
// the nucleus crossing (first prefix reaching ceil(top_p * S * 2^40)) and the
// value holding the k-th payload id; the elements of those values (ties are
// taken in id order, which is the order-value order) are collected and ranked
// in shared memory.  Declines, having written nothing, when a needed value lies
// below the window (VH_BELOW: the depth histogram then takes the row) or when a
// set to collect exceeds VH_CAP (VH_FULL, where the depth histogram's lists
// would not hold it either: the binned path does).
enum { VH_DONE, VH_BELOW, VH_FULL };
constexpr int VH_W = 4096;    // values below the max with a count
constexpr int VH_CAP = 1024;  // collected ids per set (payload values, crossing value)
constexpr int DH_XCAP = 1536; // depth histogram: listed ids around the crossing
constexpr int DH_PCAP = 768;  // listed ids of the payload's bins
static_assert(DH_PCAP <= VH_CAP, "a payload set too large for the value histogram is too large for the depth histogram");
constexpr int VH_U = 4;       // 16-byte loads per thread in flight in the counting pass

struct ValHist {
    uint32_t cnt[VH_W];                // elements of value key16(max) - d
    unsigned long long pay[VH_CAP];    // order values of the payload values
    unsigned long long tie[VH_CAP];    // order values of the crossing value
    int npay, ntie;
    int dstar, dk, j;                  // crossing value, last payload value, ids of dstar in the nucleus
    unsigned long long above, cnt_above, npay_need;
    unsigned long long above_cut;      // the cut: order value of the crossing value's j-th id
};

// 16-bit order key of a bfloat16 value: 0x8000 plus the value's signed
// magnitude, so keys sort like values and -0 and +0 share one key (-inf has
// 0x80, the finite values 0x81..0xFF7F); and the value of a key
__device__ __forceinline__ uint32_t bkey16(uint32_t b) {
    const uint32_t mag = b & 0x7FFFu;
    return (b & 0x8000u) ? 0x8000u - mag : 0x8000u + mag;
}
__device__ __forceinline__ float bval16(uint32_t k) {
    const uint32_t b = k >= 0x8000u ? k - 0x8000u : (0x8000u | (0x8000u - k));
    return __uint_as_float(b << 16);
}

// appends o to arr[*n] for every lane with take (one atomic per warp); *n
// may pass cap, entries beyond it are dropped
__device__ __forceinline__ void warp_append_cap(unsigned long long *arr, int *n, bool take, unsigned long long o,
                                                int cap) {
    const unsigned bal = __ballot_sync(0xffffffffu, take);
    if (bal == 0u) return;
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == __ffs(bal) - 1) base = atomicAdd(n, __popc(bal));
    base = __shfl_sync(0xffffffffu, base, __ffs(bal) - 1);
    const int pos = base + __popc(bal & ((1u << lane) - 1u));
    if (take && pos < cap) arr[pos] = o;
}

// (bfloat16 rows; all threads of the CTA)
// S: the row's exp-sum in units of 2^kref.  *n_fin_out gets the row's count of
// finite ids when top_p = 1 (its only use), even when the row is declined.
__device__ int valhist_row(const RowArgs &a, int r, const RowChunks<ACES_BF16> &rc, float m, float kref, double S,
                            unsigned long long *n_fin_out, ValHist *vh, unsigned long long *buf, double *redd,
                            unsigned long long *redu) {
    using E = Elem<ACES_BF16>;
    const int tid = threadIdx.x, lane = tid & 31;
    const bool all_in = a.top_p >= 1.0f;
    const char *row = rc.row();
    const uint32_t km = bkey16(__float_as_uint(m) >> 16);  // m is a bfloat16 value
    for (int i = tid; i < VH_W; i += NT) vh->cnt[i] = 0u;
    if (tid == 0) {
        vh->npay = 0;
        vh->ntie = 0;
        vh->dstar = all_in ? -1 : -2;  // -2: not (yet) found in the window
        vh->dk = -2;
    }
    // the window: values km - d for d <= D (never -inf, whose key is 0x80)
    uint32_t D = km - 0x81u < (uint32_t)(VH_W - 1) ? km - 0x81u : (uint32_t)(VH_W - 1);
    if (!all_in) {
        // Every id below a value of mass e_lo = (1 - top_p) S / (16 V) has
        // less mass than that, so all of them together hold less than a
        // sixteenth of the mass outside the nucleus and the crossing lies at
        // or above that value; an id whose fixed-point mass is 0 (below
        // 2^-40) is never needed either.  D is the last value reaching it.
        const float g = fmaxf(log2f((1.0f - a.top_p) * (float)S / (16.0f * (float)a.V)), -41.0f);
        const float vt = (kref + g) / a.c;
        uint32_t lo = 0u, hi = D;  // bval16(km) = m >= vt
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1u) >> 1;
            if (bval16(km - mid) >= vt) lo = mid;
            else hi = mid - 1u;
        }
        D = lo;
    }
    __syncthreads();
    // ---- pass 1: counts per value (top_p = 1: and of the finite ids) ----
    unsigned long long nfin = 0ull;
    const int nch = rc.nch;
    // (-inf words outside the row count nowhere)
    auto count_pass = [&](auto with_nfin) {
        constexpr bool WN = decltype(with_nfin)::value;
        for (int c0 = tid; c0 < nch; c0 += VH_U * NT) {
            uint4 wu[VH_U];
#pragma unroll
            for (int u = 0; u < VH_U; ++u) {
                const int cc = c0 + u * NT;
                wu[u] = cc < nch ? rc.load(cc) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
            }
            uint32_t nf = 0u;
#pragma unroll
            for (int u = 0; u < VH_U; ++u) {
                const uint32_t wd[4] = {wu[u].x, wu[u].y, wu[u].z, wu[u].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t b = h ? (wd[q] >> 16) : (wd[q] & 0xFFFFu);
                        if (WN) nf += b != 0xFF80u;
                        const uint32_t d = km - bkey16(b);
                        if (d <= D && ACES_IN(d, VH_W)) atomicAdd(&vh->cnt[d], 1u);
                    }
                }
            }
            if (WN) nfin += nf;
        }
    };
    if (all_in) count_pass(std::true_type());
    else count_pass(std::false_type());
    const unsigned long long n_fin = block_reduce(nfin, redu, SumU64());  // (its barriers order the counts)
    *n_fin_out = n_fin;
    const unsigned long long tg = all_in ? 0ull : (unsigned long long)ceil((double)a.top_p * S * (double)FX_SCALE);
    // ---- prefix scan over the values, PER consecutive values per thread ----
    constexpr int PER = VH_W / NT;
    static_assert(VH_W % NT == 0, "whole values per thread");
    const int d0 = tid * PER;
    // the mass of the c ids of value km - d (exact: c equal fixed-point masses)
    auto bin_mass = [&](int d, uint32_t c) -> unsigned long long {
        return c ? (unsigned long long)c * to_fx(ex2(fmaf(bval16(km - (uint32_t)d), a.c, -kref))) : 0ull;
    };
    unsigned long long bm_loc = 0ull, bc_loc = 0ull;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint32_t c = vh->cnt[d0 + i];
        bm_loc += bin_mass(d0 + i, c);
        bc_loc += c;
    }
    unsigned long long m_tot, c_tot;
    const unsigned long long m_ex = block_exscan_n<NT>(bm_loc, redu, &m_tot);
    const unsigned long long c_ex = block_exscan_n<NT>(bc_loc, redu, &c_tot);
    if (!all_in) {  // the value whose masses cross tg (at most one thread finds it)
        unsigned long long cm = m_ex, cc = c_ex;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const uint32_t c = vh->cnt[d0 + i];
            const unsigned long long bm = bin_mass(d0 + i, c);
            if (bm > 0ull && cm < tg && cm + bm >= tg) {
                const unsigned long long e = bm / c;  // one id's mass
                vh->dstar = d0 + i;
                vh->above = cm;
                vh->cnt_above = cc;
                vh->j = (int)((tg - cm + e - 1) / e);  // ids of this value in the nucleus
            }
            cm += bm;
            cc += c;
        }
    }
    __syncthreads();
    if (vh->dstar == -2) return VH_BELOW;  // the crossing lies below the window
    const unsigned long long n_nuc = all_in ? n_fin : vh->cnt_above + (unsigned long long)vh->j;
    const int L = (int)(n_nuc < (unsigned long long)a.k ? n_nuc : (unsigned long long)a.k);
    if (L > 0) {  // the value holding the L-th id (at most one thread finds it)
        unsigned long long cc = c_ex;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const unsigned long long c = vh->cnt[d0 + i];
            if (cc < (unsigned long long)L && cc + c >= (unsigned long long)L) {
                vh->dk = d0 + i;
                vh->npay_need = cc + c;  // ids of the values up to it
            }
            cc += c;
        }
    } else if (tid == 0) {
        vh->dk = -1;  // no payload
    }
    __syncthreads();
    const int dstar = vh->dstar, dk = vh->dk;
    if (dk == -2) return VH_BELOW;  // the L-th id lies below the window
    if (dk >= 0 && vh->npay_need > (unsigned long long)VH_CAP) return VH_FULL;
    if (dstar >= 0 && vh->cnt[dstar] > (uint32_t)VH_CAP) return vh->cnt[dstar] > (uint32_t)DH_XCAP ? VH_FULL : VH_BELOW;
    // ---- collect every id of the values up to dk, and those of dstar ----
    // A packed bfloat16 compare per pair of ids (value >= that of dk, or
    // == that of dstar: IEEE order, where -0 == +0 as in the keys) lets a
    // warp skip a round in which no id of its 32 chunks is wanted.
    const float vk = dk >= 0 ? bval16(km - (uint32_t)dk) : INFINITY;
    const float vs = dstar >= 0 ? bval16(km - (uint32_t)dstar) : NAN;
    const __nv_bfloat162 vk2 = __floats2bfloat162_rn(vk, vk), vs2 = __floats2bfloat162_rn(vs, vs);
    // (the next round's chunk is loaded before this round's ids are examined)
    uint4 pw = tid < nch ? rc.load(tid) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
    for (int c0 = tid & ~31; c0 < nch; c0 += NT) {  // warp-uniform rounds
        const int c = c0 + lane;
        const bool in = c < nch;
        const uint4 w = pw;
        pw = c + NT < nch ? rc.load(c + NT) : make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
        const uint32_t wd[4] = {w.x, w.y, w.z, w.w};
        uint32_t hm = 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162 *>(&wd[q]);
            hm |= __hge2_mask(x, vk2) | __heq2_mask(x, vs2);
        }
        if (!__any_sync(0xffffffffu, hm != 0u)) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t b = h ? (wd[q] >> 16) : (wd[q] & 0xFFFFu);
                const uint32_t d = km - bkey16(b);
                const bool fin = in && b != 0xFF80u;
                const bool tp = fin && dk >= 0 && d <= (uint32_t)dk;
                const bool tt = fin && dstar >= 0 && d == (uint32_t)dstar;
                if (!__any_sync(0xffffffffu, tp || tt)) continue;
                const unsigned long long o =
                    order_val(fkey(__uint_as_float(b << 16)), (uint32_t)(c * E::EPC + 2 * q + h - rc.head));
                warp_append_cap(vh->pay, &vh->npay, tp, o, VH_CAP);
                warp_append_cap(vh->tie, &vh->ntie, tt, o, VH_CAP);
            }
        }
    }
    __syncthreads();
    const int npay = vh->npay, ntie = vh->ntie;
    // ---- rank by direct counting (order values are distinct; descending
    // order, ties by ascending id): the first L payload ids go straight to
    // buf, and the cut is the crossing value's id of rank j - 1 ----
    const int LL = L < npay ? L : npay;
    for (int i = tid; i < npay; i += NT) {
        const unsigned long long key = vh->pay[i];
        int rank = 0;
#pragma unroll 4
        for (int t = 0; t < npay; ++t) rank += vh->pay[t] > key;
        if (rank < LL && ACES_IN(rank, ACES_MAX_TOPK)) buf[rank] = key;
    }
    const int jt = dstar >= 0 ? vh->j - 1 : -1;
    for (int i = tid; i < ntie; i += NT) {
        const unsigned long long key = vh->tie[i];
        int rank = 0;
#pragma unroll 4
        for (int t = 0; t < ntie; ++t) rank += vh->tie[t] > key;
        if (rank == jt) vh->above_cut = key;
    }
    __syncthreads();
    double S_nuc = S;
    unsigned long long cut = 0ull;
    if (dstar >= 0) {
        cut = vh->above_cut;
        const unsigned long long ed = to_fx(ex2(fmaf(bval16(km - (uint32_t)dstar), a.c, -kref)));
        S_nuc = (double)(vh->above + (unsigned long long)vh->j * ed) * FX_INV;
    }
    if (tid == 0) atomicAdd(&a.ws.fb_count[6], 1);
    finish_row<ACES_BF16>(a, r, row, kref, S_nuc, cut, all_in ? RS_ALL_IN : 0, buf, LL, redd);
    return VH_DONE;
}

// ---------------------------------------------------------------------------
// Depth-histogram path (the row's max m and exp-sum S_in are known):
// the float32 counterpart of the value histogram, and the second try for
// bfloat16.  One read counts the ids in DH_W equal bins of depth below the
// max, down to a value the crossing cannot lie below (top_p = 1: to where an
// id's mass is below 2^-41), and sums the row's 2^-40 masses; a bin's ids each
// carry at least its lower and at most its upper edge's mass, so bounds of the cumulative mass give a first
// and a last bin between which the crossing lies (about 0.5% of the mass apart
// with bins of T / 200).  A second read sums the exact 2^-40 masses of the ids
// above that range and lists those inside it and the payload's; the ordered
// list gives the crossing id.  Returns false, having written nothing, when a
// list would be too long (known after the first read) or the payload ends below
// the bins; the binned path then takes the row (it sums a 64-bit mass per id with shared-memory atomics).  256
// rows of 128256 float32 logits, about 200 of them handed over: 297 us a call
// with the binned path, 158 with this one, 147 with the second read's work
// done per hit and fewer rows handed over, 153 with the row's exact mass summed
// in the first read (as the binned path does; with the row kernel's float32 sum
// 117 of 46080 rows were cut one id away from float64, 34 with the exact one;
// 157 since the row kernel reads the rows it finishes again where the cut
// depends on that sum's error).
// What is left is two more reads of those rows by one CTA each.
constexpr int DH_W = 4096;    // bins
constexpr int DH_PAD = 32;    // counters of the ids below them, one per lane
constexpr int DH_U = 4;       // 16-byte loads in flight per thread

struct DepthHist {
    union {
        uint32_t cnt[DH_W + DH_PAD];
        struct {  // (once the counts are read)
            unsigned long long xs[2048];  // (a power of two for the sort)
        };
    };
    unsigned long long ps[DH_PCAP];
    alignas(16) unsigned long long fx[DH_XCAP];  // masses of the ordered crossing list
    float wu[NWARP], wl[NWARP];
    uint32_t wc[NWARP];
    int b_hi, b_lo, b_k, nx, np;
    uint32_t above_cnt;
    unsigned long long above;
    int ix;
    unsigned long long cum;
};
static_assert(offsetof(DepthHist, fx) % 16 == 0, "the payload's 32-bit keys are read 16 bytes at a time");

template <int DT>
__device__ bool depth_row(const RowArgs &a, int r, const RowChunks<DT> &rc, float m, float kref, double S_in, DepthHist *h,
                          unsigned long long *buf, double *redd, unsigned long long *redu) {
    constexpr int EPC = Elem<DT>::EPC;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool all_in = a.top_p >= 1.0f;
    // no id below vt holds the crossing (as in the value histogram)
    const float g = all_in ? -41.0f : fmaxf(log2f((1.0f - a.top_p) * (float)S_in / (16.0f * (float)a.V)), -41.0f);
    const float depth = fmaxf(m - (kref + g) / a.c, a.T * 1e-3f);
    const float inv = (float)(DH_W - 4) / depth, wid_b = depth / (float)(DH_W - 4);
    // the bin of v is round(C + 1 - v * inv) with the integer C = round(m * inv):
    // one multiply-add onto 2^23 leaves it in the low bits
    if (!(fabsf(m * inv) < 4.0e6f)) return false;  // (uniform) the index needs 23 bits
    const float C = rintf(m * inv), c0 = 8388608.0f + C + 1.0f, cmax = 8388608.0f + (float)(DH_W + lane);
    auto bin_of = [&](float v) -> int {
        return (int)(__float_as_uint(fminf(fmaf(v, -inv, c0), cmax)) - 0x4B000000u);
    };
    for (int i = tid; i < DH_W + DH_PAD; i += NT) h->cnt[i] = 0u;
    if (tid == 0) {
        h->b_hi = all_in ? -1 : INT_MAX;
        h->b_lo = all_in ? -1 : INT_MAX;
        h->b_k = INT_MAX;
        h->nx = 0;
        h->np = 0;
        h->ix = -1;
    }
    __syncthreads();
    const uint32_t NI = Elem<DT>::NEG_INF_WORD;
    uint32_t ah = 0u, al = 0u;  // the row's exact mass (20-bit parts: at most 2^11 + 4 ids a thread)
    static_assert(ACES_MAX_V / NT + 2 * EPC < 1 << 12, "the parts' sums fit");
    for (int c0i = tid; c0i < rc.nch; c0i += NT * DH_U) {
        uint4 w[DH_U];
#pragma unroll
        for (int u = 0; u < DH_U; ++u) {
            const int c = c0i + u * NT;
            w[u] = c < rc.nch ? rc.load(c) : make_uint4(NI, NI, NI, NI);
        }
#pragma unroll
        for (int u = 0; u < DH_U; ++u)
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
                const float v = Elem<DT>::get(w[u], e);
                const int bn = bin_of(v);
                if (ACES_IN(bn, DH_W + DH_PAD)) atomicAdd(&h->cnt[bn], 1u);
                uint32_t fh, fl;
                to_fx_parts(ex2(fmaf(v, a.c, -kref)), fh, fl);
                ah += fh;
                al += fl;
            }
    }
    const unsigned long long all_fx = block_reduce(((unsigned long long)ah << 20) + al, redu, SumU64());
    const double S = (double)all_fx * FX_INV;
    const unsigned long long tg = all_in ? 0ull : (unsigned long long)ceil((double)a.top_p * (double)all_fx);
    __syncthreads();
    // ---- the bins around the crossing and the payload's last ----
    int b_hi, b_lo, b_k;
    {
        constexpr int PER = DH_W / NT;
        uint32_t cn[PER], lc = 0u;
        float lu = 0.0f, ll = 0.0f, mu[PER], ml[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int bn = tid * PER + i;
            cn[i] = h->cnt[bn];
            // v * inv lies within [C + 0.5 - bn, C + 1.5 - bn]
            const float vu = fminf((C + 1.5f - (float)bn) * wid_b, m), vl = (C + 0.5f - (float)bn) * wid_b;
            mu[i] = (float)cn[i] * ex2(fmaf(vu, a.c, -kref)) * (1.0f + 1e-4f);
            ml[i] = (float)cn[i] * ex2(fmaf(vl, a.c, -kref)) * (1.0f - 1e-4f);
            lu += mu[i];
            ll += ml[i];
            lc += cn[i];
        }
        float iu = lu, il = ll;
        uint32_t ic = lc;
        for (int o = 1; o < 32; o <<= 1) {
            const float tu = __shfl_up_sync(0xffffffffu, iu, o), tl = __shfl_up_sync(0xffffffffu, il, o);
            const uint32_t tc = __shfl_up_sync(0xffffffffu, ic, o);
            if (lane >= o) {
                iu += tu;
                il += tl;
                ic += tc;
            }
        }
        if (lane == 31) {
            h->wu[wid] = iu;
            h->wl[wid] = il;
            h->wc[wid] = ic;
        }
        __syncthreads();
        for (int i = 0; i < wid; ++i) {
            iu += h->wu[i];
            il += h->wl[i];
            ic += h->wc[i];
        }
        float cu = iu - lu, cl = il - ll;
        uint32_t cc = ic - lc;
        const float tgf = (float)tg * (1.0f / FX_SCALE);
        const uint32_t ku = (uint32_t)a.k;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int bn = tid * PER + i;
            cu += mu[i];
            cl += ml[i];
            cc += cn[i];
            if (!all_in) {  // (1e-4: the rounding of the sums and of the target)
                if (cu >= tgf * (1.0f - 1e-4f)) atomicMin(&h->b_hi, bn);
                if (cl >= tgf * (1.0f + 1e-4f)) atomicMin(&h->b_lo, bn);
            }
            if (cc >= ku) atomicMin(&h->b_k, bn);
        }
        __syncthreads();
        b_hi = h->b_hi;
        b_lo = h->b_lo;
        if (b_lo == INT_MAX || (all_in && h->b_k == INT_MAX)) return false;
        b_k = a.k == 0 ? -1 : (all_in ? h->b_k : min(h->b_k, b_lo));
        // the lists' lengths (the crossing's in the upper half): a row whose lists
        // do not fit (values alike: logits that were bfloat16 once) is declined
        // before the second read.  (256 rows of 128256 equal float32 logits: 2134
        // us a call with that read, 1942 without.)
        unsigned long long len = 0ull;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int bn = tid * PER + i;
            if (!all_in && bn >= b_hi && bn <= b_lo) len += (unsigned long long)cn[i] << 32;
            if (bn <= b_k) len += cn[i];
        }
        // (its barriers: every bin is read, the lists may take the counters' place)
        len = block_reduce(len, redu, SumU64());
        if ((len >> 32) > (unsigned long long)DH_XCAP || (uint32_t)len > (uint32_t)DH_PCAP) return false;
    }
    // ---- exact masses above the range, the ids inside it and the payload's ----
    // (ids are looked at one by one only from a value just below the lowest
    // needed bin: their number per lane, not the row's length, is what costs)
    const int b_top = max(b_lo, b_k);
    const float v_min = fminf((C + 0.5f - (float)b_top) * wid_b, m) - 2.0f * wid_b;
    uint32_t hs = 0u, ls = 0u, na = 0u;
    for (int c0i = tid & ~31; c0i < rc.nch; c0i += NT * DH_U) {  // warp-uniform rounds
        uint4 w[DH_U];
#pragma unroll
        for (int u = 0; u < DH_U; ++u) {
            const int c = c0i + lane + u * NT;
            w[u] = c < rc.nch ? rc.load(c) : make_uint4(NI, NI, NI, NI);
        }
#pragma unroll
        for (int u = 0; u < DH_U; ++u) {
            uint32_t mk = 0u;
#pragma unroll
            for (int e = 0; e < EPC; ++e) mk |= (uint32_t)(Elem<DT>::get(w[u], e) >= v_min) << e;
            while (__any_sync(0xffffffffu, mk != 0u)) {
                const bool on = mk != 0u;
                const int e = on ? __ffs(mk) - 1 : 0;
                mk &= mk - 1u;
                const float v = chunk_at<DT>(w[u], e);
                const int bn = on ? bin_of(v) : INT_MAX;
                if (bn < b_hi) {
                    uint32_t fh, fl;
                    to_fx_parts(ex2(fmaf(v, a.c, -kref)), fh, fl);
                    hs += fh;
                    ls += fl;
                    ++na;
                }
                const bool tx = bn >= b_hi && bn <= b_lo, tp = bn <= b_k;
                if (__any_sync(0xffffffffu, tx || tp)) {
                    const unsigned long long o = order_val(fkey(v), (uint32_t)((c0i + lane + u * NT) * EPC + e - rc.head));
                    warp_append_cap(h->xs, &h->nx, tx, o, DH_XCAP);
                    warp_append_cap(h->ps, &h->np, tp, o, DH_PCAP);
                }
            }
        }
    }
    const unsigned long long above = block_reduce(((unsigned long long)hs << 20) + ls, redu, SumU64());
    const unsigned long long n_above = block_reduce((unsigned long long)na, redu, SumU64());
    __syncthreads();
    const int nx = h->nx, np = h->np;
    if (!all_in && above >= tg) {  // (a bin's bound of a logit far from zero was too tight)
        if (tid == 0) atomicAdd(&a.ws.fb_count[15], 1);
        return false;
    }
    // the payload's ids by rank
    const int lp = np < a.k ? np : a.k;
    rank_order_values<NT>(h->ps, np, reinterpret_cast<uint32_t *>(h->fx), [&](int rank, unsigned long long key) {
        if (rank < lp && ACES_IN(rank, ACES_MAX_TOPK)) buf[rank] = key;
    });
    double S_nuc = S;
    unsigned long long cut = 0ull;
    int L = lp;
    if (!all_in) {
        const int p2 = next_pow2(nx < 2 ? 2 : nx);
        for (int i = nx + tid; i < p2; i += NT) h->xs[i] = 0ull;
        __syncthreads();
        bitonic_sort_desc(h->xs, p2);
        for (int i = tid; i < nx; i += NT) h->fx[i] = to_fx(ex2(fmaf(order_value(h->xs[i]), a.c, -kref)));
        __syncthreads();
        const int per = (nx + NT - 1) / NT;
        const int lo = min(nx, tid * per), hi = min(nx, lo + per);
        unsigned long long loc = 0ull;
        for (int i = lo; i < hi; ++i) loc += h->fx[i];
        unsigned long long tot;
        unsigned long long cum = above + block_exscan_n<NT>(loc, redu, &tot);
        for (int i = lo; i < hi; ++i) {
            const unsigned long long prev = cum;
            cum += h->fx[i];
            if (prev < tg && cum >= tg) {  // one id crosses
                h->ix = i;
                h->cum = cum;
            }
        }
        __syncthreads();
        const int ix = h->ix;
        if (ix < 0) {
            if (tid == 0) atomicAdd(&a.ws.fb_count[15], 1);
            return false;
        }
        S_nuc = (double)h->cum * FX_INV;
        cut = ACES_IN(ix, DH_XCAP) ? h->xs[ix] : 0ull;
        const unsigned long long n_nuc = n_above + (unsigned long long)ix + 1ull;
        if (n_nuc < (unsigned long long)L) L = (int)n_nuc;
    }
    __syncthreads();
    if (tid == 0) atomicAdd(&a.ws.fb_count[14], 1);
    finish_row<DT>(a, r, rc.row(), kref, S_nuc, cut, all_in ? RS_ALL_IN : 0, buf, L, redd);
    return true;
}

template <int DT>
__global__ void __launch_bounds__(NT, 2) k_rows_general(const __grid_constant__ RowArgs a) {
    namespace cg = cooperative_groups;
    using E = Elem<DT>;
    __shared__ SelState st;
    __shared__ __align__(16) union {
        BinState bs;   // binned path
        ValHist vh;    // value-histogram path (bfloat16)
        DepthHist dh;  // depth-histogram path
    } paths;
    static_assert(sizeof(paths) >= DRAW_SCRATCH, "the draw's scratch fits");
    unsigned char *scratch = reinterpret_cast<unsigned char *>(&paths);  // (of a finished row)
    __shared__ unsigned long long buf[ACES_MAX_TOPK];
    __shared__ double redd[NWARP];
    __shared__ unsigned long long redu[NWARP];
    __shared__ int s_nbuf;
    __shared__ DrawPart part;
    __shared__ int pend[DRAW_CL];
    const int tid = threadIdx.x;
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    pdl_wait();  // after the single-pass row kernel: its fallback list is complete
    if (a.K > 0 && blockIdx.x == 0 && tid < WS_COUNTERS / 4) {
        // the hints of this call's rows, for the first rows of the next call
        // with the same shape (the row kernel reads them only when fewer than
        // its minimum of that call's rows have finished)
        int v = tid >= WS_DEPTH ? __ldcg(&a.ws.fb_count[tid]) : 0;
        if (tid == 0) v = CARRY_MAGIC;
        if (tid == 1) v = __float_as_int(a.T);
        if (tid == 2) v = __float_as_int(a.top_p);
        if (tid == 3) v = a.k;
        if (tid == 4) v = a.V;
        if (tid == 5) v = DT;
        if (tid == 6) v = __ldcg(&a.ws.fb_count[8]);
        if (tid == 7) v = __ldcg(&a.ws.fb_count[11]);
        a.ws.carry[tid] = v;
    }
    // one handed row (all threads)
    auto do_row = [&](int r) {
        const RowChunks<DT> rc(reinterpret_cast<const char *>(a.logits) + (size_t)r * a.V * E::SIZE, a.V);
        // it comes with its max and its exp-sum, and is finite
        const RowStat hs = a.ws.stats[r];
        const float m = hs.kref;
        const float kref = ceilf(m * a.c);  // masses are 2^(z*c - kref) <= 1
        // the exp-sum in units of 2^kref (its reference is the same ceil(m c); the
        // power-of-two rescale is exact)
        const double S_in = ldexp(hs.S_nuc, (int)(hs.c - kref));
        unsigned long long n_fin = 0ull;  // finite ids (top_p = 1)
        bool depth = true;
        if constexpr (DT == ACES_BF16) {
            const int vh = valhist_row(a, r, rc, m, kref, S_in, &n_fin, &paths.vh, buf, redd, redu);
            __syncthreads();
            if (vh == VH_DONE) return;
            depth = vh == VH_BELOW;
        }
        if (depth) {
            const bool done = depth_row<DT>(a, r, rc, m, kref, S_in, &paths.dh, buf, redd, redu);
            __syncthreads();
            if (done) return;
        }
        if (DT == ACES_F32 && a.top_p >= 1.0f) {
            unsigned long long nfin = 0ull;
            for_each_elem<DT>(rc, [&](int, float v) { nfin += v > -INFINITY; });
            n_fin = block_reduce(nfin, redu, SumU64());
        }
        if (binned_row<DT>(a, r, rc, m, kref, n_fin, &paths.bs, buf, redd, redu)) return;
        if (tid == 0) atomicAdd(&a.ws.fb_count[4], 1);
        const bool all_in = a.top_p >= 1.0f;
        unsigned long long cut = 0ull;
        double S_nuc;
        unsigned long long n_nuc;
        if (!all_in) {
            cut = radix_select<DT>(rc, kref, a.c, 0, (double)a.top_p, 0u, true, &st);
            S_nuc = (double)(st.above + st.found) * FX_INV;
            n_nuc = (unsigned long long)st.above_cnt + 1ull;
        } else {
            unsigned long long sfx = 0ull;
            for_each_elem<DT>(rc, [&](int, float v) {
                if (v > -INFINITY) sfx += to_fx(ex2(fmaf(v, a.c, -kref)));
            });
            S_nuc = (double)block_reduce(sfx, redu, SumU64()) * FX_INV;
            n_nuc = n_fin;
        }
        __syncthreads();
        // the payload boundary: the last nucleus id, or the k-th id when the
        // nucleus is longer than the payload
        unsigned long long lim = all_in ? 0ull : cut;
        int L = (int)(n_nuc < (unsigned long long)a.k ? n_nuc : (unsigned long long)a.k);
        if (a.k > 0 && n_nuc > (unsigned long long)a.k)
            lim = radix_select<DT>(rc, kref, a.c, 1, 0.0, (unsigned)a.k, false, &st);
        __syncthreads();
        // collect the payload ids (order value >= lim)
        if (tid == 0) s_nbuf = 0;
        __syncthreads();
        if (a.k > 0) {
            for_each_elem<DT>(rc, [&](int x, float v) {
                if (!(v > -INFINITY)) return;
                unsigned long long o = order_val(fkey(v), (uint32_t)x);
                if (o >= lim) {
                    int pos = atomicAdd(&s_nbuf, 1);
                    if (pos < ACES_MAX_TOPK) buf[pos] = o;
                }
            });
        }
        __syncthreads();
        const int nb = min(s_nbuf, ACES_MAX_TOPK);
        const int np = next_pow2(nb < 2 ? 2 : nb);
        for (int i = nb + tid; i < np; i += NT) buf[i] = 0ull;
        __syncthreads();
        bitonic_sort_desc(buf, np);
        if (L > nb) L = nb;
        finish_row<DT>(a, r, rc.row(), kref, S_nuc, cut, all_in ? RS_ALL_IN : 0, buf, L, redd);
    };
    // the handed rows, one a CTA and cluster round; the sequences a round
    // completes are then drawn by the cluster
    const int nrows = *a.ws.fb_count;
    for (int i0 = (int)(blockIdx.x / CL) * CL; i0 < nrows; i0 += (int)gridDim.x) {
        int e = -1;
        if (i0 + rank < nrows) {
            const int r = a.ws.fb_list[i0 + rank];
            if (ACES_IN(r, a.rows)) {  // (the same r in every thread)
                do_row(r);
                e = row_finished<DT, NT>(a, r, scratch);
            }
        }
        if (a.K > 0) {
            if (tid == 0) part.pend = e;
            cl.sync();
            if (tid < CL) pend[tid] = cl.map_shared_rank(&part, tid)->pend;
            cl.sync();
            for (int c = 0; c < CL; ++c)
                if (pend[c] >= 0) {
                    draw_cluster<DT, NT>(a, pend[c] >> 5, pend[c] & 31, &part, scratch);
                    __syncthreads();
                }
        }
        __syncthreads();
    }
    // the sequences the single-pass kernel completed whose draw needs a whole row
    if (a.K > 0) {
        const int nscan = a.ws.fb_count[13];
        for (int i = blockIdx.x / CL; i < nscan; i += gridDim.x / CL) {
            const int e = a.ws.scan_list[i];
            draw_cluster<DT, NT>(a, e >> 5, e & 31, &part, scratch);
            __syncthreads();
        }
    }
}

// Follows the single-pass row kernel and overlaps its drain.  Two
// CTAs an SM at most, fewer when neither the rows it may be handed nor the
// draws fill them; the CTAs of a draw's cluster: as many as let every sequence
// be drawn at once (a draw is a chain of about 20 us however few logits each
// CTA has: 128 sequences in four rounds of clusters of 8 took 120 us).
cudaError_t launch_rows_general(const RowArgs &a, int dt, int nseq, cudaStream_t s) {
    const int most = 2 * a.nsm / DRAW_CL * DRAW_CL;
    int cl = DRAW_CL;
    while (cl > 2 && (long long)cl * nseq > most) cl >>= 1;
    long long want = a.K > 0 && (long long)cl * nseq > a.rows ? (long long)cl * nseq : a.rows;
    want = (want + DRAW_CL - 1) / DRAW_CL * DRAW_CL;
    const unsigned grid = (unsigned)(want < most ? want : most);
    return launch_after(dt == ACES_BF16 ? k_rows_general<ACES_BF16> : k_rows_general<ACES_F32>, grid, NT, (unsigned)cl, s, a);
}

#ifdef ACES_CHECKED
cudaError_t check_take_rows_general(unsigned long long out[3]) { return check_take(out); }
#endif

}  // namespace aces
