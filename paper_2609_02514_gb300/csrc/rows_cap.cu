// Single-pass row kernel of the AceSpec cloud step (Sec. III-B: accept test
// and packaging of the target distribution; Sec. V-C: compact payload; the
// acceptance rule is the modified rejection sampling of Sec. II-A).
//
// One CTA per target row r = b*(K+1)+i: 256 threads, four CTAs per SM; 512 or
// 1024 threads when the launch has few rows (rows_cap_threads).  Every logit
// is read from HBM once, with 16-byte loads, eight in flight per thread; a row
// off the 16-byte grid is read through the chunks that cover it, the elements
// outside it as -inf (RAGGED).  The row is read in tiles of 32 chunks (one
// coalesced 512-byte warp load) in the order t -> (t * pstride) mod ntile, so
// that the first 64 tiles are a strided sample of the whole row.
//
//   stream    an online exp-sum in log2 units against an integer reference
//             k_t = ceil(max z * log2(e)/T) (one paired FFMA per two logits,
//             one ex2 per logit, exact power-of-two rescales), the max, and a
//             running max shared by the CTA's warps.
//   depth     D bounds how far below the row max the nucleus crossing (top_p
//             = 1: the payload's end) lies: a quantile of the depths that the
//             call's finished rows published, plus a margin (before 32 have
//             finished: those the previous call on the same workspace left,
//             for bfloat16 rows of the same shape; else NSB bins of T/4).  D
//             only decides what is kept, never a result.
//   keep      bfloat16, counting pass: every id >= (running max - D)
//             increments a shared-memory counter of its bfloat16 value (a
//             window of HW values); sketch-led pass (when nearly all finished
//             rows had short nuclei): nothing is counted while streaming.
//             Both keep the max of every group of 4 to 8 chunks in a sketch.
//             float32: every 16-byte chunk holding an id >= the threshold is
//             recorded (chunk and index).  The running max only rises, so at
//             the end every id >= (row max - D) was kept (or, sketch-led,
//             lies in a group whose max reaches it).
//   finish    from the exact row max and the exp-sum, exact 2^-40 fixed-point
//             masses give the nucleus crossing (a crossing below the kept
//             values: a second counting pass over the row; a capacity
//             exceeded: the exact general kernel; float32 rows and rows off
//             the 16-byte grid whose crossing depends on the exp-sum's rounding:
//             a second read for the exact mass):
//             bfloat16  (sketch-led: the groups reaching row max - D are read
//                       back and their ids counted first) the CTA scans the
//                       value counts for the crossing value, the number j of
//                       its ids inside the nucleus and the payload's last
//                       value; the sketch's groups whose max reaches that
//                       value are re-read and their ids at or above it
//                       ordered.  When the crossing value's ids are among them
//                       the j-th (in id order) is the cut; otherwise the row
//                       keeps (value, j) and the draw finds that id, only for
//                       the rows it draws from.
//             float32   the recorded ids are binned by (m - z)/(T/8); the bins
//                       up to the one where a lower bound of the mass reaches
//                       the target are ordered (direct ranking up to 512 ids,
//                       else bin by bin with a rank inside each bin) and the
//                       CTA finds the crossing with exact prefix sums.
//             Then the payload, the tail mass, the accept test of the draft
//             token at this position and the per-row state; the CTA that
//             finishes a sequence's last row draws its token when row pi's
//             nucleus was kept.
//
// What bounds it (GB300): 256 sequences x 17 rows of 256000 bfloat16 logits
// take 398 us, 330 us of it the bytes at the rate of a plain copy; the rest is
// each row's epilogue and the last wave.  2176 rows of 128256 (nuclei of
// thousands of ids, so nearly every chunk is counted) are bound by issue
// slots: 14.3 warp instructions per 32 logits (20.5 before the counters took
// no branch: 283 us, then 224).  Launches of one wave are one row's chain of
// dependent steps.
//
// On launches of four waves or more, the j-th CTA each SM starts with waits
// j x 10 us first, so that the first wave's epilogues do not coincide.
#include <climits>
#include <cmath>
#include <mutex>
#include <type_traits>

#include <cuda_bf16.h>

#define ACES_FILE 9  // site numbers of the checked build
#include "draw.cuh"

namespace aces {

constexpr int UC = 8;               // 16-byte chunks per thread and iteration
constexpr int TCH = 32;             // chunks per tile
constexpr int SAMPLE = 64;          // tiles of the sample: the first of the row's order
constexpr int NSB = 40;             // depth bins (of T/SPB) of the hints; D before any hint
constexpr int SPB = 4;              // depth bins per temperature
constexpr int MARGIN_BINS = 2;      // float32 first rows: theta below the sample's crossing
constexpr float LIST_FILL = 0.75f;  // of the list's room, at most, where the sample can tell
constexpr int HINT_MIN = 32;        // finished rows before their depths set D
constexpr int HINT_MARGIN = 2;      // depth bins of margin above that quantile
constexpr float HINT_Q = 0.99f;     // the quantile of the finished rows' depths D covers
// bfloat16
constexpr int HW = 1024;            // counted values (bfloat16 bit patterns) per row
constexpr int HEADROOM = 256;       // of them above the sample's max at least
constexpr int SKG = 16384;          // sketch entries (group maxima, as 16-bit order keys)
constexpr int PCAP = 1024;          // ids at or above the payload's last value
constexpr int GCAP = 1024;          // sketch groups re-read
// Values below the counted ones go to one of HPAD counters just below them,
// lane l's to the l-th: every lane adds to some counter, so that counting
// takes no branch (a predicated reduction on shared memory is compiled into
// one: 18.3 instructions a logit on flat rows) and no two lanes of a warp
// add to the same dummy.  Counters below the final limit are never read.
constexpr int HPAD = 32;
constexpr int SMEM_BF = (HPAD + HW) * 4 + SKG * 2 + PCAP * 8;
// sketch-led pass: a row is short when at most SHORT_IDS ids reach its
// crossing (top_p = 1: when k <= SHORT_IDS); later rows take the pass when
// at least SHORT_NUM / SHORT_DEN of the finished rows were short.  Its areas
// inside the sketch's (in 8-byte units): the ordered ids [0, 1024), the
// groups read back, then the kept ids [2048, 3072)
constexpr int SHORT_IDS = 256;
constexpr int SHORT_NUM = 49, SHORT_DEN = 50;
constexpr int SK_TMP = 2048;
// float32
constexpr int CREC = 1536;          // recorded chunks (16-byte chunk + its index) per row
constexpr int LCAP = 2048;          // listed ids, expanded from the records after the stream
constexpr int WCAP = 2048;          // work area: ordered candidates
constexpr int SMEM_F32 = CREC * 20 + LCAP * 8 + NBIN * 4;
// float32 rows of a launch that fits one wave at two CTAs per SM take wider
// areas (and a deeper first capture): more records and list entries per row
template <int W>
struct F32Caps {
    static constexpr int CR = W == 2 ? 3584 : CREC;  // recorded chunks
    static constexpr int LC = W == 2 ? 4096 : LCAP;  // listed ids
    static constexpr int WC = W == 2 ? 4096 : WCAP;  // ordered candidates
    static constexpr int MARGIN = W == 2 ? MARGIN_BINS + 2 : MARGIN_BINS;
    static constexpr int SMEM = CR * 20 + LC * 8 + NBIN * 4;
};

constexpr int RANK_MAX = 512;       // ids ordered by direct ranking (more: bitonic sort)
static_assert(WS_DEPTH + NSB <= WS_COUNTERS / 4, "the depth histogram fits the counters area");
static_assert(DRAW_SCRATCH <= SMEM_BF && DRAW_SCRATCH <= SMEM_F32, "the draw's scratch fits");
// (32-bit keys are read 16 bytes at a time: at hist, and after two lists of RANK_MAX)
static_assert(HPAD * 4 % 16 == 0 && CREC * 20 % 16 == 0 && F32Caps<2>::CR * 20 % 16 == 0 && 2 * RANK_MAX * 8 % 16 == 0,
              "the keys of the ranking lie on 16 bytes");
static_assert(ACES_MAX_V <= 1 << 20 && HW <= 1 << 10 && RANK_MAX <= HW, "a value and an id in 30 bits");
static_assert(GCAP * 4 <= HW * 4 && PCAP * 8 <= SKG * 2 && "the aliased areas fit");
static_assert(PCAP <= SK_TMP && SK_TMP + GCAP / 2 <= SKG / 4 && SK_TMP + PCAP <= SKG / 4, "the sketch-led areas fit");
static_assert(WCAP * 8 <= CREC * 20 && RANK_MAX * 5 / 2 <= LCAP, "the float32 work areas fit");
static_assert(F32Caps<2>::WC * 8 <= F32Caps<2>::CR * 20 && RANK_MAX * 2 <= F32Caps<2>::LC &&
                  2 * (F32Caps<2>::SMEM + 1024) <= 228 * 1024,
              "the wide float32 areas fit, two CTAs per SM");

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// 2^d for an integer-valued d <= 0, exactly
__device__ __forceinline__ float pow2_int(float d) {
    return d >= -126.0f ? __int_as_float((127 + __float2int_rn(d)) << 23) : 0.0f;
}

// Paired fp32 arithmetic (one instruction for two lanes of a 64-bit register
// pair; each lane rounds exactly like the scalar operation).
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b,
                                                    unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// (2^(lo*c + nk), 2^(hi*c + nk)) for a pair of logits
__device__ __forceinline__ unsigned long long ex2_pair(unsigned long long z2, unsigned long long c2,
                                                       unsigned long long nk2) {
    float lo, hi;
    unpack2(ffma2(z2, c2, nk2), lo, hi);
    return pack2(ex2(lo), ex2(hi));
}

// Max of one chunk, as a packed pair (bfloat16: the max of its even and of
// its odd elements, NaN when one is NaN; float32: the max of all four).
template <int DT>
__device__ __forceinline__ uint32_t chunk_max2(const uint4 &w) {
    if (DT == ACES_BF16) {
        const __nv_bfloat162 a = __hmax2_nan(*reinterpret_cast<const __nv_bfloat162 *>(&w.x),
                                             *reinterpret_cast<const __nv_bfloat162 *>(&w.y));
        const __nv_bfloat162 b = __hmax2_nan(*reinterpret_cast<const __nv_bfloat162 *>(&w.z),
                                             *reinterpret_cast<const __nv_bfloat162 *>(&w.w));
        const __nv_bfloat162 m = __hmax2_nan(a, b);
        return *reinterpret_cast<const uint32_t *>(&m);
    } else {
        return __float_as_uint(fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)),
                                     fmaxf(__uint_as_float(w.z), __uint_as_float(w.w))));
    }
}
// the max of two such maxima
template <int DT>
__device__ __forceinline__ uint32_t max2(uint32_t x, uint32_t y) {
    if (DT == ACES_BF16) {
        const __nv_bfloat162 m = __hmax2_nan(*reinterpret_cast<const __nv_bfloat162 *>(&x),
                                             *reinterpret_cast<const __nv_bfloat162 *>(&y));
        return *reinterpret_cast<const uint32_t *>(&m);
    }
    return __float_as_uint(fmaxf(__uint_as_float(x), __uint_as_float(y)));
}
template <int DT>
__device__ __forceinline__ float max2_value(uint32_t m2) {
    if (DT == ACES_BF16) return fmaxf(__uint_as_float(m2 << 16), __uint_as_float(m2 & 0xFFFF0000u));
    return __uint_as_float(m2);
}

// 2^(z*c - k) summed over one chunk, as a packed pair of partial sums
template <int DT>
__device__ __forceinline__ unsigned long long chunk_expsum2(const uint4 &x, unsigned long long c2,
                                                            unsigned long long nk2) {
    if (DT == ACES_BF16) {
        const uint32_t wd[4] = {x.x, x.y, x.z, x.w};
        unsigned long long p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            p[q] = ex2_pair(pack2(__uint_as_float(wd[q] << 16), __uint_as_float(wd[q] & 0xFFFF0000u)), c2, nk2);
        return fadd2(fadd2(p[0], p[1]), fadd2(p[2], p[3]));
    } else {
        const unsigned long long p0 = ex2_pair(pack2(__uint_as_float(x.x), __uint_as_float(x.y)), c2, nk2);
        const unsigned long long p1 = ex2_pair(pack2(__uint_as_float(x.z), __uint_as_float(x.w)), c2, nk2);
        return fadd2(p0, p1);
    }
}

// adds a chunk's pair s into the two accumulators (even and odd chunks)
__device__ __forceinline__ void acc_pair(int j, unsigned long long s, unsigned long long &acc0,
                                         unsigned long long &acc1) {
    if (j & 1) acc1 = j == 1 ? s : fadd2(acc1, s);
    else acc0 = j == 0 ? s : fadd2(acc0, s);
}

__device__ __forceinline__ float acc_total(unsigned long long acc0, unsigned long long acc1) {
    float a, b;
    unpack2(fadd2(acc0, acc1), a, b);
    return a + b;
}

// sum over the chunks of 2^(z*c - k), two logits per instruction
// (chunks U0 <= j < U1)
template <int DT, int U0, int U1>
__device__ __forceinline__ float chunks_expsum(const uint4 (&w)[UC], float c, float nk) {
    const unsigned long long c2 = pack2(c, c), nk2 = pack2(nk, nk);
    unsigned long long acc0 = 0ull, acc1 = 0ull;
#pragma unroll
    for (int j = U0; j < U1; ++j) acc_pair(j - U0, chunk_expsum2<DT>(w[j], c2, nk2), acc0, acc1);
    return acc_total(acc0, acc1);
}

// The same with the rounding error of every add in err (the two-sum of two
// logits at a time): the mass of top_p = 1 rows off the 16-byte grid, which the
// probabilities are divided by.  24 x 6 such rows of 50003 bfloat16 logits: 43 us
// a call, 41 with plain adds, 47 with a second read for the exact mass; root mean
// square error of the payload against float64 (5120 rows) 1.257e-7, 1.275e-7 and
// 1.238e-7, mean error of the tail 0.94e-8, 1.76e-8 and 1.23e-8.
template <int DT, int U0, int U1>
__device__ __forceinline__ float chunks_expsum_err(const uint4 (&w)[UC], float c, float nk, float &err) {
    err = 0.0f;
    if constexpr (U0 >= U1) return 0.0f;
    const unsigned long long c2 = pack2(c, c), nk2 = pack2(nk, nk), m1 = pack2(-1.0f, -1.0f);
    unsigned long long s = 0ull, e = 0ull;
    auto add = [&](unsigned long long x) {
        const unsigned long long t = fadd2(s, x), b = ffma2(s, m1, t);  // b = t - s
        e = fadd2(e, fadd2(ffma2(ffma2(b, m1, t), m1, s), ffma2(b, m1, x)));
        s = t;
    };
#pragma unroll
    for (int j = U0; j < U1; ++j) {
        const uint32_t wd[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (DT == ACES_BF16)
                add(ex2_pair(pack2(__uint_as_float(wd[q] << 16), __uint_as_float(wd[q] & 0xFFFF0000u)), c2, nk2));
            else if (q & 1)
                add(ex2_pair(pack2(__uint_as_float(wd[q - 1]), __uint_as_float(wd[q])), c2, nk2));
        }
    }
    float a, b, ea, eb, sm;
    unpack2(s, a, b);
    unpack2(e, ea, eb);
    two_sum(a, b, sm, err);
    err += ea + eb;
    return sm;
}

// maxima of chunks 0..3 and 4..7 (bfloat16: packed over all their pairs,
// unpacked once); returns the packed max of both
template <int DT>
__device__ __forceinline__ uint32_t group_maxima(const uint4 (&w)[UC], float &g0, float &g1) {
    uint32_t p[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        p[h] = chunk_max2<DT>(w[h * (UC / 2)]);
#pragma unroll
        for (int u = 1; u < UC / 2; ++u) p[h] = max2<DT>(p[h], chunk_max2<DT>(w[h * (UC / 2) + u]));
    }
    g0 = max2_value<DT>(p[0]);
    g1 = max2_value<DT>(p[1]);
    return max2<DT>(p[0], p[1]);
}

// element e of a chunk (e may be a run-time index)
template <int DT>
__device__ __forceinline__ float chunk_elem(const uint4 &w, int e) {
    if (DT == ACES_BF16) {
        const uint32_t lo = (e & 4) ? w.z : w.x, hi = (e & 4) ? w.w : w.y;
        const uint32_t wd = (e & 2) ? hi : lo;
        return __uint_as_float((e & 1) ? (wd & 0xFFFF0000u) : (wd << 16));
    } else {
        const uint32_t lo = (e & 2) ? w.z : w.x, hi = (e & 2) ? w.w : w.y;
        return __uint_as_float((e & 1) ? hi : lo);
    }
}

// adds 1 to the shared-memory counter at address addr
__device__ __forceinline__ void red_inc(int addr) {
    asm volatile("red.shared.add.u32 [%0], 1;" :: "r"(addr) : "memory");
}

// bfloat16 order key of a bfloat16 bit pattern (keys sort like values, -0
// and +0 share one key), and the value of a key
__device__ __forceinline__ uint32_t key16(uint32_t b) {
    const uint32_t mag = b & 0x7FFFu;
    return (b & 0x8000u) ? 0x8000u - mag : 0x8000u + mag;
}
__device__ __forceinline__ float val16(uint32_t k) {
    const uint32_t b = k >= 0x8000u ? k - 0x8000u : (0x8000u | (0x8000u - k));
    return __uint_as_float(b << 16);
}

// Hands row r to the general kernel with its max m and its exp-sum S (in
// units of 2^kref), which spare that kernel a pass and the exponentials of
// another (the row is finite: rows with NaN or +inf are marked NONFINITE
// before any handoff).
__device__ __forceinline__ void fallback_row(const RowArgs &a, int r, float m, float kref, double S) {
    RowStat s;
    s.kref = m;
    s.c = kref;
    s.S_nuc = S;
    s.cut = 0ull;
    s.flags = 0;
    s.nnuc = -1;
    a.ws.stats[r] = s;
    const int pos = atomicAdd(a.ws.fb_count, 1);
    a.ws.fb_list[pos] = r;
}

// lists a sequence for the general kernel's draw (e: row_finished's)
__device__ __forceinline__ void defer_draw(const RowArgs &a, int e) {
    if (e >= 0 && threadIdx.x == 0) a.ws.scan_list[atomicAdd(&a.ws.fb_count[13], 1)] = e;
}

// appends o to arr[*n] for every lane with take (one atomic per warp); *n
// may pass cap, entries beyond it are dropped (all lanes of the warp call it)
__device__ __forceinline__ void append_cap(unsigned long long *arr, int *n, bool take, unsigned long long o, int cap) {
    const unsigned bal = __ballot_sync(0xffffffffu, take);
    if (bal == 0u) return;
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == __ffs(bal) - 1) base = atomicAdd(n, __popc(bal));
    base = __shfl_sync(0xffffffffu, base, __ffs(bal) - 1);
    const int pos = base + __popc(bal & ((1u << lane) - 1u));
    if (take && pos < cap) arr[pos] = o;
}

// mass of one id of logit v in 2^-40 units (the same formula in every kernel)
__device__ __forceinline__ unsigned long long id_fx(float v, float c, float kref) {
    return to_fx(ex2(fmaf(v, c, -kref)));
}

// The row's mass against its reference kref as the general kernel sums it: in
// 2^-40 units, exactly (a second read of the row; all NTC threads).
template <int DT, int NTC, bool RAGGED>
__device__ __noinline__ unsigned long long exact_mass(const char *row, int V, float c, float kref, unsigned long long *red) {
    constexpr int EPC = Elem<DT>::EPC, U = 32 / EPC;  // loads in flight (32 ids: more code is slower the first time)
    const RowChunks<DT, RAGGED> rc(row, V);
    const uint32_t ni = Elem<DT>::NEG_INF_WORD;
    unsigned long long sum = 0ull;
    for (int c0 = threadIdx.x; c0 < rc.nch; c0 += NTC * U) {
        uint4 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ch = c0 + u * NTC;
            w[u] = ch < rc.nch ? rc.load(ch) : make_uint4(ni, ni, ni, ni);
        }
        uint32_t hi = 0u, lo = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
                uint32_t h, l;
                to_fx_parts(ex2(fmaf(Elem<DT>::get(w[u], e), c, -kref)), h, l);
                hi += h;
                lo += l;
            }
        sum += ((unsigned long long)hi << 20) + lo;
    }
    return block_reduce_n<NTC>(sum, red, SumU64());
}

// sum_err (see rows_cap_layout) of a row whose nucleus, P of its mass S, has n
// ids: they bound the masses' entropy and with it the mean depth (about 7
// instead of 18 bits for 900 of 128256 ids, P = 0.95, S = 15)
__device__ __noinline__ float sharp_err(float sum_err, float P, int n, int V, float S) {
    const float h = -P * log2f(P) - (1.0f - P) * log2f(1.0f - P), lv = log2f((float)V);
    const float depth = h + P * log2f((float)n) + (1.0f - P) * lv - log2f(S) + 0.01f;
    return sum_err - 2.0f * 0.6931472f * ldexpf(fmaxf(lv + 1.0f - fmaxf(depth, 0.0f), 0.0f), -24);
}

// NTC: threads per CTA, 1024 / NTC CTAs per SM
// (RAGGED: rows off the 16-byte grid; a build of its own, as the edges cost
// the other one registers: 128 x 17 rows of 128256 205 -> 213 us)
template <int DT, int W, int NTC, bool RAGGED>
__global__ void __launch_bounds__(NTC, 1024 / NTC) k_rows_cap(RowArgs a) {
    constexpr int NWC = NTC / 32;
    constexpr int TPI = NWC * UC;         // tiles per iteration
    constexpr int UCS = SAMPLE / NWC;     // this thread's chunks of iteration 0 that are in the sample
    static_assert(UCS >= 1 && UCS <= UC && HW % NTC == 0, "the sample lies in iteration 0");
    constexpr int CREC = F32Caps<W>::CR, LCAP = F32Caps<W>::LC, WCAP = F32Caps<W>::WC;
    constexpr int MARGIN_BINS = F32Caps<W>::MARGIN;
    using E = Elem<DT>;
    constexpr int EPC = E::EPC;
    constexpr bool BF = DT == ACES_BF16;
    // The cut of float32 rows, and of bfloat16 rows off the 16-byte grid, is the
    // one of the row's exact mass, whichever kernel finishes the row: the
    // float32 sum places the target within a bound, and where the cut is not the
    // same over that whole range (sharpen) the row is read again for its exact
    // mass: 5 to 12 us more on a call of one wave.  (Rows cut one id away from
    // float64, of 128000 each, by the float32 sum and by the exact one: float32
    // rows of 50000 logits 11 and 6, of 50003 7 and 9, of 20001 5 and 0; bfloat16
    // rows of 50003 9 and 6, of 20001 1 and 0.)
    constexpr bool EXACT_CUT = !BF || RAGGED;
    extern __shared__ __align__(16) unsigned char smem[];
    // bfloat16: [HPAD dummies, value counts: HW u32 | sketch: SKG u16 | ids >=
    //           the payload's last value: PCAP u64]; the list of re-read groups
    //           reuses the counts, the ordered ids the sketch, once each is read
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem) + HPAD;
    uint16_t *sk = reinterpret_cast<uint16_t *>(smem + (HPAD + HW) * 4);
    unsigned long long *pay = reinterpret_cast<unsigned long long *>(smem + (HPAD + HW) * 4 + SKG * 2);
    uint32_t *glist = hist;
    unsigned long long *sorted = reinterpret_cast<unsigned long long *>(sk);
    // float32:  [records: CREC x (16 + 4) bytes | list: LCAP u64 | bin counts:
    //           NBIN u32]; the work area reuses the records once they are expanded
    uint4 *rec_dat = reinterpret_cast<uint4 *>(smem);
    uint32_t *rec_idx = reinterpret_cast<uint32_t *>(smem + CREC * 16);
    unsigned long long *list = reinterpret_cast<unsigned long long *>(smem + CREC * 20);
    uint32_t *bcnt = reinterpret_cast<uint32_t *>(smem + CREC * 20 + LCAP * 8);
    unsigned long long *work = reinterpret_cast<unsigned long long *>(smem);

    __shared__ uint32_t sbin[NWC][NSB];  // float32 estimate: per warp, below the sample max
    __shared__ float redf[NWC], redk[NWC], redh[NWC], redl[NWC];
    __shared__ int s_nrec, s_nl, s_fb, s_n, s_bsel, s_nstar, s_L, s_npay, s_ng, s_nge, s_j, s_vs, s_vk;
    __shared__ float s_thlo, s_zx;
    __shared__ int s_dbins, s_xb;  // s_dbins: D in depth bins (-1: no hints yet)
    __shared__ int s_skm;          // bfloat16: the sketch-led pass (no counting while streaming); float32: see there
    __shared__ uint32_t s_m1, s_mr;  // order keys of the sample's max and of the running max after it
    __shared__ double s_Snuc;
    __shared__ float s_inv_S;
    __shared__ unsigned long long s_cut, s_cumL_fx;
    __shared__ unsigned long long s_tg, s_th;  // the target lies in [s_tg, s_th] (one value when it is exact)
    __shared__ unsigned long long s_redu[NWC], s_above, s_evs;
    __shared__ uint32_t s_redc[NWC], s_cab, s_cnvs;
    __shared__ int s_settled;

    const int r = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (NTC == 256 && a.stagger_ns > 0 && r < 4 * a.nsm) {
        // the j-th CTA an SM starts with (blocks are placed on the SMs in
        // turn) waits j times stagger_ns on the global timer (bounded: at
        // most 3 x stagger_ns)
        const unsigned long long wait = (unsigned long long)(r / a.nsm) * (unsigned long long)a.stagger_ns;
        const unsigned long long t0 = globaltimer_ns();
        for (int i = 0; i < 1000 && globaltimer_ns() - t0 < wait; ++i) __nanosleep(1000);
    }
    // (a row off the 16-byte grid: its chunks are cut at the boundaries, the
    // first and the last padded with -inf)
    const RowChunks<DT, RAGGED> rc(reinterpret_cast<const char *>(a.logits) + (size_t)r * a.V * E::SIZE, a.V);
    const char *row = rc.base;
    const int nch = rc.nch, ntile = a.ntile;
    const int nit = (ntile + TPI - 1) / TPI;
    const uint32_t NI = E::NEG_INF_WORD;
    const bool all_in = a.top_p >= 1.0f;

    // the draft token of this position, fetched early by thread 0 and kept
    // in shared memory across the stream (xb, bq, iq are set after it)
    int xb = -1, bq = 0, iq = 0;
    int xb0 = -1;
    if (a.K > 0 && tid == 0 && r % (a.K + 1) < a.K) xb0 = a.xt[(size_t)(r / (a.K + 1)) * a.K + r % (a.K + 1)];
    if (BF) {
        for (int i = tid; i < HW; i += NTC) hist[i] = 0u;
    } else {
        for (int i = tid; i < NWC * NSB; i += NTC) (&sbin[0][0])[i] = 0u;
    }
    if (tid == 0) {
        s_nrec = 0;
        s_nl = 0;
        s_fb = 0;
        s_nstar = INT_MAX;
        s_m1 = s_mr = fkey(-INFINITY);
    }
    __syncthreads();  // (other warps add to these before the next barrier)
    // the depths published by the call's finished rows (read by warp 0 only,
    // once: they change while this row streams)
    int hr = 0, hc0 = 0, hc1 = 0, hs = 0, hf = 0;
    if (wid == 0) {
        hr = __ldcg(&a.ws.fb_count[8]);
        hs = __ldcg(&a.ws.fb_count[11]);
        if (!BF) hf = __ldcg(&a.ws.fb_count[0]);
        hc0 = 2 * lane < NSB ? __ldcg(&a.ws.fb_count[WS_DEPTH + 2 * lane]) : 0;
        hc1 = 2 * lane + 1 < NSB ? __ldcg(&a.ws.fb_count[WS_DEPTH + 2 * lane + 1]) : 0;
        if (BF && hr < HINT_MIN) {
            // too few yet: those the previous call on this workspace carried,
            // when it had the same T, top_p, k, V and logit type (bfloat16
            // rows: a float32 row's capture from its own sample overflows
            // less often than from the carried depth)
            const int *cy = a.ws.carry;
            const bool same = __ldcg(cy) == CARRY_MAGIC && __ldcg(cy + 1) == __float_as_int(a.T) &&
                              __ldcg(cy + 2) == __float_as_int(a.top_p) && __ldcg(cy + 3) == a.k &&
                              __ldcg(cy + 4) == a.V && __ldcg(cy + 5) == DT && __ldcg(cy + 6) >= HINT_MIN;
            if (same) {
                hr = __ldcg(cy + 6);
                hs = __ldcg(cy + 7);
                hc0 = 2 * lane < NSB ? __ldcg(cy + WS_DEPTH + 2 * lane) : 0;
                hc1 = 2 * lane + 1 < NSB ? __ldcg(cy + WS_DEPTH + 2 * lane + 1) : 0;
            }
        }
    }

    // ---- stream ----
    float k_t = -1e30f, m_t = -INFINITY, s_t = 0.f, e_t = 0.f;
    uint4 w[UC];
    // this lane's byte offset of (iteration, u = 0): tile * 512 + lane * 16;
    // the next chunk's is one addition and one unsigned min away (a tile
    // index past ntile wraps around: off - tile_end is huge before that)
    uint32_t off0 = (uint32_t)(((long long)wid * a.pstride) % ntile) * (TCH * 16) + lane * 16;
    const uint32_t off_w = (uint32_t)a.pstride_w * (TCH * 16), off_it = (uint32_t)a.pstride_it * (TCH * 16);
    const uint32_t tile_end = (uint32_t)ntile * (TCH * 16);
    auto wrap = [&](uint32_t off) -> uint32_t { return min(off, off - tile_end); };
    // (iterations whose tiles all exist and are whole load without checks:
    // only the last iteration can hold fewer tiles, and only the row's last
    // tile can be partial; off the 16-byte grid also the first and the one
    // before the last)
    auto load = [&](int it) {
        uint32_t off = off0;
        if ((it + 1) * TPI > ntile || it == a.it_partial ||
            (RAGGED && (it == 0 || it == a.it_partial2))) {
#pragma unroll
            for (int u = 0; u < UC; ++u) {
                const int t = it * TPI + u * NWC + wid;
                w[u] = (t < ntile && off < (uint32_t)nch * 16u) ? rc.load((int)(off >> 4)) : make_uint4(NI, NI, NI, NI);
                off = wrap(off + off_w);
            }
        } else {
#pragma unroll
            for (int u = 0; u < UC; ++u) {
                w[u] = ldg16(row + off);
                off = wrap(off + off_w);
            }
        }
    };
    // the iteration's max im raises m_t and the reference k_t
    auto raise_ref = [&](float im) {
        m_t = fmaxf(m_t, im);
        const float gk = im * a.c;
        if (gk > k_t) {
            const float nk = ceilf(gk);
            const float sc = pow2_int(k_t - nk);
            s_t *= sc;
            e_t *= sc;
            k_t = nk;
        }
    };
    auto add_sum = [&](float gs) {
        const float t = s_t + gs;  // Neumaier
        if (fabsf(s_t) >= fabsf(gs)) e_t += (s_t - t) + gs;
        else e_t += (gs - t) + s_t;
        s_t = t;
    };
    // adds the masses of chunks U0 <= j < U1
    auto add_chunks = [&](auto u0, auto u1) {
        constexpr int U0 = decltype(u0)::value, U1 = decltype(u1)::value;
        if (RAGGED && all_in) {
            float err;
            add_sum(chunks_expsum_err<DT, U0, U1>(w, a.c, -k_t, err));
            e_t += err;
        } else {
            add_sum(chunks_expsum<DT, U0, U1>(w, a.c, -k_t));
        }
    };
    // the running max of the CTA (a lower bound of the row max at any time)
    auto publish_max = [&](float im, uint32_t *to) {
        const uint32_t wm = __reduce_max_sync(0xffffffffu, fkey(im));
        if (lane == 0 && wm > fkey(-INFINITY)) atomicMax(to, wm);
    };

    // iteration 0 begins with a strided sample (1/8 to 1/16 of a large row,
    // spread over it): chunks u < UCS
    float im, g0, g1;
    load(0);
    {
        uint32_t sm2 = chunk_max2<DT>(w[0]);
#pragma unroll
        for (int u = 1; u < UCS; ++u) sm2 = max2<DT>(sm2, chunk_max2<DT>(w[u]));
        im = max2_value<DT>(sm2);
    }
    // D: how far below the row max the nucleus crossing (top_p = 1: the
    // payload's end) can lie.  Rows of this call that have finished published
    // their depths (in bins of T/4 below their max); the HINT_Q quantile of
    // those depths, plus a margin, sets D (in bins; -1: before HINT_MIN rows
    // have finished, a fixed NSB bins).  One value for the whole CTA.
    if (wid == 0) {
        int inc = hc0 + hc1;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        const float need = HINT_Q * (float)__shfl_sync(0xffffffffu, inc, 31);
        const int hb = (float)(inc - hc1) >= need ? 2 * lane : ((float)inc >= need ? 2 * lane + 1 : NSB);
        const unsigned bal = __ballot_sync(0xffffffffu, hb < NSB);
        const int hq = bal ? __shfl_sync(0xffffffffu, hb, __ffs(bal) - 1) : NSB - 1;
        if (lane == 0) {
            s_dbins = hr >= HINT_MIN ? min(hq + HINT_MARGIN, NSB - 1) + 1 : -1;
            // bfloat16: the sketch-led pass when nearly every finished row was
            // short, and for top_p = 1 (its payload is all that is needed of
            // the row); float32: hinted rows look at their sample too once
            // one row in 16 was handed to the general kernel
            s_skm = BF ? all_in || (hr >= HINT_MIN && (long long)hs * SHORT_DEN >= (long long)hr * SHORT_NUM) : hf > hr / 16;
        }
    }
    publish_max(im, &s_m1);
    if (tid == 0) s_xb = xb0;
    __syncthreads();
    // the sample's max: the same for every warp (later maxima go to another
    // word, as the first warps publish them while the last ones read this)
    const float m1 = fkey_inv(s_m1);
    auto running_max = [&]() -> float { return fmaxf(m1, fkey_inv(*reinterpret_cast<volatile uint32_t *>(&s_mr))); };
    const bool have = m1 > -INFINITY && m1 < INFINITY;
    const int hbins = s_dbins;
    const bool hinted = have && hbins > 0;
    const float D = (float)(hinted ? hbins : NSB) * (a.T / SPB);
    if (!BF) {  // (bfloat16: with the other iterations, below)
        // one reference for all threads (the final one, unless the row max lies
        // outside the sample and across an integer of log2)
        raise_ref(have ? fmaxf(m1, im) : im);
        add_chunks(std::integral_constant<int, 0>(), std::integral_constant<int, UCS>());
    }

    // dependent loads of the accept test, consumed at the end
    float zx = 0.f, qx = 0.f, ux = 0.f;
    int L = 0;
    unsigned long long *ord = nullptr;  // the payload in order (and, when kept, the nucleus)
    int lazy = 0;
    int nnuc = -1;  // nucleus ids written to the row's list (-1: none)
    float m = -INFINITY, kref = -1e30f;
    double S = 0.0;  // (thread 0)
    float v_need = 0.0f;  // the crossing (top_p = 1: the payload's end), for the hints
    bool short_row = false;  // (bfloat16) few ids reach the crossing: published for later rows' pass

    // the nucleus target's range from S, known up to the relative error err (thread 0)
    auto set_target = [&](float err) {
        const double t = (double)a.top_p * S * (double)FX_SCALE;
        s_tg = all_in ? 0ull : (unsigned long long)ceil(t - t * (double)err);
        s_th = all_in ? 0ull : (unsigned long long)ceil(t + t * (double)err);
    };
    // every mass was summed against the final reference kref: the one of the
    // sample's max, with which all threads start
    auto one_ref = [&]() { return have && kref == ceilf(m1 * a.c); };
    // reduces the row max, the reference and the exp-sum S (fp32 two-sum tree,
    // fp64 in thread 0 only, which also leaves the nucleus target in s_tg and
    // s_th: valid after the next barrier); true when the row is not a
    // distribution (handled)
    auto finish_sums = [&]() -> bool {
        if (a.K > 0) {
            bq = r / (a.K + 1);
            iq = r % (a.K + 1);
        }
        xb = tid == 0 ? s_xb : -1;
        if (xb >= 0 && xb < a.V) {
            zx = E::load1(row + rc.head * E::SIZE, xb);
            qx = __ldg(a.q + ((size_t)bq * a.K + iq) * a.V + xb);
            ux = __ldg(a.u + (size_t)bq * (a.K + 1) + iq);
        }
        // each warp: its max, reference kw and exp-sum in units of 2^kw (a
        // compensated fp32 tree over rescales by exact powers of two)
        {
            const float mw = warp_max(m_t), kw = warp_max(k_t);
            const float f = pow2_int(fmaxf(k_t - kw, -1000.0f));
            float hi = s_t * f, lo = e_t * f;
            for (int o = 16; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
                const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
                float sm, er;
                two_sum(hi, h2, sm, er);
                lo = lo + l2 + er;
                hi = sm;
            }
            if (lane == 0) {
                redf[wid] = mw;
                redk[wid] = kw;
                redh[wid] = hi;
                redl[wid] = lo;
            }
        }
        __syncthreads();
        // every thread combines the warps' parts (fp64, exact rescales)
        // (fp32 two-sums over exact power-of-two rescales: fp64 is slow here)
        float sh = 0.0f, sl = 0.0f;
        if constexpr (NWC <= 8) {
            m = redf[0];
            kref = redk[0];
#pragma unroll
            for (int i = 1; i < NWC; ++i) {
                m = fmaxf(m, redf[i]);
                kref = fmaxf(kref, redk[i]);
            }
#pragma unroll
            for (int i = 0; i < NWC; ++i) {
                const float f = pow2_int(fmaxf(redk[i] - kref, -1000.0f));  // (an integer <= 0)
                float sm, er;
                two_sum(sh, redh[i] * f, sm, er);
                sl += er + redl[i] * f;
                sh = sm;
            }
        } else {  // one warp's part per lane, the same tree in every warp
            const int i = lane % NWC;
            m = warp_max(redf[i]);
            kref = warp_max(redk[i]);
            const float f = pow2_int(fmaxf(redk[i] - kref, -1000.0f));
            sh = redh[i] * f;
            sl = redl[i] * f;
            for (int o = NWC / 2; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, sh, o);
                const float l2 = __shfl_xor_sync(0xffffffffu, sl, o);
                float sm, er;
                two_sum(sh, h2, sm, er);
                sl = sl + l2 + er;
                sh = sm;
            }
        }
        if (tid == 0) {
            S = (double)sh + (double)sl;
            set_target(EXACT_CUT ? (one_ref() ? a.add_err : a.sum_err) : 0.0f);
        }
        if (!(sh > 0.0f && sh < INFINITY) || !(m < INFINITY) || !(kref < 1e30f)) {
            nonfinite_row<NTC>(a, r);
            defer_draw(a, row_finished<DT, NTC>(a, r, smem));
            return true;
        }
        return false;
    };
    // replaces S (thread 0) and the target by those of the row's exact mass
    // (all threads)
    bool exact_S = false, sharp = false;
    auto make_exact = [&]() {
        const unsigned long long fx = exact_mass<DT, NTC, RAGGED>(rc.row(), a.V, a.c, kref, s_redu);
        if (tid == 0) {
            S = (double)fx * FX_INV;
            s_tg = s_th = all_in ? 0ull : (unsigned long long)ceil((double)a.top_p * (double)fx);
        }
        __syncthreads();
        exact_S = true;
    };
    // the cut lies inside the target's range: the range that a nucleus of n ids
    // leaves, then the exact target (all threads)
    auto sharpen = [&](int n) {
        __syncthreads();  // (the range has been read)
        if (sharp || one_ref()) {
            make_exact();
            return;
        }
        sharp = true;
        if (tid == 0) set_target(sharp_err(a.sum_err, a.top_p, n, a.V, (float)S));
        __syncthreads();
    };
    // hands the row to the general kernel (all threads), whose value histogram
    // takes S from here
    auto hand_over = [&]() {
        if (BF && RAGGED && !all_in && !exact_S) make_exact();
        if (tid == 0) fallback_row(a, r, m, kref, S);
    };

    if constexpr (BF) {
        // ================= bfloat16: value counts and sketch =================
        // Every id >= lim(running max) is counted in the window of HW values
        // [thb0, thb0 + HW) (positive bit patterns, which sort like the
        // values); the running max only rises, so at the end every id >=
        // lim(row max) has been counted.  The sketch keeps the max of every
        // group of chunks (4 or 8 chunks of one thread and iteration, or 8
        // chunks of 2^ish iterations).
        uint32_t thb0 = 1u;
        bool count_on = false;
        // (the sketch-led pass keeps its work areas past a sketch of at most
        // SK_TMP * 4 slots)
        const int sk_slots = a.sk_gpi == 2 ? nit * NTC * 2 : ((nit + (1 << a.sk_ish) - 1) >> a.sk_ish) * NTC;
        const bool skm = s_skm != 0 && sk_slots <= SK_TMP * 4;
        if (EXACT_CUT && have) raise_ref(m1);  // (one reference for all threads)
        if (have && m1 > 0.0f && !skm) {
            const float t = m1 - D;
            int lo = t > 0.0f ? (int)__bfloat16_as_ushort(__float2bfloat16_rd(t)) : 1;
            lo = max(lo, (int)(__float_as_uint(m1) >> 16) + HEADROOM - (HW - 1));
            lo = max(lo, 1);
            if (lo + HW - 1 <= 0x7F7F) {  // (then negative values, inf and NaN fall outside)
                count_on = true;
                thb0 = (uint32_t)lo;
            }
        }
        auto lim_of = [&](float mr) -> uint32_t {
            const float t = mr - D;
            uint32_t b = t > 0.0f ? (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rd(t)) : 0u;
            b = b > thb0 ? b : thb0;
            return b < thb0 + HW ? b : thb0 + HW;
        };
        // counts the ids of a chunk that reach value thb in the counters of
        // values thb0 ... (no id of it lies above the window)
        auto count_chunk = [&](const uint4 &ch, uint32_t thb) {
            const uint32_t wd[4] = {ch.x, ch.y, ch.z, ch.w};
            // (the counts' shared-memory address, offset so that a value's
            // float bits >> 14, its bfloat16 pattern times 4, index its counter)
            const int hbase = (int)__cvta_generic_to_shared(hist) - (int)thb0 * 4;
            const int dummy = hbase + (int)thb * 4 - 4 - 4 * lane;
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
                const int v = (int)((e & 1) ? wd[e >> 1] & 0xFFFF0000u : wd[e >> 1] << 16);
                const int at = max((v >> 14) + hbase, dummy);
#ifdef ACES_CHECKED
                if (ACES_IN((at - hbase) / 4 - (int)thb0 + HPAD, HPAD + HW)) red_inc(at);
#else
                red_inc(at);
#endif
            }
        };
        const uint32_t topp = (thb0 + HW) | (thb0 + HW) << 16;  // the value above the window (at most +inf)
        const __nv_bfloat162 top2 = *reinterpret_cast<const __nv_bfloat162 *>(&topp);
        const int gpi = a.sk_gpi, ish = a.sk_ish;
        float gacc = -INFINITY;
        // the sketch holds bfloat16 bit patterns (as signed 16-bit integers
        // those of positive values sort like the values, above all others)
        auto sketch_put = [&](int it) {
            if (gpi == 2) {
                const int s2 = it * NTC + tid;
                if (ACES_IN(2 * s2 + 1, SKG))
                    reinterpret_cast<uint32_t *>(sk)[s2] = __byte_perm(__float_as_uint(g0), __float_as_uint(g1), 0x7632);
            } else {
                gacc = fmaxf(gacc, fmaxf(g0, g1));
                if (((it + 1) & ((1 << ish) - 1)) == 0 || it == nit - 1) {
                    const int s1 = (it >> ish) * NTC + tid;
                    if (ACES_IN(s1, SKG)) sk[s1] = (uint16_t)(__float_as_uint(gacc) >> 16);
                    gacc = -INFINITY;
                }
            }
        };
        // The counting loop is bound by issue slots: 14.3 warp instructions
        // per 32 logits on flat rows (whole kernel, ncu; 20.5 with a predicated
        // reduction, maxima per chunk and a divided tile order), 224 us against
        // 282 us for the call on 128 x 17 rows of 128256.  Without counting it
        // is 7.2 (8.7): there HBM and the row's other phases bound it, and
        // fewer instructions still (or L2 prefetches of the next iterations or
        // of the row one wave on) change nothing.
        auto stream = [&](auto counting) {
            constexpr bool COUNT = decltype(counting)::value;
            for (int it = 0; it < nit; ++it) {
                uint32_t thb = 0u;
                if (it > 0) {  // (iteration 0 is loaded)
                    off0 = wrap(off0 + off_it);
                    load(it);
                }
                if (COUNT) thb = lim_of(running_max());
                const uint32_t im2 = group_maxima<DT>(w, g0, g1);
                im = fmaxf(g0, g1);
                raise_ref(im);
                if (COUNT) publish_max(im, &s_mr);
                uint32_t any = 0u;  // chunk positions where some lane of the warp reaches thb
                if (COUNT) {
                    uint32_t hb = 0u;
                    const uint32_t thp = thb | thb << 16;
                    const __nv_bfloat162 t2 = *reinterpret_cast<const __nv_bfloat162 *>(&thp);
#pragma unroll
                    for (int u = 0; u < UC; ++u) {
                        const uint32_t cm = chunk_max2<DT>(w[u]);
                        hb |= (uint32_t)(__hge2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&cm), t2) != 0u) << u;
                    }
                    // a value above the window (the row is counted again) or a
                    // NaN (it is not a distribution): this iteration need not
                    // be counted, nor may it be
                    if (__hlt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&im2), top2) != 0xFFFFFFFFu) hb |= 1u << UC;
                    any = __reduce_or_sync(0xffffffffu, hb);
                    if (any >> UC) any = 0u;
                }
                if (RAGGED && all_in) {
#pragma unroll
                    for (int u = 0; u < UC; ++u)
                        if (COUNT && ((any >> u) & 1u)) count_chunk(w[u], thb);  // (warp-uniform)
                    add_chunks(std::integral_constant<int, 0>(), std::integral_constant<int, UC>());
                } else {
                    const unsigned long long c2 = pack2(a.c, a.c), nk2 = pack2(-k_t, -k_t);
                    unsigned long long acc0 = 0ull, acc1 = 0ull;
#pragma unroll
                    for (int u = 0; u < UC; ++u) {
                        if (COUNT && ((any >> u) & 1u)) count_chunk(w[u], thb);
                        acc_pair(u, chunk_expsum2<DT>(w[u], c2, nk2), acc0, acc1);
                    }
                    add_sum(acc_total(acc0, acc1));
                }
                sketch_put(it);
            }
        };
        if (count_on) stream(std::true_type());
        else stream(std::false_type());
        if (finish_sums()) return;
        const uint32_t km = __float_as_uint(m) >> 16;
        if (a.force_fb || !(m > 0.0f)) {
            hand_over();
            return;
        }
        auto vmass = [&](int idx) { return id_fx(val16(0x8000u + thb0 + (uint32_t)idx), a.c, kref); };
        // ---- the crossing, the payload's end and the values to re-read,
        // from the counts of values thc..m (all threads, VPT consecutive
        // values each, from the top).  Returns 0, or 1 when they lie below
        // the counted values, 2 when more ids than the re-read keeps share
        // the payload's last value (scan_once: 3 when the cut depends on the
        // error of S) ----
        // (L, vs, vr, j, n_nuc and nge are set when it returns 0)
        int vs = -1, vr = -1, j = 0, n_nuc = -1, nge = 0;
        auto scan_once = [&](uint32_t thc) -> int {
            constexpr int VPT = HW / NTC;
            const int top = (int)(km - thb0) - VPT * tid, lo = (int)(thc - thb0);
            uint32_t cn[VPT];
            unsigned long long e1[VPT], lm = 0ull;
            uint32_t lc = 0u;
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                cn[i] = top - i >= lo ? hist[top - i] : 0u;
                e1[i] = cn[i] ? vmass(top - i) : 0ull;
                lm += (unsigned long long)cn[i] * e1[i];
                lc += cn[i];
            }
            unsigned long long incm = lm;
            uint32_t incc = lc;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long tm = __shfl_up_sync(0xffffffffu, incm, o);
                const uint32_t tc = __shfl_up_sync(0xffffffffu, incc, o);
                if (lane >= o) {
                    incm += tm;
                    incc += tc;
                }
            }
            if (lane == 31) {
                s_redu[wid] = incm;
                s_redc[wid] = incc;
            }
            if (tid == 0) {
                s_vs = -1;
                s_j = 0;
                s_cab = s_cnvs = 0u;
                s_above = s_evs = 0ull;
            }
            __syncthreads();
            uint32_t totc = 0u;
#pragma unroll
            for (int i = 0; i < NWC; ++i) {
                if (i < wid) {
                    incm += s_redu[i];
                    incc += s_redc[i];
                }
                totc += s_redc[i];
            }
            const unsigned long long exm = incm - lm, tg = s_tg;
            const uint32_t exc = incc - lc;
            if (!all_in && exm < tg && incm >= tg) {  // (at most one thread)
                unsigned long long cm = exm;
                uint32_t cc = exc;
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const unsigned long long mm = (unsigned long long)cn[i] * e1[i];
                    if (cm < tg && cm + mm >= tg) {
                        s_vs = top - i;
                        s_above = cm;
                        s_cab = cc;
                        s_cnvs = cn[i];
                        s_evs = e1[i];
                        // the fewest ids of this value reaching the target
                        const unsigned long long rem = tg - cm;
                        unsigned long long q = (unsigned long long)((float)rem / (float)e1[i]);
                        while (q * e1[i] < rem) ++q;
                        while (q > 1ull && (q - 1ull) * e1[i] >= rem) --q;
                        s_j = (int)q;
                        s_settled = cm + q * e1[i] >= s_th;
                    }
                    cm += mm;
                    cc += cn[i];
                }
            }
            const uint32_t ku = (uint32_t)a.k;
            if (exc < ku && incc >= ku) {  // the value of the k-th id (one thread)
                unsigned long long cm = exm;
                uint32_t cc = exc;
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    if (cc < ku && cc + cn[i] >= ku) {
                        s_vk = top - i;
                        s_nge = (int)(cc + cn[i]);
                        s_cumL_fx = cm + (unsigned long long)(ku - cc) * e1[i];
                    }
                    cm += (unsigned long long)cn[i] * e1[i];
                    cc += cn[i];
                }
            }
            __syncthreads();
            // (the same in every thread)
            vs = s_vs;
            j = s_j;
            if (!all_in && vs < 0) return 1;
            if (EXACT_CUT && !all_in && !s_settled) return 3;
            const uint32_t nn = all_in ? (uint32_t)a.V : s_cab + (uint32_t)j;  // (at most V)
            const unsigned long long nuc = s_above + (unsigned long long)j * s_evs;
            n_nuc = all_in ? -1 : (int)nn;
            L = min((int)nn, a.k);
            if ((uint32_t)L > totc) return 1;  // (top_p = 1) the payload reaches below them
            // the values to re-read: down to the crossing value when the
            // nucleus is short (then it is kept and the cut is exact), else
            // down to the payload's last value
            vr = -1;
            if (!all_in && s_cab + s_cnvs <= (uint32_t)PCAP && nn <= (uint32_t)NUC_CAP) {
                vr = vs;
                nge = (int)(s_cab + s_cnvs);
            } else if (L > 0) {
                const bool at_k = all_in || nn > ku;  // else the payload ends with the nucleus, at vs
                vr = at_k ? s_vk : vs;
                nge = at_k ? s_nge : (int)(s_cab + s_cnvs);
                if (nge > PCAP) return 2;
            }
            if (tid == 0) {  // (read after later barriers)
                if (!all_in && nn <= ku) s_cumL_fx = nuc;
                if (ku == 0u) s_cumL_fx = 0ull;
                s_Snuc = all_in ? S : (double)nuc * FX_INV;
                s_inv_S = inv_mass(s_Snuc);
            }
            return 0;
        };
        auto scan = [&](uint32_t thc) -> int {
            for (;;) {
                const int f = scan_once(thc);
                if (f != 3) return f;
                // (then it is settled; a sharper range first, as for float32 rows, costs
                // more than it saves here)
                __syncthreads();
                make_exact();
            }
        };
        // ---- reading groups of the sketch back ----
        const int ng_all = gpi == 2 ? nit * NTC * 2 : ((nit + (1 << ish) - 1) >> ish) * NTC;
        // cnt items of each lane get consecutive places from *ctr (one atomic
        // per warp); returns the lane's first place (all lanes of the warp)
        auto warp_place = [&](int cnt, int *ctr) -> int {
            int inc = cnt;
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            int base = 0;
            if (lane == 31 && inc > 0) base = atomicAdd(ctr, inc);
            return __shfl_sync(0xffffffffu, base, 31) + inc - cnt;
        };
        // lists in gl the slots whose group max reaches the positive value of
        // bit pattern vb; returns their count (all threads)
        auto compact = [&](uint32_t vb, uint32_t *gl) -> int {
            if (tid == 0) s_ng = 0;
            __syncthreads();
            // this thread's slots: pairs 2 (i * NTC + tid) + {0, 1}, bits 2 i and
            // 2 i + 1 (at most 64 slots; without pairs slot i * NTC + tid)
            unsigned long long hm = 0ull;
            if (gpi == 2) {
                for (int i = 0; i < nit; ++i) {
                    const int s2 = i * NTC + tid;
                    const uint32_t g = ACES_IN(2 * s2 + 1, SKG) ? reinterpret_cast<const uint32_t *>(sk)[s2] : 0u;
                    if ((int)(g << 16) >= (int)(vb << 16)) hm |= 1ull << (2 * i);
                    if ((int)g >= (int)(vb << 16)) hm |= 2ull << (2 * i);
                }
            } else {
                for (int i = 0; i < ng_all / NTC; ++i) {
                    const int slot = i * NTC + tid;
                    if (ACES_IN(slot, SKG) && (int)(int16_t)sk[slot] >= (int)vb) hm |= 1ull << i;
                }
            }
            int at = warp_place(__popcll(hm), &s_ng);
            __syncthreads();  // (gl may overlap slots of the sketch read above)
            while (hm) {
                const int i = __ffsll((long long)hm) - 1;
                hm &= hm - 1ull;
                const int slot = gpi == 2 ? 2 * ((i >> 1) * NTC + tid) + (i & 1) : i * NTC + tid;
                if (at < GCAP && ACES_IN(at, GCAP)) gl[at] = (uint32_t)slot;
                ++at;
            }
            __syncthreads();
            return s_ng;
        };
        // reads the ng groups of gl (one per thread, four chunks at a time) and
        // hands every id whose bit pattern is >= vb (> 0) to put(place, bits,
        // id), places counted by *ctr
        auto reread = [&](const uint32_t *gl, int ng, uint32_t vb, int *ctr, auto put) {
            const int cpt = gpi == 2 ? UC / 2 : UC << ish;  // chunks per group
            for (int g0i = 0; g0i < ng; g0i += NTC) {      // warp-uniform rounds
                const int gi = g0i + tid;
                const bool has = gi < ng;
                const uint32_t slot = has ? gl[gi] : 0u;
                const int tl = gpi == 2 ? (int)((slot >> 1) % NTC) : (int)(slot % NTC);
                const int itg = gpi == 2 ? (int)((slot >> 1) / NTC) : (int)((slot / NTC) << ish);
                const int ub = gpi == 2 ? (int)(slot & 1u) * (UC / 2) : 0;
                for (int q0 = 0; q0 < cpt; q0 += 4) {
                    uint4 dat[4];
                    int cc[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int q = q0 + h;
                        const int it = itg + q / UC, u = ub + q % UC;
                        const int t = it * TPI + u * NWC + (tl >> 5);
                        cc[h] = -1;
                        if (has && it < nit && t < ntile) {
                            const int c = (int)((long long)t * a.pstride % ntile) * TCH + (tl & 31);
                            if (c < nch) cc[h] = c;
                        }
                        dat[h] = cc[h] >= 0 ? rc.load(cc[h]) : make_uint4(NI, NI, NI, NI);
                    }
                    uint32_t hm = 0u;
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const uint32_t wd[4] = {dat[h].x, dat[h].y, dat[h].z, dat[h].w};
#pragma unroll
                        for (int e = 0; e < EPC; ++e) {
                            const uint32_t bits = (e & 1) ? wd[e >> 1] >> 16 : wd[e >> 1] & 0xFFFFu;
                            hm |= (uint32_t)(bits - vb < 0x8000u - vb) << (h * EPC + e);
                        }
                    }
                    int at = warp_place(__popc(hm), ctr);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t m8 = (hm >> (h * EPC)) & 0xFFu;
                        while (m8) {
                            const int e = __ffs(m8) - 1;
                            m8 &= m8 - 1u;
                            put(at, __float_as_uint(chunk_elem<DT>(dat[h], e)) >> 16, (uint32_t)(cc[h] * EPC + e - rc.head));
                            ++at;
                        }
                    }
                }
            }
            __syncthreads();
        };
        auto put_pay = [&](int at, uint32_t bits, uint32_t id) {
            if (at < PCAP && ACES_IN(at, PCAP)) pay[at] = order_val(fkey(__uint_as_float(bits << 16)), id);
        };
        // ---- sketch-led pass (rows of a call whose finished rows were
        // short; nothing was counted while streaming).  Every id >= the
        // hinted window's lower end thb0 (row max - D) lies in a group whose
        // max reaches thb0: those groups are read back, their ids >= thb0
        // counted and kept, and the scan of those exact counts follows.
        // Returns 0 (pay holds the ids >= the scan's vr), 1 when the second
        // counting pass is needed, 2 when the row goes to the general kernel ----
        auto sketch_led = [&]() -> int {
            {
                const float t = m - D;
                const uint32_t lb = t > 0.0f ? (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rd(t)) : 1u;
                const uint32_t kfull = km > (uint32_t)(HW - 1) ? km - (uint32_t)(HW - 1) : 1u;
                thb0 = lb > kfull ? lb : kfull;
                if (all_in) {
                    // top_p = 1: the k-th largest group max, from counts of the
                    // sketch's values, is at or below the k-th id, and only the
                    // groups that reach it are read back.  (The hinted depth D
                    // spans too many groups on flat rows: 133 of 160 rows of
                    // 102400 were counted in a second pass, 10 us a row.)
                    thb0 = kfull;
                    auto add = [&](int v) {
                        const int i = v - (int)kfull;
                        if (i >= 0 && ACES_IN(i, HW)) atomicAdd(&hist[i], 1u);
                    };
                    for (int i = tid; i < (gpi == 2 ? ng_all / 2 : ng_all); i += NTC) {
                        if (gpi == 2) {
                            const uint32_t g = reinterpret_cast<const uint32_t *>(sk)[i];
                            add((int)(int16_t)(g & 0xFFFFu));
                            add((int)g >> 16);
                        } else {
                            add((int)(int16_t)sk[i]);
                        }
                    }
                    __syncthreads();
                    if (scan(kfull) != 0) return 1;  // (fewer than k groups reach the window, or far too many tie)
                    thb0 = vr >= 0 ? kfull + (uint32_t)vr : km;  // (k = 0: nothing but the max)
                    for (int i = tid; i < HW; i += NTC) hist[i] = 0u;
                    __syncthreads();
                }
            }
            uint32_t *gls = reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned long long *>(sk) + SK_TMP);
            const int nc = compact(thb0, gls);  // (ends with a barrier)
            if (nc > GCAP) return 1;
            if (tid == 0) s_npay = 0;
            __syncthreads();
            reread(gls, nc, thb0, &s_npay, [&](int at, uint32_t bits, uint32_t id) {  // (hist is clear)
                const uint32_t idx = bits - thb0;
                if (idx < (uint32_t)HW) atomicAdd(&hist[idx], 1u);
                if (at < PCAP && ACES_IN(at, PCAP)) pay[at] = order_val(fkey(__uint_as_float(bits << 16)), id);
            });
            const int nall = s_npay;
            if (nall > PCAP) return 1;
            if (tid == 0) s_ng = 0;  // (the scan's barriers come before its next use)
            const int f = scan(thb0);
            if (f != 0) return f;
            // keep in pay the ids >= the scan's vr
            if (vr >= 0) {
                const uint32_t kr = fkey(val16(0x8000u + thb0 + (uint32_t)vr));
                unsigned long long *tmp = reinterpret_cast<unsigned long long *>(sk) + SK_TMP;
                for (int i0 = 0; i0 < nall; i0 += NTC) {  // warp-uniform rounds
                    const int i = i0 + tid;
                    const unsigned long long o = i < nall ? pay[i] : 0ull;
                    const bool keep = i < nall && (uint32_t)(o >> 32) >= kr;
                    const int at = warp_place(keep ? 1 : 0, &s_ng);
                    if (keep && ACES_IN(at, PCAP)) tmp[at] = o;
                }
                __syncthreads();
                const int nk = s_ng;
                for (int i = tid; i < nk; i += NTC)
                    if (ACES_IN(i, PCAP)) pay[i] = tmp[i];
                __syncthreads();
            }
            return 0;
        };
        int fb = 1;
        bool pay_ready = false;  // (sketch-led) pay holds the ids >= vr
        if (skm) {
            fb = sketch_led();
            pay_ready = fb == 0;
            if (tid == 0 && fb == 0) atomicAdd(&a.ws.fb_count[12], 1);
        } else if (count_on && km < thb0 + HW) {
            fb = scan(lim_of(m));
        }
        if (fb == 1) {
            // the crossing (or the row max) lies outside the counted values:
            // a second pass counts the row again, from the row max down as far
            // as the window reaches
            thb0 = km > (uint32_t)(HW - 1) ? km - (uint32_t)(HW - 1) : 1u;
            for (int i = tid; i < HW; i += NTC) hist[i] = 0u;
            __syncthreads();
            for (int c0 = 0; c0 < nch; c0 += NTC * UC) {
#pragma unroll
                for (int u = 0; u < UC; ++u) {
                    const int c = c0 + u * NTC + tid;
                    w[u] = c < nch ? rc.load(c) : make_uint4(NI, NI, NI, NI);
                }
#pragma unroll
                for (int u = 0; u < UC; ++u) count_chunk(w[u], thb0);
            }
            __syncthreads();
            if (tid == 0) atomicAdd(&a.ws.fb_count[10], 1);
            fb = scan(thb0);
        }
        if (fb != 0) {
            hand_over();
            return;
        }
        const uint32_t vsb = thb0 + (uint32_t)vs;  // crossing value (bit pattern)
        const bool exact = !all_in && vr == vs;    // every id of the crossing value is read below
        if (vr >= 0) {
            // ---- the ids at or above value vr, then ordered ----
            const uint32_t vrb = thb0 + (uint32_t)vr;  // its bit pattern
            if (!pay_ready) {
                const int ng = compact(vrb, glist);
                if (ng > GCAP) {
                    hand_over();
                    return;
                }
                if (tid == 0) s_npay = 0;
                __syncthreads();
                reread(glist, ng, vrb, &s_npay, put_pay);
            }
            const int npay = pay_ready ? s_ng : s_npay;
            if (npay != nge) {  // (cannot happen: the counts and the ids agree)
                hand_over();
                return;
            }
            // order them (descending order value)
            if (npay <= RANK_MAX) {
                ord = sorted;
                // (the value in the window, then the lower id: 30 bits)
                for (int i = tid; i < ((npay + 3) & ~3); i += NTC) {
                    const unsigned long long o = i < npay ? pay[i] : 0ull;
                    const uint32_t idx = (__float_as_uint(order_value(o)) >> 16) - thb0;
                    hist[i] = i < npay ? (idx << 20 | (0xFFFFFu - order_id(o))) + 1u : 0u;
                }
                __syncthreads();
                for (int i = tid; i < npay; i += NTC) {
                    const int rank = count_above<false>(hist, npay, hist[i], nullptr);
                    if (ACES_IN(rank, PCAP)) ord[rank] = pay[i];
                }
            } else {
                if (tid == 0) atomicAdd(&a.ws.fb_count[3], 1);
                ord = pay;
                const int np = next_pow2(npay);
                for (int i = npay + tid; i < np; i += NTC)
                    if (ACES_IN(i, PCAP)) pay[i] = 0ull;
                __syncthreads();
                bitonic_sort_desc(pay, np);
            }
            __syncthreads();
        }
        if (tid == 0) {
            if (all_in) {
                s_cut = 0ull;
            } else if (exact) {
                s_cut = ord[n_nuc - 1];
            } else {
                s_cut = ((unsigned long long)fkey(val16(0x8000u + vsb)) << 32) | (unsigned long long)(uint32_t)j;
                atomicAdd(&a.ws.fb_count[5], 1);
            }
            s_zx = zx;
            s_xb = xb;
        }
        // keep the nucleus for the residual step when it fits
        if (exact && a.ws.nuc != nullptr && n_nuc <= NUC_CAP) {
            for (int i = tid; i < n_nuc; i += NTC)
                if (ACES_IN(i, NUC_CAP)) a.ws.nuc[(size_t)r * NUC_CAP + i] = ord[i];
            nnuc = n_nuc;
        }
        lazy = !all_in && !exact;
        __syncthreads();
        // the draft token's value equals the crossing value and that value's
        // ids were not read: its rank among them (ids below it) decides
        if (lazy && s_xb >= 0 && s_xb < a.V && key16(__float_as_uint(s_zx) >> 16) == 0x8000u + vsb) {
            const int xr = s_xb + rc.head;  // (a position in chunks)
            const float vsv = val16(0x8000u + vsb);
            const __nv_bfloat162 v2 = __floats2bfloat162_rn(vsv, vsv);
            uint32_t cnt = 0u;
            for (int cc = tid; cc * EPC < xr; cc += NTC) {
                const uint4 wv = rc.load(cc);
                const uint32_t wd[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t mk = __heq2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&wd[q]), v2);
                    const int x0 = cc * EPC + 2 * q;
                    cnt += ((mk & 1u) && x0 < xr) + ((mk >> 16 & 1u) && x0 + 1 < xr);
                }
            }
            const unsigned long long below = block_reduce_n<NTC>((unsigned long long)cnt, s_redu, SumU64());
            if (tid == 0) {
                atomicAdd(&a.ws.fb_count[7], 1);
                // x~ is in the nucleus iff fewer than j ids of its value precede it
                zx = below < (unsigned long long)j ? vsv : -INFINITY;
            }
        }
        v_need = all_in ? (L > 0 ? order_value(ord[L - 1]) : m) : val16(0x8000u + vsb);
        short_row = all_in ? a.k <= SHORT_IDS : (n_nuc >= 0 && n_nuc <= SHORT_IDS);
        if (tid == 0) atomicAdd(&a.ws.fb_count[2], 1);
    } else {
        // ================= float32: list mode =================
        // Chunks holding an id >= the capture threshold are recorded (16-byte
        // chunk and index).  Hinted rows: the threshold is the running max
        // minus D, so at the end every id >= (row max - D) was recorded.
        // The first rows, and those whose sample says that D would list more
        // than the areas hold: the sample's ids within NSB bins of its max are
        // binned; the bins where the sample's mass (from the exact exp-sums)
        // reaches top_p and where its count reaches nmin set a fixed
        // threshold, MARGIN_BINS lower where the areas hold that many.
        float thlo = INFINITY;
        bool by_depth = hinted;
        if (!hinted || s_skm) {
            if (have) {
#pragma unroll
                for (int u = 0; u < UCS; ++u) {
                    const float cmx = max2_value<DT>(chunk_max2<DT>(w[u]));
                    if (!__any_sync(0xffffffffu, (m1 - cmx) * a.inv_ws < (float)NSB)) continue;
#pragma unroll 1  // (unrolled, the independent atomics spill registers)
                    for (int e = 0; e < EPC; ++e) {
                        const float d = (m1 - chunk_elem<DT>(w[u], e)) * a.inv_ws;
                        if (d < (float)NSB && ACES_IN((int)d, NSB)) atomicAdd(&sbin[wid][(int)d], 1u);
                    }
                }
            }
            // the sample's mass in units of 2^((z - m1) c)
            {
                const float kw = warp_max(k_t);
                float sw = (s_t + e_t) * pow2_int(fmaxf(k_t - kw, -1000.0f));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sw += __shfl_xor_sync(0xffffffffu, sw, o);
                if (lane == 0) redh[wid] = have ? sw * ex2(kw - m1 * a.c) : 0.0f;
            }
            __syncthreads();
            if (wid == 0 && have) {
                uint32_t c0 = 0u, c1 = 0u;
                float M = 0.0f;
#pragma unroll
                for (int i = 0; i < NWC; ++i) {
                    if (2 * lane < NSB) c0 += sbin[i][2 * lane];
                    if (2 * lane + 1 < NSB) c1 += sbin[i][2 * lane + 1];
                    M += redh[i];
                }
                constexpr float L2B = 1.4426950408889634f / SPB;
                const float ms0 = (float)c0 * ex2(-(2 * lane + 0.5f) * L2B), ms1 = (float)c1 * ex2(-(2 * lane + 1.5f) * L2B);
                float pm = ms0 + ms1;
                uint32_t pc = c0 + c1;
                for (int o = 1; o < 32; o <<= 1) {
                    const float tm = __shfl_up_sync(0xffffffffu, pm, o);
                    const uint32_t tc = __shfl_up_sync(0xffffffffu, pc, o);
                    if (lane >= o) {
                        pm += tm;
                        pc += tc;
                    }
                }
                const float pm0 = pm - ms1, pc0f = (float)(pc - c1);  // cumulative through bin 2*lane
                const float f = a.samp_frac;
                // first bin whose cumulative reaches a target (NSB when none)
                auto first_bin = [&](bool h0, bool h1) -> int {
                    const int hb = h0 ? 2 * lane : (h1 ? 2 * lane + 1 : NSB);
                    const unsigned bal = __ballot_sync(0xffffffffu, hb < NSB);
                    return bal ? __shfl_sync(0xffffffffu, hb, __ffs(bal) - 1) : NSB;
                };
                auto bin_of_count = [&](float n) { return first_bin(pc0f >= n * f, (float)pc >= n * f); };
                // the first bin where the areas would be LIST_FILL full
                const int bfull = bin_of_count(LIST_FILL * (float)LCAP);
                int blo;
                if (all_in) {
                    blo = bin_of_count((float)a.nmin);
                } else {
                    const float tm = a.top_p * M;
                    const int bx = first_bin(pm0 >= tm, pm >= tm);
                    blo = max(max(min(bx + MARGIN_BINS, bfull - 1), bx + 1), bin_of_count((float)a.nmin));
                }
                blo = min(blo, NSB - 1);
                if (lane == 0) {
                    s_thlo = m1 - (float)(blo + 1) * (a.T / SPB);
                    s_fb = hinted && hbins - 1 < bfull;
                }
            }
            __syncthreads();
            if (have) {
                thlo = s_thlo;
                by_depth = s_fb != 0;
            }
        }
        // records the chunks in hb (those holding an id >= the capture
        // threshold): one vote per iteration, one warp-aggregated atomic per
        // chunk position that has any; the ids are extracted after the stream
        auto record_hits = [&](float th) {
            if (!__any_sync(0xffffffffu, im >= th)) return;
            // (past the capacity the row goes to the general kernel; the counter
            // changes meanwhile, so one lane's reading decides for its warp)
            if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile int *>(&s_nrec), 0) > CREC) return;
            uint32_t off = off0;
#pragma unroll
            for (int u = 0; u < UC; ++u) {
                const bool hit = max2_value<DT>(chunk_max2<DT>(w[u])) >= th;
                const unsigned bal = __ballot_sync(0xffffffffu, hit);
                if (bal != 0u) {
                    const int lead = __ffs(bal) - 1;
                    int base = 0;
                    if (lane == lead) base = atomicAdd(&s_nrec, __popc(bal));
                    base = __shfl_sync(0xffffffffu, base, lead);
                    if (hit) {
                        const int at = base + __popc(bal & ((1u << lane) - 1u));
                        if (at < CREC && ACES_IN(at, CREC)) {
                            rec_dat[at] = w[u];
                            rec_idx[at] = off >> 4;
                        }
                    }
                }
                off = wrap(off + off_w);
            }
        };
        {
            float th = by_depth ? m1 - D : thlo;
            for (int it = 0; it < nit; ++it) {
                if (it > 0) {  // (iteration 0 is loaded, its sample summed)
                    off0 = wrap(off0 + off_it);
                    load(it);
                    if (by_depth) th = running_max() - D;
                }
                if (it > 0 || UCS < UC) {
                    group_maxima<DT>(w, g0, g1);
                    im = fmaxf(g0, g1);
                    raise_ref(im);
                    if (it > 0) add_chunks(std::integral_constant<int, 0>(), std::integral_constant<int, UC>());
                    else add_chunks(std::integral_constant<int, UCS == UC ? 0 : UCS>(), std::integral_constant<int, UC>());
                    if (by_depth) publish_max(im, &s_mr);
                }
                record_hits(th);
            }
        }
        if (finish_sums()) return;
        const int nrec = s_nrec;
        if (a.force_fb || nrec > CREC) {
            hand_over();
            return;
        }
        const float thc = by_depth ? m - D : thlo;  // every id >= thc was recorded
        // expand the records: the ids >= thc of every recorded chunk (all such
        // ids lie in recorded chunks), as 64-bit order values
        if (tid == 0) s_nl = 0;
        __syncthreads();
        for (int i0 = 0; i0 < nrec; i0 += NTC) {  // warp-uniform rounds
            const int i = i0 + tid;
            const bool in = i < nrec;
            const uint4 dat = in ? rec_dat[i] : make_uint4(NI, NI, NI, NI);
            const uint32_t base = in ? rec_idx[i] * (uint32_t)EPC - (uint32_t)rc.head : 0u;
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
                const float v = Elem<DT>::get(dat, e);
                append_cap(list, &s_nl, in && v >= thc, order_val(fkey(v), base + (uint32_t)e), LCAP);
            }
        }
        __syncthreads();
        const int nl = s_nl;
        if (nl > LCAP) {
            hand_over();
            return;
        }
        // counts of the listed ids in bins of T/8 below m; a bin's ids each
        // carry at least its lower edge's mass, so the first bin where that
        // lower bound of the cumulative mass reaches the target holds or
        // follows the crossing (top_p = 1: the first bin where the count
        // reaches k).  The exact crossing is found below among the ids of
        // the bins up to it.
        for (int i = tid; i < NBIN; i += NTC) bcnt[i] = 0u;
        __syncthreads();
        for (int i = tid; i < nl; i += NTC) {
            const float d = (m - order_value(list[i])) * a.inv_w;
            const int bn = d < (float)(NBIN - 1) ? (int)d : NBIN - 1;
            if (ACES_IN(bn, NBIN)) atomicAdd(&bcnt[bn], 1u);
        }
        __syncthreads();
        if (wid == 0) {
            constexpr int PER = NBIN / 32;
            // lower edge of bin b in units of 2^kref: 2^(m c - kref) 2^(-(b+1) log2(e)/8)
            const float base2 = ex2(fmaf(m, a.c, -kref));
            constexpr float L2E8 = 1.4426950408889634f / BIN_PER_T;
            float lm = 0.0f;
            unsigned lc = 0u;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int bn = lane * PER + j;
                lm += (float)bcnt[bn] * base2 * ex2(-(float)(bn + 1) * L2E8);
                lc += bcnt[bn];
            }
            float pm = lm;
            unsigned pc = lc;
            for (int o = 1; o < 32; o <<= 1) {
                const float tm = __shfl_up_sync(0xffffffffu, pm, o);
                const unsigned tc = __shfl_up_sync(0xffffffffu, pc, o);
                if (lane >= o) {
                    pm += tm;
                    pc += tc;
                }
            }
            pm -= lm;
            pc -= lc;
            // 1e-4 covers the fp32 rounding of the bound and of S
            const float tgf = (float)s_tg * (1.0f / FX_SCALE) * (1.0f + 1e-4f);
            int hit = -1;
            unsigned ncand = 0u;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int bn = lane * PER + j;
                pm += (float)bcnt[bn] * base2 * ex2(-(float)(bn + 1) * L2E8) * (1.0f - 1e-4f);
                pc += bcnt[bn];
                const bool okb = all_in ? (pc >= (unsigned)a.k) : (pm >= tgf);
                if (okb && hit < 0) {
                    hit = bn;
                    ncand = pc;
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, hit >= 0);
            const int src = bal ? __ffs(bal) - 1 : 0;
            const int bsel = __shfl_sync(0xffffffffu, hit, src);
            const unsigned nc = __shfl_sync(0xffffffffu, ncand, src);
            // no bin reaches the bound: take every listed id (the exact sums
            // below still decide whether they hold the crossing); top_p = 1
            // with fewer than k listed ids goes to the exact kernel (the row
            // may hold finite ids below theta)
            if (lane == 0) {
                s_fb = all_in && bal == 0u;
                s_bsel = bal ? bsel : NBIN - 1;
                s_n = bal ? (int)nc : nl;
                s_npay = 0;
            }
        }
        __syncthreads();
        if (s_fb || s_n > WCAP) {
            hand_over();
            return;
        }
        // candidates: the listed ids in bins up to bsel
        const int bsel = s_bsel, n = s_n;
        unsigned long long *cv = work;
        for (int i0 = 0; i0 < nl; i0 += NTC) {  // warp-uniform rounds
            const int i = i0 + tid;
            unsigned long long o = 0ull;
            bool take = false;
            if (i < nl) {
                o = list[i];
                const float d = (m - order_value(o)) * a.inv_w;
                const int bn = d < (float)(NBIN - 1) ? (int)d : NBIN - 1;
                take = bn <= bsel;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, take);
            if (bal == 0u) continue;
            int base = 0;
            if (lane == __ffs(bal) - 1) base = atomicAdd(&s_npay, __popc(bal));
            base = __shfl_sync(0xffffffffu, base, __ffs(bal) - 1);
            const int at = base + __popc(bal & ((1u << lane) - 1u));
            if (take && ACES_IN(at, WCAP)) cv[at] = o;
        }
        __syncthreads();
        // order them (descending order value) into ord[], masses into efx[]
        unsigned long long *efx;
        if (n <= RANK_MAX) {
            ord = list;
            efx = list + RANK_MAX;
            rank_order_values<NTC>(cv, n, reinterpret_cast<uint32_t *>(list + 2 * RANK_MAX), [&](int rank, unsigned long long v) {
                if (ACES_IN(rank, RANK_MAX)) {
                    ord[rank] = v;
                    efx[rank] = id_fx(order_value(v), a.c, kref);
                }
            });
        } else {
            // more: bin by bin (the bins of T/8 below m order the values), and
            // inside a bin by direct ranking among its own ids
            if (tid == 0) atomicAdd(&a.ws.fb_count[3], 1);
            auto bin_of = [&](unsigned long long o) -> int {
                const float d = (m - order_value(o)) * a.inv_w;
                return d < (float)(NBIN - 1) ? (int)d : NBIN - 1;
            };
            if (wid == 0) {  // bcnt[b] <- the first place of bin b (bins 0..bsel hold the candidates)
                constexpr int PER = NBIN / 32;
                uint32_t c[PER], loc = 0u;
#pragma unroll
                for (int j = 0; j < PER; ++j) {
                    const int bn = lane * PER + j;
                    c[j] = bn <= bsel ? bcnt[bn] : 0u;
                    loc += c[j];
                }
                uint32_t inc = loc;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += t;
                }
                uint32_t run = inc - loc;
#pragma unroll
                for (int j = 0; j < PER; ++j) {
                    bcnt[lane * PER + j] = run;
                    run += c[j];
                }
            }
            __syncthreads();
            unsigned long long *binned = list;
            for (int i = tid; i < n; i += NTC) {
                const unsigned long long o = ACES_IN(i, WCAP) ? cv[i] : 0ull;
                const int bn = bin_of(o);
                const uint32_t at = ACES_IN(bn, NBIN) ? atomicAdd(&bcnt[bn], 1u) : 0u;
                if (ACES_IN(at, LCAP)) binned[at] = o;
            }
            __syncthreads();  // (bcnt[b] is now the end of bin b)
            ord = work;
            for (int i = tid; i < n; i += NTC) {
                const unsigned long long o = ACES_IN(i, LCAP) ? binned[i] : 0ull;
                const int bn = bin_of(o);
                const int st = bn > 0 && ACES_IN(bn - 1, NBIN) ? (int)bcnt[bn - 1] : 0;
                const int en = ACES_IN(bn, NBIN) ? (int)bcnt[bn] : 0;
                int rank = 0;
                for (int j = st; j < en; ++j) rank += (ACES_IN(j, LCAP) ? binned[j] : 0ull) > o;
                if (ACES_IN(st + rank, WCAP)) ord[st + rank] = o;
            }
            __syncthreads();
            efx = list;
            for (int i = tid; i < n; i += NTC)
                if (ACES_IN(i, WCAP)) efx[i] = id_fx(order_value(ord[i]), a.c, kref);
        }
        __syncthreads();
        // nucleus crossing with exact fixed-point prefix sums (consecutive
        // entries per thread; by one warp it took 3 us, up to 8 on long lists)
        {
            const int per = (n + NTC - 1) / NTC;
            const int lo = min(n, tid * per), hi = min(n, lo + per);
            unsigned long long loc = 0ull, tot;
            for (int i = lo; i < hi; ++i) loc += efx[i];
            const unsigned long long ex = block_exscan_n<NTC>(loc, s_redu, &tot);
            unsigned long long c;
            auto find = [&]() {
                const unsigned long long tg = s_tg;
                c = ex;
                for (int i = lo; i < hi; ++i) {
                    const unsigned long long prev = c;
                    c += efx[i];
                    if (prev < tg && c >= tg) {  // (one entry)
                        s_nstar = i;
                        s_above = c;
                    }
                }
                __syncthreads();
            };
            if (!all_in) {
                find();
                while (s_nstar != INT_MAX && s_above < s_th) {  // the cut depends on the error of S (at most twice)
                    sharpen(s_nstar + 1);
                    if (tid == 0) s_nstar = INT_MAX;
                    __syncthreads();
                    find();
                }
            }
            const int nstar = all_in ? n - 1 : s_nstar;  // (INT_MAX: below the list)
            if (nstar != INT_MAX) {
                const int Lw = min(nstar + 1, a.k);
                c = ex;
                for (int i = lo; i < hi && i < Lw; ++i) {
                    c += efx[i];
                    if (i == Lw - 1) s_cumL_fx = c;
                }
                if (tid == 0) {
                    s_nstar = nstar;
                    s_L = Lw;
                    if (Lw == 0) s_cumL_fx = 0ull;
                    const double sn = all_in ? S : (double)s_above * FX_INV;
                    s_Snuc = sn;
                    s_inv_S = inv_mass(sn);
                    s_cut = all_in ? 0ull : ord[nstar];
                }
            }
        }
        __syncthreads();
        if (s_nstar == INT_MAX) {
            hand_over();
            return;
        }
        // keep the nucleus for the residual step when it fits
        nnuc = (a.ws.nuc != nullptr && !all_in && s_nstar + 1 <= NUC_CAP) ? s_nstar + 1 : -1;
        if (nnuc > 0)
            for (int i = tid; i < nnuc; i += NTC)
                if (ACES_IN(i, NUC_CAP)) a.ws.nuc[(size_t)r * NUC_CAP + i] = ord[i];

        L = s_L;
        v_need = all_in ? (L > 0 ? order_value(ord[L - 1]) : m) : order_value(s_cut);
    }
    // ---- outputs ----
    if (tid == 0) {  // publish the depth this row needed, for later rows
        const float dxf = (m - v_need) * a.inv_ws;
        const int dx = dxf > 0.0f ? (int)fminf(dxf, (float)(NSB - 1)) : 0;
        if (ACES_IN(dx, NSB)) atomicAdd(&a.ws.fb_count[WS_DEPTH + dx], 1);
        atomicAdd(&a.ws.fb_count[8], 1);
        if (hinted) atomicAdd(&a.ws.fb_count[9], 1);
        if (short_row) atomicAdd(&a.ws.fb_count[11], 1);
    }
    const float inv_S = s_inv_S;
    for (int j = tid; j < a.k; j += NTC) {
        const size_t o = (size_t)r * a.k + j;
        if (j < L) {
            const unsigned long long ov = ord[j];
            a.topk_ids[o] = (int32_t)order_id(ov);
            a.topk_probs[o] = ex2(fmaf(order_value(ov), a.c, -kref)) * inv_S;
        } else {
            a.topk_ids[o] = -1;
            a.topk_probs[o] = 0.0f;
        }
    }
    if (tid == 0) {
        const double S_nuc = s_Snuc;
        const double cumL = (double)s_cumL_fx * FX_INV;
        if (a.k > 0) a.tail[r] = (float)(S_nuc - cumL) * inv_S;
        const unsigned long long cut = s_cut;
        int stt = 0;
        if (a.K > 0 && iq < a.K) {
            int accept = 0;
            if (xb < 0 || xb >= a.V) {
                stt |= ACES_ROW_BAD_Q;
            } else {
                bool in;
                if (all_in) in = zx > -INFINITY;
                else if (lazy) in = fkey(zx) >= (uint32_t)(cut >> 32);  // ties were decided above
                else in = order_val(fkey(zx), (uint32_t)xb) >= cut;
                const float e = in ? ex2(fmaf(zx, a.c, -kref)) : 0.0f;
                if (!(qx > 0.0f)) stt |= ACES_ROW_BAD_Q;
                else accept = accept_test(ux, qx, e, S_nuc);
            }
            a.ws.acc[(size_t)bq * a.K + iq] = accept;
        }
        a.row_status[r] = stt;
        RowStat rs;
        rs.kref = kref;
        rs.c = a.c;
        rs.S_nuc = S_nuc;
        rs.cut = cut;
        rs.flags = (all_in ? RS_ALL_IN : 0) | (lazy ? RS_LAZY : 0);
        rs.nnuc = nnuc;
        a.ws.stats[r] = rs;
    }
    defer_draw(a, row_finished<DT, NTC>(a, r, smem));
}

static int gcd_int(int x, int y) {
    while (y) {
        const int t = x % y;
        x = y;
        y = t;
    }
    return x;
}

// Threads per CTA.  A launch of at most one row per SM takes 1024, of at most
// two 512: one row's chain of dependent steps is then the whole time, and an
// SM's loads in flight come from that row alone (144 float32 rows of 32000:
// 73 us at 256 threads, 58 at 1024).  Not for more rows: 576 rows of 152064
// took 73 us at 256 threads, 77 at 512 and 114 at 1024.
static int rows_cap_threads(const RowArgs &a) { return a.rows <= a.nsm ? 1024 : (a.rows <= 2 * a.nsm ? 512 : 256); }

// Tile order and sample size of a row of a.V elements of type dt (ragged: its
// rows are off the 16-byte grid, up to one chunk longer): the
// stride is the smallest integer >= ntile / SAMPLE coprime with ntile, so the
// first SAMPLE tiles are spread over the whole row.
void rows_cap_layout(RowArgs &a, int dt, bool ragged) {
    const int nt = rows_cap_threads(a), nwc = nt / 32, tpi = nwc * UC;  // as in the kernel
    const int epc = dt == ACES_BF16 ? 8 : 4;
    const int nch = ragged ? (a.V + epc - 1 + epc - 1) / epc : a.V / epc;
    const int ntile = (nch + TCH - 1) / TCH;
    int p = ntile / SAMPLE;
    if (p < 1) p = 1;
    while (gcd_int(p, ntile) != 1) ++p;
    a.ntile = ntile;
    a.pstride = p;
    a.pstride_w = (int)((long long)nwc * p % ntile);
    a.pstride_it = (int)((long long)tpi * p % ntile);
    long long samp = 0;
    const int first = ntile < SAMPLE ? ntile : SAMPLE;
    for (int t = 0; t < first; ++t) {
        const long long tile = (long long)t * p % ntile;
        const long long c0 = tile * TCH, c1 = c0 + TCH < nch ? c0 + TCH : nch;
        samp += (c1 - c0) * epc;  // (off the grid: a few too many)
    }
    a.samp_frac = (float)((double)samp / (double)a.V);
    // the iterations that read the partial last tile (off the grid the row's
    // last chunk, partial itself, lies in one of the last two)
    a.it_partial = a.it_partial2 = -1;
    if (nch % TCH != 0 || ragged)
        for (int t = 0; t < ntile; ++t) {
            const long long tile = (long long)t * p % ntile;
            if (tile == ntile - 1) a.it_partial = t / tpi;
            if (ragged && tile == ntile - 2) a.it_partial2 = t / tpi;
        }
    a.inv_ws = (float)(SPB / (double)a.T);
    // Bounds of the relative difference between the row kernel's float32 sum and
    // the exact 2^-40 one.  The float32 sum rounds each mass in at most 8 adds and
    // the exact one drops less than 2^-40 of every id (add_err; the total is at
    // least 1/2).  Unless both take an id's mass against the same reference, each
    // rounds its exponent, at depth d = kref - z c, by at most d 2^-24 (d 2^-24 ln
    // 2 of its mass), and each has ex2's own error, at most 2^-22; the mean depth,
    // weighted by mass, is the masses' entropy less log2 of the total: at most
    // log2(V) + 1 (sum_err).
    a.add_err = (float)(ldexp(1.0, -21) + ldexp((double)a.V, -39));
    a.sum_err = a.add_err + (float)(2.0 * (0.6931472 * ldexp(log2((double)a.V) + 1.0, -24) + ldexp(1.0, -22)));
    a.nmin = 2 * a.k + 64 > 256 ? 2 * a.k + 64 : 256;
    // sketch groups: 4 chunks (two per thread and iteration) when they fit,
    // else 8 chunks of 2^sk_ish iterations
    const int nit = (ntile + tpi - 1) / tpi;
    a.sk_gpi = 2;
    a.sk_ish = 0;
    if ((long long)nit * nt * 2 > SKG) {
        a.sk_gpi = 1;
        while ((long long)((nit + (1 << a.sk_ish) - 1) >> a.sk_ish) * nt > SKG) ++a.sk_ish;
    }
}

// The dynamic shared memory above 48 KB needs an opt-in per device, set
// once per device on the first launch there (outside any stream capture).
template <int DT, int W, int NTC, bool RAGGED>
static cudaError_t launch_cap_dt(const RowArgs &a, cudaStream_t s) {
    constexpr int smem = DT == ACES_BF16 ? SMEM_BF : F32Caps<W>::SMEM;
    static std::mutex mu;
    static bool ready[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!ready[dev]) {
            const cudaError_t e = cudaFuncSetAttribute(k_rows_cap<DT, W, NTC, RAGGED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            ready[dev] = true;
        }
    }
    k_rows_cap<DT, W, NTC, RAGGED><<<(unsigned)a.rows, NTC, smem, s>>>(a);
    return cudaGetLastError();
}

// one CTA per row (float32: the wide areas when the launch is one wave at two
// CTAs per SM)
template <int DT, bool RAGGED>
static cudaError_t launch_cap(const RowArgs &a, cudaStream_t s) {
    constexpr int WIDE = DT == ACES_F32 ? 2 : 1;
    switch (rows_cap_threads(a)) {
        case 1024: return launch_cap_dt<DT, WIDE, 1024, RAGGED>(a, s);
        case 512: return launch_cap_dt<DT, WIDE, 512, RAGGED>(a, s);
        default: return launch_cap_dt<DT, 1, 256, RAGGED>(a, s);
    }
}
cudaError_t launch_rows_cap(const RowArgs &a, int dt, bool ragged, cudaStream_t s) {
    if (dt == ACES_BF16) return ragged ? launch_cap<ACES_BF16, true>(a, s) : launch_cap<ACES_BF16, false>(a, s);
    return ragged ? launch_cap<ACES_F32, true>(a, s) : launch_cap<ACES_F32, false>(a, s);
}

#ifdef ACES_CHECKED
cudaError_t check_take_rows_cap(unsigned long long out[3]) { return check_take(out); }
#endif

}  // namespace aces
