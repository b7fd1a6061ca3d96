// Panel simplex kernel for sm_103a: pivots are selected on single rows and
// columns of the tableau formed on demand, and the tableau itself is updated
// in place by panels of up to kPanelK pivots at a time.  Primal and dual rule,
// FP64 or FP32 tableau, one LP per launch.
//
// Arithmetic.  Step 5 (Sec. 2) gives every tableau element one fma per pivot,
//   T[i][j] <- fma(-col_t[i], prow_t[j], T[i][j])   (row p_t: prow_t[j]),
// and an element's value depends only on its own sequence of fmas.  So an
// element may be brought up to date when it is needed: the selection of pivot
// k forms just the entering column and the leaving row from the tableau of the
// last panel and the columns and rows of the pivots pending since then, and
// the other elements get the same fmas, in the same order, when the panel is
// applied.  Pivots, results and tableau are bit for bit those of updating
// everything after every pivot.  The launch ends with every pending pivot
// applied.
//
// What bounds it.  GB300 issues a warp-wide FP64 fma every 64 clocks per
// sub-partition, dependent or not (1.26 TFLOP/s in all), so a panel is bound
// by its fmas once it carries about four pivots, the tableau moving once per
// panel; the selection is a chain of two record exchanges and two dependent
// round trips to L2 per pivot, about 6 us of latency.  On small tableaus, on
// the largest and in FP32 the two alternate: nothing streams while the chain
// runs, so its loads and its few FP64 instructions never queue behind the
// panel's.  In between, where neither is small beside the other, panels of 8
// run on eight more warps and a second buffer while the next one's pivots are
// selected (OV below): the chain takes about 9 us then, the panel's time is
// hidden.  Measured, FP64, us per pivot, against the kernels that update
// everything every one or two pivots: 64^2 6.4, 256^2 7.0 (was 9.3), 501 x 703 of
// the paper's family 6.7 (10.2), 512 x 4096 8.6 (10.1; in turn 10.9), 4096 x 512
// 9.7 (41; 10.3), 2048^2 10.3 (21.6; 13.7), its dual form 12.3 (22.9; 16.1),
// 4096^2 33 (58; 36), 8192^2 118 (136; overlapped 119; 107 is its fmas at the
// FP64 peak); FP32 8192^2 18 in launches of 50 pivots, 16 of 200 (70).  In turn, panels of 8 pivots instead of 16
// were 1 to 4% slower from 512 x 4096 up; overlapped, four or six warps for the
// panels were slower than eight from 2048^2 up (13.2 and 10.4 us).
//
// Work split (G CTAs).  CTA g owns
//   the columns J_g (a contiguous strip) of the objective row and of every
//   leaving row, and the rows I_g (a contiguous slice) of the rhs and of every
//   entering column; it applies the panels to all columns of its rows.
// The panels split by rows, so the CTAs' shares stay equal whichever columns
// need no update, and a column's gather reads only rows this CTA wrote.
//
// One pivot, primal rule (dual: rows and columns change places):
//   1. pricing over J_g -> record 1 (z_q, q); all CTAs read all records (Step 2)
//   2. column q on I_g: T[i][q] with the pending pivots; ratio test on I_g
//      -> record 2 (the ratio's key, p, the variable basic in p); all CTAs read
//      all records (Step 3)
//   3. row p on J_g with the pending pivots, divided by the pivot (Step 4), the
//      objective row on J_g and the rhs on I_g updated.
// A record is 16 bytes in a 128-byte line of its own, with its pivot's number:
// readers poll the records themselves (about 2000 clocks for 152 CTAs; 16 or
// 32 bytes between records took 10 to 30% longer per pivot, and a counter
// released after the records 3960 clocks).  Polling starts once the CTA's own
// record is out: polls from the start of the pivot doubled the exchange.
// What else crosses CTAs for a pivot (single entries of pending rows and
// columns, a record's further values) carries its pivot's tag beside it, so no
// fence orders it: fences took 450 clocks alone and 3000 under the polls.  What
// a panel reads (the pending rows, plain) and writes (the tableau) has no tags
// and is ordered once per panel: the lane that publishes the record which
// announces it fences first, after the barrier that follows the writes, and the
// lanes that poll that record fence before the barrier that precedes the reads.
//
// Columns that stay basic through a panel are exact unit vectors: their
// entries in its pivot rows are zeros, and an fma with a zero product leaves a
// finite nonzero entry and +0 as they are.  The panel leaves such columns out
// (lp_options.zero_skip).  Exceptions are tracked: a pivot row divided by a
// negative pivot (dual rule) holds -0 in them, so its row is marked and marked
// rows get every column; the marks are kept in memory from launch to launch, up
// to a refresh, which writes exact unit vectors (finding such rows by a scan
// took longer than a launch of a few pivots: 512 x 4096, dual, one pivot a call,
// 1.5 times the call); and a panel with a non-finite pivot column, or with a
// nonzero pivot-row entry in a column thought to stay, gets every column in
// every row.
//
// Waits are bounded: a poll that does not succeed within the spin limit sets
// the error flag and the kernel returns with status TIMEOUT.

#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "gbs_colbits.h"
#include "gbs_device.cuh"
#include "gbs_internal.h"

namespace gbs {

namespace {

using namespace dev;

constexpr int kRec = 8;  // 16-byte units between the CTAs' records (one used: a line each)

__device__ __forceinline__ double pfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float pfma(float a, float b, float c) { return fmaf(a, b, c); }

__device__ __forceinline__ unsigned long long to_bits(double x) {
    return (unsigned long long)__double_as_longlong(x);
}
__device__ __forceinline__ unsigned long long to_bits(float x) {
    return (unsigned long long)__float_as_uint(x);
}
template <typename T>
__device__ __forceinline__ T from_bits(unsigned long long u);
template <>
__device__ __forceinline__ double from_bits<double>(unsigned long long u) {
    return __longlong_as_double((long long)u);
}
template <>
__device__ __forceinline__ float from_bits<float>(unsigned long long u) {
    return __uint_as_float((unsigned)u);
}

__device__ __forceinline__ bool is_zero(double x) {
    return (unsigned long long)__double_as_longlong(x) << 1 == 0ull;
}
__device__ __forceinline__ bool is_zero(float x) { return __float_as_uint(x) << 1 == 0u; }
__device__ __forceinline__ bool not_finite(double x) {
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) == 0x7ff00000u;
}
__device__ __forceinline__ bool not_finite(float x) {
    return (__float_as_uint(x) & 0x7f800000u) == 0x7f800000u;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// 16-byte values, written and read whole.
__device__ __forceinline__ void st_half(ulonglong2 *p, unsigned long long a, unsigned lo,
                                        unsigned hi) {
    const unsigned long long b = ((unsigned long long)hi << 32) | lo;
    asm volatile(
        "{.reg .b128 t; mov.b128 t, {%0, %1}; st.relaxed.gpu.global.b128 [%2], t;}" ::"l"(a),
        "l"(b), "l"(p)
        : "memory");
}
__device__ __forceinline__ ulonglong2 ld_half(const ulonglong2 *p) {
    ulonglong2 v;
    asm volatile("{.reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t;}"
                 : "=l"(v.x), "=l"(v.y)
                 : "l"(p)
                 : "memory");
    return v;
}

// Division of many numerators by one pivot, correctly rounded: with
// y = RN(1/b) and q within an ulp of a/b, RN(q + (a - b q) y) = RN(a/b)
// barring under- and overflow (P. Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990;
// the first correction brings q within an ulp).  Five FP64 operations instead
// of the general division's chain, which took the selection 0.3 us more per
// pivot; operands outside the middle of the exponent range take the general
// division.
struct Divisor64 {
    double b, y;
    bool mid;
    static __device__ __forceinline__ bool in_mid(double v) {
        const int e = (__double2hiint(v) >> 20) & 0x7ff;
        return e >= 1023 - 500 && e <= 1023 + 500;
    }
    // 1 / v correctly rounded, 0 where the general division is taken
    static __device__ __forceinline__ double recip(double v) {
        return in_mid(v) ? __drcp_rn(v) : 0.0;
    }
    __device__ __forceinline__ Divisor64(double v, double r) : b(v), y(r), mid(in_mid(v)) {}
    __device__ __forceinline__ double div(double a) const {
        if (mid && in_mid(a)) {
            const double q0 = __dmul_rn(a, y);
            const double q1 = fma(fma(-b, q0, a), y, q0);
            return fma(fma(-b, q1, a), y, q1);
        }
        if (mid && is_zero(a))  // a signed zero
            return __longlong_as_double(__double_as_longlong(a) ^
                                        (__double_as_longlong(b) & (long long)kSign));
        return a / b;
    }
};
struct Divisor32 {
    float b;
    static __device__ __forceinline__ float recip(float) { return 0.0f; }
    __device__ __forceinline__ Divisor32(float v, float) : b(v) {}
    __device__ __forceinline__ float div(float a) const { return a / b; }
};
template <typename T>
struct DivisorOf;
template <>
struct DivisorOf<double> {
    typedef Divisor64 type;
};
template <>
struct DivisorOf<float> {
    typedef Divisor32 type;
};

// Screening key of num / den (num >= +0, den > 0): the bits of a float within
// a relative 2^-20 of the quotient, whose order as integers is the floats'
// order, for operands with exponents within 2^+-60 (the quotient is then a
// normal float); kWide marks operands outside, which have to be divided
// exactly.  kNear steps of a key are a relative 2^-16 (significand near 2) to
// 2^-15 (near 1), more than twice a key's error: a row whose exactly rounded
// ratio is the smallest has a key at most kNear above the smallest key, so rows
// further off need no division.
constexpr unsigned kNone = 0xffffffffu;  // not a candidate
constexpr unsigned kNear = 256;
__device__ __forceinline__ unsigned ratio_key(double num, double den, bool *wide) {
    const int nh = __double2hiint(num), dh = __double2hiint(den);
    if ((nh | __double2loint(num)) == 0) return 0u;
    const int ne = nh >> 20, de = dh >> 20;
    if (ne < 1023 - 60 || ne > 1023 + 60 || de < 1023 - 60 || de > 1023 + 60) {
        *wide = true;
        return 0u;
    }
    // (truncated to the float's 23 bits)
    const float a = __int_as_float(((nh - ((1023 - 127) << 20)) << 3) |
                                   (int)((unsigned)__double2loint(num) >> 29));
    const float b = __int_as_float(((dh - ((1023 - 127) << 20)) << 3) |
                                   (int)((unsigned)__double2loint(den) >> 29));
    return __float_as_uint(__fdividef(a, b));
}
__device__ __forceinline__ unsigned ratio_key(float num, float den, bool *wide) {
    const int nb = __float_as_int(num), db = __float_as_int(den);
    if (nb == 0) return 0u;
    const int ne = nb >> 23, de = db >> 23;
    if (ne < 127 - 60 || ne > 127 + 60 || de < 127 - 60 || de > 127 + 60) {
        *wide = true;
        return 0u;
    }
    return __float_as_uint(__fdividef(num, den));
}

// One warp's entry of a selection across warps.
struct alignas(16) Slot {
    unsigned long long vk, x;
    int key, idx, aux, flag;
    unsigned sk, sk2;
    int src;
};

// A selected record, the same in every thread: its value (exchange 1) or its
// tie word (exchange 2), index (-1: none) and CTA.
struct Pick {
    unsigned long long x;
    int idx, aux, cta, zero;
};

__device__ __forceinline__ void group_sync(int id, int warps) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(warps * 32) : "memory");
}
__device__ __forceinline__ void group_arrive(int id, int warps) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(warps * 32) : "memory");
}

// The lane with the smallest (vk, key), lowest on equal pairs.  The high words
// nearly always decide.
__device__ __forceinline__ int min_lane(unsigned long long vk, int key) {
    const unsigned hi = (unsigned)(vk >> 32);
    unsigned b = __ballot_sync(0xffffffffu, hi == __reduce_min_sync(0xffffffffu, hi));
    if (b & (b - 1)) {
        const bool in = b >> (threadIdx.x & 31) & 1u;
        const unsigned lo = in ? (unsigned)vk : 0xffffffffu;
        const unsigned ml = __reduce_min_sync(0xffffffffu, lo);
        const unsigned ky = in && lo == ml ? (unsigned)key : 0xffffffffu;
        const unsigned mk = __reduce_min_sync(0xffffffffu, ky);
        b = __ballot_sync(0xffffffffu, in && lo == ml && ky == mk);
    }
    return __ffs(b) - 1;
}

// Pending pivots of one row or column entry lie side by side in shared memory,
// kStride apart from the next entry's, so that a lane fetches all of its own
// with 16-byte loads at constant offsets and 8 lanes' loads cover the banks.
__host__ __device__ constexpr int entry_stride(int esz, int K) { return esz == 8 ? K + 2 : K + 4; }

// v <- fma(-c[t], p[t], v) for t in [0, k), in order (c, p: shared memory, at
// least entry_stride).  A loop, with the next entries fetched ahead: the
// fmas' latency is its only cost (unrolled and predicated, all 16 ran).
template <typename T>
__device__ __forceinline__ T fma_chain(T v, int k, const T *c, const T *p) {
    typedef typename Vec<T>::type V;
    constexpr int VW = Vec<T>::W;
    V c0 = *reinterpret_cast<const V *>(c), p0 = *reinterpret_cast<const V *>(p);
    int t = 0;
#pragma unroll 1
    for (; t + VW <= k; t += VW) {
        c += VW;
        p += VW;
        const V c1 = *reinterpret_cast<const V *>(c), p1 = *reinterpret_cast<const V *>(p);
#pragma unroll
        for (int u = 0; u < VW; ++u) v = pfma(-getc(c0, u), getc(p0, u), v);
        c0 = c1;
        p0 = p1;
    }
#pragma unroll
    for (int u = 0; u < VW - 1; ++u)
        if (t + u < k) v = pfma(-getc(c0, u), getc(p0, u), v);
    return v;
}

// Shared-memory layout of a CTA, shared by the kernel and the host's sizing.
struct PanelLayout {
    int R, W, nvec, nwords;
    size_t zs, prs, cs, rh, bas, lastp, rowz, bb, stay, prev, out, list, total;
};

// (slots: pending pivots at most; ov: with the bitmaps of the overlapped panels)
__host__ __device__ inline PanelLayout panel_layout(int m, int N, int G, int esz, int vw, int slots,
                                                    bool ov) {
    PanelLayout L;
    const int stride = entry_stride(esz, slots);
    L.R = (m + G - 1) / G + 1;  // slices differ by at most one row
    L.W = (N + G - 1) / G + 1;
    L.nvec = (N + vw - 1) / vw;
    L.nwords = (N + 31) / 32;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t p = at;
        at = (at + bytes + 15) / 16 * 16;
        return p;
    };
    L.prs = take((size_t)stride * L.W * esz);
    L.cs = take((size_t)stride * L.R * esz);
    L.zs = take((size_t)L.W * esz);
    L.rh = take((size_t)L.R * esz);
    L.bas = take((size_t)L.R * sizeof(int));
    L.lastp = take((size_t)L.R);
    L.rowz = take((size_t)L.R);
    L.bb = take((size_t)L.nwords * sizeof(unsigned));
    L.stay = take((size_t)L.nwords * sizeof(unsigned));
    L.prev = take(ov ? (size_t)L.nwords * sizeof(unsigned) : 0);
    L.out = take(ov ? (size_t)L.nwords * sizeof(unsigned) : 0);
    L.list = take((size_t)L.nwords * (32 / vw) * sizeof(int));
    L.total = at;
    return L;
}

// Pitch of the tagged values: an odd number of 128-byte lines, so that the
// pending pivots' entries at one row or column, which every CTA reads at once,
// are spread over the L2's slices.
__host__ __device__ inline long long tag_pitch(long long n) { return ((n + 7) / 8 | 1) * 8; }

// Warps of a CTA: columns of the strip from warp 0 on, rows of the slice from
// the last warp down, the records of the other CTAs on the middle ones (two
// per lane), so that the three kinds of work of a small slice run at once, on
// different sub-partitions.
constexpr int kWarps = kPanelThreads / 32;
constexpr int kPollFirst = 3, kPollWarps = 3;
constexpr int kPollRecs = (kPanelMaxCtas + 32 * kPollWarps - 1) / (32 * kPollWarps);

// A record's third word: index + 1 (0: none) and flags.
constexpr unsigned kIdxMask = 0x1fffffffu;
constexpr unsigned kFlagAll = 1u << 31;   // this panel gets every column
constexpr unsigned kFlagZero = 1u << 30;  // the ratio rounds to zero
constexpr unsigned kFlagWide = 1u << 29;  // a ratio key out of range

// Overlapped panels: what the other warps do next.
enum : int { kJobEnd = 0, kJobCopy = 1, kJobPanel = 2, kJobInPlace = 3 };

// One LP on a group of G co-resident CTAs, this one its g-th, with panels of up
// to K pivots.
//
// OV: panels overlapped with the selection.  The CTA has eight more warps,
// which apply one panel from the current tableau buffer into the other while
// the first eight select the next panel's pivots on the current one, with the
// pivots of both panels pending.  The buffers change places when every CTA's
// panel is done, which its next record 1 says.  A column that did not change
// in this panel and the one before is the same in both buffers and is left
// out; the launch starts by copying the tableau (under the first panel's
// selection) and ends by applying the last pivots in place.
template <typename T, bool DUAL, int K, bool OV>
__device__ __forceinline__ void panel_solve(LpDesc *__restrict__ d, int G, int g,
                                            long long spin_limit, long long budget, int drop,
                                            unsigned nonce, unsigned last_epoch, long long limit_ns,
                                            unsigned char *smem_raw) {
    typedef typename Vec<T>::type V;
    typedef typename DivisorOf<T>::type Divisor;
    constexpr int VW = Vec<T>::W;
    constexpr int NS = OV ? 2 * K : K;  // slots of pending pivots
    constexpr int B = kPanelThreads, nw = kWarps, KS = entry_stride(sizeof(T), NS);
    constexpr int RS = sizeof(T) == 8 || NS < kPanelK ? 4 : 8;  // rows of a panel step per warp
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ Slot s_loc[nw], s_ex1[kPollWarps], s_ex2[kPollWarps], s_ex3[kPollWarps];
    __shared__ __align__(16) T s_at[nw][KS];  // a warp's pending entries at one row or column
    __shared__ int s_flag, s_fail[2], s_nflag, s_task, s_scan[nw];
    __shared__ int s_prow[NS];  // pivot rows of the pending pivots
    __shared__ int s_job[5];    // OV: the panel to apply
    __shared__ ulonglong2 s_rec[2];
    __shared__ unsigned long long s_aux[2][2][4];

    const int tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    T *const bufs[2] = {reinterpret_cast<T *>(d->T), reinterpret_cast<T *>(OV ? d->T2 : d->T)};
    T *Tab = bufs[0];  // the tableau of the last panel applied
    const long long P = d->P;
    const int m = d->m, N = d->N;
    const long long Mp = tag_pitch(m), Np = tag_pitch(N);
    // pending columns (NS x Mp) and rows (NS x Np) and the records' further values
    // (by pivot parity, 2 exchanges x G x 4) as 16-byte values with the tag of their pivot, for
    // single entries (with one CTA they are all in its shared memory); and the
    // rows plain, for the panels
    ulonglong2 *const CT = reinterpret_cast<ulonglong2 *>(d->panel);
    ulonglong2 *const PT = CT + (G > 1 ? NS * Mp : 0);
    ulonglong2 *const AX = PT + (G > 1 ? NS * Np : 0);
    T *const PR = reinterpret_cast<T *>(AX + (G > 1 ? 16 * G : 0));
    unsigned char *const marks = reinterpret_cast<unsigned char *>(PR + NS * P);  // rowz, between launches
    ulonglong2 *const recs = reinterpret_cast<ulonglong2 *>(d->recs);
    int *const err = d->err;

    const PanelLayout L = panel_layout(m, N, G, sizeof(T), VW, NS, OV);
    T *const zs = reinterpret_cast<T *>(smem_raw + L.zs);
    T *const prs = reinterpret_cast<T *>(smem_raw + L.prs);
    T *const cs = reinterpret_cast<T *>(smem_raw + L.cs);
    T *const rh = reinterpret_cast<T *>(smem_raw + L.rh);
    int *const bas = reinterpret_cast<int *>(smem_raw + L.bas);
    signed char *const lastp = reinterpret_cast<signed char *>(smem_raw + L.lastp);
    unsigned char *const rowz = smem_raw + L.rowz;
    unsigned *const bb = reinterpret_cast<unsigned *>(smem_raw + L.bb);      // basic columns
    unsigned *const stay = reinterpret_cast<unsigned *>(smem_raw + L.stay);  // basic since the last panel
    unsigned *const prev = reinterpret_cast<unsigned *>(smem_raw + L.prev);  // OV: in the panel before
    unsigned *const out = reinterpret_cast<unsigned *>(smem_raw + L.out);    // OV: left out of the panel
    int *const list = reinterpret_cast<int *>(smem_raw + L.list);
    // every selection thread (OV: half of the CTA)
    auto cta_sync = [&]() {
        if (OV) group_sync(5, nw);
        else __syncthreads();
    };
    const int nvec = L.nvec, nwords = L.nwords;

    const int i0 = (int)((long long)m * g / G), R = (int)((long long)m * (g + 1) / G) - i0;
    const int c0 = (int)((long long)N * g / G), W = (int)((long long)N * (g + 1) / G) - c0;
    const int cw = min(nw, (W + 31) / 32);          // warps with columns (W >= 1)
    const int rw = min(nw, max(1, (R + 31) / 32));  // warps with rows
    const bool col_warp = wid < cw, row_warp = nw - 1 - wid < rw;
    const bool poll_warp = wid >= kPollFirst && wid < kPollFirst + kPollWarps;
    const int rt = (nw - 1 - wid) * 32 + lane;      // this thread's first row
    const int ct = tid;                             // and column

    const int bland_after = d->bland_after;
    const unsigned long long lim_p = okey((T)d->eps_p);
    const unsigned long long lim_np = okey((T)(-d->eps_p));
    const unsigned long long lim_d = okey((T)(-d->eps_d));
    const unsigned long long lim_r = okey((T)(-d->eps_r));
    const unsigned long long zero_k = okey((T)0);
    long long iters = d->iters;
    const long long iter_limit =
        iters > 0x3fffffffffffffffll - budget ? 0x3fffffffffffffffll : iters + budget;
    int deg = d->deg;
    int status = ST_RUNNING;
    const bool marked = iters > 0 && !(d->negz & 2);
    const int *const abort_word = d->abort;
    const unsigned long long t_start = limit_ns > 0 ? global_ns() : 0ull;
    const long long trace_cap = d->trace_cap;

    // ------------------------------------------------------------- start --
    if (!OV || tid < B) {
        const T *z = Tab + (long long)m * P;
        for (int c = tid; c < W; c += B) zs[c] = lds(z + c0 + c);
        for (int r = tid; r < R; r += B) {
            rh[r] = lds(Tab + (long long)(i0 + r) * P + (N - 1));
            bas[r] = __ldcg(d->basis + i0 + r);
            rowz[r] = marked ? __ldcg(marks + i0 + r) : 0;
            lastp[r] = -1;
        }
        for (int w = tid; w < nwords; w += B) bb[w] = 0;
        // the padding of the last vector of the pending rows (other CTAs read
        // it once a record or the barrier has announced the rows)
        if (g == 0 && tid < NS)
            for (int j = N; j < nvec * VW; ++j) __stcg(PR + tid * P + j, (T)0);
        const int bas0 = tid < m ? __ldcg(d->basis + tid) : -1;
        if (tid == 0) {
            s_fail[0] = s_fail[1] = 0;
            s_nflag = 0;
        }
        cta_sync();
        for (int i = tid; i < m; i += B) {
            const int j = i == tid ? bas0 : __ldcg(d->basis + i);
            atomicOr(&bb[j >> 5], 1u << (j & 31));
        }
        cta_sync();
        for (int w = tid; w < nwords; w += B) {
            // (columns past the last one never need an update)
            bb[w] |= past_end(w, N);
            stay[w] = bb[w];
            if (OV) prev[w] = ~0u;  // (the copy makes the buffers equal)
        }
        for (int r = tid; r < R; r += B)
            if (rowz[r]) s_nflag = 1;
        cta_sync();
    }

    int k = 0;            // pending pivots of this panel
    int kold = 0;         // OV: and of the panel that is being applied,
    int ho = 0, hn = 0;   // in the slots from ho; this panel's from hn
    int cur = 0, jobs = 0;
    // the slot of the pos-th pending pivot, oldest first
    auto slot = [&](int pos) { return !OV ? pos : pos < kold ? ho + pos : hn + pos - kold; };
    unsigned epoch = last_epoch + 1;  // number of the pivot whose records are awaited
    unsigned ecur = epoch;            // number of the pivot being made
    int nodrop = 0;       // this panel gets every column
    int ab_next = 0;
    int last_p = d->last_p, last_q = d->last_q;
    unsigned long long upd = 0, left = 0;  // vectors x pivots, for d->work

    // NR rows of one 16-byte vector column: kk pending pivots on each.
    const long long pv = P / VW;
    auto panel_rows = [&](auto nr_tag, V(&a)[decltype(nr_tag)::value], V *at, int r, int h, int kk,
                          const V(&pr)[K], bool act) {
        constexpr int NR = decltype(nr_tag)::value;
#pragma unroll
        for (int t0 = 0; t0 < K; t0 += VW) {
            if (t0 >= kk) break;
            V c[NR];
#pragma unroll
            for (int u = 0; u < NR; ++u)
                c[u] = *reinterpret_cast<const V *>(cs + (r + u) * KS + h + t0);
#pragma unroll
            for (int t = t0; t < t0 + VW; ++t) {
                if (t >= kk) break;
                const int lp = s_prow[h + t] - i0 - r;
                if ((unsigned)lp < (unsigned)NR) {
#pragma unroll
                    for (int u = 0; u < NR; ++u) {
                        V x = a[u];
                        vfma(x, getc(c[u], t - t0), pr[t]);
                        a[u] = u == lp ? pr[t] : x;
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < NR; ++u) vfma(a[u], getc(c[u], t - t0), pr[t]);
                }
            }
        }
        if (act) {
#pragma unroll
            for (int u = 0; u < NR; ++u) at[u * pv] = a[u];
        }
    };

    // Apply the kk pending pivots in the slots from h to this CTA's rows, from
    // src to dst, but to the columns in the bitmap `left_out` (none with `all`)
    // only on marked rows.  Thread bt of nw warps; sync() is their barrier.
    auto panel_job = [&](const T *src, T *dst, int h, int kk, bool all, const unsigned *left_out,
                         int bt, auto &&sync) {
        const int bw = bt >> 5;
        // the vectors to update, in order
        int nact;
        if (bt == 0) s_task = 0;
        if (all) {
            for (int v = bt; v < nvec; v += B) list[v] = v;
            nact = nvec;
            sync();
        } else {
            const int per = (nwords + B - 1) / B;
            const int w0 = min(nwords, bt * per), w1 = min(nwords, w0 + per);
            int cnt = 0;
            for (int w = w0; w < w1; ++w) {
                const unsigned s = left_out[w];
                for (int u = 0; u < 32 / VW; ++u) cnt += vector_kept(s, u, VW);
            }
            int pre = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kAll, pre, o);
                if (lane >= o) pre += y;
            }
            if (lane == 31) s_scan[bw] = pre;
            sync();
            int base = 0;
            nact = 0;
            for (int w = 0; w < nw; ++w) {
                if (w < bw) base += s_scan[w];
                nact += s_scan[w];
            }
            int at = base + pre - cnt;
            for (int w = w0; w < w1; ++w) {
                const unsigned s = left_out[w];
                for (int u = 0; u < 32 / VW; ++u)
                    if (vector_kept(s, u, VW)) list[at++] = w * (32 / VW) + u;
            }
            sync();
        }
        upd += (unsigned long long)(all ? P / VW : nact) * kk;
        left += (unsigned long long)(all ? 0 : P / VW - nact) * kk;
        // tasks of 32 vectors x RB rows, taken by the warps in turn; the pivot
        // rows' entries in registers
        const int nchunk = (nact + 31) / 32;
        int S = nchunk > 0 ? ((sizeof(T) == 8 ? 6 : 12) * nw + nchunk - 1) / nchunk : 1;
        S = max(1, min(S, (R + RS - 1) / RS));
        const int RB = ((R + S - 1) / S + 1) / 2 * 2;
        S = RB > 0 ? (R + RB - 1) / RB : 0;
        for (;;) {
            int task = 0;
            if (lane == 0) task = atomicAdd(&s_task, 1);
            task = __shfl_sync(kAll, task, 0);
            if (task >= nchunk * S) break;
            const int sub = task / nchunk, ch = task - sub * nchunk;
            const int e = ch * 32 + lane;
            const bool act = e < nact;
            const int v = list[act ? e : nact - 1];
            V pr[K];
#pragma unroll
            for (int t = 0; t < K; ++t)
                if (t < kk) pr[t] = ldv(reinterpret_cast<const V *>(PR + (h + t) * P) + v);
            int r = sub * RB;
            const int rb1 = min(R, r + RB);
            const V *from = reinterpret_cast<const V *>(src + (long long)(i0 + r) * P) + v;
            V *at = reinterpret_cast<V *>(dst + (long long)(i0 + r) * P) + v;
            // RS rows at a time (with registers to spare the next RS in flight);
            // then 4, 2 and 1
            auto load_rows = [&](auto nr_tag, V(&x)[decltype(nr_tag)::value], const V *q) {
#pragma unroll
                for (int u = 0; u < decltype(nr_tag)::value; ++u) x[u] = ldv(q + u * pv);
            };
            const std::integral_constant<int, RS> rs;
            V a[RS];
            if constexpr (NS == kPanelK) {
                V b[RS];
                if (r + RS <= rb1) load_rows(rs, a, from);
                for (; r + RS <= rb1; r += RS, at += RS * pv, from += RS * pv) {
                    const bool more = r + 2 * RS <= rb1;
                    if (more) load_rows(rs, b, from + RS * pv);
                    panel_rows(rs, a, at, r, h, kk, pr, act);
                    if (more) {
#pragma unroll
                        for (int u = 0; u < RS; ++u) a[u] = b[u];
                    }
                }
            } else {
                for (; r + RS <= rb1; r += RS, at += RS * pv, from += RS * pv) {
                    load_rows(rs, a, from);
                    panel_rows(rs, a, at, r, h, kk, pr, act);
                }
            }
            auto rest = [&](auto nr_tag) {
                constexpr int NR = decltype(nr_tag)::value;
                V c[NR];
                if (r + NR > rb1) return;
                load_rows(nr_tag, c, from);
                panel_rows(nr_tag, c, at, r, h, kk, pr, act);
                r += NR;
                at += NR * pv;
                from += NR * pv;
            };
            if (RS == 8) rest(std::integral_constant<int, 4>());
            rest(std::integral_constant<int, 2>());
            rest(std::integral_constant<int, 1>());
        }
        // the other columns of marked rows
        if (!all && s_nflag) {
            for (int r = 0; r < R; ++r) {
                if (!rowz[r]) continue;
                const V *const from = reinterpret_cast<const V *>(src + (long long)(i0 + r) * P);
                V *const to = reinterpret_cast<V *>(dst + (long long)(i0 + r) * P);
                for (int v = bt; v < nvec; v += B) {
                    const int j = v * VW;
                    if (vector_kept(left_out[j >> 5], (j & 31) / VW, VW)) continue;
                    V x = ldv(from + v);
                    for (int t = 0; t < kk; ++t) {
                        const V pt = ldv(reinterpret_cast<const V *>(PR + (h + t) * P) + v);
                        if (s_prow[h + t] == i0 + r) x = pt;
                        else vfma(x, cs[r * KS + h + t], pt);
                    }
                    to[v] = x;
                }
            }
        }
        // other CTAs read these rows after this CTA's next record: whichever
        // thread publishes it, its fence follows every thread's writes (a launch
        // that ends publishes no more)
        sync();
        if (OV || status == ST_RUNNING) __threadfence();
    };
    // The pending pivots of a full or last panel, in place (not OV).
    auto apply_panel = [&](int kk) {
        panel_job(Tab, Tab, 0, kk, !drop || nodrop, stay, tid, cta_sync);
        for (int w = tid; w < nwords; w += B) stay[w] = bb[w];
        for (int r = tid; r < R; r += B) lastp[r] = -1;
        nodrop = 0;
        cta_sync();
    };

    // OV, the other eight warps: jobs as the selection warps post them.
    if (OV && tid >= B) {
        const int bt = tid - B;
        auto sync = [&]() { group_sync(6, nw); };
        for (;;) {
            group_sync(7, 2 * nw);
            const int kind = s_job[0];
            if (kind == kJobEnd) break;
            if (kind == kJobCopy) {
                const V *src = reinterpret_cast<const V *>(bufs[0] + (long long)i0 * P);
                V *dst = reinterpret_cast<V *>(bufs[1] + (long long)i0 * P);
                const long long cnt = (long long)R * pv;
#pragma unroll 4
                for (long long e = bt; e < cnt; e += B) dst[e] = ldv(src + e);
                sync();
                __threadfence();
            } else {
                T *const src = bufs[s_job[3]];
                panel_job(src, kind == kJobPanel ? bufs[s_job[3] ^ 1] : src, s_job[1], s_job[2],
                          s_job[4] != 0, out, bt, sync);
            }
            group_arrive(8, 2 * nw);
        }
        if (g == 0 && bt == 0 && d->work) {
            d->work[0] += upd;
            d->work[1] += left;
        }
        return;
    }
    // OV: post a job (every selection thread).
    auto post = [&](int kind, int h, int kk, bool all) {
        if (tid == 0) {
            s_job[0] = kind, s_job[1] = h, s_job[2] = kk, s_job[3] = cur, s_job[4] = all;
        }
        cta_sync();
        group_arrive(7, 2 * nw);
        ++jobs;
    };
    // OV: wait until the job posted last is done (once per job, every selection
    // warp; one that does not read what the job wrote only arrives).  A barrier:
    // polling a flag in shared memory would be a wait without a limit, and no
    // job may be posted while one is under way.
    auto wait_job = [&](bool here) {
        __syncwarp();
        if (here) group_sync(8, 2 * nw);
        else group_arrive(8, 2 * nw);
    };
    // Every CTA of the group; false when a wait ran out.
    auto group_barrier = [&]() {
        if (!OV) return grid_sync(d->bar, err, G, spin_limit, &s_flag);
        cta_sync();
        if (tid == 0) {
            int ok = 1;
            if (G > 1) {
                const unsigned g0 = ld_acquire(d->bar + 32);
                __threadfence();
                if (atom_add_acq_rel(d->bar, 1u) == (unsigned)G - 1u) {
                    atomicExch(d->bar, 0u);
                    st_release(d->bar + 32, g0 + 1u);
                } else {
                    const long long t0 = clock64();
                    while (ld_acquire(d->bar + 32) == g0) {
                        if (clock64() - t0 > spin_limit || *(volatile int *)err) {
                            atomicExch(err, 1);
                            break;
                        }
                    }
                }
                __threadfence();
            }
            if (*(volatile int *)err) ok = 0;
            s_flag = ok;
        }
        cta_sync();
        return s_flag != 0;
    };

    // A value written by another CTA, once it carries the tag of pivot e.
    auto tagged = [&](const ulonglong2 *at, unsigned e, int which) {
        const unsigned long long tag = ((unsigned long long)nonce << 32) | e;
        ulonglong2 v = ld_half(at);
        if (v.y != tag) {
            const long long t0 = clock64();
            do {
                if (clock64() - t0 > spin_limit || *(volatile int *)err) {
                    atomicExch(err, 1);
                    s_fail[which] = 1;
                    break;
                }
                v = ld_half(at);
            } while (v.y != tag);
        }
        return v.x;
    };
    // A record's further values: record 1 of the dual rule has the rhs of the
    // leaving row and the leaving variable, record 2 the numerator and the
    // denominator (the pivot) of its ratio and the pivot's reciprocal.  By
    // parity: they are read up to the next selection, and the next but one's
    // records come only after that.
    auto further_at = [&](unsigned e, int which, int cta) {
        return AX + 4 * (((int)(e & 1) * 2 + which) * G + cta);
    };
    auto set_further = [&](int which, int i, unsigned long long v) {
        if (G == 1) s_aux[epoch & 1][which][i] = v;
        else st_half(further_at(epoch, which, g) + i, v, epoch, nonce);
    };
    // A record: its first 8 bytes, index (-1: none) and flags.
    auto publish = [&](int which, unsigned long long x, int idx, unsigned flags) {
        const unsigned ix = (unsigned)(idx + 1) | flags;
        if (G == 1) s_rec[which] = make_ulonglong2(x, ix);
        else st_half(recs + (which * G + g) * kRec, x, ix, epoch);
    };
    // One round trip for what a warp needs of this pivot: pending entries
    // (lane t: slot t's at pend + t * step, or own[t] with one CTA) into its
    // s_at, and in the lanes below the further values of cta1's record 1 and
    // cta2's record 2 (-1: not wanted).  A value is waited for until it
    // carries its pivot's tag: it was stored before a record already seen, so
    // it has nearly always arrived.
    constexpr int kRhs1 = 24, kVar1 = 25, kNum2 = 28, kDen2 = 29, kRcp2 = 30;
    auto fetch = [&](const ulonglong2 *pend, long long step, const T *own, int cta1, int cta2,
                     int fail) {
        unsigned long long v = 0;
        const int npend = kold + k, sl = slot(lane);
        const bool pnd = own != nullptr && lane < npend;
        if (G == 1) {
            v = pnd ? to_bits(own[sl]) : s_aux[ecur & 1][lane >= kNum2][lane & 3];
        } else {
            // (one address per lane, kept apart from how it was chosen: three
            // branches with a load each would wait for three round trips)
            unsigned long long at = 0;
            unsigned e = ecur;
            if (cta1 >= 0 && lane >= kRhs1 && lane <= kVar1)
                at = (unsigned long long)(further_at(e, 0, cta1) + lane - kRhs1);
            if (cta2 >= 0 && lane >= kNum2 && lane <= kRcp2)
                at = (unsigned long long)(further_at(e, 1, cta2) + lane - kNum2);
            if (pnd) at = (unsigned long long)(pend + sl * step), e = ecur - npend + lane;
            asm volatile("" : "+l"(at), "+r"(e));
            if (at) v = tagged(reinterpret_cast<const ulonglong2 *>(at), e, fail);
        }
        if (pnd) s_at[wid][sl] = from_bits<T>(v);
        __syncwarp();
        return v;
    };
    auto lane_value = [&](unsigned long long v, int l) {
        return from_bits<T>(__shfl_sync(kAll, v, l));
    };

    // The poll warps start once their CTA's own record is out (its group of
    // warps arrives at barrier id 3, columns, or 4, rows): polls while the
    // records are being worked out would only delay them.
    const int gate3 = cw + max(0, kPollFirst + kPollWarps - max(cw, kPollFirst));
    const int gate4 = rw + max(0, min(nw - rw, kPollFirst + kPollWarps) - kPollFirst);
    auto open_gate = [&](int id) {
        if (G > 1 && !poll_warp) group_arrive(id, id == 3 ? gate3 : gate4);
    };
    // The records of this lane in a poll warp, of pivot `epoch`; acquire: they
    // announce untagged data.  (One failure
    // flag per exchange: one exchange's flag is read by every thread before a
    // warp can be polling in the same exchange again.)
    auto poll = [&](int which, ulonglong2 (&v)[kPollRecs], bool acquire) {
        const int id = (which != 0) == DUAL ? 3 : 4;
        group_sync(id, id == 3 ? gate3 : gate4);
        const int e0 = (wid - kPollFirst) * 32 + lane;
        const ulonglong2 *rec = recs + which * G * kRec;
        const long long t0 = clock64();
        for (int spin = 0;; ++spin) {
            bool ok = true;
#pragma unroll
            for (int u = 0; u < kPollRecs; ++u)  // (past the last CTA: the last one's)
                v[u] = ld_half(rec + min(e0 + u * 32 * kPollWarps, G - 1) * kRec);
#pragma unroll
            for (int u = 0; u < kPollRecs; ++u) ok = ok && (unsigned)(v[u].y >> 32) == epoch;
            if (ok) break;
            if (clock64() - t0 > spin_limit || ((spin & 15) == 15 && *(volatile int *)err)) {
                atomicExch(err, 1);
                s_fail[which] = 1;
                break;
            }
        }
        if (acquire) __threadfence();
    };

    // Exchange 1: the smallest record 1 (Dantzig: by value, ties smallest
    // index; Bland: by index, the dual's by the leaving variable, which is
    // then the record's value).
    auto exchange1 = [&](bool bland) {
        Pick r;
        r.aux = r.zero = 0;
        // (the abort word is asked for a pivot ahead: it is in host memory)
        int ab = ab_next;
        if (tid == 32 * kPollFirst) {
            ab_next = abort_peek(abort_word);
            // (the wall-clock limit, in case the host is late with the word)
            if (limit_ns > 0 && global_ns() - t_start > (unsigned long long)limit_ns) ab = 1;
        }
        if (ab) {
            atomicExch(err, 1);
            s_fail[0] = 1;
        }
        if (G == 1) {
            cta_sync();
            const unsigned ix = (unsigned)s_rec[0].y;
            r.x = s_rec[0].x;
            r.idx = (int)(ix & kIdxMask) - 1;
            r.cta = 0;
            nodrop |= (int)(ix >> 31);
            return r;
        }
        if (poll_warp) {
            ulonglong2 v[kPollRecs];
            poll(0, v, k == K);  // (a full panel is applied next)
            const int e0 = (wid - kPollFirst) * 32 + lane;
            unsigned long long vk = ~0ull, x = 0;
            int key = 0x7fffffff, idx = -1, e = e0, flag = 0;
#pragma unroll
            for (int u = 0; u < kPollRecs; ++u) {
                if (e0 + u * 32 * kPollWarps >= G) continue;
                const unsigned ix = (unsigned)v[u].y;
                const int j = (int)(ix & kIdxMask) - 1;
                flag |= (int)(ix >> 31);
                if (j < 0) continue;
                const unsigned long long w = bland ? zero_k : okey(from_bits<T>(v[u].x));
                const int ky = DUAL && bland ? (int)(unsigned)v[u].x : j;
                if (w < vk || (w == vk && ky < key))
                    vk = w, key = ky, idx = j, x = v[u].x, e = e0 + u * 32 * kPollWarps;
            }
            const int l = min_lane(vk, key);
            flag = __any_sync(kAll, flag);
            if (lane == l) {
                Slot &s = s_ex1[wid - kPollFirst];
                s.vk = vk, s.key = key, s.idx = idx, s.x = x, s.src = e, s.flag = flag;
            }
        }
        cta_sync();
        int w = 0;
        unsigned long long bv = s_ex1[0].vk;
        int bk = s_ex1[0].key, fl = s_ex1[0].flag;
#pragma unroll
        for (int q = 1; q < kPollWarps; ++q) {
            const unsigned long long v = s_ex1[q].vk;
            const int ky = s_ex1[q].key;
            fl |= s_ex1[q].flag;
            if (v < bv || (v == bv && ky < bk)) bv = v, bk = ky, w = q;
        }
        nodrop |= fl;
        r.x = s_ex1[w].x;
        r.idx = s_ex1[w].idx;
        r.cta = s_ex1[w].src;
        return r;
    };

    // Exchange 2: the record 2 with the smallest ratio.  The records carry the
    // ratios' keys; numerators and denominators are fetched and divided only
    // when several keys are near the smallest, or one is out of range.
    auto exchange2 = [&](bool bland_keys) {
        Pick r;
        r.x = 0;
        if (G == 1) {
            cta_sync();
            const unsigned ix = (unsigned)s_rec[1].y;
            r.aux = (int)(s_rec[1].x >> 32);
            r.idx = (int)(ix & kIdxMask) - 1;
            r.cta = 0;
            r.zero = (ix & kFlagZero) != 0;
            nodrop |= (int)(ix >> 31);
            return r;
        }
        ulonglong2 v[kPollRecs];
        unsigned sk[kPollRecs];
        const int e0 = (wid - kPollFirst) * 32 + lane;
        if (poll_warp) {
            // (in turn: row p is read next, perhaps as the panel just left it; the
            // dual rule has read it already, behind a barrier)
            poll(1, v, !OV && !DUAL && k == 0);
            unsigned b1 = kNone, b2 = kNone, flag = 0;
            int at = 0;
#pragma unroll
            for (int u = 0; u < kPollRecs; ++u) {
                sk[u] = kNone;
                if (e0 + u * 32 * kPollWarps >= G) continue;
                flag |= (unsigned)v[u].y & (kFlagAll | kFlagWide);
                if (((unsigned)v[u].y & kIdxMask) == 0u) continue;
                sk[u] = (unsigned)v[u].x;
                if (sk[u] < b1) b2 = b1, b1 = sk[u], at = u;
                else if (sk[u] < b2) b2 = sk[u];
            }
            const unsigned m1 = __reduce_min_sync(kAll, b1);
            const int l = __ffs(__ballot_sync(kAll, b1 == m1)) - 1;
            const unsigned m2 = __reduce_min_sync(kAll, lane == l ? b2 : b1);
            flag = __reduce_or_sync(kAll, flag);
            if (lane == l) {
                Slot &s = s_ex2[wid - kPollFirst];
                ulonglong2 o = v[0];
#pragma unroll
                for (int u = 1; u < kPollRecs; ++u)
                    if (at == u) o = v[u];
                s.sk = m1, s.sk2 = m2, s.flag = (int)flag;
                s.idx = (int)(unsigned)o.y, s.aux = (int)(o.x >> 32);
                s.src = e0 + at * 32 * kPollWarps;
            }
        }
        cta_sync();
        r.idx = -1;
        r.aux = r.zero = r.cta = 0;
        int w = 0;
        unsigned fl = (unsigned)s_ex2[0].flag, bv = s_ex2[0].sk;
#pragma unroll
        for (int q = 1; q < kPollWarps; ++q) {
            fl |= (unsigned)s_ex2[q].flag;
            if (s_ex2[q].sk < bv) bv = s_ex2[q].sk, w = q;
        }
        nodrop |= (int)(fl >> 31);
        const bool wide = (fl & kFlagWide) != 0;
        if (bv == kNone) return r;
        int near = 0;
#pragma unroll
        for (int q = 0; q < kPollWarps; ++q)
            near += (s_ex2[q].sk <= bv + kNear) + (s_ex2[q].sk2 <= bv + kNear);
        const Slot *win = s_ex2 + w;
        if (near != 1 || wide) {
            if (poll_warp) {
                unsigned long long ek = ~0ull;
                int key = 0x7fffffff;
                unsigned ix = 0;
                int aux = 0, e = 0;
#pragma unroll
                for (int u = 0; u < kPollRecs; ++u) {
                    if (sk[u] == kNone || (!wide && sk[u] > bv + kNear)) continue;
                    const int c = e0 + u * 32 * kPollWarps;
                    unsigned long long q = zero_k;  // (in range, a zero key is a zero ratio)
                    if (wide || sk[u] != 0u) {
                        const ulonglong2 *ax = further_at(ecur, 1, c);
                        const T num = from_bits<T>(tagged(ax, ecur, 1));
                        const T den = from_bits<T>(tagged(ax + 1, ecur, 1));
                        q = okey(pos_part(num) / (DUAL ? neg(den) : den));
                    }
                    const int j = (int)((unsigned)v[u].y & kIdxMask) - 1;
                    const int ax1 = (int)(v[u].x >> 32), ky = bland_keys ? ax1 : j;
                    if (q < ek || (q == ek && ky < key))
                        ek = q, key = ky, ix = (unsigned)v[u].y, aux = ax1, e = c;
                }
                const int l = min_lane(ek, key);
                if (lane == l) {
                    Slot &s = s_ex3[wid - kPollFirst];
                    s.vk = ek, s.key = key, s.idx = (int)ix, s.aux = aux, s.src = e;
                }
            }
            cta_sync();
            win = s_ex3;
#pragma unroll
            for (int q = 1; q < kPollWarps; ++q)
                if (s_ex3[q].vk < win->vk || (s_ex3[q].vk == win->vk && s_ex3[q].key < win->key))
                    win = s_ex3 + q;
        }
        const unsigned ix = (unsigned)win->idx;
        r.idx = (int)(ix & kIdxMask) - 1;
        r.zero = (ix & kFlagZero) != 0;
        r.aux = win->aux;
        r.cta = win->src;
        return r;
    };

    // The smallest of the candidates (vk, key) of a group of nwarp warps
    // (this warp its w-th), whose lane publishes it as record 1: pub(loc,
    // flags), loc -1 for none.
    auto local_min = [&](int id, int w, int nwarp, unsigned long long vk, int key, int loc,
                         int flag, auto &&pub) {
        const int l = min_lane(vk, key);
        flag = __any_sync(kAll, flag);
        int win = 0;
        if (nwarp > 1) {
            if (lane == l) {
                Slot &s = s_loc[w];
                s.vk = vk, s.key = key, s.flag = flag;
            }
            group_sync(id, nwarp);
            unsigned long long bv = s_loc[0].vk;
            int bk = s_loc[0].key;
            flag = s_loc[0].flag;
            for (int q = 1; q < nwarp; ++q) {
                flag |= s_loc[q].flag;
                if (s_loc[q].vk < bv || (s_loc[q].vk == bv && s_loc[q].key < bk))
                    bv = s_loc[q].vk, bk = s_loc[q].key, win = q;
            }
        }
        if (w == win && lane == l) pub(loc, flag ? kFlagAll : 0u);
    };

    // The smallest ratio among a group's candidates, published as record 2.
    // sk1 (at loc) and sk2: this lane's two smallest ratio keys; wide: a
    // candidate was out of their range; each(f) calls f(loc, key) for this
    // lane's candidates; exact(loc, div, &key): the exactly divided ratio's key
    // (zero's where div is not set) and the tie key; pub(loc, key, flags), loc -1 for none.  Returns the published
    // loc in the lane that published it, -1 elsewhere.
    auto local_ratio = [&](int id, int w, int nwarp, unsigned sk1, unsigned sk2, int loc,
                           bool wide, int flag, auto &&each, auto &&exact, auto &&pub) {
        unsigned m1 = __reduce_min_sync(kAll, sk1);
        const int l = __ffs(__ballot_sync(kAll, sk1 == m1)) - 1;
        const unsigned m2 = __reduce_min_sync(kAll, lane == l ? sk2 : sk1);
        flag = __any_sync(kAll, flag);
        wide = __any_sync(kAll, wide);
        int win = 0, near = 0;
        if (nwarp > 1) {
            if (lane == 0) {
                Slot &s = s_loc[w];
                s.sk = m1, s.sk2 = m2, s.flag = flag, s.aux = wide;
            }
            group_sync(id, nwarp);
            m1 = kNone;
            flag = 0;
            for (int q = 0; q < nwarp; ++q) {
                flag |= s_loc[q].flag;
                wide |= s_loc[q].aux != 0;
                if (s_loc[q].sk < m1) m1 = s_loc[q].sk, win = q;
            }
            for (int q = 0; q < nwarp; ++q)
                near += (s_loc[q].sk <= m1 + kNear) + (s_loc[q].sk2 <= m1 + kNear);
        } else {
            near = 1 + (m2 <= m1 + kNear);
        }
        if (m1 == kNone) near = 0;
        const unsigned fl = (flag ? kFlagAll : 0u) | (wide ? kFlagWide : 0u);
        if (near <= 1 && !wide) {
            // (in range, a ratio is zero where its numerator is)
            if (w != win || lane != l) return -1;
            if (!near) loc = -1;
            pub(loc, m1, fl | (m1 == 0u ? kFlagZero : 0u));
            return loc;
        }
        unsigned long long ek = ~0ull;
        int key = 0x7fffffff, at = -1;
        each([&](int c, unsigned sk) {
            if (!wide && sk > m1 + kNear) return;
            int ky;  // (in range, a zero key is a zero ratio)
            const unsigned long long v = exact(c, wide || sk != 0u, &ky);
            if (v < ek || (v == ek && ky < key)) ek = v, key = ky, at = c, sk1 = sk;
        });
        const int l2 = min_lane(ek, key);
        win = 0;
        if (nwarp > 1) {
            group_sync(id, nwarp);  // s_loc was read
            if (lane == l2) {
                s_loc[w].vk = ek;
                s_loc[w].key = key;
            }
            group_sync(id, nwarp);
            for (int q = 1; q < nwarp; ++q)
                if (s_loc[q].vk < s_loc[win].vk ||
                    (s_loc[q].vk == s_loc[win].vk && s_loc[q].key < s_loc[win].key))
                    win = q;
        }
        if (w != win || lane != l2) return -1;
        pub(at, sk1, fl | (ek == zero_k ? kFlagZero : 0u));
        return at;
    };

    // The pending pivots on one entry.
    auto pending_chain = [&](T v, const T *c, const T *q) {
        if (OV && kold > 0) v = fma_chain(v, kold, c + ho, q + ho);
        return fma_chain(v, k, c + hn, q + hn);
    };
    // Column q on this CTA's rows (row warps), the pending pivots applied to
    // the tableau of the last panel.  Returns whether an entry is not finite.
    // f: what fetch() returned, for the caller.
    auto form_col = [&](int q, int cta1, int cta2, int which, unsigned long long *f) {
        int bad = 0;
        const int r1 = rt < R ? rt : 0;
        T v = R > 0 ? lds(Tab + (long long)(i0 + r1) * P + q) : (T)0;
        *f = fetch(PT + q, Np, prs + (G == 1 ? q * KS : 0), cta1, cta2, which);
        for (int r0 = rt - lane; r0 < R; r0 += B) {
            const int r = r0 + lane;
            const int rr = r < R ? r : 0;
            if (r0 != rt - lane) v = lds(Tab + (long long)(i0 + rr) * P + q);
            const int lp = lastp[rr];
            const T *c = cs + rr * KS;
            if (!__any_sync(kAll, lp >= 0)) {
                v = pending_chain(v, c, s_at[wid]);
            } else {  // a row that was a pivot row starts from that pivot's row
                if (lp >= 0) v = s_at[wid][lp];
                int pos = lp < 0 ? 0 : 1 + (OV && kold > 0 && (lp & K) == ho ? lp - ho : kold + lp - hn);
                for (; pos < kold + k; ++pos) {
                    const int t = slot(pos);
                    v = pfma(-c[t], s_at[wid][t], v);
                }
            }
            if (r < R) {
                cs[r * KS + hn + k] = v;
                if (G > 1) st_half(CT + (hn + k) * Mp + i0 + r, to_bits(v), ecur, nonce);
                bad |= not_finite(v);
            }
        }
        __syncwarp();
        return bad;
    };
    // An entry of row p (column c of the strip), from its value v in the last
    // panel's tableau; tp: the position of the last pending pivot with pivot row
    // p, or -1.
    auto form_row_elem = [&](T v, int tp, int c) {
        const T *pr = prs + c * KS;
        if (tp < 0) return pending_chain(v, s_at[wid], pr);
        v = pr[slot(tp)];
        for (int pos = tp + 1; pos < kold + k; ++pos) {
            const int t = slot(pos);
            v = pfma(-s_at[wid][t], pr[t], v);
        }
        return v;
    };
    auto last_pending = [&](int p) {
        const unsigned b =
            __ballot_sync(kAll, lane < kold + k && s_prow[slot(lane) & (NS - 1)] == p);
        return 31 - __clz((int)b);
    };
    // The rhs and the basis on this CTA's rows (row warps): the pivot in slot kk,
    // row p, entering column q.
    auto update_rhs = [&](int kk, int p, int q, T rhs_p, const Divisor &dv) {
        if (rt - lane >= R) return;
        const T rp = dv.div(rhs_p);
        for (int r = rt; r < R; r += B) {
            if (i0 + r == p) {
                rh[r] = rp;
                bas[r] = q;
                lastp[r] = (signed char)kk;
                if (DUAL) {
                    rowz[r] = 1;
                    s_nflag = 1;
                }
            } else {
                rh[r] = pfma(-cs[r * KS + kk], rp, rh[r]);
            }
        }
    };
    // Records 1 of the dual rule (row warps): the leaving row.  release: it
    // announces untagged data.
    auto publish_leaving = [&](bool bland, int flag, bool release) {
        unsigned long long vk = ~0ull;
        int key = 0x7fffffff, loc = -1;
        for (int r = rt; r < R; r += B) {
            const unsigned long long rk = okey(rh[r]);
            if (rk >= lim_r) continue;
            const unsigned long long v = bland ? zero_k : rk;
            const int ky = bland ? bas[r] : i0 + r;
            if (v < vk || (v == vk && ky < key)) vk = v, key = ky, loc = r;
        }
        local_min(2, nw - 1 - wid, rw, vk, key, loc, flag, [&](int l, unsigned fl) {
            if (release && G > 1) __threadfence();
            if (l < 0) {
                publish(0, 0ull, -1, fl);
            } else {
                const unsigned long long v = (unsigned)bas[l], x = to_bits(rh[l]);
                set_further(0, 0, x);
                set_further(0, 1, v);
                publish(0, bland ? v : x, i0 + l, fl);
            }
        });
    };
    // Records 1 of the primal rule (column warps): the entering column.
    auto publish_entering = [&](unsigned long long vk, int loc, int flag, bool release) {
        local_min(1, wid, cw, vk, loc < 0 ? 0x7fffffff : loc, loc, flag, [&](int c, unsigned fl) {
            if (release && G > 1) __threadfence();
            publish(0, c < 0 ? 0ull : to_bits(zs[c]), c < 0 ? -1 : c0 + c, fl);
        });
    };

    // ------------------------------------------------------------- pivots --
    if (OV) post(kJobCopy, 0, 0, false);
    if (!DUAL && col_warp) {
        const bool bland = deg >= bland_after;
        unsigned long long vk = ~0ull;
        int loc = -1;
        for (int c = ct; c < W; c += B) {
            const unsigned long long zk = okey(zs[c]);
            if (c0 + c >= N - 1 || zk >= lim_d) continue;
            const unsigned long long v = bland ? zero_k : zk;
            if (v < vk) vk = v, loc = c;
        }
        publish_entering(vk, loc, 0, false);
        open_gate(3);
    }
    if (DUAL && row_warp) {
        publish_leaving(deg >= bland_after, 0, false);
        open_gate(4);
    }

    for (;;) {
        const bool bland = deg >= bland_after;
        ecur = epoch;
        const Pick e1 = exchange1(bland);
        if (s_fail[0]) {
            status = ST_TIMEOUT;
            break;
        }
        if (e1.idx < 0) {
            status = ST_OPTIMAL;
            break;
        }
        if (iters >= iter_limit) {
            status = ST_ITER_LIMIT;
            break;
        }
        if (k == K) {
            if constexpr (OV) {
                // every CTA's panel (or copy) is done: its record says so
                if (jobs > 1) cur ^= 1, Tab = bufs[cur];
                const bool all = !drop || nodrop;
                for (int w = tid; w < nwords; w += B) {
                    out[w] = left_out_of_panel(prev[w], stay[w], all, past_end(w, N));
                    stay[w] = bb[w];
                }
                for (int r = tid; r < R; r += B)  // (the other half's slots are used again)
                    if (lastp[r] >= 0 && (lastp[r] & K) != hn) lastp[r] = -1;
                ho = hn;
                hn ^= K;
                kold = K;
                k = 0;
                nodrop = 0;
                post(kJobPanel, ho, K, all);
            } else {
                apply_panel(k);
                k = 0;
                // (the dual rule reads other CTAs' rows next)
                if (DUAL && !group_barrier()) {
                    status = ST_TIMEOUT;
                    break;
                }
            }
        }
        int p, q, var = 0;            // leaving row, entering column, leaving variable
        T zq = (T)0;                  // objective entry of q
        if (!DUAL) {
            q = e1.idx;
            zq = from_bits<T>(e1.x);
            if (row_warp) {
                // column q and the ratio test over this CTA's rows (Step 3)
                unsigned long long f;
                const int bad = form_col(q, -1, -1, 1, &f);
                unsigned sk1 = kNone, sk2 = kNone;
                bool wide = false;
                int loc = -1;
                for (int r = rt; r < R; r += B) {
                    const T a = cs[r * KS + hn + k];
                    if (okey(a) <= lim_p) continue;
                    const unsigned sk = ratio_key(pos_part(rh[r]), a, &wide);
                    if (sk < sk1) sk2 = sk1, sk1 = sk, loc = r;
                    else if (sk < sk2) sk2 = sk;
                }
                const int mine = local_ratio(
                    2, nw - 1 - wid, rw, sk1, sk2, loc, wide, bad,
                    [&](auto &&f) {
                        for (int r = rt; r < R; r += B) {
                            const T a = cs[r * KS + hn + k];
                            bool w;
                            if (okey(a) > lim_p) f(r, ratio_key(pos_part(rh[r]), a, &w));
                        }
                    },
                    [&](int r, bool div, int *key) {
                        *key = bland ? bas[r] : i0 + r;
                        return div ? okey(pos_part(rh[r]) / cs[r * KS + hn + k]) : zero_k;
                    },
                    [&](int r, unsigned sk, unsigned fl) {
                        publish(1, r < 0 ? 0ull : ((unsigned long long)(unsigned)bas[r] << 32) | sk,
                                r < 0 ? -1 : i0 + r, fl);
                        if (r < 0) return;
                        set_further(1, 0, to_bits(rh[r]));
                        set_further(1, 1, to_bits(cs[r * KS + hn + k]));
                    });
                open_gate(4);
                // (the reciprocal follows while the records are exchanged)
                if (mine >= 0) set_further(1, 2, to_bits(Divisor::recip(cs[mine * KS + hn + k])));
                __syncwarp();
            }
        } else {
            p = e1.idx;
            if (col_warp) {
                // row p and the ratio test over this CTA's columns
                const T first = lds(Tab + (long long)p * P + c0 + min(ct, W - 1));
                const unsigned long long f =
                    fetch(CT + p, Mp, cs + (G == 1 ? p * KS : 0), e1.cta, -1, 1);
                const int tp = last_pending(p);
                var = (int)__shfl_sync(kAll, f, kVar1);
                int bad = 0;
                unsigned sk1 = kNone, sk2 = kNone;
                bool wide = false;
                int loc = -1;
                for (int q0 = ct - lane; q0 < W; q0 += B) {
                    const int c = q0 + lane;
                    const bool act = c < W;
                    const int cc = act ? c : W - 1, j = c0 + cc;
                    T v = q0 == ct - lane ? first : lds(Tab + (long long)p * P + j);
                    v = form_row_elem(v, tp, cc);
                    if (!act) continue;
                    prs[c * KS + hn + k] = v;
                    bad |= j != var && (stay[j >> 5] >> (j & 31) & 1u) && !is_zero(v);
                    if (j >= N - 1 || okey(v) >= lim_np) continue;
                    const unsigned sk = ratio_key(pos_part(zs[c]), neg(v), &wide);
                    if (sk < sk1) sk2 = sk1, sk1 = sk, loc = c;
                    else if (sk < sk2) sk2 = sk;
                }
                __syncwarp();
                const int mine = local_ratio(
                    1, wid, cw, sk1, sk2, loc, wide, bad,
                    [&](auto &&f) {
                        for (int c = ct; c < W; c += B) {
                            bool w;
                            const T v = prs[c * KS + hn + k];
                            if (c0 + c < N - 1 && okey(v) < lim_np)
                                f(c, ratio_key(pos_part(zs[c]), neg(v), &w));
                        }
                    },
                    [&](int c, bool div, int *key) {
                        *key = c0 + c;
                        return div ? okey(pos_part(zs[c]) / neg(prs[c * KS + hn + k])) : zero_k;
                    },
                    [&](int c, unsigned sk, unsigned fl) {
                        publish(1, sk, c < 0 ? -1 : c0 + c, fl);
                        if (c < 0) return;
                        set_further(1, 0, to_bits(zs[c]));
                        set_further(1, 1, to_bits(prs[c * KS + hn + k]));
                    });
                open_gate(3);
                if (mine >= 0) set_further(1, 2, to_bits(Divisor::recip(prs[mine * KS + hn + k])));
                __syncwarp();
            }
        }
        const Pick e2 = exchange2(!DUAL && bland);
        if (s_fail[1]) {
            status = ST_TIMEOUT;
            break;
        }
        if (e2.idx < 0) {
            status = DUAL ? ST_INFEASIBLE : ST_UNBOUNDED;
            break;
        }
        if (!DUAL) {
            p = e2.idx;
            var = e2.aux;
        } else {
            q = e2.idx;
        }
        deg = e2.zero ? deg + 1 : 0;
        const bool nbland = deg >= bland_after;  // rule of the next selection
        ++epoch;
        const int kc = k;  // this pivot's number in the panel
        ++iters;
        last_p = p;
        last_q = q;
        if (wid == kPollFirst) {
            if (DUAL)
                var = (int)__shfl_sync(kAll, fetch(nullptr, 0, nullptr, e1.cta, -1, 0), kVar1);
            if (lane == 0) {
                change_basis(bb, stay, var, q, N);
                if (g == 0 && iters <= trace_cap) {
                    d->trace[2 * iters - 2] = p;
                    d->trace[2 * iters - 1] = q;
                }
            }
            __syncwarp();
        }
        // ---- Step 4 on this CTA's columns, the objective row, pricing ----
        if (col_warp) {
            const T *rowp = Tab + (long long)p * P + c0;
            T first = (T)0;
            int tp = -1;
            unsigned long long f;
            if (!DUAL) {
                first = lds(rowp + min(ct, W - 1));
                f = fetch(CT + p, Mp, cs + (G == 1 ? p * KS : 0), -1, e2.cta, 0);
                tp = last_pending(p);
            } else {
                f = fetch(nullptr, 0, nullptr, -1, e2.cta, 0);
                zq = lane_value(f, kNum2);
            }
            const Divisor dv(lane_value(f, kDen2), lane_value(f, kRcp2));
            unsigned long long vk = ~0ull;
            int loc = -1, flag = 0;
            for (int q0 = ct - lane; q0 < W; q0 += B) {
                const int c = q0 + lane;
                const bool act = c < W;
                const int cc = act ? c : W - 1, j = c0 + cc;
                T v;
                if (!DUAL) {
                    v = q0 == ct - lane ? first : lds(rowp + cc);
                    v = form_row_elem(v, tp, cc);
                } else {
                    v = prs[cc * KS + hn + kc];
                }
                if (!act) continue;
                if (!DUAL) flag |= j != var && (stay[j >> 5] >> (j & 31) & 1u) && !is_zero(v);
                const T pr = dv.div(v);
                prs[c * KS + hn + kc] = pr;
                if (G > 1) st_half(PT + (hn + kc) * Np + j, to_bits(pr), ecur, nonce);
                __stcg(PR + (hn + kc) * P + j, pr);
                const T z = pfma(-zq, pr, zs[c]);
                zs[c] = z;
                if (!DUAL) {
                    const unsigned long long zk = okey(z);
                    if (j >= N - 1 || zk >= lim_d) continue;
                    const unsigned long long w = nbland ? zero_k : zk;
                    if (w < vk) vk = w, loc = c;
                }
            }
            __syncwarp();
            // a full panel is applied after the next records: this CTA's
            // announces the rows it reads, and what the panel before it wrote
            if (!DUAL) {
                if (OV && kc + 1 == K) wait_job(true);
                k = kc + 1;
                publish_entering(vk, loc, flag, kc + 1 == K);
                open_gate(3);
            }
        }
        if (DUAL) {
            int bad = 0;
            k = kc;
            unsigned long long f = 0;
            if (row_warp) bad = form_col(q, e1.cta, e2.cta, 0, &f);
            // (as above; the row warps publish, the column warps wrote the rows)
            if (kc + 1 == K) {
                if (OV) wait_job(true);
                cta_sync();
            }
            k = kc + 1;
            if (row_warp) {
                update_rhs(hn + kc, p, q, lane_value(f, kRhs1),
                           Divisor(lane_value(f, kDen2), lane_value(f, kRcp2)));
                __syncwarp();
                publish_leaving(nbland, bad, kc + 1 == K);
                open_gate(4);
            }
        } else if (row_warp) {
            const unsigned long long f = fetch(nullptr, 0, nullptr, -1, e2.cta, 0);
            update_rhs(hn + kc, p, q, lane_value(f, kNum2),
                       Divisor(lane_value(f, kDen2), lane_value(f, kRcp2)));
        }
        if (OV && !DUAL && !col_warp && kc + 1 == K) wait_job(false);
        k = kc + 1;
        if (tid == 0) s_prow[hn + kc] = p;
    }

    // --------------------------------------------------------------- end --
    if constexpr (OV) {
        if (k < K) wait_job(true);  // (at the last pivot of a panel it was waited for)
        // (every CTA takes this branch: the records decide, and they agree)
        if (status != ST_TIMEOUT && !group_barrier()) status = ST_TIMEOUT;
        if (status != ST_TIMEOUT) {
            if (jobs > 1) cur ^= 1, Tab = bufs[cur];
            if (k > 0) {
                for (int w = tid; w < nwords; w += B) out[w] = stay[w];
                post(kJobInPlace, hn, k, !drop || nodrop);
                wait_job(true);
            }
        }
        post(kJobEnd, 0, 0, false);
    } else if (status != ST_TIMEOUT && k > 0) {
        if (group_barrier()) apply_panel(k);
        else status = ST_TIMEOUT;
    }
    cta_sync();
    {
        T *z = Tab + (long long)m * P;
        for (int c = tid; c < W; c += B) z[c0 + c] = zs[c];
        for (int r = tid; r < R; r += B) d->basis[i0 + r] = bas[r], marks[i0 + r] = rowz[r];
    }
    if (g == 0 && tid == 0) {
        d->status = (*(volatile int *)err) ? ST_TIMEOUT : status;
        d->iters = iters;
        d->iter_limit = iter_limit;
        d->deg = deg;
        d->last_p = last_p;
        d->last_q = last_q;
        d->epoch = epoch;
        if (OV) {
            if (status != ST_TIMEOUT) d->T = Tab, d->T2 = bufs[cur ^ 1];
        } else if (d->work) {
            d->work[0] += upd;
            d->work[1] += left;
        }
    }
}

// The tags of one load's launches: its nonce, and pivot numbers that go on from
// launch to launch.  Both are in the descriptor, not among the launch's
// arguments, so a launch that was captured once and runs many times meets no
// tag of an earlier run.
__device__ __forceinline__ unsigned numbers_used(const LpDesc *d) {
    return d->epoch < 0x80000000u ? d->epoch : 0u;
}

template <typename T, bool DUAL>
__global__ void __launch_bounds__(kPanelThreads, 1)
    panel_kernel(LpDesc *__restrict__ d, long long spin_limit, long long budget, int drop,
                 long long limit_ns) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    panel_solve<T, DUAL, kPanelK, false>(d, gridDim.x, blockIdx.x, spin_limit, budget, drop, d->nonce,
                                         numbers_used(d), limit_ns, smem_raw);
}

template <bool DUAL>
__global__ void __launch_bounds__(2 * kPanelThreads, 1)
    panel_overlap_kernel(LpDesc *__restrict__ d, long long spin_limit, long long budget, int drop,
                         long long limit_ns) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    panel_solve<double, DUAL, kPanelOverlapK, true>(d, gridDim.x, blockIdx.x, spin_limit, budget,
                                                    drop, d->nonce, numbers_used(d), limit_ns,
                                                    smem_raw);
}

// Many LPs in one launch.  items[] lists (lp, rank) pairs, the ranks of one LP
// consecutive, largest LPs first; CTAs pop items in order from *queue, and the
// d->group CTAs that pop the ranks of one LP solve it together.  A group waits
// only on CTAs that hold earlier items, whose groups are complete, so every
// group forms (the launch has at least max(group) co-resident CTAs).  Two CTAs
// per SM (128 registers a thread, panels of 8): one LP's selection chain
// overlaps another's panels.  Columns that stay basic are always left out, whatever
// lp_options.zero_skip: with every column updated 6 LPs of 800 x 800 take 7.7 ms, 3.8
// without, 4.5 with the kernel that updates the tableau every pivot.
template <typename T>
__global__ void __launch_bounds__(kPanelThreads, 2)
    panel_batch_kernel(LpDesc *__restrict__ descs, const int2 *__restrict__ items, int nitems,
                       unsigned *queue, long long spin_limit, long long budget, unsigned nonce) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (int)atomicAdd(queue, 1u);
        __syncthreads();
        const int it = s_item;
        if (it >= nitems) break;
        const int2 w = items[it];
        LpDesc *d = descs + w.x;
        if (d->sense)
            panel_solve<T, true, kPanelBatchK, false>(d, d->group, w.y, spin_limit, budget, 1, nonce, 0,
                                                      0, smem_raw);
        else
            panel_solve<T, false, kPanelBatchK, false>(d, d->group, w.y, spin_limit, budget, 1, nonce, 0,
                                                       0, smem_raw);
    }
}

}  // namespace

unsigned panel_nonce() {
    static std::atomic<unsigned> taken{0};
    return ++taken;
}

PivotShape choose_panel_shape(int prec, int M, int N, int sms, int ctas, int dual, int drop,
                              bool overlap) {
    PivotShape sh;
    const int m = M - 1;
    // Default grid: every SM, on small LPs one CTA per two rows or 32 columns,
    // whichever gives more (one row per CTA measured no faster: 64^2 6.4 us per
    // pivot on 32 CTAs, 6.5 on 16 and 64, 6.7 on 152, 6.8 on one; 256^2 7.1 on 114
    // and on 152).
    int G = ctas > 0 ? ctas : std::max((m + 1) / 2, (N + 31) / 32);
    G = std::min(G, std::min(sms, kPanelMaxCtas));
    G = std::max(1, std::min(G, N));
    const size_t smem = panel_smem(prec, m, N, G, kPanelK, overlap);
    sh.ctas = G;
    sh.threads = overlap ? 2 * kPanelThreads : kPanelThreads;
    sh.dual = dual;
    sh.drop = drop;
    sh.use_smem = 1;
    sh.smem_bytes = smem;
    sh.pipe = smem > kMaxDynSmem ? 0 : overlap ? 5 : 4;
    return sh;
}

size_t panel_workspace(int prec, int m, long long N, long long P, int G, int K) {
    const size_t esz = prec == PREC_FP64 ? 8 : 4;
    return panel_tagged(m, N, G, K) + (size_t)K * (size_t)P * esz + (size_t)m;
}

size_t panel_tagged(int m, long long N, int G, int K) {
    return G > 1 ? (size_t)K * (size_t)(tag_pitch(m) + tag_pitch(N)) * 16 + 256 * (size_t)G : 0;
}

size_t panel_smem(int prec, int m, int N, int G, int K, bool overlap) {
    return panel_layout(m, N, G, prec == PREC_FP64 ? 8 : 4, prec == PREC_FP64 ? 2 : 4, K, overlap).total;
}

cudaError_t launch_panel(int prec, LpDesc *d_desc, const PivotShape &sh, long long spin_limit,
                         long long budget, cudaStream_t s) {
    int drop = sh.drop;
    long long limit_ns = sh.limit_ns;
    void *args[] = {&d_desc, &spin_limit, &budget, &drop, &limit_ns};
    const void *fn = sh.pipe == 5 ? (sh.dual ? (const void *)panel_overlap_kernel<true>
                                             : (const void *)panel_overlap_kernel<false>)
                     : prec == PREC_FP64 ? (sh.dual ? (const void *)panel_kernel<double, true>
                                                    : (const void *)panel_kernel<double, false>)
                                         : (sh.dual ? (const void *)panel_kernel<float, true>
                                                    : (const void *)panel_kernel<float, false>);
    cudaError_t e = allow_dyn_smem(fn);
    if (e != cudaSuccess) return e;
    // A cooperative launch fails instead of running when the grid cannot be
    // co-resident, which the record exchanges need.
    return cudaLaunchCooperativeKernel(fn, dim3(sh.ctas), dim3(sh.threads), args, sh.smem_bytes, s);
}

cudaError_t launch_panel_batch(int prec, LpDesc *descs, const int2 *items, int nitems,
                               unsigned *queue, int ctas, size_t smem, long long spin_limit,
                               long long budget, cudaStream_t s) {
    unsigned nonce = panel_nonce();
    void *args[] = {&descs, &items, &nitems, &queue, &spin_limit, &budget, &nonce};
    const void *fn = prec == PREC_FP64 ? (const void *)panel_batch_kernel<double>
                                       : (const void *)panel_batch_kernel<float>;
    cudaError_t e = allow_dyn_smem(fn);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(fn, dim3(ctas), dim3(kPanelThreads), args, smem, s);
}

int max_coresident_panel_batch_ctas(int prec, size_t smem, int sms) {
    const void *fn = prec == PREC_FP64 ? (const void *)panel_batch_kernel<double>
                                       : (const void *)panel_batch_kernel<float>;
    allow_dyn_smem(fn);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kPanelThreads, smem) !=
        cudaSuccess)
        return 0;
    return per_sm * sms;
}

}  // namespace gbs
