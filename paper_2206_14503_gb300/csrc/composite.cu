// Phase 2: compositing of K compact sub-VDIs into one regular VDI (sec. 5.2,
// Eq. 2, Algorithm S1).
//
// The paper's all-to-all exchange becomes a gather: pixel p's input is its K
// spans [offsets_e[p], offsets_e[p] + counts_e[p]) in the K PEs' record
// arrays.  A depth sweep over the K lists (each depth-sorted, sec. 5.2) cuts
// the records at every front and back depth and yields the pieces in order:
//   - a gap between records: a transparent sample;
//   - an interval covered by one record whole: that record, unchanged;
//   - part of one record: opacity by Eq. 2, 1 - (1 - A)^(dt / l);
//   - an interval covered by several records: their emission-absorption
//     mixture (extinctions add; colour is the extinction-weighted mean), summed
//     exactly in 128-bit fixed point so that every schedule gets the same bits.
// The pieces feed the supersegment state machine (Eq. 1) inside the per-pixel
// bisection search for gamma: a march evaluates several midpoints at once and
// the sequential bisection is replayed from their counts, marching again only
// for a midpoint without one, so the result is that of plain bisection.  The
// flat search evaluates the four likeliest midpoints (vdi_search.cuh); the
// direct sweeps the next two levels (midpoint and both children), recording per
// candidate the interval of gamma over which all of its decisions repeat, and
// count the non-transparent pieces (the count at gamma = 0) in their first
// march.  A final sweep emits at most n_s supersegments into the regular layout with a
// zero tail.
//
// Schedules (the same result, bit for bit; chosen per request by the
// autotuner, vdi_composite_autotune; the default is the lane schedule for
// K <= 8 and the staged one above):
//   VDI_SCHED_LANE (5, K <= 8): composite_lane_kernel copies a warp's 32
//     pixels' records into shared memory with asynchronous coalesced copies
//     and sweeps each pixel there once (a lane each; depth-disjoint lists, as
//     every box decomposition gives, without the K-head merge): the pixels
//     whose gamma = 0 count is within n_s are emitted, the others' pieces go
//     to a pool in the workspace; the list of those pixels is sorted by piece
//     count (list_hist / list_offsets / list_scatter) and
//     composite_flat_kernel searches and emits them;
//   VDI_SCHED_STAGED (4): composite_build_kernel builds each pixel's pieces
//     with a warp, or four for long lists (coalesced span loads, merge-path sort
//     of the bounds, exact prefix scan of the mixture terms) into the pool, and
//     composite_flat_kernel searches and emits every pixel; the host runs the
//     pixels in chunks whose pieces fit the pool;
//   both list pixels they cannot stage (more than 480 / 1024 records, pieces
//     beyond the pool, lists out of depth order, values that the packed search
//     does not take: packable) for composite_marked_kernel, the direct sweep;
//   1, 2, 3 (direct, composite_kernel): one thread per pixel re-sweeps its K
//     lists on every march, heads in registers (1, K <= 8) or in shared memory
//     under a winner tree (2; 3 with three levels per march).
// composite_flat_kernel runs the search and the emission as one loop whose
// body handles four pieces of a lane's current march, so lanes at different
// marches or pixels execute the same instructions; lanes at the end of a
// march wait for others to end theirs together, and a lane that finishes its
// pixel takes the next one.
//
// The batched path runs many requests (different sizes, K, N_S) as the pooled
// staged schedule does: composite_batched_build_kernel pulls (request, 32-pixel
// batch) items from an atomic counter and builds them into the pool,
// composite_batched_flat_kernel searches and emits, and requests with a direct
// schedule (and pixels the stage cannot hold) go to
// composite_batched_marked_kernel.
#include <climits>

#include "vdi_search.cuh"

namespace vdi {

struct PeIn {
    const uint32_t* counts;
    const uint64_t* offsets;
    const void* rgba;
    const float2* fb;
};

struct OutDev {
    uint32_t* counts;
    void* rgba;
    float2* fb;
    float* gamma;
    int n_s;
    int prec;
};

struct CompArgs {
    PeIn pe[VDI_MAX_PE];
    OutDev out;
    int k, npix, iters;
    unsigned int* status;
};

struct Piece {
    float f, b;
    float P[3];
    float a;
    float lgT;  // log2(1 - a)
};

template <int PREC>
__device__ __forceinline__ void load_fb(const PeIn& pe, uint64_t idx, float& f, float& b) {
    if (PREC == VDI_PREC_F32) {
        float2 v = __ldg(pe.fb + idx);
        f = v.x;
        b = v.y;
    } else {
        float2 v = __ldg(reinterpret_cast<const float2*>(reinterpret_cast<const uint4*>(pe.rgba) + idx));
        f = v.x;
        b = v.y;
    }
}

// A record's premultiplied colour and opacity, and its optical depth tau =
// -log2(1 - A): computed from A for FP32 records, stored for FP16 ones.  A
// record is opaque iff tau is not finite (A >= 1 for FP32 records).
struct RecC {
    float4 c;
    float tau;
};

template <int PREC>
__device__ __forceinline__ RecC load_rec(const PeIn& pe, uint64_t idx) {
    RecC r;
    if (PREC == VDI_PREC_F32) {
        r.c = __ldg(reinterpret_cast<const float4*>(pe.rgba) + idx);
        r.tau = -lg2_approx(__fsub_rn(1.f, r.c.w));
    } else {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const uint4*>(pe.rgba) + idx) + 1);
        f16_unpack_col(v, r.c, r.tau);
    }
    return r;
}

__device__ __forceinline__ bool rec_opaque(const RecC& r) { return !(r.tau < INFINITY); }

// ---------------------------------------------------------------------------
// Piece sweep
// ---------------------------------------------------------------------------
// The pieces of a pixel are the intervals between consecutive distinct record
// bounds of its K lists.  A sweep keeps one head per PE (its current record)
// and processes the bounds in depth order as events: a record's front starts
// it, its back ends it and moves the head to the PE's next record with b > f.
// The emission-absorption mixture of the active records is kept as exact
// running sums, updated once per event: the extinction mu = -log2(1 - A) / l
// and mu times the unpremultiplied colour of every non-opaque record are
// summed in 128-bit fixed point (64 integer and 64 fraction bits; a record's
// terms are computed the same way at its start and at its end, so the sum of
// the active records is exact however many events came before).  Opaque
// records (A >= 1) are counted, with their colours summed.

struct U128 {
    unsigned long long hi, lo;
};

__device__ __forceinline__ void u128_add(U128& s, const U128& x) {
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(s.lo), "+l"(s.hi) : "l"(x.lo), "l"(x.hi));
}

__device__ __forceinline__ void u128_sub(U128& s, const U128& x) {
    asm("sub.cc.u64 %0, %0, %2;\n\tsubc.u64 %1, %1, %3;" : "+l"(s.lo), "+l"(s.hi) : "l"(x.lo), "l"(x.hi));
}

// s + x, or s - x where neg is all ones (s + ~x + 1), without a branch
__device__ __forceinline__ void u128_add_signed(U128& s, const U128& x, unsigned long long neg) {
    asm("{\n\t.reg .u64 t;\n\tadd.cc.u64 t, %4, %4;\n\taddc.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;\n\t}"
        : "+l"(s.lo), "+l"(s.hi)
        : "l"(x.lo ^ neg), "l"(x.hi ^ neg), "l"(neg));
}

// The conversions between FP32 and this format, v in [0, 2^56] as fixed point: exact for v >= 2^-41 (the 24-bit
// significand fits the 64 fraction bits), truncated below.
__device__ __forceinline__ U128 to_fixed(float v) {
    const float ip = truncf(v);
    U128 r;
    r.hi = __float2ull_rz(ip);
    r.lo = __float2ull_rz(__fmul_rn(__fsub_rn(v, ip), 18446744073709551616.f));
    return r;
}

__device__ __forceinline__ float from_fixed(const U128& s) {
    return __fmaf_rn(__ull2float_rn(s.lo), 5.421010862427522e-20f, __ull2float_rn(s.hi));
}

// The same conversions (the same bits) in 32-bit integer operations, for the pooled build, whose warps are full: the
// hardware's conversions to and from 64-bit integers run on the FP64 pipe, 2 lanes an SM on this chip (16 cycles a
// warp for each, 8 of them per bound and per piece: more than half of the pooled build's time).  The sweeps keep the
// hardware's: they convert in code of its own for each of up to eight heads, with few lanes at work, and the integer
// form makes that code several times as long (320 x 240, K = 8, lane schedule: N_S = 32 dense 264 ms with the integer
// form, 122 with the hardware's; N_S = 4 ragged 1.68 and 1.32; N_S = 12 dense 14.1 and 16.5).

// the significand shifted to its place
__device__ __forceinline__ U128 to_fixed_int(float v) {
    const uint32_t bits = __float_as_uint(v);
    const int sh = (int)(bits >> 23) - 86;  // of the significand's last bit, from the last fraction bit
    const uint32_t m = (bits & 0x7FFFFFu) | 0x800000u;
    const uint32_t lo = sh < 0 ? (sh > -32 ? m >> -sh : 0u) : m << (sh & 31);
    const uint32_t hi = sh < 0 ? 0u : __funnelshift_l(m, 0u, sh & 31);
    const int w = sh < 0 ? 0 : sh >> 5;  // the 32-bit word that lo falls in (at most 3)
    const uint32_t w0 = w == 0 ? lo : 0u, w1 = w == 0 ? hi : (w == 1 ? lo : 0u);
    const uint32_t w2 = w == 1 ? hi : (w == 2 ? lo : 0u), w3 = w == 2 ? hi : (w == 3 ? lo : 0u);
    U128 r;
    r.lo = (unsigned long long)w1 << 32 | w0;
    r.hi = (unsigned long long)w3 << 32 | w2;
    return r;
}

// x rounded to nearest even: its top 32 bits, the rest folded into the last of them, converted and scaled
__device__ __forceinline__ float u64_to_float(unsigned long long x) {
    const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    const int z = __clz(hi);  // 32 where hi is 0
    const uint32_t top = hi ? __funnelshift_l(lo, hi, z) : lo;
    const uint32_t sticky = hi && (lo << (z & 31)) != 0u ? 1u : 0u;
    return __fmul_rn(__uint2float_rn(top | sticky), __uint_as_float((uint32_t)(159 - z) << 23));  // 2^(32 - z)
}

__device__ __forceinline__ float from_fixed_int(const U128& s) {
    return __fmaf_rn(u64_to_float(s.lo), 5.421010862427522e-20f, u64_to_float(s.hi));
}

// Clamp of a record's extinction terms (per unit depth): a record shorter than
// ~3e-16 depth units with non-zero opacity is treated as having mu = 2^56, so
// that 64 PEs' sums stay below 2^64.
constexpr float kMuMax = 72057594037927936.f;  // 2^56

// A record's terms: extinction mu = -log2(1 - A) / (b - f) and mu times the
// unpremultiplied colour (non-opaque records), or its colour (opaque records).
struct Contrib {
    U128 M, MC[3], OC[3];
    int op;  // 1 if opaque
};

__device__ __forceinline__ void u128_zero(U128& x) { x.hi = x.lo = 0ull; }

__device__ __forceinline__ Contrib contrib(const RecC& x, float f, float b) {
    Contrib r;
    u128_zero(r.M);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        u128_zero(r.MC[q]);
        u128_zero(r.OC[q]);
    }
    r.op = 0;
    const float4& c = x.c;
    const float col[3] = {c.x, c.y, c.z};
    if (rec_opaque(x)) {
        r.op = 1;
#pragma unroll
        for (int q = 0; q < 3; ++q) r.OC[q] = to_fixed(fminf(fmaxf(col[q], 0.f), kMuMax));
    } else if (c.w > 0.f) {
        const float ia = rcp_approx(c.w);
        const float mu = fminf(__fmul_rn(x.tau, rcp_approx(__fsub_rn(b, f))), kMuMax);
        r.M = to_fixed(mu);
#pragma unroll
        for (int q = 0; q < 3; ++q) r.MC[q] = to_fixed(fminf(fmaxf(__fmul_rn(mu, __fmul_rn(col[q], ia)), 0.f), kMuMax));
    }
    return r;
}

// A record's terms before their conversion to fixed point, as contrib computes them: extinction mu and mu times the
// colour (all 0 for a transparent record), or -1 and the colour of an opaque one.
__device__ __forceinline__ float4 record_terms(const RecC& x, float f, float b) {
    const float col[3] = {x.c.x, x.c.y, x.c.z};
    float t[3] = {0.f, 0.f, 0.f}, mu = 0.f;
    if (rec_opaque(x)) {
        mu = -1.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) t[q] = fminf(fmaxf(col[q], 0.f), kMuMax);
    } else if (x.c.w > 0.f) {
        const float ia = rcp_approx(x.c.w);
        mu = fminf(__fmul_rn(x.tau, rcp_approx(__fsub_rn(b, f))), kMuMax);
#pragma unroll
        for (int q = 0; q < 3; ++q) t[q] = fminf(fmaxf(__fmul_rn(mu, __fmul_rn(col[q], ia)), 0.f), kMuMax);
    }
    return make_float4(t[0], t[1], t[2], mu);
}

template <bool OPQ>
__device__ __forceinline__ Contrib contrib_of(const float4& t) {
    Contrib r;
    const bool op = OPQ && t.w < 0.f;
    r.op = op ? 1 : 0;
    const float v[3] = {t.x, t.y, t.z};
    r.M = to_fixed_int(op ? 0.f : t.w);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const U128 x = to_fixed_int(v[q]);
        u128_zero(r.MC[q]);
        u128_zero(r.OC[q]);
        if (op) r.OC[q] = x;
        else r.MC[q] = x;
    }
    return r;
}

// Sums over the active records.
struct MixSums {
    U128 M, MC[3], OC[3];
    int nop, nact;
};

__device__ __forceinline__ void sums_reset(MixSums& m) {
    u128_zero(m.M);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        u128_zero(m.MC[q]);
        u128_zero(m.OC[q]);
    }
    m.nop = m.nact = 0;
}

// OPQ = false: the caller knows that no record is opaque (the OC sums stay 0)
template <bool ADD, bool OPQ = true>
__device__ __forceinline__ void sums_update(MixSums& m, const Contrib& x) {
    if (ADD) {
        u128_add(m.M, x.M);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            u128_add(m.MC[q], x.MC[q]);
            if (OPQ) u128_add(m.OC[q], x.OC[q]);
        }
        m.nop += x.op;
        ++m.nact;
    } else {
        u128_sub(m.M, x.M);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            u128_sub(m.MC[q], x.MC[q]);
            if (OPQ) u128_sub(m.OC[q], x.OC[q]);
        }
        m.nop -= x.op;
        --m.nact;
    }
}

// The piece [t, t1] of an active set with sums m; `whole` when exactly one
// record is active and it spans [t, t1] (its colour and opacity are wc).
// INT: with the integer conversion.
template <bool INT = false>
__device__ __forceinline__ void piece_from(const MixSums& m, bool whole, const RecC& wr, float t, float t1,
                                           Piece& x) {
    const auto value = [](const U128& v) { return INT ? from_fixed_int(v) : from_fixed(v); };
    x.f = t;
    x.b = t1;
    if (whole) {
        // one record covering the piece exactly: the record itself
        x.P[0] = wr.c.x;
        x.P[1] = wr.c.y;
        x.P[2] = wr.c.z;
        x.a = wr.c.w;
        x.lgT = -wr.tau;
        return;
    }
    if (m.nop > 0) {
        // opaque records: the mean of their colours
        const float inv = 1.f / (float)m.nop;
        x.a = 1.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) x.P[q] = __fmul_rn(value(m.OC[q]), inv);
        x.lgT = -INFINITY;
        return;
    }
    const float M = m.nact > 0 ? value(m.M) : 0.f;
    if (M > 0.f) {
        // emission-absorption mixture (Eq. 2 when one record covers the piece in part)
        x.lgT = -__fmul_rn(M, __fsub_rn(t1, t));
        x.a = __fsub_rn(1.f, ex2_approx(x.lgT));
        const float s = __fmul_rn(x.a, rcp_approx(M));
#pragma unroll
        for (int q = 0; q < 3; ++q) x.P[q] = __fmul_rn(value(m.MC[q]), s);
    } else {
        // a gap, or only fully transparent records
        x.P[0] = x.P[1] = x.P[2] = 0.f;
        x.a = 0.f;
        x.lgT = 0.f;
    }
}

// Direct sweeps: the sums plus the record started last (for the whole-record case).
struct Mix {
    MixSums s;
    float lt_f, lt_b;  // bounds of the record started last
    RecC lt_c;         // and its colour, opacity and optical depth
};

__device__ __forceinline__ void mix_reset(Mix& m) {
    sums_reset(m.s);
    m.lt_f = m.lt_b = -1.f;
    m.lt_c.c = make_float4(0.f, 0.f, 0.f, 0.f);
    m.lt_c.tau = 0.f;
}

__device__ __forceinline__ void mix_piece(const Mix& m, float t, float t1, Piece& x) {
    piece_from(m.s, m.s.nact == 1 && m.lt_f == t && m.lt_b == t1, m.lt_c, t, t1, x);
}

__device__ __forceinline__ void mix_start(Mix& m, const RecC& c, float f, float b) {
    sums_update<true>(m.s, contrib(c, f, b));
    m.lt_f = f;
    m.lt_b = b;
    m.lt_c = c;
}

__device__ __forceinline__ void mix_end(Mix& m, const RecC& c, float f, float b) {
    sums_update<false>(m.s, contrib(c, f, b));
}

constexpr float kNoEvent = 3.0e38f;

// list words 2 and 3: pieces taken from the pool (64 bits: what the lists ask for may exceed any pool)
__device__ __forceinline__ unsigned long long* pool_used(uint32_t* list) {
    return reinterpret_cast<unsigned long long*>(list + 2);
}

// Takes `need` slots of a pool of `cap`, if it has them.  One that plainly does not fit takes nothing, so that smaller
// ones still do; one that others overtake at the pool's end is lost.  (Taking nothing in that case either, by compare
// and swap, costs a retry for every taker in between: the build of 640 x 480 pixels, K = 9, N_S = 4 took 2.5 times as
// long.)
__device__ __forceinline__ bool pool_take(unsigned long long* used, uint32_t need, uint32_t cap, uint32_t& at) {
    if (*reinterpret_cast<volatile unsigned long long*>(used) + need > cap) return false;
    const unsigned long long first = atomicAdd(used, (unsigned long long)need);
    at = (uint32_t)first;
    return first + need <= cap;
}

// slots of a pixel's run of n pieces in the pool (the search reads four pieces at once)
__device__ __forceinline__ uint32_t run_slots(uint32_t n) { return (n + 3u) & ~3u; }

// Heads in registers (K <= KMAX, fully unrolled; KMAX <= 8).
template <int KMAX>
struct RegHeads {
    uint64_t cur[KMAX];
    uint32_t rem[KMAX];
    float hf[KMAX], hb[KMAX];
};

// advance PE e's head to its next record with b > f (records with b <= f are ignored)
template <int KMAX, int PREC>
__device__ __forceinline__ void reg_next_valid(const PeIn* pe, RegHeads<KMAX>& h, int e) {
    while (h.rem[e] > 0) {
        float f, b;
        load_fb<PREC>(pe[e], h.cur[e], f, b);
        if (b > f) {
            h.hf[e] = f;
            h.hb[e] = b;
            return;
        }
        ++h.cur[e];
        --h.rem[e];
    }
}


struct ActiveRec {
    uint64_t cur;
    float f, b;
    int e;
};

// The piece [t, t1] covered by the n active records ar: the opaque records'
// colour sum if any is opaque, else the extinction sums (each in exact fixed
// point, as the running sums of the other sweeps).
template <int PREC>
__device__ __forceinline__ void mixture_piece(const PeIn* pe, const ActiveRec* ar, int n, float t, float t1,
                                              Piece& x) {
    MixSums m;
    sums_reset(m);
    m.nact = n;
    for (int i = 0; i < n; ++i) {
        if (rec_opaque(load_rec<PREC>(pe[ar[i].e], ar[i].cur))) ++m.nop;
    }
    if (m.nop > 0) {
        for (int i = 0; i < n; ++i) {
            const RecC r = load_rec<PREC>(pe[ar[i].e], ar[i].cur);
            if (rec_opaque(r)) {
                const float col[3] = {r.c.x, r.c.y, r.c.z};
#pragma unroll
                for (int q = 0; q < 3; ++q) u128_add(m.OC[q], to_fixed(fminf(fmaxf(col[q], 0.f), kMuMax)));
            }
        }
    } else {
        for (int i = 0; i < n; ++i) {
            const Contrib c = contrib(load_rec<PREC>(pe[ar[i].e], ar[i].cur), ar[i].f, ar[i].b);
            u128_add(m.M, c.M);
#pragma unroll
            for (int q = 0; q < 3; ++q) u128_add(m.MC[q], c.MC[q]);
        }
    }
    piece_from(m, false, RecC{make_float4(0.f, 0.f, 0.f, 0.f), 0.f}, t, t1, x);
}

// Calls visit(piece) for every piece of one pixel in depth order; returns the
// number of pieces.  The heads' bounds give each piece; the mixture sums of a
// piece covered by several records (or part of one) are summed from its
// active records (exactly, so the result equals the running sums of the other
// sweeps), which costs nothing for the common piece that is a whole record
// or a gap.
template <int KMAX, int PREC, typename V>
__device__ __forceinline__ int sweep_reg(const PeIn* pe, int k, const uint32_t* cnt0, const uint64_t* off0, V& visit) {
    RegHeads<KMAX> h;
    float t = kNoEvent;
#pragma unroll
    for (int e = 0; e < KMAX; ++e) {
        h.rem[e] = 0;
        if (e < k) {
            h.cur[e] = off0[e];
            h.rem[e] = cnt0[e];
            reg_next_valid<KMAX, PREC>(pe, h, e);
            if (h.rem[e] > 0) t = fminf(t, h.hf[e]);
        }
    }
    int npieces = 0;
    while (true) {
        float t1 = kNoEvent;
        int nact = 0, last = 0;
        unsigned act = 0u;
#pragma unroll
        for (int e = 0; e < KMAX; ++e) {
            if (e < k && h.rem[e] > 0) {
                if (h.hf[e] <= t) {
                    ++nact;
                    last = e;
                    act |= 1u << e;
                    t1 = fminf(t1, h.hb[e]);
                } else {
                    t1 = fminf(t1, h.hf[e]);
                }
            }
        }
        if (t1 >= kNoEvent) break;
        Piece x;
        if (nact == 0) {
            x.f = t;
            x.b = t1;
            x.P[0] = x.P[1] = x.P[2] = 0.f;
            x.a = 0.f;
            x.lgT = 0.f;
        } else {
            float lf = 0.f, lb = 0.f;
            uint64_t lc = 0;
#pragma unroll
            for (int e = 0; e < KMAX; ++e) {
                if (e == last) {
                    lf = h.hf[e];
                    lb = h.hb[e];
                    lc = h.cur[e];
                }
            }
            if (nact == 1 && lf == t && lb == t1) {
                MixSums m;
                sums_reset(m);
                piece_from(m, true, load_rec<PREC>(pe[last], lc), t, t1, x);
            } else {
                ActiveRec ar[KMAX];
                int na = 0;
#pragma unroll
                for (int e = 0; e < KMAX; ++e) {
                    if ((act >> e) & 1u) {
                        ar[na].cur = h.cur[e];
                        ar[na].f = h.hf[e];
                        ar[na].b = h.hb[e];
                        ar[na].e = e;
                        ++na;
                    }
                }
                mixture_piece<PREC>(pe, ar, na, t, t1, x);
            }
        }
        visit(x);
        ++npieces;
        // advance the heads that end at t1
#pragma unroll
        for (int e = 0; e < KMAX; ++e) {
            if (((act >> e) & 1u) && h.hb[e] <= t1) {
                ++h.cur[e];
                --h.rem[e];
                reg_next_valid<KMAX, PREC>(pe, h, e);
            }
        }
        t = t1;
    }
    return npieces;
}

// Heads in shared memory with a winner tree over P leaves (K <= P <= 64), one
// lane's arrays interleaved with its warp's other lanes (element i of lane l
// at word i * 32 + l), so that every access is free of bank conflicts.
template <int P>
struct SmemHeads {
    float* key;      // next event depth of each head (kNoEvent when exhausted)
    float* oth;      // the other bound of the head's record
    uint32_t* pos;   // record index within the PE's list; top bit: record active
    uint32_t* node;  // node[n], 1 <= n < P: winning head of the subtree n
    __device__ __forceinline__ float& K(int i) const { return key[i * 32]; }
    __device__ __forceinline__ float& O(int i) const { return oth[i * 32]; }
    __device__ __forceinline__ uint32_t& S(int i) const { return pos[i * 32]; }
    __device__ __forceinline__ uint32_t& N(int i) const { return node[i * 32]; }
};

constexpr uint32_t kActive = 0x80000000u;

// words of dynamic shared memory per thread for P leaves
template <int P>
constexpr int smem_words_per_thread() {
    return 4 * P;
}

template <int P>
__device__ __forceinline__ SmemHeads<P> smem_heads(uint32_t* smem) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* base = smem + (size_t)warp * (4 * P * 32) + lane;
    SmemHeads<P> h;
    h.key = reinterpret_cast<float*>(base);
    h.oth = reinterpret_cast<float*>(base + P * 32);
    h.pos = base + 2 * P * 32;
    h.node = base + 3 * P * 32;
    return h;
}

template <int P>
__device__ __forceinline__ int tree_winner_of(const SmemHeads<P>& h, int n) {
    return n >= P ? n - P : (int)h.N(n);
}

// recompute the winners on the path from leaf e to the root
template <int P>
__device__ __forceinline__ void tree_update(const SmemHeads<P>& h, int e) {
    int c = P + e;
    int w = e;
    float kw = h.K(e);
#pragma unroll
    for (int lev = 0; lev < 6; ++lev) {
        if ((P >> lev) <= 1) break;
        const int ws = tree_winner_of(h, c ^ 1);
        const float ks = h.K(ws);
        if (ks < kw || (ks == kw && ws < w)) {
            w = ws;
            kw = ks;
        }
        c >>= 1;
        h.N(c) = (uint32_t)w;
    }
}

template <int P>
__device__ __forceinline__ void tree_build(const SmemHeads<P>& h) {
    for (int n = P - 1; n >= 1; --n) {
        const int a = tree_winner_of(h, 2 * n), b = tree_winner_of(h, 2 * n + 1);
        const float ka = h.K(a), kb = h.K(b);
        h.N(n) = (uint32_t)((kb < ka || (kb == ka && b < a)) ? b : a);
    }
}

// move head e to its first record at or after index j with b > f
template <int P, int PREC>
__device__ __forceinline__ void smem_seek(const SmemHeads<P>& h, const PeIn& pe, uint32_t p, int e, uint32_t j) {
    const uint32_t cnt = __ldg(pe.counts + p);
    const uint64_t base = __ldg(pe.offsets + p);
    while (j < cnt) {
        float f, b;
        load_fb<PREC>(pe, base + j, f, b);
        if (b > f) {
            h.K(e) = f;
            h.O(e) = b;
            h.S(e) = j;
            return;
        }
        ++j;
    }
    h.K(e) = kNoEvent;
    h.S(e) = j;
}

template <int P, int PREC, typename V>
__device__ __forceinline__ int sweep_smem(const PeIn* pe, int k, uint32_t p, const SmemHeads<P>& h, V& visit) {
    for (int e = 0; e < P; ++e) {
        if (e < k) smem_seek<P, PREC>(h, pe[e], p, e, 0u);
        else h.K(e) = kNoEvent;
    }
    tree_build<P>(h);
    Mix m;
    mix_reset(m);
    int npieces = 0;
    float t = h.K(h.N(1));
    while (t < kNoEvent) {
        // events at depth t, in ascending PE order (the tree breaks ties by index)
        float t1;
        while (true) {
            const int e = (int)h.N(1);
            t1 = h.K(e);
            if (t1 != t) break;
            const uint32_t s = h.S(e);
            const uint32_t j = s & ~kActive;
            const RecC c = load_rec<PREC>(pe[e], __ldg(pe[e].offsets + p) + j);
            if (!(s & kActive)) {
                const float b = h.O(e);
                mix_start(m, c, t, b);
                h.K(e) = b;
                h.O(e) = t;
                h.S(e) = s | kActive;
            } else {
                mix_end(m, c, h.O(e), t);
                smem_seek<P, PREC>(h, pe[e], p, e, j + 1);
            }
            tree_update<P>(h, e);
        }
        if (t1 >= kNoEvent) break;
        Piece x;
        mix_piece(m, t, t1, x);
        visit(x);
        ++npieces;
        t = t1;
    }
    return npieces;
}

// Work census of the compositing kernels (VDI_FLAG_CENSUS).
struct CompCensus {
    unsigned long long pixels = 0, searched = 0, sweeps = 0, pieces = 0, cand_steps = 0, records = 0,
                       table_hits = 0;
};

// Counting state of one gamma candidate over pieces of arbitrary length.
struct CompCount {
    float P[3], A, L2, fS, bS;
    int cnt;
    bool open;
};

// Counting with decision intervals (see GenCountQ): qlo / qhi bound the
// gamma^2 for which every decision of the march repeats.
struct CompCountQ {
    float P[3], A, L2, fS, bS;
    float qlo, qhi;
    int cnt;
    bool open;
};

__device__ __forceinline__ void cq_step(CompCountQ& s, const Piece& x, float g2) {
    if (!s.open) {
        if (x.a > 0.f) {
            s.P[0] = x.P[0]; s.P[1] = x.P[1]; s.P[2] = x.P[2];
            s.A = x.a; s.L2 = x.lgT; s.fS = x.f; s.bS = x.b; s.open = true;
            ++s.cnt;
        }
        return;
    }
    float lx = __fsub_rn(x.b, x.f), lS = __fsub_rn(s.bS, s.fS);
    float r = (lx > 0.f && lS > 0.f) ? __fmul_rn(lx, rcp_approx(lS)) : 1.f;
    float q;
    if (criterion_q(s.P, s.A, s.L2, r, x.P, g2, q)) {
        s.qhi = fminf(s.qhi, q);
        if (x.a > 0.f) {
            s.P[0] = x.P[0]; s.P[1] = x.P[1]; s.P[2] = x.P[2];
            s.A = x.a; s.L2 = x.lgT; s.fS = x.f; s.bS = x.b;
            ++s.cnt;
        } else {
            s.open = false;
        }
    } else {
        s.qlo = fmaxf(s.qlo, q);
        absorb(s.P, s.A, s.L2, x.P, x.a, x.lgT);
        s.bS = x.b;
    }
}

template <int NC>
struct CountVisitorQ {
    CompCountQ st[NC];
    float g2[NC];
    int nt;
    __device__ __forceinline__ void reset() {
        nt = 0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            st[c].cnt = 0;
            st[c].open = false;
            st[c].qlo = -1.f;
            st[c].qhi = 3.0e38f;
        }
    }
    __device__ __forceinline__ void operator()(const Piece& x) {
        nt += x.a > 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) cq_step(st[c], x, g2[c]);
    }
};

struct EmitVisitor {
    CompCount s;
    float g2;
    int cap;
    float bt;
    int written;
    size_t base;  // first slot of the pixel
    const OutDev* out;

    // L2 = log2(1 - A), the record's optical depth (stored by the FP16 form)
    __device__ __forceinline__ void store(float f, float b, const float P[3], float A, float L2) {
        size_t idx = base + written;
        if (out->prec == VDI_PREC_F32) {
            reinterpret_cast<float4*>(out->rgba)[idx] = make_float4(P[0], P[1], P[2], A);
            out->fb[idx] = make_float2(f, b);
        } else {
            reinterpret_cast<uint4*>(out->rgba)[idx] = f16_pack(f, b, P[0], P[1], P[2], L2);
        }
        ++written;
    }

    __device__ __forceinline__ void operator()(const Piece& x) {
        if (!s.open) {
            if (x.a > 0.f) {
                s.P[0] = x.P[0]; s.P[1] = x.P[1]; s.P[2] = x.P[2];
                s.A = x.a; s.L2 = x.lgT; s.fS = x.f; s.bS = x.b; s.open = true;
                bt = x.b;
                ++s.cnt;
            }
            return;
        }
        float lx = __fsub_rn(x.b, x.f), lS = __fsub_rn(s.bS, s.fS);
        float r = (lx > 0.f && lS > 0.f) ? __fmul_rn(lx, rcp_approx(lS)) : 1.f;
        if (s.cnt < cap && criterion(s.P, s.A, s.L2, r, x.P, g2)) {
            if (written < cap) store(s.fS, bt, s.P, s.A, s.L2);
            if (x.a > 0.f) {
                s.P[0] = x.P[0]; s.P[1] = x.P[1]; s.P[2] = x.P[2];
                s.A = x.a; s.L2 = x.lgT; s.fS = x.f; s.bS = x.b;
                bt = x.b;
                ++s.cnt;
            } else {
                s.open = false;
            }
        } else {
            absorb(s.P, s.A, s.L2, x.P, x.a, x.lgT);
            s.bS = x.b;
            if (x.a > 0.f) bt = x.b;
        }
    }
};

// Midpoints of the complete bisection subtree of NLEV levels below [lo, hi]
// in heap order (node 1 = midpoint, node 2i / 2i+1 = its left / right child).
template <int NLEV>
__device__ __forceinline__ void tree_candidates(float lo, float hi, float g[(1 << NLEV) - 1]) {
    float L[(1 << NLEV)], H[(1 << NLEV)];
    L[1] = lo;
    H[1] = hi;
#pragma unroll
    for (int i = 1; i < (1 << NLEV); ++i) {
        float m = 0.5f * (L[i] + H[i]);
        g[i - 1] = m;
        if (2 * i + 1 < (1 << NLEV)) {
            L[2 * i] = L[i]; H[2 * i] = m;
            L[2 * i + 1] = m; H[2 * i + 1] = H[i];
        }
    }
}

// One pixel's sweeps: heads in registers (KMAX > 0, K <= KMAX) or in shared
// memory with P leaves (KMAX == 0, K <= P).
template <int KMAX, int P, int PREC>
struct Sweeper {
    const PeIn* pe;
    int k;
    uint32_t p;
    uint32_t cnt0[KMAX > 0 ? KMAX : 1];
    uint64_t off0[KMAX > 0 ? KMAX : 1];
    SmemHeads<P> sh;

    __device__ __forceinline__ void init(const PeIn* pe_, int k_, uint32_t p_, uint32_t* smem) {
        pe = pe_;
        k = k_;
        p = p_;
        if constexpr (KMAX > 0) {
#pragma unroll
            for (int e = 0; e < KMAX; ++e) {
                if (e < k) {
                    cnt0[e] = __ldg(pe[e].counts + p);
                    off0[e] = __ldg(pe[e].offsets + p);
                }
            }
        } else {
            sh = smem_heads<P>(smem);
        }
    }
    __device__ __forceinline__ unsigned long long records() const {
        unsigned long long n = 0;
        for (int e = 0; e < k; ++e) n += __ldg(pe[e].counts + p);
        return n;
    }
    template <typename V>
    __device__ __forceinline__ int run(V& v) {
        if constexpr (KMAX > 0) return sweep_reg<KMAX, PREC>(pe, k, cnt0, off0, v);
        else return sweep_smem<P, PREC>(pe, k, p, sh, v);
    }
};

// The whole per-pixel composite: search, emission, zero tail.
// The whole per-pixel composite over the pieces that sw.run(visit) produces:
// search, emission, zero tail.
template <int NLEV, bool CENSUS, typename SW>
__device__ __forceinline__ void composite_search_emit(SW& sw, const OutDev& out, int iters, unsigned int* status,
                                                      uint32_t p, CompCensus* cs) {
    constexpr int NC = (1 << NLEV) - 1;
    // search (sec. 2.4 applied to the pieces, sec. 5.2): sequential bisection;
    // a midpoint's count comes from the table of earlier marches when one of
    // their decision intervals holds it, else from a march over the NLEV-level
    // subtree below the current bracket.
    float gamma = 0.f;
    int count;
    {
        CountTable t;
        t.n = 0;
        CountVisitorQ<NC> v;
        float g[NC];
        v.reset();
        tree_candidates<NLEV>(0.f, 2.f, g);
#pragma unroll
        for (int q = 0; q < NC; ++q) v.g2[q] = __fmul_rn(g[q], g[q]);
        {
            const int np = sw.run(v);
            if (CENSUS) {
                cs->sweeps += 1;
                cs->pieces += (unsigned long long)np;
                cs->cand_steps += (unsigned long long)np * NC;
            }
        }
#pragma unroll
        for (int q = 0; q < NC; ++q) t.add(v.g2[q], v.st[q].qlo, v.st[q].qhi, v.st[q].cnt);
        if (v.nt <= out.n_s) {
            count = v.nt;
        } else {
            if (CENSUS) cs->searched += 1;
            float lo = 0.f, hi = 2.f;
            int cnt_hi = 1;  // the distance never reaches 2: one supersegment
            for (int it = 0; it < iters; ++it) {
                float mid = 0.5f * (lo + hi);
                int c = t.lookup(__fmul_rn(mid, mid));
                if (c < 0) {
                    tree_candidates<NLEV>(lo, hi, g);
                    v.reset();
#pragma unroll
                    for (int q = 0; q < NC; ++q) v.g2[q] = __fmul_rn(g[q], g[q]);
                    const int np = sw.run(v);
                    if (CENSUS) {
                        cs->sweeps += 1;
                        cs->pieces += (unsigned long long)np;
                        cs->cand_steps += (unsigned long long)np * NC;
                    }
#pragma unroll
                    for (int q = 0; q < NC; ++q) t.add(v.g2[q], v.st[q].qlo, v.st[q].qhi, v.st[q].cnt);
                    c = v.st[0].cnt;
                } else if (CENSUS) {
                    cs->table_hits += 1;
                }
                if (c <= out.n_s) {
                    hi = mid;
                    cnt_hi = c;
                    if (c == out.n_s) break;
                } else {
                    lo = mid;
                }
            }
            gamma = hi;
            count = cnt_hi;
        }
    }
    EmitVisitor em;
    em.s.cnt = 0;
    em.s.open = false;
    em.g2 = __fmul_rn(gamma, gamma);
    em.cap = out.n_s;
    em.bt = 0.f;
    em.written = 0;
    em.base = (size_t)p * out.n_s;
    em.out = &out;
    {
        const int np = sw.run(em);
        if (CENSUS) {
            cs->sweeps += 1;
            cs->pieces += (unsigned long long)np;
        }
    }
    if (em.s.open && em.written < out.n_s) em.store(em.s.fS, em.bt, em.s.P, em.s.A, em.s.L2);
    for (int j = em.written; j < out.n_s; ++j) {
        size_t idx = (size_t)p * out.n_s + j;
        if (out.prec == VDI_PREC_F32) {
            reinterpret_cast<float4*>(out.rgba)[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
            out.fb[idx] = make_float2(0.f, 0.f);
        } else {
            reinterpret_cast<uint4*>(out.rgba)[idx] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    out.counts[p] = (uint32_t)em.written;
    if (out.gamma) out.gamma[p] = gamma;
    if (em.written != count) atomicCAS(status, 0u, (unsigned)VDI_ERR_CUDA);
}

// Direct path: the pieces are swept from the K lists on every march.
template <int KMAX, int P, int NLEV, int PREC, bool CENSUS = false>
__device__ __forceinline__ void composite_pixel(const PeIn* pe, int k, const OutDev& out, int iters,
                                                unsigned int* status, uint32_t p, uint32_t* smem,
                                                CompCensus* cs = nullptr) {
    Sweeper<KMAX, P, PREC> sw;
    sw.init(pe, k, p, smem);
    if (CENSUS) {
        cs->pixels += 1;
        cs->records += sw.records();
    }
    composite_search_emit<NLEV, CENSUS>(sw, out, iters, status, p, cs);
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void census_flush(const CompCensus& cs, unsigned long long* ctr) {
    const unsigned long long v[7] = {cs.pixels, cs.searched, cs.sweeps, cs.pieces, cs.cand_steps, cs.records,
                                     cs.table_hits};
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const unsigned long long w = warp_sum(v[i]);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(ctr + i, w);
    }
}

template <int KMAX, int P, int NLEV, int PREC, bool CENSUS>
__global__ void __launch_bounds__(128, NLEV > 2 ? 2 : 3) composite_kernel(const __grid_constant__ CompArgs a) {
    extern __shared__ uint32_t smem[];
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    CompCensus cs;
    if (p < (uint32_t)a.npix)
        composite_pixel<KMAX, P, NLEV, PREC, CENSUS>(a.pe, a.k, a.out, a.iters, a.status, p, smem, &cs);
    if (CENSUS) census_flush(cs, reinterpret_cast<WsHeader*>(a.status)->counters);
}


// storage of the pieces of the pixels the lane and pooled staged paths search
struct PiecePool {
    float4* A;  // (P.rgb, a)
    float2* B;  // (b, log2(1 - a))
    uint32_t cap;
};

// list entry of a pixel for the flat search: pixel (top bit: composite it by the direct sweep), first
// piece in the pool (a multiple of 4: four pieces are read at once), packed numbers of pieces, of non-transparent
// pieces and of columns of its part of the pool (groups of four pieces lie that many groups apart), front of the
// first piece
struct FlatEntry {
    uint32_t p, base, n_nt;
    float f0;
};

// n and nt below 2048 (a stage of 1024 records has at most 2047 pieces, a lane's slab of 480 at most 959), 32 columns
__device__ __forceinline__ uint32_t pieces_of(uint32_t n_nt) { return n_nt & 0x7FFu; }
__device__ __forceinline__ uint32_t nontransparent_of(uint32_t n_nt) { return n_nt >> 11 & 0x7FFu; }
__device__ __forceinline__ uint32_t columns_of(uint32_t n_nt) { return (n_nt >> 22) + 1u; }
__device__ __forceinline__ uint32_t pack_pieces(uint32_t n, uint32_t nt, int ncol) {
    return n | nt << 11 | (uint32_t)(ncol - 1) << 22;
}

// Whether the packed search takes a piece as the direct sweep does, bit for bit.  It clears a closed supersegment by
// multiplying with 0 (which an infinity or a NaN outlives, and which turns -0 into +0), subtracts depths without a
// look at their order, and takes log2(1 - a) = -inf as -1e34 (which a length ratio below 2^-105 would undo).  So a
// pixel whose pieces are all of finite non-negative colours up to 2^64, opacities in [0, 1] and lengths from 2^-60 at
// depths within 2^40 is searched in the pool; any other is left to the direct sweep.
__device__ __forceinline__ bool packable(const Piece& x) {
    const uint32_t c = max(max(__float_as_uint(x.P[0]), __float_as_uint(x.P[1])), __float_as_uint(x.P[2]));
    return c <= __float_as_uint(0x1p64f) && __float_as_uint(x.a) <= __float_as_uint(1.f) && x.lgT <= 0.f &&
           x.f >= -0x1p40f && x.b <= 0x1p40f && __fsub_rn(x.b, x.f) >= 0x1p-60f &&
           __float_as_uint(x.f) != 0x80000000u;
}

// writes the zero tail, count and gamma of pixel p after an emission of `written` records
__device__ __forceinline__ void finish_pixel(const OutDev& out, uint32_t p, int written, float gamma) {
    for (int j = written; j < out.n_s; ++j) {
        const size_t idx = (size_t)p * out.n_s + j;
        if (out.prec == VDI_PREC_F32) {
            reinterpret_cast<float4*>(out.rgba)[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
            out.fb[idx] = make_float2(0.f, 0.f);
        } else {
            reinterpret_cast<uint4*>(out.rgba)[idx] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    out.counts[p] = (uint32_t)written;
    if (out.gamma) out.gamma[p] = gamma;
}

// ---------------------------------------------------------------------------
// Staged path
// ---------------------------------------------------------------------------
// A warp (or a CTA of four, for long lists) takes 32 consecutive pixels at a time and builds the pieces of each of
// them in turn, every thread on one pixel: they load the pixel's records from all K lists, drop those with b <= f,
// sort their bounds (each list's bounds are already in order, so a stable merge of the K runs: log2 K rounds in which
// every bound finds its place in its partner run by binary search; ties go to the lower PE) and obtain the active
// set's sums after every bound by an exact prefix scan of the records' terms.  The pieces go to the pixel's column of
// the pool, and the pixel to the list of the flat search (a later launch).  They are bit for bit those of the direct
// sweep, which takes the pixels that this path cannot (the file's header lists them).

// A pixel is built by one warp when its 32-pixel batch's lists are short, by a CTA of four when they are long: the
// steps are chains of dependent shared-memory reads, so what counts is the warps an SM holds.  A warp's stage of 1024
// records (20 KB, a 172 KB CTA of 8 warps) left 8 warps per SM, 17% of the issue slots used; four warps on such a
// stage (38 KB with the records' terms, five CTAs) make 20, and a stage of 288 records for each warp (46 KB a CTA,
// four CTAs) 16 without barriers.  The line lies where the two are equal: 131,072 pixels, K = 12, dense, of 144
// records one warp takes 4.53 ms and four 5.02, of 240 7.09 and 7.36, of 276 8.22 and 8.25, of 288 8.65 and 8.55.
// (A stage of 284 records lets a fifth CTA in: 4.51, 7.19, 8.17 ms.)
constexpr int kStageRMax = 1024;   // records per pixel held by the largest stage
constexpr int kStageRSmall = 288;  // records per pixel of a batch that single warps build
constexpr int kStageWarps = 4;     // warps per CTA, of either kind
constexpr uint64_t kPoolPiecesPerPixel = 2 * kStageRMax;  // pieces that a pixel may need

#ifndef VDI_BUILD_MIN_BLOCKS
#define VDI_BUILD_MIN_BLOCKS 5
#endif

struct ScanState;

template <int RMAX>
struct StageSmem {
    uint16_t pay[2][2 * RMAX];      // bounds: (valid record << 1) | is_back
    float2 rfb[RMAX];               // bounds of the valid records
    float4 term[RMAX];              // their terms (record_terms)
    uint32_t rloc[RMAX];            // (PE << 16) | index in the PE's list, of the valid records
    uint32_t pref[VDI_MAX_PE + 1];  // records before PE e
    uint32_t vpref[VDI_MAX_PE + 1]; // valid records before PE e
    uint64_t off[VDI_MAX_PE];       // start of PE e's list for the pixel
    uint32_t nv, nt;
};

// NW warps working on one pixel: their threads' rank, barrier and vote
template <int NW>
__device__ __forceinline__ int group_rank() {
    return NW == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
}
template <int NW>
__device__ __forceinline__ void group_sync() {
    if (NW == 1) __syncwarp();
    else __syncthreads();
}
template <int NW>
__device__ __forceinline__ bool group_any(bool v) {
    return NW == 1 ? __any_sync(0xffffffffu, v) : __syncthreads_or(v) != 0;
}

template <int RMAX>
__device__ __forceinline__ float bound_key(const StageSmem<RMAX>& S, uint32_t w) {
    return reinterpret_cast<const float*>(S.rfb)[w];  // w = 2 record + is_back
}

__device__ __forceinline__ uint32_t warp_incl_scan_u32(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += o;
    }
    return v;
}

__device__ __forceinline__ U128 shfl_up_u128(const U128& v, int d) {
    U128 r;
    r.hi = __shfl_up_sync(0xffffffffu, v.hi, d);
    r.lo = __shfl_up_sync(0xffffffffu, v.lo, d);
    return r;
}

// running state of the stage's scan
struct ScanState {
    MixSums s;
    uint32_t xr;   // xor of the active records' indices
    uint32_t nb;   // bounds followed by a larger one (pieces)
};

__device__ __forceinline__ void scan_reset(ScanState& a) {
    sums_reset(a.s);
    a.xr = 0u;
    a.nb = 0u;
}

// a + b (element-wise, modulo 2^128 for the sums)
template <bool OPQ>
__device__ __forceinline__ void scan_add(ScanState& a, const ScanState& b) {
    u128_add(a.s.M, b.s.M);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        u128_add(a.s.MC[q], b.s.MC[q]);
        if (OPQ) u128_add(a.s.OC[q], b.s.OC[q]);
    }
    a.s.nop += b.s.nop;
    a.s.nact += b.s.nact;
    a.xr ^= b.xr;
    a.nb += b.nb;
}

template <bool OPQ>
__device__ __forceinline__ ScanState shfl_up_state(const ScanState& v, int d) {
    ScanState r;
    r.s.M = shfl_up_u128(v.s.M, d);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        r.s.MC[q] = shfl_up_u128(v.s.MC[q], d);
        if (OPQ) r.s.OC[q] = shfl_up_u128(v.s.OC[q], d);
        else u128_zero(r.s.OC[q]);
    }
    r.s.nop = __shfl_up_sync(0xffffffffu, v.s.nop, d);
    r.s.nact = __shfl_up_sync(0xffffffffu, v.s.nact, d);
    r.xr = __shfl_up_sync(0xffffffffu, v.xr, d);
    r.nb = __shfl_up_sync(0xffffffffu, v.nb, d);
    return r;
}

// applies bound w, of the record with terms t, to the state
template <bool OPQ>
__device__ __forceinline__ void stage_apply(uint32_t w, const float4& t, ScanState& a) {
    const Contrib x = contrib_of<OPQ>(t);
    const int sign = 1 - 2 * (int)(w & 1u);
    const unsigned long long neg = (unsigned long long)((long long)sign >> 1);  // fronts add, backs subtract
    u128_add_signed(a.s.M, x.M, neg);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        u128_add_signed(a.s.MC[q], x.MC[q], neg);
        if (OPQ) u128_add_signed(a.s.OC[q], x.OC[q], neg);
    }
    if (OPQ) a.s.nop += sign * x.op;
    a.s.nact += sign;
    a.xr ^= w >> 1;
}

// Walks the sorted bounds [i0, i1) of the stage: visit(w, terms, key, next key, there is a next), each bound's values
// read a bound ahead of their use and its place in the order two ahead (the three reads depend on each other).
template <int RMAX, typename F>
__device__ __forceinline__ void stage_walk(const StageSmem<RMAX>& S, const uint16_t* srt, uint32_t E, uint32_t i0,
                                           uint32_t i1, F&& visit) {
    if (i0 >= i1) return;
    uint32_t w = srt[i0], w1 = srt[min(i0 + 1, E - 1)];
    float key = bound_key(S, w);
    float4 t = S.term[w >> 1];
    for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t w2 = srt[min(i + 2, E - 1)];
        const float key1 = bound_key(S, w1);
        const float4 t1 = S.term[w1 >> 1];
        visit(w, t, key, key1, i + 1 < E);
        w = w1;
        w1 = w2;
        key = key1;
        t = t1;
    }
}

// Where phase G writes a pixel's pieces: a column of its batch's part of the pool, rows of 4 pieces by `ncol`
// columns.  A lane of the search then reads whole sectors, and the lanes that search a batch's pixels together read
// neighbouring ones.  (One run per pixel, allocated as it was built, put the runs of a batch 60 MB apart: every lane
// of the search in pages of its own.)  A run of its own is a column of one (build_batch says when).
struct PoolColumn {
    uint32_t base;  // slot of the first piece
    int ncol;
    __device__ __forceinline__ size_t at(uint32_t row) const {
        return (size_t)base + (size_t)(row >> 2) * ncol * 4 + (row & 3);
    }
};

// Phase G after the merge: exact prefix scan of the records' terms over the
// sorted bounds (srt, E of them; nv valid records), in contiguous chunks per
// thread, and the pieces written to the column that place(number of pieces, column) gives.  tot: scratch for the
// warps' totals.  Returns false when it gives none or a piece is not packable.
template <int NW, int PREC, bool OPQ, int RMAX, typename PLACE>
__device__ __forceinline__ bool stage_scan(const PeIn* pe, StageSmem<RMAX>& S, ScanState* tot, const uint16_t* srt,
                                           uint32_t E, uint32_t nv, const PiecePool& pool, const PLACE& place,
                                           PoolColumn& out, int& npieces, int& nt, float& f0) {
    constexpr uint32_t T = 32 * NW;
    const int lane = threadIdx.x & 31, rank = group_rank<NW>();
    const uint32_t chunk = ((E + T - 1) / T) | 1u;  // (odd: the threads' reads of their chunks spread over the banks)
    const uint32_t i0 = min(E, rank * chunk), i1 = min(E, i0 + chunk);
    ScanState loc;
    scan_reset(loc);
    stage_walk(S, srt, E, i0, i1, [&](uint32_t w, const float4& t, float key, float next, bool more) {
        stage_apply<OPQ>(w, t, loc);
        if (more && key < next) ++loc.nb;
    });
    // exclusive prefix of the threads' totals
    ScanState inc = loc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const ScanState o = shfl_up_state<OPQ>(inc, d);
        if (lane >= d) {
            ScanState t = o;
            scan_add<OPQ>(t, inc);
            inc = t;
        }
    }
    ScanState st = shfl_up_state<OPQ>(inc, 1);
    if (lane == 0) scan_reset(st);
    uint32_t total_pieces;
    if constexpr (NW == 1) {
        total_pieces = __shfl_sync(0xffffffffu, inc.nb, 31);
    } else {
        if (lane == 31) tot[threadIdx.x >> 5] = inc;
        __syncthreads();
        total_pieces = 0;
        for (int w = NW - 1; w >= 0; --w) {
            total_pieces += tot[w].nb;
            if (w < (int)(threadIdx.x >> 5)) {
                ScanState t = tot[w];
                scan_add<OPQ>(t, st);
                st = t;
            }
        }
    }
    if (!place(total_pieces, out)) return false;
    // the pieces: after bound i the active set is that of [key_i, key_{i+1}]
    uint32_t my_nt = 0;  // non-transparent pieces; from bit 16 on: pieces that are not packable
    uint32_t row = st.nb;
    stage_walk(S, srt, E, i0, i1, [&](uint32_t w, const float4& term, float t, float t1, bool more) {
        stage_apply<OPQ>(w, term, st);
        if (!more || !(t < t1)) return;
        bool whole = false;
        RecC wc{make_float4(0.f, 0.f, 0.f, 0.f), 0.f};
        if (st.s.nact == 1) {
            const uint32_t c = min(st.xr, nv - 1);
            const float2 fb = S.rfb[c];
            if (fb.x == t && fb.y == t1) {
                const uint32_t l = S.rloc[c];
                const int e = (int)(l >> 16);
                wc = load_rec<PREC>(pe[e], S.off[e] + (l & 0xFFFFu));
                whole = true;
            }
        }
        Piece x;
        piece_from<true>(st.s, whole, wc, t, t1, x);
        const size_t at = out.at(row);
        pool.A[at] = make_float4(x.P[0], x.P[1], x.P[2], x.a);
        pool.B[at] = make_float2(x.b, x.lgT);
        my_nt += (x.a > 0.f ? 1u : 0u) + (packable(x) ? 0u : 1u << 16);
        ++row;
    });
    my_nt = __reduce_add_sync(0xffffffffu, my_nt);
    npieces = (int)total_pieces;
    f0 = bound_key(S, srt[0]);
    if constexpr (NW > 1) {
        if (lane == 0) atomicAdd(&S.nt, my_nt);
        __syncthreads();
        my_nt = S.nt;
    }
    nt = (int)(my_nt & 0xFFFFu);
    return my_nt < 1u << 16;
}

// Phase G for pixel p (at most RMAX records) by NW warps, its pieces to the column `out` of place.  Returns false when
// a list is out of depth order, a piece is not packable or place gives no column.
template <int NW, int PREC, int RMAX, typename PLACE>
__device__ __forceinline__ bool stage_pixel(const PeIn* pe, int k, uint32_t p, StageSmem<RMAX>& S, ScanState* tot,
                                            const PiecePool& pool, const PLACE& place, PoolColumn& out, int& npieces,
                                            int& nt, float& f0) {
    constexpr uint32_t T = 32 * NW;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = (uint32_t)group_rank<NW>();
    npieces = nt = 0;
    f0 = 0.f;
    // counts and list starts, prefix over PEs
    if (NW == 1 || threadIdx.x < 32) {
        uint32_t c0 = 0, c1 = 0;
        if (lane < k) {
            c0 = __ldg(pe[lane].counts + p);
            S.off[lane] = __ldg(pe[lane].offsets + p);
        }
        if (lane + 32 < k) {
            c1 = __ldg(pe[lane + 32].counts + p);
            S.off[lane + 32] = __ldg(pe[lane + 32].offsets + p);
        }
        const uint32_t x0 = warp_incl_scan_u32(c0);
        const uint32_t t0 = __shfl_sync(0xffffffffu, x0, 31);
        const uint32_t x1 = warp_incl_scan_u32(c1);
        S.pref[lane] = x0 - c0;
        S.pref[lane + 32] = t0 + x1 - c1;
        if (lane == 31) S.pref[VDI_MAX_PE] = t0 + x1;
        if (lane == 0) S.nt = 0;
    }
    group_sync<NW>();
    const uint32_t R = S.pref[VDI_MAX_PE];
    // every record's bounds, in list order
    bool opaque = false, empty = false;
    for (uint32_t r = rank; r < R; r += T) {
        int lo = 0, hi = k - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (S.pref[mid] <= r) lo = mid;
            else hi = mid - 1;
        }
        const uint32_t j = r - S.pref[lo];
        float f, b;
        load_fb<PREC>(pe[lo], S.off[lo] + j, f, b);
        S.rfb[r] = make_float2(f, b);
        S.rloc[r] = ((uint32_t)lo << 16) | j;
        if (b > f) {
            const RecC x = load_rec<PREC>(pe[lo], S.off[lo] + j);
            opaque |= rec_opaque(x);
            S.term[r] = record_terms(x, f, b);
        } else {
            empty = true;
        }
    }
    uint32_t nv = R;
    if (group_any<NW>(empty)) {
        // drop the records with b <= f: the others move forward, in order
        group_sync<NW>();
        if (NW == 1 || threadIdx.x < 32) {
            uint32_t n = 0;
            for (uint32_t r0 = 0; r0 < R; r0 += 32) {
                const uint32_t r = r0 + lane;
                const float2 fb = r < R ? S.rfb[r] : make_float2(0.f, 0.f);
                const uint32_t loc = r < R ? S.rloc[r] : 0u;
                const float4 term = r < R ? S.term[r] : make_float4(0.f, 0.f, 0.f, 0.f);
                const bool valid = fb.y > fb.x;
                const unsigned m = __ballot_sync(0xffffffffu, valid);
                __syncwarp();  // every lane has read its slot (a ballot orders no memory)
                if (valid) {
                    const uint32_t c = n + __popc(m & ((1u << lane) - 1u));
                    S.rfb[c] = fb;
                    S.rloc[c] = loc;
                    S.term[c] = term;
                }
                n += __popc(m);
                __syncwarp();
            }
            if (lane == 0) S.nv = n;
        }
        group_sync<NW>();
        nv = S.nv;
        // valid records before PE e: the first compacted record of a PE >= e
        for (int e = (int)rank; e <= k; e += (int)T) {
            uint32_t lo = 0, hi = nv;
            const uint32_t key = (uint32_t)e << 16;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (S.rloc[mid] < key) lo = mid + 1;
                else hi = mid;
            }
            S.vpref[e] = lo;
        }
    } else {
        for (int e = (int)rank; e <= k; e += (int)T) S.vpref[e] = e < k ? S.pref[e] : R;
    }
    group_sync<NW>();
    // each list must be in depth order (b of a record <= f of the next): else
    // the merge below would not be a permutation; such pixels go to the
    // direct path
    bool unsorted = false;
    for (uint32_t c = rank + 1; c < nv; c += T)
        unsorted |= (S.rloc[c] >> 16) == (S.rloc[c - 1] >> 16) && !(S.rfb[c].x >= S.rfb[c - 1].y);
    const uint32_t E = 2 * nv;
    for (uint32_t i = rank; i < E; i += T) S.pay[0][i] = (uint16_t)i;
    if (group_any<NW>(unsorted)) return false;
    opaque = group_any<NW>(opaque);
    group_sync<NW>();
    if (E == 0) return true;
    // stable merge of the PEs' runs of bounds: round r merges the groups of
    // 2^r PEs pairwise (merge path: every thread takes an equal share of the
    // output, finds where it starts in the two runs by binary search and
    // merges sequentially from there; ties go to the lower run)
    int src = 0;
    for (int r = 0; (1 << r) < k; ++r) {
        const uint16_t* in = S.pay[src];
        uint16_t* outp = S.pay[src ^ 1];
        const int span = 2 << r;
        const int ngroups = (k + span - 1) / span;
        const uint32_t per = ((E + T - 1) / T) | 1u;  // (odd, as stage_scan's)
        uint32_t o = min(E, rank * per);
        const uint32_t o_end = min(E, o + per);
        while (o < o_end) {
            // the merged group holding output o: the last one starting at or before o
            int qlo = 0, qhi = ngroups - 1;
            while (qlo < qhi) {
                const int mid = (qlo + qhi + 1) >> 1;
                if (2u * S.vpref[mid * span] <= o) qlo = mid;
                else qhi = mid - 1;
            }
            const int e0 = qlo * span, em = min(e0 + (span >> 1), k), e1 = min(e0 + span, k);
            const uint32_t a0 = 2u * S.vpref[e0], b0 = 2u * S.vpref[em], b1 = 2u * S.vpref[e1];
            const uint32_t la = b0 - a0, lb = b1 - b0, d = o - a0;
            uint32_t lo = d > lb ? d - lb : 0u, hi = min(d, la);
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (bound_key(S, in[a0 + mid]) <= bound_key(S, in[b0 + d - mid - 1])) lo = mid + 1;
                else hi = mid;
            }
            uint32_t i = lo, j = d - lo;
            float ka = i < la ? bound_key(S, in[a0 + i]) : 0.f;
            float kb = j < lb ? bound_key(S, in[b0 + j]) : 0.f;
            const uint32_t stop = min(o_end, b1);
            for (; o < stop; ++o) {
                if (i < la && (j >= lb || ka <= kb)) {
                    outp[o] = in[a0 + i];
                    ++i;
                    if (i < la) ka = bound_key(S, in[a0 + i]);
                } else {
                    outp[o] = in[b0 + j];
                    ++j;
                    if (j < lb) kb = bound_key(S, in[b0 + j]);
                }
            }
        }
        src ^= 1;
        group_sync<NW>();
    }
    const uint16_t* srt = S.pay[src];
    const bool ok = opaque ? stage_scan<NW, PREC, true>(pe, S, tot, srt, E, nv, pool, place, out, npieces, nt, f0)
                           : stage_scan<NW, PREC, false>(pe, S, tot, srt, E, nv, pool, place, out, npieces, nt, f0);
    group_sync<NW>();
    return ok;
}

// One batch of 32 pixels (from p0 on, at most p1) of a request: if its longest pixel is this kernel's (more than
// RMIN and at most RMAX records, or beyond every stage), takes columns of the pool for the batch (its longest pixel's
// bound for each) and builds the pixels one by one.  RUNS: the pool is not sized for the worst case but for
// `share` slots a pixel, and a batch whose columns would be longer takes a run for each pixel instead, of the slots
// that its pieces need; so does a batch that the pool has no columns for.  (One pixel of 960 records among 31 of 64
// took 32 columns of 1920, and most of the other batches went to the direct sweep: 256 x 256, K = 16, 62 ms, with
// runs 8.1.)  emit(pixel, entry) is called by the lane of
// warp 0 that has the pixel, for pixels with pieces and for those left to the direct sweep (the pixel's top bit);
// pixels without records are finished here.
struct BatchPixel {
    bool have;
    uint32_t p, base, n_nt;
    float f0;
};

template <int NW, int PREC, int RMIN, int RMAX, bool RUNS>
__device__ __forceinline__ bool build_batch(const PeIn* pe, int k, uint32_t p0, uint32_t p1, const OutDev& out,
                                            const PiecePool& pool, unsigned long long* used, uint32_t share,
                                            StageSmem<RMAX>& S, ScanState* tot, uint32_t* base_of_all,
                                            BatchPixel& mine) {
    const int lane = threadIdx.x & 31;
    const int ncol = (int)min(32u, p1 - p0);
    // (every warp of the group sums the counts for itself)
    uint32_t R = 0;
    if (lane < ncol)
        for (int e = 0; e < k; ++e) R += __ldg(pe[e].counts + p0 + lane);
    const uint32_t fit = R <= (uint32_t)kStageRMax ? R : 0u;
    const uint32_t longest = __reduce_max_sync(0xffffffffu, fit);
    if (longest > (uint32_t)RMAX || (RMIN > 0 && longest <= (uint32_t)RMIN)) return false;
    // slots for every thread of the group, kNoSlots where the pool has not that many
    constexpr uint32_t kNoSlots = 0xFFFFFFFFu;
    auto take = [&](uint32_t need) {
        uint32_t at = kNoSlots;
        if (group_rank<NW>() == 0 && !pool_take(used, need, pool.cap, at)) at = kNoSlots;
        if constexpr (NW == 1) {
            at = __shfl_sync(0xffffffffu, at, 0);
        } else {
            if (threadIdx.x == 0) *base_of_all = at;
            __syncthreads();
            at = *base_of_all;
        }
        return at;
    };
    uint32_t base = kNoSlots;
    if (longest > 0) {
        const uint32_t rows = run_slots(2 * longest - 1);
        if (!RUNS || rows <= share) base = take(rows * (uint32_t)ncol);
    }
    mine.have = false;
    for (int col = 0; col < ncol; ++col) {
        const uint32_t p = p0 + (uint32_t)col;
        const uint32_t n_rec = __shfl_sync(0xffffffffu, R, col);
        int n = 0, nt = 0;
        float f0 = 0.f;
        bool ok = n_rec <= (uint32_t)kStageRMax;
        PoolColumn at{0u, 1};
        auto place = [&](uint32_t n_pieces, PoolColumn& c) {
            if (!RUNS || base != kNoSlots) {
                c = PoolColumn{base + (uint32_t)col * 4u, ncol};
            } else {
                group_sync<NW>();  // the last run's first slot has been read
                c = PoolColumn{take(run_slots(n_pieces)), 1};
            }
            return RUNS ? c.base != kNoSlots : true;
        };
        if (ok && n_rec > 0)
            ok = (RUNS || base != kNoSlots) && stage_pixel<NW, PREC>(pe, k, p, S, tot, pool, place, at, n, nt, f0);
        if (lane == col) {
            if (!ok) {
                mine = BatchPixel{true, p | 0x80000000u, 0u, 0u, 0.f};
            } else if (n == 0) {
                if (NW == 1 || threadIdx.x < 32) finish_pixel(out, p, 0, 0.f);  // no record: an empty list
            } else {
                mine = BatchPixel{true, p, at.base, pack_pieces((uint32_t)n, (uint32_t)nt, at.ncol), f0};
            }
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// Lane-staged path (short lists: K <= kLaneKMax).  Two passes.
//
// Batch pass (composite_lane_kernel): a warp takes 32 consecutive pixels,
// reads their counts and offsets (coalesced over the pixels) and copies their
// records into its shared-memory slab with asynchronous copies (cp.async:
// every copy of a round is in flight before the warp waits once), PE by PE:
// the spans of consecutive pixels of one PE are consecutive in the PE's record
// array (the layout generation writes), so the copies are coalesced 16- and
// 8-byte runs; other layouts find each record's pixel by a binary search over
// the lanes.  A lane sweeps its pixel's K lists in the slab into pieces and
// counts the non-transparent ones: at most n_s means gamma = 0 (sec. 2.4: the
// count at gamma = 0 is within the budget), and a second sweep emits the
// pixel's records straight away.  A pixel that needs the gamma search gets
// its pieces written, once, to a pool in the workspace and is listed.
//
// Search pass (composite_flat_kernel, below): the listed pixels' searches and
// emissions over their pooled pieces, a lane per pixel, lanes taking new
// pixels as they finish.  Pixels whose records exceed the slab, or whose
// pieces do not fit the pool, are listed for the direct sweep
// (composite_marked_kernel).  The pieces are those of every other schedule,
// bit for bit, so is the result.
// ---------------------------------------------------------------------------
constexpr int kLaneKMax = 8;        // PEs the lane path handles (heads in registers)
constexpr int kLaneWarps = 4;       // warps per CTA
constexpr int kLaneRCap = 480;      // records per warp slab

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A warp's slab of CAP records: F32 as rgba[] then fb[], F16 as the raw
// 16-byte records.
template <int PREC, int CAP>
struct LaneSlab;
template <int CAP>
struct LaneSlab<VDI_PREC_F32, CAP> {
    float4 rgba[CAP];
    float2 fb[CAP];
    __device__ __forceinline__ float2 bounds(uint32_t i) const { return fb[i]; }
    __device__ __forceinline__ RecC rec(uint32_t i) const {
        RecC r;
        r.c = rgba[i];
        r.tau = -lg2_approx(__fsub_rn(1.f, r.c.w));
        return r;
    }
    __device__ __forceinline__ void copy(const PeIn& pe, uint64_t src, uint32_t dst) {
        cp_async16(rgba + dst, reinterpret_cast<const float4*>(pe.rgba) + src);
        cp_async8(fb + dst, pe.fb + src);
    }
};
template <int CAP>
struct LaneSlab<VDI_PREC_F16, CAP> {
    uint4 raw[CAP];
    __device__ __forceinline__ float2 bounds(uint32_t i) const {
        return make_float2(__uint_as_float(raw[i].x), __uint_as_float(raw[i].y));
    }
    __device__ __forceinline__ RecC rec(uint32_t i) const {
        RecC r;
        f16_unpack_col(make_uint2(raw[i].z, raw[i].w), r.c, r.tau);
        return r;
    }
    __device__ __forceinline__ void copy(const PeIn& pe, uint64_t src, uint32_t dst) {
        cp_async16(raw + dst, reinterpret_cast<const uint4*>(pe.rgba) + src);
    }
};

// moves a head to its next record with b > f (records with b <= f are ignored)
template <class SLAB>
__device__ __forceinline__ void slab_next_valid(const SLAB& S, uint32_t& cur, uint32_t& rem, float& hf, float& hb) {
    while (rem > 0) {
        const float2 fb = S.bounds(cur);
        if (fb.y > fb.x) {
            hf = fb.x;
            hb = fb.y;
            return;
        }
        ++cur;
        --rem;
    }
}

// The pieces of one pixel from its K lists in the slab (list e: slab entries
// [st[e], st[e] + cnt[e])), in depth order: the sweep of sweep_reg with the
// records read from shared memory.
template <class SLAB, typename V>
__device__ __forceinline__ int sweep_slab(const SLAB& S, int k, const uint32_t st[kLaneKMax],
                                          const uint32_t cnt[kLaneKMax], V& visit) {
    uint32_t cur[kLaneKMax], rem[kLaneKMax];
    float hf[kLaneKMax], hb[kLaneKMax];
    float t = kNoEvent;
#pragma unroll
    for (int e = 0; e < kLaneKMax; ++e) {
        rem[e] = 0;
        hf[e] = hb[e] = 0.f;
        cur[e] = 0;
        if (e < k) {
            cur[e] = st[e];
            rem[e] = cnt[e];
            slab_next_valid(S, cur[e], rem[e], hf[e], hb[e]);
            if (rem[e] > 0) t = fminf(t, hf[e]);
        }
    }
    int npieces = 0;
    while (true) {
        float t1 = kNoEvent;
        int nact = 0, last = 0;
        unsigned act = 0u;
#pragma unroll
        for (int e = 0; e < kLaneKMax; ++e) {
            if (e < k && rem[e] > 0) {
                if (hf[e] <= t) {
                    ++nact;
                    last = e;
                    act |= 1u << e;
                    t1 = fminf(t1, hb[e]);
                } else {
                    t1 = fminf(t1, hf[e]);
                }
            }
        }
        if (t1 >= kNoEvent) break;
        Piece x;
        if (nact == 0) {
            x.f = t;
            x.b = t1;
            x.P[0] = x.P[1] = x.P[2] = 0.f;
            x.a = 0.f;
            x.lgT = 0.f;
        } else {
            float lf = 0.f, lb = 0.f;
            uint32_t lc = 0;
#pragma unroll
            for (int e = 0; e < kLaneKMax; ++e) {
                if (e == last) {
                    lf = hf[e];
                    lb = hb[e];
                    lc = cur[e];
                }
            }
            MixSums m;
            sums_reset(m);
            if (nact == 1 && lf == t && lb == t1) {
                piece_from(m, true, S.rec(lc), t, t1, x);
            } else {
                // the active records' mixture, summed exactly (as mixture_piece)
                m.nact = nact;
#pragma unroll
                for (int e = 0; e < kLaneKMax; ++e)
                    if ((act >> e) & 1u) m.nop += rec_opaque(S.rec(cur[e])) ? 1 : 0;
                if (m.nop > 0) {
#pragma unroll
                    for (int e = 0; e < kLaneKMax; ++e) {
                        if ((act >> e) & 1u) {
                            const RecC r = S.rec(cur[e]);
                            if (rec_opaque(r)) {
                                const float col[3] = {r.c.x, r.c.y, r.c.z};
#pragma unroll
                                for (int q = 0; q < 3; ++q)
                                    u128_add(m.OC[q], to_fixed(fminf(fmaxf(col[q], 0.f), kMuMax)));
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < kLaneKMax; ++e) {
                        if ((act >> e) & 1u) {
                            const Contrib c = contrib(S.rec(cur[e]), hf[e], hb[e]);
                            u128_add(m.M, c.M);
#pragma unroll
                            for (int q = 0; q < 3; ++q) u128_add(m.MC[q], c.MC[q]);
                        }
                    }
                }
                piece_from(m, false, RecC{make_float4(0.f, 0.f, 0.f, 0.f), 0.f}, t, t1, x);
            }
        }
        visit(x);
        ++npieces;
#pragma unroll
        for (int e = 0; e < kLaneKMax; ++e) {
            if (((act >> e) & 1u) && hb[e] <= t1) {
                ++cur[e];
                --rem[e];
                slab_next_valid(S, cur[e], rem[e], hf[e], hb[e]);
            }
        }
        t = t1;
    }
    return npieces;
}

// One pixel's sweeps over the slab.  When the pixel's K lists are disjoint
// in depth -- each list sorted with
// non-overlapping records, and the PEs' depth ranges not overlapping (every
// convex decomposition gives such lists: a ray crosses each box in one
// stretch) -- no interval is covered by two records, so the pieces are the
// records themselves, in the order of the PEs' ranges, with a transparent gap
// piece wherever one record ends before the next begins: exactly the pieces
// the sweep would cut, without comparing K list heads per piece.  Other
// pixels take the sweep.
template <class SLAB>
struct SlabSweeper {
    const SLAB* S;
    int k;
    uint32_t st[kLaneKMax], cnt[kLaneKMax];
    bool sorted;     // every list's records in depth order
    bool disjoint;
    uint32_t order;  // PEs by the front of their first record, 4 bits each
    int nonempty;    // PEs with a record of positive length
    int nvalid;      // records of positive length
    int nto;         // of them, those of positive opacity (the non-transparent pieces, if disjoint)

    __device__ __forceinline__ void prepare() {
        float lo[kLaneKMax], hi[kLaneKMax];
        bool ok = true;
        int nz = 0;
        nvalid = 0;
        nto = 0;
#pragma unroll
        for (int e = 0; e < kLaneKMax; ++e) {
            lo[e] = kNoEvent;
            hi[e] = -kNoEvent;
            if (e < k) {
                float prev = -kNoEvent;
                for (uint32_t r = st[e]; r < st[e] + cnt[e]; ++r) {
                    const float2 fb = S->bounds(r);
                    if (!(fb.y > fb.x)) continue;
                    ++nvalid;
                    nto += S->rec(r).c.w > 0.f;
                    ok = ok && fb.x >= prev;
                    prev = fb.y;
                    lo[e] = fminf(lo[e], fb.x);
                    hi[e] = fb.y;
                }
                nz += lo[e] < kNoEvent;
            }
        }
        sorted = ok;
        // insertion sort of the PEs by their first front (ties by index, as the sweep's heads)
        uint32_t ord = 0;
        int n = 0;
#pragma unroll
        for (int e = 0; e < kLaneKMax; ++e) {
            if (e < k && lo[e] < kNoEvent) {
                int pos = n;
                while (pos > 0) {
                    const int q = (int)((ord >> (4 * (pos - 1))) & 15u);
                    float lq = lo[0];
#pragma unroll
                    for (int w = 1; w < kLaneKMax; ++w)
                        if (w == q) lq = lo[w];
                    if (!(lq > lo[e])) break;
                    const uint32_t sh = 4u * (uint32_t)pos;
                    ord = (ord & ~(15u << sh)) | ((uint32_t)q << sh);
                    --pos;
                }
                const uint32_t sh = 4u * (uint32_t)pos;
                ord = (ord & ~(15u << sh)) | ((uint32_t)e << sh);
                ++n;
            }
        }
        // consecutive ranges must not overlap
        float end = -kNoEvent;
        for (int i = 0; i < n; ++i) {
            const int e = (int)((ord >> (4 * i)) & 15u);
            float le = lo[0], he = hi[0];
#pragma unroll
            for (int w = 1; w < kLaneKMax; ++w)
                if (w == e) {
                    le = lo[w];
                    he = hi[w];
                }
            ok = ok && le >= end;
            end = he;
        }
        disjoint = ok;
        order = ord;
        nonempty = n;
    }

    template <typename V>
    __device__ __forceinline__ int run(V& v) const {
        if (!disjoint) return sweep_slab(*S, k, st, cnt, v);
        const int n = nonempty;
        int np = 0;
        float t = 0.f;
        bool first = true;
        for (int i = 0; i < n; ++i) {
            const int e = (int)((order >> (4 * i)) & 15u);
            uint32_t s0 = st[0], c0 = cnt[0];
#pragma unroll
            for (int w = 1; w < kLaneKMax; ++w)
                if (w == e) {
                    s0 = st[w];
                    c0 = cnt[w];
                }
            for (uint32_t r = s0; r < s0 + c0; ++r) {
                const float2 fb = S->bounds(r);
                if (!(fb.y > fb.x)) continue;
                Piece x;
                if (!first && fb.x > t) {
                    x.f = t;
                    x.b = fb.x;
                    x.P[0] = x.P[1] = x.P[2] = 0.f;
                    x.a = 0.f;
                    x.lgT = 0.f;
                    v(x);
                    ++np;
                }
                MixSums m;
                sums_reset(m);
                piece_from(m, true, S->rec(r), fb.x, fb.y, x);
                v(x);
                ++np;
                t = fb.y;
                first = false;
            }
        }
        return np;
    }
};

struct NtVisitor {
    int nt;
    __device__ __forceinline__ void operator()(const Piece& x) { nt += x.a > 0.f; }
};

// One sweep of the batch pass for every lane, whichever way its pixel goes.  A pixel whose
// non-transparent pieces number at most N_S takes gamma = 0 (sec. 2.4), and then every
// non-transparent piece is one output record, itself: each one terminates the open supersegment
// (Eq. 1 with gamma = 0: the distance is >= 0, reading G2) and each transparent piece closes it,
// so EmitVisitor with gamma = 0 stores exactly these pieces' values.  A pixel that needs the search
// writes all its pieces to its pool run.
struct LaneSink {
    const OutDev* out;
    size_t base;  // first output slot of the pixel
    int written;
    bool emit;
    float4* A;  // the pixel's pool run
    float2* B;
    bool pool;
    bool odd;  // a piece written to the pool is not packable
    float f0;  // front of the first piece
    uint32_t np;
    __device__ __forceinline__ void operator()(const Piece& x) {
        if (np == 0) f0 = x.f;
        if (pool) {
            A[np] = make_float4(x.P[0], x.P[1], x.P[2], x.a);
            B[np] = make_float2(x.b, x.lgT);
            odd = odd || !packable(x);
        }
        if (emit && x.a > 0.f) {
            const size_t idx = base + written;
            if (out->prec == VDI_PREC_F32) {
                reinterpret_cast<float4*>(out->rgba)[idx] = make_float4(x.P[0], x.P[1], x.P[2], x.a);
                out->fb[idx] = make_float2(x.f, x.b);
            } else {
                reinterpret_cast<uint4*>(out->rgba)[idx] = f16_pack(x.f, x.b, x.P[0], x.P[1], x.P[2], x.lgT);
            }
            ++written;
        }
        ++np;
    }
};

// list: [0] entries, [1] next entry for the search pass, [2], [3] pieces taken from the pool,
// then FlatEntry entries from word 4
struct LaneArgs {
    unsigned int* counter;  // batch counter of the batch pass
    uint32_t* list;
    PiecePool pool;
};


// appends an entry for each lane with `flag` set (one atomic per warp)
__device__ __forceinline__ void list_push(uint32_t* list, bool flag, const FlatEntry& en) {
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(list, (uint32_t)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (flag) reinterpret_cast<FlatEntry*>(list + 4)[base + __popc(m & ((1u << lane) - 1u))] = en;
}

// Copies the records of the lanes with `take` set into the slab, PE-major,
// and sets st[e] to each lane's first slab entry of PE e.  The copies are
// asynchronous; the caller waits once for all of them.
template <class SLAB>
__device__ __forceinline__ void slab_stage(const PeIn* pe, int k, SLAB& S, bool take, const uint32_t cnt[kLaneKMax],
                                           const uint64_t off[kLaneKMax], uint32_t st[kLaneKMax]) {
    const int lane = threadIdx.x & 31;
    uint32_t base_e = 0;
#pragma unroll
    for (int e = 0; e < kLaneKMax; ++e) {
        st[e] = 0;
        if (e < k) {
            const uint32_t ce = take ? cnt[e] : 0u;
            const uint32_t ie = warp_incl_scan_u32(ce);
            const uint32_t pre = ie - ce;
            const uint32_t n_e = __shfl_sync(0xffffffffu, ie, 31);
            st[e] = base_e + pre;
            // PE e's spans of this round are one run of its record array iff every non-empty span starts
            // where the previous ones leave off
            const unsigned nz = __ballot_sync(0xffffffffu, ce > 0);
            if (nz) {
                const int f = __ffs(nz) - 1;
                const uint64_t o0 = __shfl_sync(0xffffffffu, off[e], f);
                const bool run = !__any_sync(0xffffffffu, ce > 0 && off[e] != o0 + pre);
                for (uint32_t r0 = 0; r0 < n_e; r0 += 32) {
                    const uint32_t r = r0 + (uint32_t)lane;
                    uint64_t src = o0 + r;
                    if (!run) {
                        // the lane whose span holds record r: the last with pre <= r
                        int lo = 0, hi = 31;
#pragma unroll
                        for (int it = 0; it < 5; ++it) {
                            const int mid = (lo + hi + 1) >> 1;
                            const uint32_t pm = __shfl_sync(0xffffffffu, pre, mid);
                            if (pm <= r) lo = mid;
                            else hi = mid - 1;
                        }
                        const uint64_t oq = __shfl_sync(0xffffffffu, off[e], lo);
                        const uint32_t pq = __shfl_sync(0xffffffffu, pre, lo);
                        src = oq + (r - pq);
                    }
                    if (r < n_e) S.copy(pe[e], src, base_e + r);
                }
            }
            base_e += n_e;
        }
    }
}

// the listed pixels marked for the direct sweep (records beyond a slab, pieces beyond the pool or not packable, lists
// out of depth order), list heads in registers (KMAX > 0) or in shared memory under a winner tree of P
// leaves (KMAX == 0)
template <int KMAX, int P, int PREC, bool CENSUS>
__global__ void __launch_bounds__(128) composite_marked_kernel(const __grid_constant__ CompArgs a,
                                                               const uint32_t* __restrict__ list) {
    extern __shared__ uint32_t smem[];
    const uint32_t n = *list;
    const FlatEntry* entries = reinterpret_cast<const FlatEntry*>(list + 4);
    CompCensus cs;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i - threadIdx.x < n; i += gridDim.x * blockDim.x) {
        const uint32_t v = i < n ? entries[i].p : 0u;
        if (v & 0x80000000u)
            composite_pixel<KMAX, P, 2, PREC, CENSUS>(a.pe, a.k, a.out, a.iters, a.status, v & 0x7FFFFFFFu, smem,
                                                      &cs);
    }
    if (CENSUS) census_flush(cs, reinterpret_cast<WsHeader*>(a.status)->counters);
}

template <int PREC, int CAP>
constexpr size_t lane_smem_bytes() {
    return kLaneWarps * sizeof(LaneSlab<PREC, CAP>);
}

// Four CTAs per SM, as many as their slabs (46 KB each) allow: the sweeps' serial chains want every warp, and a
// kernel of 136 registers kept three (320 x 240, FP16 records: K = 4, N_S = 12 dense 4.64 -> 3.30 ms with four,
// K = 2, N_S = 32 dense 5.76 -> 4.02).
template <int PREC, bool CENSUS>
__global__ void __launch_bounds__(kLaneWarps * 32, 4) composite_lane_kernel(const __grid_constant__ CompArgs a,
                                                                        const __grid_constant__ LaneArgs la) {
    using Slab = LaneSlab<PREC, kLaneRCap>;
    extern __shared__ __align__(16) unsigned char lane_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Slab& S = reinterpret_cast<Slab*>(lane_smem)[warp];
    const int k = a.k;
    const uint32_t nitems = ((uint32_t)a.npix + 31u) / 32u;
    CompCensus cs;
    while (true) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(la.counter, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= nitems) break;
        const uint32_t p = item * 32u + (uint32_t)lane;
        const bool valid = p < (uint32_t)a.npix;
        uint32_t cnt[kLaneKMax];
        uint64_t off[kLaneKMax];
        uint32_t tot = 0;
#pragma unroll
        for (int e = 0; e < kLaneKMax; ++e) {
            cnt[e] = 0;
            off[e] = 0;
            if (e < k && valid) {
                cnt[e] = __ldg(a.pe[e].counts + p);
                off[e] = __ldg(a.pe[e].offsets + p);
                tot += cnt[e];
            }
        }
        // records beyond the slab: the direct sweep composites the pixel
        const bool big = valid && tot > (uint32_t)kLaneRCap;
        list_push(la.list, big, FlatEntry{p | 0x80000000u, 0u, 0u, 0.f});
        bool pending = valid && !big;
        while (__any_sync(0xffffffffu, pending)) {
            // this round: the pending lanes, in order, whose records fit the slab together
            const uint32_t incl = warp_incl_scan_u32(pending ? tot : 0u);
            const bool take = pending && incl <= (uint32_t)kLaneRCap;
            pending = pending && !take;
            uint32_t st[kLaneKMax];
            slab_stage(a.pe, k, S, take, cnt, off, st);
            cp_async_wait_all();
            __syncwarp();
            SlabSweeper<Slab> sw;
            sw.S = &S;
            sw.k = k;
#pragma unroll
            for (int e = 0; e < kLaneKMax; ++e) {
                sw.st[e] = st[e];
                sw.cnt[e] = take ? cnt[e] : 0u;
            }
            sw.prepare();
            bool emit = false, search = false;
            uint32_t bound = 0;  // pieces the pixel's pool run must hold
            int nt = 0;
            if (take) {
                if (sw.disjoint) {
                    // the pieces are the valid records with a gap between some of them
                    nt = sw.nto;
                    bound = sw.nvalid > 0 ? 2u * (uint32_t)sw.nvalid - 1u : 0u;
                } else {
                    NtVisitor nv{0};
                    bound = (uint32_t)sw.run(nv);
                    nt = nv.nt;
                }
                emit = nt <= a.out.n_s;
                search = !emit;
            }
            // the searching lanes' pool runs (one atomic per warp).  Lists out of depth order are left to the direct
            // sweep: their sweep can step back, so a slab's records can give any number of pieces (an entry holds
            // 2047), of lengths that are not positive.
            const bool pooled = search && sw.sorted;
            unsigned long long base = 0;
            bool fits = false;
            if (__any_sync(0xffffffffu, pooled)) {
                const uint32_t mine = pooled ? run_slots(bound) : 0u;
                const uint32_t inc = warp_incl_scan_u32(mine);
                if (lane == 31) base = atomicAdd(pool_used(la.list), (unsigned long long)inc);
                base = __shfl_sync(0xffffffffu, base, 31) + inc - mine;
                fits = pooled && base + mine <= (unsigned long long)la.pool.cap;
                if (!fits) base = 0;
            }
            // one sweep: the gamma = 0 pixels' records, the searched pixels' pieces
            LaneSink snk{&a.out, (size_t)p * a.out.n_s, 0, emit, la.pool.A + base, la.pool.B + base, fits, false, 0.f, 0u};
            if (emit || fits) sw.run(snk);
            fits = fits && !snk.odd;
            if (emit) {
                if (snk.written != nt) atomicCAS(a.status, 0u, (unsigned)VDI_ERR_CUDA);
                finish_pixel(a.out, p, snk.written, 0.f);
                if (CENSUS) {
                    const unsigned sweeps = sw.disjoint ? 1u : 2u;
                    cs.pixels += 1;
                    cs.records += tot;
                    cs.sweeps += sweeps;
                    cs.pieces += (unsigned long long)sweeps * snk.np;
                }
            }
            if (__any_sync(0xffffffffu, search))
                list_push(la.list, search,
                          fits ? FlatEntry{p, (uint32_t)base, pack_pieces(snk.np, (uint32_t)nt, 1), snk.f0}
                               : FlatEntry{p | 0x80000000u, 0u, 0u, 0.f});
            __syncwarp();
        }
    }
    if (CENSUS) census_flush(cs, reinterpret_cast<WsHeader*>(a.status)->counters);
}

// ---------------------------------------------------------------------------
// Pooled staged path (K > kLaneKMax): two launches of composite_build_kernel
// (build_batch's warps and CTAs of four) build the pixels' pieces into their
// batches' columns of the pool and list the pixels; composite_flat_kernel then
// searches and emits every listed pixel, a lane each.  The host runs the pixels
// in chunks whose pieces fit the pool.
// ---------------------------------------------------------------------------
struct BuildArgs {
    unsigned int* counter;  // batch counter
    uint32_t* list;         // as LaneArgs::list
    PiecePool pool;
    uint32_t p0, p1;        // the chunk's pixels
};

// shared memory of a build CTA: four warps' stages, or one stage for four warps
template <int NW, int RMAX>
struct BuildShared {
    StageSmem<RMAX> stage[NW == 1 ? kStageWarps : 1];
    ScanState tot[NW == 1 ? 1 : NW];
    uint32_t base, item;
    __device__ BuildShared() {}
};

// the next item for a warp (NW = 1) or the CTA
template <int NW>
__device__ __forceinline__ uint32_t next_item(unsigned int* counter, uint32_t* share) {
    uint32_t item = 0;
    if (group_rank<NW>() == 0) item = atomicAdd(counter, 1u);
    if constexpr (NW == 1) return __shfl_sync(0xffffffffu, item, 0);
    __syncthreads();
    if (threadIdx.x == 0) *share = item;
    __syncthreads();
    return *share;
}

template <int NW, int PREC, bool CENSUS>
__global__ void __launch_bounds__(kStageWarps * 32, VDI_BUILD_MIN_BLOCKS) composite_build_kernel(const __grid_constant__ CompArgs a,
                                                                          const __grid_constant__ BuildArgs ba) {
    constexpr int RMAX = NW == 1 ? kStageRSmall : kStageRMax, RMIN = NW == 1 ? 0 : kStageRSmall;
    __shared__ BuildShared<NW, RMAX> sh;
    const uint32_t nbatch = (ba.p1 - ba.p0 + 31u) / 32u;
    CompCensus cs;
    while (true) {
        const uint32_t batch = next_item<NW>(ba.counter + (NW == 1 ? 0 : 1), &sh.item);
        if (batch >= nbatch) break;
        BatchPixel px;
        if (!build_batch<NW, PREC, RMIN, RMAX, false>(a.pe, a.k, ba.p0 + batch * 32u, ba.p1, a.out, ba.pool,
                                                      pool_used(ba.list), 0u, sh.stage[NW == 1 ? threadIdx.x >> 5 : 0],
                                                      sh.tot, &sh.base, px))
            continue;
        if (NW > 1 && threadIdx.x >= 32) continue;
        list_push(ba.list, px.have, FlatEntry{px.p, px.base, px.n_nt, px.f0});
        if (CENSUS) {
            const uint32_t p = ba.p0 + batch * 32u + (threadIdx.x & 31);
            cs.pixels += !px.have && p < ba.p1;
        }
    }
    if (CENSUS) census_flush(cs, reinterpret_cast<WsHeader*>(a.status)->counters);
}

// ---------------------------------------------------------------------------
// Flat search: the search and the emission of one pixel per lane, written as one
// loop whose body handles four pieces of the lane's current march.  Lanes at
// different marches, or at different pixels, execute the same loop body, so
// a warp's lanes stay busy however many marches their pixels need; a lane
// that finishes its pixel takes the next one from the list.  The decisions
// are those of composite_search_emit, step for step, and the bisection is
// replayed from the marches' counts (vdi_search.cuh), so the output is the
// same, bit for bit.  The pieces come from a pool in the workspace: a pixel's
// column of its batch's rows (the pooled builds), or a run of its own, which is
// a column of one (the lane path).
//
// What bounds it: instructions per piece (640 x 480, K = 32 dense: the search pass's two chunks of 131,072 pixels
// took 35 ms each with three candidates value by value and a load per piece; the whole call 171 -> 70 ms with the
// build's changes).  Four candidates run as two packed
// pairs in the form that takes the fewest operations:
//   - a closed S is P = A = L2 = 0, and the next non-transparent piece opens a new
//     one;
//   - opening is absorbing into the zeroed state (T = 1 - 0, fma(1, x, 0) = x):
//     the state is multiplied by 0 or 1 instead of selected value by value, and
//     a transparent piece that terminates S leaves the closed state;
//   - the pieces are contiguous, so S's back is the next piece's front;
//   - nA = -A saves the negations, products and sums keeping their bits;
//   - an opaque piece's log2(1 - a) = -inf becomes -1e34, whose products with a
//     length ratio give 2^x = 0 as well and which 0 clears.
// The rounded operations that decide are cq_step's, in its order; pixels with
// values for which one of these does not hold do not come here (packable).
// ---------------------------------------------------------------------------
#ifndef VDI_FLAT_END_BATCH
#define VDI_FLAT_END_BATCH 16
#endif
// resident CTAs of the flat pass per SM over the dense pieces of the pooled and batched paths: 4 and 5 measured alike
// (72.5 and 73.0 ms for the dense call), 6 spills (78.5)
#ifndef VDI_FLAT_CTAS_PER_SM
#define VDI_FLAT_CTAS_PER_SM 5
#endif

#ifndef VDI_FLAT_MIN_BLOCKS
#define VDI_FLAT_MIN_BLOCKS 5
#endif

struct FlatPair {
    f32x2 P[3], nA, L2, f, kept;  // kept: non-transparent pieces absorbed (the others each opened an S)
};

// the closed state before a first piece with front f0 (any front of S before f0 will do)
__device__ __forceinline__ void fp_reset(FlatPair& s, float f0) {
    s.P[0] = s.P[1] = s.P[2] = s.nA = s.L2 = s.kept = pk(0.f);
    s.f = pk(f0 - fmaxf(fabsf(f0), 1.f));
}

// A piece's values, each in both halves
struct PieceX {
    f32x2 P[3], na, lgT, f, lx, nt;
};

// where S goes on (1), or is closed or terminated by the piece (0); `last`: the first candidate's S is never terminated
__device__ __forceinline__ f32x2 fp_keep(const FlatPair& s, const PieceX& x, f32x2 g2, bool last) {
    float l0, l1, t0, t1, d0, d1, a0, a1;
    unpk(fma2(s.f, pk(-1.f), x.f), l0, l1);
    unpk(mul2(s.L2, mul2(x.lx, pk(rcp_approx(l0), rcp_approx(l1)))), t0, t1);
    const f32x2 at = fma2(pk(ex2_approx(t0), ex2_approx(t1)), pk(-1.f), pk(1.f));
    const f32x2 e0 = fma2(s.P[0], at, mul2(s.nA, x.P[0]));
    const f32x2 e1 = fma2(s.P[1], at, mul2(s.nA, x.P[1]));
    const f32x2 e2 = fma2(s.P[2], at, mul2(s.nA, x.P[2]));
    unpk(fma2(e2, e2, fma2(e1, e1, mul2(e0, e0))), d0, d1);
    unpk(mul2(g2, mul2(s.nA, s.nA)), t0, t1);
    unpk(s.nA, a0, a1);
    return pk(a0 == 0.f || (d0 >= t0 && !last) ? 0.f : 1.f, a1 == 0.f || d1 >= t1 ? 0.f : 1.f);
}

__device__ __forceinline__ void fp_apply(FlatPair& s, const PieceX& x, f32x2 k) {
    const f32x2 A = mul2(s.nA, k);
    const f32x2 T = add2(A, pk(1.f));
#pragma unroll
    for (int c = 0; c < 3; ++c) s.P[c] = fma2(T, x.P[c], mul2(s.P[c], k));
    s.nA = fma2(T, x.na, A);
    s.L2 = add2(mul2(s.L2, k), x.lgT);
    s.f = fma2(s.f, k, mul2(x.f, fma2(k, pk(-1.f), pk(1.f))));
    s.kept = fma2(k, x.nt, s.kept);
}

struct FlatLane {
    const OutDev* out;  // the pixel's output (its request's, in a batch)
    uint32_t p, base;
    int n, nt, ncol;
    float f0;
};

__device__ __forceinline__ void flat_store(const OutDev& out, uint32_t p, int written, float f, float b,
                                           const float P[3], float A, float L2) {
    const size_t idx = (size_t)p * out.n_s + written;
    if (out.prec == VDI_PREC_F32) {
        reinterpret_cast<float4*>(out.rgba)[idx] = make_float4(P[0], P[1], P[2], A);
        out.fb[idx] = make_float2(f, b);
    } else {
        reinterpret_cast<uint4*>(out.rgba)[idx] = f16_pack(f, b, P[0], P[1], P[2], L2);
    }
}

// the first candidate's open supersegment as a record that ends at bt
__device__ __forceinline__ void flat_record(const FlatLane& L, const FlatPair& s, int written, float bt) {
    float P[3], nA, L2, f, u;
#pragma unroll
    for (int c = 0; c < 3; ++c) unpk(s.P[c], P[c], u);
    unpk(s.nA, nA, u);
    unpk(s.L2, L2, u);
    unpk(s.f, f, u);
    flat_store(*L.out, L.p, written, f, bt, P, -nA, L2);
}

__device__ __forceinline__ bool flat_open(const FlatPair& s) {
    float nA, u;
    unpk(s.nA, nA, u);
    return nA != 0.f;
}

// Where the flat loop finds its pixels: the list's entries (one request) ...
struct FlatSrcOne {
    const FlatEntry* entries;
    const OutDev* out;
    const PeIn* pe;
    int k;
    __device__ __forceinline__ bool get(uint32_t i, FlatLane& L) const {
        const FlatEntry en = entries[i];
        if (en.p & 0x80000000u) return false;  // the direct sweep's
        L.p = en.p;
        L.base = en.base;
        L.n = (int)pieces_of(en.n_nt);
        L.nt = (int)nontransparent_of(en.n_nt);
        L.ncol = (int)columns_of(en.n_nt);
        L.f0 = en.f0;
        L.out = out;
        return true;
    }
    __device__ __forceinline__ unsigned long long records(uint32_t p) const {
        unsigned long long r = 0;
        for (int e = 0; e < k; ++e) r += __ldg(pe[e].counts + p);
        return r;
    }
};

// Shared memory of a flat CTA: the lanes' bisections, and their next pieces, two groups of four each, copied
// asynchronously while the groups before them are worked on: a lane's pieces come from L2 or DRAM once per march,
// and loads into registers left it waiting (25% of the issue slots used, against 8.7 stalls on a load per
// instruction).  Element i of lane l at i * 128 + l: 16-byte accesses without bank conflicts.
constexpr int kFlatThreads = 128;
struct FlatShared {
    float4 A[2 * 4][kFlatThreads];
    float4 B[2 * 2][kFlatThreads];  // (b, log2(1 - a)) of two pieces
    GammaSearch search[kFlatThreads];
};

// starts the copy of group q of the lane's run (an empty group at its end keeps the count of groups in flight)
__device__ __forceinline__ void flat_fetch(FlatShared& S, const PiecePool& pool, const FlatLane& L, int q) {
    if (q * 4 < L.n) {
        const size_t at = (size_t)L.base + (size_t)q * 4 * L.ncol;
        const float4* a = pool.A + at;
        const float4* b = reinterpret_cast<const float4*>(pool.B + at);
#pragma unroll
        for (int i = 0; i < 4; ++i) cp_async16(&S.A[(q & 1) * 4 + i][threadIdx.x], a + i);
#pragma unroll
        for (int i = 0; i < 2; ++i) cp_async16(&S.B[(q & 1) * 2 + i][threadIdx.x], b + i);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The search and emission of the listed pixels, a lane each (list: [count, next-entry counter, ...]
// then the entries SRC reads).
template <bool CENSUS, class SRC>
__device__ __forceinline__ void flat_loop(const SRC& src, const PiecePool& pool, uint32_t* list, int iters,
                                          unsigned int* status, FlatShared& S, CompCensus& cs) {
    GammaSearch& sh = S.search[threadIdx.x];
    const uint32_t n_list = list[0];
    const int lane = threadIdx.x & 31;
    FlatLane L;
    L.out = nullptr;
    L.p = L.base = 0;
    L.n = L.nt = L.ncol = 0;
    L.f0 = 0.f;
    FlatPair st[kCand / 2];
    f32x2 g2[kCand / 2];
    int j = 0, written = 0;
    float f = 0.f, bt = 0.f;
    bool has = false, emitting = false, exhausted = false, last = false;
#pragma unroll
    for (int w = 0; w < kCand / 2; ++w) {
        fp_reset(st[w], 0.f);
        g2[w] = 0ull;
    }
    while (true) {
        const unsigned act = __ballot_sync(0xffffffffu, has || !exhausted);
        if (!act) break;
        // a lane at the end of its march, or without a pixel, waits until VDI_FLAT_END_BATCH lanes (or all
        // active ones) are there: the divergent end of a march (the replay of bisection levels, the next
        // march's candidates, a new pixel) runs once for all of them instead of once per lane while the others idle
        const bool at_end = has ? j >= L.n : !exhausted;
        const unsigned pend = __ballot_sync(0xffffffffu, at_end);
        if (pend != 0u && (pend == act || __popc(pend) >= VDI_FLAT_END_BATCH)) {
            bool count = false, emit = false;  // the next march
            if (has && at_end) {
                if (CENSUS) {
                    cs.sweeps += 1;
                    cs.pieces += L.n;
                    if (!emitting) cs.cand_steps += (unsigned long long)L.n * kCand;
                }
                if (emitting) {
                    // the open supersegment, the zero tail, count and gamma
                    if (flat_open(st[0]) && written < L.out->n_s) {
                        flat_record(L, st[0], written, bt);
                        ++written;
                    }
                    finish_pixel(*L.out, L.p, written, sh.ghi);
                    if (written != sh.cnt_hi) atomicCAS(status, 0u, (unsigned)VDI_ERR_CUDA);
                    has = false;
                } else {
                    float k0, k1, k2, k3;
                    unpk(st[0].kept, k0, k1);
                    unpk(st[1].kept, k2, k3);
                    search_end_march(sh, L.nt - (int)k0, L.nt - (int)k1, L.nt - (int)k2, L.nt - (int)k3, L.out->n_s);
                    emit = sh.done != 0;
                    count = !emit;
                }
            }
            // lanes without a pixel take the next entries, one atomic per warp (in a list sorted by piece
            // count, the entries one fetch hands to a warp's lanes have nearly equal counts)
            const unsigned need = __ballot_sync(0xffffffffu, !has && !exhausted);
            if (need) {
                const int leader = __ffs(need) - 1;
                uint32_t first = 0;
                if (lane == leader) first = atomicAdd(list + 1, (uint32_t)__popc(need));
                first = __shfl_sync(0xffffffffu, first, leader);
                if ((need >> lane) & 1u) {
                    const uint32_t idx = first + (uint32_t)__popc(need & ((1u << lane) - 1u));
                    if (idx >= n_list) {
                        exhausted = true;
                    } else if (src.get(idx, L)) {  // (a marked entry leaves the lane idle: it takes another)
                        has = true;
                        if (CENSUS) {
                            cs.pixels += 1;
                            cs.records += src.records(L.p);
                        }
                        if (L.nt <= L.out->n_s) {  // gamma = 0 meets the budget
                            sh.ghi = 0.f;
                            sh.cnt_hi = L.nt;
                            emit = true;
                        } else {
                            if (CENSUS) cs.searched += 1;
                            search_start(sh, L.out->n_s, iters, L.nt);
                            count = true;
                        }
                    }
                }
            }
            if (count || emit) {
                emitting = emit;
                const float ge = __fmul_rn(sh.ghi, sh.ghi);
#pragma unroll
                for (int w = 0; w < kCand / 2; ++w) {
                    g2[w] = emit ? pk(ge) : pk(sh.g2[2 * w], sh.g2[2 * w + 1]);
                    fp_reset(st[w], L.f0);
                }
                j = 0;
                f = L.f0;
                written = 0;
                bt = 0.f;
                last = emit && L.out->n_s <= 1;
                flat_fetch(S, pool, L, 0);
                flat_fetch(S, pool, L, 1);
            }
            continue;
        }
        if (!has || at_end) continue;
        // four pieces of the lane's march
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        const int q = j >> 2, stop = min(L.n, j + 4);
#pragma unroll 1
        for (; j < stop; ++j) {
            const float4 A = S.A[j & 7][threadIdx.x];
            const float2 B = reinterpret_cast<const float2*>(&S.B[(j >> 1) & 3][threadIdx.x])[j & 1];
            const float b = B.x;
            const bool seen = A.w > 0.f;
            const PieceX x{{pk(A.x), pk(A.y), pk(A.z)},
                           pk(-A.w),
                           pk(fmaxf(B.y, -1e34f)),
                           pk(f),
                           pk(__fsub_rn(b, f)),
                           pk(seen ? 1.f : 0.f)};
            // one instruction stream for counting and emitting lanes: an emitting lane's first candidate carries
            // the budget and writes the supersegment a termination closes
            const f32x2 k = fp_keep(st[0], x, g2[0], last);
            if (emitting) {
                float k0, u1;
                unpk(k, k0, u1);
                if (k0 == 0.f && flat_open(st[0])) {
                    if (written < L.out->n_s) flat_record(L, st[0], written, bt);
                    ++written;
                    last = written + 1 >= L.out->n_s;
                }
                bt = seen ? b : bt;
            }
            fp_apply(st[0], x, k);
#pragma unroll
            for (int w = 1; w < kCand / 2; ++w) fp_apply(st[w], x, fp_keep(st[w], x, g2[w], false));
            f = b;
        }
        flat_fetch(S, pool, L, q + 2);
    }
}

template <bool CENSUS>
__global__ void __launch_bounds__(kFlatThreads, VDI_FLAT_MIN_BLOCKS) composite_flat_kernel(
    const __grid_constant__ CompArgs a, const __grid_constant__ PiecePool pool, uint32_t* list) {
    __shared__ FlatShared S;
    CompCensus cs;
    const FlatSrcOne src{reinterpret_cast<const FlatEntry*>(list + 4), &a.out, a.pe, a.k};
    flat_loop<CENSUS>(src, pool, list, a.iters, a.status, S, cs);
    if (CENSUS) census_flush(cs, reinterpret_cast<WsHeader*>(a.status)->counters);
}

// ---------------------------------------------------------------------------
// Order of the search pass: the listed pixels sorted by piece count, longest
// first (a counting sort into a second list with the same header).  A warp's
// lanes then take pixels of (nearly) equal piece counts, so their marches end
// together and no lane waits for the others at the end of a march; the
// longest pixels start first, so the last wave holds the shortest.  The order
// of pixels with equal counts is that of the atomics, which is free to vary:
// each pixel's result is independent of when it runs.  Marked pixels (the
// direct sweep's) stay out of the sorted list.
// ---------------------------------------------------------------------------
constexpr int kSortBins = 2048;

__device__ __forceinline__ uint32_t sort_bin(uint32_t n) {
    return (uint32_t)(kSortBins - 1) - (n < (uint32_t)(kSortBins - 1) ? n : (uint32_t)(kSortBins - 1));
}

// hist[b] += entries of bin b (hist zeroed by the caller)
template <class E, int HW>
__global__ void __launch_bounds__(256) list_hist_kernel(const uint32_t* __restrict__ list, uint32_t* hist) {
    __shared__ uint32_t h[kSortBins];
    for (int i = threadIdx.x; i < kSortBins; i += blockDim.x) h[i] = 0u;
    __syncthreads();
    const uint32_t n = list[0];
    const E* en = reinterpret_cast<const E*>(list + HW);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const E e = en[i];
        if (!(e.p & 0x80000000u)) atomicAdd(&h[sort_bin(pieces_of(e.n_nt))], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSortBins; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// hist -> exclusive offsets (in place); the sorted list's header: [0] entries, [1] next entry = 0
__global__ void __launch_bounds__(1024) list_offsets_kernel(uint32_t* hist, uint32_t* sorted) {
    __shared__ uint32_t wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kPer = kSortBins / 1024;
    uint32_t v[kPer], s = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        v[q] = hist[tid * kPer + q];
        s += v[q];
    }
    const uint32_t incl = warp_incl_scan_u32(s);
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = warp_incl_scan_u32(wsum[lane]);
        wsum[lane] = w;
    }
    __syncthreads();
    uint32_t ex = (warp > 0 ? wsum[warp - 1] : 0u) + incl - s;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        hist[tid * kPer + q] = ex;
        ex += v[q];
    }
    if (tid == 0) {
        sorted[0] = wsum[31];
        sorted[1] = 0u;
    }
}

// every unmarked entry to its bin's next slot (one atomic per bin and warp)
template <class E, int HW>
__global__ void __launch_bounds__(256) list_scatter_kernel(const uint32_t* __restrict__ list, uint32_t* pos,
                                                           uint32_t* sorted) {
    const uint32_t n = list[0];
    const E* en = reinterpret_cast<const E*>(list + HW);
    E* out = reinterpret_cast<E*>(sorted + HW);
    const int lane = threadIdx.x & 31;
    for (uint32_t i0 = blockIdx.x * blockDim.x; i0 < n; i0 += gridDim.x * blockDim.x) {
        const uint32_t i = i0 + threadIdx.x;
        E e{};
        bool take = false;
        if (i < n) {
            e = en[i];
            take = !(e.p & 0x80000000u);
        }
        const unsigned act = __ballot_sync(0xffffffffu, take);
        if (take) {
            const uint32_t b = sort_bin(pieces_of(e.n_nt));
            const unsigned grp = __match_any_sync(act, b);
            const int leader = __ffs(grp) - 1;
            uint32_t slot = 0;
            if (lane == leader) slot = atomicAdd(&pos[b], (uint32_t)__popc(grp));
            slot = __shfl_sync(grp, slot, leader) + (uint32_t)__popc(grp & ((1u << lane) - 1u));
            out[slot] = e;
        }
    }
}

static int device_sms();

// bytes of the sort's scratch: the histogram / offsets
constexpr size_t kSortScratch = kSortBins * sizeof(uint32_t);

// sorts list (HW header words, entries E) into sorted; hist: kSortScratch bytes
template <class E, int HW>
static cudaError_t launch_sort(const uint32_t* list, uint32_t* sorted, uint32_t* hist, uint64_t max_entries,
                               cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(hist, 0, kSortScratch, st);
    if (e != cudaSuccess) return e;
    uint64_t b = (max_entries + 255) / 256;
    const uint64_t cap = (uint64_t)device_sms() * 4u;
    if (b > cap) b = cap;
    if (b == 0) b = 1;
    list_hist_kernel<E, HW><<<(unsigned)b, 256, 0, st>>>(list, hist);
    list_offsets_kernel<<<1, 1024, 0, st>>>(hist, sorted);
    list_scatter_kernel<E, HW><<<(unsigned)b, 256, 0, st>>>(list, hist, sorted);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Batched persistent compositing
// ---------------------------------------------------------------------------
struct ReqDev {
    OutDev out;
    uint32_t npix;
    uint32_t item_begin;  // first 32-pixel batch of the request
    uint32_t pe_begin;    // index of its first PE descriptor
    int k, schedule;
};

struct BatchArgs {
    const ReqDev* reqs;
    const PeIn* pes;
    int n;
    uint32_t total_items;
    unsigned int* status;
    int iters;
};

__device__ __forceinline__ int request_of(const BatchArgs& a, uint32_t item) {
    int lo = 0, hi = a.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&a.reqs[mid].item_begin) <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Pooled batched path: composite_batched_build_kernel takes (request,
// 32-pixel batch) items of a chunk from an atomic counter and builds the
// pixels' pieces into the pool as composite_build_kernel does, into columns or
// into runs (build_batch; requests with a direct schedule, and pixels the stage cannot hold, are listed for the
// direct sweep); composite_batched_flat_kernel searches and emits the listed
// pixels, a lane each, each into its request's output; composite_batched_
// marked_kernel sweeps the pixels listed for the direct path.
struct BatchEntry {
    uint32_t p, base, n_nt;  // as FlatEntry's
    float f0;
    uint32_t req, pad0, pad1, pad2;
};

// Pieces that a request's pixel is expected to need: its K lists of at most N_S records cut into at most
// 2 K N_S - 1 pieces, rounded up to the groups of four that a run takes, at most the stage's.  (Lists may be longer:
// the table does not say by how much.)
__host__ __device__ static uint64_t batch_pixel_pieces(const ReqDev& r) {
    const uint64_t est = (2ull * (uint64_t)r.k * (uint64_t)(r.out.n_s > 0 ? r.out.n_s : 1) + 2) / 4 * 4;
    return est < kPoolPiecesPerPixel ? est : kPoolPiecesPerPixel;
}

struct BatchBuildArgs {
    unsigned int* counter;  // item counter
    uint32_t* list;         // [0] entries, [1] next entry of the flat pass, [2], [3] pool pieces taken; entries from word 8
    PiecePool pool;
    uint32_t item0, item1;  // the chunk's items
};

__device__ __forceinline__ void batch_push(uint32_t* list, bool flag, const BatchEntry& en) {
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(list, (uint32_t)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (flag) reinterpret_cast<BatchEntry*>(list + 8)[base + __popc(m & ((1u << lane) - 1u))] = en;
}

template <int NW, int PREC>
__global__ void __launch_bounds__(kStageWarps * 32, VDI_BUILD_MIN_BLOCKS) composite_batched_build_kernel(
    const __grid_constant__ BatchArgs a, const __grid_constant__ BatchBuildArgs bb) {
    constexpr int RMAX = NW == 1 ? kStageRSmall : kStageRMax, RMIN = NW == 1 ? 0 : kStageRSmall;
    __shared__ BuildShared<NW, RMAX> sh;
    while (true) {
        const uint32_t item = bb.item0 + next_item<NW>(bb.counter + (NW == 1 ? 0 : 1), &sh.item);
        if (item >= bb.item1) break;
        const int rq = request_of(a, item);
        const ReqDev& r = a.reqs[rq];
        const uint32_t base = (item - r.item_begin) * 32u;
        BatchPixel px;
        if (r.schedule == VDI_SCHED_STAGED) {
            if (!build_batch<NW, PREC, RMIN, RMAX, true>(a.pes + r.pe_begin, r.k, base, r.npix, r.out, bb.pool,
                                                         pool_used(bb.list), (uint32_t)batch_pixel_pieces(r),
                                                         sh.stage[NW == 1 ? threadIdx.x >> 5 : 0], sh.tot, &sh.base, px))
                continue;
            if (NW > 1 && threadIdx.x >= 32) continue;
        } else {
            if (NW > 1) continue;
            const uint32_t p = base + (threadIdx.x & 31);
            px = BatchPixel{p < r.npix, p | 0x80000000u, 0u, 0u, 0.f};
        }
        batch_push(bb.list, px.have, BatchEntry{px.p, px.base, px.n_nt, px.f0, (uint32_t)rq, 0u, 0u, 0u});
    }
}

struct FlatSrcBatch {
    const BatchEntry* entries;
    const ReqDev* reqs;
    __device__ __forceinline__ bool get(uint32_t i, FlatLane& L) const {
        const BatchEntry en = entries[i];
        if (en.p & 0x80000000u) return false;  // the direct sweep's
        L.p = en.p;
        L.base = en.base;
        L.n = (int)pieces_of(en.n_nt);
        L.nt = (int)nontransparent_of(en.n_nt);
        L.ncol = (int)columns_of(en.n_nt);
        L.f0 = en.f0;
        L.out = &reqs[en.req].out;
        return true;
    }
    __device__ __forceinline__ unsigned long long records(uint32_t) const { return 0; }
};

__global__ void __launch_bounds__(kFlatThreads, VDI_FLAT_MIN_BLOCKS) composite_batched_flat_kernel(
    const __grid_constant__ BatchArgs a, const __grid_constant__ PiecePool pool, uint32_t* list) {
    __shared__ FlatShared S;
    CompCensus cs;
    const FlatSrcBatch src{reinterpret_cast<const BatchEntry*>(list + 8), a.reqs};
    flat_loop<false>(src, pool, list, a.iters, a.status, S, cs);
}

template <int P, int PREC>
__global__ void __launch_bounds__(128) composite_batched_marked_kernel(const __grid_constant__ BatchArgs a,
                                                                       const uint32_t* __restrict__ list) {
    extern __shared__ uint32_t smem[];
    // a warp collects the marked entries among the others until it has one for every lane (where the pool runs out
    // within batches, a quarter of the entries are marked: 256 x 256, K = 16, lists 1.4 N_S long, 16.4 -> 11.3 ms)
    __shared__ uint32_t queue[4][64];
    uint32_t* q = queue[threadIdx.x >> 5];
    const uint32_t n = *list;
    const BatchEntry* entries = reinterpret_cast<const BatchEntry*>(list + 8);
    const uint32_t lane = threadIdx.x & 31, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    uint32_t queued = 0;
    for (uint32_t i0 = warp * 32; i0 < n || queued > 0; i0 += warps * 32) {
        const bool more = i0 < n, marked = more && i0 + lane < n && (entries[i0 + lane].p & 0x80000000u);
        const unsigned m = __ballot_sync(0xffffffffu, marked);
        if (marked) q[queued + __popc(m & ((1u << lane) - 1u))] = i0 + lane;
        queued += __popc(m);
        __syncwarp();
        if (more && queued < 32) continue;
        if (lane < queued) {
            const BatchEntry en = entries[q[lane]];
            const ReqDev& r = a.reqs[en.req];
            composite_pixel<0, P, 2, PREC>(a.pes + r.pe_begin, r.k, r.out, a.iters, a.status, en.p & 0x7FFFFFFFu,
                                           smem);
        }
        const uint32_t rest = queued > 32 ? queued - 32 : 0u;
        const uint32_t next = lane < rest ? q[32 + lane] : 0u;
        __syncwarp();
        if (lane < rest) q[lane] = next;
        queued = rest;
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
int default_schedule(int k) { return k <= kLaneKMax ? VDI_SCHED_LANE : VDI_SCHED_STAGED; }

static OutDev out_dev(const vdi_regular* out) {
    OutDev o;
    o.counts = out->counts;
    o.rgba = out->rgba;
    o.fb = reinterpret_cast<float2*>(out->fb);
    o.gamma = out->gamma;
    o.n_s = out->n_s;
    o.prec = out->prec;
    return o;
}

// leaves of the winner tree for K PEs
static int tree_leaves(int k) { return k <= 16 ? 16 : (k <= 32 ? 32 : 64); }

template <int P>
static size_t heads_smem_bytes(int threads) {
    return (size_t)threads * smem_words_per_thread<P>() * sizeof(uint32_t);
}

static int device_sms() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    return sms;
}

// CTAs of a build launch over `batches` 32-pixel batches
template <int NW, typename K>
static cudaError_t build_ctas(K kernel, uint64_t batches, unsigned& ctas) {
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kStageWarps * 32, 0);
    const uint64_t need = NW == 1 ? (batches + kStageWarps - 1) / kStageWarps : batches;
    const uint64_t most = (uint64_t)device_sms() * (uint64_t)(per_sm > 0 ? per_sm : 1);
    ctas = (unsigned)(need < most ? (need > 0 ? need : 1) : most);
    return e;
}

template <int NW, int PREC>
static cudaError_t launch_build(bool census, const CompArgs& a, const BuildArgs& ba, cudaStream_t st) {
    auto kb = census ? composite_build_kernel<NW, PREC, true> : composite_build_kernel<NW, PREC, false>;
    unsigned ctas = 0;
    cudaError_t e = build_ctas<NW>(kb, (ba.p1 - ba.p0 + 31) / 32, ctas);
    if (e != cudaSuccess) return e;
    kb<<<ctas, kStageWarps * 32, 0, st>>>(a, ba);
    return cudaGetLastError();
}

// pixels per chunk of the pooled staged path that the queried workspace holds at the stage's worst case
constexpr uint64_t kPoolChunkPixels = 131072;

size_t composite_workspace_bytes(int w, int h) {
    const uint64_t npix = (uint64_t)w * (uint64_t)h;
    const size_t piece = sizeof(float4) + sizeof(float2);
    // pooled staged path: a chunk of up to kPoolChunkPixels pixels, each with room for the stage's pieces
    const uint64_t chunk = npix < kPoolChunkPixels ? npix : kPoolChunkPixels;
    const size_t pooled = kWsHeader + 512 + (size_t)chunk * (sizeof(FlatEntry) + 2 * kStageRMax * piece);
    // lane path: the list of every pixel, its sorted copy and a pool of 16 pieces per pixel
    const size_t lane = kWsHeader + 256 + 2 * align_up(16 + npix * sizeof(FlatEntry), 256) + kSortScratch +
                        (size_t)npix * 16 * piece;
    return pooled > lane ? pooled : lane;
}


template <int KMAX, int P, int NLEV, int PREC>
static cudaError_t launch_cs(bool census, unsigned blocks, int threads, cudaStream_t st, const CompArgs& a) {
    const size_t sm = KMAX > 0 ? 0 : heads_smem_bytes<P>(threads);
    auto kern = census ? composite_kernel<KMAX, P, NLEV, PREC, true> : composite_kernel<KMAX, P, NLEV, PREC, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<blocks, threads, sm, st>>>(a);
    return cudaGetLastError();
}

template <int PREC>
static cudaError_t launch_sched(int schedule, int k, bool census, unsigned blocks, int threads, cudaStream_t st,
                                const CompArgs& a) {
    if (schedule == 1) return launch_cs<8, 16, 2, PREC>(census, blocks, threads, st, a);
    const int P = tree_leaves(k);
    if (schedule == 3) {
        if (P == 16) return launch_cs<0, 16, 3, PREC>(census, blocks, threads, st, a);
        if (P == 32) return launch_cs<0, 32, 3, PREC>(census, blocks, threads, st, a);
        return launch_cs<0, 64, 3, PREC>(census, blocks, threads, st, a);
    }
    if (P == 16) return launch_cs<0, 16, 2, PREC>(census, blocks, threads, st, a);
    if (P == 32) return launch_cs<0, 32, 2, PREC>(census, blocks, threads, st, a);
    return launch_cs<0, 64, 2, PREC>(census, blocks, threads, st, a);
}


template <int KMAX, int P, int PREC>
static cudaError_t launch_marked(bool census, const CompArgs& a, const uint32_t* list, uint64_t npix,
                                 cudaStream_t st) {
    const size_t sm = KMAX > 0 ? 0 : heads_smem_bytes<P>(128);
    auto kern = census ? composite_marked_kernel<KMAX, P, PREC, true> : composite_marked_kernel<KMAX, P, PREC, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    unsigned b = (unsigned)((npix + 127) / 128);
    const unsigned cap = (unsigned)device_sms() * 2u;
    if (b > cap) b = cap;
    kern<<<b, 128, sm, st>>>(a, list);
    return cudaGetLastError();
}

static cudaError_t launch_flat(bool census, const CompArgs& a, const PiecePool& pool, uint32_t* list, uint64_t lanes,
                               cudaStream_t st, int max_per_sm = 0) {
    auto k2 = census ? composite_flat_kernel<true> : composite_flat_kernel<false>;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k2, 128, 0);
    if (e != cudaSuccess) return e;
    if (max_per_sm > 0 && per_sm > max_per_sm) per_sm = max_per_sm;
    uint64_t b = (uint64_t)device_sms() * (uint64_t)(per_sm > 0 ? per_sm : 1);
    const uint64_t need = (lanes + 127) / 128;
    if (b > need) b = need > 0 ? need : 1;
    k2<<<(unsigned)b, 128, 0, st>>>(a, pool, list);
    return cudaGetLastError();
}

template <int PREC>
static cudaError_t launch_staged_pool(bool census, const CompArgs& a, void* workspace, size_t ws_bytes,
                                     cudaStream_t st) {
    // workspace: [header][counters][list: 4 words, entries of a chunk][pool: float4 x cap][pool: float2 x cap]
    // (the list stays in build order: dense pixels have equal piece counts, and a warp's lanes then read
    // neighbouring columns of a batch)
    const uint64_t npix = (uint64_t)a.npix;
    char* base = static_cast<char*>(workspace);
    // the chunk: as many pixels as the pool holds at the stage's worst case, all of them if they fit
    const size_t head = kWsHeader + 256;
    if (ws_bytes < head + 256) return cudaErrorInvalidValue;
    const size_t per_pixel = sizeof(FlatEntry) + kPoolPiecesPerPixel * (sizeof(float4) + sizeof(float2));
    uint64_t chunk = (ws_bytes - head - 256) / per_pixel;
    if (chunk > npix) chunk = npix;
    if (chunk == 0) return cudaErrorInvalidValue;
    const size_t list_bytes = align_up(16 + chunk * sizeof(FlatEntry), 256);
    size_t cap = (ws_bytes - head - list_bytes) / (sizeof(float4) + sizeof(float2));
    if (cap > 0x7FFFFFFFu) cap = 0x7FFFFFFFu;
    BuildArgs ba;
    ba.counter = reinterpret_cast<unsigned int*>(base + kWsHeader);
    ba.list = reinterpret_cast<uint32_t*>(base + head);
    ba.pool.cap = (uint32_t)cap;
    ba.pool.A = reinterpret_cast<float4*>(base + head + list_bytes);
    ba.pool.B = reinterpret_cast<float2*>(base + head + list_bytes + cap * sizeof(float4));
    cudaError_t e;
    const int P = tree_leaves(a.k);
    for (uint64_t p0 = 0; p0 < npix; p0 += chunk) {
        const uint64_t p1 = p0 + chunk < npix ? p0 + chunk : npix;
        ba.p0 = (uint32_t)p0;
        ba.p1 = (uint32_t)p1;
        e = cudaMemsetAsync(ba.counter, 0, 256, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(ba.list, 0, 16, st);
        if (e != cudaSuccess) return e;
        e = launch_build<1, PREC>(census, a, ba, st);
        if (e == cudaSuccess) e = launch_build<kStageWarps, PREC>(census, a, ba, st);
        if (e == cudaSuccess) e = launch_flat(census, a, ba.pool, ba.list, p1 - p0, st, VDI_FLAT_CTAS_PER_SM);
        if (e == cudaSuccess) {
            if (P == 16) e = launch_marked<0, 16, PREC>(census, a, ba.list, p1 - p0, st);
            else if (P == 32) e = launch_marked<0, 32, PREC>(census, a, ba.list, p1 - p0, st);
            else e = launch_marked<0, 64, PREC>(census, a, ba.list, p1 - p0, st);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int PREC>
static cudaError_t launch_lane(bool census, const CompArgs& a, void* workspace, size_t ws_bytes, cudaStream_t st) {
    // workspace: [header][counters][list: 4 words, npix entries][the list sorted][sort scratch]
    // [pool: float4 x cap][pool: float2 x cap]
    const uint64_t npix = (uint64_t)a.npix;
    const size_t list_bytes = align_up(16 + npix * sizeof(FlatEntry), 256);
    const size_t fixed = kWsHeader + 256 + 2 * list_bytes + kSortScratch;
    if (ws_bytes < fixed) return cudaErrorInvalidValue;
    char* base = static_cast<char*>(workspace);
    LaneArgs la;
    la.counter = reinterpret_cast<unsigned int*>(base + kWsHeader);
    la.list = reinterpret_cast<uint32_t*>(base + kWsHeader + 256);
    uint32_t* sorted = reinterpret_cast<uint32_t*>(base + kWsHeader + 256 + list_bytes);
    uint32_t* hist = reinterpret_cast<uint32_t*>(base + kWsHeader + 256 + 2 * list_bytes);
    size_t cap = (ws_bytes - fixed) / (sizeof(float4) + sizeof(float2));
    if (cap > 0x7FFFFFFFu) cap = 0x7FFFFFFFu;
    la.pool.cap = (uint32_t)cap;
    la.pool.A = reinterpret_cast<float4*>(base + fixed);
    la.pool.B = reinterpret_cast<float2*>(base + fixed + cap * sizeof(float4));
    cudaError_t e = cudaMemsetAsync(la.counter, 0, 256 + 16, st);
    if (e != cudaSuccess) return e;
    // batch pass
    const size_t sm = lane_smem_bytes<PREC, kLaneRCap>();
    auto k1 = census ? composite_lane_kernel<PREC, true> : composite_lane_kernel<PREC, false>;
    e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k1, kLaneWarps * 32, sm);
    if (e != cudaSuccess) return e;
    const uint64_t batches = (npix + 31) / 32;
    uint64_t blocks = (uint64_t)device_sms() * (uint64_t)(per_sm > 0 ? per_sm : 1);
    const uint64_t need = (batches + kLaneWarps - 1) / kLaneWarps;
    if (blocks > need) blocks = need > 0 ? need : 1;
    k1<<<(unsigned)blocks, kLaneWarps * 32, sm, st>>>(a, la);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // search pass over the list sorted by piece count: a persistent grid; the list's length is known
    // only on the device
    e = launch_sort<FlatEntry, 4>(la.list, sorted, hist, npix, st);
    if (e == cudaSuccess) e = launch_flat(census, a, la.pool, sorted, npix, st);
    if (e != cudaSuccess) return e;
    return launch_marked<kLaneKMax, 16, PREC>(census, a, la.list, npix, st);
}

vdi_status launch_composite(const vdi_compact* pe, int k, int w, int h, const vdi_regular* out, int iters,
                            int schedule, unsigned int* status, void* workspace, size_t ws_bytes, cudaStream_t st,
                            bool census) {
    CompArgs a;
    for (int e = 0; e < k; ++e) {
        a.pe[e].counts = pe[e].counts;
        a.pe[e].offsets = pe[e].offsets;
        a.pe[e].rgba = pe[e].rgba;
        a.pe[e].fb = reinterpret_cast<const float2*>(pe[e].fb);
    }
    a.k = k;
    a.npix = w * h;
    a.iters = iters;
    a.out = out_dev(out);
    a.status = status;
    const int prec_in = pe[0].prec;
    const bool automatic = schedule == 0;
    if (schedule == 0 || (schedule == 1 && k > 8)) schedule = default_schedule(k);
    // an automatic choice falls back to a direct schedule when the workspace holds no list or stage
    if (automatic && schedule == VDI_SCHED_LANE &&
        ws_bytes < kWsHeader + 256 + 2 * align_up(16 + (uint64_t)w * h * sizeof(FlatEntry), 256) + kSortScratch)
        schedule = 1;
    if (automatic && schedule == VDI_SCHED_STAGED && ws_bytes < composite_workspace_bytes(1, 1)) schedule = 2;
    if (a.npix == 0) return VDI_OK;
    const bool f32 = prec_in == VDI_PREC_F32;
    cudaError_t e;
    if (schedule == VDI_SCHED_LANE && k > kLaneKMax) schedule = VDI_SCHED_STAGED;
    if (schedule == VDI_SCHED_STAGED) {
        e = f32 ? launch_staged_pool<VDI_PREC_F32>(census, a, workspace, ws_bytes, st)
                : launch_staged_pool<VDI_PREC_F16>(census, a, workspace, ws_bytes, st);
    } else if (schedule == VDI_SCHED_LANE) {
        e = f32 ? launch_lane<VDI_PREC_F32>(census, a, workspace, ws_bytes, st)
                : launch_lane<VDI_PREC_F16>(census, a, workspace, ws_bytes, st);
    } else {
        const int threads = 128;
        const unsigned blocks = (unsigned)((a.npix + threads - 1) / threads);
        e = f32 ? launch_sched<VDI_PREC_F32>(schedule, k, census, blocks, threads, st, a)
                : launch_sched<VDI_PREC_F16>(schedule, k, census, blocks, threads, st, a);
    }
    return cuda_check(e, "composite launch");
}

// Device table: [BatchHeader][ReqDev x n][PeIn x sum k]
struct BatchHeader {
    uint32_t n, total_items, total_pes, prec_in;
    uint32_t max_k, pad;
    uint64_t total_pixels;
    uint64_t reqs_off, pes_off;
};

size_t batch_table_bytes(const vdi_request* reqs, int n) {
    size_t pes = 0;
    for (int r = 0; r < n; ++r) pes += (size_t)reqs[r].k;
    return align_up(sizeof(BatchHeader), 64) + align_up(sizeof(ReqDev) * (size_t)n, 64) + sizeof(PeIn) * pes;
}

vdi_status batch_table_pack(const vdi_request* reqs, int n, void* host_table, size_t bytes) {
    if (bytes < batch_table_bytes(reqs, n)) return set_error(VDI_ERR_INVALID_ARG, "batch table: buffer too small");
    char* base = static_cast<char*>(host_table);
    BatchHeader* hd = reinterpret_cast<BatchHeader*>(base);
    hd->reqs_off = align_up(sizeof(BatchHeader), 64);
    hd->pes_off = hd->reqs_off + align_up(sizeof(ReqDev) * (size_t)n, 64);
    ReqDev* rd = reinterpret_cast<ReqDev*>(base + hd->reqs_off);
    PeIn* pd = reinterpret_cast<PeIn*>(base + hd->pes_off);
    uint64_t items = 0, pes = 0, pixels = 0;
    uint32_t max_k = 0;
    for (int r = 0; r < n; ++r) {
        const vdi_request& q = reqs[r];
        rd[r].out = out_dev(&q.out);
        rd[r].npix = (uint32_t)((uint64_t)q.w * (uint64_t)q.h);
        rd[r].item_begin = (uint32_t)items;
        rd[r].pe_begin = (uint32_t)pes;
        rd[r].k = q.k;
        rd[r].schedule =
            q.schedule == VDI_SCHED_STAGED || q.schedule == VDI_SCHED_LANE || q.schedule == 0 ? VDI_SCHED_STAGED : 2;
        for (int e = 0; e < q.k; ++e) {
            pd[pes + e].counts = q.pe[e].counts;
            pd[pes + e].offsets = q.pe[e].offsets;
            pd[pes + e].rgba = q.pe[e].rgba;
            pd[pes + e].fb = reinterpret_cast<const float2*>(q.pe[e].fb);
        }
        pes += (uint64_t)q.k;
        pixels += rd[r].npix;
        items += ((uint64_t)rd[r].npix + 31) / 32;
        if ((uint32_t)q.k > max_k) max_k = (uint32_t)q.k;
    }
    if (items > 0xFFFFFFFFull) return set_error(VDI_ERR_INVALID_ARG, "batch table: too many work items");
    hd->n = (uint32_t)n;
    hd->total_items = (uint32_t)items;
    hd->total_pes = (uint32_t)pes;
    hd->prec_in = n > 0 ? (uint32_t)reqs[0].pe[0].prec : 0u;
    hd->max_k = max_k;
    hd->pad = 0;
    hd->total_pixels = pixels;
    return VDI_OK;
}

// Pooled batched path, its workspace: [header][counter][list: 8 words, kBatchListCap entries at most][pool]
constexpr uint64_t kBatchListCap = 1u << 22;
constexpr uint64_t kBatchPoolCap = 1u << 28;

static size_t batch_list_bytes(const BatchHeader* hd) {
    const uint64_t n = hd->total_pixels < kBatchListCap ? hd->total_pixels : kBatchListCap;
    return align_up(32 + n * sizeof(BatchEntry), 256);
}

size_t batched_workspace_bytes(const void* host_table) {
    const BatchHeader* hd = static_cast<const BatchHeader*>(host_table);
    const ReqDev* rd = reinterpret_cast<const ReqDev*>(static_cast<const char*>(host_table) + hd->reqs_off);
    uint64_t est = 0;
    for (uint32_t q = 0; q < hd->n; ++q) est += (uint64_t)rd[q].npix * batch_pixel_pieces(rd[q]);
    if (est > kBatchPoolCap) est = kBatchPoolCap;
    if (est < kPoolPiecesPerPixel * 32) est = kPoolPiecesPerPixel * 32;
    return kWsHeader + 256 + batch_list_bytes(hd) + (size_t)est * (sizeof(float4) + sizeof(float2));
}

template <int PREC>
static cudaError_t launch_batched(const BatchArgs& a, const BatchHeader* hd, const ReqDev* rd, void* workspace,
                                  size_t ws_bytes, cudaStream_t st) {
    // workspace: [header][counter][list][pool: float4 x cap][pool: float2 x cap] (the list in build order, as
    // the pooled path's)
    char* base = static_cast<char*>(workspace);
    const size_t fixed = kWsHeader + 256 + batch_list_bytes(hd);
    if (ws_bytes < fixed) return cudaErrorInvalidValue;
    uint64_t cap = (ws_bytes - fixed) / (sizeof(float4) + sizeof(float2));
    if (cap > 0x7FFFFFFFu) cap = 0x7FFFFFFFu;
    if (cap < kPoolPiecesPerPixel * 32) return cudaErrorInvalidValue;  // one item's worst case
    const uint64_t list_cap = hd->total_pixels < kBatchListCap ? hd->total_pixels : kBatchListCap;
    BatchBuildArgs bb;
    bb.counter = reinterpret_cast<unsigned int*>(base + kWsHeader);
    bb.list = reinterpret_cast<uint32_t*>(base + kWsHeader + 256);
    bb.pool.cap = (uint32_t)cap;
    bb.pool.A = reinterpret_cast<float4*>(base + fixed);
    bb.pool.B = reinterpret_cast<float2*>(base + fixed + cap * sizeof(float4));
    cudaError_t e;
    const int P = tree_leaves((int)hd->max_k);
    const size_t smd = P == 16 ? heads_smem_bytes<16>(128) : (P == 32 ? heads_smem_bytes<32>(128)
                                                                        : heads_smem_bytes<64>(128));
    auto km = P == 16 ? composite_batched_marked_kernel<16, PREC>
                      : (P == 32 ? composite_batched_marked_kernel<32, PREC> : composite_batched_marked_kernel<64, PREC>);
    e = cudaFuncSetAttribute(km, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smd);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, composite_batched_flat_kernel, 128, 0);
    if (e != cudaSuccess) return e;
    if (VDI_FLAT_CTAS_PER_SM > 0 && per_sm > VDI_FLAT_CTAS_PER_SM) per_sm = VDI_FLAT_CTAS_PER_SM;
    // chunks of whole items whose expected pieces fit the pool and whose pixels fit the list
    uint32_t item = 0;
    int q = 0;
    while (item < hd->total_items) {
        const uint32_t item0 = item;
        uint64_t pieces = 0, pixels = 0;
        while (item < hd->total_items) {
            while (q + 1 < (int)hd->n && rd[q + 1].item_begin <= item) ++q;
            const uint64_t px = 32;
            const uint64_t pc = px * batch_pixel_pieces(rd[q]);
            if (item > item0 && (pieces + pc > cap || pixels + px > list_cap)) break;
            pieces += pc;
            pixels += px;
            ++item;
        }
        BatchBuildArgs c = bb;
        c.item0 = item0;
        c.item1 = item;
        e = cudaMemsetAsync(bb.counter, 0, 256, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(bb.list, 0, 32, st);
        if (e != cudaSuccess) return e;
        unsigned ctas = 0;
        e = build_ctas<1>(composite_batched_build_kernel<1, PREC>, item - item0, ctas);
        if (e != cudaSuccess) return e;
        composite_batched_build_kernel<1, PREC><<<ctas, kStageWarps * 32, 0, st>>>(a, c);
        e = build_ctas<kStageWarps>(composite_batched_build_kernel<kStageWarps, PREC>, item - item0, ctas);
        if (e != cudaSuccess) return e;
        composite_batched_build_kernel<kStageWarps, PREC><<<ctas, kStageWarps * 32, 0, st>>>(a, c);
        uint64_t b = (uint64_t)device_sms() * (uint64_t)(per_sm > 0 ? per_sm : 1);
        const uint64_t need = (pixels + 127) / 128;
        if (b > need) b = need > 0 ? need : 1;
        composite_batched_flat_kernel<<<(unsigned)b, 128, 0, st>>>(a, bb.pool, bb.list);
        unsigned b3 = (unsigned)((pixels + 127) / 128);
        const unsigned cap3 = (unsigned)device_sms() * 2u;
        if (b3 > cap3) b3 = cap3;
        km<<<b3, 128, smd, st>>>(a, bb.list);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

vdi_status launch_composite_batched(const void* dev_table, const void* host_table, int iters, unsigned int* status,
                                    void* workspace, size_t ws_bytes, cudaStream_t st) {
    const BatchHeader* hd = static_cast<const BatchHeader*>(host_table);
    if (hd->n == 0 || hd->total_items == 0) return VDI_OK;
    BatchArgs a;
    a.reqs = reinterpret_cast<const ReqDev*>(static_cast<const char*>(dev_table) + hd->reqs_off);
    a.pes = reinterpret_cast<const PeIn*>(static_cast<const char*>(dev_table) + hd->pes_off);
    a.n = (int)hd->n;
    a.total_items = hd->total_items;
    a.status = status;
    a.iters = iters;
    const ReqDev* rd = reinterpret_cast<const ReqDev*>(static_cast<const char*>(host_table) + hd->reqs_off);
    const cudaError_t e = hd->prec_in == VDI_PREC_F32
                              ? launch_batched<VDI_PREC_F32>(a, hd, rd, workspace, ws_bytes, st)
                              : launch_batched<VDI_PREC_F16>(a, hd, rd, workspace, ws_bytes, st);
    return cuda_check(e, "composite_batched launch");
}

}  // namespace vdi
