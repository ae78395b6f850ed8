// The bisection search for gamma over a list of samples or pieces, as generation's and compositing's lanes run it:
// which gammas a march evaluates, and the replay of sequential bisection from their counts (sec. 2.4).
#pragma once

#include "vdi_device.cuh"

namespace vdi {

// A lane's bisection.  A march over the samples (pieces) evaluates four midpoints:
// the next one and the three that the bisection is most likely to visit after
// it.  The likelihood comes from where the count, taken as a power of gamma
// between the bracket's ends, crosses n_s (a logistic belief in log2 gamma about
// that point).  It only chooses what is evaluated: the bisection's own steps are
// replayed from the counts, and a step without a count waits for the next march.
// (The midpoint and both its children, three candidates, always give two levels.)
// With `probe` the first march starts at gamma = 1/2: a count of `runs` there
// means that S was never terminated, so every larger gamma takes the same steps
// and the count at 1 is the same.
constexpr int kCand = 4;  // two packed pairs

enum : int { kBisTop = 0, kBisBracket = 1, kBisSearch = 2, kBisDone = 3 };

// the learned bracket: its width in octaves of gamma and its levels of bisection (1024^3, K = 16,
// N_S = 32: 4 octaves in 6 levels give 1.43% supersegment-count error against the search; 4 levels,
// one cached march fewer, 1.14x faster but 5.3-6.2% count error at 2-4 octaves; 5 levels cost as much
// as 6)
#ifndef VDI_LEARNED_OCTAVES
#define VDI_LEARNED_OCTAVES 4.f
#endif
#ifndef VDI_LEARNED_LEVELS
#define VDI_LEARNED_LEVELS 6
#endif

struct GammaSearch {
    int phase;
    float lo, hi, ghi;  // the bracket (log2 gamma in the learned phases), the upper end's gamma
    float llo, lhi;     // log2 of the counts at the bracket's ends (lo: of nt while the lower end is 0)
    int cnt_hi, it, levels;
    int runs;           // the count at gamma = 2
    float x[kCand];     // the march's candidates
    float g2[kCand];    // and their gamma^2
    int quarter;        // kBisTop: the next level is the bracket's lower quarter, as taken from its bottom
    int probe;          // the first march of a search
    int fell;           // the learned bracket fell back to the search
};
static_assert(sizeof(GammaSearch) % 8 == 4, "an odd number of words: a warp's copies in shared memory lie in different banks");

__device__ __forceinline__ float search_gamma(int phase, float x) { return phase == kBisSearch ? x : exp2f(x); }

__device__ __forceinline__ float search_mid(const GammaSearch& s) {
    return s.quarter ? s.lo + 0.25f * VDI_LEARNED_OCTAVES : 0.5f * (s.lo + s.hi);
}

__device__ __forceinline__ void search_begin(GammaSearch& s, int iters, int nt, int runs, bool probe) {
    s.phase = kBisSearch;
    s.lo = 0.f;
    s.hi = 2.f;
    s.ghi = 2.f;
    s.cnt_hi = runs;  // the distance never reaches 2: one supersegment per domain run
    s.it = 0;
    s.levels = iters;
    s.runs = runs;
    s.llo = lg2_approx((float)nt);
    s.lhi = lg2_approx((float)runs);
    s.quarter = 0;
    s.probe = probe ? 1 : 0;
}

// the next march's candidates
__device__ __forceinline__ void search_plan(GammaSearch& s, float lns) {
    if (s.phase == kBisTop) {
        s.x[0] = s.hi;
        s.x[1] = s.lo + 0.5f * VDI_LEARNED_OCTAVES;
        s.x[2] = s.lo + 0.25f * VDI_LEARNED_OCTAVES;
        s.x[3] = 0.5f * (s.x[1] + s.hi);
        return;
    }
    const bool lin = s.phase == kBisSearch;
    const float a = s.lo, b = s.probe ? 1.f : s.hi;
    // the crossing in log2 gamma; a lower end of 0 counts as a sixteenth of the upper end
    const float ub = lin ? lg2_approx(s.hi) : s.hi;
    const float ua = lin ? (a > 0.f ? lg2_approx(a) : ub - 4.f) : a;
    const float uc = ua + (ub - ua) * __fdividef(s.llo - lns, fmaxf(s.llo - s.lhi, 1e-3f));
    const float inv = __fdividef(8.75f, fmaxf(ub - ua, 1e-3f));  // 1 / (0.165 ln 2) of the bracket
    auto F = [&](float u) { return rcp_approx(1.f + ex2_approx((uc - u) * inv)); };
    auto G = [&](float x) { return F(lin ? lg2_approx(x) : x); };
    const float m1 = s.probe ? 0.5f : search_mid(s);
    const float fa = F(ua), fb = F(ub), f1 = G(m1);
    // the more likely half C, the other S
    const bool l1 = f1 - fa >= fb - f1;
    const float pS = l1 ? fb - f1 : f1 - fa, mS = l1 ? 0.5f * (m1 + b) : 0.5f * (a + m1);
    const float Ca = l1 ? a : m1, Cb = l1 ? m1 : b, fCa = l1 ? fa : f1, fCb = l1 ? f1 : fb;
    const float m2 = 0.5f * (Ca + Cb), f2 = G(m2);
    s.x[0] = m1;
    s.x[1] = m2;
    // C's more likely half D, the other O
    const bool l2 = f2 - fCa >= fCb - f2;
    const float pD = l2 ? f2 - fCa : fCb - f2, pO = l2 ? fCb - f2 : f2 - fCa;
    const float Da = l2 ? Ca : m2, Db = l2 ? m2 : Cb, fDa = l2 ? fCa : f2, fDb = l2 ? f2 : fCb;
    const float mD = 0.5f * (Da + Db), mO = l2 ? 0.5f * (m2 + Cb) : 0.5f * (Ca + m2);
    const float f3 = G(mD);
    const bool l3 = f3 - fDa >= fDb - f3;
    const float pE = l3 ? f3 - fDa : fDb - f3, mE = l3 ? 0.5f * (Da + mD) : 0.5f * (mD + Db);
    s.x[2] = mD;
    s.x[3] = pS >= fmaxf(pO, pE) || pS > pD ? mS : (pO > pE ? mO : mE);
}

// replays the bisection from the counts c at the march's candidates; plans the next march or ends
__device__ __forceinline__ void search_replay(GammaSearch& s, const int c[kCand], int n_s, int iters, int nt, float lns) {
    bool above = false;  // the count at gamma = 1 is c[0]
    if (s.phase == kBisTop) {
        if (c[0] > n_s) {  // no feasible gamma in the bracket: the full search
            s.fell = 1;
            search_begin(s, iters, nt, s.runs, true);
            search_plan(s, lns);
            return;
        }
        s.phase = kBisBracket;
        s.hi = s.x[0];
        s.ghi = search_gamma(s.phase, s.hi);
        s.cnt_hi = c[0];
        s.lhi = lg2_approx((float)c[0]);
        ++s.it;
        if (c[1] <= n_s) {
            s.hi = s.x[1];
            s.ghi = search_gamma(s.phase, s.hi);
            s.cnt_hi = c[1];
            s.lhi = lg2_approx((float)c[1]);
            s.quarter = 1;
        } else {
            s.lo = s.x[1];
            s.llo = lg2_approx((float)c[1]);
        }
        if (s.cnt_hi == n_s) s.it = s.levels;
    } else if (s.probe) {
        above = c[0] == s.runs;
        s.probe = 0;
    }
#pragma unroll 1
    for (int q = 0; q <= kCand; ++q) {  // the level above a probe, and one level per candidate
        if (s.it >= s.levels) break;
        const float mid = search_mid(s);
        int v = -1;
#pragma unroll
        for (int w = 0; w < kCand; ++w) v = mid == s.x[w] ? c[w] : v;
        if (v < 0) {
            if (!(above && mid == 1.f)) break;
            v = c[0];
        }
        ++s.it;
        s.quarter = 0;
        const float lv = lg2_approx((float)v);
        if (v <= n_s) {
            s.hi = mid;
            s.ghi = search_gamma(s.phase, mid);
            s.cnt_hi = v;
            s.lhi = lv;
            if (v == n_s) s.it = s.levels;
        } else {
            s.lo = mid;
            s.llo = lv;
        }
    }
    if (s.it >= s.levels) s.phase = kBisDone;
    else search_plan(s, lns);
}

// the candidates' gamma^2 for the march
__device__ __forceinline__ void search_store(GammaSearch& sh, GammaSearch& s) {
#pragma unroll
    for (int w = 0; w < kCand; ++w) {
        const float g = search_gamma(s.phase, s.x[w]);
        s.g2[w] = __fmul_rn(g, g);
    }
    sh = s;
}

// The end of a lane's march, and the start of a ray's search, out of line: seldom, and of many values.  Both work
// on the lane's state in shared memory and leave the next march's candidates there.
__device__ __noinline__ void search_end_march(GammaSearch& sh, int c0, int c1, int c2, int c3, int n_s, int iters,
                                              int nt) {
    const int c[4] = {c0, c1, c2, c3};
    GammaSearch s = sh;
    search_replay(s, c, n_s, iters, nt, lg2_approx((float)n_s + 0.3f));
    search_store(sh, s);
}

// starts the search of a list whose counts at gamma = 0 and 2 are nt > n_s and runs
__device__ __noinline__ void search_start(GammaSearch& sh, int n_s, int iters, int nt, int runs, bool probe) {
    GammaSearch s;
    s.fell = 0;
    search_begin(s, iters, nt, runs, probe);
    search_plan(s, lg2_approx((float)n_s + 0.3f));
    search_store(sh, s);
}


}  // namespace vdi
