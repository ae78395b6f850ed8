// The bisection search for gamma over a pixel's pieces, as the compositing search's lanes run it: which gammas a march
// evaluates, and the replay of sequential bisection from their counts (sec. 2.4).
#pragma once

#include "vdi_device.cuh"

namespace vdi {

// A march over the pieces evaluates four midpoints: the next one and the three
// that the bisection is most likely to visit after it.  The likelihood comes
// from where the count, taken as a power of gamma between the bracket's ends,
// crosses n_s (a logistic belief in log2 gamma about that point).  It only
// chooses what is evaluated: the bisection's own steps are replayed from the
// counts, and a step without a count waits for the next march.  (The midpoint
// and both its children, three candidates, always give two levels; these four
// gave 2.6 on the searched samples of the 512^3 frame, in two packed pairs.)
constexpr int kCand = 4;

struct GammaSearch {
    int done;
    float lo, hi, ghi;  // the bracket, the result
    float llo, lhi;     // log2 of the counts at the bracket's ends (lo: of nt while the lower end is 0)
    int cnt_hi, it, levels;
    float x[kCand];     // the march's candidates
    float g2[kCand];    // and their gamma^2
};
static_assert(sizeof(GammaSearch) % 8 == 4, "an odd number of words: a warp's copies in shared memory lie in different banks");

// the next march's candidates
__device__ __forceinline__ void search_plan(GammaSearch& s, float lns) {
    // the crossing in log2 gamma; a lower end of 0 counts as a sixteenth of the upper end
    const float ub = lg2_approx(s.hi), ua = s.lo > 0.f ? lg2_approx(s.lo) : ub - 4.f;
    const float uc = ua + (ub - ua) * __fdividef(s.llo - lns, fmaxf(s.llo - s.lhi, 1e-3f));
    const float inv = __fdividef(8.75f, fmaxf(ub - ua, 1e-3f));  // the belief's width: 0.3 of the bracket
    auto F = [&](float u) { return rcp_approx(1.f + ex2_approx((uc - u) * inv)); };
    auto G = [&](float x) { return F(lg2_approx(x)); };
    const float a = s.lo, b = s.hi, m1 = 0.5f * (a + b);
    const float fa = F(ua), fb = F(ub), f1 = G(m1);
    // the more likely half C, the other S
    const bool l1 = f1 - fa >= fb - f1;
    const float pS = l1 ? fb - f1 : f1 - fa, mS = l1 ? 0.5f * (m1 + b) : 0.5f * (a + m1);
    const float Ca = l1 ? a : m1, Cb = l1 ? m1 : b, fCa = l1 ? fa : f1, fCb = l1 ? f1 : fb;
    const float m2 = 0.5f * (Ca + Cb), f2 = G(m2);
    // C's more likely half D, the other O
    const bool l2 = f2 - fCa >= fCb - f2;
    const float pD = l2 ? f2 - fCa : fCb - f2, pO = l2 ? fCb - f2 : f2 - fCa;
    const float Da = l2 ? Ca : m2, Db = l2 ? m2 : Cb, fDa = l2 ? fCa : f2, fDb = l2 ? f2 : fCb;
    const float mD = 0.5f * (Da + Db), mO = l2 ? 0.5f * (m2 + Cb) : 0.5f * (Ca + m2);
    const float f3 = G(mD);
    const bool l3 = f3 - fDa >= fDb - f3;
    const float pE = l3 ? f3 - fDa : fDb - f3, mE = l3 ? 0.5f * (Da + mD) : 0.5f * (mD + Db);
    s.x[0] = m1;
    s.x[1] = m2;
    s.x[2] = mD;
    s.x[3] = pS >= fmaxf(pO, pE) || pS > pD ? mS : (pO > pE ? mO : mE);
#pragma unroll
    for (int w = 0; w < kCand; ++w) s.g2[w] = __fmul_rn(s.x[w], s.x[w]);
}

// The start of a pixel's search (nt > n_s: the count at gamma = 0) and the end of a lane's march, out of line: seldom,
// and of many values.  Both work on the lane's state in shared memory and leave the next march's candidates there.
static __device__ __noinline__ void search_start(GammaSearch& sh, int n_s, int iters, int nt) {
    GammaSearch s;
    s.done = 0;
    s.lo = 0.f;
    s.hi = s.ghi = 2.f;
    s.cnt_hi = 1;  // the distance never reaches 2: one supersegment
    s.it = 0;
    s.levels = iters;
    s.llo = lg2_approx((float)nt);
    s.lhi = 0.f;
    search_plan(s, lg2_approx((float)n_s + 0.3f));
    sh = s;
}

// replays the bisection from the counts at the march's candidates; plans the next march or ends
static __device__ __noinline__ void search_end_march(GammaSearch& sh, int c0, int c1, int c2, int c3, int n_s) {
    const int c[kCand] = {c0, c1, c2, c3};
    GammaSearch s = sh;
#pragma unroll 1
    for (int q = 0; q < kCand && s.it < s.levels; ++q) {
        const float mid = 0.5f * (s.lo + s.hi);
        int v = -1;
#pragma unroll
        for (int w = 0; w < kCand; ++w) v = mid == s.x[w] ? c[w] : v;
        if (v < 0) break;
        ++s.it;
        const float lv = lg2_approx((float)v);
        if (v <= n_s) {
            s.hi = s.ghi = mid;
            s.cnt_hi = v;
            s.lhi = lv;
            if (v == n_s) s.it = s.levels;
        } else {
            s.lo = mid;
            s.llo = lv;
        }
    }
    s.done = s.it >= s.levels;
    if (!s.done) search_plan(s, lg2_approx((float)n_s + 0.3f));
    sh = s;
}

}  // namespace vdi
