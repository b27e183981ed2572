// ns_plan.h -- the products of a Newton-Schulz run, as a list of operations.
//
// Two forms compute the same polynomial of the p x q frame X:
//
//  * iterated: k times A = X X^T, B' = aI + bA + cA^2, X <- B' X, all in bf16
//    (3 p^2 q + p^3 multiply-adds per iteration with the symmetric products
//    counted once).
//  * grouped: the first iteration as above, then the remaining ones in groups
//    that go back to X once.  Inside a group A stays a p x p matrix: with
//    H = aI + bA + cA^2 the next iterate is H X and its Gram matrix is H A H,
//    so an iteration costs four p x p products (H, H A, (H A) H and the running
//    product Q of the H's) instead of a Gram and a B*X product over q.  All
//    these are polynomials of one symmetric matrix, so they commute and are
//    symmetric themselves, and every one is computed as an upper triangle.
//    With q = 4 p a merged iteration costs 4 p^3 in place of 13 p^3.
//
// Rounding.  In bf16 the grouped form loses accuracy, since A carries the squared
// singular values (1.5 times the iterated form's error, 2 in the worst row), so the
// p x p matrices of a group are fp16: 11 significant bits in place of 8.  Their
// entries are bounded (|p(x)| stays near 1), so each is stored times the power of two
// that brings its bound near fp16's largest value (ns_grouped_run): A and H A times
// 2^14, H times 2^13 with the default coefficients.  The iterates X are
//  * fp16 times 2^15 for preconditioned frames (MALT, MALTER: L M R, whose rows and
//    columns are drawn together);
//  * bf16, which has fp32's range, for frames as they are (Muon).  A column 1e-10 of
//    the others leaves fp16 with an error of 1 at any scale.  The running product that
//    is applied to X goes out in X's type; bf16 costs it accuracy, and at k = 3 the
//    worst column gets 1.0 - 1.3 times the iterated form's error, so these runs stay
//    iterated.
// The first iteration keeps bf16, because Mt's scale is not known before it.
//
// Error against fp64 in terms of the iterated form's, on frames with log-normal scales
// of sigma 0 to 3 (geometric means over 64 x 128 to 512 x 2048, k = 3 to 8): preconditioned,
// fp16, the whole frame 0.3 - 0.65, the worst row and column 0.2 - 0.7; as they are,
// bf16, 0.6 - 0.9 and 0.5 - 0.95.  Rows and columns far smaller than the rest: half
// of them 1e-8 of the others have errors of 0.005 - 0.015 (iterated 0.01 - 0.03; k = 3:
// the same down to 1e-7).  Below that the range of fp16 ends: at 1e-9 0.03 - 0.14, at 1e-10
// 0.3 - 1; with X in bf16 columns have no such limit and rows 0.005 - 0.08 at 1e-9.
// An update that small against the others moves W by less than W's own fp32 rounding.
// tests/test_ns_plan.py reads the plan from the library and runs its arithmetic on
// the CPU, on these frames and on geometric, low-rank, graded and blocked ones.
//
// Which form runs (ns_grouped_run, ns_grouped_shape) follows from k, from the
// coefficients, from whether the frames are preconditioned, from the shape and from
// the size of the set.
#pragma once
#include <cmath>
#include <cstdint>

#include "common.cuh"

namespace malt {

// Groups of a k-iteration run after the first iteration (k = 3 .. 8), zero
// ended.  Pairs; three at a time loses accuracy on ill-conditioned frames, so
// it is taken only where it ends the longest run.
constexpr int kMinGroupedSteps = 3, kMinGroupedStepsRaw = 4, kMaxGroupedSteps = 8;
constexpr int kNsGroups[kMaxGroupedSteps + 1][4] = {
    {0}, {0}, {0}, {2, 0}, {2, 1, 0}, {2, 2, 0}, {2, 2, 1, 0}, {2, 2, 2, 0}, {2, 2, 3, 0}};

// Factors (powers of two) by which the fp16 matrices are stored: X, A, H A, and the
// product of 1, 2 or 3 H.
struct NsScales {
    float x = 1.f, a = 1.f, ha = 1.f, h[3] = {1.f, 1.f, 1.f};
};

// The largest power of two that keeps a bound below 2^15.5, 0.7 of fp16's largest
// value: the bounds have 1/64 to spare per iteration, rounding moves values by less.
inline float ns_scale_to_fp16(double bound) {
    return static_cast<float>(std::exp2(std::floor(15.5 - std::log2(std::fmax(bound, 1.0)))));
}

// Whether a run of k iterations with these coefficients may take the grouped
// form (raw: on frames that are not preconditioned), and its scales: the fp16
// values must stay in range.  The singular values of the first iterate are at most
// 1 (X is divided by its Frobenius norm), so the range of every later one follows
// from the extrema of x h(x^2) and of h, h(t) = a + b t + c t^2.  Coefficients that let values grow or
// that amplify small ones further than 8 iterations of a = 3.4445 do stay in the
// iterated form.
inline bool ns_grouped_run(int k, double a, double b, double c, bool raw, NsScales* scales = nullptr) {
    if (k < (raw ? kMinGroupedStepsRaw : kMinGroupedSteps) || k > kMaxGroupedSteps) return false;
    if (!(std::isfinite(a) && std::isfinite(b) && std::isfinite(c))) return false;
    double m = 1.0 + 1.0 / 64, amp = 1.0;       // bound of the singular values; of the gain so far
    double x_max = 0.0, a_max = 0.0, h_max = 0.0, ha_max = 0.0;   // of X (once iterated), A, H and H A
    for (int i = 0; i < k; ++i) {
        // extrema of h on [0, m^2] and of x h(x^2) on [0, m]
        auto h = [&](double t) { return std::fabs(a + b * t + c * t * t); };
        double hmax = std::fmax(h(0.0), h(m * m));
        if (c != 0.0) {
            const double t = -b / (2.0 * c);
            if (t > 0.0 && t < m * m) hmax = std::fmax(hmax, h(t));
        }
        double pmax = m * h(m * m);
        const double disc = 9.0 * b * b - 20.0 * a * c;   // roots of a + 3 b t + 5 c t^2
        if (c != 0.0 && disc >= 0.0) {
            for (double s : {-1.0, 1.0}) {
                const double t = (-3.0 * b + s * std::sqrt(disc)) / (10.0 * c);
                if (t > 0.0 && t < m * m) pmax = std::fmax(pmax, std::sqrt(t) * h(t));
            }
        } else if (c == 0.0 && b != 0.0) {
            const double t = -a / (3.0 * b);
            if (t > 0.0 && t < m * m) pmax = std::fmax(pmax, std::sqrt(t) * h(t));
        }
        if (!(hmax <= 16.0) || !(pmax <= 3.0) || !(m * pmax <= 8.0)) return false;
        amp *= hmax;
        if (!(amp <= 32768.0)) return false;
        a_max = std::fmax(a_max, m * m);
        h_max = std::fmax(h_max, hmax);
        ha_max = std::fmax(ha_max, m * pmax);
        x_max = std::fmax(x_max, pmax * (1.0 + 1.0 / 64));
        m = std::fmax(pmax, 1e-3) * (1.0 + 1.0 / 64);
    }
    if (scales != nullptr)
        *scales = {ns_scale_to_fp16(x_max), ns_scale_to_fp16(a_max), ns_scale_to_fp16(ha_max),
                   {ns_scale_to_fp16(h_max), ns_scale_to_fp16(h_max * h_max),
                    ns_scale_to_fp16(h_max * h_max * h_max)}};
    return true;
}

// Frames that take the grouped form when the run may.  A merged iteration
// replaces 3 p^2 q + p^3 by 4 p^3, which are equal at q = p, in more and less
// efficient products (short reductions): at q = 1.5 p it gains 2 - 3 % in large
// sets and loses 2 - 4 % in small ones (1280 x 1920, iterated / grouped: 32 of them
// 1259 / 1230 us, 8 of them 369 / 386), so q >= 2 p.  Where a set is only a few
// tiles, a product takes its latency plus its reduction, and the grouped form has
// two products more: it pays once the q - 2 p that a merged iteration saves are
// long enough or the set is large.  Measured at k = 5, us of Newton-Schulz per
// step, iterated / grouped: one 512 x 1024 108 / 114, 32 of them 204 / 206, one
// 512 x 2048 127 / 128, one 256 x 4096 155 / 133, 16 of 1024 x 2048 439 / 400,
// one 2048 x 4096 383 / 339, 8 of 1280 x 5120 727 / 570 (at the line itself, as
// with the 512 x 2048, it is a percent either way).
// tiles: 256 x 256 tiles of one symmetric product over the set.
inline bool ns_grouped_shape(int64_t p, int64_t q, int64_t tiles) {
    return q >= 2 * p && 50 * (q - 2 * p) + tiles * p >= 50000;
}

// The grouped form's operations; returns their number (at most kMaxGroupedOps).
// (a run that may not take the form: the same products, scales 1)
inline int ns_grouped_ops(int k, float a, float b, float c, bool raw, NsOp* ops) {
    NsScales sc;
    ns_grouped_run(k, a, b, c, raw, &sc);
    const bool x16 = !raw;
    const float xs = x16 ? sc.x : 1.f;
    int n = 0;
    for (int kind = kGram; kind <= kBX; ++kind) ops[n++] = ns_iterated_op(0, kind, false, a, b, c);
    ops[n - 1].out16 = x16;
    ops[n - 1].gamma = xs;
    int cur = 1;                                  // the iterate that the next group reads
    for (const int* g = kNsGroups[k]; *g > 0; ++g) {
        const bool last = g[1] == 0;
        auto op = [&](int kind, int x, int y, int out, bool f16, bool out16, float gamma) {
            NsOp o = ns_iterated_op(1, kind, false, a, b, c);
            o.f16 = f16;
            o.out16 = out16;
            o.a = static_cast<int8_t>(x);
            o.b = static_cast<int8_t>(y);
            o.e = kBufNone;
            o.out = static_cast<int8_t>(out);
            o.alpha = o.beta = 0.f;
            o.gamma = gamma;
            ops[n++] = o;
        };
        op(kGram, kBufX + cur, kBufX + cur, 0, x16, true, sc.a / (xs * xs));
        int q = -1;                               // buffer of the running product Q
        float q_scale = 1.f;
        for (int j = 0; j < *g; ++j) {
            const bool end = j + 1 == *g;         // Q is complete: X's type
            const bool to16 = !end || x16;
            const float s = to16 ? sc.h[j] : 1.f;    // of Q
            const int h = q == 1 ? 2 : 1;         // H next to A (buffer 0) and Q
            const float hs = q < 0 ? s : sc.h[0];
            op(kPoly, 0, 0, h, true, q >= 0 || to16, hs * c / (sc.a * sc.a));
            ops[n - 1].e = 0;
            ops[n - 1].alpha = hs * a;
            ops[n - 1].beta = hs * b / sc.a;
            int free_buf = 6 - h - (q < 0 ? 3 : q);   // buffers 1 .. 3 without h and q
            if (q < 0) {
                q = h;
                free_buf = h == 1 ? 2 : 1;
            } else {
                op(kPoly, h, q, free_buf, true, to16, s / (hs * q_scale));
                const int old = q;
                q = free_buf;
                free_buf = old;
            }
            q_scale = s;
            if (!end) {
                op(kPoly, h, 0, free_buf, true, true, sc.ha / (hs * sc.a));   // H A
                op(kPoly, free_buf, h, 0, true, true, sc.a / (sc.ha * hs));   // (H A) H over A
            }
        }
        // (O is bf16)
        op(kBX, q, kBufX + cur, last ? kBufO : kBufX + (cur ^ 1), x16, x16 && !last,
           1.f / (last ? q_scale * xs : q_scale));
        cur ^= 1;
    }
    return n;
}

}  // namespace malt
