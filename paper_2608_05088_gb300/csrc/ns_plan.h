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
// Rounding.  In bf16 the grouped form loses accuracy (A carries the squared
// singular values), so from the second iterate on it works in fp16: 11
// significant bits in place of 8.  The iterates are bounded (|p(x)| stays near
// 1), so the range is known: X is stored times kScaleX and A times kScaleA
// (powers of two), which puts fp16's smallest step 2^-24 at 2^-32 and 2^-34 of
// a unit singular value.  The first iteration keeps bf16, because Mt's scale is
// not known before it.  Against fp64 the grouped form is closer than the
// iterated one: 0.30-0.55e-2 in place of 0.7-1.7e-2 relative on frames with
// log-normal scales (sigma 0 to 3, k = 5), and no worse on the geometric,
// low-rank and graded spectra of tests/test_ns_plan.py, which reads the plan
// from the library and runs its arithmetic on the CPU.
//
// Which form runs (ns_grouped_run, ns_grouped_shape) follows from k, from the
// coefficients, from the shape and from the size of the set.
#pragma once
#include <cmath>
#include <cstdint>

#include "common.cuh"

namespace malt {

// Groups of a k-iteration run after the first iteration (k = 3 .. 8), zero
// ended.  Pairs; three at a time loses accuracy on ill-conditioned frames, so
// it is taken only where it ends the longest run.
constexpr int kMinGroupedSteps = 3, kMaxGroupedSteps = 8;
constexpr int kNsGroups[kMaxGroupedSteps + 1][4] = {
    {0}, {0}, {0}, {2, 0}, {2, 1, 0}, {2, 2, 0}, {2, 2, 1, 0}, {2, 2, 2, 0}, {2, 2, 3, 0}};

constexpr float kScaleX = 256.f;      // fp16 iterates hold kScaleX * X
constexpr float kScaleA = 1024.f;     // fp16 Gram matrices hold kScaleA * A (and H A the same)

// Whether a run of k iterations with these coefficients may take the grouped
// form: the fp16 values must stay in range and above its smallest step.  The
// singular values of the first iterate are at most 1 (X is divided by its
// Frobenius norm), so the range of every later one follows from the extrema of
// x h(x^2), h(t) = a + b t + c t^2.  Coefficients that let values grow or that
// amplify small ones further than 8 iterations of a = 3.4445 do stay in bf16,
// which has fp32's range.
inline bool ns_grouped_run(int k, double a, double b, double c) {
    if (k < kMinGroupedSteps || k > kMaxGroupedSteps) return false;
    if (!(std::isfinite(a) && std::isfinite(b) && std::isfinite(c))) return false;
    double m = 1.0 + 1.0 / 64, amp = 1.0;       // bound of the singular values; of the gain so far
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
        // H and Q (a product of up to three H) below 2^12, kScaleA * (H A) and
        // kScaleX * X below 2^14.
        if (!(hmax <= 16.0) || !(pmax <= 3.0) || !(m * pmax <= 8.0)) return false;
        amp *= hmax;
        if (!(amp <= 32768.0)) return false;
        m = std::fmax(pmax, 1e-3) * (1.0 + 1.0 / 64);
    }
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
// one 2048 x 4096 383 / 339, 8 of 1280 x 5120 727 / 570.
// tiles: 256 x 256 tiles of one symmetric product over the set.
inline bool ns_grouped_shape(int64_t p, int64_t q, int64_t tiles) {
    return q >= 2 * p && 50 * (q - 2 * p) + tiles * p >= 50000;
}

// The grouped form's operations; returns their number (at most kMaxGroupedOps).
inline int ns_grouped_ops(int k, float a, float b, float c, NsOp* ops) {
    int n = 0;
    for (int kind = kGram; kind <= kBX; ++kind) ops[n++] = ns_iterated_op(0, kind, false, a, b, c);
    // The first iterate goes out as fp16, scaled.
    ops[n - 1].out16 = 1;
    ops[n - 1].gamma = kScaleX;
    int cur = 1;                                  // the iterate that the next group reads
    for (const int* g = kNsGroups[k]; *g > 0; ++g) {
        const bool last = g[1] == 0;
        auto op = [&](int kind, int x, int y, int out, float gamma) {
            NsOp o = ns_iterated_op(1, kind, false, a, b, c);
            o.f16 = o.out16 = 1;
            o.a = static_cast<int8_t>(x);
            o.b = static_cast<int8_t>(y);
            o.e = kBufNone;
            o.out = static_cast<int8_t>(out);
            o.alpha = o.beta = 0.f;
            o.gamma = gamma;
            ops[n++] = o;
        };
        op(kGram, kBufX + cur, kBufX + cur, 0, kScaleA / (kScaleX * kScaleX));
        int q = -1;                               // buffer of the running product Q
        for (int j = 0; j < *g; ++j) {
            const int h = q == 1 ? 2 : 1;         // H next to A (buffer 0) and Q
            op(kPoly, 0, 0, h, c / (kScaleA * kScaleA));
            ops[n - 1].e = 0;
            ops[n - 1].alpha = a;
            ops[n - 1].beta = b / kScaleA;
            int free_buf = 6 - h - (q < 0 ? 3 : q);   // buffers 1 .. 3 without h and q
            if (q < 0) {
                q = h;
                free_buf = h == 1 ? 2 : 1;
            } else {
                op(kPoly, h, q, free_buf, 1.f);
                const int old = q;
                q = free_buf;
                free_buf = old;
            }
            if (j + 1 < *g) {
                op(kPoly, h, 0, free_buf, 1.f);   // H A
                op(kPoly, free_buf, h, 0, 1.f);   // (H A) H over A
            }
        }
        op(kBX, q, kBufX + cur, last ? kBufO : kBufX + (cur ^ 1), last ? 1.f / kScaleX : 1.f);
        if (last) ops[n - 1].out16 = 0;           // O is bf16
        cur ^= 1;
    }
    return n;
}

}  // namespace malt
