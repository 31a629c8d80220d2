// Sums, products and the unit normal in two-float arithmetic: a value is the sum
// of an FP32 number and a rest below half a unit of its last place.  Plain C++
// too (compiled without contraction), so that it can be checked on the host.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define LBE_HD __host__ __device__ __forceinline__
#else
#define LBE_HD static inline
#endif

namespace lbe {

// a b rounded, never fused with what follows
LBE_HD float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

// Error-free transformations: a + b = s + e exactly (Knuth's two-sum; the fast
// variant needs |a| >= |b|).
LBE_HD void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
LBE_HD void fast_two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  e = b - (s - a);
}

struct Two {
  float h, l;
};
LBE_HD Two two_add(Two a, Two b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  Two r;
  fast_two_sum(s, e + (a.l + b.l), r.h, r.l);
  return r;
}
LBE_HD Two two_square(Two a) {
  Two r;
  r.h = mul_rn(a.h, a.h);
  r.l = fmaf(a.h, a.h, -r.h) + 2.f * a.h * a.l;
  return r;
}

// The unit normal grad c / sqrt(|grad c|^2 + eta_n^2) (Eq. 3), of c = c + cl at
// entry k of a field whose rows are w entries apart; e = 144 eta_n^2.  kappa is
// the difference of normals that differ by 1/R, so a normal that is off by a
// unit of its last place costs R units of kappa.  Formed to 2^-40 (and 2^-44 of
// the differences that cancel in grad c), the result is the exact normal
// rounded, but for one in some ten thousand next to a tie.
LBE_HD void unit_normal(const float* c, const float* cl, int k, int w, Two e, float& nx,
                        float& ny) {
  auto diff = [&](int p, int m) {
    Two a, b;
    two_sum(c[k + p], -c[k + m], a.h, a.l);
    two_sum(cl[k + p], -cl[k + m], b.h, b.l);
    return two_add(a, b);
  };
  auto four = [](Two a) { return Two{4.f * a.h, 4.f * a.l}; };
  // g = 12 grad c
  const Two d1 = diff(w + 1, -w - 1), d2 = diff(1 - w, w - 1);
  const Two gx = two_add(four(diff(1, -1)), two_add(d1, d2));
  const Two gy = two_add(four(diff(w, -w)), two_add(d1, Two{-d2.h, -d2.l}));
  const Two s = two_add(two_add(two_square(gx), two_square(gy)), e);
  // 1/sqrt(s) = y (1 + t/2 + 3 t^2/8 + ...), t = 1 - s y^2 of 2^-21 at most
  const float y = 1.f / sqrtf(s.h);
  const Two q = two_square(Two{y, 0.f});
  const float p = mul_rn(s.h, q.h);
  const float t = (1.f - p) - (fmaf(s.h, q.h, -p) + (s.h * q.l + s.l * q.h));
  auto scaled = [&](Two g) {
    const float n = mul_rn(g.h, y);
    return n + (fmaf(g.h, y, -n) + (g.l * y + n * (0.5f * t)));
  };
  nx = scaled(gx);
  ny = scaled(gy);
}

}  // namespace lbe
