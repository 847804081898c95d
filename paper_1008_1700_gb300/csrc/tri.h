// Unevaluated sums of three floats: about 70 bits in FP32 arithmetic (products by fused
// multiply-add, sums by Knuth's two-sum), for sums and scalars where FP64 is too slow.
// Host code includes it too (compile without contraction of a product and a sum).
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define DDPS_TRI __device__ __forceinline__
#else
#define DDPS_TRI inline
#endif

namespace ddps {

#ifdef __CUDACC__
DDPS_TRI float add_rn(float a, float b) { return __fadd_rn(a, b); }
DDPS_TRI float sub_rn(float a, float b) { return __fsub_rn(a, b); }
DDPS_TRI float mul_rn(float a, float b) { return __fmul_rn(a, b); }
DDPS_TRI float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
DDPS_TRI float add_rn(float a, float b) { return a + b; }
DDPS_TRI float sub_rn(float a, float b) { return a - b; }
DDPS_TRI float mul_rn(float a, float b) { return a * b; }
DDPS_TRI float fma_rn(float a, float b, float c) { return std::fma(a, b, c); }
#endif

struct Two {
  float x, y;
};
struct alignas(16) Tri {
  float h, m, l;  // normalised: |m| <= ulp(h) / 2, |l| <= ulp(m) / 2
};
DDPS_TRI Two two_sum(float a, float b) {  // a + b = x + y exactly
  const float s = add_rn(a, b), t = sub_rn(s, a);
  return {s, add_rn(sub_rn(a, sub_rn(s, t)), sub_rn(b, t))};
}
DDPS_TRI Two two_prod(float a, float b) {  // a b = x + y exactly
  const float p = mul_rn(a, b);
  return {p, fma_rn(a, b, -p)};
}
DDPS_TRI Tri settle(Tri x) {
  const Two a = two_sum(x.m, x.l), b = two_sum(x.h, a.x), c = two_sum(b.y, a.y);
  return {b.x, c.x, c.y};
}
// running sums: left unnormalised (the lower words stay far below the terms' last bits)
DDPS_TRI Tri sum(Tri x, Tri y) {
  const Two a = two_sum(x.h, y.h), b = two_sum(x.m, y.m), c = two_sum(b.x, a.y);
  return {a.x, c.x, add_rn(add_rn(x.l, y.l), add_rn(b.y, c.y))};
}
DDPS_TRI Tri mul(float a, float b) {
  const Two p = two_prod(a, b);
  return {p.x, p.y, 0.f};
}
DDPS_TRI Tri mul(Tri s, Tri b) {
  const Two p = two_prod(s.h, b.h), q = two_prod(s.h, b.m), r = two_prod(s.m, b.h);
  const Two c = two_sum(q.x, r.x), d = two_sum(c.x, p.y);
  const float low = fma_rn(s.h, b.l, fma_rn(s.l, b.h, fma_rn(s.m, b.m, add_rn(q.y, r.y))));
  return settle({p.x, d.x, add_rn(low, add_rn(c.y, d.y))});
}
DDPS_TRI Tri neg(Tri x) { return {-x.h, -x.m, -x.l}; }
// a - b q for a q near a / b, not normalised
DDPS_TRI Tri left(Tri a, Tri b, float q) {
  const Two p = two_prod(b.h, -q), f = two_prod(b.m, -q), s = two_sum(a.h, p.x);
  const Two c = two_sum(a.m, p.y), d = two_sum(c.x, f.x), e = two_sum(s.y, d.x);
  const Two u = two_sum(s.x, e.x);
  const float low = fma_rn(-q, b.l, add_rn(add_rn(a.l, f.y), add_rn(c.y, d.y)));
  return {u.x, u.y, add_rn(e.y, low)};
}
// quotient, a float at a time: each of what the ones before leave
DDPS_TRI Tri quot(Tri a, Tri b) {
  const float inv = 1.f / b.h, q = a.h * inv;
  const Tri r = left(a, b, q);
  const float t = r.h * inv;
  const Tri w = left(r, b, t);
  return settle({q, t, add_rn(w.h, add_rn(w.m, w.l)) * inv});
}
// r + a x and r + a x + b y rounded once to a float: the leading products and sums with their
// errors, these and the middle words' products as a second sum with its errors, and the rest.
DDPS_TRI float lin(float r, Tri a, float x) {
  const Two p = two_prod(a.h, x), q = two_prod(a.m, x), s = two_sum(p.x, r);
  const Two c = two_sum(p.y, q.x), d = two_sum(c.x, s.y), u = two_sum(s.x, d.x);
  const float rest = add_rn(add_rn(c.y, d.y), fma_rn(a.l, x, q.y));
  return add_rn(u.x, add_rn(u.y, rest));
}
DDPS_TRI float lin(float r, Tri a, float x, Tri b, float y) {
  const Two p = two_prod(a.h, x), q = two_prod(b.h, y), f = two_prod(a.m, x), g = two_prod(b.m, y);
  const Two s = two_sum(p.x, q.x), t = two_sum(s.x, r);
  const Two c = two_sum(p.y, q.y), d = two_sum(s.y, t.y), e = two_sum(f.x, g.x);
  const Two i = two_sum(c.x, d.x), j = two_sum(i.x, e.x), u = two_sum(t.x, j.x);
  const float rest = add_rn(add_rn(add_rn(c.y, d.y), add_rn(e.y, add_rn(i.y, j.y))),
                            fma_rn(a.l, x, fma_rn(b.l, y, add_rn(f.y, g.y))));
  return add_rn(u.x, add_rn(u.y, rest));
}
DDPS_TRI float value(Tri x) { return x.h; }
DDPS_TRI bool less(Tri a, Tri b) {
  return a.h < b.h || (a.h == b.h && (a.m < b.m || (a.m == b.m && a.l < b.l)));
}
DDPS_TRI bool at_most(Tri a, Tri b) {  // false for NaN
  return a.h < b.h || (a.h == b.h && (a.m < b.m || (a.m == b.m && a.l <= b.l)));
}

// the same in FP64
DDPS_TRI double lin(double r, double a, double x) { return r + a * x; }
DDPS_TRI double lin(double r, double a, double x, double b, double y) {
  return r + (a * x + b * y);
}
DDPS_TRI double sum(double x, double y) { return x + y; }
DDPS_TRI double settle(double x) { return x; }
DDPS_TRI double mul(double a, double b) { return a * b; }
DDPS_TRI double neg(double x) { return -x; }
DDPS_TRI double quot(double a, double b) { return a / b; }
DDPS_TRI double value(double x) { return x; }
DDPS_TRI bool less(double a, double b) { return a < b; }
DDPS_TRI bool at_most(double a, double b) { return a <= b; }

}  // namespace ddps
