// The fixed-point primitives of su2_fixed.cuh on the host, for
// tests/test_fixed_point.py.
#include <cstring>

#include "su2_fixed.cuh"

using namespace su2;

static FixQuat link(const double* v, int conj, FixBad& bad, bool any = false) {
  uint32_t w[8];
  std::memcpy(w, v, sizeof w);
  return any ? fix_any_link(w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7], conj ? -1 : 0, bad)
             : fix_link(w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7], conj ? -1 : 0, bad);
}

extern "C" {
int fixed_frac() { return kFixFrac; }
int fixed_log_entry_alignment() { return (int)alignof(FixLog); }
int fixed_log_entry_size() { return (int)sizeof(FixLog); }
// out[4]: the converted components, v = h 2^29 + l; returns fix_ok
static int convert(const double* v, int conj, int64_t* out, bool any) {
  FixBad bad{0, 0};
  const FixQuat q = link(v, conj, bad, any);
  const Fix f[4] = {q.w, q.x, q.y, q.z};
  for (int i = 0; i < 4; ++i) out[i] = (int64_t)f[i].h * (1 << kFixLow) + f[i].l;
  return fix_ok(bad);
}
int fixed_link(const double* v, int conj, int64_t* out) { return convert(v, conj, out, false); }
int fixed_any_link(const double* v, int conj, int64_t* out) { return convert(v, conj, out, true); }
int64_t fixed_any(double v) {
  uint32_t w[2];
  std::memcpy(w, &v, 8);
  const Fix f = fix_from_any(w[0], w[1]);
  return (int64_t)f.h * (1 << kFixLow) + f.l;
}
// out[4] = sum over n of a b c, in units of 2^-58; a, b, c: n quaternions
int fixed_triples(const double* a, const double* b, const double* c, int n, int64_t* out) {
  FixBad bad{0, 0};
  FixSum s = fix_zero();
  for (int i = 0; i < n; ++i)
    fix_mac(s, fix_mul(link(a + 4 * i, 0, bad), link(b + 4 * i, 0, bad)), link(c + 4 * i, 0, bad));
  out[0] = fix_fold(s.hw, s.mw);
  out[1] = fix_fold(s.hx, s.mx);
  out[2] = fix_fold(s.hy, s.my);
  out[3] = fix_fold(s.hz, s.mz);
  return fix_ok(bad);
}
int64_t fixed_neg_log(uint32_t x) { return fix_neg_log(x); }
uint64_t fixed_cos2(uint32_t x) { return fix_cos2(x); }
void fixed_sincos(uint32_t x, int64_t* sc) { fix_sincos(x, sc, sc + 1); }
}
