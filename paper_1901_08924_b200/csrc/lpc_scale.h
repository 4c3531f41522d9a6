// The reciprocals that the scale rule (the c * std threshold and Eq. 2) uses, made on the host.
#pragma once
#include <stdint.h>

namespace lpc {

struct ScaleRule {
  int64_t len;                 // values of the vector
  float inv_len, inv_len_low;  // 1 / len as the unrounded sum of two floats
  float levels, inv_levels;    // 2^(b-1) - 1 (b = 1, 32: 1) and its reciprocal, rounded
};
inline ScaleRule scale_rule(int64_t len, int b) {
  ScaleRule r;
  r.len = len;
  const double inv = 1.0 / (double)len;
  r.inv_len = (float)inv;
  r.inv_len_low = (float)(inv - (double)r.inv_len);
  r.levels = (b == 1 || b == 32) ? 1.f : (float)((1 << (b - 1)) - 1);
  r.inv_levels = 1.f / r.levels;
  return r;
}

}  // namespace lpc
