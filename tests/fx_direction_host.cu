// Host program of test_fx_direction.py: fx_direction (su3_fx_kp.cuh, the device's own function) on projections whose
// largest component is at or next to a power of two, against long double.  Prints the largest error of a direction
// in units of 2^-53, and of |2r| times its reciprocal.
#include <cmath>
#include <cstdio>

#include "su3_fx_kp.cuh"

using namespace su3dev;
typedef long double Q;

static Q value(const fx& a) { return std::ldexp((Q)a.h, -30) + std::ldexp((Q)a.l, -62); }

int main() {
  Q dir = 0, length = 0;
  const long long off[] = {0, 1, -1, 2, 127, -128, 1LL << 20, -(1LL << 20), 3LL << 28, -(3LL << 28)};
  for (int s = 0; s < 62; ++s)
    for (int axis = 0; axis < 4; ++axis)
      for (long long d : off)
        for (int sign = -1; sign <= 1; sign += 2)
          for (int side = 0; side < 3; ++side) {  // the other components: none, one by one part in 2^16, in 2^10
            long long r[4] = {0, 0, 0, 0};
            if ((1LL << s) + d <= 0) continue;
            r[axis] = sign * ((1LL << s) + d);
            if (side) r[(axis + 1) & 3] = (side == 1 ? 1LL << s >> 16 : -(1LL << s >> 10));
            Q k = 0;
            for (long long c : r) k += (Q)c * c;
            k = std::sqrt(k);
            fx v[4];
            double ik;
            if (!fx_direction(r, v, &ik)) {
              std::printf("a direction was refused\n");
              return 1;
            }
            for (int c = 0; c < 4; ++c) dir = std::fmax(dir, std::fabs(value(v[c]) - r[c] / k) * std::ldexp((Q)1, 53));
            length = std::fmax(length, std::fabs(ik * std::ldexp(k, -58) - 1) * std::ldexp((Q)1, 53));
          }
  std::printf("direction %.3Lf length %.3Lf\n", dir, length);
  return 0;
}
