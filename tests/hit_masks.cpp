// Random splats against the tile's pixels: blocks that a mask leaves out although
// a pixel of theirs would blend the splat. Arguments: least and largest major
// sigma (pixels), splats. Prints blending blocks, blocks left out, masked blocks.
#include "gsr_hit.h"

#include <cstdio>
#include <cstdlib>
#include <random>

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  const double s0 = atof(argv[1]), s1 = atof(argv[2]);
  const long n = atol(argv[3]);
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  long hits = 0, missed = 0, masked = 0;
  for (long i = 0; i < n; ++i) {
    const double major = s0 * std::pow(s1 / s0, U(rng)), minor = 0.55 + 1.45 * U(rng), th = M_PI * U(rng);
    const double c = std::cos(th), s = std::sin(th), v0 = major * major, v1 = minor * minor;
    // covariance and conic in binary32, as the shading pass forms them
    const float ca = (float)(c * c * v0 + s * s * v1), cb = (float)(c * s * (v0 - v1)), cc = (float)(s * s * v0 + c * c * v1);
    const float bb = cb * cb, e = fmaf(-cb, cb, bb), f = fmaf(ca, cc, -bb), inv = 1.0f / (f + e);
    const float A = cc * inv, B = -cb * inv, C = ca * inv;
    // a tile that the splat may cross: the centre up to 3 sigma away along the axis, a little beside it
    const double along = 3.0 * major * (2.0 * U(rng) - 1.0), beside = 3.0 * minor * (2.0 * U(rng) - 1.0);
    const float x = (float)(16.0 * U(rng) + along * c - beside * s), y = (float)(16.0 * U(rng) + along * s + beside * c);
    const float o = (float)(0.05 + 0.94 * U(rng));
    const uint32_t mask = gsr::warp_hit_mask(make_float4(x, y, A, B), C, gsr::floor_threshold(o));
    for (int w = 0; w < gsr::kWarps; ++w) {
      bool blends = false;
      for (int k = 0; k < 32 && !blends; ++k) {
        const float px = 8 * (w & 1) + (k & 7) + 0.5f, py = 4 * (w >> 1) + (k >> 3) + 0.5f;
        const float p = gsr::gs_power(A, B, C, x - px, y - py);
        blends = !(p > 0.0f) && !(o * std::exp(p) < 1.0f / 255.0f);
      }
      hits += blends;
      missed += blends && !(mask >> w & 1u);
      masked += mask >> w & 1u;
    }
  }
  std::printf("%ld %ld %ld\n", hits, missed, masked);
  return 0;
}
