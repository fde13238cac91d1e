/* The steps of the device generator's square root (neg_sqrt_neg_x2 in
 * paper_2603_20966_gb300/csrc/sk_rng.cuh) in C with explicit fmaf and IEEE
 * single-precision rounding, on every radicand the Box-Muller step can
 * produce (u = 2 ln u1, u1 = j 2^-24, j = 1 .. 2^24), from the correctly
 * rounded reciprocal square root and from its neighbours, compared with the
 * IEEE square root.  Prints how many radicands miss their root from the rounded
 * seed, and from at least one of its neighbours. */
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

float orc_ln1(float x); /* the oracle's ln: the radicands are -2 ln u1 */

static float u2f(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static uint32_t f2u(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }

static float neg_sqrt_neg(float u, float y) {
  float ng = u * y;
  float h = 0.5f * y;
  float nd = fmaf(ng, ng, u);
  return fmaf(nd, h, ng);
}

int main(void) {
  long bad = 0, bad_near = 0;
  for (uint32_t j = 1; j <= (1u << 24); ++j) {
    float u = 2.0f * orc_ln1((float)j * 0x1p-24f);
    if (u == 0.0f) u = 0.0f; /* u1 = 1: +0 on the device */
    float want = u == 0.0f ? 0.0f : -sqrtf(-u);
    float rn = (float)(1.0 / sqrt((double)fmaxf(-u, 1e-30f)));
    if (f2u(neg_sqrt_neg(u, rn)) != f2u(want)) ++bad;
    if (f2u(neg_sqrt_neg(u, u2f(f2u(rn) - 1))) != f2u(want) ||
        f2u(neg_sqrt_neg(u, u2f(f2u(rn) + 1))) != f2u(want))
      ++bad_near;
  }
  printf("rounded seed %ld neighbours %ld\n", bad, bad_near);
  return 0;
}
