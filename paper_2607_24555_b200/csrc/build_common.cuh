// Parameters and arithmetic shared by the summary-build kernels (build.cu: bulk; build_page.cu: the pages that a decode step
// has just filled).
#pragma once
#include "locks_internal.cuh"

struct BuildParams {
  const void *k;
  int64_t sb, sh, st;
  const int32_t *block_table;
  const int32_t *seq_lens;
  const int32_t *page_begin, *page_end;
  uint8_t *summ;
  int32_t *status;
  int batch, Hkv, Pmax, num_blocks, r, S;
  int fmt, esz;            // LOCKS_FMT_*, bytes per cache element (build_page.cu)
  // decode step only: where to leave the scan-partition suggestion for these lengths, and the scan's geometry
  int32_t *hint;
  int kpages, hint_wpp, hint_rounds, hint_W;
  // decode step only: the token appended by this step is read from the caller's buffer, not from the cache
  // (the append runs in another kernel at the same time); append_pos[b] = its position or -1
  const void *k_new;
  const int32_t *append_pos;
  // decode step whose build starts beside the scan, before any length is published: the token is counted here (seq_inc = 1),
  // and the caller's length is stored by whoever comes last of the request's page-heads, which have read it by then, and the
  // selector (arrivals[b] counts them; zero between steps).  seq_commit == nullptr: seq_lens are the step's.
  int32_t *seq_commit, *arrivals;
  // the same build: a summary that is ready before the step's scores are waits in stage[page-head] (S bytes each), since another
  // request may hold the page's block.  staged[page-head] counts the page-head and the selector, which comes when the scan is over;
  // the second of them puts the summary in place and leaves a zero.  stage == nullptr: the scan is over, summaries go in place.
  uint8_t *stage;
  int32_t *staged;
  // bulk build of several layers in one launch: per-layer key caches and summary buffers (device arrays), or null
  const void *const *k_layers;
  void *const *summ_layers;
};

// The pages that a decode step has just filled.  Adds its launch to c->last_launches.
int locks_launch_build_pages(locks_ctx *c, const BuildParams &p, cudaStream_t st);

#define LOCKS_BUILD_COS_TOL 1e-3f   // a Jacobi sweep that met no pair above this |cosine| was the last (it left them near 1e-6: quadratic convergence)
#define LOCKS_BUILD_SWEEPS 16       // upper bound (twice that for 32- and 64-token pages)

#ifdef __CUDACC__
// code = clamp(rint(x / scale)); `inv` = 1 / scale correctly rounded (0 for a zero scale: all codes 0).  The
// product differs from the quotient by at most an ulp, which matters only within an ulp of a rounding boundary.
__device__ __forceinline__ float inv_scale(float scale) { return scale == 0.f ? 0.f : __frcp_rn(scale); }
__device__ __forceinline__ float round_code(float x, float inv, float qmax) {
  return fminf(fmaxf(rintf(x * inv), -qmax), qmax);
}

// packed fp32 pairs (two independent lanes of arithmetic per instruction)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(*reinterpret_cast<unsigned long long *>(&d))
      : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)),
        "l"(*reinterpret_cast<unsigned long long *>(&c)));
  return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(*reinterpret_cast<unsigned long long *>(&d))
      : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
  return d;
}

// The plane rotation that makes two columns p, q orthogonal, from a = |p|^2, b = |q|^2, g = p . q (smaller angle):
// with d = |b - a| and h = d^2 + 4 g^2, cos 2x = d / sqrt(h) and sin 2x = 2 g / sqrt(h) (with the sign of b - a), so
// c = sqrt((1 + cos 2x) / 2), s = sin 2x / (2 c) and t = s / c: two reciprocal square roots in a row (approximate ones
// are enough for the angle; c^2 + s^2 = 1 holds to their rounding).  p' = c p - s q, q' = s p + c q, |p'|^2 = a - t g,
// |q'|^2 = b + t g.  Matrices come at unit scale; the 1e-18 makes equal, orthogonal columns an identity rotation and is
// below the rounding of any norm that counts.
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void jacobi_angle(float a, float b, float g, float &c, float &sn, float &tn) {
  const float d = b - a, ad = fabsf(d) + 1e-18f, g2 = g + g;
  const float rs = rsqrt_approx(fmaf(g2, g2, ad * ad));
  const float x = fmaf(0.5f * ad, rs, 0.5f), r2 = rsqrt_approx(x);
  const float u = __uint_as_float(__float_as_uint(g * rs) ^ (__float_as_uint(d) & 0x80000000u));
  c = x * r2;
  sn = u * r2;
  tn = sn * r2;
}
#endif
