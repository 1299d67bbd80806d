// Summary build (Sec. 4 "Build (once, when a page completes)"), bulk, 16-token pages (build_page.cu has the rest).
//
// One warp takes 8 (page, KV head) items through three phases:
//   1. per item, all lanes: centre the page's 16 keys and form the Gram matrix M = D D^T (16 x 16) on the tensor cores; M
//      goes to shared memory
//   2. all 8 items at once: eigendecomposition of M by one-sided Jacobi in fp32.  Four lanes hold one item's matrix (4
//      columns of 16 entries each, in registers).  A QR factorisation with column pivoting comes first; the columns of
//      R^T are then rotated in pairs until they are mutually orthogonal: column norms are the eigenvalues, normalised
//      columns the eigenvectors.
//   3. per item, all lanes: modes above the zero-mode thresholds, V = D^T U_r Sigma_r^-1, C = U_r Sigma_r, sign: largest
//      |V| entry positive; store or quantise: symmetric abs-max, fp16 scale, round-half-even codes (int4 basis per column,
//      int8 coefficients per row, int8 centroid) packed in the blob layout
// build_i4_kernel: bf16 keys, int4 summaries.  build_kernel: everything else (fp32 keys, the other formats).
//
// Bound by instruction issue and its latencies, not by bytes: an eigenproblem per 4 KB page.  131 008 page-heads of 8 x 32K
// tokens: 1347 us with 8.2 Jacobi sweeps and all phases through shared memory (6 960 warp instructions per page-head), 908
// us with the factorisation in front (5.0 sweeps) and build_i4_kernel's phases 1 and 3 (3 930), 870 us with every pair
// rotated in one lane, by shears.  10 CTAs of 96 registers per SM instead of 8 of 128: 957 us (spills).
#include "build_common.cuh"

namespace {

constexpr int kBuildWarps = 2;
constexpr int kBuildItems = 8;                                   // (page, KV head) items per warp
constexpr int kBuildCtasPerSm = 8;                               // 16 warps per SM
constexpr int kBuildScratch = 2 * LOCKS_B * 128;                 // 4096 B: bf16 half-tiles of D (hi | lo); later the blob
constexpr int kMat = LOCKS_B * LOCKS_B + 16;                     // floats per item's matrix: items on different banks
constexpr int kBuildMat = kBuildItems * kMat * 4;                // 8704 B: Gram matrices, then R^T, then the leading eigenvectors
constexpr int kBuildSmemPerWarp = kBuildScratch + kBuildMat + 64 + kBuildItems * LOCKS_B * 4;   // + key norms, eigenvalues
constexpr int kUs = 20;                                          // build_i4_kernel: floats per eigenvector
constexpr int kPiv = 2 * kBuildItems * LOCKS_B;                  // floats: pivot columns of two steps; later an item's centroid
constexpr int kBuildI4SmemPerWarp = kPiv * 4 + kBuildMat + kBuildItems * LOCKS_B * 4;

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One-sided Jacobi on 8 matrices at once.  Lane (item = lane / 4, j = lane % 4) holds columns 4 j .. 4 j + 3 of its item's
// matrix W, w[c][i] = rows 2i, 2i+1 of column 4 j + c as a packed pair, and their squared norms: two pairs of columns.
// Odd-even transposition (16 steps per sweep meet every two columns once): every step rotates all pairs and passes one
// column of each to a neighbour, half of the time within the lane.
// W starts as R^T of M's QR factorisation with column pivoting (modified Gram-Schmidt, only R kept: Drmac and Veselic's
// preconditioning; R^T's left singular vectors are M's eigenvectors): half a sweep's work that saves three of eight
// (emulated in fp32 on this repository's synthetic pages, worst of 8 items: 8.2 -> 5.0 sweeps; the worst eigenvector
// entry falls from 1.1e-4 to 3.5e-5 from fp64).
// Result: the columns ranked by norm (descending, ties to the lower position), the 16 eigenvalues to lam_s[item][mode],
// unit eigenvectors of the leading min(r, 8) modes to us: PAIRS = false us[item][mode][token], kUs floats per mode; PAIRS =
// true [item][token][mode] as pairs (u, u) (r > 8: all 16, plain entries, [token][16]).
template <bool PAIRS>
__device__ __forceinline__ void jacobi_phase(float *mat, float *piv, float *us, float *lam_s, uint32_t live, int r, int lane) {
  constexpr int CPL = 4, LPI = LOCKS_B / CPL;
  const int item = lane / LPI, j = lane % LPI;
  const bool item_live = (live >> item) & 1u;   // lanes of an absent item compute on zeros
  float *mine = mat + item * kMat;
  float2 w[CPL][8];
  auto load = [&](bool live_item) {
    const float4 *src = reinterpret_cast<const float4 *>(mine + CPL * j * LOCKS_B);
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        const float4 f = live_item ? src[c * 4 + q4] : make_float4(0.f, 0.f, 0.f, 0.f);
        w[c][2 * q4] = make_float2(f.x, f.y);
        w[c][2 * q4 + 1] = make_float2(f.z, f.w);
      }
  };
  load(item_live);
  auto seg_max = [&](float v) {   // maximum over the lanes of the item
#pragma unroll
    for (int o = 1; o < LPI; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  };
  // The rotations square matrix entries: bring the matrix to unit scale first (an exact power of two, taken
  // from its largest entry and undone on the eigenvalues), so that keys of any magnitude are handled alike.
  float unscale = 1.f;
  {
    float amax = 0.f;
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
      for (int i = 0; i < 8; ++i) amax = fmaxf(amax, fmaxf(fabsf(w[c][i].x), fabsf(w[c][i].y)));
    amax = seg_max(amax);
    if (amax > 0.f && amax < INFINITY) {
      int ex;
      (void)frexpf(amax, &ex);
      ex = max(-120, min(120, ex));
      const float sc = ldexpf(1.f, -ex);
      unscale = ldexpf(1.f, ex);
      const float2 sc2 = make_float2(sc, sc);
#pragma unroll
      for (int c = 0; c < CPL; ++c)
#pragma unroll
        for (int i = 0; i < 8; ++i) w[c][i] = mul2(w[c][i], sc2);
    }
  }
  float n[CPL];
  auto norms = [&]() {
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc = fma2(w[c][i], w[c][i], acc);
      n[c] = acc.x + acc.y;
    }
  };
  auto dot = [&](const float2 (&a)[8], const float2 (&b)[8]) {
    float2 acc0 = mul2(a[0], b[0]), acc1 = mul2(a[1], b[1]);
#pragma unroll
    for (int i = 2; i < 8; i += 2) { acc0 = fma2(a[i], b[i], acc0); acc1 = fma2(a[i + 1], b[i + 1], acc1); }
    return (acc0.x + acc1.x) + (acc0.y + acc1.y);
  };
  norms();
  // ---- QR with column pivoting.  The norms that choose the pivot are downdated; the pivot's own is exact.
  {
    uint32_t used = 0u;
#pragma unroll 1
    for (int k = 0; k < LOCKS_B; ++k) {
      // largest remaining column: the norm's bits with the column in the lowest four; + 16 so that 0 means "used"
      uint32_t best = 0u;
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const uint32_t key = ((__float_as_uint(fmaxf(n[c], 0.f)) & ~15u) + 16u) | (uint32_t)(CPL * j + c);
        best = max(best, ((used >> c) & 1u) ? 0u : key);
      }
      best = max(best, __shfl_xor_sync(0xffffffffu, best, 1));
      best = max(best, __shfl_xor_sync(0xffffffffu, best, 2));
      float4 *pb = reinterpret_cast<float4 *>(piv + ((k & 1) * kBuildItems + item) * LOCKS_B);
      const int pc = (int)(best & 15u) - CPL * j;   // this lane's column of that number, if 0 .. 3
#pragma unroll
      for (int c = 0; c < CPL; ++c)
        if (c == pc) {
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) pb[q4] = make_float4(w[c][2 * q4].x, w[c][2 * q4].y, w[c][2 * q4 + 1].x, w[c][2 * q4 + 1].y);
        }
      __syncwarp();   // (the buffer of step k - 1 is not written before every lane has passed here)
      float2 pv[8];
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        const float4 f = pb[q4];
        pv[2 * q4] = make_float2(f.x, f.y);
        pv[2 * q4 + 1] = make_float2(f.z, f.w);
      }
      const float pp = dot(pv, pv), ir = pp > 1e-37f ? rsqrt_approx(pp) : 0.f;
      float rk[CPL];
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        rk[c] = ((used >> c) & 1u) ? 0.f : (c == pc ? pp : dot(w[c], pv)) * ir;
        const float f = -rk[c] * ir;
        const float2 f2 = make_float2(f, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) w[c][i] = fma2(f2, pv[i], w[c][i]);
        n[c] = fmaf(-rk[c], rk[c], n[c]);
      }
      if (pc >= 0 && pc < CPL) used |= 1u << pc;
      *reinterpret_cast<float4 *>(mine + k * LOCKS_B + CPL * j) = make_float4(rk[0], rk[1], rk[2], rk[3]);   // column k of R^T
    }
    __syncwarp();
    load(true);
  }
  // The stop test: no pair above the tolerance in a whole sweep.  With few modes kept only pairs with one of the r largest
  // columns count (r = 2: 5.4 -> 3.3 sweeps); with 8 the others add a fifth of a sweep, less than finding the r-th norm.
  const float tol = r >= 8 ? 3.f * LOCKS_BUILD_COS_TOL : LOCKS_BUILD_COS_TOL, tol2 = tol * tol;
  int bad = 0;
  float floor_n = 0.f, top = 0.f;
  int rank[CPL];
  auto ranks = [&]() {
#pragma unroll
    for (int c = 0; c < CPL; ++c) rank[c] = 0;
#pragma unroll
    for (int jj = 0; jj < LPI; ++jj)
#pragma unroll
      for (int cc = 0; cc < CPL; ++cc) {
        const float o = __shfl_sync(0xffffffffu, n[cc], (lane & ~(LPI - 1)) + jj);
#pragma unroll
        for (int c = 0; c < CPL; ++c) rank[c] += (int)(o > n[c]) | ((int)(o == n[c]) & (int)(jj * CPL + cc < j * CPL + c));
      }
  };
  // A pair holds a column that it kept from the step before (a) and one that it has been passed (b).  Which of the two is the
  // lower position alternates from step to step, and so do the signs of the rotation and of the swap that follows it,
  // which leaves one formula: passed on c a + s b (in a), kept c b - s a (in b).
  struct Angle { float c, s; };
  auto angle = [&](const float2 (&a)[8], const float2 (&b)[8], float &na, float &nb, bool there) {
    const float g = dot(a, b);
    // columns whose norm is rounding noise beside the largest (null directions) do not hold up convergence
    bad |= (int)there & (int)(g * g > tol2 * na * nb) & (int)(fminf(na, nb) > floor_n) & (int)(fmaxf(na, nb) >= top);
    Angle r;
    float tn;
    jacobi_angle(nb, na, g, r.c, r.s, tn);
    tn = there ? tn * g : nb - na;   // (no pair: the two change places)
    na = fmaxf(na + tn, 0.f);
    nb = fmaxf(nb - tn, 0.f);
    return r;
  };
  // as three shears (tau = tan(angle / 2) = s / (1 + c)): three packed operations per row instead of four
  auto rotate = [&](float2 (&a)[8], float2 (&b)[8], float &na, float &nb) {
    const Angle r = angle(a, b, na, nb, true);
    const float tau = r.s * rcp_approx(1.f + r.c);
    const float2 T2 = make_float2(tau, tau), S2 = make_float2(-r.s, -r.s);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      a[i] = fma2(T2, b[i], a[i]);
      b[i] = fma2(S2, a[i], b[i]);
      a[i] = fma2(T2, b[i], a[i]);
    }
  };
  const int up = (lane & ~(LPI - 1)) | ((j + 1) & (LPI - 1)), down = (lane & ~(LPI - 1)) | ((j - 1) & (LPI - 1));
  for (int sweep = 0; sweep < LOCKS_BUILD_SWEEPS; ++sweep) {
    norms();
    {
      float nm = n[0];
#pragma unroll
      for (int c = 1; c < CPL; ++c) nm = fmaxf(nm, n[c]);
      floor_n = 1e-11f * seg_max(nm);   // squared norm = squared eigenvalue: modes below 3e-6 of the largest
    }
    if (r < 8) {
      ranks();
      float least = INFINITY;
#pragma unroll
      for (int c = 0; c < CPL; ++c) least = rank[c] < r ? fminf(least, n[c]) : least;
      top = -0.999f * seg_max(-least);
    }
    bad = 0;
#pragma unroll 2
    for (int st2 = 0; st2 < 8; ++st2) {
      // even step: the lane's pairs (w[1], w[0]) and (w[3], w[2])
      rotate(w[1], w[0], n[1], n[0]);
      rotate(w[3], w[2], n[3], n[2]);
      // a pair passes to the one before it: w[3] to w[0]'s, w[1] to the lane below
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        w[1][i].x = __shfl_sync(0xffffffffu, w[1][i].x, up);
        w[1][i].y = __shfl_sync(0xffffffffu, w[1][i].y, up);
      }
      n[1] = __shfl_sync(0xffffffffu, n[1], up);
      // odd step: (w[0], w[3]) and (w[2], w[1]); the item's last pair has the two ends of the row, which do not meet
      rotate(w[0], w[3], n[0], n[3]);
      {
        Angle r = angle(w[2], w[1], n[2], n[1], j != LPI - 1);
        if (j == LPI - 1) { r.c = 0.f; r.s = 1.f; }
        const float2 C2 = make_float2(r.c, r.c), S2 = make_float2(r.s, r.s), nS2 = make_float2(-r.s, -r.s);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 a = fma2(C2, w[2][i], mul2(S2, w[1][i]));
          w[1][i] = fma2(C2, w[1][i], mul2(nS2, w[2][i]));
          w[2][i].x = __shfl_sync(0xffffffffu, a.x, down);   // a pair passes to the one after it: w[0] to w[1]'s, w[2] to the lane above
          w[2][i].y = __shfl_sync(0xffffffffu, a.y, down);
        }
        n[2] = __shfl_sync(0xffffffffu, n[2], down);
      }
      // the lane's pairs are now (w[3], w[2]) and (w[1], w[0]), in this order: exchange the names
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int i = 0; i < 8; ++i) { const float2 y = w[c][i]; w[c][i] = w[c + 2][i]; w[c + 2][i] = y; }
        const float y = n[c];
        n[c] = n[c + 2];
        n[c + 2] = y;
      }
    }
    if (!__any_sync(0xffffffffu, bad != 0)) break;
  }
  norms();
  ranks();
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    lam_s[item * LOCKS_B + rank[c]] = sqrtf(n[c]) * unscale;
    const float inv = n[c] > 0.f ? rsqrtf(n[c]) : 0.f;
    if (!PAIRS) {
      if (rank[c] < 8) {
        float4 *dst = reinterpret_cast<float4 *>(us + (item * 8 + rank[c]) * kUs);
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4)
          dst[q4] = make_float4(w[c][2 * q4].x * inv, w[c][2 * q4].y * inv, w[c][2 * q4 + 1].x * inv, w[c][2 * q4 + 1].y * inv);
      }
    } else if (r > 8) {   // ranks above 8 (fp32 summaries): all 16 modes, plain entries
      float *dst = us + item * LOCKS_B * LOCKS_B + rank[c];
#pragma unroll
      for (int i = 0; i < 8; ++i) { dst[(2 * i) * LOCKS_B] = w[c][i].x * inv; dst[(2 * i + 1) * LOCKS_B] = w[c][i].y * inv; }
    } else if (rank[c] < 8) {
      float2 *dst = reinterpret_cast<float2 *>(us) + item * LOCKS_B * 8 + rank[c];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float u0 = w[c][i].x * inv, u1 = w[c][i].y * inv;
        dst[(2 * i) * 8] = make_float2(u0, u0);
        dst[(2 * i + 1) * 8] = make_float2(u1, u1);
      }
    }
  }
  __syncwarp();
}

// Physical block of item `lane` (< 8) of this warp, -1 if there is none; page ranges as locks_build_summaries has them.
__device__ __forceinline__ int item_block(const BuildParams &p, int warp, int lane) {
  if (lane >= kBuildItems) return -1;
  const int b = blockIdx.z % p.batch;
  const int complete = p.seq_lens[b] / LOCKS_B;
  const int p0 = p.page_begin ? p.page_begin[b] : 0;
  const int p1 = min(p.page_end ? p.page_end[b] : complete, complete);
  const int page = p0 + (blockIdx.x * kBuildWarps + warp) * kBuildItems + lane;
  if (page < 0 || page >= p1 || page >= p.Pmax) return -1;
  const int block = p.block_table[(int64_t)b * p.Pmax + page];
  if (block >= 0 && block < p.num_blocks) return block;
  set_status(p.status, LOCKS_ERR_BAD_BLOCK);
  return -1;
}

__device__ __forceinline__ uint32_t bf16x2_add(uint32_t a, uint32_t b) {
  const __nv_bfloat162 d = __hadd2_rn(*reinterpret_cast<__nv_bfloat162 *>(&a), *reinterpret_cast<__nv_bfloat162 *>(&b));
  return *reinterpret_cast<const uint32_t *>(&d);
}
__device__ __forceinline__ uint32_t bf16x2_sub(uint32_t a, uint32_t b) {
  const __nv_bfloat162 d = __hsub2_rn(*reinterpret_cast<__nv_bfloat162 *>(&a), *reinterpret_cast<__nv_bfloat162 *>(&b));
  return *reinterpret_cast<const uint32_t *>(&d);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(*reinterpret_cast<unsigned long long *>(&d))
      : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
  return d;
}
// fp16 scale of codes -qmax .. qmax for values up to `best`, and its reciprocal (0 for a zero scale: all codes 0)
__device__ __forceinline__ __half code_scale(float best, float inv_qmax, float &inv) {
  const __half s = __float2half_rn(best * inv_qmax);
  const float f = __half2float(s);
  inv = f == 0.f ? 0.f : rcp_approx(f);
  return s;
}

// bf16 keys, int4 summaries.  Neither phase 1 nor phase 3 touches shared memory for the keys: a lane loads from global
// memory the 16-byte chunks that are its own MMA fragments (any assignment of dimensions to fragment positions will do in
// phase 1, where they are summed over; in phase 3 it decides which dimensions of the basis a lane receives).
//   Phase 1: the keys minus c = bf16(mean) split exactly into two bf16 terms H + L (Knuth's TwoSum in bf16 pairs), M' =
//   (H + L)(H + L)^T, and M = M' centred in both directions (c is not quite the mean).
//   Phase 3: V Sigma = U^T D = (U - mean U)^T K, U in three bf16 terms (24 bits, rows 0-7 and 8-15 of one A operand and rows
//   0-7 of another whose rows 8-15 are 1/16 and give the centroid), K as stored: products exact, sums fp32.
__global__ void __launch_bounds__(kBuildWarps * 32, kBuildCtasPerSm) build_i4_kernel(BuildParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x = lane >> 2, t = lane & 3, h = blockIdx.y, r = p.r;
  const int it_block = item_block(p, warp, lane);
  const uint32_t live = __ballot_sync(0xffffffffu, it_block >= 0);
  if (!live) return;
  const int layer = blockIdx.z / p.batch;
  const __nv_bfloat16 *kbase = reinterpret_cast<const __nv_bfloat16 *>(p.k_layers ? p.k_layers[layer] : p.k);
  uint8_t *sbase = p.summ_layers ? reinterpret_cast<uint8_t *>(p.summ_layers[layer]) : p.summ;
  float *piv = reinterpret_cast<float *>(smem_raw + warp * kBuildI4SmemPerWarp), *mat = piv + kPiv, *lam_s = mat + kBuildItems * kMat;
  auto page_keys = [&](int s) {
    return kbase + (int64_t)__shfl_sync(0xffffffffu, it_block, s) * p.sb + (int64_t)h * p.sh;
  };

  // ---- 1. Gram matrices: lane (x, t) holds dimensions 8t .. 8t+7 (+ 32 j) of tokens x and x + 8
#pragma unroll 1
  for (int s = 0; s < kBuildItems; ++s) {
    if (!((live >> s) & 1u)) continue;
    const __nv_bfloat16 *K = page_keys(s) + (int64_t)x * p.st + 8 * t;
    uint32_t ka[16], kb[16], nc[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 a = *reinterpret_cast<const uint4 *>(K + 32 * j), b = *reinterpret_cast<const uint4 *>(K + 8 * p.st + 32 * j);
      ka[4 * j] = a.x; ka[4 * j + 1] = a.y; ka[4 * j + 2] = a.z; ka[4 * j + 3] = a.w;
      kb[4 * j] = b.x; kb[4 * j + 1] = b.y; kb[4 * j + 2] = b.z; kb[4 * j + 3] = b.w;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) nc[i] = bf16x2_add(ka[i], kb[i]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
      for (int i = 0; i < 16; ++i) nc[i] = bf16x2_add(nc[i], __shfl_xor_sync(0xffffffffu, nc[i], o));
    float X0[4] = {0.f, 0.f, 0.f, 0.f}, X1[4] = {0.f, 0.f, 0.f, 0.f}, Y0[4] = {0.f, 0.f, 0.f, 0.f}, Y1[4] = {0.f, 0.f, 0.f, 0.f};
    auto split = [&](uint32_t k, uint32_t n, uint32_t &hi, uint32_t &lo) {   // k + n = hi + lo exactly
      hi = bf16x2_add(k, n);
      const uint32_t bb = bf16x2_sub(hi, k);
      lo = bf16x2_add(bf16x2_sub(k, bf16x2_sub(hi, bb)), bf16x2_sub(n, bb));
    };
#pragma unroll
    for (int i = 0; i < 16; i += 2) {   // one k-step: registers i, i + 1 of both tokens are the A and the B operand
      uint32_t H[4], L[4];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const __nv_bfloat162 m = __hmul2(*reinterpret_cast<__nv_bfloat162 *>(&nc[i + u]), __floats2bfloat162_rn(-1.f / LOCKS_B, -1.f / LOCKS_B));
        const uint32_t n = *reinterpret_cast<const uint32_t *>(&m);
        split(ka[i + u], n, H[2 * u], L[2 * u]);
        split(kb[i + u], n, H[2 * u + 1], L[2 * u + 1]);
      }
      mma_bf16(X0, H[0], H[1], H[2], H[3], H[0], H[2]);
      mma_bf16(X1, H[0], H[1], H[2], H[3], H[1], H[3]);
      mma_bf16(Y0, H[0], H[1], H[2], H[3], L[0], L[2]);
      mma_bf16(Y1, H[0], H[1], H[2], H[3], L[1], L[3]);
      mma_bf16(X0, L[0], L[1], L[2], L[3], L[0], L[2]);
      mma_bf16(X1, L[0], L[1], L[2], L[3], L[1], L[3]);
      mma_bf16(Y0, L[0], L[1], L[2], L[3], H[0], H[2]);
      mma_bf16(Y1, L[0], L[1], L[2], L[3], H[1], H[3]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) { X0[i] += Y0[i]; X1[i] += Y1[i]; }   // [0..1]: row x, columns 2t, 2t+1 (X1: + 8); [2..3]: row x + 8
    float r0 = (X0[0] + X0[1]) + (X1[0] + X1[1]), r1 = (X0[2] + X0[3]) + (X1[2] + X1[3]);
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) { r0 += __shfl_xor_sync(0xffffffffu, r0, o); r1 += __shfl_xor_sync(0xffffffffu, r1, o); }
    r0 *= 1.f / LOCKS_B;   // means of rows x and x + 8; by symmetry also of those columns
    r1 *= 1.f / LOCKS_B;
    float c0 = __shfl_sync(0xffffffffu, r0, 8 * t), c1 = __shfl_sync(0xffffffffu, r0, 8 * t + 4);
    float c8 = __shfl_sync(0xffffffffu, r1, 8 * t), c9 = __shfl_sync(0xffffffffu, r1, 8 * t + 4);
    float g = (c0 + c1) + (c8 + c9);
    g += __shfl_xor_sync(0xffffffffu, g, 1);
    g += __shfl_xor_sync(0xffffffffu, g, 2);
    g *= 1.f / LOCKS_B;
    r0 -= g;
    r1 -= g;
    float *dst = mat + s * kMat + x * LOCKS_B + 2 * t;
    *reinterpret_cast<float2 *>(dst) = make_float2(X0[0] - (r0 + c0), X0[1] - (r0 + c1));
    *reinterpret_cast<float2 *>(dst + 8) = make_float2(X1[0] - (r0 + c8), X1[1] - (r0 + c9));
    *reinterpret_cast<float2 *>(dst + 8 * LOCKS_B) = make_float2(X0[2] - (r1 + c0), X0[3] - (r1 + c1));
    *reinterpret_cast<float2 *>(dst + 8 * LOCKS_B + 8) = make_float2(X1[2] - (r1 + c8), X1[3] - (r1 + c9));
  }
  __syncwarp();

  // ---- 2. eigenvectors and eigenvalues of all the warp's items at once
  jacobi_phase<false>(mat, piv, mat, lam_s, live, r, lane);

  // ---- 3. basis, coefficients, centroid.  Lane (x, t) receives mode x, dimensions 16 t .. 16 t + 15 (+ 64)
#pragma unroll 1
  for (int s = 0; s < kBuildItems; ++s) {
    if (!((live >> s) & 1u)) continue;
    const __nv_bfloat16 *K = page_keys(s) + (int64_t)(2 * t) * p.st + 8 * x;
    uint4 kk[2][4];   // tokens 2t, 2t + 1, 2t + 8, 2t + 9; dimensions 8 x .. 8 x + 7 (+ 64)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int hc = 0; hc < 2; ++hc) kk[hc][i] = *reinterpret_cast<const uint4 *>(K + (int64_t)((i & 1) + 8 * (i >> 1)) * p.st + 64 * hc);
    const float *U = mat + s * 8 * kUs, *lam = lam_s + s * LOCKS_B;
    uint32_t A[4], Lo[2];
    {
      const float2 ua = *reinterpret_cast<const float2 *>(U + x * kUs + 2 * t), ub = *reinterpret_cast<const float2 *>(U + x * kUs + 8 + 2 * t);
      float m = (ua.x + ua.y) + (ub.x + ub.y);
      m += __shfl_xor_sync(0xffffffffu, m, 1);
      m += __shfl_xor_sync(0xffffffffu, m, 2);
      m *= 1.f / LOCKS_B;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        float a = (i ? ub.x : ua.x) - m, b = (i ? ub.y : ua.y) - m;
        if (x >= r) a = b = 0.f;
        A[2 * i] = pack_bf16(a, b);
        a -= __uint_as_float(A[2 * i] << 16);
        b -= __uint_as_float(A[2 * i] & 0xFFFF0000u);
        A[2 * i + 1] = pack_bf16(a, b);
        a -= __uint_as_float(A[2 * i + 1] << 16);
        b -= __uint_as_float(A[2 * i + 1] & 0xFFFF0000u);
        Lo[i] = pack_bf16(a, b);
      }
    }
    const uint32_t kOne = 0x3D803D80u;   // 1/16
    float2 v[2][8];   // [hc][j]: dimensions 64 hc + 16 t + j and + 8
    float *mu_s = piv;
#pragma unroll
    for (int hc = 0; hc < 2; ++hc) {
      float2 mu[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        auto word = [&](const uint4 &q) { return j < 2 ? q.x : (j < 4 ? q.y : (j < 6 ? q.z : q.w)); };
        const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
        const uint32_t b0 = __byte_perm(word(kk[hc][0]), word(kk[hc][1]), sel), b1 = __byte_perm(word(kk[hc][2]), word(kk[hc][3]), sel);
        float C1[4] = {0.f, 0.f, 0.f, 0.f}, C2[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(C1, A[0], A[1], A[2], A[3], b0, b1);
        mma_bf16(C2, Lo[0], kOne, Lo[1], kOne, b0, b1);
        v[hc][j] = add2(add2(make_float2(C2[0], C2[1]), make_float2(C1[2], C1[3])), make_float2(C1[0], C1[1]));
        mu[j] = make_float2(C2[2], C2[3]);
      }
      if (x == 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          *reinterpret_cast<float4 *>(mu_s + 64 * hc + 16 * t + 4 * q) = make_float4(mu[4 * q].x, mu[4 * q + 1].x, mu[4 * q + 2].x, mu[4 * q + 3].x);
          *reinterpret_cast<float4 *>(mu_s + 64 * hc + 16 * t + 8 + 4 * q) = make_float4(mu[4 * q].y, mu[4 * q + 1].y, mu[4 * q + 2].y, mu[4 * q + 3].y);
        }
      }
    }
    __syncwarp();
    uint8_t *gout = sbase + ((int64_t)__shfl_sync(0xffffffffu, it_block, s) * p.Hkv + h) * p.S;
    // ---- centroid: dimensions 4 lane .. + 3
    const float4 mu4 = *reinterpret_cast<const float4 *>(mu_s + 4 * lane);
    {
      const float mx = fmaxf(fmaxf(fabsf(mu4.x), fabsf(mu4.y)), fmaxf(fabsf(mu4.z), fabsf(mu4.w)));
      float inv;
      const __half sh = code_scale(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx))), 1.f / 127.f, inv);
      auto code = [&](float v) { return (uint32_t)((int)round_code(v, inv, 127.f) + 128); };
      // dim offset c = 2*half + e -> byte e*2 + half
      *reinterpret_cast<uint32_t *>(gout + i4_off_mu(r) + lane * 4) = code(mu4.x) | (code(mu4.z) << 8) | (code(mu4.y) << 16) | (code(mu4.w) << 24);
      if (lane == 0) *reinterpret_cast<__half *>(gout + i4_off_smu(r)) = sh;
      if (lane < 16 && i4_off_smu(r) + 2 + lane < p.S) gout[i4_off_smu(r) + 2 + lane] = 0;   // bytes between the payload and the stride
    }
    // ---- the mode's place among those above the zero-mode thresholds (eigenvalues descend: no gaps)
    const float knorm2 = warp_sum((float)LOCKS_B * (mu4.x * mu4.x + mu4.y * mu4.y + mu4.z * mu4.z + mu4.w * mu4.w) +
                                  (lane < LOCKS_B ? lam[lane] : 0.f));
    const float lam0 = lam[0], lx = lam[x];
    const bool keep = x < r && lam0 > 0.f && lx > 1e-6f * lam0 && lx > 1e-10f * knorm2;
    // ---- basis: largest magnitude and its sign (lowest dimension on ties)
    float mx = v[0][0].x, mn = v[0][0].x;
#pragma unroll
    for (int hc = 0; hc < 2; ++hc)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mx = fmaxf(mx, fmaxf(v[hc][j].x, v[hc][j].y));
        mn = fminf(mn, fminf(v[hc][j].x, v[hc][j].y));
      }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    }
    bool neg = -mn > mx;
    if (__any_sync(0xffffffffu, keep && mx == -mn)) {   // opposite entries of the same magnitude
      int at = LOCKS_D << 1;   // 2 * dimension + (negative)
#pragma unroll
      for (int hc = 1; hc >= 0; --hc)
#pragma unroll
        for (int i = 15; i >= 0; --i) {
          const float y = i < 8 ? v[hc][i & 7].x : v[hc][i & 7].y;
          if (fabsf(y) == mx) at = 2 * (64 * hc + 16 * t + i) + (y < 0.f ? 1 : 0);
        }
      at = min(at, __shfl_xor_sync(0xffffffffu, at, 1));
      at = min(at, __shfl_xor_sync(0xffffffffu, at, 2));
      if (mx == -mn) neg = at & 1;
    }
    const float isig = keep ? rsqrtf(lx) : 0.f;
    float inv;
    const __half sv = code_scale(fmaxf(mx, -mn) * isig, 1.f / 7.f, inv);
    inv *= neg ? -isig : isig;   // (a unit vector's largest entry is at least 0.088: the scale is a normal fp16, no code leaves -7 .. 7)
    // code + 8 in the low bits of 1.5 * 2^23 + code + 8; a word's nibbles from the top: dimensions 7 5 3 1 6 4 2 0
    if (x < r) {
#pragma unroll
      for (int hc = 0; hc < 2; ++hc) {
        uint32_t wx = 0u, wy = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int j = q < 4 ? 7 - 2 * q : 14 - 2 * q;
          wx = wx * 16u + __float_as_uint(fmaf(v[hc][j].x, inv, 12582920.f));
          wy = wy * 16u + __float_as_uint(fmaf(v[hc][j].y, inv, 12582920.f));
        }
        *reinterpret_cast<uint2 *>(gout + x * 64 + 32 * hc + 8 * t) = make_uint2(wx - 0x3F400000u, wy - 0x3F400000u);
      }
      if (t == 0) *reinterpret_cast<__half *>(gout + i4_off_sv(r) + 2 * x) = sv;
    }
    // ---- coefficients C = U Sigma: tokens x and x + 8, modes 2t and 2t + 1
    const float sg = keep ? (neg ? -sqrtf(lx) : sqrtf(lx)) : 0.f;
    const float g0 = __shfl_sync(0xffffffffu, sg, 8 * t), g1 = __shfl_sync(0xffffffffu, sg, 8 * t + 4);
    const float *Ut = U + 2 * t * kUs + x;
    const float ca = g0 * Ut[0], cb = g1 * Ut[kUs], cc = g0 * Ut[8], cd = g1 * Ut[kUs + 8];
    float ma = fmaxf(fabsf(ca), fabsf(cb)), mb = fmaxf(fabsf(cc), fabsf(cd));
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
      mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    }
    float ia, ib;
    const __half sa = code_scale(ma, 1.f / 127.f, ia), sb = code_scale(mb, 1.f / 127.f, ib);
    if (t < r / 2) {
      auto code = [&](float v, float inv) { return (uint32_t)((int)round_code(v, inv, 127.f) + 128); };
      *reinterpret_cast<uint32_t *>(gout + i4_off_coef(r) + (x * (r / 2) + t) * 4) =
          code(ca, ia) | (code(cb, ia) << 8) | (code(cc, ib) << 16) | (code(cd, ib) << 24);
    }
    if (t == 0) {
      __half *dst = reinterpret_cast<__half *>(gout + i4_off_sc(r)) + (x >> 1) * 4 + (x & 1);
      dst[0] = sa;
      dst[2] = sb;
    }
    __syncwarp();   // the centroid's shared memory is written again for the next item
  }
}

template <typename T, int FMT>
__global__ void __launch_bounds__(kBuildWarps * 32, kBuildCtasPerSm) build_kernel(BuildParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int h = blockIdx.y;
  const int it_block = item_block(p, warp, lane);   // the warp's items: lane s < 8 works out item s
  const uint32_t live = __ballot_sync(0xffffffffu, it_block >= 0);
  if (!live) return;

  const int layer = blockIdx.z / p.batch;
  const void *kbase = p.k_layers ? p.k_layers[layer] : p.k;
  uint8_t *sbase = p.summ_layers ? reinterpret_cast<uint8_t *>(p.summ_layers[layer]) : p.summ;
  uint8_t *scratch = smem_raw + warp * kBuildSmemPerWarp;                        // D half-tiles; phase 3: the blob
  float *mat = reinterpret_cast<float *>(scratch + kBuildScratch);              // [8][16][16] Gram; then [8][16][8] pairs (u, u) of U_r
  float *kn_s = mat + kBuildItems * kMat;                          // [8] squared norm of the page's keys
  float *lam_s = kn_s + 16;                                                     // [8][16] eigenvalues, descending
  float2 *us = reinterpret_cast<float2 *>(mat);
  const int r = p.r;

  // keys of item s: v[i][c] = key i, dim 4 lane + c, as fp32
  auto load_item = [&](int s, float (&v)[LOCKS_B][4]) {
    const int block = __shfl_sync(0xffffffffu, it_block, s);
    const T *K = reinterpret_cast<const T *>(kbase) + ((int64_t)block * p.sb + (int64_t)h * p.sh) + 4 * lane;
#pragma unroll
    for (int i = 0; i < LOCKS_B; ++i) {
      const T *src = K + (int64_t)i * p.st;
      if (sizeof(T) == 2) {
        const uint2 w = *reinterpret_cast<const uint2 *>(src);
        v[i][0] = __uint_as_float(w.x << 16); v[i][1] = __uint_as_float(w.x & 0xFFFF0000u);
        v[i][2] = __uint_as_float(w.y << 16); v[i][3] = __uint_as_float(w.y & 0xFFFF0000u);
      } else {
        const float4 w = *reinterpret_cast<const float4 *>(src);
        v[i][0] = w.x; v[i][1] = w.y; v[i][2] = w.z; v[i][3] = w.w;
      }
    }
  };
  auto centre = [&](float (&v)[LOCKS_B][4], float (&mu)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) mu[c] = 0.f;
#pragma unroll
    for (int i = 0; i < LOCKS_B; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) mu[c] += v[i][c];
#pragma unroll
    for (int c = 0; c < 4; ++c) mu[c] *= (1.f / LOCKS_B);
#pragma unroll
    for (int i = 0; i < LOCKS_B; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[i][c] -= mu[c];
  };

  // ---- 1. Gram matrices M = D D^T on the tensor cores.  D = H + L with H = bf16(D), L = bf16(D - H) (16 significant
  // bits; the bf16 products are exact and accumulate in fp32): M = (H H^T + L L^T) + H L^T + (H L^T)^T.  The A
  // operand (tokens x dims) and the B operand (dims x tokens) of an m16n8k16 step are the same registers.
  // Two passes over 64 dims each: the half-tiles of H and L (16 rows x 128 bytes, 16-byte chunks XOR-swizzled with
  // the row so that ldmatrix reads are conflict-free) share the 4 KB of scratch; in a pass the 16 lanes that own
  // the half's dims write it.
#pragma unroll 1
  for (int s = 0; s < kBuildItems; ++s) {
    if (!((live >> s) & 1u)) continue;
    uint32_t hl[LOCKS_B][4];   // h01, h23, l01, l23 of this lane's 4 dims, per key
    {
      float v[LOCKS_B][4], mu[4];
      load_item(s, v);
      float knorm2 = 0.f;
#pragma unroll
      for (int i = 0; i < LOCKS_B; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) knorm2 = fmaf(v[i][c], v[i][c], knorm2);
      knorm2 = warp_sum(knorm2);
      if (lane == 0) kn_s[s] = knorm2;
      centre(v, mu);
#pragma unroll
      for (int i = 0; i < LOCKS_B; ++i) {
        const uint32_t h01 = pack_bf16(v[i][0], v[i][1]), h23 = pack_bf16(v[i][2], v[i][3]);
        hl[i][0] = h01; hl[i][1] = h23;
        hl[i][2] = pack_bf16(v[i][0] - __uint_as_float(h01 << 16), v[i][1] - __uint_as_float(h01 & 0xFFFF0000u));
        hl[i][3] = pack_bf16(v[i][2] - __uint_as_float(h23 << 16), v[i][3] - __uint_as_float(h23 & 0xFFFF0000u));
      }
    }
    float X0[4] = {0.f, 0.f, 0.f, 0.f}, X1[4] = {0.f, 0.f, 0.f, 0.f}, Y0[4] = {0.f, 0.f, 0.f, 0.f}, Y1[4] = {0.f, 0.f, 0.f, 0.f};
    const int c16 = lane & 15;                                          // writer: dims 4 c16 .. + 3 of the half
    const int mq = lane >> 3, rr = lane & 7, tok = (mq & 1) * 8 + rr;   // reader (ldmatrix address lanes)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      if ((lane >> 4) == hf) {
#pragma unroll
        for (int row = 0; row < LOCKS_B; ++row) {
          uint8_t *dst = scratch + row * 128 + ((((c16 >> 1) ^ (row & 7)) << 4) | ((c16 & 1) << 3));
          *reinterpret_cast<uint2 *>(dst) = make_uint2(hl[row][0], hl[row][1]);
          *reinterpret_cast<uint2 *>(dst + 2048) = make_uint2(hl[row][2], hl[row][3]);
        }
      }
      __syncwarp();
#pragma unroll
      for (int s4 = 0; s4 < 4; ++s4) {
        uint32_t Hf[4], Lf[4];
        const uint8_t *src = scratch + tok * 128 + (((2 * s4 + (mq >> 1)) ^ (tok & 7)) << 4);
        ldsm_x4(Hf, src);
        ldsm_x4(Lf, src + 2048);
        mma_bf16(X0, Hf[0], Hf[1], Hf[2], Hf[3], Hf[0], Hf[2]);
        mma_bf16(X1, Hf[0], Hf[1], Hf[2], Hf[3], Hf[1], Hf[3]);
        mma_bf16(X0, Lf[0], Lf[1], Lf[2], Lf[3], Lf[0], Lf[2]);
        mma_bf16(X1, Lf[0], Lf[1], Lf[2], Lf[3], Lf[1], Lf[3]);
        mma_bf16(Y0, Hf[0], Hf[1], Hf[2], Hf[3], Lf[0], Lf[2]);
        mma_bf16(Y1, Hf[0], Hf[1], Hf[2], Hf[3], Lf[1], Lf[3]);
      }
      __syncwarp();
    }
    // accumulator (x = lane / 4, t = lane % 4): [0..1] = row x, columns 2t, 2t+1; [2..3] = row x + 8.
    // M = sym(X) + Y + Y^T, assembled through two padded 16 x 17 arrays in the (now free) scratch
    {
      float *XA = reinterpret_cast<float *>(scratch), *YA = XA + LOCKS_B * 17;
      const int x = lane >> 2, t = lane & 3;
      XA[x * 17 + 2 * t] = X0[0]; XA[x * 17 + 2 * t + 1] = X0[1]; XA[(x + 8) * 17 + 2 * t] = X0[2]; XA[(x + 8) * 17 + 2 * t + 1] = X0[3];
      XA[x * 17 + 8 + 2 * t] = X1[0]; XA[x * 17 + 9 + 2 * t] = X1[1]; XA[(x + 8) * 17 + 8 + 2 * t] = X1[2]; XA[(x + 8) * 17 + 9 + 2 * t] = X1[3];
      YA[x * 17 + 2 * t] = Y0[0]; YA[x * 17 + 2 * t + 1] = Y0[1]; YA[(x + 8) * 17 + 2 * t] = Y0[2]; YA[(x + 8) * 17 + 2 * t + 1] = Y0[3];
      YA[x * 17 + 8 + 2 * t] = Y1[0]; YA[x * 17 + 9 + 2 * t] = Y1[1]; YA[(x + 8) * 17 + 8 + 2 * t] = Y1[2]; YA[(x + 8) * 17 + 9 + 2 * t] = Y1[3];
      __syncwarp();
      const int i = lane >> 1, j0 = 8 * (lane & 1);
      float g[8];
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int j = j0 + jj;
        g[jj] = 0.5f * (XA[i * 17 + j] + XA[j * 17 + i]) + YA[i * 17 + j] + YA[j * 17 + i];
      }
      float4 *dst = reinterpret_cast<float4 *>(mat + s * kMat + i * LOCKS_B + j0);
      dst[0] = make_float4(g[0], g[1], g[2], g[3]);
      dst[1] = make_float4(g[4], g[5], g[6], g[7]);
      __syncwarp();
    }
  }

  // ---- 2. eigenvectors and eigenvalues of all the warp's items at once
  jacobi_phase<true>(mat, reinterpret_cast<float *>(scratch), mat, lam_s, live, r, lane);

  // ---- 3. per item: modes, basis, coefficients, quantisation
  uint8_t *blob = scratch;
#pragma unroll 1
  for (int s = 0; s < kBuildItems; ++s) {
    if (!((live >> s) & 1u)) continue;
    float dv[LOCKS_B][4], mu[4];
    load_item(s, dv);
    centre(dv, mu);
    const int block = __shfl_sync(0xffffffffu, it_block, s);
    const float knorm2 = kn_s[s];
    const float2 *U = us + s * LOCKS_B * 8;      // [token][mode], (u, u); ranks above 8: Uw[token][16 modes]
    const float *Uw = reinterpret_cast<const float *>(us) + s * LOCKS_B * LOCKS_B;
    const float *lamv = lam_s + s * LOCKS_B;     // eigenvalues, descending
    // ---- choose r_eff
    const float lam0 = lamv[0];
    int r_eff = 0;
    const int rmax = min(r, LOCKS_B - 1);
    for (int l = 0; l < rmax; ++l) {
      const float ll = lamv[l];
      if (lam0 > 0.f && ll > 1e-6f * lam0 && ll > 1e-10f * knorm2) r_eff = l + 1; else break;
    }
    // ---- per mode: basis entries of this lane's 4 dims, sign, quantise
    if (FMT == LOCKS_FMT_I4) {
      for (int e = lane; e < i4_stride(8) / 4; e += 32) reinterpret_cast<uint32_t *>(blob)[e] = 0u;
      __syncwarp();
    }
    uint8_t *gout = sbase + ((int64_t)block * p.Hkv + h) * p.S;
    float *fout = reinterpret_cast<float *>(gout);
    uint32_t sign_bits = 0u;   // bit l: mode l was flipped
#pragma unroll 1
    for (int l = 0; l < r; ++l) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      float best = 0.f;   // largest magnitude of the mode's basis vector
      if (l < r_eff) {
        const float inv = rsqrtf(lamv[l]);
        float2 va = make_float2(0.f, 0.f), vb = make_float2(0.f, 0.f);
        if (r > 8) {
#pragma unroll
          for (int i = 0; i < LOCKS_B; ++i) {
            const float u1 = Uw[i * LOCKS_B + l];
            const float2 u = make_float2(u1, u1);
            va = fma2(make_float2(dv[i][0], dv[i][1]), u, va);
            vb = fma2(make_float2(dv[i][2], dv[i][3]), u, vb);
          }
        } else {
#pragma unroll
          for (int i = 0; i < LOCKS_B; ++i) {
            const float2 u = U[i * 8 + l];
            va = fma2(make_float2(dv[i][0], dv[i][1]), u, va);
            vb = fma2(make_float2(dv[i][2], dv[i][3]), u, vb);
          }
        }
        v[0] = va.x * inv; v[1] = va.y * inv; v[2] = vb.x * inv; v[3] = vb.y * inv;
        // sign: entry of largest magnitude (lowest dim on ties) positive.  Magnitudes order like their bit
        // patterns; the lowest lane that holds the maximum owns the lowest such dim.
        best = fabsf(v[0]); float bv = v[0];
#pragma unroll
        for (int c = 1; c < 4; ++c) if (fabsf(v[c]) > best) { best = fabsf(v[c]); bv = v[c]; }
        const uint32_t mxb = __reduce_max_sync(0xffffffffu, __float_as_uint(best));
        const uint32_t who = __ballot_sync(0xffffffffu, __float_as_uint(best) == mxb);
        bv = __shfl_sync(0xffffffffu, bv, __ffs(who) - 1);
        best = __uint_as_float(mxb);
        if (bv < 0.f) {
          sign_bits |= 1u << l;
#pragma unroll
          for (int c = 0; c < 4; ++c) v[c] = -v[c];
        }
      }
      if (FMT == LOCKS_FMT_F32) {
        *reinterpret_cast<float4 *>(fout + LOCKS_D + l * LOCKS_D + lane * 4) = make_float4(v[0], v[1], v[2], v[3]);
      } else if (FMT == LOCKS_FMT_BF16) {   // row-major bf16 basis, straight to global memory
        *reinterpret_cast<uint2 *>(gout + 2 * (l * LOCKS_D + lane * 4)) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
      } else if (FMT == LOCKS_FMT_I8) {     // row-major int8 basis, one scale per mode
        const __half sh = __float2half_rn(best / 127.f);
        const float sc = inv_scale(__half2float(sh));
        if (lane == 0) *reinterpret_cast<__half *>(gout + wb_off_sv(r, 1) + 2 * l) = sh;
        uint32_t wd = 0u;
#pragma unroll
        for (int c = 0; c < 4; ++c) wd |= (uint32_t)((int)round_code(v[c], sc, 127.f) + 128) << (8 * c);
        *reinterpret_cast<uint32_t *>(gout + l * LOCKS_D + lane * 4) = wd;
      } else {
        const __half sh = __float2half_rn(best / 7.f);
        const float sc = inv_scale(__half2float(sh));
        if (lane == 0) *reinterpret_cast<__half *>(blob + i4_off_sv(r) + 2 * l) = sh;
        // lane = 8 t + s8 owns dims 32 t + 4 s8 + {0,1,2,3} = (half, e) in {0,1}^2 of k-step s8
        const int t = lane >> 3, s8 = lane & 7, i0 = (s8 & 1) << 1;
        uint32_t nb[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) nb[c] = (uint32_t)((int)round_code(v[c], sc, 7.f) + 8);
        // dim offset c = 2*half + e -> nibble i0 + half + 4 e
        uint32_t pw = (nb[0] << (4 * i0)) | (nb[1] << (4 * (i0 + 4))) | (nb[2] << (4 * (i0 + 1))) | (nb[3] << (4 * (i0 + 5)));
        pw |= __shfl_xor_sync(0xffffffffu, pw, 1);
        if ((s8 & 1) == 0) *reinterpret_cast<uint32_t *>(blob + (l * 4 + t) * 16 + (s8 >> 1) * 4) = pw;
      }
    }
    // coefficients: lane i < 16 owns token i
    if (lane < LOCKS_B) {
      float cf[16];
      float mx = 0.f;
      for (int l = 0; l < r; ++l) {
        float c = 0.f;
        if (l < r_eff) {
          c = sqrtf(lamv[l]) * (r > 8 ? Uw[lane * LOCKS_B + l] : U[lane * 8 + l].x);
          if ((sign_bits >> l) & 1u) c = -c;
        }
        cf[l & 15] = c;
        mx = fmaxf(mx, fabsf(c));
      }
      if (FMT == LOCKS_FMT_F32) {
        for (int l = 0; l < r; ++l) fout[LOCKS_D + r * LOCKS_D + lane * r + l] = cf[l & 15];
      } else if (FMT == LOCKS_FMT_I8 || FMT == LOCKS_FMT_BF16) {
        constexpr int W = FMT == LOCKS_FMT_BF16 ? 2 : 1;
        const __half sh = __float2half_rn(mx / 127.f);
        const float sc = inv_scale(__half2float(sh));
        *reinterpret_cast<__half *>(gout + wb_off_sc(r, W) + 2 * lane) = sh;
        for (int l = 0; l < r; ++l) gout[wb_off_coef(r, W) + lane * r + l] = (uint8_t)((int)round_code(cf[l & 15], sc, 127.f) + 128);
      } else {
        const __half sh = __float2half_rn(mx / 127.f);
        const float sc = inv_scale(__half2float(sh));
        const int tpos = ((lane & 7) >> 1) * 4 + (lane >> 3) * 2 + (lane & 1);
        *reinterpret_cast<__half *>(blob + i4_off_sc(r) + 2 * tpos) = sh;
        const int xx = lane & 7, hi = lane >> 3;
        for (int l = 0; l < r; ++l)
          blob[i4_off_coef(r) + (xx * (r / 2) + (l >> 1)) * 4 + hi * 2 + (l & 1)] =
              (uint8_t)((int)round_code(cf[l & 15], sc, 127.f) + 128);
      }
    }
    // centroid
    if (FMT == LOCKS_FMT_F32) {
      *reinterpret_cast<float4 *>(fout + lane * 4) = make_float4(mu[0], mu[1], mu[2], mu[3]);
    } else if (FMT == LOCKS_FMT_I8 || FMT == LOCKS_FMT_BF16) {
      constexpr int W = FMT == LOCKS_FMT_BF16 ? 2 : 1;
      float mx = fmaxf(fmaxf(fabsf(mu[0]), fabsf(mu[1])), fmaxf(fabsf(mu[2]), fabsf(mu[3])));
      mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
      const __half sh = __float2half_rn(mx / 127.f);
      const float sc = inv_scale(__half2float(sh));
      if (lane == 0) *reinterpret_cast<__half *>(gout + wb_off_smu(r, W)) = sh;
      uint32_t wd = 0u;
#pragma unroll
      for (int c = 0; c < 4; ++c) wd |= (uint32_t)((int)round_code(mu[c], sc, 127.f) + 128) << (8 * c);
      *reinterpret_cast<uint32_t *>(gout + wb_off_mu(r, W) + lane * 4) = wd;
      // bytes between the payload and the 16-byte padded stride stay zero (the buffer is the caller's; clear them)
      for (int e = wb_off_smu(r, W) + 2 + lane; e < p.S; e += 32) gout[e] = 0;
    } else {
      float mx = fmaxf(fmaxf(fabsf(mu[0]), fabsf(mu[1])), fmaxf(fabsf(mu[2]), fabsf(mu[3])));
      mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
      const __half sh = __float2half_rn(mx / 127.f);
      const float sc = inv_scale(__half2float(sh));
      if (lane == 0) *reinterpret_cast<__half *>(blob + i4_off_smu(r)) = sh;
      uint32_t bytes[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) bytes[c] = (uint32_t)((int)round_code(mu[c], sc, 127.f) + 128);
      // dim offset c = 2*half + e -> byte e*2 + half
      const uint32_t wd = bytes[0] | (bytes[2] << 8) | (bytes[1] << 16) | (bytes[3] << 24);
      *reinterpret_cast<uint32_t *>(blob + i4_off_mu(r) + lane * 4) = wd;
      __syncwarp();
      uint4 *dst = reinterpret_cast<uint4 *>(gout);
      for (int e = lane; e < p.S / 16; e += 32) dst[e] = reinterpret_cast<const uint4 *>(blob)[e];
      __syncwarp();   // the blob is cleared again for the next item
    }
  }
}

}  // namespace

int locks_launch_build(locks_ctx *c, const locks_kv *kv, int batch, const int32_t *pb, const int32_t *pe,
                       int just_filled, void *summaries, const void *k_new, const int32_t *append_pos,
                       cudaStream_t st, const void *const *k_layers, void *const *summ_layers, int num_layers) {
  BuildParams p;
  p.k = kv->k; p.sb = kv->stride_block; p.sh = kv->stride_head; p.st = kv->stride_token;
  p.block_table = kv->block_table; p.seq_lens = kv->seq_lens; p.page_begin = pb; p.page_end = pe;
  p.summ = reinterpret_cast<uint8_t *>(summaries); p.status = c->status;
  p.batch = batch; p.Hkv = c->cfg.num_kv_heads; p.Pmax = c->Pmax; p.num_blocks = kv->num_blocks;
  p.r = c->cfg.rank; p.S = c->S; p.fmt = c->cfg.summary_fmt; p.esz = c->cfg.kv_dtype == LOCKS_BF16 ? 2 : 4;
  p.k_layers = just_filled ? nullptr : k_layers; p.summ_layers = just_filled ? nullptr : summ_layers;
  p.k_new = just_filled ? k_new : nullptr; p.append_pos = just_filled ? append_pos : nullptr;
  p.hint = nullptr; p.kpages = c->k; p.hint_wpp = 1; p.hint_rounds = 1; p.hint_W = 1;
  if (just_filled && c->hint_dev && c->cfg.summary_fmt == LOCKS_FMT_I4 && c->cfg.q_dtype == LOCKS_BF16) {
    const locks_scan_geom geo = locks_scan_geometry(c, batch);
    p.hint = c->hint_dev; p.hint_wpp = geo.wpp; p.hint_rounds = geo.rounds; p.hint_W = geo.W;
  }
  if (c->B != LOCKS_B && k_layers) return LOCKS_ERR_UNSUPPORTED;   // one layer per launch
  // A step's few pages, where latency counts, and the page sizes that the bulk kernel does not know: one CTA per page
  if (just_filled || c->B != LOCKS_B) return locks_launch_build_pages(c, p, just_filled, st);
  constexpr int kPer = kBuildWarps * kBuildItems;   // items per CTA (bulk)
  const dim3 grid((c->Pmax + kPer - 1) / kPer, p.Hkv, batch * (k_layers ? num_layers : 1));
  const bool bf = c->cfg.kv_dtype == LOCKS_BF16;
  const int smem = kBuildWarps * kBuildSmemPerWarp;
#define LOCKS_BUILD_CASE(F_)                                                                                                \
  do {                                                                                                                     \
    if (bf) build_kernel<__nv_bfloat16, F_><<<grid, kBuildWarps * 32, smem, st>>>(p);                                       \
    else build_kernel<float, F_><<<grid, kBuildWarps * 32, smem, st>>>(p);                                                 \
  } while (0)
  switch (c->cfg.summary_fmt) {
    case LOCKS_FMT_I4:
      if (bf) build_i4_kernel<<<grid, kBuildWarps * 32, kBuildWarps * kBuildI4SmemPerWarp, st>>>(p);
      else build_kernel<float, LOCKS_FMT_I4><<<grid, kBuildWarps * 32, smem, st>>>(p);
      break;
    case LOCKS_FMT_I8: LOCKS_BUILD_CASE(LOCKS_FMT_I8); break;
    case LOCKS_FMT_BF16: LOCKS_BUILD_CASE(LOCKS_FMT_BF16); break;
    default: LOCKS_BUILD_CASE(LOCKS_FMT_F32); break;
  }
#undef LOCKS_BUILD_CASE
  return locks_check_launch(c);
}
