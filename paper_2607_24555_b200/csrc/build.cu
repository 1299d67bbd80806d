// Summary build (Sec. 4 "Build (once, when a page completes)"), bulk (build_page.cu has the page that a decode step fills).
//
// 16-token pages: one warp takes 8 (page, KV head) items through three phases.
//   1. per item, all lanes: load the page's 16 keys (lane owns 4 consecutive dims of every key), centroid mu,
//      deviations D, and the Gram matrix M = D D^T (16 x 16) on the tensor cores; M goes to shared memory
//   2. all 8 items at once: eigendecomposition of M by one-sided Jacobi in fp32.  Four lanes hold one item's
//      matrix (4 columns of 16 entries each, in registers); columns are rotated in pairs until they are mutually
//      orthogonal, which leaves M W = U Lambda: column norms are the eigenvalues, normalised columns the
//      eigenvectors.
//   3. per item, all lanes: reload the keys, rank the modes by eigenvalue, keep r_eff <= min(r, 15) modes above
//      the zero-mode thresholds, V = D^T U_r Sigma_r^-1 (lane's 4 dims), C = U_r Sigma_r, sign: largest |V| entry
//      positive; store fp32 (F32 format) or quantise: symmetric abs-max, fp16 scale, round-half-even codes
//      (int4 basis per column, int8 coefficients per row, int8 centroid) packed in the blob layout
// build_i4_kernel: bf16 keys, int4 summaries.  build_kernel: everything else (fp32 keys, the other formats), one instruction
// sequence for all of them.  Both round alike.
//
// The bytes of a summary decide near-ties between pages, so what is computed and in which order is kept exactly: a
// preconditioned solver (build_page.cu's; 5 sweeps for 8) builds 131 008 page-heads in 870 us and is as accurate, but one
// byte in ten thousand comes out differently, and one request in a few hundred then keeps another page.  The page that a step
// fills is built with that solver: a bulk build of the same page gives other bytes at that rate.
// A mode between 1e-6 and 3e-6 of the largest is kept, but does not hold up the sweeps (floor_n), so its basis vector may be too
// long; on such pages the step build is the more accurate one.
// Bound by instruction issue, fetch and latency, not by bytes (an eigenproblem per 4 KB page).  131 008 page-heads: 1348 us
// with the pair that straddles two lanes rotated by both and all formats in one kernel (6 960 warp instructions each), 1281
// us with every pair rotated once and build_i4_kernel's phases (5 370), 1095 us with the body of a sweep kept to two steps.
// Smaller builds are one or two waves long and bound by the latency of a group (8 pages of a KV head) and by how the groups
// lie on the SMs; see build_i4_kernel: 16 .. 384 groups 99 -> 79 .. 93 us, 1024: 197 -> 131, 4096 (a prompt chunk of 2048
// tokens in 32 layers): 385 -> 345, and chunks of 9 .. 40 pages in 32 layers, 130 .. 205 us before, 76 .. 131.
#include <algorithm>
#include <type_traits>
#include "build_common.cuh"

namespace {

constexpr int kBuildWarps = 2;
constexpr int kBuildItems = 8;                                   // (page, KV head) items per warp
constexpr int kBuildCtasPerSm = 8;                               // 16 warps per SM
constexpr int kBuildScratch = 2 * LOCKS_B * 128;                 // 4096 B: bf16 half-tiles of D (hi | lo); later the blob
constexpr int kMat = LOCKS_B * LOCKS_B + 16;                     // floats per item's matrix: items on different banks
constexpr int kBuildMat = kBuildItems * kMat * 4;                // 8704 B: Gram matrices; later the leading eigenvectors, every entry twice
constexpr int kBuildSmemPerWarp = kBuildScratch + kBuildMat + 64 + kBuildItems * LOCKS_B * 4;   // + key norms, eigenvalues

// The plane rotation that makes two columns p, q orthogonal, from a = |p|^2, b = |q|^2, g = p . q (smaller angle):
// with d = b - a and h = d^2 + 4 g^2, cos 2t = |d| / sqrt(h) and sin 2t = 2 g sign(d) / sqrt(h), so
// c = sqrt((1 + cos 2t) / 2) and s = sin 2t / (2 c): two reciprocal square roots in a row (approximate ones are
// enough for the angle; c^2 + s^2 = 1 holds to their rounding).  p' = c p - s q, q' = s p + c q.  Inputs too small
// or too large to square are left alone.
__device__ __forceinline__ void plane_rotation(float a, float b, float g, float &c, float &sn) {
  const float d = b - a, hh = fmaf(d, d, 4.f * g * g);
  const bool ok = hh > 1e-37f && hh < 1e37f;   // branch-free: independent pairs interleave in one basic block
  const float rs = rsqrt_approx(ok ? hh : 1.f);
  const float x = fmaf(0.5f * fabsf(d), rs, 0.5f);
  const float r2 = rsqrt_approx(x);
  const float s0 = copysignf(g * rs * r2, d == 0.f ? g : g * d);
  c = ok ? x * r2 : 1.f;
  sn = ok ? s0 : 0.f;
}

// One-sided Jacobi on 8 matrices at once.  Lane (item = lane / 4, j = lane % 4) holds columns 4 j .. 4 j + 3 of its item's
// matrix W (initially M, symmetric: the columns are read as rows), w[c][i] = rows 2i, 2i+1 of column 4 j + c as a packed
// pair, and their squared norms: two pairs of columns.  Odd-even transposition: 16 steps per sweep meet every two columns
// once; every step rotates all pairs, a rotated pair swaps places, and one column of each pair is passed to a neighbour,
// half of the time within the lane.
// Result: the columns ranked by norm (descending, ties to the lower position), the 16 eigenvalues to lam_s[item][mode],
// unit eigenvectors of the leading min(r, 8) modes to us as pairs (u, u): BY_MODE [item][mode][token], else
// [item][token][mode] (r > 8: all 16, plain entries, [token][16]).
template <bool BY_MODE, int CPL, typename Vote>
__device__ __forceinline__ void jacobi_phase(const float *mat, float *us, float *lam_s, uint32_t live, int r, int lane, int item0,
                                             Vote vote) {
  constexpr int LPI = LOCKS_B / CPL;
  const int item = item0 + lane / LPI, j = lane % LPI;
  const bool item_live = (live >> item) & 1u;   // lanes of an absent item compute on zeros
  float2 w[CPL][8];
  {
    const float4 *src = reinterpret_cast<const float4 *>(mat + item * kMat + CPL * j * LOCKS_B);
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        const float4 f = item_live ? src[c * 4 + q4] : make_float4(0.f, 0.f, 0.f, 0.f);
        w[c][2 * q4] = make_float2(f.x, f.y);
        w[c][2 * q4 + 1] = make_float2(f.z, f.w);
      }
  }
  __syncwarp();   // every lane holds its columns: the matrices' shared memory may be overwritten from here on
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
  const float tol2 = LOCKS_BUILD_COS_TOL * LOCKS_BUILD_COS_TOL;
  int bad = 0;
  float floor_n = 0.f;
  // columns whose norm is rounding noise beside the largest (null directions) do not hold up convergence
  // One pair: a is the column that it kept from the step before, b the one that it has been passed; in even steps b is the
  // lower position (p), in odd ones a.  The lower position receives q' = s p + c q, the upper one p' = c p - s q.  What is
  // kept ends in a, what is passed on in b.  `there` = false: the two ends of the row, which do not meet: a stays, b moves on.
  auto rotate = [&](auto odd, float2 (&a)[8], float2 (&b)[8], float &na, float &nb, bool there) {
    constexpr bool kOdd = decltype(odd)::value;
    const float g = dot(a, b), np = kOdd ? na : nb, nq = kOdd ? nb : na;
    bad |= (int)there & (int)(g * g > tol2 * np * nq) & (int)(fminf(np, nq) > floor_n);
    float c, sn;
    plane_rotation(np, nq, g, c, sn);
    float x2 = 2.f * c * sn * g;
    if (kOdd && !there) { c = 0.f; sn = 1.f; x2 = 0.f; }
    const float2 C2 = make_float2(c, c), S2 = make_float2(sn, sn), nS2 = make_float2(-sn, -sn);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 p = kOdd ? a[i] : b[i], q = kOdd ? b[i] : a[i];
      const float2 pp = fma2(C2, p, mul2(nS2, q)), qq = fma2(S2, p, mul2(C2, q));
      a[i] = kOdd ? qq : pp;
      b[i] = kOdd ? pp : qq;
    }
    const float cc = c * c, ss = sn * sn;
    const float n_p = fmaxf(fmaf(cc, np, fmaf(ss, nq, -x2)), 0.f), n_q = fmaxf(fmaf(ss, np, fmaf(cc, nq, x2)), 0.f);
    na = kOdd ? n_q : n_p;
    nb = kOdd ? n_p : n_q;
  };
  const int up = (lane & ~(LPI - 1)) | ((j + 1) & (LPI - 1)), down = (lane & ~(LPI - 1)) | ((j - 1) & (LPI - 1));
  auto fetch = [&](float2 (&col)[8], float &norm, int from) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      col[i].x = __shfl_sync(0xffffffffu, col[i].x, from);
      col[i].y = __shfl_sync(0xffffffffu, col[i].y, from);
    }
    norm = __shfl_sync(0xffffffffu, norm, from);
  };
  constexpr std::false_type even{};
  constexpr std::true_type odd{};
  for (int sweep = 0; sweep < LOCKS_BUILD_SWEEPS; ++sweep) {
    norms();
    {
      float nm = n[0];
#pragma unroll
      for (int c = 1; c < CPL; ++c) nm = fmaxf(nm, n[c]);
      floor_n = 1e-11f * seg_max(nm);   // squared norm = squared eigenvalue: modes below 3e-6 of the largest
    }
    bad = 0;
#pragma unroll 1
    for (int st2 = 0; st2 < 8; ++st2) {   // (a body of this size: twice unrolled, a quarter of the warps wait for instructions)
      rotate(even, w[1], w[0], n[1], n[0], true);
      if constexpr (CPL == 4) rotate(even, w[3], w[2], n[3], n[2], true);
      fetch(w[0], n[0], up);     // a pair passes to the one before it: w[2] to the lane's first, w[0] to the lane below
      if constexpr (CPL == 4) rotate(odd, w[1], w[2], n[1], n[2], true);
      rotate(odd, w[CPL - 1], w[0], n[CPL - 1], n[0], j != LPI - 1);
      fetch(w[0], n[0], down);   // ... and then to the one after it: w[2] to the lane's second, w[0] to the lane above
    }
    if (!vote(bad != 0)) break;
  }
  norms();
  int rank[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) rank[c] = 0;
#pragma unroll
  for (int jj = 0; jj < LPI; ++jj)
#pragma unroll
    for (int cc = 0; cc < CPL; ++cc) {
      const float o = __shfl_sync(0xffffffffu, n[cc], (lane & ~(LPI - 1)) + jj);
#pragma unroll
      for (int c = 0; c < CPL; ++c) rank[c] += (o > n[c]) || (o == n[c] && (jj * CPL + cc) < (j * CPL + c));
    }
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    lam_s[item * LOCKS_B + rank[c]] = sqrtf(n[c]) * unscale;
    const float inv = n[c] > 0.f ? rsqrtf(n[c]) : 0.f;
    if (BY_MODE) {
      if (rank[c] < 8) {
        float4 *dst = reinterpret_cast<float4 *>(us + item * kMat + rank[c] * 2 * LOCKS_B);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float u0 = w[c][i].x * inv, u1 = w[c][i].y * inv;
          dst[i] = make_float4(u0, u0, u1, u1);
        }
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

// Physical block of item `lane` (< 8) of warp `warp` among those of request b, -1 if there is none; page ranges as
// locks_build_summaries has them.
__device__ __forceinline__ int item_block(const BuildParams &p, int b, int warp, int lane) {
  if (lane >= kBuildItems) return -1;
  const int complete = p.seq_lens[b] / LOCKS_B;
  const int p0 = p.page_begin ? p.page_begin[b] : 0;
  const int p1 = min(p.page_end ? p.page_end[b] : complete, complete);
  const int page = p0 + warp * kBuildItems + lane;
  if (page < 0 || page >= p1 || page >= p.Pmax) return -1;
  const int block = p.block_table[(int64_t)b * p.Pmax + page];
  if (block >= 0 && block < p.num_blocks) return block;
  set_status(p.status, LOCKS_ERR_BAD_BLOCK);
  return -1;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(*reinterpret_cast<unsigned long long *>(&d))
      : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
  return d;
}

// bf16 keys, int4 summaries: build_kernel's arithmetic with its phases 1 and 3 arranged for the common case.  Packed fp32
// pairs; M leaves the MMA accumulators through one transposed array instead of two; all modes' basis vectors are formed
// before any is quantised, so that their scales (a division, an fp16 rounding and a reciprocal each) are worked out by a
// lane per mode, once; codes go straight to global memory.
//
// A group is 8 pages of one (layer, request, KV head); W warps of a CTA work on it.  One keeps every lane busy all the time.
// Of two, each takes 4 of the items in phases 1 and 3, and 8 lanes hold a matrix in phase 2: a group is done in 79 us on an
// idle chip where one warp takes 99.  Whether a group's sweeps go on is one decision of all its warps, so that the bytes are
// the same either way.
constexpr int kI4Warps = 2, kI4CtasPerSm = 8, kI4Waves = 32, kI4Pairs = 22;
constexpr int kI4Group = kBuildMat + 64 + kBuildItems * LOCKS_B * 4;   // bytes: matrices, key norms, eigenvalues
constexpr int kI4Smem = kI4Warps * (kBuildScratch + kI4Group);
constexpr int kI4SmemCount = kI4Smem + 64;   // + the number of groups, a group's blocks and KV head

__device__ __forceinline__ int build_pages(const BuildParams &p, int b, int &p0) {   // pages of request b to build, from p0 on
  const int complete = p.seq_lens[b] / LOCKS_B;
  p0 = p.page_begin ? p.page_begin[b] : 0;
  const int p1 = min(min(p.page_end ? p.page_end[b] : complete, complete), p.Pmax);
  return (int)max((int64_t)0, min((int64_t)p1 - p0, (int64_t)p.Pmax + LOCKS_B));
}

// kbase, sbase: the layer's keys and summaries at the group's KV head
template <int W>
__device__ __forceinline__ void build_i4_group(const BuildParams &p, uint8_t *smem_raw, int tid, int it_block, uint32_t live,
                                               const __nv_bfloat16 *kbase, uint8_t *sbase) {
  constexpr int kItems = kBuildItems / W;   // items of this warp
  const int lane = tid & 31, warp = tid >> 5, wg = warp % W, r = p.r;
  uint8_t *scratch = smem_raw + warp * kBuildScratch;   // D half-tiles, then Y
  float *mat = reinterpret_cast<float *>(smem_raw + kI4Warps * kBuildScratch + warp / W * kI4Group);   // [8][16][16] Gram; then [8][8][16] pairs (u, u) of U_r by mode
  float *kn_s = mat + kBuildItems * kMat;   // [8] squared norm of the page's keys
  float *lam_s = kn_s + 16;                 // [8][16] eigenvalues, descending
  // deviations of item s: v[i][e] = key i minus the centroid, dims 4 lane + 2 e, + 1; knorm2: this lane's share
  auto load_centred = [&](int s, float2 (&v)[LOCKS_B][2], float2 (&mu)[2], bool want_norm, float &knorm2) {
    const __nv_bfloat16 *K = kbase + (int64_t)__shfl_sync(0xffffffffu, it_block, s) * p.sb + 4 * lane;
#pragma unroll
    for (int i = 0; i < LOCKS_B; ++i) {
      const uint2 w = *reinterpret_cast<const uint2 *>(K + (int64_t)i * p.st);
      v[i][0] = make_float2(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u));
      v[i][1] = make_float2(__uint_as_float(w.y << 16), __uint_as_float(w.y & 0xFFFF0000u));
    }
    if (want_norm) {
      float2 n0 = make_float2(0.f, 0.f), n1 = n0;
#pragma unroll
      for (int i = 0; i < LOCKS_B; ++i) { n0 = fma2(v[i][0], v[i][0], n0); n1 = fma2(v[i][1], v[i][1], n1); }
      knorm2 = (n0.x + n0.y) + (n1.x + n1.y);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      mu[e] = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < LOCKS_B; ++i) mu[e] = add2(mu[e], v[i][e]);
      mu[e] = mul2(mu[e], make_float2(1.f / LOCKS_B, 1.f / LOCKS_B));
      const float2 neg = make_float2(-mu[e].x, -mu[e].y);
#pragma unroll
      for (int i = 0; i < LOCKS_B; ++i) v[i][e] = add2(v[i][e], neg);
    }
  };

  // ---- 1. Gram matrices (see build_kernel)
#pragma unroll 1
  for (int s = wg * kItems; s < (wg + 1) * kItems; ++s) {
    if (!((live >> s) & 1u)) continue;
    uint32_t hl[LOCKS_B][4];   // h01, h23, l01, l23 of this lane's 4 dims, per key
    {
      float2 v[LOCKS_B][2], mu[2];
      float knorm2 = 0.f;
      load_centred(s, v, mu, true, knorm2);
      knorm2 = warp_sum(knorm2);
      if (lane == 0) kn_s[s] = knorm2;
#pragma unroll
      for (int i = 0; i < LOCKS_B; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint32_t hh = pack_bf16(v[i][e].x, v[i][e].y);
          const float2 lo = add2(v[i][e], make_float2(-__uint_as_float(hh << 16), -__uint_as_float(hh & 0xFFFF0000u)));
          hl[i][e] = hh;
          hl[i][2 + e] = pack_bf16(lo.x, lo.y);
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
    // accumulator (x = lane / 4, t = lane % 4): [0..1] = row x, columns 2t, 2t+1 (X1: + 8); [2..3] = row x + 8.  X is symmetric
    // as computed; M = X + Y + Y^T, the transpose through a padded 16 x 17 array in the (now free) scratch
    {
      float *YA = reinterpret_cast<float *>(scratch);
      const int x = lane >> 2, t = lane & 3;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        YA[x * 17 + 2 * t + e] = Y0[e]; YA[(x + 8) * 17 + 2 * t + e] = Y0[2 + e];
        YA[x * 17 + 8 + 2 * t + e] = Y1[e]; YA[(x + 8) * 17 + 8 + 2 * t + e] = Y1[2 + e];
      }
      __syncwarp();
      float *dst = mat + s * kMat + x * LOCKS_B + 2 * t;
      const float *yt = YA + 2 * t * 17 + x;   // column 2t of Y^T's row x
      *reinterpret_cast<float2 *>(dst) = make_float2(X0[0] + Y0[0] + yt[0], X0[1] + Y0[1] + yt[17]);
      *reinterpret_cast<float2 *>(dst + 8) = make_float2(X1[0] + Y1[0] + yt[8 * 17], X1[1] + Y1[1] + yt[9 * 17]);
      *reinterpret_cast<float2 *>(dst + 8 * LOCKS_B) = make_float2(X0[2] + Y0[2] + yt[8], X0[3] + Y0[3] + yt[17 + 8]);
      *reinterpret_cast<float2 *>(dst + 8 * LOCKS_B + 8) = make_float2(X1[2] + Y1[2] + yt[8 * 17 + 8], X1[3] + Y1[3] + yt[9 * 17 + 8]);
      __syncwarp();
    }
  }

  // ---- 2. eigenvectors and eigenvalues of all the warp's items at once
  if constexpr (W == 1) {
    jacobi_phase<true, 4>(mat, mat, lam_s, live, r, lane, 0, [](bool bad) { return __any_sync(0xffffffffu, bad) != 0; });
  } else {
    // the two warps' votes meet at a barrier of theirs
    auto vote = [](bool bad) {
      int any;
      asm volatile("{\n .reg .pred a, b;\n setp.ne.s32 a, %1, 0;\n bar.red.or.pred b, 1, 64, a;\n selp.s32 %0, 1, 0, b;\n}\n"
                   : "=r"(any) : "r"((int)bad) : "memory");
      return any != 0;
    };
    jacobi_phase<true, 2>(mat, mat, lam_s, live, r, lane, wg * 4, vote);
  }

  // ---- 3. basis, coefficients, centroid
#pragma unroll 1
  for (int s = wg * kItems; s < (wg + 1) * kItems; ++s) {
    if (!((live >> s) & 1u)) continue;
    const float *U = mat + s * kMat, *lam = lam_s + s * LOCKS_B;   // U[mode][token] as pairs
    // lane l < r: mode l
    const float lam0 = lam[0], lx = lam[lane & 15];
    // modes above the zero-mode thresholds (eigenvalues descend).  The 16th is nothing but rounding (D sums to zero), but not always
    // below them: where the diagonal of M swallows many small products (one large entry per key) it reads 3e-6 of the first.
    const uint32_t above = __ballot_sync(0xffffffffu, lam0 > 0.f && lx > 1e-6f * lam0 && lx > 1e-10f * kn_s[s]) & 0x7fffu;
    const int r_eff = min(r, __ffs(~above) - 1);
    const float isig = lane < r_eff ? rsqrtf(lx) : 0.f;
    float2 v[8][2], mu[2];   // basis vectors of this lane's 4 dims
    {
      float2 dv[LOCKS_B][2];
      float unused;
      load_centred(s, dv, mu, false, unused);
#pragma unroll
      for (int l = 0; l < 8; ++l) {
        v[l][0] = v[l][1] = make_float2(0.f, 0.f);
        if (l < r_eff) {
          const float4 *u4 = reinterpret_cast<const float4 *>(U + l * 2 * LOCKS_B);
#pragma unroll
          for (int i = 0; i < LOCKS_B; i += 2) {
            const float4 u = u4[i / 2];
            v[l][0] = fma2(dv[i][0], make_float2(u.x, u.y), v[l][0]);
            v[l][1] = fma2(dv[i][1], make_float2(u.x, u.y), v[l][1]);
            v[l][0] = fma2(dv[i + 1][0], make_float2(u.z, u.w), v[l][0]);
            v[l][1] = fma2(dv[i + 1][1], make_float2(u.z, u.w), v[l][1]);
          }
        }
      }
    }
    uint8_t *gout = sbase + (int64_t)__shfl_sync(0xffffffffu, it_block, s) * p.Hkv * p.S;
    // sign: the entry of largest magnitude (lowest dim on ties) is positive.  Magnitudes order like their bit patterns; the
    // lowest lane that holds the maximum owns the lowest such dim.
    float best_mode = 0.f;         // lane l: largest magnitude of mode l
    uint32_t neg = 0u;             // bit l: mode l is flipped
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      if (l >= r_eff) break;
      const float is = __shfl_sync(0xffffffffu, isig, l);
      const float2 is2 = make_float2(is, is);
      v[l][0] = mul2(v[l][0], is2);
      v[l][1] = mul2(v[l][1], is2);
      float best = fabsf(v[l][0].x), bv = v[l][0].x;
      if (fabsf(v[l][0].y) > best) { best = fabsf(v[l][0].y); bv = v[l][0].y; }
      if (fabsf(v[l][1].x) > best) { best = fabsf(v[l][1].x); bv = v[l][1].x; }
      if (fabsf(v[l][1].y) > best) { best = fabsf(v[l][1].y); bv = v[l][1].y; }
      const uint32_t mxb = __reduce_max_sync(0xffffffffu, __float_as_uint(best));
      const uint32_t who = __ballot_sync(0xffffffffu, __float_as_uint(best) == mxb), minus = __ballot_sync(0xffffffffu, bv < 0.f);
      if (minus & who & -who) neg |= 1u << l;
      if (lane == l) best_mode = __uint_as_float(mxb);
    }
    const __half sv = __float2half_rn(best_mode / 7.f);
    const float sc_mode = inv_scale(__half2float(sv)) * ((neg >> (lane & 7)) & 1u ? -1.f : 1.f);
    if (lane < r) *reinterpret_cast<__half *>(gout + i4_off_sv(r) + 2 * lane) = sv;
    // codes: lane = 8 t + s8 owns dims 32 t + 4 s8 + {0,1,2,3} = (half, e) in {0,1}^2 of k-step s8; dim offset c = 2 half + e ->
    // nibble 2 (s8 & 1) + half + 4 e.  x + 1.5 2^23 + 8 rounds half to even and leaves code + 8 in the low bits (a scale would have
    // to be below 7 steps of fp16 for a code to leave -7 .. 7; the smallest that pages of noise modes gave is 13).  The product is
    // rounded by itself: packed, the two become one fma, and what rounds to a tie first gets another code (a byte in 8 million).
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      if (l >= r) break;
      const float sc = __shfl_sync(0xffffffffu, sc_mode, l);
      auto magic = [&](float x) { return __fadd_rn(__fmul_rn(x, sc), 12582920.f); };
      const float2 a = make_float2(magic(v[l][0].x), magic(v[l][0].y)), b = make_float2(magic(v[l][1].x), magic(v[l][1].y));
      uint32_t pw = (__float_as_uint(a.x) & 15u) | (__float_as_uint(a.y) & 15u) << 16 | (__float_as_uint(b.x) & 15u) << 4 |
                    (__float_as_uint(b.y) & 15u) << 20;
      pw <<= 8 * (lane & 1);
      pw |= __shfl_xor_sync(0xffffffffu, pw, 1);
      if ((lane & 1) == 0) *reinterpret_cast<uint32_t *>(gout + l * 64 + lane * 2) = pw;
    }
    // coefficients C = U Sigma: lane (x, t) has tokens x and x + 8, modes 2t and 2t + 1
    {
      const int x = lane >> 2, t = lane & 3;
      const float sg = lane < r_eff ? ((neg >> lane) & 1u ? -sqrtf(lx) : sqrtf(lx)) : 0.f;
      const float g0 = __shfl_sync(0xffffffffu, sg, 2 * t), g1 = __shfl_sync(0xffffffffu, sg, 2 * t + 1);
      const float *u0 = U + 2 * t * 2 * LOCKS_B + 2 * x, *u1 = u0 + 2 * LOCKS_B;
      const float ca = 2 * t < r_eff ? g0 * u0[0] : 0.f, cb = 2 * t + 1 < r_eff ? g1 * u1[0] : 0.f;
      const float cc = 2 * t < r_eff ? g0 * u0[16] : 0.f, cd = 2 * t + 1 < r_eff ? g1 * u1[16] : 0.f;
      float ma = fmaxf(fabsf(ca), fabsf(cb)), mb = fmaxf(fabsf(cc), fabsf(cd));
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
        mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
      }
      const __half sa = __float2half_rn(ma / 127.f), sb = __float2half_rn(mb / 127.f);
      const float ia = inv_scale(__half2float(sa)), ib = inv_scale(__half2float(sb));
      auto code = [&](float v, float inv) { return (uint32_t)((int)round_code(v, inv, 127.f) + 128); };
      if (t < r / 2)
        *reinterpret_cast<uint32_t *>(gout + i4_off_coef(r) + (x * (r / 2) + t) * 4) =
            code(ca, ia) | (code(cb, ia) << 8) | (code(cc, ib) << 16) | (code(cd, ib) << 24);
      if (t == 0) {
        __half *dst = reinterpret_cast<__half *>(gout + i4_off_sc(r)) + (x >> 1) * 4 + (x & 1);
        dst[0] = sa;
        dst[2] = sb;
      }
    }
    // centroid: dim offset c = 2*half + e -> byte e*2 + half
    {
      const float mx = fmaxf(fmaxf(fabsf(mu[0].x), fabsf(mu[0].y)), fmaxf(fabsf(mu[1].x), fabsf(mu[1].y)));
      const __half sh = __float2half_rn(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx))) / 127.f);
      const float sc = inv_scale(__half2float(sh));
      auto code = [&](float v) { return (uint32_t)((int)round_code(v, sc, 127.f) + 128); };
      *reinterpret_cast<uint32_t *>(gout + i4_off_mu(r) + lane * 4) = code(mu[0].x) | (code(mu[1].x) << 8) | (code(mu[0].y) << 16) | (code(mu[1].y) << 24);
      if (lane == 0) *reinterpret_cast<__half *>(gout + i4_off_smu(r)) = sh;
      if (lane < 16 && i4_off_smu(r) + 2 + lane < p.S) gout[i4_off_smu(r) + 2 + lane] = 0;   // bytes between the payload and the stride
    }
  }}

// The groups by the table's rows: of 16 pages of a row, 8 a warp.  For tables that are about full, but nothing says that they are:
// the first pages of all rows come first in the grid, so that the CTAs of pages that are not there start, and end, while the
// others work (8 requests of 2K tokens in rows of 34 816, us: 119, row after row 146, dealt out 88; 32 of 4K in rows of 32K: 500, 573
// and 518; rows of 32K that are full: 967, 956 and 991).
__global__ void __launch_bounds__(kI4Warps * 32, kI4CtasPerSm) build_i4_table_kernel(BuildParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, h = blockIdx.x, layer = blockIdx.y / p.batch;
  const int it_block = item_block(p, blockIdx.y % p.batch, blockIdx.z * kI4Warps + (threadIdx.x >> 5), lane);   // lane s < 8: item s
  const uint32_t live = __ballot_sync(0xffffffffu, it_block >= 0);
  if (!live) return;
  build_i4_group<1>(p, smem_raw, threadIdx.x, it_block, live,
                    reinterpret_cast<const __nv_bfloat16 *>(p.k_layers ? p.k_layers[layer] : p.k) + (int64_t)h * p.sh,
                    (p.summ_layers ? reinterpret_cast<uint8_t *>(p.summ_layers[layer]) : p.summ) + (int64_t)h * p.S);
}

// The groups that there are, counted from the lengths and page ranges and dealt to the CTAs without gaps.
template <int W>
__device__ __forceinline__ void build_i4_groups(const BuildParams &p, uint8_t *smem_raw, const volatile int *count, int layers) {
#pragma unroll 1
  for (int round = 0;; ++round) {
    int tid = threadIdx.x;
    asm volatile("" : "+r"(tid));   // nothing that follows from it is worth a register across groups
    const int lane = tid & 31, warp = tid >> 5;
    int *blk_s = reinterpret_cast<int *>(smem_raw + kI4Warps * (kBuildScratch + kI4Group)) + 4;   // W > 1: blocks of the 8 items, KV head
    const int groups = *count;   // of a layer
    const int64_t g = ((int64_t)round * gridDim.x + blockIdx.x) * (kI4Warps / W) + warp / W;
    const int layer = (int)(g / groups);
    if (layer >= layers) break;
    int it_block = -1, h = 0;   // lane s < 8: item s
    if (W == 1 || warp == 0) {
      int n = (int)(g - (int64_t)layer * groups);   // the group's place in its layer: by request, KV head, page
      for (int b0 = 0; b0 < p.batch; b0 += 32) {
        int p0 = 0;
        const int have = b0 + lane < p.batch ? build_pages(p, b0 + lane, p0) : 0, mine = (have + kBuildItems - 1) / kBuildItems * p.Hkv;
        int upto = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, upto, o);
          if (lane >= o) upto += v;
        }
        const uint32_t past = __ballot_sync(0xffffffffu, n < upto);
        if (past) {
          const int src = __ffs(past) - 1;
          const int end = __shfl_sync(0xffffffffu, have, src), per_head = (end + kBuildItems - 1) / kBuildItems;
          n -= __shfl_sync(0xffffffffu, upto - mine, src);
          h = n / per_head;
          const int first = (n - h * per_head) * kBuildItems + lane, page = __shfl_sync(0xffffffffu, p0, src) + first;
          if (lane < kBuildItems && first < end && page >= 0) {
            it_block = p.block_table[(int64_t)(b0 + src) * p.Pmax + page];
            if (it_block < 0 || it_block >= p.num_blocks) { it_block = -1; set_status(p.status, LOCKS_ERR_BAD_BLOCK); }
          }
          break;
        }
        n -= __shfl_sync(0xffffffffu, upto, 31);
      }
    }
    if (W > 1) {   // one warp looks the items up: the warps of a group agree on them, whatever happens to the table meanwhile
      if (warp == 0 && lane < kBuildItems) blk_s[lane] = it_block;
      if (warp == 0 && lane == 0) blk_s[kBuildItems] = h;
      __syncthreads();
      it_block = lane < kBuildItems ? blk_s[lane] : -1;
      h = blk_s[kBuildItems];
    }
    const uint32_t live = __ballot_sync(0xffffffffu, it_block >= 0);
    if (live)
      build_i4_group<W>(p, smem_raw, tid, it_block, live,
                        reinterpret_cast<const __nv_bfloat16 *>(p.k_layers ? p.k_layers[layer] : p.k) + (int64_t)h * p.sh,
                        (p.summ_layers ? reinterpret_cast<uint8_t *>(p.summ_layers[layer]) : p.summ) + (int64_t)h * p.S);
    if (W > 1) __syncthreads();   // the group's shared memory is free
    else __syncwarp();
  }
}

__global__ void __launch_bounds__(kI4Warps * 32, kI4CtasPerSm) build_i4_kernel(BuildParams p, int layers, int sms) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  int *count = reinterpret_cast<int *>(smem_raw + kI4Warps * (kBuildScratch + kI4Group));
  if (threadIdx.x < 32) {
    int n = 0, p0;
    for (int b = threadIdx.x; b < p.batch; b += 32) n += (build_pages(p, b, p0) + kBuildItems - 1) / kBuildItems * p.Hkv;
    n = __reduce_add_sync(0xffffffffu, n);
    if (threadIdx.x == 0) *count = n;
  }
  __syncthreads();
  const int groups = *count;
  if (groups == 0) return;
  // Two warps a group up to 22 groups per SM (1.4 waves of single ones, 2.8 of pairs): us with one / two at 128 groups 104 / 80,
  // 1024: 168 / 131, 2048: 216 / 201, 3072: 294 / 284, 4096: 348 / 349, 16 376: 1126 / 1153.
  if ((int64_t)groups * layers <= (int64_t)kI4Pairs * sms) build_i4_groups<2>(p, smem_raw, count, layers);
  else build_i4_groups<1>(p, smem_raw, count, layers);
}

template <typename T, int FMT>
__global__ void __launch_bounds__(kBuildWarps * 32, kBuildCtasPerSm) build_kernel(BuildParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int h = blockIdx.y;
  const int it_block = item_block(p, blockIdx.z % p.batch, blockIdx.x * kBuildWarps + warp, lane);   // the warp's items: lane s < 8 works out item s
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
  jacobi_phase<false, 4>(mat, mat, lam_s, live, r, lane, 0, [](bool bad) { return __any_sync(0xffffffffu, bad) != 0; });

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

// ------------------------------------------------------------------------------------------------
// Pages of 32 and 64 tokens (App. D "Page size"): one warp per (page, KV head), everything in fp32 from shared
// memory, the row-major summary formats only.  The same method as above (centre, Gram, one-sided Jacobi by
// odd-even transposition, rank, project, quantise), written for brevity rather than speed: lane m rotates the
// column pair m of a step.
// ------------------------------------------------------------------------------------------------
constexpr int kWideDStride = LOCKS_D + 4;   // floats per staged key row (16-byte aligned rows, no bank conflicts)
__host__ __device__ constexpr int build_wide_smem(int B) {
  return (B * kWideDStride + B * (B + 1) + 2 * B + 32) * 4;   // keys, W (column-major, padded), norms, order, misc
}

template <typename T, int FMT>
__global__ void __launch_bounds__(32) build_wide_kernel(BuildParams p, int B) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int lane = threadIdx.x;
  const int b = blockIdx.z, h = blockIdx.y;
  const int complete = p.seq_lens[b] / B;
  const int p0 = p.page_begin ? p.page_begin[b] : 0;
  const int p1 = min(p.page_end ? p.page_end[b] : complete, complete);
  const int page = p0 + blockIdx.x;
  if (page < 0 || page >= p1) return;
  if (page >= p.Pmax) return;
  const int block = p.block_table[(int64_t)b * p.Pmax + page];
  if (block < 0 || block >= p.num_blocks) {
    if (lane == 0) set_status(p.status, LOCKS_ERR_BAD_BLOCK);
    return;
  }
  float *Ds = reinterpret_cast<float *>(smem_raw);   // [B][kWideDStride] deviations
  float *W = Ds + B * kWideDStride;                  // [B columns][B + 1]
  float *nr = W + B * (B + 1);                       // [B] squared column norms
  int *order = reinterpret_cast<int *>(nr + B);      // [B] column of rank l
  const int WS = B + 1, r = p.r;
  // ---- keys, centroid, deviations
  float mu[4] = {0.f, 0.f, 0.f, 0.f}, knorm2 = 0.f;
  {
    const T *K = reinterpret_cast<const T *>(p.k) + ((int64_t)block * p.sb + (int64_t)h * p.sh) + 4 * lane;
    for (int i = 0; i < B; ++i) {
      const T *src = K + (int64_t)i * p.st;
      float v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = ldf<T>(src, c);
#pragma unroll
      for (int c = 0; c < 4; ++c) { mu[c] += v[c]; knorm2 = fmaf(v[c], v[c], knorm2); }
      *reinterpret_cast<float4 *>(Ds + i * kWideDStride + 4 * lane) = make_float4(v[0], v[1], v[2], v[3]);
    }
    knorm2 = warp_sum(knorm2);
#pragma unroll
    for (int c = 0; c < 4; ++c) mu[c] /= (float)B;
    for (int i = 0; i < B; ++i) {
      float4 *d4 = reinterpret_cast<float4 *>(Ds + i * kWideDStride + 4 * lane);
      float4 v = *d4;
      v.x -= mu[0]; v.y -= mu[1]; v.z -= mu[2]; v.w -= mu[3];
      *d4 = v;
    }
    __syncwarp();
  }
  // ---- Gram matrix: lane j (and j + 32) computes column j of M, row by row
  float amax = 0.f;
  for (int jj = lane; jj < B; jj += 32) {
    for (int i = 0; i < B; ++i) {
      const float4 *di = reinterpret_cast<const float4 *>(Ds + i * kWideDStride);
      const float4 *dj = reinterpret_cast<const float4 *>(Ds + jj * kWideDStride);
      float acc = 0.f;
#pragma unroll 8
      for (int c = 0; c < LOCKS_D / 4; ++c) {
        const float4 x = di[c], y = dj[c];
        acc = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, acc))));
      }
      W[jj * WS + i] = acc;
      amax = fmaxf(amax, fabsf(acc));
    }
  }
  amax = warp_max(amax);
  // unit scale (an exact power of two, undone on the eigenvalues)
  float unscale = 1.f;
  if (amax > 0.f && amax < INFINITY) {
    int ex;
    (void)frexpf(amax, &ex);
    ex = max(-120, min(120, ex));
    const float sc = ldexpf(1.f, -ex);
    unscale = ldexpf(1.f, ex);
    for (int jj = lane; jj < B; jj += 32)
      for (int i = 0; i < B; ++i) W[jj * WS + i] *= sc;
  }
  __syncwarp();
  // ---- one-sided Jacobi, odd-even transposition, rotate then swap
  const float tol2 = LOCKS_BUILD_COS_TOL * LOCKS_BUILD_COS_TOL;
  for (int sweep = 0; sweep < 2 * LOCKS_BUILD_SWEEPS; ++sweep) {
    float nm = 0.f;
    for (int jj = lane; jj < B; jj += 32) {
      float a = 0.f;
      for (int i = 0; i < B; ++i) a = fmaf(W[jj * WS + i], W[jj * WS + i], a);
      nr[jj] = a;
      nm = fmaxf(nm, a);
    }
    const float floor_n = 1e-11f * warp_max(nm);
    __syncwarp();
    int bad = 0;
    for (int st = 0; st < B; ++st) {
      const int pc = 2 * lane + (st & 1), qc = pc + 1;   // the pair of this lane
      if (qc < B) {
        float *wp = W + pc * WS, *wq = W + qc * WS;
        const float a = nr[pc], bq = nr[qc];
        float g = 0.f;
        for (int i = 0; i < B; ++i) g = fmaf(wp[i], wq[i], g);
        bad |= (int)(g * g > tol2 * a * bq) & (int)(fminf(a, bq) > floor_n);
        float c, sn;
        plane_rotation(a, bq, g, c, sn);
        for (int i = 0; i < B; ++i) {
          const float x = wp[i], y = wq[i];
          wp[i] = fmaf(sn, x, c * y);    // q' takes p's place
          wq[i] = fmaf(c, x, -sn * y);   // p' takes q's place
        }
        nr[pc] = fmaxf(fmaf(sn * sn, a, fmaf(c * c, bq, 2.f * c * sn * g)), 0.f);
        nr[qc] = fmaxf(fmaf(c * c, a, fmaf(sn * sn, bq, -2.f * c * sn * g)), 0.f);
      }
      __syncwarp();
    }
    if (!__any_sync(0xffffffffu, bad != 0)) break;
  }
  // ---- exact norms, ranking (descending, ties to the lower position)
  for (int jj = lane; jj < B; jj += 32) {
    float a = 0.f;
    for (int i = 0; i < B; ++i) a = fmaf(W[jj * WS + i], W[jj * WS + i], a);
    nr[jj] = a;
  }
  __syncwarp();
  for (int jj = lane; jj < B; jj += 32) {
    const float mine = nr[jj];
    int rk = 0;
    for (int o = 0; o < B; ++o) rk += (nr[o] > mine) || (nr[o] == mine && o < jj);
    order[rk] = jj;
  }
  __syncwarp();
  const float lam0 = sqrtf(nr[order[0]]) * unscale;
  int r_eff = 0;
  const int rmax = min(r, B - 1);
  for (int l = 0; l < rmax; ++l) {
    const float ll = sqrtf(nr[order[l]]) * unscale;
    if (lam0 > 0.f && ll > 1e-6f * lam0 && ll > 1e-10f * knorm2) r_eff = l + 1; else break;
  }
  uint8_t *gout = p.summ + ((int64_t)block * p.Hkv + h) * p.S;
  float *fout = reinterpret_cast<float *>(gout);
  constexpr int WD = FMT == LOCKS_FMT_BF16 ? 2 : 1;
  uint32_t sign_bits = 0u;
  for (int l = 0; l < r; ++l) {
    float v[4] = {0.f, 0.f, 0.f, 0.f}, best = 0.f;
    if (l < r_eff) {
      const int col = order[l];
      const float n2 = nr[col], lam = sqrtf(n2) * unscale;
      const float inv = rsqrtf(n2) * rsqrtf(lam);   // unit eigenvector entries, then 1 / sigma
      for (int i = 0; i < B; ++i) {
        const float u = W[col * WS + i];
        const float4 d4 = *reinterpret_cast<const float4 *>(Ds + i * kWideDStride + 4 * lane);
        v[0] = fmaf(d4.x, u, v[0]); v[1] = fmaf(d4.y, u, v[1]); v[2] = fmaf(d4.z, u, v[2]); v[3] = fmaf(d4.w, u, v[3]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] *= inv;
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
    } else if (FMT == LOCKS_FMT_BF16) {
      *reinterpret_cast<uint2 *>(gout + 2 * (l * LOCKS_D + lane * 4)) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
    } else if (FMT == LOCKS_FMT_I8) {
      const __half sh = __float2half_rn(best / 127.f);
      const float sc = inv_scale(__half2float(sh));
      if (lane == 0) *reinterpret_cast<__half *>(gout + wb_off_sv(r, 1, B) + 2 * l) = sh;
      uint32_t wd = 0u;
#pragma unroll
      for (int c = 0; c < 4; ++c) wd |= (uint32_t)((int)round_code(v[c], sc, 127.f) + 128) << (8 * c);
      *reinterpret_cast<uint32_t *>(gout + l * LOCKS_D + lane * 4) = wd;
    } else {   // int4 basis: the same nibble order as at B = 16
      const __half sh = __float2half_rn(best / 7.f);
      const float sc = inv_scale(__half2float(sh));
      if (lane == 0) *reinterpret_cast<__half *>(gout + i4_off_sv(r, B) + 2 * l) = sh;
      const int t = lane >> 3, s8 = lane & 7, i0 = (s8 & 1) << 1;
      uint32_t nb[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) nb[c] = (uint32_t)((int)round_code(v[c], sc, 7.f) + 8);
      uint32_t pw = (nb[0] << (4 * i0)) | (nb[1] << (4 * (i0 + 4))) | (nb[2] << (4 * (i0 + 1))) | (nb[3] << (4 * (i0 + 5)));
      pw |= __shfl_xor_sync(0xffffffffu, pw, 1);
      if ((s8 & 1) == 0) *reinterpret_cast<uint32_t *>(gout + (l * 4 + t) * 16 + (s8 >> 1) * 4) = pw;
    }
  }
  // coefficients: lane owns tokens lane and lane + 32
  for (int tok = lane; tok < B; tok += 32) {
    float mx = 0.f;
    for (int l = 0; l < r; ++l) {
      float c = 0.f;
      if (l < r_eff) {
        const int col = order[l];
        c = W[col * WS + tok] * rsqrtf(nr[col]) * sqrtf(sqrtf(nr[col]) * unscale);
        if ((sign_bits >> l) & 1u) c = -c;
      }
      mx = fmaxf(mx, fabsf(c));
      if (FMT == LOCKS_FMT_F32) fout[LOCKS_D + r * LOCKS_D + tok * r + l] = c;
    }
    if (FMT != LOCKS_FMT_F32) {
      const __half sh = __float2half_rn(mx / 127.f);
      const float sc = inv_scale(__half2float(sh));
      *reinterpret_cast<__half *>(gout + (FMT == LOCKS_FMT_I4 ? i4_off_sc(r, B) : wb_off_sc(r, WD, B)) + 2 * tok) = sh;
      for (int l = 0; l < r; ++l) {
        float c = 0.f;
        if (l < r_eff) {
          const int col = order[l];
          c = W[col * WS + tok] * rsqrtf(nr[col]) * sqrtf(sqrtf(nr[col]) * unscale);
          if ((sign_bits >> l) & 1u) c = -c;
        }
        gout[(FMT == LOCKS_FMT_I4 ? i4_off_coef(r) : wb_off_coef(r, WD)) + tok * r + l] = (uint8_t)((int)round_code(c, sc, 127.f) + 128);
      }
    }
  }
  // centroid
  if (FMT == LOCKS_FMT_F32) {
    *reinterpret_cast<float4 *>(fout + lane * 4) = make_float4(mu[0], mu[1], mu[2], mu[3]);
  } else {
    float mx = fmaxf(fmaxf(fabsf(mu[0]), fabsf(mu[1])), fmaxf(fabsf(mu[2]), fabsf(mu[3])));
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
    const __half sh = __float2half_rn(mx / 127.f);
    const float sc = inv_scale(__half2float(sh));
    const int osmu = FMT == LOCKS_FMT_I4 ? i4_off_smu(r, B) : wb_off_smu(r, WD, B);
    if (lane == 0) *reinterpret_cast<__half *>(gout + osmu) = sh;
    uint32_t by[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) by[c] = (uint32_t)((int)round_code(mu[c], sc, 127.f) + 128);
    if (FMT == LOCKS_FMT_I4)   // dim offset c = 2*half + e -> byte e*2 + half, as at B = 16
      *reinterpret_cast<uint32_t *>(gout + i4_off_mu(r, B) + lane * 4) = by[0] | (by[2] << 8) | (by[1] << 16) | (by[3] << 24);
    else
      *reinterpret_cast<uint32_t *>(gout + wb_off_mu(r, WD, B) + lane * 4) = by[0] | (by[1] << 8) | (by[2] << 16) | (by[3] << 24);
    for (int e = osmu + 2 + lane; e < p.S; e += 32) gout[e] = 0;
  }
}

}  // namespace

int locks_launch_build(locks_ctx *c, const locks_kv *kv, int batch, const int32_t *pb, const int32_t *pe,
                       int just_filled, void *summaries, const void *k_new, const int32_t *append_pos,
                       cudaStream_t st, bool early, int32_t *seq_commit, const void *const *k_layers, void *const *summ_layers, int num_layers) {
  BuildParams p;
  p.k = kv->k; p.sb = kv->stride_block; p.sh = kv->stride_head; p.st = kv->stride_token;
  p.block_table = kv->block_table; p.seq_lens = kv->seq_lens; p.page_begin = pb; p.page_end = pe;
  p.summ = reinterpret_cast<uint8_t *>(summaries); p.status = c->status;
  p.batch = batch; p.Hkv = c->cfg.num_kv_heads; p.Pmax = c->Pmax; p.num_blocks = kv->num_blocks;
  p.r = c->cfg.rank; p.S = c->S; p.fmt = c->cfg.summary_fmt; p.esz = c->cfg.kv_dtype == LOCKS_BF16 ? 2 : 4;
  p.k_layers = just_filled ? nullptr : k_layers; p.summ_layers = just_filled ? nullptr : summ_layers;
  p.k_new = just_filled ? k_new : nullptr; p.append_pos = just_filled ? append_pos : nullptr;
  p.seq_commit = early ? seq_commit : nullptr; p.arrivals = c->arrivals;
  p.stage = early ? reinterpret_cast<uint8_t *>(c->stage_summ) : nullptr; p.staged = c->staged;
  p.hint = nullptr; p.kpages = c->k; p.hint_wpp = 1; p.hint_rounds = 1; p.hint_W = 1;
  if (just_filled && c->hint_dev && c->cfg.summary_fmt == LOCKS_FMT_I4 && c->cfg.q_dtype == LOCKS_BF16) {
    const locks_scan_geom geo = locks_scan_geometry(c, batch);
    p.hint = c->hint_dev; p.hint_wpp = geo.wpp; p.hint_rounds = geo.rounds; p.hint_W = geo.W;
  }
  if (just_filled) return locks_launch_build_pages(c, p, st);   // a step's few pages: latency counts
  if (c->B != LOCKS_B) {   // pages of 32 / 64 tokens: the plain kernel (row-major formats; one layer per launch)
    if (k_layers) return LOCKS_ERR_UNSUPPORTED;
    const int B = c->B, smem = build_wide_smem(B);
    const dim3 grid(c->Pmax, p.Hkv, batch);
    const bool bf16kv = c->cfg.kv_dtype == LOCKS_BF16;
#define LOCKS_WIDE_CASE(F_)                                                                                              \
  do {                                                                                                                  \
    if (locks_attrs_needed(LOCKS_ATTR_BUILD_WIDE + F_)) {                                                                \
      cudaFuncSetAttribute(build_wide_kernel<__nv_bfloat16, F_>, cudaFuncAttributeMaxDynamicSharedMemorySize, build_wide_smem(64)); \
      cudaFuncSetAttribute(build_wide_kernel<float, F_>, cudaFuncAttributeMaxDynamicSharedMemorySize, build_wide_smem(64));         \
    }                                                                                                                   \
    if (bf16kv) build_wide_kernel<__nv_bfloat16, F_><<<grid, 32, smem, st>>>(p, B);                        \
    else build_wide_kernel<float, F_><<<grid, 32, smem, st>>>(p, B);                                       \
  } while (0)
    switch (c->cfg.summary_fmt) {
      case LOCKS_FMT_I4: LOCKS_WIDE_CASE(LOCKS_FMT_I4); break;
      case LOCKS_FMT_I8: LOCKS_WIDE_CASE(LOCKS_FMT_I8); break;
      case LOCKS_FMT_BF16: LOCKS_WIDE_CASE(LOCKS_FMT_BF16); break;
      default: LOCKS_WIDE_CASE(LOCKS_FMT_F32); break;
    }
#undef LOCKS_WIDE_CASE
    return locks_check_launch(c);
  }
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
      if (bf) {
        // Rows that can all be full (no page ranges, and a pool that holds them) and are many waves long are taken as they
        // are: finding a group's place costs 3 % (8 x 32K tokens, 8 KV heads: 1094 us against 1126).  A pool can hold more than
        // the batch uses; the grid's order then keeps most of what dealing out would save (build_i4_table_kernel).  Otherwise the
        // CTAs of empty rows cost more, in launches and in how the others are spread: a chunk of 128 of 512 pages in 32
        // layers, 386 us by rows against 343.
        const int layers = k_layers ? num_layers : 1;
        const int64_t rows = (int64_t)batch * c->Pmax, most = (int64_t)((c->Pmax + kBuildItems - 1) / kBuildItems) * p.Hkv * batch * layers;
        if (!pb && 4 * rows <= 5 * (int64_t)kv->num_blocks && most > 64 * (int64_t)c->num_sms && grid.x <= 65535)
          build_i4_table_kernel<<<dim3(p.Hkv, batch * layers, grid.x), kI4Warps * 32, kI4Smem, st>>>(p);
        else
        {
          // A CTA per two groups, as many as the pool's blocks can make up: rounds of a smaller grid let the warps drift apart
          // (163 840 groups in 16 waves of CTAs 14.9 ms, in one round 13.4).  With page ranges few of the rows' groups may
          // be there: at most 32 waves, so that the empty ones cost no more than some 30 us.
          const int64_t groups = std::min(most, (kv->num_blocks / kBuildItems + (int64_t)batch) * p.Hkv * layers);
          int64_t ctas = std::max((groups + 1) / 2, std::min<int64_t>(groups, (int64_t)kI4Pairs * c->num_sms));
          if (pb) ctas = std::min<int64_t>(ctas, (int64_t)kI4Waves * kI4CtasPerSm * c->num_sms);
          build_i4_kernel<<<(unsigned)std::min<int64_t>(ctas, INT32_MAX), kI4Warps * 32, kI4SmemCount, st>>>(p, layers, c->num_sms);
        }
      }
      else build_kernel<float, LOCKS_FMT_I4><<<grid, kBuildWarps * 32, smem, st>>>(p);
      break;
    case LOCKS_FMT_I8: LOCKS_BUILD_CASE(LOCKS_FMT_I8); break;
    case LOCKS_FMT_BF16: LOCKS_BUILD_CASE(LOCKS_FMT_BF16); break;
    default: LOCKS_BUILD_CASE(LOCKS_FMT_F32); break;
  }
#undef LOCKS_BUILD_CASE
  return locks_check_launch(c);
}
