// Summary build of the pages that a decode step has just filled (any page size).  The method is that of build.cu (Sec. 4
// "Build"); here the latency of one page counts, because the step that filled it ends with its summary.  The solver is another
// one, so a bulk build of the same page differs in about one byte in ten thousand (this one is the nearer to fp64: 7e-5 of the
// bytes differ from such a build, of the bulk build's 1.2e-4).
//
// What bounds it is one dependent chain, the eigenproblem of the B x B Gram matrix M.  One warp solves it by one-sided
// Jacobi in registers: a pair of columns belongs to L lanes that hold B / L rows of both, so a step (B / 2 pairs at once)
// is a dot product, log2(L) shuffles, the angle, the rotation, and one column passed to the neighbouring pair.  Two
// things keep the number of sweeps down: a QR factorisation with column pivoting first (Drmac and Veselic's
// preconditioning: Jacobi then runs on the columns of R^T, whose left singular vectors are the eigenvectors of M), and a
// stop test that looks only at pairs with one of the r modes that are kept (emulated in fp32 on this repository's
// synthetic pages: 7.7 -> 4.9 sweeps at B = 16 and r = 8, 3.0 at r = 2, 8.5 -> 5.1 at B = 32; worst eigenvector entry
// 1e-4 -> 4e-5 from fp64).  Measured beside a running selector and attention, from the launch to the last store: B = 16,
// r = 8 31 -> 22 us, of it the Jacobi sweeps 19 -> 10 (226 cycles a step), the factorisation 3, the basis 3.5; r = 2 27 -> 18
// us; B = 32 400 -> 47 us.  Steps that a page fills: 8 x 32K 64.5 -> 59.2 us, 32 x 16K at r = 2 75.3 -> 62.4, 4 x 16K with
// 32-token pages 497 -> 176.
//
// The other phases use all of the page's threads (keys and centroid: one or two dimensions each; Gram matrix: dimensions
// dealt to the warps; basis and quantisation: a warp per mode), in short loops: a freshly filled page finds this code in
// no cache.
#include "build_common.cuh"

namespace {

// A page belongs to 64 (B = 64: 128) threads; a CTA takes several, so that a step's build displaces few of the attention
// CTAs that run beside it (24 requests, 2 of them filling a page, 576 attention CTAs in 592 slots: step 65.1 us with a CTA
// of 128 threads per page).
__host__ __device__ constexpr int page_threads(int B) { return B == 64 ? 128 : 64; }
__host__ __device__ constexpr int page_ctas(int B) { return 64 / B; }   // pages per CTA
__host__ __device__ constexpr int dt_stride(int B) { return B + 4; }   // floats per dimension: 16-byte aligned rows, no bank conflicts

template <int B> struct PageShared {
  static constexpr int KS = B == 64 ? 1 : 2;   // slices of the dimensions in the Gram matrix
  float dt[LOCKS_D * dt_stride(B)];   // deviations, [dimension][token]
  float m[2][B * B];                  // Gram matrix (partial sums; the total in m[0]); R^T of its QR factorisation in m[1]
  float us[16 * B];                   // unit eigenvectors, [mode][token]
  float lam[B];                       // eigenvalues, descending
  float sig[16];                      // singular values with the sign of their mode
  float mx[4], kn[4];
  uint8_t codes[16 * LOCKS_D];        // int4 codes before packing
  int early, solved, pad[2];          // the summary has to wait (BuildParams::stage); the modes are there; a CTA's pages start on 16 bytes
};

static_assert(sizeof(PageShared<16>) % 16 == 0 && sizeof(PageShared<32>) % 16 == 0, "");

// Eigenvectors and eigenvalues of the symmetric matrix m0 * 2^-ex (unit scale), by one warp: sh.us[mode][token] and
// sh.lam[mode] of the modes in descending order (the first min(r, B) are accurate, the rest are not needed).
template <int B> __device__ __forceinline__ void solve_modes(PageShared<B> &sh, float scale, float unscale, int r, int lane) {
  constexpr int L = 64 / B, R = B / L, R2 = R / 2;   // lanes per pair of columns; rows, and packed pairs of rows, per lane
  const int pair = lane / L, row0 = (lane % L) * R;
  const float *m0 = sh.m[0];
  float *lt = sh.m[1];   // [k][j]: column k of R^T
  float2 w[2][R2];   // rows row0 .. of the columns at positions 2 pair, 2 pair + 1
  auto over_rows = [&](float v) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  auto dot = [&](const float2 (&a)[R2], const float2 (&b)[R2]) {
    float2 s0 = mul2(a[0], b[0]), s1 = mul2(a[1], b[1]);
#pragma unroll
    for (int i = 2; i < R2; i += 2) { s0 = fma2(a[i], b[i], s0); s1 = fma2(a[i + 1], b[i + 1], s1); }
    return over_rows((s0.x + s1.x) + (s0.y + s1.y));
  };
  auto load = [&](const float *src, float sc) {
    const float2 sc2 = make_float2(sc, sc);
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int i = 0; i < R2; i += 2) {
        const float4 f = *reinterpret_cast<const float4 *>(src + (2 * pair + c) * B + row0 + 2 * i);
        w[c][i] = mul2(make_float2(f.x, f.y), sc2);
        w[c][i + 1] = mul2(make_float2(f.z, f.w), sc2);
      }
  };
  load(m0, scale);
  float n[2];
  n[0] = dot(w[0], w[0]);
  n[1] = dot(w[1], w[1]);
  __syncwarp();
  // ---- QR with column pivoting (modified Gram-Schmidt; only R is kept).  The norms that choose the pivot are downdated;
  // the pivot's own is exact.
  {
    bool used[2] = {false, false};
#pragma unroll 1
    for (int k = 0; k < B; ++k) {
      // largest remaining column: the norm's bits with the column's index in the lowest six; + 64 so that 0 means "used"
      uint32_t key[2];
#pragma unroll
      for (int c = 0; c < 2; ++c)
        key[c] = used[c] ? 0u : ((__float_as_uint(fmaxf(n[c], 0.f)) & ~63u) + 64u) | (uint32_t)(2 * pair + c);
      const uint32_t best = __reduce_max_sync(0xffffffffu, max(key[0], key[1]));
      const int col = (int)(best & 63u), src = (col >> 1) * L + lane % L;
      float2 pv[R2];
#pragma unroll
      for (int i = 0; i < R2; ++i) {
        const float2 mine = (best & 1u) ? w[1][i] : w[0][i];
        pv[i].x = __shfl_sync(0xffffffffu, mine.x, src);
        pv[i].y = __shfl_sync(0xffffffffu, mine.y, src);
      }
      const float pp = dot(pv, pv), g0 = dot(w[0], pv), g1 = dot(w[1], pv);
      const float ir = pp > 1e-37f ? rsqrt_approx(pp) : 0.f;
      float rk[2] = {g0 * ir, g1 * ir};
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (used[c]) rk[c] = 0.f;
        if (2 * pair + c == col) { used[c] = true; rk[c] = pp * ir; }
        const float f = -rk[c] * ir;
        const float2 f2 = make_float2(f, f);
#pragma unroll
        for (int i = 0; i < R2; ++i) w[c][i] = fma2(f2, pv[i], w[c][i]);
        n[c] = fmaf(-rk[c], rk[c], n[c]);
      }
      if (lane % L == 0) *reinterpret_cast<float2 *>(lt + k * B + 2 * pair) = make_float2(rk[0], rk[1]);
    }
  }
  __syncwarp();
  load(lt, 1.f);
  const float tol2 = LOCKS_BUILD_COS_TOL * LOCKS_BUILD_COS_TOL;
  int rank[2];
  auto ranks = [&]() {   // norms, and the positions of this lane's columns in descending order of norm
    uint32_t *keys = reinterpret_cast<uint32_t *>(sh.codes), key[2];   // the norm's bits, ties broken by the column
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      n[c] = dot(w[c], w[c]);
      rank[c] = 0;
      key[c] = (__float_as_uint(n[c]) & ~63u) | (uint32_t)(2 * pair + c);
    }
    __syncwarp();
    if (row0 == 0) *reinterpret_cast<uint2 *>(keys + 2 * pair) = make_uint2(key[0], key[1]);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < B / 4; ++q) {
      const uint4 o = reinterpret_cast<const uint4 *>(keys)[q];
#pragma unroll
      for (int c = 0; c < 2; ++c) rank[c] += (int)(o.x > key[c]) + (int)(o.y > key[c]) + (int)(o.z > key[c]) + (int)(o.w > key[c]);
    }
  };
#pragma unroll 1
  for (int sweep = 0; sweep < (B == LOCKS_B ? 1 : 2) * LOCKS_BUILD_SWEEPS; ++sweep) {
    ranks();
    // pairs count for the stop test if one of them is among the r largest columns and neither is below the modes that are
    // kept (squared norm = squared eigenvalue: those above 1e-6 of the largest are).  A mode that is kept before its column has met
    // the largest one leans on it, and its basis vector, divided by its own small singular value, grows up to 300 times too long.
    const uint32_t b0 = __float_as_uint(n[0]), b1 = __float_as_uint(n[1]);
    const float top = __uint_as_float(__reduce_min_sync(0xffffffffu, min(rank[0] < r ? b0 : 0x7F7FFFFFu, rank[1] < r ? b1 : 0x7F7FFFFFu))) * 0.999f;
    const float floor_n = 5e-13f * __uint_as_float(__reduce_max_sync(0xffffffffu, max(b0, b1)));
    // Odd-even transposition: a rotated pair swaps places, which lets every two columns meet once in B steps.  w[0] is the
    // column that a pair keeps from the step before, w[1] the one that it has been passed; which of the two is the lower
    // position alternates, and so do the signs of the rotation and of the swap, which leaves one formula for every step.
    // In odd steps the last pair holds the two ends of the row, which do not meet.
    int bad = 0;
#pragma unroll 1
    for (int st = 0; st < B; ++st) {
      const float na = n[0], nb = n[1];
      const float g = dot(w[0], w[1]);
      const bool live = !((st & 1) && pair == B / 2 - 1);
      bad |= (int)live & (int)(g * g > tol2 * na * nb) & (int)(fminf(na, nb) > floor_n) & (int)(fmaxf(na, nb) >= top);
      float c, sn, tn;
      jacobi_angle(nb, na, g, c, sn, tn);
      c = live ? c : 0.f;
      sn = live ? sn : -1.f;
      tn = live ? tn * g : nb - na;
      const float2 C2 = make_float2(c, c), S2 = make_float2(sn, sn), F2 = make_float2(-sn, -sn);
      const int from = (st & 1) ? lane - L : lane + L;
#pragma unroll
      for (int i = 0; i < R2; ++i) {
        const float2 keep = fma2(C2, w[1][i], mul2(F2, w[0][i])), pass = fma2(C2, w[0][i], mul2(S2, w[1][i]));
        w[0][i] = keep;
        w[1][i].x = __shfl_sync(0xffffffffu, pass.x, from);
        w[1][i].y = __shfl_sync(0xffffffffu, pass.y, from);
      }
      n[0] = fmaxf(nb - tn, 0.f);
      n[1] = __shfl_sync(0xffffffffu, fmaxf(na + tn, 0.f), from);
    }
    if (!__any_sync(0xffffffffu, bad != 0)) break;
  }
  ranks();
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float inv = n[c] > 0.f ? rsqrtf(n[c]) : 0.f;
    if (row0 == 0) sh.lam[rank[c]] = sqrtf(n[c]) * unscale;
    if (rank[c] < 16)
#pragma unroll
      for (int i = 0; i < R2; i += 2)
        *reinterpret_cast<float4 *>(sh.us + rank[c] * B + row0 + 2 * i) =
            make_float4(w[c][i].x * inv, w[c][i].y * inv, w[c][i + 1].x * inv, w[c][i + 1].y * inv);
  }
}

template <int B>
__global__ void __launch_bounds__(page_threads(B) * page_ctas(B)) build_page_kernel(BuildParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  constexpr int NT = page_threads(B), PPC = page_ctas(B), DS = dt_stride(B), NW = NT / 32, DPT = LOCKS_D / NT;
  const int sub = threadIdx.x / NT, tid = threadIdx.x % NT, lane = tid & 31, warp = tid >> 5, r = p.r;
  PageShared<B> &sh = reinterpret_cast<PageShared<B> *>(smem_raw)[sub];
  auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(sub + 1), "n"(NT) : "memory"); };   // the page's threads
  if (p.seq_commit) {
    // The lengths are about to change, and the suggestion does not depend on them: a tensor scan that leaves room for this kernel
    // has a warp for every group, and then the strided partition takes one round.
    if (p.hint && blockIdx.x == 0 && threadIdx.x == 0) *p.hint = LOCKS_PARTITION_STRIDED;
  } else if (p.hint && blockIdx.x == 0 && threadIdx.x < 32)
    locks_update_partition_hint(p.hint, p.seq_lens, p.batch, p.Hkv, p.kpages, p.hint_wpp, p.hint_rounds, p.hint_W, lane);
  const int prob = blockIdx.x * PPC + sub;
  if (prob >= p.batch * p.Hkv) return;
  const int b = prob / p.Hkv, h = prob - b * p.Hkv;
  int Tb = p.seq_lens[b], at_new = p.append_pos ? p.append_pos[b] : -1;
  if (p.seq_commit) {
    sync();   // every thread of the page has read the length
    const bool room = Tb < p.Pmax * B;   // a sequence that has no room for the token keeps its length
    at_new = room ? Tb : -1;
    Tb += room;
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(p.arrivals + b, 1) == p.Hkv) { p.arrivals[b] = 0; p.seq_commit[b] = Tb; }
    }
  }
  if (Tb <= 0 || (Tb & (B - 1)) != 0) return;
  const int page = Tb / B - 1;
  const bool last_from_new = p.k_new && at_new == Tb - 1;   // the last row is this step's token
  if (page >= p.Pmax) return;
  const int block = p.block_table[(int64_t)b * p.Pmax + page];
  if (block < 0 || block >= p.num_blocks) {
    if (tid == 0) set_status(p.status, LOCKS_ERR_BAD_BLOCK);
    return;
  }
  // ---- keys (thread t: dimensions t, t + NT ..), centroid, deviations
  float mu[DPT];
  {
    float v[DPT][B], kn = 0.f;
    const int64_t base = (int64_t)block * p.sb + (int64_t)h * p.sh + tid, nbase = ((int64_t)b * p.Hkv + h) * LOCKS_D + tid;
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const bool nw = last_from_new && i == B - 1;
      const void *src = nw ? p.k_new : p.k;
      const int64_t at = nw ? nbase : base + (int64_t)i * p.st;
#pragma unroll
      for (int u = 0; u < DPT; ++u)
        v[u][i] = p.esz == 2 ? __uint_as_float((uint32_t)reinterpret_cast<const uint16_t *>(src)[at + u * NT] << 16)
                             : reinterpret_cast<const float *>(src)[at + u * NT];
    }
#pragma unroll
    for (int u = 0; u < DPT; ++u) {
      mu[u] = 0.f;
#pragma unroll
      for (int i = 0; i < B; ++i) { mu[u] += v[u][i]; kn = fmaf(v[u][i], v[u][i], kn); }
      mu[u] *= 1.f / B;
#pragma unroll
      for (int i = 0; i < B; i += 4)
        *reinterpret_cast<float4 *>(sh.dt + (tid + u * NT) * DS + i) =
            make_float4(v[u][i] - mu[u], v[u][i + 1] - mu[u], v[u][i + 2] - mu[u], v[u][i + 3] - mu[u]);
    }
    kn = warp_sum(kn);
    if (lane == 0) sh.kn[warp] = kn;
    if (tid == 0) sh.solved = 0;
  }
  sync();
  float knorm2 = 0.f;
#pragma unroll
  for (int w = 0; w < NW; ++w) knorm2 += sh.kn[w];
  // ---- Gram matrix: KS slices of the dimensions, a thread owns TI x TJ entries of its slice's sum
  // (a dimension's entries in 8- and 16-byte loads, the additions in the same order: a step that fills a page of 16 tokens, 1 x 8016
  // tokens, 27.6 -> 26.7 us; entry by entry before, bound by the latency of 64 short iterations)
  {
    constexpr int KS = PageShared<B>::KS, TN = NT / KS, TJ = B == 16 ? 4 : 8, TI = B * B / TN / TJ, NJ = B / TJ;
    const int ks = tid / TN, tt = tid % TN, i0 = (tt / NJ) * TI, j0 = (tt % NJ) * TJ;
    float acc[TI][TJ];
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
      for (int j = 0; j < TJ; ++j) acc[i][j] = 0.f;
    const float *d = sh.dt + ks * (LOCKS_D / KS) * DS;
#pragma unroll(B == 16 ? 8 : 4)
    for (int cc = 0; cc < LOCKS_D / KS; ++cc, d += DS) {
      __align__(16) float x[TI], y[TJ];
#pragma unroll
      for (int i = 0; i < TI; i += 2) *reinterpret_cast<float2 *>(x + i) = *reinterpret_cast<const float2 *>(d + i0 + i);
#pragma unroll
      for (int j = 0; j < TJ; j += 4) *reinterpret_cast<float4 *>(y + j) = *reinterpret_cast<const float4 *>(d + j0 + j);
#pragma unroll
      for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < TJ; ++j) acc[i][j] = fmaf(x[i], y[j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
      for (int j = 0; j < TJ; j += 4)
        *reinterpret_cast<float4 *>(&sh.m[ks][(i0 + i) * B + j0 + j]) = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
    sync();
    float amax = 0.f;
#pragma unroll 2
    for (int e = tid; e < B * B; e += NT) {
      float s = sh.m[0][e];
#pragma unroll
      for (int k = 1; k < KS; ++k) s += sh.m[k][e];
      sh.m[0][e] = s;
      amax = fmaxf(amax, fabsf(s));
    }
    amax = warp_max(amax);
    if (lane == 0) sh.mx[warp] = amax;
  }
  sync();
  if (warp == 0) {   // unit scale (an exact power of two, undone on the eigenvalues)
    float amax = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) amax = fmaxf(amax, sh.mx[w]);
    float scale = 0.f, unscale = 1.f;
    if (amax > 0.f && amax < INFINITY) {
      const int ex = max(-120, min(120, (int)(__float_as_uint(amax) >> 23) - 126));   // amax <= 2^ex
      scale = __uint_as_float((uint32_t)(127 - ex) << 23);
      unscale = __uint_as_float((uint32_t)(127 + ex) << 23);
    }
    solve_modes<B>(sh, scale, unscale, r, lane);
    if (lane == 0) *reinterpret_cast<volatile int *>(&sh.solved) = 1;
  } else if (warp == 1 && lane == 0) {
    // Has the selector come (BuildParams::stage)?  It usually does long before the modes are there; asked here, the answer costs them
    // no time (asked by the warp that solves, at its end, 4 x 16K tokens with 32-token pages: 57.9 us a step, now 56.5).
    int come = p.stage == nullptr;
    for (int i = 0; !come && i < LOCKS_SPIN_LIMIT; ++i) {   // (until the modes are there: nothing waits for the selector)
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(come) : "l"(p.staged + prob) : "memory");
      if (*reinterpret_cast<volatile int *>(&sh.solved)) break;
    }
    sh.early = !come;
  }
  sync();
  // ---- modes kept
  const float lam0 = sh.lam[0];
  int r_eff = 0;
  const int rmax = min(r, B - 1);
  for (int l = 0; l < rmax; ++l) {
    const float ll = sh.lam[l];
    if (lam0 > 0.f && ll > 1e-6f * lam0 && ll > 1e-10f * knorm2) r_eff = l + 1; else break;
  }
  const int fmt = p.fmt, wide = fmt == LOCKS_FMT_BF16 ? 2 : 1;
  uint8_t *const place = p.summ + ((int64_t)block * p.Hkv + h) * p.S, *const gout = sh.early ? p.stage + (int64_t)prob * p.S : place;
  float *fout = reinterpret_cast<float *>(gout);
  // ---- basis V = D^T U Sigma^-1: a warp per mode, a lane owns dimensions lane, lane + 32 ..
#pragma unroll 1
  for (int l = warp; l < r; l += NW) {
    float x[4] = {0.f, 0.f, 0.f, 0.f}, sigma = 0.f;
    if (l < r_eff) {
#pragma unroll 4
      for (int i = 0; i < B; i += 4) {
        const float4 uv = *reinterpret_cast<const float4 *>(sh.us + l * B + i);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 dv = *reinterpret_cast<const float4 *>(sh.dt + (lane + 32 * u) * DS + i);
          x[u] = fmaf(dv.x, uv.x, fmaf(dv.y, uv.y, fmaf(dv.z, uv.z, fmaf(dv.w, uv.w, x[u]))));
        }
      }
      const float inv = rsqrtf(sh.lam[l]);
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] *= inv;
      sigma = sqrtf(sh.lam[l]);
    }
    // sign: the entry of largest magnitude (lowest dimension on ties) is positive
    float best = fabsf(x[0]), bv = x[0];
#pragma unroll
    for (int u = 1; u < 4; ++u) if (fabsf(x[u]) > best) { best = fabsf(x[u]); bv = x[u]; }
    const uint32_t mine = __float_as_uint(best), mx = __reduce_max_sync(0xffffffffu, mine);
    int dim = LOCKS_D;   // this lane's lowest dimension that holds the maximum
#pragma unroll
    for (int u = 3; u >= 0; --u) if (__float_as_uint(fabsf(x[u])) == mx) { dim = lane + 32 * u; bv = x[u]; }
    const int first = __reduce_min_sync(0xffffffffu, dim);
    const float sgn = __shfl_sync(0xffffffffu, bv, first & 31) < 0.f ? -1.f : 1.f;
    best = __uint_as_float(mx);
    if (lane == 0) sh.sig[l] = sgn * sigma;
    if (fmt == LOCKS_FMT_F32) {
#pragma unroll
      for (int u = 0; u < 4; ++u) fout[LOCKS_D + l * LOCKS_D + lane + 32 * u] = sgn * x[u];
    } else if (fmt == LOCKS_FMT_BF16) {
#pragma unroll
      for (int u = 0; u < 4; ++u) reinterpret_cast<__nv_bfloat16 *>(gout)[l * LOCKS_D + lane + 32 * u] = __float2bfloat16_rn(sgn * x[u]);
    } else {
      const float qmax = fmt == LOCKS_FMT_I8 ? 127.f : 7.f;
      const __half s = __float2half_rn(best / qmax);
      const float inv = inv_scale(__half2float(s)) * sgn;
      if (lane == 0) *reinterpret_cast<__half *>(gout + (fmt == LOCKS_FMT_I8 ? wb_off_sv(r, 1, B) : i4_off_sv(r, B)) + 2 * l) = s;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int code = (int)round_code(x[u], inv, qmax);
        if (fmt == LOCKS_FMT_I8) gout[l * LOCKS_D + lane + 32 * u] = (uint8_t)(code + 128);
        else sh.codes[l * LOCKS_D + lane + 32 * u] = (uint8_t)(code + 8);
      }
      if (fmt == LOCKS_FMT_I4) {   // eight consecutive dimensions' codes make one 32-bit word of the basis
        __syncwarp();
        if (lane < 16) {
          const uint2 by = *reinterpret_cast<const uint2 *>(sh.codes + l * LOCKS_D + 8 * lane);
          uint32_t word = 0u;
#pragma unroll
          for (int q = 0; q < 8; ++q) {   // dimension q: s = q >> 2, half = (q >> 1) & 1, e = q & 1
            const uint32_t code = ((q < 4 ? by.x : by.y) >> (8 * (q & 3))) & 15u;
            word |= code << (4 * ((q >> 1) + 4 * (q & 1)));
          }
          reinterpret_cast<uint32_t *>(gout)[l * 16 + lane] = word;
        }
      }
    }
  }
  float mm = 0.f;
#pragma unroll
  for (int u = 0; u < DPT; ++u) mm = fmaxf(mm, fabsf(mu[u]));
  mm = warp_max(mm);
  if (lane == 0) sh.mx[warp] = mm;
  sync();
  // ---- coefficients C = U Sigma: a thread per token
  if (tid < B) {
    float mx = 0.f;
#pragma unroll 4
    for (int l = 0; l < r; ++l) mx = fmaxf(mx, l < r_eff ? fabsf(sh.sig[l] * sh.us[l * B + tid]) : 0.f);
    auto coef = [&](int l) { return l < r_eff ? sh.sig[l] * sh.us[l * B + tid] : 0.f; };
    if (fmt == LOCKS_FMT_F32) {
      for (int l = 0; l < r; ++l) fout[LOCKS_D + r * LOCKS_D + tid * r + l] = coef(l);
    } else {
      const __half s = __float2half_rn(mx / 127.f);
      const float sc = inv_scale(__half2float(s));
      const bool inter = fmt == LOCKS_FMT_I4 && B == LOCKS_B;   // fragment order of the tensor-core scan
      const int spos = inter ? ((tid & 7) >> 1) * 4 + (tid >> 3) * 2 + (tid & 1) : tid;
      *reinterpret_cast<__half *>(gout + (fmt == LOCKS_FMT_I4 ? i4_off_sc(r, B) : wb_off_sc(r, wide, B)) + 2 * spos) = s;
      uint8_t *cd = gout + (fmt == LOCKS_FMT_I4 ? i4_off_coef(r) : wb_off_coef(r, wide));
#pragma unroll 2
      for (int l = 0; l < r; ++l) {
        const int at = inter ? ((tid & 7) * (r / 2) + (l >> 1)) * 4 + (tid >> 3) * 2 + (l & 1) : tid * r + l;
        cd[at] = (uint8_t)((int)round_code(coef(l), sc, 127.f) + 128);
      }
    }
  }
  // ---- centroid
  const int osmu = fmt == LOCKS_FMT_I4 ? i4_off_smu(r, B) : wb_off_smu(r, wide, B);
  mm = sh.mx[0];
#pragma unroll
  for (int w = 1; w < NW; ++w) mm = fmaxf(mm, sh.mx[w]);
  const __half s = __float2half_rn(mm / 127.f);
  const float inv = inv_scale(__half2float(s));
#pragma unroll
  for (int u = 0; u < DPT; ++u) {
    const int c = tid + u * NT;
    const uint8_t code = (uint8_t)((int)round_code(mu[u], inv, 127.f) + 128);
    if (fmt == LOCKS_FMT_F32) fout[c] = mu[u];
    else if (fmt == LOCKS_FMT_I4)   // dim 32 t + 4 s + 2 half + e -> byte 32 t + 4 s + 2 e + half
      gout[i4_off_mu(r, B) + (c & ~3) + 2 * (c & 1) + ((c >> 1) & 1)] = code;
    else
      gout[wb_off_mu(r, wide, B) + c] = code;
  }
  if (fmt != LOCKS_FMT_F32) {
    if (tid == 0) *reinterpret_cast<__half *>(gout + osmu) = s;
    if (osmu + 2 + tid < p.S) gout[osmu + 2 + tid] = 0;   // bytes between the payload and the padded stride stay zero
  }
  if (!p.stage) return;
  if (sh.early) {   // the scan may have ended meanwhile; if not, the selector will find the summary
    sync();
    if (tid == 0) {
      __threadfence();
      sh.early = atomicAdd(p.staged + prob, 1) == 0;
      __threadfence();
    }
    sync();
    if (sh.early) return;
    for (int i = tid; i < p.S / 16; i += NT) reinterpret_cast<uint4 *>(place)[i] = reinterpret_cast<const uint4 *>(gout)[i];
  }
  if (tid == 0) p.staged[prob] = 0;
}

template <int B> int launch_pages(locks_ctx *c, const BuildParams &p, cudaStream_t st) {
  constexpr int PPC = page_ctas(B), smem = PPC * (int)sizeof(PageShared<B>);
  const dim3 grid((p.batch * p.Hkv + PPC - 1) / PPC);
  if (locks_attrs_needed(LOCKS_ATTR_BUILD_PAGE + B / 32))
    cudaFuncSetAttribute(build_page_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  build_page_kernel<B><<<grid, PPC * page_threads(B), smem, st>>>(p);
  return locks_check_launch(c);
}

}  // namespace

int locks_launch_build_pages(locks_ctx *c, const BuildParams &p, cudaStream_t st) {
  return c->B == 64 ? launch_pages<64>(c, p, st) : (c->B == 32 ? launch_pages<32>(c, p, st) : launch_pages<16>(c, p, st));
}
