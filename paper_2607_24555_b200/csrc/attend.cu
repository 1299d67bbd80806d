// Stage B: sparse paged attention over the selected pages (Sec. 3 "Decode-time attention", App. E):
//   o_g = sum_i softmax_i(q_g . k_i / sqrt(d)) v_i   over tokens i < T of the pages in the table,
// computed split-K: every CTA takes a slice of the page list, every warp streams tiles of 16 tokens
// (K 16x128 + V 16x128) through its own two-stage shared-memory ring with 16-byte async
// copies into an XOR-swizzled layout, scores them with m16n8k16 bf16 MMAs (tokens are the rows, the G query heads
// of the KV head the columns), keeps a running (max, sum, O) per head, and the CTA merges its warps by
// log-sum-exp.  The splits of a problem are merged by the thread-block cluster that they form, by the CTA that
// arrives last, or by a second small kernel.  fp32 caches: attend_f32_kernel.
// A NULL page table means "all pages": the same kernels are the dense flash-decode baseline.
#include <mutex>
#include "locks_internal.cuh"

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct AttParams {
  const void *q;
  const void *k, *v;
  int64_t sb, sh, st;
  const int32_t *block_table;
  const int32_t *seq_lens;
  const int32_t *ids, *cnt;
  float *part_o, *part_lse;
  void *out;
  float *lse;
  int32_t *status;
  int32_t *done;   // [batch*Hkv] split-arrival counters (zero between launches)
  int batch, Hq, Hkv, G, Pmax, kbud, num_blocks, splits;
  int B;             // tokens per page
  int sub_shift;     // bf16 kernel, wide pages: a page is 2^sub_shift tiles of 16 tokens (1, 2 for pages of 32, 64 tokens)
  int kvdiv;         // the KV head of problem h is h / kvdiv (1; per-head page tables: G, with G = 1 and Hkv = Hq here)
  int fused_merge;   // 1: the last CTA of a problem merges its splits; 0: a separate merge kernel follows
  uint64_t per_split;   // 2^32 / splits + 1
  int cluster;       // 1: the splits of a problem form one thread-block cluster and merge through its shared memory
  float sm_scale;
};

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

constexpr int kTile = LOCKS_B * LOCKS_D * 2;                 // 4096 B: one K or V page tile in bf16
constexpr int kAttStage = 2 * kTile;                         // K + V
constexpr int kAttStages = LOCKS_ATT_STAGES;                  // ring depth per warp
constexpr int kAttSmem = LOCKS_ATT_WARPS * kAttStages * kAttStage;
// Clusters: behind the rings a CTA keeps room for its slice of the other CTAs' partials (see attend_bf16_kernel).  At most 8 KB, so
// that four CTAs still fit on an SM: 16 heads in slices of at most 15 / 16 of 8 KB, and the (max, sum) of the slice's heads.
constexpr int kAttSmemMost = kAttSmem + 8192;
constexpr int kWarpRow = LOCKS_D + 4;   // floats per head of a warp's partial: the four lanes of a quad on different banks
__host__ __device__ constexpr int slice_heads(int slice) { return (slice + LOCKS_D - 1) / LOCKS_D + 1; }
constexpr int cluster_smem(int G, int splits) {
  const int slice = G * LOCKS_D / splits;   // (at most 16 splits, so a multiple of 8)
  return kAttSmem + ((splits - 1) * slice * 4 + splits * slice_heads(slice) * 8 + 127) / 128 * 128;
}
static_assert(cluster_smem(16, 16) <= kAttSmemMost && cluster_smem(16, 8) <= kAttSmemMost && cluster_smem(15, 16) <= kAttSmemMost, "");
// A single CTA merging many splits of many heads is a serial tail: beyond 64 (head, split) pairs the splits of a problem
// go to the parallel merge kernel.
constexpr int kFusedMerge = 64;

// Length of a slice when n list entries are cut into p.splits: ceil(n / p.splits), n below 2^25, without a division (the kernel for
// more than 8 heads takes 8.4 us for 4 x 32 pages and 37.4 for 131K tokens with this; with a division, which costs it registers in
// the loop, 8.7 and 39.1).  Taken from the lengths that the device sees: the table's row (what the host could slice) is
// usually longer than the sequence, and equal slices of the row leave the last CTAs of a problem idle.
__device__ __forceinline__ int slice_length(const AttParams &p, int n) {
  return (int)(((uint64_t)(uint32_t)(n + p.splits - 1) * p.per_split) >> 32);
}

// Resolve a logical page of request b: physical block, valid tokens.
__device__ __forceinline__ bool resolve_page(const AttParams &p, int b, int page, int T, int &block, int &ntok) {
  if (page < 0 || page >= p.Pmax) { set_status(p.status, LOCKS_ERR_BAD_BLOCK); return false; }
  block = p.block_table[(int64_t)b * p.Pmax + page];
  if (block < 0 || block >= p.num_blocks) { set_status(p.status, LOCKS_ERR_BAD_BLOCK); return false; }
  ntok = min(p.B, T - page * p.B);
  return ntok > 0;
}

// ---- thread-block clusters: an address of this CTA's shared memory in CTA `rank` of the cluster, stores to it, the barrier
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_st4(uint32_t a, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void cluster_st2(uint32_t a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t movm_trans_b16(uint32_t v) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(v));
  return d;
}

// Orientation: tokens are the MMA rows.  Per page (16 tokens):
//   S^T[16 tokens x 8 heads]  = K[16 x 128] . q^T[128 x 8]          (8 k-steps, A = K via ldmatrix)
//   O^T[128 dims x 8 heads]  += V^T[128 x 16] . P^T[16 x 8]          (8 row tiles, A = V via ldmatrix.trans,
//                                                                   B = P^T after an 8x8 movmatrix transpose)
// so both products use all 16 rows of the tile and the accumulator is 32 registers per 8 heads.
//
// WIDE: pages of 32 and 64 tokens are two and four such tiles, and the page list is walked tile by tile.  Their weights and sums
// are those of fp32 arithmetic: P goes in as three bf16 parts (24 bits), and since the tensor core truncates what it adds to an
// accumulator, every product starts from zero and is added to the running sum by a rounding fp32 addition.  Against fp64, over 18
// batches at both sizes: outputs 1.38e-3 .. 1.70e-3, all of it the rounding of the result (P in bf16: up to 2.29e-3), log-sum-exp
// 3.3e-7 on average, as an fp32 kernel has it (3.4e-7).  4 x 128 pages of 32 tokens: 12.6 us; P in bf16 11.1, plain fp32 arithmetic
// 18.9 (sums by halves) and 40.6 (a warp reduction per token).
template <int NH, bool CONTIG, bool WIDE>
__global__ void __launch_bounds__(LOCKS_ATT_WARPS * 32, LOCKS_ATT_CTAS_PER_SM) attend_bf16_kernel(AttParams p) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x = lane >> 2, t = lane & 3;
  const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int64_t prob = (int64_t)b * p.Hkv + h;
  const int hkv = h / p.kvdiv;   // head of the cache this problem reads
  uint8_t *ring = smem + warp * kAttStages * kAttStage;
  const uint8_t *Kb = reinterpret_cast<const uint8_t *>(p.k);
  const uint8_t *Vb = reinterpret_cast<const uint8_t *>(p.v);
  pdl_trigger();
  if (p.cluster) cluster_arrive_relaxed();   // "this CTA has started": its shared memory may be written to from here on

  // query as the B operand: lane (x, t) holds head x (+8), dims 16 s + 2t.. and 16 s + 8 + 2t..
  uint32_t qb[NH][8][2];
  {
    const __nv_bfloat16 *q = reinterpret_cast<const __nv_bfloat16 *>(p.q);
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) {
      const int g = x + 8 * hh;
      const uint32_t *qr = reinterpret_cast<const uint32_t *>(q + ((int64_t)b * p.Hq + h * p.G + g) * LOCKS_D);
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        qb[hh][s][0] = (g < p.G) ? __ldg(qr + 8 * s + t) : 0u;
        qb[hh][s][1] = (g < p.G) ? __ldg(qr + 8 * s + 4 + t) : 0u;
      }
    }
  }
  const float c2 = p.sm_scale * kLog2e;
  pdl_wait();   // page table from the selector, appended K/V rows, sequence lengths
  const int T = p.seq_lens[b];
  const int B = WIDE ? p.B : LOCKS_B;
  int npages = p.ids ? p.cnt[prob] : 0;
  const int row = p.ids ? p.kbud : p.Pmax, sub_shift = WIDE ? p.sub_shift : 0;
  // A sparse list is nearly always as long as its row: the page ids that this warp starts with are then fetched together with
  // length and count instead of after them.
  int id_ahead = 0;
  if (p.ids) {
    const int idx = (split * slice_length(p, row << sub_shift) + warp + lane * LOCKS_ATT_WARPS) >> sub_shift;
    if (idx < row) id_ahead = p.ids[prob * p.kbud + idx];
  } else {
    npages = max((T + B - 1) / B, 0);
  }
  if ((p.ids && npages < 0) || npages > row) {   // a count or a length beyond the table's row: use the row, report it
    if (threadIdx.x == 0) set_status(p.status, LOCKS_ERR_BAD_BLOCK);
    npages = npages < 0 ? 0 : row;
  }
  // Dense attention slices all requests by the longest of them, so that the CTAs have equally much to do (16 requests of 3K .. 12K
  // tokens: 82 us in rows of 12K and of 32K tokens; each by its own length 87, by rows of 32K 144).  Not with more than 8 heads:
  // there the loop over the lengths costs the other loop more (131K tokens 37.3 -> 39.7).
  int longest = npages;
  if (NH == 1 && !p.ids) {
#pragma unroll 1
    for (int i = lane; i < p.batch; i += 32) longest = max(longest, (p.seq_lens[i] + B - 1) / B);
    longest = min(__reduce_max_sync(0xffffffffu, longest), p.Pmax);
  }
  const int per = slice_length(p, longest << sub_shift);
  const int lo = split * per, hi = min(lo + per, npages << sub_shift);

  float oacc[8][NH][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) oacc[i][hh][0] = oacc[i][hh][1] = oacc[i][hh][2] = oacc[i][hh][3] = 0.f;
  float mrun[NH][2], lrun[NH][2];   // per head column 2t, 2t+1 (+8): running max, this lane's partial sum
#pragma unroll
  for (int hh = 0; hh < NH; ++hh) { mrun[hh][0] = mrun[hh][1] = -INFINITY; lrun[hh][0] = lrun[hh][1] = 0.f; }

  // per-lane constants of the 16-byte copies: copy i moves chunk (lane & 15) of token (lane >> 4) + 2 i
  const int tok0 = lane >> 4, ch0 = lane & 15;
  const int64_t goff0 = ((int64_t)tok0 * p.st + ch0 * 8) * 2;       // bytes
  const int64_t gstep = p.st * 4;                                    // two token rows, bytes
  uint32_t sw[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) sw[i] = (uint32_t)(tok0 * 256 + (((ch0 ^ tok0) ^ ((2 * i) & 7)) << 4));

  // page ids and physical blocks of this warp's pages are resolved 32 at a time, one lane each, so the
  // two dependent global loads are paid once per batch instead of once per page
  const int first = lo + warp, sub_mask = (1 << sub_shift) - 1;
  auto resolve_batch = [&](int jb, int &blk, int &nt) {
    const int idx = first + (jb + lane) * LOCKS_ATT_WARPS;
    blk = 0;
    nt = 0;
    if (idx < hi) {
      const int page = !p.ids ? idx >> sub_shift : (jb == 0 && npages == row ? id_ahead : p.ids[prob * p.kbud + (idx >> sub_shift)]);
      if (!resolve_page(p, b, page, T, blk, nt)) nt = 0;
    }
    if constexpr (WIDE) nt = min(LOCKS_B, nt - (idx & sub_mask) * LOCKS_B);   // tokens of this tile (none past the sequence's end)
  };
  int blk_cur, nt_cur, blk_nxt = 0, nt_nxt = 0;
  resolve_batch(0, blk_cur, nt_cur);

  const uint64_t pol_stream = l2_policy_evict_first();
  auto issue = [&](int j, int stage) -> int {  // j-th page of this warp; returns its valid tokens
    const int block = __shfl_sync(0xffffffffu, blk_cur, j & 31);
    const int ntok = __shfl_sync(0xffffffffu, nt_cur, j & 31);
    uint8_t *kt = ring + stage * kAttStage, *vt = kt + kTile;
    const int sub = WIDE ? (first + j * LOCKS_ATT_WARPS) & sub_mask : 0;   // tile within its page
    const int64_t base = ((int64_t)block * p.sb + (int64_t)hkv * p.sh + (int64_t)(sub * LOCKS_B) * p.st) * 2 + goff0;
    const uint8_t *kp = Kb + base, *vp = Vb + base;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t so = sw[i & 3] + 512 * i;
      const bool valid = tok0 + 2 * i < ntok;   // rows past the sequence end are zero-filled
      if (LOCKS_ATT_HINT_LOAD) {   // K and V stream through L2 once: they should not push out the small
                                   // tables (lengths, block table, page ids) every kernel of the step re-reads
        if (CONTIG) {   // token rows are 256 bytes apart: immediate offsets
          cp_async16_hint(kt + so, kp + i * 512, valid, pol_stream);
          cp_async16_hint(vt + so, vp + i * 512, valid, pol_stream);
        } else {
          cp_async16_hint(kt + so, kp + i * gstep, valid, pol_stream);
          cp_async16_hint(vt + so, vp + i * gstep, valid, pol_stream);
        }
      } else if (CONTIG) {
        cp_async16(kt + so, kp + i * 512, valid);
        cp_async16(vt + so, vp + i * 512, valid);
      } else {
        cp_async16(kt + so, kp + i * gstep, valid);
        cp_async16(vt + so, vp + i * gstep, valid);
      }
    }
    cp_async_commit();
    return ntok;
  };

  // ring of kAttStages pages per warp: pages j+1 .. j+kAttStages-1 are in flight while page j is used
  const int npg = (hi > first) ? (hi - first + LOCKS_ATT_WARPS - 1) / LOCKS_ATT_WARPS : 0;   // this warp's pages
  int ntok_ring[kAttStages];
#pragma unroll
  for (int s2 = 0; s2 < kAttStages - 1; ++s2) {
    ntok_ring[s2] = 0;
    if (s2 < npg) ntok_ring[s2] = issue(s2, s2); else cp_async_commit();
  }
  ntok_ring[kAttStages - 1] = 0;
  for (int j = 0; j < npg; ++j) {
    const int stage = j % kAttStages;
    if ((j & 31) == 15) resolve_batch((j & ~31) + 32, blk_nxt, nt_nxt);   // next batch, half a batch early
    {
      const int jn = j + kAttStages - 1;   // refill the slot freed by page j-1
      if (((jn) & 31) == 0 && jn > 0) { blk_cur = blk_nxt; nt_cur = nt_nxt; }
      int nt_new = 0;
      if (jn < npg) nt_new = issue(jn, jn % kAttStages); else cp_async_commit();
#pragma unroll
      for (int s2 = 0; s2 < kAttStages; ++s2) if (s2 == jn % kAttStages) ntok_ring[s2] = nt_new;
    }
    cp_async_wait<kAttStages - 1>();
    int ntok_cur = 0;
#pragma unroll
    for (int s2 = 0; s2 < kAttStages; ++s2) if (s2 == stage) ntok_cur = ntok_ring[s2];
    __syncwarp();
    const uint8_t *kt = ring + stage * kAttStage, *vt = kt + kTile;
    const int ntok = ntok_cur;
    const int m = lane >> 3, rr = lane & 7;
    // ---- S^T = K q^T
    float sacc[NH][4];
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) sacc[hh][0] = sacc[hh][1] = sacc[hh][2] = sacc[hh][3] = 0.f;
    {
      const int tok = (m & 1) * 8 + rr;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int ch = 2 * s + (m >> 1);
        uint32_t r[4];
        ldsm_x4(r, kt + tok * 256 + ((ch ^ (tok & 7)) << 4));
#pragma unroll
        for (int hh = 0; hh < NH; ++hh) {
          if constexpr (WIDE) {
            float c[4];
            mma_bf16_z(c, r[0], r[1], r[2], r[3], qb[hh][s][0], qb[hh][s][1]);
#pragma unroll
            for (int e = 0; e < 4; ++e) sacc[hh][e] = s > 0 ? sacc[hh][e] + c[e] : c[e];
          } else {
            mma_bf16(sacc[hh], r[0], r[1], r[2], r[3], qb[hh][s][0], qb[hh][s][1]);
          }
        }
      }
    }
    // ---- online softmax down the token rows; this lane: tokens x, x + 8, heads 2t, 2t+1 (+8)
    uint32_t pb0[NH], pb1[NH], rest0[NH][2], rest1[NH][2];   // P^T; wide pages: its leading and its further parts
    const bool v0ok = x < ntok, v1ok = x + 8 < ntok;
#pragma unroll
    for (int hh = 0; hh < NH; ++hh) {
      float sv[4];
      sv[0] = v0ok ? sacc[hh][0] * c2 : -INFINITY;
      sv[1] = v0ok ? sacc[hh][1] * c2 : -INFINITY;
      sv[2] = v1ok ? sacc[hh][2] * c2 : -INFINITY;
      sv[3] = v1ok ? sacc[hh][3] * c2 : -INFINITY;
      float cm0 = fmaxf(sv[0], sv[2]), cm1 = fmaxf(sv[1], sv[3]);
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        cm0 = fmaxf(cm0, __shfl_xor_sync(0xffffffffu, cm0, o));
        cm1 = fmaxf(cm1, __shfl_xor_sync(0xffffffffu, cm1, o));
      }
      const float mn0 = fmaxf(mrun[hh][0], cm0), mn1 = fmaxf(mrun[hh][1], cm1);
      const float ms0 = (mn0 == -INFINITY) ? 0.f : mn0, ms1 = (mn1 == -INFINITY) ? 0.f : mn1;
      const bool moved = (mn0 != mrun[hh][0]) || (mn1 != mrun[hh][1]);
      if (__any_sync(0xffffffffu, moved)) {   // rescale only when some running max rose
        const float a0 = ex2f(mrun[hh][0] - ms0), a1 = ex2f(mrun[hh][1] - ms1);
        lrun[hh][0] *= a0;
        lrun[hh][1] *= a1;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          oacc[i][hh][0] *= a0; oacc[i][hh][2] *= a0;
          oacc[i][hh][1] *= a1; oacc[i][hh][3] *= a1;
        }
      }
      mrun[hh][0] = mn0;
      mrun[hh][1] = mn1;
      const float p00 = ex2f(sv[0] - ms0), p01 = ex2f(sv[1] - ms1), p10 = ex2f(sv[2] - ms0), p11 = ex2f(sv[3] - ms1);
      lrun[hh][0] += p00 + p10;
      lrun[hh][1] += p01 + p11;
      // P^T rows (tokens) -> B fragment (k = tokens 2t, 2t+1 | 8 + 2t.., n = head x)
      if constexpr (!WIDE) {
        pb0[hh] = movm_trans_b16(pack_bf16(p00, p01));
        pb1[hh] = movm_trans_b16(pack_bf16(p10, p11));
      } else {
        // truncated, so that no part is negative; and none but the first is zero: an infinite value stays infinite
        float w[4] = {p00, p01, p10, p11};
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const uint32_t a = movm_trans_b16(__byte_perm(__float_as_uint(w[0]), __float_as_uint(w[1]), 0x7632));
          const uint32_t c = movm_trans_b16(__byte_perm(__float_as_uint(w[2]), __float_as_uint(w[3]), 0x7632));
          if (u == 0) { pb0[hh] = a; pb1[hh] = c; }
          else { rest0[hh][u - 1] = a; rest1[hh][u - 1] = c; }
#pragma unroll
          for (int e = 0; e < 4; ++e) w[e] = fmaxf(w[e] - __uint_as_float(__float_as_uint(w[e]) & 0xFFFF0000u), 1.17549435e-38f);
        }
      }
    }
    // ---- O^T += V^T P^T
    {
      const int tok = (m >> 1) * 8 + rr;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        const int ch = 2 * mt + (m & 1);
        uint32_t r[4];
        ldsm_x4_trans(r, vt + tok * 256 + ((ch ^ (tok & 7)) << 4));
#pragma unroll
        for (int hh = 0; hh < NH; ++hh) {
          if constexpr (WIDE) {   // the smallest part first
            float c[4];
            mma_bf16_z(c, r[0], r[1], r[2], r[3], rest0[hh][1], rest1[hh][1]);
            mma_bf16(c, r[0], r[1], r[2], r[3], rest0[hh][0], rest1[hh][0]);
            mma_bf16(c, r[0], r[1], r[2], r[3], pb0[hh], pb1[hh]);
#pragma unroll
            for (int e = 0; e < 4; ++e) oacc[mt][hh][e] += c[e];
          } else {
            mma_bf16(oacc[mt][hh], r[0], r[1], r[2], r[3], pb0[hh], pb1[hh]);
          }
        }
      }
    }
    __syncwarp();
  }
  cp_async_wait<0>();
#pragma unroll
  for (int hh = 0; hh < NH; ++hh)
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) lrun[hh][c] += __shfl_xor_sync(0xffffffffu, lrun[hh][c], o);
  __syncthreads();  // every warp is done with its ring: reuse it for the merge
  // a warp's partial: [16 heads][kWarpRow] fp32, then (max, sum) of the 16 heads
  constexpr int NT = LOCKS_ATT_WARPS * 32, kWarpBytes = kAttStages * kAttStage;
  float *wo = reinterpret_cast<float *>(ring);
  float2 *ws = reinterpret_cast<float2 *>(wo + 16 * kWarpRow);
#pragma unroll
  for (int hh = 0; hh < NH; ++hh) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int row = 8 * hh + 2 * t + c;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        wo[row * kWarpRow + 16 * mt + x] = oacc[mt][hh][c];
        wo[row * kWarpRow + 16 * mt + 8 + x] = oacc[mt][hh][2 + c];
      }
      if (x == 0) ws[row] = make_float2(mrun[hh][c], lrun[hh][c]);
    }
  }
  __syncthreads();
  // the CTA's (max, sum) of head g, and the factors of its warps' partials
  auto fold_head = [&](int g, float (&sc)[LOCKS_ATT_WARPS]) -> float2 {
    float2 v[LOCKS_ATT_WARPS];
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int w = 0; w < LOCKS_ATT_WARPS; ++w) {
      v[w] = reinterpret_cast<const float2 *>(smem + w * kWarpBytes + 16 * kWarpRow * 4)[g];
      M = fmaxf(M, v[w].x);
    }
#pragma unroll
    for (int w = 0; w < LOCKS_ATT_WARPS; ++w) {
      sc[w] = M > -INFINITY ? ex2f(v[w].x - M) : 0.f;
      L += v[w].y * sc[w];
    }
    return make_float2(M, L);
  };
  auto fold_dims = [&](int g, int d4, const float (&sc)[LOCKS_ATT_WARPS]) -> float4 {   // dims d4 .. d4 + 3, unnormalised
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < LOCKS_ATT_WARPS; ++w) {
      const float4 v = *reinterpret_cast<const float4 *>(smem + w * kWarpBytes + (g * kWarpRow + d4) * 4);
      o.x += v.x * sc[w]; o.y += v.y * sc[w]; o.z += v.z * sc[w]; o.w += v.w * sc[w];
    }
    return o;
  };
  if (p.cluster) {
    // The splits of this (request, KV head) are the CTAs of one cluster, and CTA r finishes a slice of the problem's G x 128
    // outputs.  Every CTA folds its warps and stores the folded partial, slice by slice, straight into the shared memory of the
    // CTA that finishes it; after one cluster barrier every CTA reads its slice's partials from its own memory, and nobody's
    // memory is touched from outside any more.  Bound by the latency of one chain: stores to peers, barrier, local loads.  Steps, with
    // the peers' partials read remotely after a barrier, and a second barrier to keep the peers alive, and now: 8 x 32K tokens 56.8
    // -> 54.7 us, 24 chat requests 53.0 -> 51.4, 1 x 1M (16 heads) 73.3 -> 72.0, 11 x 14K 49.4 -> 47.8.
    const int slice = p.G * LOCKS_D / p.splits, nh = slice_heads(slice);
    float *rx = reinterpret_cast<float *>(smem + kAttSmem);                    // [splits - 1][slice]: the peers' partials
    float2 *rms = reinterpret_cast<float2 *>(rx + (p.splits - 1) * slice);     // [splits][nh]: (max, sum) of the slice's heads
    // idle tails of two rings: this CTA's own slice; [nh][splits] the CTAs' factors, and their share of the denominator
    float *own = reinterpret_cast<float *>(smem + (LOCKS_ATT_WARPS - 1) * kWarpBytes) + 16 * kWarpRow + 32;
    float2 *factor = reinterpret_cast<float2 *>(smem + 16 * kWarpRow * 4 + 128);
    const float inv_slice = 1.f / (float)slice;   // e / slice for e < 2048: (e + 1/2) / slice is at least 1 / 2048 from a whole number
    cluster_wait();   // the peers have started
    for (int i = threadIdx.x; i < p.G * (LOCKS_D / 4); i += NT) {
      const int g = i / (LOCKS_D / 4), d4 = 4 * (i % (LOCKS_D / 4)), e = g * LOCKS_D + d4, r = (int)(((float)e + 0.5f) * inv_slice);
      float sc[LOCKS_ATT_WARPS];
      (void)fold_head(g, sc);
      const float4 o = fold_dims(g, d4, sc);
      if (r == split) *reinterpret_cast<float4 *>(own + e - r * slice) = o;
      else cluster_st4(cluster_addr(rx + (split - (split > r)) * slice + e - r * slice, r), o);
    }
    for (int i = threadIdx.x; i < p.splits * nh; i += NT) {
      const int r = i / nh, j = i - r * nh, g = r * slice / LOCKS_D + j;
      if (g * LOCKS_D < (r + 1) * slice) {
        float sc[LOCKS_ATT_WARPS];
        cluster_st2(cluster_addr(rms + split * nh + j, r), fold_head(g, sc));
      }
    }
    cluster_arrive();
    cluster_wait();
    const int lg = __ffs(p.splits) - 1;   // splits is a power of two
    for (int i = threadIdx.x; i < p.splits * nh; i += NT) {
      const int j = i >> lg, c = i & (p.splits - 1);
      if ((split * slice / LOCKS_D + j) * LOCKS_D >= (split + 1) * slice) continue;
      float M = -INFINITY;
#pragma unroll 8
      for (int u = 0; u < p.splits; ++u) M = fmaxf(M, rms[u * nh + j].x);
      const float2 v = rms[c * nh + j];
      const float sc = M > -INFINITY ? ex2f(v.x - M) : 0.f;
      factor[i] = make_float2(sc, v.y * sc);
    }
    __syncthreads();
    const int g0 = split * slice / LOCKS_D;
    for (int e = threadIdx.x; e < slice; e += NT) {
      const int g = (split * slice + e) / LOCKS_D, dim = split * slice + e - g * LOCKS_D;
      const float2 *fc = factor + (g - g0) * p.splits;
      float L = 0.f, o = 0.f;
#pragma unroll 4
      for (int c = 0; c < p.splits; ++c) {
        const float2 f = fc[c];
        L += f.y;
        o = fmaf(c == split ? own[e] : rx[(c - (c > split)) * slice + e], f.x, o);
      }
      if (L != 0.f) o /= L;   // (0: no tokens)
      const int64_t row = (int64_t)b * p.Hq + h * p.G + g;
      reinterpret_cast<__nv_bfloat16 *>(p.out)[row * LOCKS_D + dim] = __float2bfloat16_rn(o);
      if (p.lse && dim == 0) {
        float M = -INFINITY;
        for (int c = 0; c < p.splits; ++c) M = fmaxf(M, rms[c * nh + g - g0].x);
        p.lse[row] = (M > -INFINITY) ? (M + log2f(L)) * kLn2 : -INFINITY;
      }
    }
    return;
  }
  for (int i = threadIdx.x; i < p.G * (LOCKS_D / 4); i += NT) {
    const int g = i / (LOCKS_D / 4), d4 = 4 * (i % (LOCKS_D / 4));
    float sc[LOCKS_ATT_WARPS];
    const float2 ML = fold_head(g, sc);
    float4 o = fold_dims(g, d4, sc);
    if (ML.x > -INFINITY) { o.x /= ML.y; o.y /= ML.y; o.z /= ML.y; o.w /= ML.y; }
    const int hq = h * p.G + g;
    const float lse2 = (ML.x > -INFINITY) ? ML.x + log2f(ML.y) : -INFINITY;
    if (p.splits == 1) {
      const int64_t row = (int64_t)b * p.Hq + hq;
      __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(p.out) + row * LOCKS_D + d4;
      if ((uintptr_t)p.out % 8 == 0) {   // (the caller's buffer need not be aligned)
        *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf16(o.x, o.y), pack_bf16(o.z, o.w));
      } else {
        dst[0] = __float2bfloat16_rn(o.x); dst[1] = __float2bfloat16_rn(o.y);
        dst[2] = __float2bfloat16_rn(o.z); dst[3] = __float2bfloat16_rn(o.w);
      }
      if (p.lse && d4 == 0) p.lse[row] = lse2 * kLn2;
    } else {
      const int64_t slot = ((int64_t)b * p.Hq + hq) * p.splits + split;
      *reinterpret_cast<float4 *>(p.part_o + slot * LOCKS_D + d4) = o;
      if (d4 == 0) p.part_lse[slot] = lse2;
    }
  }
  if (p.splits == 1 || !p.fused_merge) return;
  // the last CTA of this (request, KV head) to arrive merges the splits' partials by log-sum-exp
  int &sh_last = *reinterpret_cast<int *>(smem + kWarpBytes - 16);   // idle tail of a ring
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) sh_last = (atomicAdd(&p.done[prob], 1) == p.splits - 1);
  __syncthreads();
  if (!sh_last) return;
  __threadfence();
  // weights of the splits: sh_w[g][s] = 2^(lse_s - max), then normalised by their sum
  float *sh_w = reinterpret_cast<float *>(smem);   // [G][splits] <= 16 x 64 floats, the rings are idle now
  for (int e = threadIdx.x; e < p.G * p.splits; e += NT) {
    const int g = e / p.splits, s2 = e - g * p.splits;
    sh_w[e] = __ldcg(p.part_lse + ((int64_t)b * p.Hq + h * p.G + g) * p.splits + s2);
  }
  __syncthreads();
  if (threadIdx.x < p.G) {
    float *w = sh_w + threadIdx.x * p.splits;
    float M = -INFINITY;
    for (int s2 = 0; s2 < p.splits; ++s2) M = fmaxf(M, w[s2]);
    float L = 0.f;
    for (int s2 = 0; s2 < p.splits; ++s2) { const float v = (M > -INFINITY) ? ex2f(w[s2] - M) : 0.f; w[s2] = v; L += v; }
    const float inv = L > 0.f ? 1.f / L : 0.f;
    for (int s2 = 0; s2 < p.splits; ++s2) w[s2] *= inv;
    if (p.lse) p.lse[(int64_t)b * p.Hq + h * p.G + threadIdx.x] = (M > -INFINITY) ? (M + log2f(L)) * kLn2 : -INFINITY;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < p.G * (LOCKS_D / 4); e += NT) {   // four dims per thread, loads batched by 4 splits
    const int g = e / (LOCKS_D / 4), d4 = e - g * (LOCKS_D / 4);
    const int64_t row = (int64_t)b * p.Hq + h * p.G + g;
    const float4 *po = reinterpret_cast<const float4 *>(p.part_o + row * p.splits * LOCKS_D) + d4;
    const float *w = sh_w + g * p.splits;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < p.splits; s0 += 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        v[u] = (s0 + u < p.splits) ? __ldcg(po + (int64_t)(s0 + u) * (LOCKS_D / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float ww = (s0 + u < p.splits) ? w[s0 + u] : 0.f;
        acc.x += ww * v[u].x; acc.y += ww * v[u].y; acc.z += ww * v[u].z; acc.w += ww * v[u].w;
      }
    }
    __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(reinterpret_cast<__nv_bfloat16 *>(p.out) + row * LOCKS_D + 4 * d4);
    dst[0] = __floats2bfloat162_rn(acc.x, acc.y);
    dst[1] = __floats2bfloat162_rn(acc.z, acc.w);
  }
  if (threadIdx.x == 0) p.done[prob] = 0;   // ready for the next launch
}

// fp32 caches, in fp32 arithmetic: a CTA of four warps takes a split's pages for NH query heads of a KV head at a time, a warp
// every fourth page in tiles of 8 tokens.  A lane owns 4 dims of every row; the 8 NH partial dot products of a tile are summed
// by halves (each step a lane passes on the half that is not its own: 31 shuffles for 32 sums), after which a lane holds the
// score of one (head, token).  Bound by the latency of a tile's chain (16 rows in flight a warp) and by its shuffles.
// Steps with fp32 caches, before (a warp per head, token after token, each with a warp reduction of its own) and after this
// kernel and scan_f32_kernel: 30 requests x 32 pages, 4 heads, 226 -> 70 us; 25 x 169..666 tokens, all pages, 122 -> 41; 48 x
// 237..968, 5 heads, 377 -> 114; 3 x 31K, 8 heads, 357 -> 99.
constexpr int kF32CtasPerSm = 3;
template <int NH>
__global__ void __launch_bounds__(128, kF32CtasPerSm) attend_f32_kernel(AttParams p) {
  constexpr int kTok = 8, NV = kTok * NH, kDup = 32 / NV;   // kDup lanes hold the same score
  static_assert(NH == 1 || NH == 4, "scores have to fill or divide a warp");
  __shared__ float so[4][NH][LOCKS_D];
  __shared__ float sm[4][NH], sl[4][NH];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int parts = (p.G + NH - 1) / NH;
  const int split = blockIdx.x, h = blockIdx.y / parts, g0 = blockIdx.y % parts * NH, b = blockIdx.z;
  pdl_wait();
  const int64_t prob = (int64_t)b * p.Hkv + h;
  const int Tn = p.seq_lens[b];
  int npages = p.ids ? p.cnt[prob] : max((Tn + p.B - 1) / p.B, 0);
  const int row = p.ids ? p.kbud : p.Pmax;
  if ((p.ids && npages < 0) || npages > row) {
    if (threadIdx.x == 0) set_status(p.status, LOCKS_ERR_BAD_BLOCK);
    npages = npages < 0 ? 0 : row;
  }
  const int per = slice_length(p, npages), lo = split * per, hi = min(lo + per, npages);
  const float *K = reinterpret_cast<const float *>(p.k), *V = reinterpret_cast<const float *>(p.v);
  const int64_t row0 = (int64_t)b * p.Hq + h * p.G + g0;   // first of the CTA's query heads
  float4 q[NH], o[NH];
#pragma unroll
  for (int g = 0; g < NH; ++g) {
    q[g] = o[g] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g0 + g < p.G) q[g] = reinterpret_cast<const float4 *>(p.q)[(row0 + g) * (LOCKS_D / 4) + lane];
  }
  const int tok = lane / kDup % kTok;   // this lane's score: head lane / (kDup kTok), token tok of the tile
  float m = -INFINITY, l = 0.f;         // of the lane's head; l: its tokens' share
  const float c2 = p.sm_scale * kLog2e;
  int block = 0, ntok = 0;
  auto page_at = [&](int idx) { return p.ids ? p.ids[prob * p.kbud + idx] : idx; };
  bool good = lo + warp < hi && resolve_page(p, b, page_at(lo + warp), Tn, block, ntok);
  for (int idx = lo + warp; idx < hi; idx += 4) {
    int next_block = 0, next_ntok = 0;   // resolved one page ahead
    const bool next_good = idx + 4 < hi && resolve_page(p, b, page_at(idx + 4), Tn, next_block, next_ntok);
    if (good) {
      const int64_t base = (int64_t)block * p.sb + (int64_t)(h / p.kvdiv) * p.sh + 4 * lane;
      for (int t0 = 0; t0 < ntok; t0 += kTok) {
        float4 k[kTok], v[kTok];
#pragma unroll
        for (int t = 0; t < kTok; ++t) {   // rows past the end: the last row again, with a weight of zero
          const int64_t at = base + (int64_t)min(t0 + t, ntok - 1) * p.st;
          k[t] = *reinterpret_cast<const float4 *>(K + at);
          v[t] = *reinterpret_cast<const float4 *>(V + at);
        }
        if (t0 + kTok > ntok) {   // ... and values of zero: an infinite one times zero is not zero
#pragma unroll
          for (int t = 1; t < kTok; ++t)
            if (t0 + t >= ntok) v[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float s[NV];
#pragma unroll
        for (int g = 0; g < NH; ++g)
#pragma unroll
          for (int t = 0; t < kTok; ++t)
            s[g * kTok + t] = fmaf(q[g].w, k[t].w, fmaf(q[g].z, k[t].z, fmaf(q[g].y, k[t].y, q[g].x * k[t].x)));
        halving_sum<NV>(s, lane);
        const float sc = t0 + tok < ntok ? s[0] * c2 : -INFINITY;
        float mn = sc;
#pragma unroll
        for (int x = kDup; x < kDup * kTok; x <<= 1) mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, x));
        mn = fmaxf(mn, m);
        if (__any_sync(0xffffffffu, mn > m)) {
          const float alpha = exp2f(m - mn);
          l *= alpha;
          m = mn;
#pragma unroll
          for (int g = 0; g < NH; ++g) {
            const float a = __shfl_sync(0xffffffffu, alpha, g * kTok * kDup);
            o[g].x *= a; o[g].y *= a; o[g].z *= a; o[g].w *= a;
          }
        }
        const float pw = exp2f(sc - mn);
        l += pw;
#pragma unroll
        for (int t = 0; t < kTok; ++t)
#pragma unroll
          for (int g = 0; g < NH; ++g) {
            const float w = __shfl_sync(0xffffffffu, pw, (g * kTok + t) * kDup);
            o[g].x = fmaf(w, v[t].x, o[g].x); o[g].y = fmaf(w, v[t].y, o[g].y);
            o[g].z = fmaf(w, v[t].z, o[g].z); o[g].w = fmaf(w, v[t].w, o[g].w);
          }
      }
    }
    good = next_good; block = next_block; ntok = next_ntok;
  }
#pragma unroll
  for (int x = kDup; x < kDup * kTok; x <<= 1) l += __shfl_xor_sync(0xffffffffu, l, x);
#pragma unroll
  for (int g = 0; g < NH; ++g) *reinterpret_cast<float4 *>(&so[warp][g][4 * lane]) = o[g];
  if (lane % (kDup * kTok) == 0) { sm[warp][lane / (kDup * kTok)] = m; sl[warp][lane / (kDup * kTok)] = l; }
  __syncthreads();
  const int dim = threadIdx.x;
#pragma unroll
  for (int g = 0; g < NH; ++g) {
    if (g0 + g >= p.G) break;
    const float M = fmaxf(fmaxf(sm[0][g], sm[1][g]), fmaxf(sm[2][g], sm[3][g]));
    float L = 0.f, acc = 0.f;
    if (M > -INFINITY) {
      for (int w = 0; w < 4; ++w) {
        const float sc = exp2f(sm[w][g] - M);
        L += sl[w][g] * sc;
        acc += so[w][g][dim] * sc;
      }
      acc /= L;
    }
    const float lse2 = (M > -INFINITY) ? M + log2f(L) : -INFINITY;
    if (p.splits == 1) {
      reinterpret_cast<float *>(p.out)[(row0 + g) * LOCKS_D + dim] = acc;
      if (p.lse && dim == 0) p.lse[row0 + g] = lse2 * kLn2;
    } else {
      const int64_t slot = (row0 + g) * p.splits + split;
      p.part_o[slot * LOCKS_D + dim] = acc;
      if (dim == 0) p.part_lse[slot] = lse2;
    }
  }
}

// Merge of the split-K partials of one query head: 128 threads = 4 split slices x 32 four-dim columns.
template <typename T>
__global__ void __launch_bounds__(128) attend_merge_kernel(const float *part_o, const float *part_lse, int splits,
                                                           T *out, float *lse, int Hq) {
  __shared__ float sw[LOCKS_ATT_MAX_SPLITS];
  __shared__ float4 sacc[4][32];
  const int hq = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
  pdl_wait();
  const int64_t row = (int64_t)b * Hq + hq;
  for (int s = tid; s < splits; s += 128) sw[s] = part_lse[row * splits + s];
  __syncthreads();
  if (tid < 32) {
    float M = -INFINITY;
    for (int s = lane; s < splits; s += 32) M = fmaxf(M, sw[s]);
    M = warp_max(M);
    float L = 0.f;
    for (int s = lane; s < splits; s += 32) { const float w = (M > -INFINITY) ? exp2f(sw[s] - M) : 0.f; sw[s] = w; L += w; }
    L = warp_sum(L);
    const float inv = L > 0.f ? 1.f / L : 0.f;
    __syncwarp();
    for (int s = lane; s < splits; s += 32) sw[s] *= inv;
    if (lse && lane == 0) lse[row] = (M > -INFINITY) ? (M + log2f(L)) * kLn2 : -INFINITY;
  }
  __syncthreads();
  const int sl = tid >> 5;
  const float4 *po = reinterpret_cast<const float4 *>(part_o + row * splits * LOCKS_D) + lane;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = sl; s0 < splits; s0 += 16) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = (s0 + 4 * u < splits) ? __ldcg(po + (int64_t)(s0 + 4 * u) * (LOCKS_D / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float w = (s0 + 4 * u < splits) ? sw[s0 + 4 * u] : 0.f;
      acc.x += w * v[u].x; acc.y += w * v[u].y; acc.z += w * v[u].z; acc.w += w * v[u].w;
    }
  }
  sacc[sl][lane] = acc;
  __syncthreads();
  if (sl == 0) {
    const float4 a1 = sacc[1][lane], a2 = sacc[2][lane], a3 = sacc[3][lane];
    acc.x += a1.x + a2.x + a3.x; acc.y += a1.y + a2.y + a3.y; acc.z += a1.z + a2.z + a3.z; acc.w += a1.w + a2.w + a3.w;
    stf<T>(out, row * LOCKS_D + 4 * lane + 0, acc.x);
    stf<T>(out, row * LOCKS_D + 4 * lane + 1, acc.y);
    stf<T>(out, row * LOCKS_D + 4 * lane + 2, acc.z);
    stf<T>(out, row * LOCKS_D + 4 * lane + 3, acc.w);
  }
}

// Merge of the attention partials of several shards of one sequence (each normalised over its own pages, with
// its natural-log lse): out = sum_r w_r o_r, w_r = exp(lse_r - LSE), LSE = log sum_r exp(lse_r).
template <typename T>
__global__ void __launch_bounds__(LOCKS_D) merge_shards_kernel(const T *part_out, const float *part_lse, int nparts, int rows,
                                                              T *out, float *lse) {
  const int row = blockIdx.x, dim = threadIdx.x;
  float M = -INFINITY;
  for (int r = 0; r < nparts; ++r) M = fmaxf(M, part_lse[(int64_t)r * rows + row]);
  float L = 0.f, acc = 0.f;
  if (M > -INFINITY) {
    for (int r = 0; r < nparts; ++r) {
      const float l = part_lse[(int64_t)r * rows + row];
      if (l == -INFINITY) continue;
      const float w = __expf(l - M);
      L += w;
      acc += w * ldf<T>(part_out, ((int64_t)r * rows + row) * LOCKS_D + dim);
    }
    acc /= L;
  }
  stf<T>(out, (int64_t)row * LOCKS_D + dim, acc);
  if (lse && dim == 0) lse[row] = M > -INFINITY ? M + __logf(L) : -INFINITY;
}

}  // namespace

int locks_launch_merge_shards(locks_ctx *c, const void *part_out, const float *part_lse, int nparts, int batch, void *out,
                              float *lse, cudaStream_t st) {
  const int rows = batch * c->cfg.num_q_heads;
  if (c->cfg.q_dtype == LOCKS_BF16)
    merge_shards_kernel<__nv_bfloat16><<<rows, LOCKS_D, 0, st>>>(reinterpret_cast<const __nv_bfloat16 *>(part_out), part_lse, nparts,
                                                                rows, reinterpret_cast<__nv_bfloat16 *>(out), lse);
  else
    merge_shards_kernel<float><<<rows, LOCKS_D, 0, st>>>(reinterpret_cast<const float *>(part_out), part_lse, nparts, rows,
                                                        reinterpret_cast<float *>(out), lse);
  return locks_check_launch(c);
}

namespace {

// How the problems of a launch are cut: splits per problem, and how these are merged.
struct AttGeom { int splits, cluster, fused_merge; };

AttGeom attend_geometry(locks_ctx *c, int batch, int Hkv, int G, bool dense) {
  const bool bf = c->cfg.kv_dtype == LOCKS_BF16;   // tensor-core kernel
  const int sub_shift = !bf ? 0 : (c->B == 64 ? 2 : (c->B == 32 ? 1 : 0));
  // one wave: as many splits per problem as resident CTA slots allow, at least one tile (fp32 kernel: page) per warp
  const int ntiles = (dense ? c->Pmax : c->k) << sub_shift;
  int slots = c->num_sms * LOCKS_ATT_CTAS_PER_SM;
  if (slots > LOCKS_ATT_SLOT_BOUND) slots = LOCKS_ATT_SLOT_BOUND;
  int splits = slots / (batch * Hkv);
  const int most = (ntiles + LOCKS_ATT_WARPS - 1) / LOCKS_ATT_WARPS;
  if (splits > most) splits = most;
  if (splits > LOCKS_ATT_MAX_SPLITS) splits = LOCKS_ATT_MAX_SPLITS;
  if (splits < 1) splits = 1;
  // With clearly more problems than SMs every SM streams for several CTAs already: splitting a problem in
  // two only adds the merge (config 2, 256 problems: -1.5 to -2 us per step with one CTA per problem)
  if (bf && !dense && 2 * batch * Hkv >= 3 * c->num_sms) splits = 1;
  AttGeom g = {splits, 0, 0};
  // Preferred: the splits of a problem as one thread-block cluster (2, 4, 8 or 16 CTAs) that merges through
  // distributed shared memory, as long as a CTA then has at most 12 tiles per warp to stream (12 x 9K tokens, budget 128
  // pages, 96 problems: step 47.3 us as five splits that the last CTA merges, 43.8 as clusters of four; no case of 14 .. 64
  // requests slower), or 8 where the cluster leaves more than half of the CTAs that there is room for unused (dense, 1 x 8K
  // tokens: 13.2 us as clusters of 16, 12.4 as 72 splits; with 16 heads, whose splits cost more to merge, 20.5 and 21.4).
  if (c->att_clusters[0] < 0) {   // clusters of 2, 4, 8, 16 CTAs of this kernel that fit the device at once (probed once)
    cudaFuncSetAttribute(attend_bf16_kernel<1, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemMost);
    cudaFuncSetAttribute(attend_bf16_kernel<1, true, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int i = 0; i < 4; ++i) {
      cudaLaunchConfig_t lc = {};
      lc.gridDim = dim3(2 << i, 1, 1);
      lc.blockDim = dim3(LOCKS_ATT_WARPS * 32);
      lc.dynamicSmemBytes = kAttSmemMost;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 2 << i; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      lc.attrs = at;
      lc.numAttrs = 1;
      int nclusters = 0;
      if (cudaOccupancyMaxActiveClusters(&nclusters, attend_bf16_kernel<1, true, false>, &lc) != cudaSuccess) nclusters = 0;
      c->att_clusters[i] = nclusters;
    }
    (void)cudaGetLastError();   // a refused probe is not an error of this call
  }
  if (bf && splits >= 2) {
    // The largest size of which every problem's cluster is resident in one wave.  A cluster's CTAs have to share a GPC, so
    // fewer large clusters fit than CTAs do: 32 problems as clusters of 16 (512 CTAs in 592 slots) take two waves, 36.7 us a
    // step (4 x 8K tokens, budget 128 pages) against 30.8 as clusters of 8; 24 problems fit, 29.2 against 30.0.
    int i = 3;
    while (i >= 0 && ((2 << i) > splits || c->att_clusters[i] < batch * Hkv)) --i;
    const int most_tiles = i >= 0 && ((4 << i) >= splits || G > 8) ? 12 : 8;
    if (i >= 0 && (ntiles + (2 << i) - 1) / (2 << i) <= most_tiles * LOCKS_ATT_WARPS) {
      g.cluster = 1;
      g.splits = 2 << i;
      g.fused_merge = 1;   // no merge launch follows
    }
  }
  if (!g.cluster) {   // as many slices as the longest list has: 8 problems of 901 pages 24.2 us as 70 splits, 26.7 as 74
    const int per = (ntiles + splits - 1) / splits;
    g.splits = (ntiles + per - 1) / per;
    g.fused_merge = (G * g.splits <= kFusedMerge) ? 1 : 0;
  }
  return g;
}

}  // namespace

// Called at once, attention's CTAs wait in their slots while the selector works, and a build that starts when the scan ends has what
// they leave.  Worth it between about 7/8 and 19/20 of the slots.  Steps that append, called when the keys are there -> at once; CTAs
// of attention + of the build, of 592 slots: 512 + 16 (8 x 24K) 50.0 -> 53.0 us, (8 x 32K) 53.7 ->
// 53.5; 512 + 32 (16 x 8K) 51.6 -> 51.7; 528 + 17 (11 x 8K, 6 KV heads) 41.0 -> 38.4; 528 + 33 (33 x 8K, 4) 55.3 -> 56.7; 532 + 34 (19 x 8K,
// 7) 55.4 -> 53.0; 544 + 34 (17 x 8K) 58.5 -> 53.6, when all 17 fill a page 61.1 -> 75.3; 560 + 18 (10 x 8K, 7) 43.0 -> 42.4; 560 + 35
// (20 x 8K, 7) 60.8 -> 54.9; 576 + 18 (9 x
// 32K) 56.0 -> 57.0; 576 + 36 (18 x 8K) 55.8 -> 58.4, (18 x 30K) 87.5 -> 90.8; 592 + 37 (37 x 8K, 4) 66.4 -> 77.6.  fp32 caches (three CTAs on
// an SM, always more than fit): 8 x 8K 91.4 -> 94.5, 16 x 8K 144.6 -> 148.8.
bool locks_attend_fills(locks_ctx *c, int batch) {
  const int Hkv = c->cfg.num_kv_heads, slots = c->num_sms * (c->cfg.kv_dtype == LOCKS_BF16 ? LOCKS_ATT_CTAS_PER_SM : kF32CtasPerSm);
  const int ctas = attend_geometry(c, batch, Hkv, c->G, false).splits * Hkv * batch;
  return 8 * ctas > 7 * slots && 20 * ctas <= 19 * slots;
}

int locks_launch_attend(locks_ctx *c, const void *q, const locks_kv *kv, int batch, const int32_t *ids,
                        const int32_t *cnt, void *out, float *lse, cudaStream_t st) {
  AttParams p;
  p.q = q; p.k = kv->k; p.v = kv->v; p.sb = kv->stride_block; p.sh = kv->stride_head; p.st = kv->stride_token;
  p.block_table = kv->block_table; p.seq_lens = kv->seq_lens; p.ids = ids; p.cnt = cnt;
  p.part_o = c->att_o; p.part_lse = c->att_lse; p.out = out; p.lse = lse; p.status = c->status;
  p.batch = batch; p.Hq = c->cfg.num_q_heads; p.Hkv = c->cfg.num_kv_heads; p.G = c->G; p.Pmax = c->Pmax;
  p.kbud = c->k; p.num_blocks = kv->num_blocks; p.sm_scale = c->cfg.sm_scale; p.B = c->B; p.kvdiv = 1;
  if (c->cfg.combine == LOCKS_COMBINE_PER_HEAD && ids) {   // one page table per query head: groups of one
    p.kvdiv = p.G; p.Hkv = p.Hq; p.G = 1;
  }
  const bool bf = c->cfg.kv_dtype == LOCKS_BF16;   // tensor-core kernel
  const bool wide = c->B != LOCKS_B;
  p.sub_shift = !bf ? 0 : (c->B == 64 ? 2 : (c->B == 32 ? 1 : 0));
  p.done = c->att_done;
  const AttGeom geo = attend_geometry(c, batch, p.Hkv, p.G, ids == nullptr);
  p.splits = geo.splits; p.cluster = geo.cluster; p.fused_merge = geo.fused_merge;
  p.per_split = (1ull << 32) / p.splits + 1;
  if (bf) {
    const bool contig = kv->stride_token == LOCKS_D;
    const dim3 grid(p.splits, p.Hkv, batch), blk(LOCKS_ATT_WARPS * 32);
    const bool attrs = locks_attrs_needed(LOCKS_ATTR_ATTEND);
#define LOCKS_ATT_CASE(NH_, CONTIG_, WIDE_)                                                                                  \
  do {                                                                                                                      \
    if (attrs) {                                                                                                            \
      cudaFuncSetAttribute(attend_bf16_kernel<NH_, CONTIG_, WIDE_>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemMost); \
      cudaFuncSetAttribute(attend_bf16_kernel<NH_, CONTIG_, WIDE_>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);     \
    }                                                                                                                       \
    if ((p.G > 8) != (NH_ == 2) || contig != CONTIG_ || wide != WIDE_) break;                                               \
    if (p.cluster) locks_launch_pdl_cluster(attend_bf16_kernel<NH_, CONTIG_, WIDE_>, grid, blk, cluster_smem(p.G, p.splits), p.splits, st, p); \
    else locks_launch_pdl(attend_bf16_kernel<NH_, CONTIG_, WIDE_>, grid, blk, kAttSmem, st, p);                             \
  } while (0)
    LOCKS_ATT_CASE(1, true, false);
    LOCKS_ATT_CASE(1, false, false);
    LOCKS_ATT_CASE(2, true, false);
    LOCKS_ATT_CASE(2, false, false);
    LOCKS_ATT_CASE(1, true, true);
    LOCKS_ATT_CASE(1, false, true);
    LOCKS_ATT_CASE(2, true, true);
    LOCKS_ATT_CASE(2, false, true);
#undef LOCKS_ATT_CASE
  } else {
    if (p.G == 1) locks_launch_pdl(attend_f32_kernel<1>, dim3(p.splits, p.Hkv, batch), dim3(128), 0, st, p);
    else locks_launch_pdl(attend_f32_kernel<4>, dim3(p.splits, p.Hkv * ((p.G + 3) / 4), batch), dim3(128), 0, st, p);
  }
  int rc = locks_check_launch(c);
  if (rc != LOCKS_OK || p.splits == 1 || (bf && p.fused_merge)) return rc;
  const dim3 mg(c->cfg.num_q_heads, batch);
  if (bf) locks_launch_pdl(attend_merge_kernel<__nv_bfloat16>, mg, dim3(128), 0, st, (const float *)c->att_o, (const float *)c->att_lse,
                           p.splits, reinterpret_cast<__nv_bfloat16 *>(out), lse, p.Hq);
  else locks_launch_pdl(attend_merge_kernel<float>, mg, dim3(128), 0, st, (const float *)c->att_o, (const float *)c->att_lse, p.splits,
                        reinterpret_cast<float *>(out), lse, p.Hq);
  return locks_check_launch(c);
}

// ------------------------------------------------------------------------------------------------
// Sparse attention for callers that cannot allocate device memory.
//
// The split-K partials and the split-arrival counters of attend_bf16_kernel normally live in the
// workspace the caller allocates for locks_create().  This variant keeps them in a fixed array that is
// part of the library image instead, so nothing has to be allocated at all.
// ------------------------------------------------------------------------------------------------

namespace {

constexpr int kNoAllocMaxRows = LOCKS_NOALLOC_MAX_ROWS;          // batch * Hq
constexpr int kNoAllocMaxSplits = LOCKS_NOALLOC_MAX_SPLITS;
constexpr size_t kNoAllocO = (size_t)kNoAllocMaxRows * kNoAllocMaxSplits * LOCKS_D * sizeof(float);
constexpr size_t kNoAllocLse = (size_t)kNoAllocMaxRows * kNoAllocMaxSplits * sizeof(float);
constexpr size_t kNoAllocDone = (size_t)kNoAllocMaxRows * sizeof(int32_t);   // >= batch * Hkv
constexpr size_t kNoAllocBytes = kNoAllocO + kNoAllocLse + kNoAllocDone + 256;

// About 2.1 MB held by every GPU that loads the library, until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

struct NoAllocDevice {
  unsigned char *scratch;   // device address of g_noalloc_scratch on this device (not the host symbol!)
  int num_sms;
  bool ready;
};
NoAllocDevice g_noalloc_dev[64] = {};
std::mutex g_noalloc_mu;   // guards the per-device set-up (two host threads may make a device's first call)

}  // namespace

extern "C" int locks_sparse_attend_noalloc(const locks_config *cfg, const void *q, const locks_kv *kv, int batch,
                                           const int32_t *page_ids, const int32_t *page_count, void *out, float *lse,
                                           locks_stream stream) {
  if (!cfg || !q || !kv || !out || !kv->k || !kv->v || !kv->block_table || !kv->seq_lens) return LOCKS_ERR_INVALID_ARG;
  if ((page_ids == nullptr) != (page_count == nullptr) || batch <= 0 || kv->num_blocks <= 0) return LOCKS_ERR_INVALID_ARG;
  if (cfg->num_q_heads <= 0 || cfg->num_kv_heads <= 0 || cfg->num_q_heads % cfg->num_kv_heads) return LOCKS_ERR_INVALID_ARG;
  if (cfg->max_pages_per_seq <= 0 || cfg->budget_tokens <= 0 || !(cfg->sm_scale > 0.f)) return LOCKS_ERR_INVALID_ARG;
  if (cfg->head_dim != LOCKS_D || cfg->page_size != LOCKS_B || cfg->kv_dtype != LOCKS_BF16 || cfg->q_dtype != LOCKS_BF16)
    return LOCKS_ERR_UNSUPPORTED;
  const int G = cfg->num_q_heads / cfg->num_kv_heads;
  if (G > 16) return LOCKS_ERR_UNSUPPORTED;
  if ((kv->stride_block | kv->stride_head | kv->stride_token) % 8 || kv->stride_token < LOCKS_D) return LOCKS_ERR_INVALID_ARG;
  if (((uintptr_t)kv->k | (uintptr_t)kv->v | (uintptr_t)q) % 16) return LOCKS_ERR_INVALID_ARG;
  // the built-in scratch bounds the problem: reject anything that would not fit
  if ((int64_t)batch * cfg->num_q_heads > kNoAllocMaxRows) return LOCKS_ERR_TOO_LARGE;

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LOCKS_ERR_CUDA;
  NoAllocDevice &nd = g_noalloc_dev[dev];
  std::unique_lock<std::mutex> setup_lock(g_noalloc_mu);
  if (!nd.ready) {
    // first call on this device: ask the runtime where the array lives on the CURRENT device
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || ptr == nullptr) return LOCKS_ERR_CUDA;
    if (cudaDeviceGetAttribute(&nd.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return LOCKS_ERR_CUDA;
    cudaFuncSetAttribute(attend_bf16_kernel<1, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemMost);
    cudaFuncSetAttribute(attend_bf16_kernel<2, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemMost);
    cudaFuncSetAttribute(attend_bf16_kernel<1, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemMost);
    cudaFuncSetAttribute(attend_bf16_kernel<2, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemMost);
    nd.scratch = reinterpret_cast<unsigned char *>(ptr);
    nd.ready = true;
  }
  setup_lock.unlock();
  cudaStream_t st = (cudaStream_t)stream;
  AttParams p;
  p.q = q; p.k = kv->k; p.v = kv->v; p.sb = kv->stride_block; p.sh = kv->stride_head; p.st = kv->stride_token;
  p.block_table = kv->block_table; p.seq_lens = kv->seq_lens; p.ids = page_ids; p.cnt = page_count;
  p.part_o = reinterpret_cast<float *>(nd.scratch);
  p.part_lse = reinterpret_cast<float *>(nd.scratch + kNoAllocO);
  p.done = reinterpret_cast<int32_t *>(nd.scratch + kNoAllocO + kNoAllocLse);
  p.status = reinterpret_cast<int32_t *>(nd.scratch + kNoAllocO + kNoAllocLse + kNoAllocDone);
  p.out = out; p.lse = lse;
  p.batch = batch; p.Hq = cfg->num_q_heads; p.Hkv = cfg->num_kv_heads; p.G = G; p.Pmax = cfg->max_pages_per_seq;
  p.kbud = (cfg->budget_tokens + LOCKS_B - 1) / LOCKS_B; p.num_blocks = kv->num_blocks; p.sm_scale = cfg->sm_scale; p.B = LOCKS_B; p.kvdiv = 1;
  const int npages = page_ids ? p.kbud : p.Pmax;
  int splits = nd.num_sms * LOCKS_ATT_CTAS_PER_SM / (batch * p.Hkv);
  const int most = (npages + LOCKS_ATT_WARPS - 1) / LOCKS_ATT_WARPS;
  if (splits > most) splits = most;
  if (splits > kNoAllocMaxSplits) splits = kNoAllocMaxSplits;
  if (splits < 1) splits = 1;
  const int per = (npages + splits - 1) / splits;
  p.splits = (npages + per - 1) / per;
  p.per_split = (1ull << 32) / p.splits + 1;
  p.sub_shift = 0;
  p.fused_merge = 1;
  p.cluster = 0;
  // the array keeps whatever the last call left: the arrival counters and the status word must start at zero
  if (cudaMemsetAsync(p.done, 0, kNoAllocDone + 256, st) != cudaSuccess) return LOCKS_ERR_CUDA;
  dim3 grid(p.splits, p.Hkv, batch);
  const bool contig = kv->stride_token == LOCKS_D;
  if (G <= 8) {
    if (contig) attend_bf16_kernel<1, true, false><<<grid, LOCKS_ATT_WARPS * 32, kAttSmem, st>>>(p);
    else attend_bf16_kernel<1, false, false><<<grid, LOCKS_ATT_WARPS * 32, kAttSmem, st>>>(p);
  } else {
    if (contig) attend_bf16_kernel<2, true, false><<<grid, LOCKS_ATT_WARPS * 32, kAttSmem, st>>>(p);
    else attend_bf16_kernel<2, false, false><<<grid, LOCKS_ATT_WARPS * 32, kAttSmem, st>>>(p);
  }
  return cudaPeekAtLastError() == cudaSuccess ? LOCKS_OK : LOCKS_ERR_CUDA;
}
