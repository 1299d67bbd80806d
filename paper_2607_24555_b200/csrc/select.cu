// Stage A, part 2: share-average combine and budgeted page selection (Sec. 4 of the paper):
//   log Z_g   = log sum_{j in 1..P-2} exp s^_j(q_g)                       (candidates only)
//   log m_bar_j = log( (1/G) sum_g exp(s^_j(q_g) - log Z_g) )
//   S = {0, P-1}  U  top-(k-2) candidates by log m_bar_j (ties: lower page index), ids ascending.
// One 512-thread CTA ranks a chunk of 512 .. 8192 pages of a (request, KV head): it turns the chunk's scores into
// order-preserving 32-bit keys in shared memory and emits the K = k-2 largest in page order (emit_winners: a histogram that
// finds the bin of the K-th largest key, an exact ranking of that bin's few keys, and a bit map of the winners, whose prefix
// counts are the output positions).  With one chunk per problem that is the final table.  With several, each chunk emits
// its own top-(k-2) (key, page) list, and the CTA of a problem that finishes last ranks the lists the same way in the same
// launch (a chunk's local top-(k-2) always contains the chunk's share of the global top-(k-2), ties included, because both
// rounds use the same lower-index tie rule and lists stay in page order).
// Pages are dealt to threads round-robin (element i of thread t is page i*512 + t), so loads are
// coalesced and every thread is busy whatever the context length.
// The kernel runs once through its code on at most a few dozen SMs, so instruction fetch is a visible part
// of its latency: loops over a thread's elements stay rolled (keys live in shared memory, not in
// registers), and the ranking is a real call (select_emit) in the kernels that need it twice.
#include "locks_internal.cuh"

namespace {

constexpr int kNW = LOCKS_SEL_THREADS / 32;
constexpr int kMaxKeys = LOCKS_SEL_MAX_EPT * LOCKS_SEL_THREADS;   // keys one CTA ranks at most
constexpr int kMaxWin = 4 * LOCKS_SEL_THREADS;                    // k - 2 at most (checked on the host)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct SelParams {
  const float *shat;
  const float2 *part;
  const int32_t *seq_lens;
  const int32_t *part_cnt;   // partials per head of each problem, or nullptr: part_slots for all
  int pc_div;                // rankings per entry of part_cnt (1; per-head arm: G)
  int32_t *ids, *cnt;
  float *logshare;
  uint32_t *cand_key;  // [batch][Hkv][chunks][kc] chunk lists (chunked selection only): keys, 0 = no entry
  int32_t *cand_idx;
  int32_t *sel_done;   // [batch][Hkv] chunk-arrival counters (zero between launches)
  int32_t *status;
  int batch, Hq, Hkv, G, Pmax, max_groups, k, chunks, kc, chunk_pages, part_slots;
  int combine;       // LOCKS_COMBINE_*
  int attend_first;  // let the next kernel be scheduled at once
  int Bshift;        // log2 of the page size (4, 5 or 6)
  int place;         // `staged` is given (asked for in a line of parameters that is read anyway)
  locks_append app;  // decode step only: the new token's K/V rows, written here beside the ranking
  locks_staged staged;  // decode step only: summaries that were ready before the scores
};

// Decode step: the CTA of (request b, KV head h) writes the new token's K and V rows of that head into the
// cache (one warp, a few independent loads and stores beside the ranking's own loads), and the CTA of
// head 0 stores the step's length back to the caller's array.  Nothing reads the caller's array between
// the scan (complete before this kernel passes its wait) and the end of the step, except a build that started
// beside the scan: the step's other kernels take lengths from the published copy.  With such a build (a.arrivals) the
// last to arrive of this CTA and the request's page-heads stores the length.
__device__ __noinline__ void append_token(const SelParams &p, int b, int h, int lane, int T) {
  const locks_append &a = p.app;
  const int batch = p.batch, Hkv = p.Hkv, Pmax = p.Pmax, Bshift = p.Bshift;
  int32_t *status = p.status;
  if (h == 0 && lane == 0) {
    if (!a.arrivals || atomicAdd(a.arrivals + b, 1) == Hkv) {   // the last to arrive stores (BuildParams::seq_commit)
      if (a.arrivals) a.arrivals[b] = 0;
      a.seq_commit[b] = T;
    }
  }
  const int at = a.seq_eff[batch + b];
  if (at < 0) return;
  const int page = at >> Bshift, slot = at & ((1 << Bshift) - 1);
  const int block = a.block_table[(int64_t)b * Pmax + page];
  if (block < 0 || block >= a.num_blocks) {
    if (lane == 0) set_status(status, LOCKS_ERR_BAD_BLOCK);
    return;
  }
  const int64_t dst = (int64_t)block * a.sb + (int64_t)h * a.sh + (int64_t)slot * a.st;
  const int64_t src = ((int64_t)b * Hkv + h) * LOCKS_D;
  if (a.esz == 2) {
    const uint2 kk = reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(a.k_new) + src)[lane];
    const uint2 vv = reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(a.v_new) + src)[lane];
    reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(a.k) + dst)[lane] = kk;
    reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(a.v) + dst)[lane] = vv;
  } else {
    const uint4 kk = reinterpret_cast<const uint4 *>(reinterpret_cast<const uint32_t *>(a.k_new) + src)[lane];
    const uint4 vv = reinterpret_cast<const uint4 *>(reinterpret_cast<const uint32_t *>(a.v_new) + src)[lane];
    reinterpret_cast<uint4 *>(reinterpret_cast<uint32_t *>(a.k) + dst)[lane] = kk;
    reinterpret_cast<uint4 *>(reinterpret_cast<uint32_t *>(a.v) + dst)[lane] = vv;
  }
}

// The summary of the page that request b has filled in this step, if its build was done before the scan: put in place now that no
// score reads it any more.  If the build is not done it will do so itself.
__device__ __noinline__ void place_staged(const SelParams &p, int b, int h, int lane, int T) {
  const locks_staged &s = p.staged;
  const int page = (T >> p.Bshift) - 1, prob = b * p.Hkv + h;
  if (T <= 0 || (T & ((1 << p.Bshift) - 1)) || page >= p.Pmax) return;   // as build_page_kernel has it
  const int block = s.block_table[(int64_t)b * p.Pmax + page];
  if (block < 0 || block >= s.num_blocks) return;
  int done = 0;
  if (lane == 0) {
    __threadfence();
    done = atomicAdd(s.staged + prob, 1);
    if (done) s.staged[prob] = 0;
    __threadfence();
  }
  __syncwarp();
  if (!__shfl_sync(0xffffffffu, done, 0)) return;
  const uint4 *src = reinterpret_cast<const uint4 *>(s.stage + (int64_t)prob * s.S);
  uint4 *dst = reinterpret_cast<uint4 *>(s.summ + ((int64_t)block * p.Hkv + h) * s.S);
  for (int i = lane; i < s.S / 16; i += 32) dst[i] = __ldcg(src + i);
}

constexpr int kListMax = 256;    // keys of the threshold bin that are ranked pair by pair
constexpr int kElemBits = 13;    // kMaxKeys = 2^13 elements

struct SelShared {
  uint32_t key[kMaxKeys];             // order-preserving keys, element i of thread t at i*512 + t; 0 = not a candidate
  int hist[3 * 256];                  // histograms of the key offsets' leading bits, rotating
  __align__(16) uint32_t gt[256];     // winners, one bit per element in element order
  __align__(16) uint32_t eq[256];     // elements of the threshold bin, where it holds equal keys or wins whole
  __align__(16) uint32_t list[kListMax];
  int nlist;
  int misc[16];                       // arrival flag
  float lzm[kNW], lzs[kNW];           // per-warp (max, sum) of the log Z reduction
  uint32_t red[2 * kNW];              // per-warp smallest and largest valid key
};

extern __shared__ __align__(16) uint8_t sel_smem[];
// Routines that are real calls take the block's shared state from the symbol itself (a reference argument would turn every
// access into a generic one) and their inputs by value (no stack).
__device__ __forceinline__ SelShared &shared_state() { return *reinterpret_cast<SelShared *>(sel_smem); }

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2f(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t order_key(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// smallest and largest valid key of this thread -> sh.red (read by emit_winners after its first barrier)
__device__ __forceinline__ void publish_range(SelShared &sh, uint32_t kmin, uint32_t kmax) {
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if ((threadIdx.x & 31) == 0) { sh.red[threadIdx.x >> 5] = kmin; sh.red[kNW + (threadIdx.x >> 5)] = kmax; }
}

// The K largest of the keys sh.key[i*512 + t], i < nslab (1 <= K <= number of valid keys; the range of the keys is in
// sh.red), in element order and with ties to the lower element.  Winner number pos of element e is written as
//   kEmitIds:   ids[1 + pos] = c0 + e                         (final table of a single-chunk problem)
//   kEmitList:  list_key[pos] = key, list_idx[pos] = c0 + e   (a chunk's candidate list)
//   kEmitFinal: ids[1 + pos] = page of entry e                (final table from the problem's lists; pages at sh.key[4096 + e])
//   kEmitEntry: sh.key[pos] = e                               (the same from more than 4096 entries: see select_finish)
// The keys' offsets from the smallest one need far fewer than 32 bits (page masses lie within a few units of each other),
// and one pass over their leading 8 bits usually leaves a few dozen keys in the bin of the K-th largest: these are ranked
// pair by pair.  A fuller bin is divided again; a bin of equal keys, or one that wins whole, needs no ranking.
// What bounds this is the chain of barriers, shuffles and instruction fetches (every phase runs once, on few SMs), not the
// keys: four barriers here, where three 8-bit radix passes and an ordered compaction by ballots and a scan of counts took
// eleven.  Steps, before and after: 1 x 8K tokens 27.8 -> 26.6 us, 8 x 32K 59.3 -> 57.1, 32 x 16K with a budget of 16 pages
// 62.0 -> 58.1, 24 chat requests 59.4 -> 57.1, 1 x 128K (lists of 9 chunks, ranked twice) 42.4 -> 41.2.  Running this code
// once on made-up keys before the wait for the scan, to have it in the instruction caches, costs 1 .. 6 us: the selector's
// CTAs become resident only when the scan is nearly over.
enum { kEmitIds = 0, kEmitList = 1, kEmitFinal = 2, kEmitEntry = 3 };
constexpr int kFinalPages = kMaxKeys / 2;

__device__ __forceinline__ void emit_winners(int nslab, int K, int mode, int c0, int32_t *ids, uint32_t *list_key, int32_t *list_idx) {
  SelShared &sh = shared_state();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 256) sh.hist[tid] = 0;
  if (tid == 0) sh.nlist = 0;
  __syncthreads();
  const uint32_t kmin = __reduce_min_sync(0xffffffffu, sh.red[lane & (kNW - 1)]);
  const uint32_t kmax = __reduce_max_sync(0xffffffffu, sh.red[kNW + (lane & (kNW - 1))]);
  int left = 32 - __clz(kmax - kmin);   // undecided bits of the offsets (0: all valid keys are equal)
  uint32_t prefix = 0u;                 // decided leading bits of the offset of the K-th largest key, in place
  int remaining = K;                    // of the keys with that prefix, how many win
  bool rank = false;                    // they are to be ranked (else: all of them equal, or all of them win)
#pragma unroll 1
  for (int cur = 0; left > 0;) {
    const int width = min(8, left), shift = left - width;
    const int nxt = cur == 2 ? 0 : cur + 1;
    int *hc = sh.hist + cur * 256;
    if (tid < 256) sh.hist[nxt * 256 + tid] = 0;   // last read two passes ago
    const uint32_t above = left < 32 ? prefix >> left : 0u;
#pragma unroll 4
    for (int i = 0; i < nslab; ++i) {
      const uint32_t k = sh.key[i * LOCKS_SEL_THREADS + tid], d = k - kmin;
      if (k && (left < 32 ? d >> left : 0u) == above) atomicAdd(&hc[(d >> shift) & ((1u << width) - 1u)], 1);
    }
    __syncthreads();
    // every warp for itself (one warp alone, and a barrier, take 2300 cycles where this takes 1100): lane l owns bins 8 (31 - l) .. + 7,
    // so lane order is descending digit order
    const int base = 8 * (31 - lane);
    const int4 lo = *reinterpret_cast<const int4 *>(hc + base), hi = *reinterpret_cast<const int4 *>(hc + base + 4);
    const int c[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    const int tot = (c[0] + c[1]) + (c[2] + c[3]) + (c[4] + c[5]) + (c[6] + c[7]);
    int incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const bool hit = incl - tot < remaining && remaining <= incl;   // the K-th largest falls in this lane's bins
    uint32_t found = 0u;   // digit (8 bits), count in its bin (12), rank wanted within it (12; at most the count)
    int acc = incl - tot;
#pragma unroll
    for (int j = 7; j >= 0; --j) {
      if (hit && acc < remaining && remaining <= acc + c[j]) found = (uint32_t)(base + j) << 24 | (uint32_t)min(c[j], 4095) << 12 | (uint32_t)min(remaining - acc, 4095);
      acc += c[j];
    }
    const uint32_t who = __ballot_sync(0xffffffffu, hit);
    found = __shfl_sync(0xffffffffu, found, who ? __ffs(who) - 1 : 0);
    const int count = (int)((found >> 12) & 4095u);
    remaining = (int)(found & 4095u);   // (K is below 4096)
    prefix |= (found >> 24) << shift;
    left = shift;
    cur = nxt;
    if (count == remaining && count < 4095) break;
    rank = count <= kListMax && left + kElemBits <= 32;
    if (rank) break;
  }
  if (left == 0) rank = false;
  // ---- winners above the bin, and the bin's own keys
  const uint32_t at = left < 32 ? prefix >> left : 0u;
#pragma unroll 2
  for (int i = 0; i < nslab; ++i) {
    const int e = i * LOCKS_SEL_THREADS + tid;
    const uint32_t k = sh.key[e], d = k - kmin, top = left < 32 ? d >> left : 0u;
    const uint32_t g = __ballot_sync(0xffffffffu, k && top > at), q = __ballot_sync(0xffffffffu, k && top == at);
    if (lane == 0) { sh.gt[i * kNW + warp] = g; sh.eq[i * kNW + warp] = q; }
    if (rank && k && top == at)   // the rest of the offset, then the element: larger is better, no two alike
      sh.list[min(atomicAdd(&sh.nlist, 1), kListMax - 1)] = (d & ((1u << left) - 1u)) << kElemBits | (uint32_t)(kMaxKeys - 1 - e);
  }
  __syncthreads();
  if (rank) {
    const int n = min(sh.nlist, kListMax);
    if (tid < n) {
      const uint32_t mine = sh.list[tid];
      int better = 0;
      for (int j = 0; j < n; j += 4) {
        const uint4 o = *reinterpret_cast<const uint4 *>(sh.list + j);
        better += (int)(o.x > mine) + (int)(o.y > mine && j + 1 < n) + (int)(o.z > mine && j + 2 < n) + (int)(o.w > mine && j + 3 < n);
      }
      const int e = kMaxKeys - 1 - (int)(mine & (kMaxKeys - 1));
      if (better < remaining) atomicOr(&sh.gt[e >> 5], 1u << (e & 31));
    }
    __syncthreads();
  }
  const int nw = nslab * kNW;
  if (K < 24 * nslab) {
    // ---- few winners: a thread per 32 elements finds the position of its first winner and walks its winners (8192 pages, 126
    // winners: 0.7 us, the other way 2.4)
    if (warp * 32 >= nw) return;
    int before = 0, eq_before = 0;   // winners, and unranked keys of the bin, in the words of the warps before this one
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int w = u * 32 + lane;
      if (w < warp * 32) { before += __popc(sh.gt[w]); eq_before += __popc(sh.eq[w]); }
    }
    const int w = warp * 32 + lane;
    uint32_t won = w < nw ? sh.gt[w] : 0u, q = w < nw && !rank ? sh.eq[w] : 0u;
    int incl = __popc(won) | __popc(q) << 16;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    eq_before = __reduce_add_sync(0xffffffffu, eq_before);
    int pos = before + (incl & 0xffff) - __popc(won);
    if (!rank) {
      eq_before += (incl >> 16) - __popc(q);
      pos += min(eq_before, remaining);
      for (int take = remaining - eq_before; q && take > 0; --take) { won |= q & -q; q &= q - 1; }
    }
    for (; won; won &= won - 1, ++pos) {
      const int e = w * 32 + __ffs(won) - 1;
      if (mode == kEmitIds) ids[1 + pos] = c0 + e;
      else if (mode == kEmitList) { list_key[pos] = sh.key[e]; list_idx[pos] = c0 + e; }
      else if (mode == kEmitFinal) ids[1 + pos] = (int32_t)sh.key[kFinalPages + e];
      else sh.key[pos] = (uint32_t)e;   // (the keys are bits of sh.gt and sh.eq by now)
    }
    return;
  }
  // ---- positions: every warp counts the winners (and the bin's unranked keys) before each of its words; lane l owns words
  // 8 l .. 8 l + 7, and word i * kNW + warp is the same one of lane 2 i or 2 i + 1 for every i (512 pages, 126 winners: 0.8 us,
  // the other way 1.4)
  const int mine = warp & 7, half = warp >> 3;
  uint32_t g8[8], q8[8];
  {
    const uint4 *gp = reinterpret_cast<const uint4 *>(sh.gt + 8 * lane), *qp = reinterpret_cast<const uint4 *>(sh.eq + 8 * lane);
    const bool in = 8 * lane < nw;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u), a = in ? gp[0] : z, b = in ? gp[1] : z, c = in && !rank ? qp[0] : z, d = in && !rank ? qp[1] : z;
    g8[0] = a.x; g8[1] = a.y; g8[2] = a.z; g8[3] = a.w; g8[4] = b.x; g8[5] = b.y; g8[6] = b.z; g8[7] = b.w;
    q8[0] = c.x; q8[1] = c.y; q8[2] = c.z; q8[3] = c.w; q8[4] = d.x; q8[5] = d.y; q8[6] = d.z; q8[7] = d.w;
  }
  int before = 0, total = 0;   // packed: winners | unranked keys << 16; before this lane's word `mine`, and in all of its words
  uint32_t g = 0u, q = 0u;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    if (u == mine) { before = total; g = g8[u]; q = q8[u]; }
    total += __popc(g8[u]) | __popc(q8[u]) << 16;
  }
  int incl = total;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  before += incl - total;
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll 2
  for (int i = 0; i < nslab; ++i) {
    const int src = 2 * i + half;
    const uint32_t gw = __shfl_sync(0xffffffffu, g, src), qw = __shfl_sync(0xffffffffu, q, src);
    const int pre = __shfl_sync(0xffffffffu, before, src);
    const int eq_before = (pre >> 16) + __popc(qw & lt);
    const bool won = ((gw >> lane) & 1u) || (((qw >> lane) & 1u) && eq_before < remaining);
    if (won) {
      const int e = i * LOCKS_SEL_THREADS + tid, pos = (pre & 0xffff) + __popc(gw & lt) + min(eq_before, remaining);
      if (mode == kEmitIds) ids[1 + pos] = c0 + e;
      else if (mode == kEmitList) { list_key[pos] = sh.key[e]; list_idx[pos] = c0 + e; }
      else if (mode == kEmitFinal) ids[1 + pos] = (int32_t)sh.key[kFinalPages + e];
      else sh.key[pos] = (uint32_t)e;   // (the keys are bits of sh.gt and sh.eq by now)
    }
  }
}

// The same as a real call, where a kernel needs it twice
__device__ __noinline__ void select_emit(int nslab, int K, int mode, int c0, int32_t *ids, uint32_t *list_key, int32_t *list_idx) {
  emit_winners(nslab, K, mode, c0, ids, list_key, list_idx);
}

// What a launch's rankings have in common before the length is known: a CTA's scores and partials sit at addresses that do not
// depend on it, so one round trip fetches them together with it.
struct KeyInputs {
  const float *shat0;      // scores of the group's head 0, page 0
  const float2 *part0;     // partials of head 0
  const int32_t *seq_len, *part_cnt;   // part_cnt: this problem's, or nullptr
  int G, Pmax, max_groups, part_slots, c0, chunk_pages, Bshift, combine;
};

// Keys of a chunk: log m_bar of page c0 + i*512 + t as an order-preserving integer in sh.key[i*512 + t] (0 for pages that are not
// candidates), and their range in sh.red.  A thread takes the scores of all HB >= G heads of SB = 16 / HB slabs at once, 16 loads in
// flight, the next batch while the current one is reduced.  log Z_g comes from the scan's partials (max_i, sum_i):
// log2 Z = M + log2 sum_i sum_i 2^(max_i - M), M = max_i max_i; the block's warps are dealt to (head, slice) pairs.
// combine: share-average (the paper's rule) subtracts log Z_g per head and averages; group-mass sums the raw masses (log Z_g = 0,
// no 1/G); group-max keeps the largest raw score.
// `begin(T, P)` is called once the length is there; false: nothing to rank (returns 0 slabs).
// Bound by a chain of round trips: the length, the first batch of scores and the first partials travel together (before, the length
// alone came first, then 2000 cycles of address arithmetic with a 64-bit division, then the rest).
template <int HB, typename Begin>
__device__ __forceinline__ int chunk_keys(const KeyInputs &in, Begin begin, float *logshare_row) {
  constexpr int SB = 16 / HB, NP = HB == 16 ? 5 : 4;   // NP: partials in flight per lane
  constexpr int NSLICE = kNW / HB;                     // warps per head
  SelShared &sh = shared_state();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = in.G;
  const float *row0 = in.shat0 + in.c0 + tid;
  float cur[HB][SB], nxt[HB][SB];
  auto load = [&](int i0, int last, float (&x)[HB][SB]) {   // pages 1 .. last
    const float *r = row0 + i0 * LOCKS_SEL_THREADS;   // offsets within one request fit 32 bits
#pragma unroll
    for (int sl = 0; sl < SB; ++sl) {
      const int page = in.c0 + (i0 + sl) * LOCKS_SEL_THREADS + tid;
      const bool ok = page >= 1 && page <= last && (i0 + sl) * LOCKS_SEL_THREADS < in.chunk_pages;
#pragma unroll
      for (int u = 0; u < HB; ++u) x[u][sl] = (ok && u < G) ? r[u * in.Pmax + sl * LOCKS_SEL_THREADS] : -INFINITY;
    }
  };
  const int T = *in.seq_len;
  const int counted = in.part_cnt ? *in.part_cnt : in.part_slots;
  load(0, in.Pmax - 1, cur);
  const int slice = warp / HB, g = warp % HB;
  const bool has_head = g < G && in.combine == LOCKS_COMBINE_SHARE_AVG;
  const float2 *pp = in.part0 + (int64_t)g * in.max_groups;
  constexpr int pstep = 32 * NSLICE;
  const int p0 = slice * 32 + lane;
  const int most = in.part_cnt ? in.max_groups : in.part_slots;   // what may be read before the count is known
  float2 v[NP];
#pragma unroll
  for (int u = 0; u < NP; ++u) v[u] = (has_head && p0 + pstep * u < most) ? pp[p0 + pstep * u] : make_float2(-INFINITY, 0.f);
  // ---- the length is there
  const int P = (T + (1 << in.Bshift) - 1) >> in.Bshift;
  if (!begin(T, P)) return 0;
  // slabs of 512 pages that hold at least one candidate of this chunk (the configured maximum context is usually longer)
  const int nslab = (min(P - 1, in.c0 + in.chunk_pages) - in.c0 + LOCKS_SEL_THREADS - 1) / LOCKS_SEL_THREADS;
  const int nparts = in.part_cnt ? min(max(counted, 0), in.max_groups) : min(counted, (P - 1 + LOCKS_GROUP - 1) / LOCKS_GROUP);
  if (in.combine == LOCKS_COMBINE_SHARE_AVG) {
    float m = -INFINITY, s = 0.f;
    if (has_head) {
#pragma unroll 1
      for (int i0 = p0;;) {
        float nm = m;
#pragma unroll
        for (int u = 0; u < NP; ++u) {
          if (i0 + pstep * u >= nparts) v[u] = make_float2(-INFINITY, 0.f);
          nm = fmaxf(nm, v[u].x);
        }
        if (nm > -INFINITY) {
          s *= ex2f((m - nm) * kLog2e);
#pragma unroll
          for (int u = 0; u < NP; ++u) s = fmaf(v[u].y, ex2f((v[u].x - nm) * kLog2e), s);
          m = nm;
        }
        i0 += NP * pstep;
        if (i0 - lane >= nparts) break;   // (the whole warp leaves together)
#pragma unroll
        for (int u = 0; u < NP; ++u) v[u] = i0 + pstep * u < nparts ? pp[i0 + pstep * u] : make_float2(-INFINITY, 0.f);
      }
      const uint32_t top = __reduce_max_sync(0xffffffffu, order_key(m));
      const float M = __uint_as_float((top & 0x80000000u) ? top & 0x7FFFFFFFu : ~top);
      s = M > -INFINITY ? s * ex2f((m - M) * kLog2e) : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      m = M;
    }
    if (lane == 0) { sh.lzm[warp] = m; sh.lzs[warp] = s; }
  }
  __syncthreads();
  // every warp for itself: lanes g, g + HB .. hold the slices of head g
  float lz[HB];
  {
    const int w = lane % kNW;
    float m = sh.lzm[w], s = sh.lzs[w], M = m;
#pragma unroll
    for (int o = HB; o < kNW; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    if (NSLICE > 1) s = M > -INFINITY ? s * ex2f((m - M) * kLog2e) : 0.f;
#pragma unroll
    for (int o = HB; o < kNW; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float l2 = in.combine == LOCKS_COMBINE_SHARE_AVG && lane < G ? M * kLog2e + lg2f(s) : 0.f;
#pragma unroll
    for (int u = 0; u < HB; ++u) lz[u] = __shfl_sync(0xffffffffu, l2, u);
  }
  const float logG = in.combine == LOCKS_COMBINE_SHARE_AVG ? __logf((float)G) : 0.f;
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll 1
  for (int i0 = 0; i0 < nslab; i0 += SB) {
    if (i0 + SB < nslab) load(i0 + SB, P - 2, nxt);
#pragma unroll
    for (int sl = 0; sl < SB; ++sl) {
      const int i = i0 + sl, page = in.c0 + i * LOCKS_SEL_THREADS + tid;
      if (i >= nslab) break;
      float m = -INFINITY;
#pragma unroll
      for (int u = 0; u < HB; ++u) {
        cur[u][sl] = fmaf(cur[u][sl], kLog2e, -lz[u]);   // heads past the group stay -inf
        m = fmaxf(m, cur[u][sl]);
      }
      float acc = 0.f;
#pragma unroll
      for (int u = 0; u < HB; ++u) acc += ex2f(cur[u][sl] - m);
      const bool valid = page >= 1 && page <= P - 2;
      const float val = (in.combine == LOCKS_COMBINE_GROUP_MAX ? m : m + lg2f(acc)) * kLn2 - logG;
      const uint32_t key = order_key(val);
      sh.key[i * LOCKS_SEL_THREADS + tid] = valid ? key : 0u;
      if (valid) {
        kmin = min(kmin, key);
        kmax = max(kmax, key);
        if (logshare_row) logshare_row[page] = val;
      }
    }
#pragma unroll
    for (int u = 0; u < HB; ++u)
#pragma unroll
      for (int sl = 0; sl < SB; ++sl) cur[u][sl] = nxt[u][sl];
  }
  publish_range(sh, kmin, kmax);
  return nslab;
}

// Several chunks per problem: the chunk that arrives last ranks the problem's candidate lists.
__device__ __noinline__ void select_finish(int32_t *done, int chunks, int kc, int k, int32_t *ids, int32_t *count,
                                           const uint32_t *ck, const int32_t *ci, int P) {
  SelShared &sh = shared_state();
  const int tid = threadIdx.x;
  __threadfence();   // this chunk's list before its arrival
  __syncthreads();
  if (tid == 0) {
    const int ticket = atomicAdd(done, 1);
    const bool last = ticket == chunks - 1;
    if (last) *done = 0;   // every chunk has arrived: ready for the next launch
    sh.misc[8] = last;
  }
  __syncthreads();
  if (!sh.misc[8]) return;
  __threadfence();
  const int K2 = k - 2;
  // entries in list order (chunk, position) = page order; element i of thread t is entry i*512 + t
  const int N = chunks * kc;
  const int nslab = (N + LOCKS_SEL_THREADS - 1) / LOCKS_SEL_THREADS;
  const bool pages_too = N <= kFinalPages;
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll 4
  for (int i = 0; i < nslab; ++i) {
    const int e = i * LOCKS_SEL_THREADS + tid;
    const uint32_t key = e < N ? __ldcg(ck + e) : 0u;
    sh.key[e] = key;
    if (pages_too) sh.key[kFinalPages + e] = e < N ? (uint32_t)__ldcg(ci + e) : 0u;
    if (key) { kmin = min(kmin, key); kmax = max(kmax, key); }
  }
  publish_range(sh, kmin, kmax);
  if (K2 > 0) {
    select_emit(nslab, K2, pages_too ? kEmitFinal : kEmitEntry, 0, ids, nullptr, nullptr);
    if (!pages_too) {   // the winners' pages, four loads in flight a thread
      __syncthreads();
      for (int j0 = tid; j0 < K2; j0 += 4 * LOCKS_SEL_THREADS) {
        int page[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) page[u] = j0 + u * LOCKS_SEL_THREADS < K2 ? __ldcg(ci + sh.key[j0 + u * LOCKS_SEL_THREADS]) : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) if (j0 + u * LOCKS_SEL_THREADS < K2) ids[1 + j0 + u * LOCKS_SEL_THREADS] = page[u];
      }
    }
  }
  if (tid == 0) {
    ids[0] = 0;
    ids[k - 1] = P - 1;
    *count = k;
  }
}

// HB: 4, 8 or 16 >= heads per KV head.  ONE: a CTA ranks its whole problem.
template <int HB, bool ONE>
__global__ void __launch_bounds__(LOCKS_SEL_THREADS, 2) select_kernel(const __grid_constant__ SelParams p) {
  const int chunk = ONE ? 0 : blockIdx.x, h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int prob = b * p.Hkv + h, c0 = chunk * p.chunk_pages;   // first page of this chunk
  int32_t *ids = p.ids + (int64_t)prob * p.k;
  const int64_t list0 = (int64_t)prob * p.chunks * p.kc;
  KeyInputs in;
  in.shat0 = p.shat + ((int64_t)b * p.Hq + h * p.G) * p.Pmax;
  in.part0 = p.part + ((int64_t)b * p.Hq + h * p.G) * p.max_groups;
  in.seq_len = p.seq_lens + b;
  in.part_cnt = p.part_cnt ? p.part_cnt + (p.pc_div == 1 ? prob : prob / p.pc_div) : nullptr;
  in.G = p.G; in.Pmax = p.Pmax; in.max_groups = p.max_groups; in.part_slots = p.part_slots; in.c0 = c0;
  in.chunk_pages = p.chunk_pages; in.Bshift = p.Bshift; in.combine = p.combine;
  if (p.attend_first) pdl_trigger();
  pdl_wait();   // the scan's scores and partials
  int P = 0;
  const int nslab = chunk_keys<HB>(in, [&](int T, int np) {
    P = np;
    if (p.app.k_new && chunk == 0 && tid >= LOCKS_SEL_THREADS - 32)
      append_token(p, b, h, tid & 31, T);
    if (p.place && (T & ((1 << p.Bshift) - 1)) == 0 && chunk == 0 && tid >= LOCKS_SEL_THREADS - 32) place_staged(p, b, h, tid & 31, T);
    if (P <= p.k) {  // every page is kept
      if (chunk == 0) {
        for (int j = tid; j < p.k; j += LOCKS_SEL_THREADS) ids[j] = j < P ? j : -1;
        if (tid == 0) p.cnt[prob] = P;
      }
      return false;
    }
    return c0 <= P - 2;
  }, p.logshare ? p.logshare + (int64_t)prob * p.Pmax : nullptr);
  // Attention's CTAs are called when the keys are there, not at once: waiting, they would hold the slots in which the step's build
  // starts when the scan ends (32 x 16K tokens, budget 16 pages: 59.4 -> 53.3 us a step, 8 x 24K 59.2 -> 52.9).  Where attention
  // itself needs most of the slots, but leaves some, it comes first (locks_attend_fills).
  pdl_trigger();
  if (P <= p.k) return;
  if (nslab == 0) {  // chunk past the candidates: an empty list
    if constexpr (!ONE) {
      for (int j = tid; j < p.kc; j += LOCKS_SEL_THREADS) p.cand_key[list0 + (int64_t)chunk * p.kc + j] = 0u;
      select_finish(p.sel_done + prob, p.chunks, p.kc, p.k, ids, p.cnt + prob, p.cand_key + list0, p.cand_idx + list0, P);
    }
    return;
  }
  const int cand_in_chunk = min(P - 2, c0 + p.chunk_pages - 1) - max(1, c0) + 1;
  const int K = min(p.k - 2, cand_in_chunk);
  if constexpr (ONE) {
    if (K > 0) emit_winners(nslab, K, kEmitIds, c0, ids, nullptr, nullptr);
    if (tid == 0) {
      ids[0] = 0;
      ids[p.k - 1] = P - 1;
      p.cnt[prob] = p.k;
    }
  } else {
    uint32_t *lk = p.cand_key + list0 + (int64_t)chunk * p.kc;
    for (int j = K + tid; j < p.kc; j += LOCKS_SEL_THREADS) lk[j] = 0u;   // fewer candidates than list slots
    if (K > 0) select_emit(nslab, K, kEmitList, c0, nullptr, lk, p.cand_idx + list0 + (int64_t)chunk * p.kc);
    select_finish(p.sel_done + prob, p.chunks, p.kc, p.k, ids, p.cnt + prob, p.cand_key + list0, p.cand_idx + list0, P);
  }
}

// ---- page-sharded selection (one long request whose pages are dealt to several GPUs) -----------------------
// log Z_g of the pages one shard scanned, from the scan's partials: one warp per (request, query head)
__global__ void __launch_bounds__(32) head_logz_kernel(const float2 *part, const int32_t *part_cnt, const int32_t *seq_lens,
                                                       float *logz, int Hq, int Hkv, int max_groups, int part_slots, int k) {
  const int hq = blockIdx.x, b = blockIdx.y, lane = threadIdx.x;
  pdl_wait();
  const int P = (seq_lens[b] + LOCKS_B - 1) / LOCKS_B;
  const int64_t prob = (int64_t)b * Hkv + hq / (Hq / Hkv);
  int nparts = part_cnt ? min(max(part_cnt[prob], 0), max_groups) : min(part_slots, (P - 1 + LOCKS_GROUP - 1) / LOCKS_GROUP);
  if (P <= k) nparts = 0;
  const float2 *pp = part + ((int64_t)b * Hq + hq) * max_groups;
  float m = -INFINITY, s = 0.f;
  for (int i = lane; i < nparts; i += 32) {
    const float2 x = pp[i];
    const float nm = fmaxf(m, x.x);
    if (nm > -INFINITY) { s = s * __expf(m - nm) + x.y * __expf(x.x - nm); m = nm; }
  }
  const float M = warp_max(m);
  s = warp_sum(M > -INFINITY ? s * __expf(m - M) : 0.f);
  if (lane == 0) logz[(int64_t)b * Hq + hq] = M > -INFINITY ? M + __logf(s) : -INFINITY;
}

// the shards' log Z values as the selector's partials: slot r of head g holds (log Z_g of shard r, 1)
__global__ void __launch_bounds__(128) ext_partials_kernel(const float *logz_parts, int nparts, float2 *part, int32_t *part_cnt,
                                                           int batch, int Hq, int Hkv, int max_groups) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < batch * Hkv) part_cnt[i] = nparts;
  if (i >= batch * Hq) return;
  for (int r = 0; r < nparts; ++r) {
    const float v = logz_parts[(int64_t)r * batch * Hq + i];
    part[(int64_t)i * max_groups + r] = make_float2(v, v > -INFINITY ? 1.f : 0.f);
  }
}

// Global top-(k-2) of the shards' candidate lists (each in page order, shards in page order, so that list order
// is page order and the lower-page tie rule carries over): one CTA per (request, KV head).
__global__ void __launch_bounds__(LOCKS_SEL_THREADS) merge_selection_kernel(const float *cand_key, const int32_t *cand_page, int nparts,
                                                                           int batch, int Hkv, int kc, int32_t *ids, int32_t *cnt) {
  SelShared &sh = shared_state();
  const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  const int64_t prob = (int64_t)b * Hkv + h, nprob = (int64_t)batch * Hkv;
  const int N = nparts * kc, nslab = (N + LOCKS_SEL_THREADS - 1) / LOCKS_SEL_THREADS;
  int32_t *out = ids + prob * kc;
  __shared__ int s_valid;
  if (tid == 0) s_valid = 0;
  __syncthreads();
  int mine = 0;
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
  for (int i = 0; i < nslab; ++i) {
    const int e = i * LOCKS_SEL_THREADS + tid;
    uint32_t key = 0u;
    if (e < N) {
      const int r = e / kc, j = e - r * kc;
      const int64_t at = ((int64_t)r * nprob + prob) * kc + j;
      if (cand_page[at] >= 0) {
        key = order_key(cand_key[at]);
        kmin = min(kmin, key);
        kmax = max(kmax, key);
        ++mine;
      }
    }
    sh.key[e] = key;
  }
  for (int j = tid; j < kc; j += LOCKS_SEL_THREADS) out[j] = -1;
  if (mine) atomicAdd(&s_valid, mine);
  publish_range(sh, kmin, kmax);
  __syncthreads();
  const int K = min(kc, s_valid);
  if (K > 0) {
    select_emit(nslab, K, kEmitIds, 0, out - 1, nullptr, nullptr);   // out[pos] = winning entry, in list order
    __syncthreads();
    int page[(kMaxWin + LOCKS_SEL_THREADS - 1) / LOCKS_SEL_THREADS];
#pragma unroll
    for (int u = 0; u < (kMaxWin + LOCKS_SEL_THREADS - 1) / LOCKS_SEL_THREADS; ++u) {
      const int j = tid + u * LOCKS_SEL_THREADS;
      page[u] = -1;
      if (j < K) {
        const int e = out[j], rr = e / kc, jj = e - rr * kc;
        page[u] = cand_page[((int64_t)rr * nprob + prob) * kc + jj];
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < (kMaxWin + LOCKS_SEL_THREADS - 1) / LOCKS_SEL_THREADS; ++u)
      if (tid + u * LOCKS_SEL_THREADS < K) out[tid + u * LOCKS_SEL_THREADS] = page[u];
  }
  if (tid == 0) cnt[prob] = K;
}

}  // namespace

int locks_launch_head_logz(locks_ctx *c, const locks_kv *kv, int batch, float *logz, cudaStream_t st) {
  locks_launch_pdl(head_logz_kernel, dim3(c->cfg.num_q_heads, batch), dim3(32), 0, st, (const float2 *)c->part,
                   (const int32_t *)(c->part_balanced ? c->part_cnt : nullptr), (const int32_t *)kv->seq_lens, logz,
                   c->cfg.num_q_heads, c->cfg.num_kv_heads, c->max_groups, c->part_slots, c->k);
  return locks_check_launch(c);
}

int locks_launch_ext_partials(locks_ctx *c, const float *logz_parts, int nparts, int batch, cudaStream_t st) {
  if (nparts < 1 || nparts > c->max_groups) return LOCKS_ERR_INVALID_ARG;
  const int n = batch * c->cfg.num_q_heads;
  ext_partials_kernel<<<(n + 127) / 128, 128, 0, st>>>(logz_parts, nparts, c->part, c->part_cnt, batch, c->cfg.num_q_heads,
                                                       c->cfg.num_kv_heads, c->max_groups);
  c->part_slots = nparts;
  c->part_balanced = 1;   // the selector takes the count from part_cnt
  return locks_check_launch(c);
}

int locks_launch_merge_selection(locks_ctx *c, const float *cand_key, const int32_t *cand_page, int nparts, int batch,
                                 int32_t *ids, int32_t *cnt, cudaStream_t st) {
  if (nparts < 1 || (int64_t)nparts * c->sel_kc > kMaxKeys) return LOCKS_ERR_UNSUPPORTED;
  merge_selection_kernel<<<dim3(c->cfg.num_kv_heads, batch), LOCKS_SEL_THREADS, sizeof(SelShared), st>>>(
      cand_key, cand_page, nparts, batch, c->cfg.num_kv_heads, c->sel_kc, ids, cnt);
  return locks_check_launch(c);
}

int locks_launch_select(locks_ctx *c, const float *shat, const locks_kv *kv, int batch, int32_t *ids,
                        int32_t *cnt, float *logshare, const locks_append *app, cudaStream_t st, bool attend_first,
                        const locks_staged *staged) {
  SelParams p;
  p.attend_first = attend_first;
  if (app) p.app = *app;
  else p.app.k_new = nullptr;
  if (staged) p.staged = *staged;
  else p.staged.stage = nullptr;
  p.place = p.staged.stage != nullptr;
  p.status = c->status;
  p.shat = shat; p.part = c->part; p.seq_lens = kv->seq_lens; p.ids = ids; p.cnt = cnt; p.logshare = logshare;
  p.cand_key = reinterpret_cast<uint32_t *>(c->cand_val); p.cand_idx = c->cand_idx; p.sel_done = c->sel_done;
  p.batch = batch; p.Hq = c->cfg.num_q_heads; p.Hkv = c->cfg.num_kv_heads; p.G = c->G; p.Pmax = c->Pmax;
  p.max_groups = c->max_groups; p.k = c->k; p.chunks = c->sel_chunks; p.kc = c->sel_kc;
  p.chunk_pages = c->sel_ept * LOCKS_SEL_THREADS;
  p.part_slots = c->part_slots;
  p.combine = c->cfg.combine;
  p.pc_div = 1;
  if (p.combine == LOCKS_COMBINE_PER_HEAD) {   // every query head is a group of one with a page table of its own
    if (app) return LOCKS_ERR_UNSUPPORTED;
    p.pc_div = p.G; p.Hkv = p.Hq; p.G = 1; p.combine = LOCKS_COMBINE_SHARE_AVG;
  }
  p.Bshift = c->B == 64 ? 6 : (c->B == 32 ? 5 : 4);
  p.part_cnt = c->part_balanced ? c->part_cnt : nullptr;
  if (p.chunk_pages > kMaxKeys || (int64_t)c->sel_chunks * c->sel_kc > kMaxKeys || p.G > 16) return LOCKS_ERR_UNSUPPORTED;
  // Two CTAs fit on an SM (64 registers per thread).  As long as every CTA can have an SM of its own it asks for enough shared memory
  // to get one: the block scheduler otherwise stacks pairs on the SMs that drain first (8 x 32K tokens 56.9 us a step, in pairs
  // 58.1).  More CTAs than SMs run in pairs, in one wave (192 CTAs of 24 chat requests 52.4 -> 48.3 us, 216 of 27 requests 81.2 ->
  // 77.5; 144 CTAs 60.2 alone, 60.7 in pairs).
  constexpr int kSmemAlone = 116 * 1024;
  const int64_t nctas = (int64_t)c->sel_chunks * p.Hkv * batch;
  const size_t smem = nctas <= c->num_sms ? (size_t)kSmemAlone : sizeof(SelShared);
  const dim3 grid(c->sel_chunks, p.Hkv, batch), blk(LOCKS_SEL_THREADS);
  const bool attrs = locks_attrs_needed(LOCKS_ATTR_SELECT), one = c->sel_chunks == 1;
#define LOCKS_SELECT_CASE(HB_, ONE_, FITS_)                                                                                  \
  do {                                                                                                                      \
    if (attrs) cudaFuncSetAttribute(select_kernel<HB_, ONE_>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAlone);     \
    if ((FITS_) && one == ONE_) locks_launch_pdl(select_kernel<HB_, ONE_>, grid, blk, smem, st, p);                         \
  } while (0)
  LOCKS_SELECT_CASE(4, true, p.G <= 4);
  LOCKS_SELECT_CASE(8, true, p.G > 4 && p.G <= 8);
  LOCKS_SELECT_CASE(16, true, p.G > 8);
  LOCKS_SELECT_CASE(4, false, p.G <= 4);
  LOCKS_SELECT_CASE(8, false, p.G > 4 && p.G <= 8);
  LOCKS_SELECT_CASE(16, false, p.G > 8);
#undef LOCKS_SELECT_CASE
  return locks_check_launch(c);
}
