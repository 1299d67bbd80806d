// The CUDA runtime calls and kernel launchers that locks_decode_step uses, as fakes that write down what is enqueued on which
// stream.  Linked with the library's own api.cu, they show the order of a step's work, without a GPU and with any call failing.
//   step_order EARLY APPEND CALL NTH      two steps; the NTH occurrence of CALL in the first one reports an error ("none": nothing does)
// A launch that reports an error is enqueued all the same: the error may be one that another library left pending.
#include <cuda_runtime_api.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>

#include "locks.h"

struct locks_append;
struct locks_staged;

static bool early_build = false;
static std::string fail_call;
static int fail_nth = 0, seen = 0;
static bool failing(const char *call) { return fail_call == call && ++seen == fail_nth; }
static const char *stream_name(cudaStream_t s) { return s == (cudaStream_t)0x10 ? "main" : s == (cudaStream_t)0x20 ? "side" : "default"; }
static int launch(const char *name, cudaStream_t st) {
  printf("op %s %s\n", name, stream_name(st));
  return failing(name) ? LOCKS_ERR_CUDA : LOCKS_OK;
}

extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)0x20; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { static size_t n = 0; *e = (cudaEvent_t)++n; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  if (failing("record")) return cudaErrorUnknown;
  printf("record %zu %s\n", (size_t)e, stream_name(s));
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (failing("wait")) return cudaErrorUnknown;
  printf("wait %zu %s\n", (size_t)e, stream_name(s));
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *, int, size_t n, cudaStream_t s) { if (s) printf("op clear %s %zu\n", stream_name(s), n); return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
// registration of the file's kernels, none of which runs
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
}

bool locks_scan_leaves_room(const locks_ctx *, int) { return early_build; }
bool locks_attend_fills(locks_ctx *, int) { return false; }
int locks_launch_scan(locks_ctx *, const void *, const void *, const locks_kv *, int, float *, int, cudaStream_t st) { return launch("scan", st); }
int locks_launch_select(locks_ctx *, const float *, const locks_kv *, int, int32_t *, int32_t *, float *, const locks_append *, cudaStream_t st, bool, const locks_staged *) { return launch("select", st); }
int locks_launch_attend(locks_ctx *, const void *, const locks_kv *, int, const int32_t *, const int32_t *, void *, float *, cudaStream_t st) { return launch("attend", st); }
int locks_launch_build(locks_ctx *, const locks_kv *, int, const int32_t *, const int32_t *, int, void *, const void *, const int32_t *, cudaStream_t st, bool, int32_t *,
                       const void *const *, void *const *, int) { return launch("build", st); }

int main(int argc, char **argv) {
  if (argc != 5) return 2;
  early_build = atoi(argv[1]);
  void *row = atoi(argv[2]) ? (void *)0x1000 : nullptr;
  locks_config cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.head_dim = 128; cfg.page_size = 16; cfg.num_q_heads = 8; cfg.num_kv_heads = 2; cfg.rank = 8; cfg.summary_fmt = LOCKS_FMT_I4;
  cfg.kv_dtype = cfg.q_dtype = LOCKS_BF16; cfg.max_batch = 3; cfg.max_pages_per_seq = 64; cfg.budget_tokens = 256; cfg.sm_scale = 0.1f;
  const size_t bytes = locks_workspace_bytes(&cfg);
  locks_ctx *ctx = nullptr;
  if (locks_create(&cfg, aligned_alloc(256, (bytes + 255) / 256 * 256), bytes, &ctx) != LOCKS_OK) return 3;
  locks_kv kv;
  memset(&kv, 0, sizeof kv);
  kv.k = kv.v = (void *)0x2000; kv.block_table = (int32_t *)0x3000; kv.seq_lens = (int32_t *)0x4000; kv.num_blocks = 100;
  kv.stride_block = 4096; kv.stride_head = 2048; kv.stride_token = 128;
  fail_call = argv[3]; fail_nth = atoi(argv[4]);
  for (int step = 0; step < 2; ++step) {
    printf("step %d\n", step);
    const int rc = locks_decode_step(ctx, (void *)0x5000, row, row, &kv, (void *)0x6000, 3, (void *)0x7000, nullptr, nullptr, (cudaStream_t)0x10);
    printf("returns %d\n", rc);
    fail_call = "none";
  }
  return 0;
}
