// What locks_launch_scan decides on the host, with the CUDA runtime replaced by fakes: one line for every line of the input.
//   input   B  Hq  Hkv  rank  format  dtype  batch  max_pages  partition
//   output  partials that a problem may have, slots in a row of them, CTAs of the scan, whether a step's build starts beside it
#include <cuda_runtime.h>
#include <cstdio>
#include <cstring>

#include "locks_internal.cuh"

static long ctas = 0;
extern "C" {
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **) {
  ctas = (long)c->gridDim.x * c->gridDim.y * c->gridDim.z;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **, unsigned long long, cudaDriverEntryPointQueryResult *) { return cudaErrorUnknown; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 0; }
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
}
bool locks_attrs_needed(int) { return false; }

int main() {
  int B, Hq, Hkv, rank, fmt, dtype, batch, pages, partition;
  while (scanf("%d %d %d %d %d %d %d %d %d", &B, &Hq, &Hkv, &rank, &fmt, &dtype, &batch, &pages, &partition) == 9) {
    locks_ctx c;
    memset((void *)&c, 0, sizeof c);
    c.cfg.page_size = c.B = B; c.cfg.num_q_heads = Hq; c.cfg.num_kv_heads = Hkv; c.cfg.rank = rank; c.cfg.summary_fmt = fmt;
    c.cfg.q_dtype = c.cfg.kv_dtype = dtype; c.cfg.max_batch = batch; c.cfg.max_pages_per_seq = c.Pmax = pages; c.cfg.sm_scale = 0.1f;
    c.G = Hq / Hkv; c.k = 8; c.S = locks_fmt_stride(fmt, rank, B); c.max_groups = (pages + LOCKS_GROUP - 1) / LOCKS_GROUP; c.num_sms = 148;
    c.scan_partition = partition; c.scorer = LOCKS_SCORER_SUMMARY;
    locks_kv kv;
    memset(&kv, 0, sizeof kv);
    kv.num_blocks = 100;
    if (locks_launch_scan(&c, nullptr, nullptr, &kv, batch, nullptr, 0, nullptr) != LOCKS_OK) return 1;
    printf("%d %d %ld %d\n", c.part_slots, c.max_groups, ctas, (int)locks_scan_leaves_room(&c, batch));
  }
  return 0;
}
