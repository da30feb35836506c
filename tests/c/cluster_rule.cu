/* The cluster kernel's host code with the runtime's current device faked (no
 * GPU needed): device ordinals past its table, and the form that the cost rule
 * takes for launch shapes read from stdin. */
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

static int fake_current = 0;
static cudaError_t fake_get_device(int *d) {
  *d = fake_current;
  return cudaSuccess;
}
#define cudaGetDevice fake_get_device
#include "../../paper_2607_10582_gb300/csrc/md_attn_cluster.cu"

int main() {
  using namespace md;
  AttnBase p = AttnBase();
  p.L = p.L_launch = p.Hkv = p.n_seqs = 1;
  p.ps = 16;
  p.n_tokens[0] = 430;
  p.n_pages[0] = 27;
  for (int dev : {64, 127, 500}) {
    fake_current = dev;
    const cudaError_t e = cluster_prepare();
    printf("device %d: %d, %d\n", dev, (int)e, cluster_plan(p, 0).C);
  }
  /* what cluster_prepare finds on a GB300 (152 SMs) */
  const int w4[3][5] = {{152, 152, 144, 120, 112}, {304, 304, 296, 288, 224}, {456, 456, 440, 408, 336}};
  fake_current = 0;
  memcpy(g_slots[0].w4, w4, sizeof(w4));
  memcpy(g_slots[0].w8, w4[0], sizeof(w4[0]));
  g_slots[0].ready = true;
  /* a line: layers, KV heads, page size, floats of scratch, sequences, their tokens */
  long long scratch;
  while (scanf("%d %d %d %lld %d", &p.L_launch, &p.Hkv, &p.ps, &scratch, &p.n_seqs) == 5) {
    for (int b = 0; b < p.n_seqs; ++b) {
      if (scanf("%d", &p.n_tokens[b]) != 1) return 1;
      p.n_pages[b] = (p.n_tokens[b] + p.ps - 1) / p.ps;
    }
    const ClusterPlan f = cluster_plan(p, (size_t)scratch);
    printf("form %d %d %d\n", f.C, f.warps, (int)f.spill);
  }
  return 0;
}
