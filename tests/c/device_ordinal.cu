/* The cluster kernel's host code under a device ordinal past its table, with
 * the runtime's current device faked (no GPU needed). */
#include <cuda_runtime.h>
#include <stdio.h>

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
  return 0;
}
