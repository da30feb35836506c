/* md_host.cpp with a fake CUDA runtime, to show on a machine without a GPU
 * which route a call takes.  Launchers that the checks do not reach stay
 * unresolved. */
#include <cuda_runtime.h>
#include <stdio.h>

static int fake_current = 0, fake_owner = 0, n_memcpy = 0, n_kernel = 0;
static cudaError_t fake_get_device(int *d) {
  *d = fake_current;
  return cudaSuccess;
}
static cudaError_t fake_attributes(cudaPointerAttributes *a, const void *) {
  *a = cudaPointerAttributes();
  a->type = cudaMemoryTypeDevice;
  a->device = fake_owner;
  return cudaSuccess;
}
static cudaError_t fake_memcpy(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) {
  ++n_memcpy;
  return cudaSuccess;
}
#define cudaGetDevice fake_get_device
#define cudaPointerGetAttributes fake_attributes
#define cudaMemcpyAsync fake_memcpy
#include "../../paper_2607_10582_gb300/csrc/md_host.cpp"

cudaError_t md::launch_copy(const CopyParams &, cudaStream_t) {
  ++n_kernel;
  return fake_current == 0 ? cudaSuccess : cudaErrorInvalidResourceHandle;   // a stream of device 0
}

int main() {
  md_ctx c;
  c.cfg = md_config();
  c.cfg.num_layers = c.cfg.num_kv_heads = c.cfg.num_q_heads = 1;
  c.cfg.head_dim = 128;
  c.cfg.page_size = 16;
  c.cfg.max_batch = 2;
  c.cfg.max_pages_per_seq = c.cfg.num_phys_pages = 8;
  compute_layout(c.cfg, &c.lay);
  c.ws = (uint8_t *)(uintptr_t)(1 << 20);
  c.device = 0;
  const size_t n = (size_t)c.cfg.num_phys_pages * c.cfg.page_size * 4;
  void *dst = (void *)(uintptr_t)(1 << 16);
  for (int current = 0; current < 2; ++current)
    for (int owner = 0; owner < 2; ++owner) {
      fake_current = current;
      fake_owner = owner;
      n_memcpy = n_kernel = 0;
      const md_status st = md_get_state(&c, MD_STATE_A, dst, n);
      printf("get_state current %d owner %d: %d %s%s\n", current, owner, (int)st, n_kernel ? "kernel" : "",
             n_memcpy ? "copy" : "");
    }
  return 0;
}
