/* Device code shared by the two attention kernels (the persistent one and the
 * cluster one): bounded waits, the stage layout, the new token's rows and
 * state, a token's mass. */
#ifndef MD_ATTN_CUH
#define MD_ATTN_CUH

#include "md_internal.h"
#include "md_ptx.cuh"

namespace md {

/* NEW (a template parameter): this launch appends the step's new tokens.
 * Free-stack index of sequence b's last page when the step opens it, or -1:
 * the block table holds every page. */
template <bool NEW>
__device__ __forceinline__ int tail_pop(const AttnBase &p, int b) {
  return NEW ? p.nt.tail_pop[b] : -1;
}

__device__ __forceinline__ void raise_status(const AttnBase &p, int code, int diag) {
  atomicCAS(&p.status[ST_CODE], 0, code);
  atomicExch(&p.status[ST_DIAG], diag);
  atomicExch(&p.status[ST_ABORT], 1);
}

/* The wait for copies that a CTA has issued, before it exits: one still in
 * flight would write shared memory that the next CTA owns.  Not the handle's
 * wait limit, which may be set below the time a copy takes (1 us at least). */
constexpr long long DRAIN_LIMIT_NS = 2000000000LL;

/* Bounded wait on an mbarrier phase; false on abort or timeout. */
static __device__ __noinline__ bool wait_phase(uint32_t bar, uint32_t parity, const AttnBase &p,
                                        int diag, bool honour_abort, long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (honour_abort && ld_volatile(&p.status[ST_ABORT])) return false;
    if (globaltimer() - t0 > limit_ns) {
      raise_status(p, MD_ERR_DEVICE_TIMEOUT, diag);
      return false;
    }
  }
}

/* Address of the 16-byte chunk holding (row, d..d+7) of a stage stored as two
 * 64-column halves of 128-byte rows with the TMA 128-byte swizzle. */
template <int PS>
__device__ __forceinline__ uint32_t swz(uint32_t stage, int row, int d) {
  const int half = d >> 6;
  const int chunk = (d & 63) >> 3;
  return stage + half * (2 * PS * 128) + row * 128 + ((chunk ^ (row & 7)) << 4);
}

/* The V row that a lane's ldmatrix reads (row PS + v of a stage), as the row's
 * address in either 64-column half: the stage's while token v is one of its
 * `valid` cached tokens, else a row of zeros.  A masked token's weight is 0,
 * but the MMA would multiply it with whatever its slot holds, and 0 times a
 * stale Inf or NaN (an uninitialised row of a caller's pool, a page another
 * sequence left) is NaN in every head's output.  Choosing the address costs a
 * few instructions per tile; zeroing the stale rows in the stage, in code that
 * only a partial tile runs, took 0.25 to 0.4 us of a 6.4 us layer launch (a
 * cold branch), masking the fragments 0.16. */
struct VRow {
  uint32_t half0, half1;
};
template <int PS>
__device__ __forceinline__ VRow v_row(uint32_t stage, uint32_t zero_row, int v, int valid) {
  const uint32_t row = stage + (PS + v) * 128;
  return {v < valid ? row : zero_row, v < valid ? row + 2 * PS * 128 : zero_row};
}
/* Address of the 16-byte chunk holding dims d .. d+7 of such a row. */
__device__ __forceinline__ uint32_t v_chunk(const VRow &r, int v, int d) {
  return (d < 64 ? r.half0 : r.half1) + ((((d & 63) >> 3) ^ (v & 7)) << 4);
}

/* A decode step's new token: one warp writes the K and V rows (16 bytes per
 * lane: K in lanes 0..15, V in 16..31) to token `off` of page `phys`; lane 0
 * of the first layer's KV head 0 starts the token's state. */
__device__ __forceinline__ void store_new_token(const AttnBase &p, int b, int l, int kvh, int ps, int off, int phys,
                                                const uint4 &v, int lane) {
  const int row = (lane < 16 ? 0 : ps) + off;
  *(uint4 *)(p.nt.pool + ((((size_t)l * p.P_phys + phys) * p.Hkv + kvh) * 2 * ps + row) * D + (lane & 15) * 8) = v;
  if (p.nt.init_state && l == p.l0 && kvh == 0 && lane == 0) {
    const size_t slot = (size_t)phys * ps + off, last = (size_t)b * p.P_max + p.n_pages[b] - 1;
    p.nt.region[slot] = p.nt.tail_region[b];
    p.nt.t_ref[slot] = p.nt.insert_step;
    p.nt.t_ins[slot] = p.nt.insert_step;
    p.nt.a[slot] = 0.f;
    p.nt.window[slot] = 0.f;
    p.nt.ahat[slot] = 0.f;
    p.nt.prio[slot] = 0.f;
    if (p.nt.tail_pop[b] >= 0) p.nt.block_table[last] = phys;
    p.nt.page_fill[last] = (uint8_t)(off + 1);
    p.nt.seq_tokens[b] += 1;
  }
}

/* sum over the heads of exp2(score - max) / Z: the mass one token receives
 * from the query heads of one KV head (padded heads: 1/Z = 0). */
__device__ __forceinline__ float token_mass(const float4 &s0, const float4 &s1, const float (&fm)[GP],
                                            const float (&fz)[GP]) {
  float m = exp2f(s0.x - fm[0]) * fz[0] + exp2f(s0.y - fm[1]) * fz[1] + exp2f(s0.z - fm[2]) * fz[2] +
            exp2f(s0.w - fm[3]) * fz[3];
  m += exp2f(s1.x - fm[4]) * fz[4] + exp2f(s1.y - fm[5]) * fz[5] + exp2f(s1.z - fm[6]) * fz[6] +
       exp2f(s1.w - fm[7]) * fz[7];
  return m;
}

}  // namespace md

#endif
