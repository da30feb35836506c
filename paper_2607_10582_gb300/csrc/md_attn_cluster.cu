/* Stage 1 for launches of one to a few waves of CTAs (cluster_plan draws the
 * line): the same attention and exact mass as attn_mass_kernel, with one CTA per
 * chunk of a (sequence, layer, KV head) item and the item's chunks in one
 * thread-block cluster.
 *
 * What bounds these launches is latency, not HBM: a layer of a 32-sequence
 * batch at a 430-token budget reads 12 MB (1.8 us at 6.8 TB/s).  The
 * persistent kernel puts a producer, a score round trip through L2, partials
 * in global memory and a polled counter on that path.  Here
 *   - a warp issues the TMA copies of its own 16-token tiles (tile i of the
 *     chunk belongs to warp i % NW) and refills its own stages, so there is no
 *     producer, no empty barrier and no block barrier before the merge;
 *   - raw scores stay in shared memory;
 *   - every chunk pushes its (m, Z) and the slices of its O into the shared
 *     memory of the item's other CTAs; after one cluster barrier each CTA has
 *     everything for its slice of the output and its own tokens' masses.
 * LONG: chunks whose scores do not fit shared memory keep them in the
 * workspace's scratch (L2), and a lane's page ids are loaded 32 tiles at a time.
 * A cluster's CTAs are co-scheduled by the hardware, so nothing polls; the
 * only software waits are the bounded ones on the CTA's own copies. */
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "md_attn.cuh"

namespace md {

namespace {

constexpr int TILE_BYTES = 2 * TILE * D * 2;      // 16 K rows and 16 V rows
constexpr int HALF_BYTES = TILE_BYTES / 2;        // their 64-column halves
constexpr int OS = D + 4;                         // padded row of a warp's O^T (conflict-free stores)
constexpr int SCORE_BYTES = TILE * GP * 4;        // one tile's raw scores
constexpr int STAGES = 2;                         // tiles in flight per warp
constexpr int ZERO_BYTES = 128;                   // a row of zeros in place of stale V rows
/* zeros, barriers, wm, wl [warps][8], fin [16] */
constexpr int misc_bytes(int warps) { return ZERO_BYTES + warps * STAGES * 8 + (2 * warps * GP + 2 * GP) * 4; }
/* from every CTA of the cluster: (m, Z) per head, its O over this CTA's slice */
constexpr int XCH_BYTES = (MAX_CLUSTER * GP * 2 + GP * D) * 4;
constexpr int CLUSTER_SMEM = 227 * 1024, SM_SMEM = 228 * 1024;   // most a block may have, an SM has
constexpr double LONG_SCORES = 48e6;              // most bytes of spilled scores (L2 is 129 MB, K/V stream through it)
static_assert(GP * OS * 4 <= TILE_BYTES, "a warp's O^T fits one of its stages");
static_assert(D % (8 * MAX_CLUSTER) == 0, "8 consecutive elements of O lie in one slice");

}  // namespace

/* warp_tiles: tiles per warp whose scores are kept here (LONG: 0) */
static size_t cluster_smem(int warps, int C, int warp_tiles) {
  return 1024 + (size_t)warps * (STAGES * TILE_BYTES + warp_tiles * SCORE_BYTES) + misc_bytes(warps) +
         (C > 1 ? XCH_BYTES : 0);
}

template <bool ALIGNED, bool ROWS, int NW, bool LONG>
__global__ void __launch_bounds__(32 * NW, NW == 4 ? 3 : 2)
    attn_cluster_kernel(const __grid_constant__ ClusterParams p, const __grid_constant__ CUtensorMap tmap) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *ring = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float *scores = (float *)(ring + NW * STAGES * TILE_BYTES);
  float *zero_row = scores + (LONG ? 0 : (size_t)NW * p.warp_tiles * TILE * GP);
  float *wm = zero_row + ZERO_BYTES / 4;
  float *wl = wm + NW * GP;
  float *fin = wl + NW * GP;      // [16] the item's per-head max, then 1/Z (one chunk per item)
  uint64_t *full = (uint64_t *)(fin + 2 * GP);
  float *xml = (float *)(full + NW * STAGES);   // [C][8][2]
  float *xo = xml + MAX_CLUSTER * GP * 2;           // [C][G * 128 / C]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int mi = lane >> 3, rr = lane & 7;
  const uint32_t ring_u32 = smem_u32(ring) + warp * STAGES * TILE_BYTES;   // this warp's stages
  const uint32_t bar_u32 = smem_u32(full + warp * STAGES);
  const uint32_t zero_u32 = smem_u32(zero_row);
  const int G = p.G, C = p.C;
  const float NEG_INF = -INFINITY;

  if (lane < STAGES) {   // each barrier is made visible by the lane that initialised it
    mbar_init(bar_u32 + lane * 8, 1);
    fence_barrier_init();
  }
  if (lane == 0) tma_prefetch_desc(&tmap);
  if (lane < ZERO_BYTES / 16) ((uint4 *)zero_row)[lane] = make_uint4(0, 0, 0, 0);   // every warp: all write the same
  __syncwarp();
  if (C > 1) cluster_arrive();   // this CTA runs: the others may write its shared memory

  /* the unit: (sequence, layer, KV head, chunk) and its tiles [t0, t1) */
  const int item = blockIdx.x / C, rank = blockIdx.x - item * C;
  const int lh = p.L_launch * p.Hkv;
  const int b = item / lh;
  const int l = p.l0 + (item - b * lh) / p.Hkv;
  const int kvh = item % p.Hkv;
  const int n_tok = p.n_tokens[b];
  const int tpp = p.ps / TILE, shift = tpp - 1;      // tiles per page: 1 or 2
  const int last = p.n_pages[b] - 1;
  const bool add = !ROWS && p.nt.free_stack != nullptr;   // this launch appends the new tokens
  const int pop = add ? p.nt.tail_pop[b] : -1;
  const int tail_fill = add ? p.nt.tail_fill[b] : 0;
  /* contiguous pages: the tiles that hold tokens; region-aligned pages: all
   * tiles of all pages, each masked by its page's fill */
  const int tiles = ALIGNED ? (last + 1) * tpp : (n_tok + TILE - 1) / TILE;
  const int t0 = (int)((long long)rank * tiles / C), t1 = (int)((long long)(rank + 1) * tiles / C);
  const int nt = t1 - t0 > warp ? (t1 - t0 - warp + NW - 1) / NW : 0;   // this warp's tiles (not LONG: at most 32)

  /* Lane i keeps the page id and the token count of the warp's tile i (LONG:
   * 32 k + i, and id2, fill2 those of the next 32).
   * Layers after a step's first one only read pages and table entries that
   * were complete before that first layer's launch (the new token's own rows
   * and table entry come from the launch parameters), so their K/V copies
   * start before the kernel ahead has finished. */
  if (!p.early) pdl_wait();
  auto load_ids = [&](int n0, int &page, int &valid) {   // of tiles n0 .. n0 + 31
    page = valid = 0;
    const int tile = t0 + warp + NW * (n0 + lane);
    if (n0 + lane < nt) {
      const int pg = tile >> shift;
      page = *(pop >= 0 && pg == last ? p.nt.free_stack + pop : p.block_table + (size_t)b * p.P_max + pg);
      if (ALIGNED)
        valid = (add && pg == last ? tail_fill : p.page_fill[(size_t)b * p.P_max + pg]) - (tile & (tpp - 1)) * TILE;
      else
        valid = n_tok - tile * TILE;
    }
  };
  int id, fill, id2 = 0, fill2 = 0;
  load_ids(0, id, fill);
  if (LONG) load_ids(32, id2, fill2);
  const uint64_t pol = policy_evict_first();
  auto copy_tile = [&](int n, int tile, int page) {
    const uint32_t st = ring_u32 + (n % STAGES) * TILE_BYTES, bar = bar_u32 + (n % STAGES) * 8;
    const int y = (tile & (tpp - 1)) * TILE, row = (l * p.P_phys + page) * p.Hkv + kvh;
    mbar_arrive_expect_tx(bar, TILE_BYTES);
    tma_load_4d(st, &tmap, 0, y, 0, row, bar, pol);
    tma_load_4d(st + HALF_BYTES, &tmap, 64, y, 0, row, bar, pol);
  };
  if (p.early) {
    if (lane < STAGES && lane < nt) copy_tile(lane, t0 + warp + NW * lane, id);
    pdl_wait();
  }
  pdl_trigger();

  /* Q^T fragments (B operand): head g, dims 16kk + {2t, 2t+1} and + 8 */
  uint32_t qf[8][2];
  {
    const uint16_t *qrow =
        p.q + (((size_t)b * p.q_layers + (l - p.l0)) * p.Hq + (size_t)kvh * G + g) * D + 2 * t;
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      qf[kk][0] = g < G ? *(const uint32_t *)(qrow + 16 * kk) : 0u;
      qf[kk][1] = g < G ? *(const uint32_t *)(qrow + 16 * kk + 8) : 0u;
    }
  }
  if (!p.early && lane < STAGES && lane < nt) copy_tile(lane, t0 + warp + NW * lane, id);
  /* the new token's rows (16 bytes per lane: K, then V), if this warp has its tile */
  int n_tail = -1, off = 0;
  uint4 row_new = make_uint4(0, 0, 0, 0);
  if (add) {
    off = tail_fill - 1;
    const int x = last * tpp + off / TILE - t0 - warp;
    if (x >= 0 && x % NW == 0 && x / NW < nt) {
      n_tail = x / NW;
      const long long src = b * p.nt.sb + (l - p.l0) * p.nt.sl + kvh * D + (lane & 15) * 8;
      row_new = *(const uint4 *)((lane < 16 ? p.nt.k_new : p.nt.v_new) + src);
    }
  }

  float m0 = NEG_INF, m1 = NEG_INF, l0 = 0.f, l1 = 0.f;
  float o[8][4];
#pragma unroll
  for (int mt = 0; mt < 8; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f;
  const bool hv0 = 2 * t < G, hv1 = 2 * t + 1 < G;
  float *sc = (LONG ? p.scratch + (size_t)blockIdx.x * NW * p.warp_tiles * TILE * GP : scores) +
              (size_t)warp * p.warp_tiles * TILE * GP;
  const uint64_t acc_pol = policy_evict_last();
  int issued = min(nt, STAGES);
  int n = 0;
  for (; n < nt; ++n) {
    const uint32_t st = ring_u32 + (n % STAGES) * TILE_BYTES;
    /* the call, and the fetch of its code, only if the copy has not landed in
     * the first try: 32 sequences of 430 tokens layer by layer 229.9 -> 225.7 us */
    const uint32_t bar = bar_u32 + (n % STAGES) * 8, parity = (n / STAGES) & 1;
    const bool landed = mbar_try_wait(bar, parity) || wait_phase(bar, parity, p, 4, false, p.spin_limit_ns);
    if (!__all_sync(0xffffffffu, landed)) break;
    if (LONG && n > 0 && n % 32 == 0) {
      id = id2;
      fill = fill2;
      load_ids(n + 32, id2, fill2);
    }
    const int valid = __shfl_sync(0xffffffffu, fill, n & 31);
    if (n == n_tail) {
      const int r = off % TILE + (lane < 16 ? 0 : TILE);
      *(uint4 *)(ring + (swz<TILE>(st, r, (lane & 15) * 8) - smem_u32(ring))) = row_new;
      store_new_token(p, b, l, kvh, p.ps, off, __shfl_sync(0xffffffffu, id, n & 31), row_new, lane);
      __syncwarp();
    }
    /* two accumulators: half the chain of dependent MMAs */
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      uint32_t a0, a1, a2, a3;
      ldmatrix_x4(swz<TILE>(st, (mi & 1) * 8 + rr, kk * 16 + (mi >> 1) * 8), a0, a1, a2, a3);
      mma_bf16(kk & 1 ? acc2 : acc, a0, a1, a2, a3, qf[kk][0], qf[kk][1]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] += acc2[i];
    const bool va = g < valid, vb = g + 8 < valid;
    acc[0] = (va && hv0) ? acc[0] * p.scale_log2 : NEG_INF;
    acc[1] = (va && hv1) ? acc[1] * p.scale_log2 : NEG_INF;
    acc[2] = (vb && hv0) ? acc[2] * p.scale_log2 : NEG_INF;
    acc[3] = (vb && hv1) ? acc[3] * p.scale_log2 : NEG_INF;
    float *srow = sc + ((size_t)n * TILE + g) * GP + 2 * t;
    if (LONG) {
      st_v2_hint(srow, acc[0], acc[1], acc_pol);
      st_v2_hint(srow + 8 * GP, acc[2], acc[3], acc_pol);
    } else {
      *(float2 *)srow = make_float2(acc[0], acc[1]);
      *(float2 *)(srow + 8 * GP) = make_float2(acc[2], acc[3]);
    }
    float mx0 = fmaxf(acc[0], acc[2]), mx1 = fmaxf(acc[1], acc[3]);
#pragma unroll
    for (int x = 4; x < 32; x <<= 1) {
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, x));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, x));
    }
    const float n0 = fmaxf(m0, mx0), n1 = fmaxf(m1, mx1);
    const float r0 = n0 == NEG_INF ? 0.f : n0, r1 = n1 == NEG_INF ? 0.f : n1;
    const float al0 = exp2f(m0 - r0), al1 = exp2f(m1 - r1);
    m0 = n0;
    m1 = n1;
    l0 *= al0;
    l1 *= al1;
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
      o[mt][0] *= al0;
      o[mt][1] *= al1;
      o[mt][2] *= al0;
      o[mt][3] *= al1;
    }
    const float p00 = exp2f(acc[0] - r0), p01 = exp2f(acc[1] - r1);
    const float p10 = exp2f(acc[2] - r0), p11 = exp2f(acc[3] - r1);
    l0 += p00 + p10;
    l1 += p01 + p11;
    const uint32_t b0 = movmatrix_trans(pack_bf16(p00, p01));
    const uint32_t b1 = movmatrix_trans(pack_bf16(p10, p11));
    const VRow vr = v_row<TILE>(st, zero_u32, (mi >> 1) * 8 + rr, valid);
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
      uint32_t a0, a1, a2, a3;
      ldmatrix_x4_trans(v_chunk(vr, rr, mt * 16 + (mi & 1) * 8), a0, a1, a2, a3);
      mma_bf16(o[mt], a0, a1, a2, a3, b0, b1);
    }
    /* refill the stage; its reads (generic proxy) come before the copy (async) */
    __syncwarp();
    if (n + STAGES < nt) {
      const int m = n + STAGES;
      const int page = __shfl_sync(0xffffffffu, LONG && m / 32 != n / 32 ? id2 : id, m & 31);
      if (lane == 0) {
        fence_proxy_async_smem();
        copy_tile(n + STAGES, t0 + warp + NW * (n + STAGES), page);
      }
      ++issued;
    }
  }
  if (n < nt)   // a wait ran out: the copies still in flight must land before the CTA exits
    for (; n < issued; ++n) wait_phase(bar_u32 + (n % STAGES) * 8, (n / STAGES) & 1, p, 2, false, DRAIN_LIMIT_NS);

  /* ---- merge the warps: (m, Z, O) of the chunk ---- */
#pragma unroll
  for (int x = 4; x < 32; x <<= 1) {
    l0 += __shfl_xor_sync(0xffffffffu, l0, x);
    l1 += __shfl_xor_sync(0xffffffffu, l1, x);
  }
  if (g == 0) {
    wm[warp * GP + 2 * t] = m0;
    wm[warp * GP + 2 * t + 1] = m1;
    wl[warp * GP + 2 * t] = l0;
    wl[warp * GP + 2 * t + 1] = l1;
  }
  {
    float *wo = (float *)(ring + warp * STAGES * TILE_BYTES);   // this warp's first stage: its tiles are done
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
      wo[(2 * t) * OS + 16 * mt + g] = o[mt][0];
      wo[(2 * t + 1) * OS + 16 * mt + g] = o[mt][1];
      wo[(2 * t) * OS + 16 * mt + g + 8] = o[mt][2];
      wo[(2 * t + 1) * OS + 16 * mt + g + 8] = o[mt][3];
    }
  }
  __syncthreads();
  const size_t out0 = (((size_t)b * p.q_layers + (l - p.l0)) * p.Hq + (size_t)kvh * G) * D;
  {
    constexpr int DPT = GP / (NW / 4), TPH = D / DPT;   // dims per thread, threads per head
    const int h = threadIdx.x / TPH, x = threadIdx.x % TPH, d0 = x * DPT;
    float M = NEG_INF, Z = 0.f, acc[DPT];
#pragma unroll
    for (int w = 0; w < NW; ++w) M = fmaxf(M, wm[w * GP + h]);
    const float Mr = M == NEG_INF ? 0.f : M;
#pragma unroll
    for (int i = 0; i < DPT; ++i) acc[i] = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float f = exp2f(wm[w * GP + h] - Mr);
      Z += f * wl[w * GP + h];
      const float *wo = (const float *)(ring + w * STAGES * TILE_BYTES) + h * OS + d0;
#pragma unroll
      for (int i = 0; i < DPT; ++i) acc[i] += f * wo[i];
    }
    if (C == 1) {
      const float inv = Z > 0.f ? 1.f / Z : 0.f;
      if (x == 0) {
        fin[h] = Mr;
        fin[GP + h] = inv;
      }
      if (h < G) {
        uint32_t w[DPT / 2];
#pragma unroll
        for (int i = 0; i < DPT / 2; ++i) w[i] = pack_bf16(acc[2 * i] * inv, acc[2 * i + 1] * inv);
        uint16_t *dst = p.out + out0 + h * D + d0;
        if (p.out16) {
#pragma unroll
          for (int i = 0; i < DPT / 2; i += 2) *(uint2 *)(dst + 2 * i) = make_uint2(w[i], w[i + 1]);
        } else {
#pragma unroll
          for (int i = 0; i < DPT; ++i) dst[i] = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
        }
      }
    } else {
      /* push: (m, Z) of head h to CTA x from thread x of the head's, and these
       * elements to the CTA whose output slice they are in */
      cluster_wait();
      const int SE = G * D / C;
      if (x < C) st_cluster_v2(cluster_map(smem_u32(xml + (rank * GP + h) * 2), x), M, Z);
      if (h < G) {
        const int e = h * D + d0, to = e / SE;
        const uint32_t dst = cluster_map(smem_u32(xo + rank * SE + (e - to * SE)), to);
#pragma unroll
        for (int i = 0; i < DPT; i += 4) st_cluster_v4(dst + 4 * i, acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
      }
      __syncwarp();
      cluster_arrive();
    }
  }

  /* ---- the item's softmax over the cluster's chunks ---- */
  float fm[GP], fz[GP];
  if (C == 1) {
    __syncthreads();
#pragma unroll
    for (int h = 0; h < GP; ++h) {
      fm[h] = fin[h];
      fz[h] = h < G ? fin[GP + h] : 0.f;
    }
  } else {
    cluster_wait();
    /* every warp: lane (h, part) has chunks part, part + 4, ... */
    const int h = lane & 7, part = lane >> 3;
    float mj[MAX_CLUSTER / 4];
    float M = NEG_INF, Z = 0.f;
#pragma unroll
    for (int i = 0; i < MAX_CLUSTER / 4; ++i) {
      const int j = part + 4 * i;
      mj[i] = j < C ? xml[(j * GP + h) * 2] : NEG_INF;
      M = fmaxf(M, mj[i]);
    }
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 8));
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 16));
    const float Mr = M == NEG_INF ? 0.f : M;
#pragma unroll
    for (int i = 0; i < MAX_CLUSTER / 4; ++i) {
      const int j = part + 4 * i;
      mj[i] = exp2f(mj[i] - Mr);      // from here on the chunk's factor
      Z += j < C ? mj[i] * xml[(j * GP + h) * 2 + 1] : 0.f;
    }
    Z += __shfl_xor_sync(0xffffffffu, Z, 8);
    Z += __shfl_xor_sync(0xffffffffu, Z, 16);
    const float inv = Z > 0.f ? 1.f / Z : 0.f;
#pragma unroll
    for (int x = 0; x < GP; ++x) {
      fm[x] = __shfl_sync(0xffffffffu, Mr, x);
      fz[x] = __shfl_sync(0xffffffffu, inv, x);
    }
    /* this chunk's slice of the item's output */
    const int SE = G * D / C;
    for (int e0 = 0; e0 < SE; e0 += 32 * NW) {
      const int e = e0 + threadIdx.x;
      const int he = min(rank * SE + e, G * D - 1) >> 7;
      float v = 0.f;
#pragma unroll
      for (int i = 0; i < MAX_CLUSTER / 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float f = __shfl_sync(0xffffffffu, mj[i], he + 8 * q);
          if (4 * i + q < C && e < SE) v += f * xo[(4 * i + q) * SE + e];
        }
      const float inv_e = __shfl_sync(0xffffffffu, inv, he);
      if (e < SE) {
        const __nv_bfloat16 bv = __float2bfloat16_rn(v * inv_e);
        p.out[out0 + rank * SE + e] = *(const uint16_t *)&bv;
      }
    }
  }

  /* ---- token masses from this warp's scores: a half warp per tile, four
   * tiles' scores loaded before the first is used ---- */
  if (LONG && nt > 32) load_ids(0, id, fill);
  for (int x = 0; x < nt; x += 8) {
    if (LONG && x > 0 && x % 32 == 0) load_ids(x, id, fill);
    const int r = lane & 15;
    float4 s0[4], s1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int nn = x + 2 * k + (lane >> 4);
      const float4 *s = (const float4 *)(sc + ((size_t)nn * TILE + r) * GP);
      if (nn < nt) {
        s0[k] = LONG ? __ldcg(s) : s[0];
        s1[k] = LONG ? __ldcg(s + 1) : s[1];
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int nn = x + 2 * k + (lane >> 4);
      const int page = __shfl_sync(0xffffffffu, id, nn & 31);
      const int valid = __shfl_sync(0xffffffffu, fill, nn & 31);
      if (nn < nt && r < valid) {
        const float m = token_mass(s0[k], s1[k], fm, fz);
        const int tile = t0 + warp + NW * nn;
        const size_t slot = (size_t)page * p.ps + (tile & (tpp - 1)) * TILE + r;
        if (ROWS)
          p.mass[(size_t)(l * p.Hkv + kvh) * p.slots + slot] = m;
        else
          red_add_u64_hint(p.mass_acc + slot, __float2ull_rn(m * MASS_SCALE), acc_pol);
      }
    }
  }
}

/* CTAs that run at once on the current device as clusters of 2^lgC, with
 * 1, 2 or 3 CTAs of 4 warps per SM (shared memory decides which) or one of 8:
 * the GPU's processing clusters hold whole thread-block clusters only (152 SMs
 * take 304 CTAs of 4 warps, 288 as clusters of 8, 224 as clusters of 16). */
struct ClusterSlots {
  int w4[3][5], w8[5];
  std::atomic<bool> ready{false};
};
static ClusterSlots g_slots[64];   // per device ordinal, filled once under g_slots_mu
static std::mutex g_slots_mu;

template <int NW>
static cudaError_t prepare_warps(int per_sm, int *slots) {
  cudaError_t e = cudaSuccess;
  for (const void *k : {(const void *)attn_cluster_kernel<false, true, NW, false>,
                        (const void *)attn_cluster_kernel<true, false, NW, false>,
                        (const void *)attn_cluster_kernel<false, false, NW, false>,
                        (const void *)attn_cluster_kernel<true, false, NW, true>,
                        (const void *)attn_cluster_kernel<false, false, NW, true>}) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, CLUSTER_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  for (int lg = 0; lg < 5 && e == cudaSuccess; ++lg) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1 << lg;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(1 << lg);
    cfg.blockDim = dim3(32 * NW);
    cfg.dynamicSmemBytes = SM_SMEM / per_sm - 1024;
    if (cfg.dynamicSmemBytes > CLUSTER_SMEM) cfg.dynamicSmemBytes = CLUSTER_SMEM;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, attn_cluster_kernel<false, false, NW, false>, &cfg);
    slots[lg] = n << lg;
  }
  return e;
}

cudaError_t cluster_prepare() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaSuccess;   // no table: cluster_plan keeps the persistent kernel
  ClusterSlots &g = g_slots[dev];
  std::lock_guard<std::mutex> lock(g_slots_mu);
  if (g.ready.load(std::memory_order_relaxed)) return cudaSuccess;
  for (int per = 3; per >= 1 && e == cudaSuccess; --per) e = prepare_warps<4>(per, g.w4[per - 1]);
  if (e == cudaSuccess) e = prepare_warps<8>(1, g.w8);
  if (e == cudaSuccess && g.w4[0][0] > 0) g.ready.store(true, std::memory_order_release);
  return e;
}

/* 16-token tiles the kernel reads of sequence b. */
static int seq_tiles(const AttnBase &p, int b) {
  return p.page_fill ? p.n_pages[b] * (p.ps / TILE) : (p.n_tokens[b] + TILE - 1) / TILE;
}

/* Which kernel, and how many CTAs and warps per item: the least of these costs
 * in us, fitted to 57 launch shapes timed on a GB300 in every form (1 to 64
 * sequences of 128 to 30,000 tokens, one layer and whole steps).  Over 48 shapes
 * (1 to 64 sequences of 30 to 100,000 tokens) its choice takes 1.4% longer than
 * the best form of each, 14% at worst (5 sequences of 700 tokens in 36 layers,
 * 33.0 and 29.1), and the persistent kernel alone 34% longer than its choice.  n: 16-token tiles per warp, N: CTAs, hbm: the K/V bytes at 6.8 TB/s.
 *   One wave (the N CTAs run at once): the CTA's time (launch chain, prologue
 *     and merge in `base`, 0.65 or 0.74 per tile of its warps; the cluster's
 *     exchange raises `base`) or HBM's, and 0.006 N.  One layer of 1 x 430
 *     tokens: 4.3 us with 8 CTAs per item, 6.7 with one, 12.8 persistent; of
 *     32 x 430: 6.8, persistent 12.7; of 32 x 4,096: 23.4, persistent 32.0.
 *   More waves, one CTA per item: the hardware hands out CTAs as others end,
 *     so the chip idles for part of one CTA at the end.  4 warps while a CTA
 *     is short (up to 96 tiles; a step of 2,304 items of 27 tiles 88 us,
 *     persistent 90; 768 of 63, 68 and 73), above that 8 warps, which stream
 *     one item twice as fast (384 of 150, 76 and 99; 392 of 100, 58 and 85).
 *   More waves of clusters: launching them costs 0.0075 N (24 items of 813
 *     tiles, 30.4 and 33.9; 100 of 250, 39.6 and 43.1).
 *   LONG, one wave: as one wave, with the score rows' way through L2 on top.  One
 *     layer of 16 x 13,001 tokens 37.0 us, persistent 44.0; of 24 x 9,000,
 *     37.5 and 44.9; of 50 x 4,000, 36.8 and 45.1; a step of 3 x 30,000 tokens
 *     in 8 layers 121 and 139.  (22 shapes of 4,000 to 100,000 tokens.)
 *   Persistent: hbm and about 14 us of split, combine, ramp and tail, which a
 *     launch of several hundred us hides (2,304 items of 107 tiles: 281 us, 286
 *     with 8 warps per item). */
ClusterPlan cluster_plan(const AttnBase &p, size_t scratch_floats) {
  ClusterPlan best;
  int dev = 0, T = 1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 ||
      !g_slots[dev].ready.load(std::memory_order_acquire))
    return best;
  long long sum = 0;
  for (int b = 0; b < p.n_seqs; ++b) {
    const int t = seq_tiles(p, b);
    T = std::max(T, t);
    sum += t;
  }
  const int lh = p.L_launch * p.Hkv;
  const long long items = (long long)p.n_seqs * lh;
  const double hbm = (double)sum * lh * TILE_BYTES / 6.8e6;
  double least = 0.97 * (1.01 * hbm + 14.0 * std::min(1.0, 100.0 / hbm));
  for (int warps = 4; warps <= 8; warps += 4)
    for (int lg = 0; lg < 5; ++lg) {
      const int C = 1 << lg, n = ((T + C - 1) / C + warps - 1) / warps;
      const size_t smem = cluster_smem(warps, C, n);
      if (n > 32 || smem > CLUSTER_SMEM) continue;
      const int per_sm = std::min(3, (int)(SM_SMEM / (smem + 1024)));
      const long long N = items * C, slots = warps == 4 ? g_slots[dev].w4[per_sm - 1][lg] : g_slots[dev].w8[lg];
      if (slots < C) continue;
      const double base = warps == 4 ? (C == 1 ? 2.25 : 3.7) : (C == 1 ? 2.85 : 4.0);
      const double cta = base + (warps == 4 ? 0.65 : 0.74) * n;
      double cost;
      if (N <= slots)
        cost = std::max(cta, hbm + 3.0) + 0.006 * N;
      else if (C > 1)
        cost = std::max((double)((N + slots - 1) / slots) * cta * 1.1, hbm + 0.6 * cta) + 1.5 + 0.0075 * N;
      else if ((warps == 4) == (T <= 96))
        cost = hbm + 2.0 + 0.003 * N + (warps == 4 ? 0.2 * cta : 0.0);
      else
        continue;
      if (cost < least) {
        least = cost;
        best.C = C;
        best.warps = warps;
        best.warp_tiles = n;
      }
    }
  /* LONG: one wave only; against the persistent kernel at its measured cost
   * for such launches, 8% of hbm above the figure that the others have to beat */
  if (best.C == 0) least += 0.08 * hbm;
  for (int warps = 4; warps <= 8 && (double)sum * lh * SCORE_BYTES < LONG_SCORES; warps += 4)
    for (int lg = 0; lg < 5; ++lg) {
      const int C = 1 << lg, n = ((T + C - 1) / C + warps - 1) / warps;
      const long long N = items * C, slots = warps == 4 ? g_slots[dev].w4[2][lg] : g_slots[dev].w8[lg];
      if (N > slots || (size_t)N * warps * n * TILE * GP > scratch_floats) continue;
      const double base = warps == 4 ? (C == 1 ? 2.25 : 3.7) : (C == 1 ? 2.85 : 4.0);
      const int shared = warps == 4 ? (int)((N - 1) / g_slots[dev].w4[0][0]) : 0;   // more CTAs on an SM
      const double cta = (base + (warps == 4 ? 0.75 : 0.85) * n) * (1.0 + 0.1 * shared);
      const double cost = std::max(cta, hbm + 4.0) + 0.003 * N + 1.0 + 0.1 * hbm;
      if (cost < least) {
        least = cost;
        best.C = C;
        best.warps = warps;
        best.warp_tiles = n;
        best.spill = true;
      }
    }
  return best;
}

ClusterPlan cluster_form(const AttnBase &p, size_t scratch_floats, int C, int warps, bool spill) {
  ClusterPlan f;
  int T = 1;
  for (int b = 0; b < p.n_seqs; ++b) T = std::max(T, seq_tiles(p, b));
  const int n = ((T + C - 1) / C + warps - 1) / warps;
  const size_t ctas = (size_t)p.n_seqs * p.L_launch * p.Hkv * C;
  if (spill ? ctas * warps * n * TILE * GP > scratch_floats : n > 32 || cluster_smem(warps, C, n) > CLUSTER_SMEM)
    return f;
  f.C = C;
  f.warps = warps;
  f.warp_tiles = n;
  f.spill = spill;
  return f;
}

template <int NW, bool LONG>
static cudaError_t launch_warps(const cudaLaunchConfig_t &cfg, const ClusterParams &p, const CUtensorMap &tmap) {
  if (!p.mass_acc)
    return LONG ? cudaErrorInvalidValue : cudaLaunchKernelEx(&cfg, attn_cluster_kernel<false, true, NW, false>, p, tmap);
  return p.page_fill ? cudaLaunchKernelEx(&cfg, attn_cluster_kernel<true, false, NW, LONG>, p, tmap)
                     : cudaLaunchKernelEx(&cfg, attn_cluster_kernel<false, false, NW, LONG>, p, tmap);
}

cudaError_t launch_cluster(const AttnBase &base, const ClusterPlan &plan, bool early, float *scratch,
                           const CUtensorMap &tmap, cudaStream_t s) {
  ClusterParams p;
  (AttnBase &)p = base;
  p.C = plan.C;
  p.warp_tiles = plan.warp_tiles;
  p.early = early;
  p.scratch = scratch;
  p.out16 = ((uintptr_t)p.out & 15) == 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.n_seqs * p.L_launch * p.Hkv * p.C);
  cfg.blockDim = dim3(32 * plan.warps);
  cfg.dynamicSmemBytes = cluster_smem(plan.warps, p.C, plan.spill ? 0 : p.warp_tiles);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = p.C;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (plan.spill) return plan.warps == 4 ? launch_warps<4, true>(cfg, p, tmap) : launch_warps<8, true>(cfg, p, tmap);
  return plan.warps == 4 ? launch_warps<4, false>(cfg, p, tmap) : launch_warps<8, false>(cfg, p, tmap);
}

}  // namespace md
