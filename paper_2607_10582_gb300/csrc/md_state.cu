/* Stages 0, 2, 3, 4 of the MemDecay step and the workspace initialiser.
 *
 *   append   write new tokens' K/V into the page pool (taking fresh pages
 *            from the free stack) and start each token's state: region label,
 *            t_ref = insertion step, a = 0 (Sec. III-A; Fig. 1 "append KV").
 *            Prompts and tool outputs, decode steps whose K/V lie in host
 *            memory, and those whose attention launch does not append.
 *   score    per page, one lane per token: Abar from the window accumulator
 *            and the step's mass summed over layers and heads (Sec. III-C;
 *            a fixed-point accumulator the attention kernel fills), the EWMA
 *            (Eq. 2), the refresh test Abar >= tau_scale/|K_t| (Eq. 3), the
 *            retention score (Eq. 4, lambda = ln2 / half-life, Eq. 7) and the
 *            page score by a shuffle reduction over the page's lanes (Eq. 5;
 *            pinned pages and the page being written score +inf).  With
 *            fold_only it only adds the step's mass into the window accumulator.
 *   select   one CTA per sequence: radix select (4 passes of 8-bit digits
 *            over order-preserving uint32 keys, ties by logical page index)
 *            of the e lowest evictable pages, stable compaction of the block
 *            table row, push of the freed ids onto the free stack
 *            (Sec. III-D, Algorithm 1: lowest S_p first; a selection, not a
 *            sort or a heap). */
#include <float.h>

#include "md_internal.h"
#include "md_ptx.cuh"

namespace md {

/* ---------------------------------------------------------------- init --- */
__global__ void init_kernel(int32_t *free_stack, int P_phys, int *status, int *counters,
                            size_t n_items) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < (size_t)P_phys; i += stride)
    free_stack[i] = P_phys - 1 - (int)i;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_items; i += stride)
    counters[i] = 0;
  if (blockIdx.x == 0 && threadIdx.x < ST_WORDS) status[threadIdx.x] = 0;
}

cudaError_t launch_init(int32_t *free_stack, int P_phys, int *status, int *counters,
                        size_t n_items, cudaStream_t s) {
  init_kernel<<<304, 256, 0, s>>>(free_stack, P_phys, status, counters, n_items);
  return cudaGetLastError();
}

/* ---------------------------------------------------------- state copy --- */
/* Device-to-device copy of a state array, 16 bytes per thread and iteration.
 * In a stream of dependent launches it starts as the kernel ahead ends, where
 * a copy node waits for that one and holds up the next: a pass over 32
 * sequences of 430 tokens that reads four arrays back, 97.9 -> 87.9 us. */
__global__ void __launch_bounds__(256) copy_kernel(const __grid_constant__ CopyParams p) {
  pdl_wait();
  pdl_trigger();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += (size_t)gridDim.x * blockDim.x)
    p.dst[i] = p.src[i];
}

cudaError_t launch_copy(const CopyParams &p, cudaStream_t s) {
  const size_t blocks = (p.n + 255) / 256;
  return launch_pdl(copy_kernel, (int)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, s, p);
}

/* -------------------------------------------------------------- append --- */
__device__ __forceinline__ void start_token(const AppendTo &d, size_t slot, int region, int step) {
  d.region[slot] = (uint8_t)region;
  d.t_ref[slot] = step;
  d.t_ins[slot] = step;
  d.a[slot] = 0.f;
  d.window[slot] = 0.f;
  d.ahat[slot] = 0.f;
  d.prio[slot] = 0.f;
}

/* One thread per 16-byte piece of a token's K or V row in one (layer, head),
 * and of the query rows where those lie in pinned host memory too.  The link
 * bounds it: 165 GB/s for a kernel, 182 for the copy engine, but a copy ahead
 * of this launch has a start and a gap of its own (4.7 MB of query rows: a step
 * of 32 sequences with host buffers 141.3 -> 134.9 us). */
__global__ void append_step_kernel(const __grid_constant__ AppendStepParams p) {
  pdl_wait();
  pdl_trigger();
  const AppendTo &d = p.to;
  const unsigned lh = p.L * d.Hkv, total = p.n_seqs * lh * 32u;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total + p.q_n; i += gridDim.x * blockDim.x) {
    if (i >= total) {
      p.q_dst[i - total] = p.q_src[i - total];
      continue;
    }
    const unsigned w = i;
    const int c = w & 15, kv = (w >> 4) & 1;
    const unsigned x = w >> 5, j = x / lh, r = x - j * lh;
    const int l = p.l0 + r / d.Hkv, h = r % d.Hkv;
    const int tok = p.tok0[j], pg = tok / d.ps, off = tok - pg * d.ps, pop = p.pop[j];
    const int phys = pop < 0 ? d.block_table[(size_t)j * d.P_max + pg] : d.free_stack[pop];
    const uint16_t *src = (kv == 0 ? p.k_src : p.v_src) + (size_t)x * D;
    uint16_t *dst = d.pool + ((((size_t)l * d.P_phys + phys) * d.Hkv + h) * 2 + kv) * (size_t)d.ps * D + (size_t)off * D;
    ((uint4 *)dst)[c] = ((const uint4 *)src)[c];
    if (p.l0 == 0 && r == 0 && kv == 0 && c == 0) {
      start_token(d, (size_t)phys * d.ps + off, p.regions[j], p.insert_step);
      if (pop >= 0) d.block_table[(size_t)j * d.P_max + pg] = phys;
      d.page_fill[(size_t)j * d.P_max + pg] = (uint8_t)(off + 1);
      d.seq_tokens[j] += 1;
    }
  }
}

cudaError_t launch_append_step(const AppendStepParams &p, cudaStream_t s) {
  const long long total = (long long)p.n_seqs * p.L * p.to.Hkv * 32 + p.q_n;
  long long blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  return launch_pdl(append_step_kernel, (int)blocks, 256, 0, s, p);
}

/* The run that token i is in. */
__device__ __forceinline__ int find_run(const AppendTokensParams &p, int i) {
  int lo = 0, hi = p.n_runs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.runs[mid].start <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

/* Slot of token i in the sequence.  ALIGNED: slots skip the rest of a page
 * where the region changes. */
template <bool ALIGNED>
__device__ __forceinline__ int token_slot(const AppendTokensParams &p, int i) {
  if (!ALIGNED) return p.tok0 + i;
  if (p.slots_dev) return p.slots_dev[i];
  const AppendRun &r = p.runs[find_run(p, i)];
  return r.slot + (i - r.start);
}

/* One warp copies the K or the V rows of 16 consecutive tokens in one (layer,
 * KV head): 4 KiB, contiguous in the source, eight 16-byte loads per lane in
 * flight before the first store.  Lane j looks up where token j goes, so the
 * index arithmetic is done once per row and not once per 16 bytes: in 64-bit
 * divisions it had the copy bound by instructions.  8,192 tokens of 36 layers,
 * 302 MB read and as much written: 165 -> 98 us, 6.2 TB/s, now bound by HBM.
 * Without the staging copies of labels ahead of it, a call of 317 tokens takes
 * 12.7 -> 5.5 us in a stream of them. */
template <bool ALIGNED>
__global__ void __launch_bounds__(256, 4) append_tokens_kernel(const __grid_constant__ AppendTokensParams p) {
  pdl_wait();
  pdl_trigger();
  const AppendTo &d = p.to;
  const int lane = threadIdx.x & 31;
  const unsigned groups = (p.n + 15) / 16, items = d.L * d.Hkv * 2u * groups;
  for (unsigned w = blockIdx.x * 8 + (threadIdx.x >> 5); w < items; w += gridDim.x * 8) {
    const unsigned x = w / groups, i0 = (w - x * groups) * 16;   // x = (l * Hkv + h) * 2 + kv
    const int l = (x >> 1) / d.Hkv, hk = x - l * d.Hkv * 2, kv = x & 1;   // hk = h * 2 + kv
    const int cnt = min(16, p.n - (int)i0);
    const uint4 *src = (const uint4 *)((kv ? p.v_src : p.k_src) + ((size_t)(x >> 1) * p.n + i0) * D) + lane;
    uint4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (2 * k + (lane >> 4) < cnt) v[k] = __ldcs(src + k * 32);
    const int i = i0 + (lane & 15);
    int pg = 0, off = 0, phys = 0;
    if (i < p.n) {
      const int slot = token_slot<ALIGNED>(p, i);
      pg = slot / d.ps;
      off = slot - pg * d.ps;
      phys = pg < p.pages_before ? d.block_table[(size_t)p.seq * d.P_max + pg]
                                 : d.free_stack[p.pop_base - (pg - p.pages_before)];
    }
    const int row = ((l * d.P_phys + phys) * d.Hkv * 2 + hk) * d.ps + off;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int to = __shfl_sync(0xffffffffu, row, 2 * k + (lane >> 4));
      if (2 * k + (lane >> 4) < cnt) ((uint4 *)(d.pool + (size_t)to * D))[lane & 15] = v[k];
    }
    if (x == 0 && lane < cnt) {
      const int run = p.regions_dev ? 0 : find_run(p, i);
      const int step = p.regions_dev ? (p.steps_dev ? p.steps_dev[i] : p.insert_step) : p.runs[run].step;
      start_token(d, (size_t)phys * d.ps + off, p.regions_dev ? p.regions_dev[i] : p.runs[run].region, step);
      if (off == 0 && pg >= p.pages_before) d.block_table[(size_t)p.seq * d.P_max + pg] = phys;
      /* the last token this append puts on a page sets the page's fill */
      if (i + 1 == p.n || token_slot<ALIGNED>(p, i + 1) / d.ps != pg)
        d.page_fill[(size_t)p.seq * d.P_max + pg] = (uint8_t)(off + 1);
      if (i == 0) d.seq_tokens[p.seq] += p.n;
    }
  }
}

cudaError_t launch_append_tokens(const AppendTokensParams &p, bool aligned, cudaStream_t s) {
  const long long items = (long long)p.to.L * p.to.Hkv * 2 * ((p.n + 15) / 16);
  const int blocks = (int)(items + 7 < 152 * 4 * 8 ? (items + 7) / 8 : 152 * 4);
  return aligned ? launch_pdl(append_tokens_kernel<true>, blocks, 256, 0, s, p)
                 : launch_pdl(append_tokens_kernel<false>, blocks, 256, 0, s, p);
}

/* ------------------------------------------------------ score / fold ----- */
__device__ __forceinline__ int find_seq(const int *start, int n, int x) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

/* Uniform draw in [0, 1) for the random-baseline score: the SplitMix64
 * finaliser (Steele, Lea and Flood, 2014) of (seed, step, slot); the top 24
 * bits scaled by 2^-24 are exact in fp32. */
__device__ __forceinline__ float random_draw(unsigned long long seed, int t, size_t slot) {
  unsigned long long z = (seed * 0x9E3779B97F4A7C15ull) ^ ((unsigned long long)(unsigned)t << 40) ^
                         (unsigned long long)slot;
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (float)(z >> 40) * 5.9604644775390625e-08f;
}

/* The calibration histogram of a block (Sec. IV-B, Eq. 6's input): observed
 * mass in fixed point, so integer atomics keep the sums order-independent. */
struct CalibSmem {
  unsigned long long sum[8 * CALIB_BUCKETS];
  unsigned int cnt[8 * CALIB_BUCKETS];
};

/* Stages 2-3 for one warp's tile of 32/PS consecutive pages, one lane per
 * token slot: this lane's slot is `off` of page pg of sequence b (page_ok:
 * there is such a page).  Returns the page's score, the same in all its lanes.
 * A token's step mass is one fixed-point accumulator (the attention kernel
 * adds every (layer, KV head) into it): read and zeroed here, loaded together
 * with the token's state. */
template <int PS, bool CALIB>
__device__ __forceinline__ float score_tile(const ScoreParams &p, int b, int pg, int off, bool page_ok, bool need_mass,
                                            CalibSmem *calib) {
  const float INF = INFINITY;
  bool valid = false;
  size_t slot = 0;
  if (page_ok) {
    valid = p.page_fill ? off < p.page_fill[(size_t)b * p.P_max + pg] : pg * PS + off < p.n_tokens[b];
    slot = (size_t)p.block_table[(size_t)b * p.P_max + pg] * PS + off;
  }
  /* the token's state and its step mass, all loads independent */
  int reg = 0, tr = 0, tins = 0, ntok = 1;
  float a = 0.f, w = 0.f;
  unsigned long long macc = 0ull;
  if (valid) {
    if (need_mass) macc = __ldcs(p.mass_acc + slot);
    if (p.fold_only) {
      w = p.window[slot];
    } else {
      reg = p.region[slot];
      a = p.a[slot];
      tr = p.t_ref[slot];
      if (p.observe) w = p.window[slot];
      if (p.observe || p.score_mode == 2) ntok = p.seq_tokens ? p.seq_tokens[b] : p.n_tokens[b];
      if (CALIB || p.score_mode == 3) tins = p.t_ins[slot];
    }
  }
  /* the sum over layers and query heads, rounded once to fp32 */
  const float msum = __ull2float_rn(macc) * MASS_UNIT;
  if (valid && need_mass) p.mass_acc[slot] = 0ull;
  float s = 0.f;
  int pinned = 0, bin = -1;
  unsigned long long fx = 0ull;
  if (valid) {
    if (p.fold_only) {
      p.window[slot] = w + msum;
    } else {
      if (p.observe) {
        if (p.mass_pending) w += msum;
        const float abar = __fdiv_rn(w, p.norm);                    // Sec. III-C
        a = p.rho * a + p.gamma * abar;                             // Eq. 2
        const float tau = __fdiv_rn(p.tau_scale, (float)ntok);
        if (abar >= tau) tr = p.t;                                  // Eq. 3
        p.window[slot] = 0.f;
        p.ahat[slot] = abar;
        p.a[slot] = a;
        p.t_ref[slot] = tr;
        if (CALIB) {
          const int age = p.t - tins;
          const int bkt = age >= 0 ? age / CALIB_WIDTH : -1;
          if (bkt >= 0 && bkt < CALIB_BUCKETS) {
            bin = reg * CALIB_BUCKETS + bkt;
            fx = __float2ull_rn(abar * 4294967296.0f);
          }
        }
      }
      const float x = __fdiv_rn((float)(p.t - tr), p.reg.half_life[reg]);
      const float d = exp2f(-x);                                    // Eqs. 4, 7
      switch (p.score_mode) {
        case 0: s = p.reg.base[reg] * d + p.alpha * a; break;       // Eq. 4
        case 1: s = (p.reg.base[reg] + p.alpha * a) * d; break;
        case 2: s = p.reg.base[reg] * d + p.alpha * a * (float)ntok; break;
        case 3: s = (float)tins; break;                             // recency
        default: s = random_draw(p.random_seed, p.t, slot); break;   // random
      }
      pinned = p.reg.pinned[reg];
      if (pinned) s = INF;
      if (p.keep_prio) p.prio[slot] = s;
    }
  }
  if (p.fold_only) return 0.f;
  if (CALIB) {
    /* one pair of shared atomics for all tokens of a bin that holds a quarter
     * of the warp's (a prompt's page has one or two bins) instead of one pair
     * per token: the histogram's share of an observation of 16 x 30,000 tokens,
     * 30 -> 3 us; of 12 x 2,400, 12 -> 4 us.  Tokens spread over more bins (a
     * page of decode steps: four to a bin) conflict less and go one by one. */
    unsigned left = __ballot_sync(0xffffffffu, bin >= 0);
    while (left) {
      const int first = __ffs(left) - 1, cur = __shfl_sync(0xffffffffu, bin, first);
      const unsigned in = __ballot_sync(0xffffffffu, bin == cur);
      if (__popc(in) < 8) {
        if ((left >> (threadIdx.x & 31)) & 1) {
          atomicAdd(&calib->sum[bin], fx);
          atomicAdd(&calib->cnt[bin], 1u);
        }
        break;
      }
      const unsigned long long v = bin == cur ? fx : 0ull;
      const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0xFFFFFFu);
      const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 24) & 0xFFFFFFu);
      const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 48));
      if ((threadIdx.x & 31) == first) {
        atomicAdd(&calib->sum[cur], (unsigned long long)lo + ((unsigned long long)mid << 24) + ((unsigned long long)hi << 48));
        atomicAdd(&calib->cnt[cur], (unsigned)__popc(in));
      }
      left &= ~in;
    }
    __syncwarp();
  }
  float sum = (valid && !pinned) ? s : 0.f;
  float mx = (valid && !pinned) ? s : -INF;
  int anyp = (valid && pinned) ? 1 : 0;
  int cnt = valid ? 1 : 0;
#pragma unroll
  for (int o = PS / 2; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o, PS);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o, PS));
    anyp |= __shfl_xor_sync(0xffffffffu, anyp, o, PS);
    cnt += __shfl_xor_sync(0xffffffffu, cnt, o, PS);
  }
  float S = INF;                                                   // pinning, tail
  if (page_ok && !anyp && pg != p.n_pages[b] - 1)
    S = (p.page_reduce == 0) ? __fdiv_rn(sum, (float)cnt) : mx;   // Eq. 5
  if (page_ok && off == 0) p.page_score[(size_t)b * p.P_max + pg] = S;
  return S;
}

/* One warp per tile; the loop count is uniform across a warp, so the segmented
 * shuffle reductions see every lane.  The launcher sizes the grid to one wave
 * of resident blocks. */
template <int PS, bool CALIB>
__global__ void __launch_bounds__(256, 6) score_kernel(const __grid_constant__ ScoreParams p) {
  pdl_wait();
  pdl_trigger();
  constexpr int PPW = 32 / PS;
  __shared__ __align__(8) uint8_t hist_mem[CALIB ? sizeof(CalibSmem) : 8];
  CalibSmem *hist = (CalibSmem *)hist_mem;
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int tiles = (p.total_pages + PPW - 1) / PPW;
  const bool need_mass = p.fold_only || (p.observe && p.mass_pending);
  if (CALIB) {
    for (int k = threadIdx.x; k < 8 * CALIB_BUCKETS; k += blockDim.x) {
      hist->sum[k] = 0ull;
      hist->cnt[k] = 0u;
    }
    __syncthreads();
  }
  for (int t0 = blockIdx.x * 8; t0 < tiles; t0 += gridDim.x * 8) {
    const int gp = (t0 + wib) * PPW + lane / PS;
    const bool page_ok = gp < p.total_pages;
    const int b = page_ok ? find_seq(p.page_start, p.n_seqs, gp) : 0;
    score_tile<PS, CALIB>(p, b, page_ok ? gp - p.page_start[b] : 0, lane % PS, page_ok, need_mass, hist);
  }
  if (CALIB) {
    __syncthreads();
    for (int k = threadIdx.x; k < 8 * CALIB_BUCKETS; k += blockDim.x)
      if (hist->cnt[k]) {
        atomicAdd(&p.calib_sum[k], hist->sum[k]);
        atomicAdd(&p.calib_cnt[k], hist->cnt[k]);
      }
  }
}

/* Blocks of the score kernel that are resident at once on the current device
 * (SMs x blocks per SM from the occupancy of the instance).  The kernel gives
 * every block an equal share of the pages, so a grid larger than one wave
 * would leave the second wave's blocks as a tail. */
template <int PS, bool CALIB>
static int score_grid_cap() {
  static int cached[64];   // per device ordinal; a racy first fill writes the same value
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152 * 4;
  if (cached[dev] > 0) return cached[dev];
  int sms = 0, per_sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, score_kernel<PS, CALIB>, 256, 0) != cudaSuccess ||
      sms <= 0 || per_sm <= 0)
    return 152 * 4;
  cached[dev] = sms * per_sm;
  return cached[dev];
}

template <int PS, bool CALIB>
static cudaError_t launch_score_ps(const ScoreParams &p, cudaStream_t s) {
  const int ppb = 256 / PS;   // pages per block and iteration: one warp per tile
  const long long blocks = (p.total_pages + ppb - 1) / ppb, cap = score_grid_cap<PS, CALIB>();
  return launch_pdl(score_kernel<PS, CALIB>, (int)(blocks < cap ? blocks : cap), 256, 0, s, p);
}

cudaError_t launch_score(const ScoreParams &p, cudaStream_t s) {
  if (p.total_pages == 0) return cudaSuccess;
  if (p.calib_on && p.observe && !p.fold_only)
    return p.ps == 16 ? launch_score_ps<16, true>(p, s) : launch_score_ps<32, true>(p, s);
  return p.ps == 16 ? launch_score_ps<16, false>(p, s) : launch_score_ps<32, false>(p, s);
}

/* -------------------------------------------------------------- select --- */
constexpr int SEL_THREADS = 1024;
constexpr uint32_t KEY_PINNED = 0xFFFFFFFFu;

/* Order-preserving map of fp32 onto uint32 (larger float -> larger key). */
__device__ __forceinline__ uint32_t order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

/* Block-wide exclusive scan of one int per thread; returns the prefix and
 * writes the block total to *total. */
__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    int s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < nw) warp_sums[lane] = s;   // inclusive sums of warps
  }
  __syncthreads();
  const int before = (wid > 0 ? warp_sums[wid - 1] : 0) + x - v;
  *total = warp_sums[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

__global__ void __launch_bounds__(SEL_THREADS) select_kernel(const __grid_constant__ SelectParams p) {
  extern __shared__ uint32_t sm[];
  uint32_t *keys = sm;                               // [P_max]
  int32_t *phys = (int32_t *)(sm + p.P_max);         // [P_max]
  uint8_t *fills = (uint8_t *)(sm + 2 * (size_t)p.P_max);   // [P_max]
  __shared__ int hist[256];
  __shared__ int warp_sums[32];
  __shared__ uint32_t s_prefix;
  __shared__ int s_k, s_bad, s_gone, s_cnt;

  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x;
  const int P = p.n_pages[b];
  const int e = p.n_evict[b];
  int32_t *row = p.block_table + (size_t)b * p.P_max;
  int32_t *uout = p.user_evicted ? p.user_evicted + (size_t)b * p.P_max : nullptr;
  if (e == 0) {
    if (uout)
      for (int i = threadIdx.x; i < p.P_max; i += blockDim.x) uout[i] = -1;
    return;
  }
  const float *sc = p.page_score + (size_t)b * p.P_max;
  uint8_t *frow = p.page_fill + (size_t)b * p.P_max;
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    const float S = sc[i];
    keys[i] = (S == INFINITY) ? KEY_PINNED : order_key(S);
    phys[i] = row[i];
    fills[i] = frow[i];
  }
  if (threadIdx.x == 0) { s_prefix = 0u; s_k = e; s_bad = 0; s_gone = 0; s_cnt = 0; }
  __syncthreads();

  /* radix select of the e-th smallest evictable key, most significant digit
   * first.  It stops early once the digit's bucket holds exactly the keys
   * still to be taken: then every key below the bucket and every key in it
   * is evicted, the same set the remaining passes would pick. */
  uint32_t mask = 0u;
  bool whole_bucket = false;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    const uint32_t prefix = s_prefix;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
      const uint32_t k = keys[i];
      if (k != KEY_PINNED && (k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      /* the digit holding the k-th smallest remaining key: one warp, eight
       * bins per lane; the lane whose cumulative range (excl, incl] holds k
       * walks its bins (the same digit and residual a serial scan finds) */
      const int lane = threadIdx.x;
      const int k = s_k;
      int c[8], sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        c[j] = hist[lane * 8 + j];
        sum += c[j];
      }
      int incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int excl = incl - sum;
      const bool mine = excl < k && k <= incl;
      if (__ballot_sync(0xffffffffu, mine) == 0u) {
        if (lane == 0) s_bad = 1;         // fewer evictable pages than e
      } else if (mine) {
        int cum = excl, digit = lane * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (cum + c[j] >= k) { digit = lane * 8 + j; break; }
          cum += c[j];
        }
        s_prefix = prefix | ((uint32_t)digit << shift);
        s_k = k - cum;
        s_cnt = hist[digit];
      }
    }
    __syncthreads();
    if (s_bad) {
      if (threadIdx.x == 0) atomicCAS(&p.status[ST_CODE], 0, (int)MD_ERR_STATE);
      return;
    }
    mask |= 0xFFu << shift;
    if (pass < 3 && s_k == s_cnt) {   // the same value in every thread
      whole_bucket = true;
      break;
    }
  }
  /* key of the e-th smallest evictable page and how many pages with key == T
   * are evicted; for a whole bucket, T is the bucket's largest key and every
   * page equal to it goes */
  const uint32_t T = whole_bucket ? (s_prefix | ~mask) : s_prefix;
  const int take_eq = whole_bucket ? P : s_k;

  /* evict: key < T, or key == T among the first take_eq in logical order;
   * compact kept pages in order; list the evicted ones in logical order */
  int carry_eq = 0, carry_ev = 0, gone = 0;
  const int base_push = p.top + p.push_off[b];
  for (int t0 = 0; t0 < P; t0 += blockDim.x) {
    const int i = t0 + threadIdx.x;
    const bool in = i < P;
    const uint32_t k = in ? keys[i] : KEY_PINNED;
    const int eq = (in && k == T) ? 1 : 0;
    int tot_eq;
    const int rank_eq = carry_eq + block_exclusive_scan(eq, warp_sums, &tot_eq);
    const int ev = (in && k != KEY_PINNED && (k < T || (eq && rank_eq < take_eq))) ? 1 : 0;
    int tot_ev;
    const int idx_ev = carry_ev + block_exclusive_scan(ev, warp_sums, &tot_ev);
    if (in) {
      const int id = phys[i];
      if (ev) {
        p.free_stack[base_push + idx_ev] = id;
        if (uout) uout[idx_ev] = id;
        gone += fills[i];
      } else {
        row[i - idx_ev] = id;
        frow[i - idx_ev] = fills[i];
      }
    }
    carry_eq += tot_eq;
    carry_ev += tot_ev;
  }
  if (gone) atomicAdd(&s_gone, gone);
  __syncthreads();
  if (threadIdx.x == 0) p.seq_tokens[b] -= s_gone;
  for (int i = P - e + threadIdx.x; i < P; i += blockDim.x) {
    row[i] = -1;
    frow[i] = 0;
  }
  if (uout)
    for (int i = e + threadIdx.x; i < p.P_max; i += blockDim.x) uout[i] = -1;
}

/* Stages 2-4 in one launch for short sequences (at most OBSERVE_PAGES pages):
 * one block scores its sequence's pages and then selects among them in shared
 * memory.  What bounds a short observation is the chain of dependent launches
 * and round trips, not the bytes: a decode step of 32 sequences of 430 tokens
 * and its observation took 102.3 us with the two kernels and their hand-over
 * through the page-score array, 97.9 with this one.  With so few keys a page's rank is counted directly (one thread per
 * page reads every key, a broadcast), instead of up to four radix passes of
 * three barriers each; ties go to the lower logical index as there. */
template <int PS>
__global__ void __launch_bounds__(1024) observe_kernel(const __grid_constant__ ObserveParams p) {
  __shared__ __align__(16) uint32_t keys[OBSERVE_PAGES];
  __shared__ int warp_ev[OBSERVE_PAGES / 32];
  __shared__ int s_gone;
  pdl_wait();
  pdl_trigger();
  constexpr int PPW = 32 / PS;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int P = p.s.n_pages[b], e = p.n_evict[b];
  int32_t *row = p.block_table + (size_t)b * p.s.P_max;
  uint8_t *frow = p.page_fill + (size_t)b * p.s.P_max;
  int32_t *uout = p.user_evicted ? p.user_evicted + (size_t)b * p.s.P_max : nullptr;
  /* thread i < P: page i's id and fill, before anything is compacted */
  const int id = tid < P ? row[tid] : 0, fill = tid < P ? frow[tid] : 0;
  if (tid == 0) s_gone = 0;
  if (tid < OBSERVE_PAGES && tid >= P) keys[tid] = KEY_PINNED;
  for (int pg0 = warp * PPW; pg0 < P; pg0 += (int)(blockDim.x >> 5) * PPW) {
    const int pg = pg0 + lane / PS;
    const float S = score_tile<PS, false>(p.s, b, pg < P ? pg : 0, lane % PS, pg < P, p.s.observe && p.s.mass_pending, nullptr);
    if (pg < P && lane % PS == 0) keys[pg] = S == INFINITY ? KEY_PINNED : order_key(S);
  }
  __syncthreads();
  if (e > 0) {
    /* page tid's rank among the evictable pages: keys below its own, and
     * equal ones at lower indices */
    const int P4 = (P + 3) / 4;
    int ev = 0;
    if (tid < P) {
      const uint32_t k = keys[tid];
      int rank = 0;
      for (int j = 0; j < P4; ++j) {
        const uint4 q = ((const uint4 *)keys)[j];
        const int i = 4 * j;
        rank += (q.x < k || (q.x == k && i < tid)) + (q.y < k || (q.y == k && i + 1 < tid)) +
                (q.z < k || (q.z == k && i + 2 < tid)) + (q.w < k || (q.w == k && i + 3 < tid));
      }
      ev = k != KEY_PINNED && rank < e;
    }
    const unsigned m = __ballot_sync(0xffffffffu, ev);
    if (lane == 0 && warp < OBSERVE_PAGES / 32) warp_ev[warp] = __popc(m);
    __syncthreads();
    int idx = __popc(m & ((1u << lane) - 1)), total = 0;
    for (int w = 0; w < (P + 31) / 32; ++w) {
      idx += w < warp ? warp_ev[w] : 0;
      total += warp_ev[w];
    }
    if (total != e) {   // fewer evictable pages than e: nothing is changed
      if (tid == 0) atomicCAS(&p.status[ST_CODE], 0, (int)MD_ERR_STATE);
      return;
    }
    if (tid < P) {
      if (ev) {
        p.free_stack[p.top + p.push_off[b] + idx] = id;
        if (uout) uout[idx] = id;
        atomicAdd(&s_gone, fill);
      } else {
        row[tid - idx] = id;
        frow[tid - idx] = (uint8_t)fill;
      }
    }
    __syncthreads();
    if (tid == 0) p.seq_tokens[b] -= s_gone;
    if (tid < P && tid >= P - e) {
      row[tid] = -1;
      frow[tid] = 0;
    }
  }
  if (uout)
    for (int i = e + tid; i < p.s.P_max; i += blockDim.x) uout[i] = -1;
}

cudaError_t launch_observe(const ObserveParams &p, cudaStream_t s) {
  int pmax = 1;
  for (int b = 0; b < p.s.n_seqs; ++b) pmax = p.s.n_pages[b] > pmax ? p.s.n_pages[b] : pmax;
  int threads = (pmax * p.s.ps + 31) / 32 * 32;   // one token slot per thread, up to a full block
  threads = threads > 1024 ? 1024 : threads;
  return p.s.ps == 16 ? launch_pdl(observe_kernel<16>, p.s.n_seqs, threads, 0, s, p)
                      : launch_pdl(observe_kernel<32>, p.s.n_seqs, threads, 0, s, p);
}

cudaError_t launch_select(const SelectParams &p, cudaStream_t s) {
  if (p.n_seqs == 0) return cudaSuccess;
  /* one thread per page of the longest sequence (whole warps, at least 128,
   * at most SEL_THREADS): fewer warps make the passes' barriers cheaper */
  int pmax = 0;
  for (int b = 0; b < p.n_seqs; ++b) pmax = p.n_pages[b] > pmax ? p.n_pages[b] : pmax;
  int threads = (pmax + 31) / 32 * 32;
  threads = threads < 128 ? 128 : (threads > SEL_THREADS ? SEL_THREADS : threads);
  const size_t smem = (size_t)p.P_max * 9;
  /* raise the kernel's dynamic shared-memory limit only when a larger table
   * needs it (a host call per launch costs more than the kernel at small
   * sizes); per device ordinal, a racy first fill sets the same value */
  static int granted[64];
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= 64 || granted[dev] < (int)smem) {
    err = cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    if (dev >= 0 && dev < 64) granted[dev] = (int)smem;
  }
  return launch_pdl(select_kernel, p.n_seqs, threads, (int)smem, s, p);
}

}  // namespace md
