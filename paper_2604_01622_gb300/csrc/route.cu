// Expert-choice top-k selection (arXiv 2604.01622, Sec. 2.2).
//
// Selection: for every expert e and group g (one sequence, Sec. 5.2) keep the k_g tokens
// with the largest S[t,e] (Sec. 2.2 TopC; capacity per group, Sec. 4.2). Ties go to the
// lower token index and the kept tokens are written in ascending index. One CTA (or cluster)
// per (e, g) runs an MSB-first radix select over order-preserving 32-bit keys of the fp32
// scores to find the k-th largest key, then compacts the column in index order with one
// scan, which makes the result unique and independent of thread timing.
#include "common.cuh"
#include "kernels.h"

namespace ecmoe {

// ------------------------------------------------------------------ top-k selection
// Order-preserving key: larger float -> larger unsigned key; -0.0 is folded onto +0.0.
__device__ __forceinline__ uint32_t score_key(float s) {
  const uint32_t u = __float_as_uint(s + 0.0f);
  return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}

// The k-th largest key is found by an MSB-first radix select over the offsets u = key - kmin
// of the column (kmin, kmax its smallest and largest key), 8 bits per pass starting at the top
// bit of kmax - kmin. Scores of one expert over a sequence span a narrow range, so digits of
// the raw key would put most of the column into a few bins of the first pass (and serialise
// its shared-memory atomics); digits of the offset spread it over the whole histogram. The
// select stops early once the bin that holds the k-th key is taken whole. The selected set
// is the one the (score desc, index asc) order defines, whatever the digit boundaries.

// One histogram bin search by a whole warp: lane l owns bins 8l .. 8l+7 (counts c), bins are
// taken from the top. Finds the bin of the `remaining`-th largest offset; returns it with the
// keys taken above it (`above`) and the keys in it (`inside`), the same in every lane; -1 if
// the histogram holds fewer keys or `remaining` is below 1.
__device__ __forceinline__ int find_bin(const int (&c)[8], int remaining, int& above,
                                        int& inside) {
  const int lane = threadIdx.x & 31;
  int local = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) local += c[j];
  int incl = local;   // bins of lanes >= this one
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += u;
  }
  int run = incl - local, bin = 0, ab = 0, in = 0;
  const bool mine = run < remaining && remaining <= incl;
#pragma unroll
  for (int j = 7; j >= 0; --j) {
    if (run < remaining && remaining <= run + c[j]) { bin = lane * 8 + j; ab = run; in = c[j]; }
    run += c[j];
  }
  const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
  if (src < 0) return -1;
  above = __shfl_sync(0xffffffffu, ab, src);
  inside = __shfl_sync(0xffffffffu, in, src);
  return __shfl_sync(0xffffffffu, bin, src);
}

// Ranks the at most kCand keys that share the k-th key's prefix against each other: thread i
// takes cand[i] and counts the larger and the equal ones; the one that is the `remaining`-th
// largest leaves itself and the number of its equals that are taken.
constexpr int kCand = 64;
__device__ __forceinline__ void rank_candidates(const uint32_t* cand, int n, int remaining,
                                                uint32_t* T, int* need, int* all = nullptr) {
  if ((int)threadIdx.x >= n) return;
  const uint32_t mine = cand[threadIdx.x];
  int gt = 0, eq = 0;
#pragma unroll 8
  for (int i = 0; i < n; ++i) {
    const uint32_t o = cand[i];
    gt += o > mine;
    eq += o == mine;
  }
  if (gt < remaining && remaining <= gt + eq) {   // the same for equal keys
    *T = mine;
    *need = remaining - gt;
    if (all) *all = remaining - gt == eq;   // whether that is all of them
  }
}

// One column (expert, group) per CTA, its keys in registers: thread i owns KPT consecutive
// scores on the 16-byte grid of the column (thread 0 starts up to 3 scores early), so every
// load is one 16-byte vector but at the column's ends. A pass is an unrolled loop over registers
// and two barriers (two histogram buffers take turns; warp 0 searches the bins). Once the bin of
// the k-th key holds at most kCand keys they are ranked against each other instead of by more
// passes.
//
// Outputs: per thread a bit mask of its selected keys, whose set bits go to a list in shared
// memory (about 2 of 16 in a top-8-of-64 selection; the loop's length is the largest count in
// the warp, not KPT); the CTA then writes the list with neighbouring threads on neighbouring
// entries, re-reading each score as the gate.
//
// What bounds it: the chain of block-wide steps, not memory: half of a 4096-score column's
// cycles are its first histogram pass, whose shared atomics cost about 14 cycles a warp. A lone
// launch on narrow scores (8 x 4096 scores, 64 experts, 512 selected): 14.5 -> 12.5 us against
// stores predicated per key; 16 x 2048, 128 experts: 18.5 -> 14.8; 8192-score columns 10.3 ->
// 8.4; 256-score columns 6.2 -> 4.2 (4 scores per thread). A bracket from a sample of the keys,
// which lets 15% of them into the histogram, cost as much as it saved here, and searching the
// bins in every warp instead of one cost 0.6 k cycles a pass.
constexpr uint32_t kNoKey = 0xFFFFFFFFu;   // offset of a register that holds no score

template <int KPT, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) topk_reg_kernel(TopkArgs p) {
  constexpr int nw = NT / 32;
  __shared__ __align__(16) int hist[2][256];
  __shared__ uint32_t s_mn[nw], s_mx[nw], s_cnt[nw], s_cand[kCand];
  __shared__ uint16_t s_list[KPT * NT];   // selected scores by place in the column
  __shared__ int s_ncand, s_bin[3], s_need;
  __shared__ uint32_t s_T;
  const int e = blockIdx.x, g = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_begin(p.ST, p.group_off, p.k_g, p.k_off);
  const int lo = p.group_off[g];
  const int L = p.group_off[g + 1] - lo;
  const int k = p.k_g[g];
  const int base = p.k_off[g];
  const float* col = p.ST + (size_t)e * p.N + lo;
  // this thread's scores: i0 + j for j in [j0, j1)
  const int i0 = tid * KPT - (int)((reinterpret_cast<uintptr_t>(col) >> 2) & 3u);
  const int j0 = max(0, -i0), j1 = min(KPT, L - i0);
  const bool full = j0 == 0 && j1 == KPT;
  uint32_t key[KPT];
  uint32_t mn = 0xFFFFFFFFu, mx = 0u;
  if (full) {
    const float4* src = reinterpret_cast<const float4*>(col + i0);
    float4 q[KPT / 4];
#pragma unroll
    for (int j = 0; j < KPT / 4; ++j) q[j] = __ldg(src + j);
    if (p.S_copy) {
      float* dst = p.S_copy + (size_t)e * p.N + lo + i0;
      if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
#pragma unroll
        for (int j = 0; j < KPT / 4; ++j) reinterpret_cast<float4*>(dst)[j] = q[j];
      } else {
#pragma unroll
        for (int j = 0; j < KPT / 4; ++j) {
          dst[4 * j] = q[j].x; dst[4 * j + 1] = q[j].y;
          dst[4 * j + 2] = q[j].z; dst[4 * j + 3] = q[j].w;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < KPT / 4; ++j) {
      key[4 * j] = score_key(q[j].x); key[4 * j + 1] = score_key(q[j].y);
      key[4 * j + 2] = score_key(q[j].z); key[4 * j + 3] = score_key(q[j].w);
    }
#pragma unroll
    for (int j = 0; j < KPT; ++j) { mn = min(mn, key[j]); mx = max(mx, key[j]); }
  } else {
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      key[j] = 0u;
      if (j >= j0 && j < j1) {
        const float v = __ldg(col + i0 + j);
        if (p.S_copy) p.S_copy[(size_t)e * p.N + lo + i0 + j] = v;
        key[j] = score_key(v);
        mn = min(mn, key[j]);
        mx = max(mx, key[j]);
      }
    }
  }
  if (k == 0) return;
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) { s_mn[warp] = mn; s_mx[warp] = mx; }
  for (int i = tid; i < 256; i += NT) hist[0][i] = 0;
  if (tid == 0) s_ncand = 0;
  __syncthreads();
  mn = __reduce_min_sync(0xffffffffu, lane < nw ? s_mn[lane] : 0xFFFFFFFFu);
  mx = __reduce_max_sync(0xffffffffu, lane < nw ? s_mx[lane] : 0u);
  // keys become offsets from the column's smallest key
  const uint32_t valid = j1 <= j0 ? 0u : (((1u << j1) - 1u) & ~((1u << j0) - 1u));
#pragma unroll
  for (int j = 0; j < KPT; ++j) key[j] = (full || (valid >> j & 1u)) ? key[j] - mn : kNoKey;

  // threshold T (an offset) and how many keys equal to it are taken (in token order)
  int hi = mx == mn ? 0 : 32 - __clz(mx - mn);   // every offset lies in [0, 2^hi)
  uint32_t prefix = 0u, mask = hi == 32 ? 0u : ~((1u << hi) - 1u);
  int remaining = k;
  bool done = hi == 0;                           // all keys equal: the first k are taken
  const bool wide = hi == 32;                    // no bit above the offsets marks kNoKey
  int b = 0;                                     // histogram buffer of this pass
  int inside = kCand + 1;                        // keys that share the prefix (first pass: many)
  while (!done && hi > 0) {
    if (inside <= kCand) {
#pragma unroll
      for (int j = 0; j < KPT; ++j)
        if (((key[j] ^ prefix) & mask) == 0u && (valid >> j & 1u))
          s_cand[atomicAdd(&s_ncand, 1)] = key[j];
      __syncthreads();
      rank_candidates(s_cand, inside, remaining, &s_T, &s_need);
      __syncthreads();
      prefix = s_T;
      remaining = s_need;
      hi = 0;
      break;
    }
    const int shift = max(hi - 8, 0);
    const uint32_t dmask = (1u << (hi - shift)) - 1u;
    // the other buffer was last read before the previous pass's second barrier
    for (int i = tid; i < 256; i += NT) hist[b ^ 1][i] = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (((key[j] ^ prefix) & mask) == 0u && (!wide || (valid >> j & 1u)))
        atomicAdd(&hist[b][(key[j] >> shift) & dmask], 1);
    __syncthreads();
    if (warp == 0) {
      const int4 x = *reinterpret_cast<const int4*>(&hist[b][lane * 8]);
      const int4 y = *reinterpret_cast<const int4*>(&hist[b][lane * 8 + 4]);
      const int c[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
      int above, in;
      const int bin = find_bin(c, remaining, above, in);
      if (lane == 0) { s_bin[0] = bin; s_bin[1] = above; s_bin[2] = in; }
    }
    __syncthreads();
    prefix |= (uint32_t)s_bin[0] << shift;
    remaining -= s_bin[1];
    inside = s_bin[2];
    done = inside == remaining;   // the whole bin is taken
    mask |= dmask << shift;
    hi = shift;
    b ^= 1;
  }
  const uint32_t T = prefix;
  // a bin taken whole: every offset >= T is selected
  const int need_eq = (done && hi > 0) ? 0x7FFFFFFF : remaining;
  // compaction in token order: this thread's keys follow those of lower threads
  uint32_t gt = 0u, eq = 0u;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    gt |= (uint32_t)(key[j] > T) << j;
    eq |= (uint32_t)(key[j] == T) << j;
  }
  gt &= valid;
  eq &= valid;
  const uint32_t cnt = (uint32_t)__popc(gt) << 16 | (uint32_t)__popc(eq);   // <= 512 each a warp
  uint32_t incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_cnt[warp] = incl;
  __syncthreads();
  const uint32_t lower = lane < warp ? s_cnt[lane] : 0u;   // keys of lower warps, then threads
  const int gt0 = (int)(__reduce_add_sync(0xffffffffu, lower >> 16) + ((incl - cnt) >> 16));
  const int eq0 = (int)(__reduce_add_sync(0xffffffffu, lower & 0xFFFFu) + ((incl - cnt) & 0xFFFFu));
  int pos = gt0 + min(eq0, need_eq);   // selected keys before this thread's
  const int take = need_eq - eq0;      // of its keys equal to T, the first `take` (<= 0: none)
  while (__popc(eq) > max(take, 0)) eq &= ~(0x80000000u >> __clz(eq));
  uint32_t sel = gt | eq;
  while (sel) {
    const int j = __ffs(sel) - 1;
    sel &= sel - 1u;
    s_list[pos++] = (uint16_t)(i0 + j);
  }
  __syncthreads();
  const size_t row = (size_t)e * p.M + base;
  for (int i = tid; i < k; i += NT) {
    const int c = s_list[i], t = lo + c;
    const float sv = __ldg(col + c);
    p.idx[row + i] = t;
    p.gate[row + i] = sv;
    if (p.idx2) p.idx2[row + i] = t;
    if (p.gate2) p.gate2[row + i] = sv;
    if (p.slot) p.slot[(size_t)t * p.E + e] = base + i;
  }
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of a shared variable of this CTA in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_shared(const void* p, int rank) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int4 ld_peer4(uint32_t addr) {
  int4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// Columns of 8193 to 49152 scores: one CTA of NT threads with the column's keys in shared memory
// (`chunk` of them, a multiple of kStep NT / 32). Warp w owns the keys [w wlen, (w+1) wlen), each
// lane 16 consecutive ones of every kStep (16-byte units swizzled so that these reads and the
// coalesced fills are free of bank conflicts).
//
// The k-th key is bracketed first: one key in 16 goes into a histogram, the sample's rank of the
// k-th key plus and minus four standard deviations gives two bins, and only the keys between
// them (6-10%) are listed, those above being counted by comparison; the radix passes then read
// the list. If the k-th key is outside, or the list overflows (many equal scores), the passes
// read all keys. Selected keys are found once, as a bit mask per lane, and compacted in order in
// place: the list of a warp's selected keys is never longer than the keys it has read.
//
// What bounds it: instructions of the block-wide steps (listing the bracket 6 k of a column's 25 k
// cycles, the selection masks 3 k, the load 4-7 k). The shared atomics of a full pass cost about
// 21 cycles a warp, a third of the time before the bracket, and a cluster of four CTAs per
// column paid 2.7 k cycles of barrier and search per pass: 256 columns of 32768 scores, 37 -> 29
// us (with the slot map instead of the copy of the scores 39 -> 33); 128 of 16384, 16.5 -> 12.4.
constexpr int kStep = 512;    // keys a warp handles at a time
constexpr int kList = 4096;   // keys of the bracket

template <int NT>
__global__ void __launch_bounds__(NT, NT <= 512 ? 2 : 1) topk_block_kernel(TopkArgs p, int chunk) {
  constexpr int nw = NT / 32, MAXS = 3;   // steps per warp: chunk <= MAXS kStep nw
  extern __shared__ uint4 skeys4[];
  uint32_t* skeys = reinterpret_cast<uint32_t*>(skeys4);
  uint32_t* s_list = skeys + chunk;
  __shared__ __align__(16) int hist[2][256];
  __shared__ uint32_t s_mn[nw], s_mx[nw], s_cand[kCand], s_T;
  __shared__ int s_gt[nw], s_eq[nw], s_bin[4], s_n, s_above, s_ncand, s_need, s_whole;
  const int e = blockIdx.x, g = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_begin(p.ST, p.group_off, p.k_g, p.k_off);
  const int lo = p.group_off[g];
  const int L = p.group_off[g + 1] - lo;
  const int k = p.k_g[g];
  const int base = p.k_off[g];
  const float* col = p.ST + (size_t)e * p.N + lo;
  // place i is score c0 + i of the column, for i in [v0, v1)
  const int v0 = (int)((reinterpret_cast<uintptr_t>(col) >> 2) & 3u), c0 = -v0, v1 = v0 + L;
  const int wlen = chunk / nw, w0 = warp * wlen;
  float* copy = p.S_copy ? p.S_copy + (size_t)e * p.N + lo + c0 : nullptr;
  const bool cvec = (reinterpret_cast<uintptr_t>(copy) & 15u) == 0;
  auto unit = [](int v) { return v ^ ((v >> 3) & 3); };   // where 16-byte unit v is kept
  uint32_t mn = 0xFFFFFFFFu, mx = 0u;
  for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
    const int i = i0 + lane * 4;
    if (i0 >= v0 && i0 + kStep <= v1) {
      float4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        x[u] = __ldg(reinterpret_cast<const float4*>(col + c0 + i + u * 128));
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (copy) {
          float* dst = copy + i + u * 128;
          if (cvec) {
            *reinterpret_cast<float4*>(dst) = x[u];
          } else {
            dst[0] = x[u].x; dst[1] = x[u].y; dst[2] = x[u].z; dst[3] = x[u].w;
          }
        }
        const uint4 q = make_uint4(score_key(x[u].x), score_key(x[u].y), score_key(x[u].z),
                                   score_key(x[u].w));
        mn = min(min(min(mn, q.x), min(q.y, q.z)), q.w);
        mx = max(max(max(mx, q.x), max(q.y, q.z)), q.w);
        skeys4[unit((i + u * 128) >> 2)] = q;
      }
    } else {
      for (int u = 0; u < 4; ++u)
        for (int j = i + u * 128; j < i + u * 128 + 4; ++j) {
          uint32_t q = 0u;
          if (j >= v0 && j < v1) {
            const float v = __ldg(col + c0 + j);
            if (copy) copy[j] = v;
            q = score_key(v);
            mn = min(mn, q);
            mx = max(mx, q);
          }
          skeys[unit(j >> 2) * 4 + (j & 3)] = q;
        }
    }
  }
  if (k == 0) return;
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) { s_mn[warp] = mn; s_mx[warp] = mx; }
  for (int i = tid; i < 512; i += NT) (&hist[0][0])[i] = 0;
  if (tid == 0) s_n = s_above = s_ncand = 0;
  __syncthreads();
  mn = __reduce_min_sync(0xffffffffu, lane < nw ? s_mn[lane] : 0xFFFFFFFFu);
  mx = __reduce_max_sync(0xffffffffu, lane < nw ? s_mx[lane] : 0u);

  // the 16 keys of this lane from place i0 + 16 lane on, and which of them exist
  auto load16 = [&](int i0, uint32_t (&q)[16]) -> uint32_t {
    const int i = i0 + lane * 16;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint4 x = skeys4[unit((i >> 2) + u)];
      q[4 * u] = x.x; q[4 * u + 1] = x.y; q[4 * u + 2] = x.z; q[4 * u + 3] = x.w;
    }
    if (i0 >= v0 && i0 + kStep <= v1) return 0xFFFFu;
    const int a = min(max(v0 - i, 0), 16), z = min(max(v1 - i, 0), 16);
    return a < z ? ((1u << z) - 1u) & ~((1u << a) - 1u) : 0u;
  };
  auto each = [&](auto f) {
    for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
      uint32_t q[16];
      const uint32_t ok = load16(i0, q);
      if (ok == 0xFFFFu) {
#pragma unroll
        for (int j = 0; j < 16; ++j) f(q[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (ok >> j & 1u) f(q[j]);
      }
    }
  };
  auto excl = [&](int v, int& total) {   // exclusive scan over the warp
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - v;
  };
  // bin of the rem-th largest key in histogram h, by one warp: out[0..2] = bin, keys above, in it
  auto search = [&](const int* h, int rem, int* out, int n_out) {
    const int4 x = *reinterpret_cast<const int4*>(h + lane * 8);
    const int4 y = *reinterpret_cast<const int4*>(h + lane * 8 + 4);
    const int c[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    int above = 0, in = 0;
    const int bin = find_bin(c, rem, above, in);
    if (lane == 0) {
      out[0] = bin;
      if (n_out > 1) { out[1] = above; out[2] = in; }
    }
  };

  int hi = mx == mn ? 0 : 32 - __clz(mx - mn);   // every offset key - org lies in [0, 2^hi)
  uint32_t org = mn;
  int remaining = k, b = 0, inside = L;
  int listed = -1;                               // keys in the list, once they are bracketed
  const int n_s = (v1 + 15) / 16 - (v0 + 15) / 16;
  if (hi > 0 && n_s >= 64) {
    const int shift = max(hi - 8, 0);
    const uint32_t dmask = (1u << (hi - shift)) - 1u;
    for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
      const int i = i0 + lane * 16;
      if (i >= v0 && i < v1) atomicAdd(&hist[0][(skeys[unit(i >> 2) * 4] - mn) >> shift], 1);
    }
    __syncthreads();
    const float c = (float)k * n_s / L, m = 4.0f * sqrtf(c * (n_s - c) / n_s) + 2.0f;
    if (warp == 0 && c - m >= 1.0f) search(hist[0], (int)(c - m), s_bin, 1);
    if (warp == 1 && c + m < n_s) search(hist[0], (int)ceilf(c + m), s_bin + 3, 1);
    __syncthreads();
    const uint32_t bhi = c - m >= 1.0f ? (uint32_t)s_bin[0] : dmask;
    const uint32_t blo = c + m < n_s ? (uint32_t)s_bin[3] : 0u;
    const uint32_t khi = (bhi << shift) + ((1u << shift) - 1u), klo = blo << shift;
    int above = 0;
    for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
      uint32_t q[16], in = 0u;
      const uint32_t ok = load16(i0, q);
      const uint32_t lowest = mn + klo, width = khi - klo, highest = mn + khi;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        above += q[j] > highest;   // (a place without a score holds key 0)
        if (q[j] - lowest <= width) in |= 1u << j;
      }
      in &= ok;
      int total;
      int at = excl(__popc(in), total);
      int first = 0;
      if (lane == 0 && total) first = atomicAdd(&s_n, total);
      at += __shfl_sync(0xffffffffu, first, 0);
      // dynamic indexing would put q into local memory: the keys are read again
      while (in) {
        const int j = __ffs(in) - 1;
        in &= in - 1u;
        const int i = i0 + lane * 16 + j;
        if (at < kList) s_list[at] = skeys[unit(i >> 2) * 4 + (i & 3)];
        ++at;
      }
    }
    above = __reduce_add_sync(0xffffffffu, above);
    if (lane == 0) atomicAdd(&s_above, above);
    if (tid < 256) hist[0][tid] = 0;
    __syncthreads();
    const int n = s_n, rem = k - s_above;
    if (n <= kList && rem >= 1 && rem <= n) {
      listed = inside = n;
      remaining = rem;
      org = mn + klo;
      hi = khi == klo ? 0 : 32 - __clz(khi - klo);
    }
  }
  uint32_t prefix = 0u, mask = hi == 32 ? 0u : ~((1u << hi) - 1u);
  bool whole = false;   // every key that shares the prefix is selected
  while (!whole && hi > 0) {
    auto keys = [&](auto f) {
      if (listed >= 0)
        for (int i = tid; i < listed; i += NT) f(s_list[i]);
      else
        each(f);
    };
    if (inside <= kCand) {
      keys([&](uint32_t key) {
        const uint32_t u = key - org;
        if (((u ^ prefix) & mask) == 0u) s_cand[atomicAdd(&s_ncand, 1)] = u;
      });
      __syncthreads();
      rank_candidates(s_cand, inside, remaining, &s_T, &s_need, &s_whole);
      __syncthreads();
      prefix = s_T;
      remaining = s_need;
      whole = s_whole;
      break;
    }
    const int shift = max(hi - 8, 0);
    const uint32_t dmask = (1u << (hi - shift)) - 1u;
    // the other buffer was last read before the previous pass's second barrier
    if (tid < 256) hist[b ^ 1][tid] = 0;
    int* h = hist[b];
    keys([&](uint32_t key) {
      const uint32_t u = key - org;
      if (((u ^ prefix) & mask) == 0u) atomicAdd(&h[(u >> shift) & dmask], 1);
    });
    __syncthreads();
    if (warp == 0) search(h, remaining, s_bin, 3);
    __syncthreads();
    prefix |= (uint32_t)s_bin[0] << shift;
    remaining -= s_bin[1];
    inside = s_bin[2];
    whole = inside == remaining;
    mask |= dmask << shift;
    hi = shift;
    b ^= 1;
  }
  // every key >= T is selected if all that share the prefix are, else those above T and the first
  // `remaining` equal to it
  const uint32_t T = prefix + org;
  const int need_eq = remaining;
  uint32_t sel[MAXS];   // per step: keys above T in the low half, equal to T in the high half
  int gt = 0, eq = 0;
#pragma unroll
  for (int t = 0; t < MAXS; ++t) {
    sel[t] = 0u;
    if (t * kStep < wlen) {
      uint32_t q[16];
      const uint32_t ok = load16(w0 + t * kStep, q);
      if (whole) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (q[j] >= T) sel[t] |= 1u << j;
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (q[j] > T) sel[t] |= 1u << j;
          if (q[j] == T) sel[t] |= 0x10000u << j;
        }
      }
      sel[t] &= ok | ok << 16;
      gt += __popc(sel[t] & 0xFFFFu);
      eq += __popc(sel[t] >> 16);
    }
  }
  gt = __reduce_add_sync(0xffffffffu, gt);
  eq = __reduce_add_sync(0xffffffffu, eq);
  if (lane == 0) { s_gt[warp] = gt; s_eq[warp] = eq; }
  __syncthreads();
  const int gt0 = __reduce_add_sync(0xffffffffu, lane < warp ? s_gt[lane] : 0);   // lower warps'
  int eq0 = __reduce_add_sync(0xffffffffu, lane < warp ? s_eq[lane] : 0);
  const int first = gt0 + min(eq0, need_eq);   // selected keys before this warp's
  int n = 0;                                   // selected keys of this warp so far
#pragma unroll
  for (int t = 0; t < MAXS; ++t) {
    if (t * kStep >= wlen) break;
    uint32_t seq = sel[t] >> 16;
    if (__any_sync(0xffffffffu, seq)) {
      int all;
      const int before = eq0 + excl(__popc(seq), all);
      eq0 += all;
      while (__popc(seq) > max(need_eq - before, 0)) seq &= ~(0x80000000u >> __clz(seq));
    }
    uint32_t m = (sel[t] & 0xFFFFu) | seq;
    int all;
    int at = w0 + n + excl(__popc(m), all);
    n += all;
    while (m) {   // the masks hold all that is still needed of the keys
      const int j = __ffs(m) - 1;
      m &= m - 1u;
      skeys[at++] = (uint32_t)(w0 + t * kStep + lane * 16 + j);
    }
  }
  __syncwarp();
  const size_t row = (size_t)e * p.M + base + first;
#pragma unroll 4
  for (int i = lane; i < n; i += 32) {
    const int c = c0 + (int)skeys[w0 + i], t = lo + c;
    const float sv = __ldg(col + c);
    p.idx[row + i] = t;
    p.gate[row + i] = sv;
    if (p.idx2) p.idx2[row + i] = t;
    if (p.gate2) p.gate2[row + i] = sv;
    if (p.slot) p.slot[(size_t)t * p.E + e] = base + first + i;
  }
}

// Columns above 49152 scores: one per cluster of CL CTAs of 256 threads, each with `chunk` keys
// (a multiple of 8 kStep) in its shared memory, so that several CTAs per SM cover one another's
// loads and barriers. The CTAs add up their histograms through distributed shared memory, one
// cluster barrier per pass; once at most kTail keys share the k-th key's prefix, each CTA lists
// its own of them and the later passes read the lists. Warp w owns the keys
// [w chunk/8, (w+1) chunk/8), each lane 16 consecutive ones of every kStep (16-byte units
// swizzled so that these reads and the coalesced fills are free of bank conflicts), and compacts
// them in order in place: the list of its selected keys is never longer than the keys it has
// read.
//
// What bounds it: the first pass's shared atomics (about 21 cycles a warp) and the cluster
// barriers (1-1.4 k cycles each with the search behind them); 64 columns of 131072 scores take
// 52 us.
constexpr int kTail = 512;
constexpr int kClusterKeys = 49152;   // 192 KB of keys per CTA

template <int CL>
__global__ void __launch_bounds__(256, 4) topk_cluster_kernel(TopkArgs p, int chunk) {
  constexpr int nw = 8, TW = nw * CL;
  extern __shared__ uint4 skeys4[];
  uint32_t* skeys = reinterpret_cast<uint32_t*>(skeys4);
  __shared__ __align__(16) int hist[3][256];
  __shared__ uint32_t s_mn[TW], s_mx[TW], s_keys[kTail];
  __shared__ int s_gt[TW], s_eq[TW], s_bin[3], s_n;
  const int rank = (int)cluster_rank();
  const int e = blockIdx.x / CL, g = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_begin(p.ST, p.group_off, p.k_g, p.k_off);
  const int lo = p.group_off[g];
  const int L = p.group_off[g + 1] - lo;
  const int k = p.k_g[g];
  const int base = p.k_off[g];
  const float* col = p.ST + (size_t)e * p.N + lo;
  cluster_arrive();   // every CTA has started before its shared memory is written
  // place i of this CTA is score c0 + i of the column, for i in [v0, v1)
  const int c0 = rank * chunk - (int)((reinterpret_cast<uintptr_t>(col) >> 2) & 3u);
  const int v0 = max(0, -c0), v1 = max(v0, min(chunk, L - c0));
  const int wlen = chunk / nw, w0 = warp * wlen;   // this warp's places [w0, w0 + wlen)
  auto unit = [](int v) { return v ^ ((v >> 3) & 3); };   // where 16-byte unit v is kept
  uint32_t mn = 0xFFFFFFFFu, mx = 0u;
  for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
    const int i = i0 + lane * 4;
    if (i0 >= v0 && i0 + kStep <= v1) {
      float4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        x[u] = __ldg(reinterpret_cast<const float4*>(col + c0 + i + u * 128));
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint4 q = make_uint4(score_key(x[u].x), score_key(x[u].y), score_key(x[u].z),
                                   score_key(x[u].w));
        mn = min(min(min(mn, q.x), min(q.y, q.z)), q.w);
        mx = max(max(max(mx, q.x), max(q.y, q.z)), q.w);
        skeys4[unit((i + u * 128) >> 2)] = q;
      }
    } else {
      for (int u = 0; u < 4; ++u)
        for (int j = i + u * 128; j < i + u * 128 + 4; ++j) {
          uint32_t q = 0u;
          if (j >= v0 && j < v1) {
            q = score_key(__ldg(col + c0 + j));
            mn = min(mn, q);
            mx = max(mx, q);
          }
          skeys[unit(j >> 2) * 4 + (j & 3)] = q;
        }
    }
  }
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  cluster_wait();
  if (lane < CL) {
    st_peer(peer_shared(&s_mn[rank * nw + warp], lane), mn);
    st_peer(peer_shared(&s_mx[rank * nw + warp], lane), mx);
  }
  hist[0][tid] = 0;
  if (tid == 0) s_n = 0;
  cluster_arrive();
  cluster_wait();
  mn = 0xFFFFFFFFu;
  mx = 0u;
  for (int i = lane; i < TW; i += 32) { mn = min(mn, s_mn[i]); mx = max(mx, s_mx[i]); }
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);

  // the 16 keys of this lane from place i0 + 16 lane on, and which of them exist
  auto load16 = [&](int i0, uint32_t (&q)[16]) -> uint32_t {
    const int i = i0 + lane * 16;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint4 x = skeys4[unit((i >> 2) + u)];
      q[4 * u] = x.x; q[4 * u + 1] = x.y; q[4 * u + 2] = x.z; q[4 * u + 3] = x.w;
    }
    if (i0 >= v0 && i0 + kStep <= v1) return 0xFFFFu;
    const int a = min(max(v0 - i, 0), 16), z = min(max(v1 - i, 0), 16);
    return a < z ? ((1u << z) - 1u) & ~((1u << a) - 1u) : 0u;
  };
  auto each = [&](auto f) {
    for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
      uint32_t q[16];
      const uint32_t ok = load16(i0, q);
      if (ok == 0xFFFFu) {
#pragma unroll
        for (int j = 0; j < 16; ++j) f(q[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (ok >> j & 1u) f(q[j]);
      }
    }
  };
  int hi = mx == mn ? 0 : 32 - __clz(mx - mn);   // every offset key - mn lies in [0, 2^hi)
  uint32_t prefix = 0u, mask = hi == 32 ? 0u : ~((1u << hi) - 1u);
  int remaining = k, b = 0, inside = L;
  int listed = -1;                               // keys in this CTA's list, once there is one
  bool done = hi == 0 || k == 0;
  while (!done && hi > 0) {
    const int shift = max(hi - 8, 0);
    const uint32_t dmask = (1u << (hi - shift)) - 1u;
    // the next pass's buffer was last read before the previous pass's barrier
    const int bn = b == 2 ? 0 : b + 1;
    hist[bn][tid] = 0;
    int* h = hist[b];
    if (listed < 0 && inside <= kTail) {
      each([&](uint32_t key) {
        if ((((key - mn) ^ prefix) & mask) == 0u) s_keys[atomicAdd(&s_n, 1)] = key;
      });
      __syncthreads();
      listed = s_n;
    }
    auto count = [&](uint32_t key) {
      const uint32_t u = key - mn;
      if (((u ^ prefix) & mask) == 0u) atomicAdd(&h[(u >> shift) & dmask], 1);
    };
    if (listed >= 0)
      for (int i = tid; i < listed; i += 256) count(s_keys[i]);
    else
      each(count);
    cluster_arrive();
    cluster_wait();
    if (warp == 0) {
      int c[8], above, in;
#pragma unroll
      for (int j = 0; j < 8; ++j) c[j] = 0;
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        const uint32_t a = peer_shared(&h[lane * 8], r);
        const int4 x = ld_peer4(a), y = ld_peer4(a + 16);
        c[0] += x.x; c[1] += x.y; c[2] += x.z; c[3] += x.w;
        c[4] += y.x; c[5] += y.y; c[6] += y.z; c[7] += y.w;
      }
      const int bin = find_bin(c, remaining, above, in);
      if (lane == 0) { s_bin[0] = bin; s_bin[1] = above; s_bin[2] = in; }
    }
    __syncthreads();
    prefix |= (uint32_t)s_bin[0] << shift;
    remaining -= s_bin[1];
    inside = s_bin[2];
    done = inside == remaining;   // the whole bin is taken
    mask |= dmask << shift;
    hi = shift;
    b = bn;   // s_bin is written again after the next cluster barrier
  }
  // every key >= T is selected if the last bin is taken whole (or nothing is: k == 0, T above
  // all); else those above T and the first `remaining` equal to it
  const uint32_t T = prefix + mn;
  const bool whole = done && hi > 0;
  const int need_eq = whole ? 0x7FFFFFFF : remaining;
  int gt = 0, eq = 0;
  if (whole)
    each([&](uint32_t key) { gt += key >= T; });
  else
    each([&](uint32_t key) {
      gt += key > T;
      eq += key == T;
    });
  gt = __reduce_add_sync(0xffffffffu, gt);
  eq = __reduce_add_sync(0xffffffffu, eq);
  if (lane < CL) {
    st_peer(peer_shared(&s_gt[rank * nw + warp], lane), (uint32_t)gt);
    st_peer(peer_shared(&s_eq[rank * nw + warp], lane), (uint32_t)eq);
  }
  cluster_arrive();
  cluster_wait();   // the last access to another CTA's shared memory is behind it
  if (k > 0) {
    int gt0 = 0, eq0 = 0;   // keys of the column's lower warps
    for (int i = lane; i < rank * nw + warp; i += 32) { gt0 += s_gt[i]; eq0 += s_eq[i]; }
    gt0 = __reduce_add_sync(0xffffffffu, gt0);
    eq0 = __reduce_add_sync(0xffffffffu, eq0);
    const int first = gt0 + min(eq0, need_eq);   // selected keys before this warp's
    auto excl = [&](int v, int& total) {
      int incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      total = __shfl_sync(0xffffffffu, incl, 31);
      return incl - v;
    };
    int n = 0;                                   // selected keys of this warp so far
    for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
      uint32_t q[16], sel = 0u, seq = 0u;
      const uint32_t ok = load16(i0, q);
      if (whole) {
#pragma unroll
        for (int j = 0; j < 16; ++j) sel |= (uint32_t)(q[j] >= T) << j;
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          sel |= (uint32_t)(q[j] > T) << j;
          seq |= (uint32_t)(q[j] == T) << j;
        }
        seq &= ok;
        int all;
        const int before = eq0 + excl(__popc(seq), all);
        eq0 += all;
        while (__popc(seq) > max(need_eq - before, 0)) seq &= ~(0x80000000u >> __clz(seq));
      }
      sel = (sel & ok) | seq;
      int all;
      int at = w0 + n + excl(__popc(sel), all);   // (a warp step: every lane has read its keys)
      n += all;
      while (sel) {
        const int j = __ffs(sel) - 1;
        sel &= sel - 1u;
        skeys[at++] = (uint32_t)(i0 + lane * 16 + j);
      }
      __syncwarp();
    }
    const size_t row = (size_t)e * p.M + base + first;
#pragma unroll 4
    for (int i = lane; i < n; i += 32) {
      const int c = c0 + (int)skeys[w0 + i], t = lo + c;
      const float sv = __ldg(col + c);
      p.idx[row + i] = t;
      p.gate[row + i] = sv;
      if (p.idx2) p.idx2[row + i] = t;
      if (p.gate2) p.gate2[row + i] = sv;
      if (p.slot) p.slot[(size_t)t * p.E + e] = base + first + i;
    }
  }
  // last, so that the cluster barriers do not wait for these stores
  if (p.S_copy) {
    float* dst = p.S_copy + (size_t)e * p.N + lo + c0;
    const bool vec = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0;
    for (int i0 = w0; i0 < w0 + wlen; i0 += kStep) {
      const int i = i0 + lane * 4;
      if (vec && i0 >= v0 && i0 + kStep <= v1) {
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          x[u] = __ldg(reinterpret_cast<const float4*>(col + c0 + i + u * 128));
#pragma unroll
        for (int u = 0; u < 4; ++u) *reinterpret_cast<float4*>(dst + i + u * 128) = x[u];
      } else {
        for (int u = 0; u < 4; ++u)
          for (int j = i + u * 128; j < i + u * 128 + 4; ++j)
            if (j >= v0 && j < v1) dst[j] = __ldg(col + c0 + j);
      }
    }
  }
}

// Exclusive scan of two counts per thread (packed as hi:lo 32-bit halves) across the block.
__device__ __forceinline__ unsigned long long block_excl_scan2(unsigned long long v,
                                                               unsigned long long* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long w = lane < nw ? s_warp[lane] : 0ull;
    unsigned long long wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += u;
    }
    if (lane < nw) s_warp[lane] = wi - w;
  }
  __syncthreads();
  return incl - v + s_warp[warp];
}

// Columns too long for a cluster's shared memory (above 393216 scores): one CTA per column,
// every pass reads the scores again.
__global__ void __launch_bounds__(512) topk_long_kernel(TopkArgs p) {
  __shared__ __align__(16) int hist[256];
  __shared__ unsigned long long s_scan[32];
  __shared__ uint32_t s_mn[32], s_mx[32];
  const int e = blockIdx.x, g = blockIdx.y;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nw = nthr >> 5;
  pdl_begin(p.ST, p.group_off, p.k_g, p.k_off);
  const int lo = p.group_off[g];
  const int L = p.group_off[g + 1] - lo;
  const int k = p.k_g[g];
  const int base = p.k_off[g];
  const float* col = p.ST + (size_t)e * p.N + lo;

  uint32_t mn = 0xFFFFFFFFu, mx = 0u;
  for (int i = tid; i < L; i += nthr) {
    const float v = col[i];
    if (p.S_copy) p.S_copy[(size_t)e * p.N + lo + i] = v;
    const uint32_t key = score_key(v);
    mn = min(mn, key);
    mx = max(mx, key);
  }
  if (k == 0) return;
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) { s_mn[warp] = mn; s_mx[warp] = mx; }
  __syncthreads();
  mn = __reduce_min_sync(0xffffffffu, lane < nw ? s_mn[lane] : 0xFFFFFFFFu);
  mx = __reduce_max_sync(0xffffffffu, lane < nw ? s_mx[lane] : 0u);
  auto off_at = [&](int i) -> uint32_t { return score_key(col[i]) - mn; };

  int hi = mx == mn ? 0 : 32 - __clz(mx - mn);
  uint32_t prefix = 0u, mask = hi == 32 ? 0u : ~((1u << hi) - 1u);
  int remaining = k;
  bool done = hi == 0;
  while (!done && hi > 0) {
    const int shift = max(hi - 8, 0);
    const uint32_t dmask = (1u << (hi - shift)) - 1u;
    for (int i = tid; i < 256; i += nthr) hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < L; i += nthr) {
      const uint32_t u = off_at(i);
      if ((u & mask) == prefix) atomicAdd(&hist[(u >> shift) & dmask], 1);
    }
    __syncthreads();
    int c[8], above, inside;
#pragma unroll
    for (int j = 0; j < 8; ++j) c[j] = hist[lane * 8 + j];
    const int bin = find_bin(c, remaining, above, inside);
    prefix |= (uint32_t)bin << shift;
    remaining -= above;
    done = inside == remaining;
    mask |= dmask << shift;
    hi = shift;
    __syncthreads();   // the histogram is cleared next
  }
  const uint32_t T = prefix;
  const int need_eq = (done && hi > 0) ? 0x7FFFFFFF : remaining;

  // compaction in token order: thread tid owns a contiguous chunk
  const int chunk = (L + nthr - 1) / nthr;
  const int i0 = min(L, tid * chunk), i1 = min(L, i0 + chunk);
  uint32_t n_gt = 0, n_eq = 0;
  for (int i = i0; i < i1; ++i) {
    const uint32_t u = off_at(i);
    n_gt += u > T;
    n_eq += u == T;
  }
  const unsigned long long before =
      block_excl_scan2(((unsigned long long)n_gt << 32) | n_eq, s_scan);
  int r = (int)(before & 0xFFFFFFFFu);                 // keys equal to T before this one
  int pos = (int)(before >> 32) + min(r, need_eq);     // selected keys before this one
  const size_t row = (size_t)e * p.M + base;
  for (int i = i0; i < i1; ++i) {
    const uint32_t u = off_at(i);
    const bool eq = u == T;
    const bool s = u > T || (eq && r < need_eq);
    r += eq;
    if (s) {
      const int t = lo + i;
      const float sv = col[i];
      p.idx[row + pos] = t;
      p.gate[row + pos] = sv;
      if (p.idx2) p.idx2[row + pos] = t;
      if (p.gate2) p.gate2[row + pos] = sv;
      if (p.slot) p.slot[(size_t)t * p.E + e] = base + pos;
      ++pos;
    }
  }
}

// The limit on a kernel's shared memory is one for the process, so every call sets it to the most
// that any call needs: a call on another thread may come between this one's setting and its launch.
template <int CL>
static cudaError_t topk_cluster(const TopkArgs& p, int G, int span, LaunchStream st) {
  auto kern = topk_cluster_kernel<CL>;
  const int chunk = ((span + CL - 1) / CL + 8 * kStep - 1) / (8 * kStep) * (8 * kStep);
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kClusterKeys * 4);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, dim3((unsigned)(p.E * CL), (unsigned)G), 256, (size_t)chunk * 4, st, CL,
                       p, chunk);
}

// Columns of at most MAXK scores (with the places before the first one).
template <int NT, int MAXK>
static cudaError_t topk_block(const TopkArgs& p, int G, int span, LaunchStream st) {
  auto kern = topk_block_kernel<NT>;
  constexpr int unit = kStep * NT / 32;
  static_assert(MAXK % unit == 0, "the longest column fills its places");
  const int chunk = (span + unit - 1) / unit * unit;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (MAXK + kList) * 4);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, dim3(p.E, G), NT, ((size_t)chunk + kList) * 4, st, 1, p, chunk);
}

cudaError_t launch_topk(const TopkArgs& p, int G, int max_group, bool aligned, LaunchStream st) {
  if (G == 0 || p.E == 0) return cudaSuccess;
  // The registers that hold the longest column: 4 scores per thread for short ones (a 256-token
  // column then uses 64 threads, not 16), else 16; 128 threads up to 2048, so that every
  // column of a 16-sequence batch is resident at once. Above 8192 scores the keys go to shared
  // memory, of one CTA up to 49152, else of a cluster of eight. Columns that start off the
  // 16-byte grid take up to 3 places more.
  const int span = max_group + (aligned ? 0 : 3);
  const dim3 grid(p.E, G);
  if (span <= 512) return launch_kernel(topk_reg_kernel<4, 128, 8>, grid, 128, 0, st, 1, p);
  if (span <= 2048) return launch_kernel(topk_reg_kernel<16, 128, 8>, grid, 128, 0, st, 1, p);
  if (span <= 4096) return launch_kernel(topk_reg_kernel<16, 256, 4>, grid, 256, 0, st, 1, p);
  if (span <= 8192) return launch_kernel(topk_reg_kernel<16, 512, 2>, grid, 512, 0, st, 1, p);
  if (span <= 16384) return topk_block<512, 16384>(p, G, span, st);
  if (span <= 49152) return topk_block<1024, 49152>(p, G, span, st);
  if (span <= 8 * kClusterKeys) return topk_cluster<8>(p, G, span, st);
  return launch_kernel(topk_long_kernel, grid, 512, 0, st, 1, p);
}

// ------------------------------------------------------------------ capacity update
// Per-sequence capacities that change every step (Sec. 4.2) without a host round trip: the
// new k_g is read from device memory, checked, and the group tables are rewritten in place.
// One CTA; thread i owns a contiguous chunk of groups.
__global__ void __launch_bounds__(1024) set_capacity_kernel(const int* __restrict__ k_new,
                                                            const int* __restrict__ group_off,
                                                            int G, int M, int* __restrict__ k_g,
                                                            int* __restrict__ k_off,
                                                            int* __restrict__ status) {
  __shared__ long long s_part[1024];
  __shared__ int s_bad;
  pdl_begin(k_new, group_off);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int chunk = (G + nthr - 1) / nthr;
  const int g0 = min(G, tid * chunk), g1 = min(G, g0 + chunk);
  if (tid == 0) s_bad = 0;
  long long sum = 0;
  bool bad = false;
  for (int g = g0; g < g1; ++g) {
    const int k = k_new[g];
    bad |= k < 0 || k > group_off[g + 1] - group_off[g];
    sum += k;
  }
  s_part[tid] = sum;
  __syncthreads();
  if (bad) s_bad = 1;
  // inclusive scan of the chunk sums (Hillis-Steele over 1024 entries)
  for (int o = 1; o < nthr; o <<= 1) {
    const long long u = tid >= o ? s_part[tid - o] : 0;
    __syncthreads();
    s_part[tid] += u;
    __syncthreads();
  }
  const long long total = s_part[nthr - 1];
  if (s_bad || total != (long long)M) {
    if (tid == 0) atomicExch(status, DEV_BAD_CAPACITY);
    return;
  }
  long long run = s_part[tid] - sum;   // exclusive prefix of this chunk
  for (int g = g0; g < g1; ++g) {
    const int k = k_new[g];
    k_g[g] = k;
    k_off[g] = (int)run;
    run += k;
  }
  if (tid == nthr - 1) k_off[G] = (int)total;
}

cudaError_t launch_set_capacity(const int* k_new, const int* group_off, int G, int M, int* k_g,
                                int* k_off, int* status, LaunchStream st) {
  if (G <= 0) return cudaSuccess;
  return launch_kernel(set_capacity_kernel, 1, 1024, 0, st, 1, k_new, group_off, G, M, k_g, k_off,
                       status);
}

}  // namespace ecmoe
