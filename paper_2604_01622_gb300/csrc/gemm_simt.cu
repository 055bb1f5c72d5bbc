// Batched fp32 CUDA-core GEMMs of the fp32 path (tensor-core TF32 would miss its 1e-4 bound).
//
// C[b] = A[b] . B[b], one output tile per CTA. Both operands may be contiguous along K or
// along their other dimension; k-slices are fetched with 16-byte loads one slice ahead into
// registers, stored k-major into one of two shared buffers (one barrier per slice), and each
// thread accumulates a TM x TN block in column pairs (one paired FMA per two products). Every
// output is one chain of fused multiply-adds in ascending k, so the tile shape does not change
// a bit of the result.
//
// What bounds it: the FMA pipes. With 8 x 8 outputs per thread they are busy 69% of an SM's
// active cycles (ncu; the most frequent stall is the pipe itself), and 35-47 TFLOP/s come out of
// the 75 that the pipes allow, the rest lost to the last wave and the edge tiles. The scalar
// 4 x 4 kernel with 4-byte loads before it ran 22 TFLOP/s on the same shapes (16 experts of 1000
// rows, d 500, d_ff 364). The row gather of H = X[idx], the SwiGLU and its derivative, and the
// second product of dH are part of the same launches, so no intermediate is written that a
// later kernel only reads back: that layer's step 2820 -> 1304 us, a 256-token layer's (24
// kernels, now 13) 195 -> 62-64 us, most of it host time by now.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace ecmoe {

namespace {

enum SimtEpi : int {
  SIMT_PLAIN = 0,       // C
  SIMT_DUAL = 1,        // column halves: C = A.B, C2 = A.B2
  SIMT_SWIGLU_FWD = 2,  // column halves a = A.B, b = A.B2: C = a, C2 = b, C3 = silu(a) b
  SIMT_SWIGLU_BWD = 3   // acc = dU, with E1 = A, E2 = B: C = dA, C2 = dB
};

__device__ __forceinline__ uint64_t pair2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void split2(uint64_t r, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Four elements of a chunk whose contiguous dimension is at `i` of `n`: one 16-byte load when
// `vec` (n, the stride and the base are multiples of 16 bytes, so a chunk is in or out whole).
__device__ __forceinline__ void load4(float (&v)[4], const float* p, int i, int n, bool vec) {
  if (vec) {
    const float4 q = i < n ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(0, 0, 0, 0);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = i + j < n ? __ldg(p + j) : 0.f;
  }
}

// G consecutive values at dst (vec: 4 * G bytes aligned and wholly inside), else guarded.
template <int G>
__device__ __forceinline__ void store_group(float* dst, const float* v, int n, int N, bool vec) {
  if (vec) {
    if (n < N) {
      if constexpr (G == 4) *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
      else *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
    }
  } else {
#pragma unroll
    for (int j = 0; j < G; ++j)
      if (n + j < N) dst[j] = v[j];
  }
}

// A_K / B_K: the operand is contiguous along k. Thread (ty, tx) of TY x TX owns rows in RG
// groups of RW and columns in CG groups of CW, spread evenly over the tile (so with two B
// operands, each half of the tile's columns, it holds the same columns of both products).
template <int BM, int BN, int BK, int TM, int TN, int MINB, bool A_K, bool B_K, int EPI>
__global__ void __launch_bounds__(BM / TM * (BN / TN), MINB)
simt_gemm_kernel(const SimtGemmArgs p0, const SimtGemmArgs p1, int z1) {
  constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
  constexpr bool DUAL = EPI == SIMT_DUAL || EPI == SIMT_SWIGLU_FWD;
  constexpr int RW = TM >= 4 ? 4 : 2, RG = TM / RW;   // rows per group, groups per thread
  constexpr int CW = TN >= 8 ? 4 : 2, CG = TN / CW;   // columns per group, groups per thread
  constexpr int KQ = BK / 4;
  constexpr int LDA = BM + 4, LDB = BN + 4;
  constexpr int NA = BM * BK / 4 / NT, NB = BN * BK / 4 / NT;   // 16-byte chunks per thread
  static_assert(NA * NT * 4 == BM * BK && NB * NT * 4 == BN * BK, "chunks divide evenly");
  static_assert(KQ % 2 == 0 && BM % 16 == 0 && BN % 16 == 0 && TX % 8 == 0 && TY % 4 == 0 &&
                CG % 2 == 0, "chunk and thread maps");
  __shared__ __align__(16) float As[2][BK][LDA];
  __shared__ __align__(16) float Bs[2][BK][LDB];
  // a warp covers 4 x 8 threads of the block, so its 16-byte reads of Bs touch one 128-byte line
  // and those of As four addresses
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ty = warp / (TX / 8) * 4 + (lane >> 3), tx = warp % (TX / 8) * 8 + (lane & 7);
  // SIMT_DUAL: a second problem of the same form from grid layer z1 on
  const bool other = EPI == SIMT_DUAL && (int)blockIdx.z >= z1;
  const SimtGemmArgs p = other ? p1 : p0;
  const int z = (int)blockIdx.z - (other ? z1 : 0);
  const int b = z / p.splits, sp = z % p.splits;
  const int m0 = blockIdx.y * BM;
  const int n0 = blockIdx.x * (DUAL ? BN / 2 : BN);
  if (EPI == SIMT_DUAL && (m0 >= p.M || n0 >= p.N)) return;   // the grid covers both problems
  const int kb = sp * p.kchunk, ke = min(p.K, kb + p.kchunk);
  const int ksl = (ke - kb + BK - 1) / BK;            // k-slices of one product
  const int nsl = p.segs * ksl;
  const int* idx = p.idx ? p.idx + (int64_t)b * p.idx_bs : nullptr;
  const float* A0 = p.A + (int64_t)b * p.a_bs;
  const float* A1 = p.A2 + (int64_t)b * p.a_bs;
  const float* B0 = p.B + (int64_t)b * p.b_bs;
  const float* B1 = p.B2 + (int64_t)b * p.b_bs;
  pdl_begin(idx, A0, A1, B0, B1);
  const bool va = p.vec_a, vb = p.vec_b;

  // Chunk c of an operand contiguous along k: a warp takes 16 rows x 2 chunks, so its loads use
  // whole 32-byte sectors and its transposed 4-byte stores fall into 32 different banks
  // (rows of 4 LDA floats are 16 banks apart).
  auto ck = [](int c) { return ((c & 1) + 2 * ((c >> 5) % (KQ / 2))) * 4; };
  auto cm = [](int c) { return (c >> 5) / (KQ / 2) * 16 + ((c & 31) >> 1); };

  // A rows of this thread's chunks (gathered through idx where given): fixed over the k loop
  int64_t arow[A_K ? NA : 1];
  if constexpr (A_K) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int gm = m0 + cm(tid + i * NT);
      arow[i] = gm < p.M ? (int64_t)(idx ? __ldg(idx + gm) : gm) * p.a_ld : -1;
    }
  }
  float ra[NA][4], rb[NB][4];
  auto fetch = [&](int s) {
    const bool second = s >= ksl;
    const int k0 = kb + (second ? s - ksl : s) * BK;
    const float* Ab = second ? A1 : A0;
    const float* Bb = second && !DUAL ? B1 : B0;
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int c = tid + i * NT;
      if constexpr (A_K) {
        const int gk = k0 + ck(c);
        load4(ra[i], Ab + arow[i] + gk, arow[i] >= 0 ? gk : ke, ke, va);
      } else {
        const int gk = k0 + c / (BM / 4), gm = m0 + (c % (BM / 4)) * 4;
        const bool ok = gk < ke;
        const int64_t r = ok ? (idx ? __ldg(idx + gk) : gk) : 0;
        load4(ra[i], Ab + r * p.a_ld + gm, ok ? gm : p.M, p.M, va);
      }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int c = tid + i * NT;
      const int nn = B_K ? cm(c) : (c % (BN / 4)) * 4;   // column of the tile
      const bool h1 = DUAL && nn >= BN / 2;
      const float* Bp = h1 ? B1 : Bb;
      const int N = h1 ? p.N2 : p.N;
      const int gn = n0 + (h1 ? nn - BN / 2 : nn);
      if constexpr (B_K) {
        const int gk = k0 + ck(c);
        load4(rb[i], Bp + (int64_t)gn * p.b_ld + gk, gn < N ? gk : ke, ke, vb);
      } else {
        const int gk = k0 + c / (BN / 4);
        load4(rb[i], Bp + (int64_t)gk * p.b_ld + gn, gk < ke ? gn : N, N, vb);
      }
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int c = tid + i * NT;
      if constexpr (A_K) {
#pragma unroll
        for (int j = 0; j < 4; ++j) As[buf][ck(c) + j][cm(c)] = ra[i][j];
      } else {
        *reinterpret_cast<float4*>(&As[buf][c / (BM / 4)][(c % (BM / 4)) * 4]) =
            make_float4(ra[i][0], ra[i][1], ra[i][2], ra[i][3]);
      }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int c = tid + i * NT;
      if constexpr (B_K) {
#pragma unroll
        for (int j = 0; j < 4; ++j) Bs[buf][ck(c) + j][cm(c)] = rb[i][j];
      } else {
        *reinterpret_cast<float4*>(&Bs[buf][c / (BN / 4)][(c % (BN / 4)) * 4]) =
            make_float4(rb[i][0], rb[i][1], rb[i][2], rb[i][3]);
      }
    }
  };

  float* C = p.C + (int64_t)b * p.c_bs + (int64_t)sp * p.c_split;
  float* C2 = (EPI == SIMT_PLAIN) ? nullptr : p.C2 + (int64_t)b * p.c_bs;
  float* C3 = (EPI == SIMT_SWIGLU_FWD) ? p.C3 + (int64_t)b * p.c_bs : nullptr;
  auto row_of = [&](int i) { return m0 + (i / RW) * (BM / RG) + ty * RW + i % RW; };
  // column group h (of CG; of a dual tile, of the CG / 2 in each half)
  auto col_of = [&](int h) { return n0 + h * (BN / CG) + tx * CW; };

  uint64_t acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;

  if (nsl > 0) {
    fetch(0);
    put(0);
  }
  __syncthreads();
  for (int s = 0; s < nsl; ++s) {
    const int buf = s & 1;
    if (s + 1 < nsl) fetch(s + 1);
    if (EPI == SIMT_PLAIN && s == ksl && s > 0) {
      // the first product is complete: it waits in C (this thread's own elements) and the
      // second one starts from zero, so the two are rounded and added as separate sums
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int gm = row_of(i);
        float v[TN];
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) {
          split2(acc[i][j], v[2 * j], v[2 * j + 1]);
          acc[i][j] = 0ull;
        }
        if (gm < p.M)
#pragma unroll
          for (int h = 0; h < CG; ++h)
            store_group<CW>(C + (int64_t)gm * p.c_ld + col_of(h), v + h * CW, col_of(h), p.N,
                            p.vec_c);
      }
    }
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM];
      uint64_t bb[TN / 2];
#pragma unroll
      for (int g = 0; g < RG; ++g) {
        const float* src = &As[buf][k][g * (BM / RG) + ty * RW];
        if constexpr (RW == 4) {
          const float4 q = *reinterpret_cast<const float4*>(src);
          a[g * RW] = q.x; a[g * RW + 1] = q.y; a[g * RW + 2] = q.z; a[g * RW + 3] = q.w;
        } else {
          const float2 q = *reinterpret_cast<const float2*>(src);
          a[g * RW] = q.x; a[g * RW + 1] = q.y;
        }
      }
#pragma unroll
      for (int h = 0; h < CG; ++h) {
        const float* src = &Bs[buf][k][h * (BN / CG) + tx * CW];
        if constexpr (CW == 4) {
          const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(src);
          bb[2 * h] = q.x;
          bb[2 * h + 1] = q.y;
        } else {
          bb[h] = *reinterpret_cast<const unsigned long long*>(src);
        }
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const uint64_t aa = pair2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = fma2(aa, bb[j], acc[i][j]);
      }
    }
    // the other buffer was last read before the previous slice's barrier
    if (s + 1 < nsl) put(buf ^ 1);
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int gm = row_of(i);
    if (gm >= p.M) continue;
    float v[TN];
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) split2(acc[i][j], v[2 * j], v[2 * j + 1]);
    const int64_t ro = (int64_t)gm * p.c_ld;
    if constexpr (EPI == SIMT_PLAIN) {
#pragma unroll
      for (int h = 0; h < CG; ++h) {
        const int n = col_of(h);
        if (p.segs == 2)
#pragma unroll
          for (int j = 0; j < CW; ++j)
            if (n + j < p.N) v[h * CW + j] += C[ro + n + j];
        store_group<CW>(C + ro + n, v + h * CW, n, p.N, p.vec_c);
      }
    } else if constexpr (DUAL) {
#pragma unroll
      for (int h = 0; h < CG / 2; ++h) {
        const int n = col_of(h);
        const float* x = v + h * CW;
        const float* y = v + (CG / 2 + h) * CW;
        store_group<CW>(C + ro + n, x, n, p.N, p.vec_c);
        store_group<CW>(C2 + ro + n, y, n, p.N2, p.vec_c);
        if constexpr (EPI == SIMT_SWIGLU_FWD) {
          float u[CW];
#pragma unroll
          for (int j = 0; j < CW; ++j) u[j] = x[j] * sigmoidf_(x[j]) * y[j];
          store_group<CW>(C3 + ro + n, u, n, p.N, p.vec_c);
        }
      }
    } else {
      const float* E1 = after_wait(p.E1) + (int64_t)b * p.c_bs + ro;
      const float* E2 = after_wait(p.E2) + (int64_t)b * p.c_bs + ro;
#pragma unroll
      for (int h = 0; h < CG; ++h) {
        const int n = col_of(h);
        float da[CW], db[CW];
#pragma unroll
        for (int j = 0; j < CW; ++j) {
          const float aj = n + j < p.N ? __ldg(E1 + n + j) : 0.f;
          const float bj = n + j < p.N ? __ldg(E2 + n + j) : 0.f;
          const float du = v[h * CW + j], sg = sigmoidf_(aj);
          da[j] = du * bj * sg * (1.0f + aj * (1.0f - sg));
          db[j] = du * aj * sg;
        }
        store_group<CW>(C + ro + n, da, n, p.N, p.vec_c);
        store_group<CW>(C2 + ro + n, db, n, p.N, p.vec_c);
      }
    }
  }
}

int simt_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

template <int BM, int BN, int BK, int TM, int TN, int MINB, bool A_K, bool B_K, int EPI>
cudaError_t go(const SimtGemmArgs& a, const SimtGemmArgs* a2, LaunchStream st) {
  constexpr bool DUAL = EPI == SIMT_DUAL || EPI == SIMT_SWIGLU_FWD;
  constexpr int cols = DUAL ? BN / 2 : BN;
  const SimtGemmArgs& o = a2 ? *a2 : a;
  const int N = a.N > o.N ? a.N : o.N, M = a.M > o.M ? a.M : o.M;
  const int z1 = a.batch * a.splits;
  const dim3 grid((N + cols - 1) / cols, (M + BM - 1) / BM, z1 + (a2 ? a2->batch * a2->splits : 0));
  return launch_kernel(simt_gemm_kernel<BM, BN, BK, TM, TN, MINB, A_K, B_K, EPI>, grid,
                       BM / TM * (BN / TN), 0, st, 1, a, o, z1);
}

// Tile shape: the one whose busiest SM has the least work, tiles per SM (rounded up) times the
// tile's outputs times its measured cost per output against 128 x 128 (the shapes below, on
// 16 problems of M 1000 and M 96, N 364 and 500, K 364 to 1000: half tiles 1.0-1.12, 64 x 64
// 1.14, 32 x 32 2.1-2.4; 16 x 8 outputs per thread were slower in every shape, and so were A
// pairs kept in shared memory and fragments loaded a step ahead). Half tiles where 128 x 128
// leaves a nearly empty last wave, tall ones where A's rows are contiguous (gate/up 260 against
// 279 us, down 123 against 140, dH 254 against 281), wide ones for the weight gradients (dWd 160
// against 193) and dU; the small tiles for a few rows per expert (96 x 500 x 364: 27 against 43).
// A grid has at most 65535 rows of tiles, which rules the small ones out from 2.1 million rows on.
template <bool A_K, bool B_K, int EPI>
cudaError_t pick(const SimtGemmArgs& a, const SimtGemmArgs* a2, LaunchStream st) {
  constexpr int half = (EPI == SIMT_DUAL || EPI == SIMT_SWIGLU_FWD) ? 2 : 1;
  constexpr bool TALL = A_K && EPI != SIMT_SWIGLU_BWD;
  const int64_t sms = simt_sms();
  auto tiles_of = [&](const SimtGemmArgs& p, int bm, int bn) {
    return (int64_t)((p.M + bm - 1) / bm) * (((int64_t)p.N * half + bn - 1) / bn) * p.batch * p.splits;
  };
  auto cost = [&](int bm, int bn, double per_output) -> double {
    const int64_t tiles = tiles_of(a, bm, bn) + (a2 ? tiles_of(*a2, bm, bn) : 0);
    if ((std::max(a.M, a2 ? a2->M : 0) - 1) / bm >= 65535) return INFINITY;
    return (double)((tiles + sms - 1) / sms) * bm * bn * per_output;
  };
  const double c[4] = {cost(128, 128, 1.0), TALL ? cost(128, 64, 1.02) : cost(64, 128, 1.06),
                       cost(64, 64, 1.14), cost(32, 32, 2.2)};
  int best = 0;
  for (int i = 1; i < 4; ++i)
    if (c[i] < c[best]) best = i;
  switch (best) {
    case 0: return go<128, 128, 16, 8, 8, 2, A_K, B_K, EPI>(a, a2, st);
    case 1:
      if constexpr (TALL)
        return go<128, 64, 16, 8, 8, EPI == SIMT_SWIGLU_FWD ? 3 : 4, A_K, B_K, EPI>(a, a2, st);
      else
        return go<64, 128, 16, 8, 8, 4, A_K, B_K, EPI>(a, a2, st);
    case 2: return go<64, 64, 16, 8, 4, 4, A_K, B_K, EPI>(a, a2, st);
  }
  return go<32, 32, 32, 2, 4, 4, A_K, B_K, EPI>(a, a2, st);
}

bool vec_ok(const void* p, int64_t bs, int64_t ld, int contiguous) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && bs % 4 == 0 && ld % 4 == 0 &&
         contiguous % 4 == 0;
}

}  // namespace

static void prepare(SimtGemmArgs& a) {
  const bool second_a = a.segs == 2;
  if (!a.A2) a.A2 = a.A;
  if (!a.B2) a.B2 = a.B;
  if (a.N2 < 0) a.N2 = a.N;
  // split boundaries are multiples of 4, so a chunk of four k never crosses one
  a.kchunk = a.splits > 1 ? ((a.K + a.splits - 1) / a.splits + 3) / 4 * 4 : a.K;
  a.vec_a = vec_ok(a.A, a.a_bs, a.a_ld, a.a_kfast ? a.K : a.M) &&
            (!second_a || vec_ok(a.A2, a.a_bs, a.a_ld, a.a_kfast ? a.K : a.M));
  a.vec_b = vec_ok(a.B, a.b_bs, a.b_ld, a.b_kfast ? a.K : a.N) &&
            vec_ok(a.B2, a.b_bs, a.b_ld, a.b_kfast ? a.K : a.N2);
  a.vec_c = vec_ok(a.C, a.c_bs, a.c_ld, a.N) && a.c_split % 4 == 0 &&
            (!a.C2 || vec_ok(a.C2, a.c_bs, a.c_ld, a.N2)) &&
            (!a.C3 || vec_ok(a.C3, a.c_bs, a.c_ld, a.N));
}

cudaError_t launch_simt_gemm(SimtGemmArgs a, LaunchStream st) {
  if (a.M == 0 || a.N == 0 || a.batch == 0) return cudaSuccess;
  prepare(a);
  if (a.C3) return pick<true, false, SIMT_SWIGLU_FWD>(a, nullptr, st);
  if (a.E1) return pick<true, true, SIMT_SWIGLU_BWD>(a, nullptr, st);
  if (a.a_kfast)
    return a.b_kfast ? pick<true, true, SIMT_PLAIN>(a, nullptr, st)
                     : pick<true, false, SIMT_PLAIN>(a, nullptr, st);
  return pick<false, false, SIMT_PLAIN>(a, nullptr, st);
}

cudaError_t launch_simt_gemm_pair(SimtGemmArgs a, SimtGemmArgs b, LaunchStream st) {
  prepare(a);
  prepare(b);
  return pick<false, false, SIMT_DUAL>(a, &b, st);
}

// ------------------------------------------------------------------ router
// Scores of RBM tokens per CTA: logits X.Wr as one FMA chain per (token, expert) in ascending
// k, kept in shared memory (never written to global), then the row softmax, S, S^T and the
// slot map's -1. Neither the chain nor the softmax depends on the tile: every variant gives the
// same bits. A CTA is bound by its shared-memory reads (3 wavefronts per k and warp), so few tokens
// want small tiles on many SMs and many tokens the larger tiles' reuse.
namespace {
constexpr int RBK = 64;

template <int RBM, int BN, int TM, int TN>
__global__ void __launch_bounds__(RBM / TM * (BN / TN))
router_f32_kernel(const float* __restrict__ X, const float* __restrict__ Wr,
                  const float* __restrict__ br, float* __restrict__ S, float* __restrict__ ST,
                  int* __restrict__ slot, int N, int d, int E, bool vx, bool vw) {
  constexpr int TX = BN / TN, TY = RBM / TM, NT = TX * TY;
  constexpr int LDA = RBM + 4, LDB = BN + 4;
  constexpr int NA = RBM * RBK / 4 / NT, NB = BN * RBK / 4 / NT;
  static_assert(NA * NT * 4 == RBM * RBK && NB * NT * 4 == BN * RBK, "chunks divide evenly");
  pdl_begin(X, Wr, br);
  extern __shared__ float4 sh4[];
  float* As = reinterpret_cast<float*>(sh4);     // [2][RBK][LDA]
  float* Bs = As + 2 * RBK * LDA;                // [2][RBK][LDB]
  float* tile = Bs + 2 * RBK * LDB;              // [RBM][E+1] logits, then scores
  const int tid = threadIdx.x, ty = tid / TX, tx = tid % TX;
  const int warp = tid >> 5, lane = tid & 31, nw = NT / 32;
  const int t0 = blockIdx.x * RBM;
  const int nsl = (d + RBK - 1) / RBK;
  float ra[NA][4], rb[NB][4];
  for (int n0 = 0; n0 < E; n0 += BN) {
    auto fetch = [&](int s) {
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int c = tid + i * NT, t = t0 + c / (RBK / 4), k = s * RBK + (c % (RBK / 4)) * 4;
        load4(ra[i], X + (int64_t)t * d + k, t < N ? k : d, d, vx);
      }
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int c = tid + i * NT, k = s * RBK + c / (BN / 4), n = n0 + (c % (BN / 4)) * 4;
        load4(rb[i], Wr + (int64_t)k * E + n, k < d ? n : E, E, vw);
      }
    };
    auto put = [&](int buf) {
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int c = tid + i * NT;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          As[(buf * RBK + (c % (RBK / 4)) * 4 + j) * LDA + c / (RBK / 4)] = ra[i][j];
      }
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int c = tid + i * NT;
        *reinterpret_cast<float4*>(Bs + (buf * RBK + c / (BN / 4)) * LDB + (c % (BN / 4)) * 4) =
            make_float4(rb[i][0], rb[i][1], rb[i][2], rb[i][3]);
      }
    };
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
    fetch(0);
    put(0);
    __syncthreads();
    for (int s = 0; s < nsl; ++s) {
      const int buf = s & 1;
      if (s + 1 < nsl) fetch(s + 1);
#pragma unroll 16
      for (int k = 0; k < RBK; ++k) {
        float a[TM], w[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) a[i] = As[(buf * RBK + k) * LDA + ty * TM + i];
#pragma unroll
        for (int j = 0; j < TN; ++j) w[j] = Bs[(buf * RBK + k) * LDB + tx * TN + j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], w[j], acc[i][j]);
      }
      if (s + 1 < nsl) put(buf ^ 1);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int e = n0 + tx * TN + j;
        if (e < E) tile[(ty * TM + i) * (E + 1) + e] = acc[i][j];
      }
  }
  __syncthreads();
  for (int r = warp; r < RBM; r += nw) {
    const int t = t0 + r;
    if (t >= N) break;
    float* row = tile + r * (E + 1);
    float mx = -INFINITY;
    for (int e = lane; e < E; e += 32) {
      const float v = row[e] + (br ? __ldg(br + e) : 0.0f);
      row[e] = v;
      mx = fmaxf(mx, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float sum = 0.f;
    for (int e = lane; e < E; e += 32) {
      const float q = expf(row[e] - mx);
      row[e] = q;
      sum += q;
    }
    sum = warp_sum(sum);
    const float inv = 1.0f / sum;
    for (int e = lane; e < E; e += 32) {
      const float q = row[e] * inv;
      row[e] = q;
      if (S) S[(size_t)t * E + e] = q;
      if (slot) slot[(size_t)t * E + e] = -1;
    }
  }
  __syncthreads();
  for (int i = tid; i < E * RBM; i += NT) {
    const int e = i / RBM, r = i % RBM;
    if (t0 + r < N) ST[(size_t)e * N + t0 + r] = tile[r * (E + 1) + e];
  }
}

template <int RBM, int BN, int TM, int TN>
cudaError_t router_go(const float* X, const float* Wr, const float* br, float* S, float* ST,
                      int* slot, int N, int d, int E, LaunchStream st) {
  auto kern = router_f32_kernel<RBM, BN, TM, TN>;
  auto bytes = [](int experts) {
    return ((size_t)2 * RBK * (RBM + 4 + BN + 4) + (size_t)RBM * (experts + 1)) * sizeof(float);
  };
  // narrow tiles are for up to BN experts; the limit, one for the process, covers every call's need
  // (a call on another thread may come between this one's setting and its launch)
  constexpr int most = BN < 128 ? BN : 512;
  const size_t smem = bytes(E);
  if (bytes(most) > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)bytes(most));
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(kern, (N + RBM - 1) / RBM, RBM / TM * (BN / TN), smem, st, 1, X, Wr, br, S,
                       ST, slot, N, d, E, vec_ok(X, 0, d, d), vec_ok(Wr, 0, E, E));
}
}  // namespace

cudaError_t launch_router_f32(const float* X, const float* Wr, const float* br, float* S,
                              float* ST, int* slot, int N, int d, int E, LaunchStream st) {
  if (N == 0) return cudaSuccess;
  // Tokens per CTA by how many 152 SMs get (1216 = 8 x 152 tokens, 4864 = 16 x 2 x 152, 9728 = 16
  // x 4 x 152); one pass over X up to 128 experts. d 656, from 32 tokens x 64 experts (x 16 for
  // E <= 16) per CTA for every size: 16 experts, 858 tokens 31 -> 19 us (16000: 47.5, and 48.5
  // with 16 tokens); 30 experts, 858 36 -> 22, 16000 97 -> 65; 64 experts, 858 36 -> 24, 3000
  // 50 -> 44, 16000 98 -> 71; 128 experts, 858 60 -> 32, 3000 89 -> 62, 16000 180 -> 120.
  if (E <= 16)
    return N <= 9728 ? router_go<16, 16, 2, 1>(X, Wr, br, S, ST, slot, N, d, E, st)
                     : router_go<32, 16, 2, 2>(X, Wr, br, S, ST, slot, N, d, E, st);
  if (E <= 32) return router_go<16, 32, 2, 2>(X, Wr, br, S, ST, slot, N, d, E, st);
  if (E <= 64)
    return N <= 1216   ? router_go<8, 64, 1, 4>(X, Wr, br, S, ST, slot, N, d, E, st)
           : N <= 4864 ? router_go<16, 64, 2, 4>(X, Wr, br, S, ST, slot, N, d, E, st)
                       : router_go<64, 64, 4, 4>(X, Wr, br, S, ST, slot, N, d, E, st);
  return N <= 1216 ? router_go<16, 128, 2, 4>(X, Wr, br, S, ST, slot, N, d, E, st)
                   : router_go<32, 128, 4, 4>(X, Wr, br, S, ST, slot, N, d, E, st);
}

}  // namespace ecmoe
