// FFMA matrix products for the fp32 precision mode (tensor cores have no fp32-operand kind), for
// shapes the tensor-core path does not take, and as an on-device cross-check of that path.
// One kernel covers forward (A W^T), dgrad (dZ W) and wgrad (dZ^T A) through element strides.
//
// Small layers with a long contraction (the weight gradient of the paper's 80- and 60-wide layers
// over a batch of 1410: one or two output tiles, 88 k-steps) would leave the GPU idle, so K can be
// split over gridDim.z CTAs per tile: every CTA stores its partial tile to a workspace, the last one
// to arrive adds the partials in split order (a fixed order: bit-reproducible), applies the epilogue
// and leaves the arrival counter at zero.
//
// gemm_ffma_kernel is the fp32 path proper: tiles of 64 x 64, both operands brought by tensor copies into a ring of shared-memory
// stages, 8 x 8 outputs per thread.  The 64 threads that hold a tile exist four times in a CTA (each group takes a quarter of
// every stage's K) and S CTAs of a cluster split K again, so that few tiles still fill the GPU; the partial tiles meet in
// shared memory and, as a reduce-scatter, in distributed shared memory, in a fixed order.  gemm_simt_kernel serves what tensor
// copies cannot take (rows that are no whole 16-byte groups), bf16 operands on the FFMA backend, and the fp32 products it is
// the faster one for (strided_is_faster).
#include <algorithm>
#include <atomic>

#include "async_copy.cuh"
#include "common.cuh"

namespace segk {
namespace {

constexpr int BM = 64, BN = 64, BK = 32, PAD = 4;

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(256)
gemm_simt_kernel(GemmDesc g, int k_per_split) {
  pdl_wait();
  pdl_trigger();
  __shared__ bool is_last;
  __shared__ __align__(16) float As[BK][BM + PAD];
  __shared__ __align__(16) float Bs[BK][BN + PAD];
  const TIn* __restrict__ A = reinterpret_cast<const TIn*>(g.A);
  const TIn* __restrict__ B = reinterpret_cast<const TIn*>(g.B);
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool a_kfast = (g.a_sk == 1), b_nfast = (g.b_sn == 1);
  float acc[4][4] = {};
  const int k_begin = blockIdx.z * k_per_split, k_end = min(g.K, k_begin + k_per_split);
  constexpr int LD = BM * BK / 256;          // elements of each operand tile a thread fetches per k-step
  float ra[LD], rb[LD];
  // fetch of one k-step into registers; the next step's fetch is issued before this step's arithmetic
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int idx = threadIdx.x + 256 * i;
      const int k = a_kfast ? (idx & (BK - 1)) : (idx / BM);
      const int m = a_kfast ? (idx / BK) : (idx & (BM - 1));
      ra[i] = 0.f;
      if (m0 + m < g.M && k0 + k < k_end) ra[i] = to_f<TIn>(A[(int64_t)(m0 + m) * g.a_sm + (int64_t)(k0 + k) * g.a_sk]);
    }
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int idx = threadIdx.x + 256 * i;
      const int n = b_nfast ? (idx & (BN - 1)) : (idx / BK);
      const int k = b_nfast ? (idx / BN) : (idx & (BK - 1));
      rb[i] = 0.f;
      if (n0 + n < g.N && k0 + k < k_end) rb[i] = to_f<TIn>(B[(int64_t)(k0 + k) * g.b_sk + (int64_t)(n0 + n) * g.b_sn]);
    }
  };
  if (k_begin < k_end) fetch(k_begin);
  for (int k0 = k_begin; k0 < k_end; k0 += BK) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int idx = threadIdx.x + 256 * i;
      As[a_kfast ? (idx & (BK - 1)) : (idx / BM)][a_kfast ? (idx / BK) : (idx & (BM - 1))] = ra[i];
      Bs[b_nfast ? (idx / BN) : (idx & (BK - 1))][b_nfast ? (idx & (BN - 1)) : (idx / BK)] = rb[i];
    }
    __syncthreads();
    if (k0 + BK < k_end) fetch(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (gridDim.z > 1) {
    const int tile = blockIdx.y * gridDim.x + blockIdx.x;
    float* slot = g.simt_scratch + ((size_t)tile * gridDim.z + blockIdx.z) * kSimtTileFloats;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<float4*>(slot + (ty * 4 + i) * BN + tx * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(g.simt_counters + tile, 1u) == gridDim.z - 1);
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    const float* base = g.simt_scratch + (size_t)tile * gridDim.z * kSimtTileFloats;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (unsigned int z = 0; z < gridDim.z; ++z) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 p = __ldcg(reinterpret_cast<const float4*>(base + (size_t)z * kSimtTileFloats + (ty * 4 + i) * BN + tx * 4));
        acc[i][0] += p.x; acc[i][1] += p.y; acc[i][2] += p.z; acc[i][3] += p.w;
      }
    }
    if (threadIdx.x == 0) g.simt_counters[tile] = 0u;
  }
  TOut* __restrict__ C = reinterpret_cast<TOut*>(g.C);
  const TOut* __restrict__ mask = reinterpret_cast<const TOut*>(g.mask);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n >= g.N) continue;
      float v = acc[i][j];
      if (g.epi == EPI_BIAS_ACT) {
        v += g.bias[n];
        if (g.relu) v = fmaxf(v, 0.f);
      } else if (g.epi == EPI_MASK) {
        if (!(to_f<TOut>(mask[(int64_t)m * g.ldmask + n]) > 0.f)) v = 0.f;
      }
      v = apply_round(v, g.c_round);
      if constexpr (sizeof(TOut) == 2) C[(int64_t)m * g.ldc + n] = __float2bfloat16_rn(v);
      else C[(int64_t)m * g.ldc + n] = v;
    }
  }
}

// ---- fp32 products by tensor copies and packed FFMA ------------------------------------------------------
// What bounds it: FFMA issue beside the loads of 8 x 8 tiles from shared memory.  Packed multiply-adds (fma.rn.f32x2, two per
// issue slot) leave slots for the loads.  At 2048^3 / 4096^3: NT 37.6 / 39.7 TFLOP/s, NN 42.2 / 43.6, TN 49.2 / 51.2, 53 to 72 %
// of the 71.5 that a loop of multiply-adds alone reaches.
constexpr int FT = 64, FK = 32;                             // tile edge, k per stage
constexpr int FGROUPS = 4, FTHREADS = 64 * FGROUPS;         // four k groups of 64 threads
// NN and TN have a ninth warp that issues the tensor copies (TN at 2048^3 falls from 49 to 43 TFLOP/s when a computing warp issues
// them); NT does without: nine warps leave a thread 168 registers, its 64 pairs of sums need more (38 TFLOP/s against 33 with
// the ninth warp and plain multiply-adds).
__host__ __device__ constexpr int ffma_threads(int form) { return FTHREADS + (form == 0 ? 0 : 32); }
constexpr int FSTAGES = 6, FSTAGE_FLOATS = 2 * FT * FK;     // 16 KiB per stage
constexpr int FPART = FT + 8;                               // row pitch of a partial tile: conflict-free stores in every form
constexpr int FRING_FLOATS = FSTAGES * FSTAGE_FLOATS;
constexpr size_t FSMEM = 1024 + (size_t)(FRING_FLOATS + FT * FT) * sizeof(float);
static_assert(FGROUPS * FT * FPART <= FRING_FLOATS, "the partial tiles take the ring's place");

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ void fma2(f32x2& c, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b)); }

struct FfmaEpi { void* C; int64_t ldc, ldmask; int c_round, epi, relu; const float* bias; const float* mask; };

template <int FORM>
__global__ void __launch_bounds__(ffma_threads(FORM), 1)
gemm_ffma_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int M, int N, int K, int S,
                 int k_per_cta, FfmaEpi e, int* dev_status) {
  extern __shared__ uint8_t raw[];
  float* sm = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
  float* recv = sm + FRING_FLOATS;                          // [source CTA][64 / S rows][64]
  __shared__ uint64_t full[FSTAGES], empty[FSTAGES];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = S > 1 ? (int)cluster_rank() : 0;
  const int tile = (int)blockIdx.x / S, tiles_m = (M + FT - 1) / FT;
  const int m0 = tile % tiles_m * FT, n0 = tile / tiles_m * FT;
  const int k0 = rank * k_per_cta, k1 = min(K, k0 + k_per_cta), steps = k1 > k0 ? (k1 - k0 + FK - 1) / FK : 0;
  if (tid == 0) {
    for (int i = 0; i < FSTAGES; ++i) { bar_init(full + i, 1); bar_init(empty + i, 2 * FGROUPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async();
  }
  __syncthreads();
  if (S > 1) cluster_arrive_release();
  pdl_wait();
  pdl_trigger();
  const int grp = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  // NT: pairs along k (even and odd partial sums of all 64 outputs); NN, TN: pairs of columns
  constexpr int NJ = FORM == FORM_NT ? 8 : 4;
  f32x2 acc[8][NJ];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = 0ull;
  auto load = [&](int s) {                                  // by the issuing thread
    const int st = s % FSTAGES, k = k0 + s * FK;
    float* a = sm + st * FSTAGE_FLOATS;
    float* b = a + FT * FK;
    bar_expect(full + st, FSTAGE_FLOATS * 4);
    if constexpr (FORM == FORM_TN) tensor_load(a, &map_a, m0, k, full + st); else tensor_load(a, &map_a, k, m0, full + st);
    if constexpr (FORM == FORM_NT) tensor_load(b, &map_b, k, n0, full + st); else tensor_load(b, &map_b, n0, k, full + st);
  };
  constexpr bool COPY_WARP = ffma_threads(FORM) > FTHREADS;
  if (!COPY_WARP && warp == 0) {
    if (elect_one())
      for (int s = 0; s < min(steps, FSTAGES); ++s) load(s);
  }
  if (COPY_WARP && warp == 2 * FGROUPS) {
    if (elect_one())
      for (int s = 0; s < steps; ++s) {
        if (s >= FSTAGES) bar_wait(empty + s % FSTAGES, (uint32_t)(s / FSTAGES - 1) & 1u, dev_status);
        load(s);
      }
  } else {
    // this group's 8 of every stage's 32 k
    for (int s = 0; s < steps; ++s) {
      const int st = s % FSTAGES;
      const float* a_s = sm + st * FSTAGE_FLOATS;
      const float* b_s = a_s + FT * FK;
      bar_wait(full + st, (uint32_t)(s / FSTAGES) & 1u, dev_status);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = 2 * grp + h;                          // four k: c * 4 ..
        if constexpr (FORM == FORM_NT) {
          // k-fast tiles: rows of 32 k, 128-byte swizzle (16-byte group c of row r at c ^ (r & 7)); a 16-byte load is two pairs
          ulonglong2 a[8];
          const float* ar = a_s + ty * FK + ((c ^ ty) << 2);
          const float* br = b_s + tx * FK + ((c ^ tx) << 2);
#pragma unroll
          for (int i = 0; i < 8; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(ar + i * 8 * FK);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(br + j * 8 * FK);
#pragma unroll
            for (int i = 0; i < 8; ++i) fma2(acc[i][j], a[i].x, b.x);
#pragma unroll
            for (int i = 0; i < 8; ++i) fma2(acc[i][j], a[i].y, b.y);
          }
        } else {
          // n-fast B: rows of 64 n; packed multiply-adds over pairs of columns 4 tx .. and 32 + 4 tx ..
          float4 a[8];                                      // NN: [row i] four k;  TN: [2 k' + half] four rows
          if constexpr (FORM == FORM_NN) {
            const float* ar = a_s + ty * FK + ((c ^ ty) << 2);
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] = *reinterpret_cast<const float4*>(ar + i * 8 * FK);
          } else {
            const float* ar = a_s + 4 * c * FT + 4 * ty;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              a[2 * k] = *reinterpret_cast<const float4*>(ar + k * FT);
              a[2 * k + 1] = *reinterpret_cast<const float4*>(ar + k * FT + 32);
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float* br = b_s + (4 * c + k) * FT + 4 * tx;
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(br), b1 = *reinterpret_cast<const ulonglong2*>(br + 32);
            const f32x2 b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float av;
              if constexpr (FORM == FORM_NN) av = k == 0 ? a[i].x : k == 1 ? a[i].y : k == 2 ? a[i].z : a[i].w;
              else { const float4 t = a[2 * k + (i >> 2)]; av = (i & 3) == 0 ? t.x : (i & 3) == 1 ? t.y : (i & 3) == 2 ? t.z : t.w; }
              const f32x2 aa = pack2(av, av);
#pragma unroll
              for (int j = 0; j < 4; ++j) fma2(acc[i][j], aa, b[j]);
            }
          }
        }
      }
      if (s + FSTAGES < steps) {
        __syncwarp();
        if (lane == 0) bar_arrive(empty + st);
      }
      if (!COPY_WARP && warp == 0 && s + FSTAGES < steps) {
        if (elect_one()) { bar_wait(empty + st, (uint32_t)(s / FSTAGES) & 1u, dev_status); load(s + FSTAGES); }
      }
    }
  }
  __syncthreads();                                          // the ring is free: partial tiles [group][64][72] take its place
  if (!COPY_WARP || warp < 2 * FGROUPS) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int m = FORM == FORM_TN ? (i >> 2) * 32 + 4 * ty + (i & 3) : ty + 8 * i;
      float* d = sm + (grp * FT + m) * FPART;
      if constexpr (FORM == FORM_NT) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float lo, hi;
          unpack2(acc[i][j], lo, hi);
          d[tx + 8 * j] = lo + hi;
        }
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float4 v;
          unpack2(acc[i][2 * h], v.x, v.y);
          unpack2(acc[i][2 * h + 1], v.z, v.w);
          *reinterpret_cast<float4*>(d + 32 * h + 4 * tx) = v;
        }
      }
    }
  }
  const int slice = FT / S;                                 // rows each CTA of the cluster finishes
  if (S > 1) cluster_wait_acquire();                        // every peer has started: its shared memory may be written
  __syncthreads();
  auto group_sum = [&](int row, int c) {
    float4 v = lds4(sm + row * FPART + 4 * c);
#pragma unroll
    for (int g = 1; g < FGROUPS; ++g) add4(v, lds4(sm + (g * FT + row) * FPART + 4 * c));
    return v;
  };
  if (S > 1) {
    if (!COPY_WARP || tid < FTHREADS) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int row = (tid >> 4) + 16 * u, c = tid & 15, owner = row / slice;
        const uint32_t off = 4u * (uint32_t)((rank * slice + row - owner * slice) * FT + 4 * c);
        store_cluster4(in_cta(smem_addr(recv), (uint32_t)owner) + off, group_sum(row, c));
      }
    }
    cluster_arrive_release();
    cluster_wait_acquire();
  }
  if (COPY_WARP && tid >= FTHREADS) return;
  float* C = reinterpret_cast<float*>(e.C);
  const bool wide = (e.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0;
  const bool mask_wide = (e.ldmask & 3) == 0 && (reinterpret_cast<uintptr_t>(e.mask) & 15u) == 0;
  for (int r = tid >> 4; r < slice; r += 16) {
    const int c = tid & 15, m = m0 + rank * slice + r, n = n0 + 4 * c;
    if (m >= M || n >= N) continue;
    float4 v4;
    if (S > 1) {
      v4 = lds4(recv + r * FT + 4 * c);
      for (int s = 1; s < S; ++s) add4(v4, lds4(recv + (s * slice + r) * FT + 4 * c));
    } else {
      v4 = group_sum(r, c);
    }
    float v[4] = {v4.x, v4.y, v4.z, v4.w};
    const bool whole = n + 3 < N;
    if (e.epi == EPI_BIAS_ACT) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (n + j < N) v[j] += __ldg(e.bias + n + j);
        if (e.relu) v[j] = fmaxf(v[j], 0.f);
      }
    } else if (e.epi == EPI_MASK) {
      const float* mr = e.mask + (int64_t)m * e.ldmask + n;
      if (whole && mask_wide) {
        const float4 q = *reinterpret_cast<const float4*>(mr);
        if (!(q.x > 0.f)) v[0] = 0.f;
        if (!(q.y > 0.f)) v[1] = 0.f;
        if (!(q.z > 0.f)) v[2] = 0.f;
        if (!(q.w > 0.f)) v[3] = 0.f;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) if (n + j < N && !(mr[j] > 0.f)) v[j] = 0.f;
      }
    }
    if (e.c_round == RND_TF32) {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = round_tf32_rne(v[j]);
    }
    float* cr = C + (int64_t)m * e.ldc + n;
    if (whole && wide) *reinterpret_cast<float4*>(cr) = make_float4(v[0], v[1], v[2], v[3]);
    else {
#pragma unroll
      for (int j = 0; j < 4; ++j) if (n + j < N) cr[j] = v[j];
    }
  }
}

// CTAs that split K of one tile.  A CTA pays about 3000 cycles of latencies (start, first stage, exchange, epilogue) and 46
// cycles per k (64 x 64 multiply-adds at 70 % of the FFMA rate); clusters of 2, 4 and 8 leave 148, 132 and 120 SMs to fill.
int ffma_split(int tiles, int K, double* cycles = nullptr) {
  int best = 1;
  double best_t = 1e30;
  for (int S : {1, 2, 4, 8}) {
    const int resident = S == 1 ? 148 : S == 2 ? 74 : S == 4 ? 33 : 15;
    const int kp = ((K + S - 1) / S + FK - 1) / FK * FK;
    if (S > 1 && kp * (S - 1) >= K) continue;               // a CTA would have nothing to do
    const double t = (double)((tiles + resident - 1) / resident) * ((S > 1 ? 4000.0 : 3000.0) + 46.0 * kp);
    if (t < best_t) { best_t = t; best = S; }
  }
  if (cycles) *cycles = best_t;
  return best;
}

template <int FORM>
cudaError_t launch_ffma(const CUtensorMap& ma, const CUtensorMap& mb, const GemmDesc& g, int* dev_status, cudaStream_t s) {
  static std::atomic<bool> allowed[64];
  auto kern = gemm_ffma_kernel<FORM>;
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!allowed[dev].load(std::memory_order_acquire)) {
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FSMEM);
    if (err != cudaSuccess) return err;
    allowed[dev].store(true, std::memory_order_release);
  }
  const int tiles = ((g.M + FT - 1) / FT) * ((g.N + FT - 1) / FT);
  const int S = ffma_split(tiles, g.K);
  const int kp = ((g.K + S - 1) / S + FK - 1) / FK * FK;
  FfmaEpi e{};
  e.C = g.C; e.ldc = g.ldc; e.ldmask = g.ldmask; e.c_round = g.c_round; e.epi = g.epi; e.relu = g.relu;
  e.bias = g.bias; e.mask = reinterpret_cast<const float*>(g.mask);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * S)); cfg.blockDim = dim3(ffma_threads(FORM)); cfg.dynamicSmemBytes = FSMEM; cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (g_use_pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (S > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)S; attr[n].val.clusterDim.y = 1; attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr; cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, ma, mb, g.M, g.N, g.K, S, kp, e, dev_status);
}

// The split of K the strided kernel takes: while it adds CTAs the GPU has room for and leaves every split at least 4 k-steps.
struct StridedSplit { int splits, k_per_split; };
StridedSplit strided_split(int tiles, int K, int slots) {
  int splits = 1;
  if (tiles <= slots) splits = std::max(1, std::min(std::min(148 / tiles, slots / tiles), K / (4 * BK)));
  const int k_per_split = std::max(BK, ((K + splits - 1) / splits + BK - 1) / BK * BK);
  return {std::max(1, (K + k_per_split - 1) / k_per_split), k_per_split};
}

// Estimated cycles of an fp32 product in each of the two kernels.  Which one takes it (strided_is_faster): two kinds of products
// are the strided kernel's - few tiles over a very long contraction (the weight gradient of narrow layers over a large batch, very
// wide inputs), which it cuts into up to 148 pieces where a cluster cuts 8, and many tiles over a short one, where two of its CTAs
// share an SM and the other kernel's fixed cost of 6500 to 8500 cycles per tile is most of its time.  Strided against tensor
// copies, us: weight gradient of 64 x 64 over 16384 / 65536 rows 29 / 50 against 56 / 207, forward 65536 x 256 over K = 8 / 64 /
// 128 78 / 117 / 205 against 111 / 138 / 189, dgrad 65536 x 784 over K = 8 / 64 / 128 297 / 410 / 660 against 555 / 637 / 793.
// The constants follow from 552 products timed in both kernels: none of them goes to one that is over 5 % and 0.6 us behind.
double copies_cycles(Form form, int tiles, int K) {
  const int S = ffma_split(tiles, K);
  const int resident = S == 1 ? 148 : S == 2 ? 74 : S == 4 ? 33 : 15, kp = ((K + S - 1) / S + FK - 1) / FK * FK;
  const double fixed = (form == FORM_NT ? 6500.0 : form == FORM_NN ? 8500.0 : 7000.0) + (S > 1 ? 1000.0 : 0.0);
  return (double)((tiles + resident - 1) / resident) * (fixed + 46.0 * kp);
}
double strided_cycles(int tiles, int K, int slots) {
  const StridedSplit sp = strided_split(tiles, K, slots);
  const int64_t ctas = (int64_t)tiles * sp.splits;
  const double t = ctas > 148 ? (double)((ctas + 295) / 296) * (4800.0 + 168.0 * sp.k_per_split) : 6000.0 + 107.0 * sp.k_per_split;
  return t + (sp.splits > 1 ? 200.0 * sp.splits : 0.0);
}
// Not for a few per cent, though: its CTAs take more of the SMs from the products of other branches (weight gradients, TN, run
// beside the dgrad chain).  Whole steps of 81 fp32 cases against tensor copies alone: 0.986 of the time with these factors, 0.995
// with 0.75 for all three forms, 1.004 with 0.75 for TN and 0 for the others; the worst case 1.05, 1.14 and 1.13.
bool strided_is_faster(Form form, int tiles, int K, int slots) {
  return strided_cycles(tiles, K, slots) < (form == FORM_TN ? 0.75 : 0.93) * copies_cycles(form, tiles, K);
}

// cudaErrorNotSupported: operands that tensor copies cannot take (the strided kernel serves them).
cudaError_t try_ffma(const GemmDesc& g, int* dev_status, cudaStream_t s) {
  if (g.a_dt != DT_F32 || g.b_dt != DT_F32 || g.c_dt != DT_F32 || g.M <= 0 || g.N <= 0 || g.K <= 0 || g.c_round == RND_BF16)
    return cudaErrorNotSupported;
  const bool a_k = g.a_sk == 1, b_k = g.b_sk == 1 && g.b_sn != 1;
  const int64_t a_pitch = a_k ? g.a_sm : g.a_sk, b_pitch = b_k ? g.b_sn : g.b_sk;
  if ((!a_k && g.a_sm != 1) || (!b_k && g.b_sn != 1) || (!a_k && b_k)) return cudaErrorNotSupported;
  if ((a_pitch & 3) || (b_pitch & 3) || ((reinterpret_cast<uintptr_t>(g.A) | reinterpret_cast<uintptr_t>(g.B)) & 15u)) return cudaErrorNotSupported;
  CUtensorMap ma, mb;
  bool ok = a_k ? make_map_f32(&ma, g.A, (uint64_t)g.K, (uint64_t)g.M, (uint64_t)a_pitch * 4, FK, FT, true)
                : make_map_f32(&ma, g.A, (uint64_t)g.M, (uint64_t)g.K, (uint64_t)a_pitch * 4, FT, FK, false);
  ok = ok && (b_k ? make_map_f32(&mb, g.B, (uint64_t)g.K, (uint64_t)g.N, (uint64_t)b_pitch * 4, FK, FT, true)
                  : make_map_f32(&mb, g.B, (uint64_t)g.N, (uint64_t)g.K, (uint64_t)b_pitch * 4, FT, FK, false));
  if (!ok) return cudaErrorNotSupported;
  if (a_k && b_k) return launch_ffma<FORM_NT>(ma, mb, g, dev_status, s);
  if (a_k) return launch_ffma<FORM_NN>(ma, mb, g, dev_status, s);
  return launch_ffma<FORM_TN>(ma, mb, g, dev_status, s);
}

}  // namespace

double ffma_estimate_us(int M, int N, int K) {
  double cycles = 0;
  ffma_split(((M + FT - 1) / FT) * ((N + FT - 1) / FT), K, &cycles);
  return cycles / 1900.0;
}

// The copy: a launch of about 3 us and 8 bytes per element at about 3 TB/s.  784-80-60 at 8192 rows, us: 85 with the strided first
// layer, 72 with the copy (63 from aligned rows).
bool fp32_staging_pays(int M, int N, int K, int slots) {
  const int tiles = ((M + FT - 1) / FT) * ((N + FT - 1) / FT);
  return strided_cycles(tiles, K, slots) / 1900.0 > copies_cycles(FORM_NT, tiles, K) / 1900.0 + 3.0 + 8.0 * M * K / 3e6;
}

// Partial tiles the split of an M x N x K product would use with an unlimited workspace (0: no split).
int gemm_simt_slots(int M, int N, int K) {
  const int tiles = ((N + BN - 1) / BN) * ((M + BM - 1) / BM);
  if (tiles < 1 || tiles > 148) return 0;
  const int splits = std::min(148 / tiles, K / (4 * BK));
  return splits > 1 ? tiles * splits : 0;
}

int fp32_slots(Form form, int M, int N, int K) {
  const int slots = gemm_simt_slots(M, N, K);
  return strided_is_faster(form, ((M + FT - 1) / FT) * ((N + FT - 1) / FT), K, slots) ? slots : 0;
}

cudaError_t launch_gemm_simt(const GemmDesc& g, int* dev_status, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.a_dt != g.b_dt) return cudaErrorInvalidValue;
  dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM);
  const int tiles = (int)(grid.x * grid.y), slots = g.simt_scratch != nullptr && g.simt_counters != nullptr ? g.simt_slots : 0;
  const Form form = g.a_sk != 1 ? FORM_TN : (g.b_sk == 1 && g.b_sn != 1) ? FORM_NT : FORM_NN;
  if (!strided_is_faster(form, tiles, g.K, slots))
    if (cudaError_t e = try_ffma(g, dev_status, s); e != cudaErrorNotSupported) return e;
  const StridedSplit sp = strided_split(tiles, g.K, slots);
  const int k_per_split = sp.k_per_split;
  grid.z = (unsigned)sp.splits;
  if (g.a_dt == DT_F32 && g.c_dt == DT_F32) launch_k(gemm_simt_kernel<float, float>, dim3(grid), dim3(256), 0, s, g, k_per_split);
  else if (g.a_dt == DT_BF16 && g.c_dt == DT_BF16)
    launch_k(gemm_simt_kernel<__nv_bfloat16, __nv_bfloat16>, dim3(grid), dim3(256), 0, s, g, k_per_split);
  else if (g.a_dt == DT_BF16 && g.c_dt == DT_F32)
    launch_k(gemm_simt_kernel<__nv_bfloat16, float>, dim3(grid), dim3(256), 0, s, g, k_per_split);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace segk
