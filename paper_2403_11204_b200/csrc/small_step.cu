// The whole training step of a small fp32 segment in two launches (Section 2: forward through the
// segment's layers, loss against the intermediate labels of the samples' classes or, in the final
// segment, against the class labels, backward, update; Section 3: layers of 80, 60 and 47 units).
//
// A segment whose layers are at most kSmallMaxWidth wide is a chain of small dependent products: what bounds it
// is not arithmetic but how few SMs and warps a chain keeps busy, how many instructions a link issues and how long
// every link takes.
//   1. small_fwd_bwd_kernel: a cluster of C CTAs owns a block of C * R rows of the batch.  A wide first layer is
//      split over K: CTA r contracts its slice of the features, at most 132 of them, for all rows of the block and
//      sends every row's partial sums to the CTA that owns the row (bulk copies through distributed shared
//      memory).  From there each CTA carries its own R rows through the rest of the chain - the other forward
//      products, the loss with dZ of the last layer, the dgrad products - with everything it needs already on its
//      way into shared memory by a handful of bulk and tensor copies; each weight matrix is loaded once for both
//      directions.  A link of the chain takes one barrier: a warp owns a block of output columns and half of the
//      rows, its lanes split the contraction in four, and the four shares meet in a shuffle reduce-scatter (a fixed
//      order: bit-reproducible).  Activations, dZ and the staged input also go to global memory for the second
//      kernel.  Forward-only calls (seg_forward) run the same kernel up to the last layer's output.
//   2. small_wgrad_update_kernel: tiles of (all outputs) x NT inputs of dW_l = dZ_l^T [A_{l-1} | 1] for all layers
//      in one grid; a cluster of S CTAs splits the batch of one tile, tensor copies bring 64 rows of both operands
//      per stage, threads hold 8 x NT/8 register tiles, the partial tiles are combined as a reduce-scatter through
//      distributed shared memory (fixed order), and every CTA applies the optimizer to the rows it received.  The
//      column of ones, which yields the bias gradient, is kept in the padding of the activation buffers.
// Register tiles: a 16-byte shared-memory load costs the SM 2 cycles when neighbouring lanes share the address and 4
// when they do not (measured), so r rows x c columns cost 2 r + 4 c cycles of loads per r c cycles of FFMA issue and
// four k.
#include <cuda.h>
#include <limits.h>

#include <algorithm>
#include <atomic>
#include <new>
#include <type_traits>

#include "async_copy.cuh"
#include "common.cuh"

namespace segk {
namespace {

constexpr int SS_THREADS = 256, SS_WARPS = SS_THREADS / 32;
constexpr size_t SS_SMEM_LIMIT = 226 * 1024;                // dynamic shared memory; the static part is below 1 KiB

__host__ __device__ constexpr int up(int v, int m) { return (v + m - 1) / m * m; }
__host__ __device__ constexpr int pitch_of(int K) { return small_weight_pitch(K); }

// ---- first kernel -----------------------------------------------------------------------------------
// Shared-memory layout and work split of one launch (offsets in floats; filled by layout_small).
struct SmallPlan {
  int C, R;                    // CTAs per cluster, rows of the batch per CTA
  int ks;                      // features per CTA (C > 1) or the input width rounded up to 4 (C = 1): row pitch of the x tile
  int late;                    // chain weights share the x and W_0 tiles' memory and are loaded once the first layer is done
  int streamed;                // chain weights go through two slots instead of one slot each
  int forward_only;            // 1: forward pass that also stores every layer's output; 2: only the last layer's, into y
  int off_x, off_w0, off_send, off_recv, off_bias, off_tgt, off_dz[2];
  int off_act[kSmallMaxLayers + 1], off_slot[kSmallMaxLayers];
  int floats;
};

// Sum over the SL lane groups (consecutive groups of 32 / SL lanes) of v[0 .. V): afterwards a lane of group b holds, in
// v[0 .. H), the complete sums of the elements b * H + i, where H = VP / SL and VP = V rounded up to a multiple of SL.
template <int V, int SL>
__device__ __forceinline__ void reduce_scatter(float (&v)[(V + SL - 1) / SL * SL], int lane) {
  constexpr int VP = (V + SL - 1) / SL * SL;
#pragma unroll
  for (int len = VP, bit = 16; len > VP / SL; len /= 2, bit /= 2) {
    const bool hi = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < VP / 2; ++i) {
      if (i < len / 2) {
        const float give = hi ? v[i] : v[i + len / 2];
        const float keep = hi ? v[i + len / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, bit);
      }
    }
  }
}
// The element a lane holds after reduce_scatter, as (row, column index) of an RT x CT tile: element e = b * H + i.
template <int CT, int H, int SL>
__device__ __forceinline__ void element_of(int i, int b, int& row, int& col) {
  row = i / CT; col = i % CT;                               // compile-time alternatives, chosen by the lane group
#pragma unroll
  for (int s = 1; s < SL; ++s)
    if (b == s) { row = (s * H + i) / CT; col = (s * H + i) % CT; }
}

// v[r * CT + j] += sum over this lane's chunks (four k each) of A[r][4c ..] . W[n_j][4c ..]; A rows `pa` apart, wp[j] the row
// of column n_j.  The lanes' chunks are c0, c0 + step, ...; all lanes make the same number of rounds (a lane without a chunk
// left multiplies zeros by zeros: a value it does not own may be infinite), so that a warp never splits.
template <int RT, int CT, int VP>
__device__ __forceinline__ void dot_chunk(float (&v)[VP], const float* A, int pa, const float4 (&w)[CT], bool own = true) {
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    float4 a = lds4(A + r * pa);
    if (!own) a = make_float4(0.f, 0.f, 0.f, 0.f);
    // component by component: the CT sums in between hide the latency of a multiply-add on the same sum
#pragma unroll
    for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.x, w[j].x, v[r * CT + j]);
#pragma unroll
    for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.y, w[j].y, v[r * CT + j]);
#pragma unroll
    for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.z, w[j].z, v[r * CT + j]);
#pragma unroll
    for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.w, w[j].w, v[r * CT + j]);
  }
}
template <int RT, int CT, int VP>
__device__ __forceinline__ void dot_rows(float (&v)[VP], const float* A, int pa, const float* const (&wp)[CT], int c0, int chunks, int step) {
  const int full = chunks / step;
  int c = c0;
#pragma unroll 2
  for (int i = 0; i < full; ++i, c += step) {
    float4 w[CT];
#pragma unroll
    for (int j = 0; j < CT; ++j) w[j] = lds4(wp[j] + 4 * c);
    dot_chunk<RT, CT, VP>(v, A + 4 * c, pa, w);
  }
  if (full * step < chunks) {
    const bool ok = c < chunks;
    c = min(c, chunks - 1);
    float4 w[CT];
#pragma unroll
    for (int j = 0; j < CT; ++j) {
      w[j] = lds4(wp[j] + 4 * c);
      if (!ok) w[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    dot_chunk<RT, CT, VP>(v, A + 4 * c, pa, w, ok);
  }
}

// A forward link for R rows: every element n < N (rounded up to 4) of A W^T.  Warp = (half of the rows, block of 8 * CT columns),
// lane = (column, quarter of the contraction).  side(r, n) is what the element's epilogue needs from shared memory, fetched
// ahead of the arithmetic; emit(r, n, value, side) finishes the element.
template <int R, int CT, typename Side, typename Emit>
__device__ __forceinline__ void link_forward(const float* A, int pa, const float* W, int pw, int K, int N, const Side& side, const Emit& emit) {
  constexpr int RP = R >= 4 ? 2 : 1, RT = R / RP, V = RT * CT, VP = (V + 3) / 4 * 4, H = VP / 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sl = lane >> 3;
  const int rp = warp % RP, n0 = warp / RP * 8 * CT + (lane & 7);
  if (warp / RP * 8 * CT >= N) return;
  float v[VP];
#pragma unroll
  for (int i = 0; i < VP; ++i) v[i] = 0.f;
  const float* wp[CT];
#pragma unroll
  for (int j = 0; j < CT; ++j) wp[j] = W + min(n0 + 8 * j, N - 1) * pw;
  const int N4 = up(N, 4);
  int er[H], en[H];
  float2 es[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    int j;
    element_of<CT, H, 4>(i, sl, er[i], j);
    en[i] = n0 + 8 * j;
    if (er[i] >= RT || en[i] >= N4) en[i] = -1;
    er[i] += rp * RT;
    if (en[i] >= 0) es[i] = side(er[i], en[i]);
  }
  dot_rows<RT, CT, VP>(v, A + rp * RT * pa, pa, wp, sl, (K + 3) >> 2, 4);
  reduce_scatter<V, 4>(v, lane);
#pragma unroll
  for (int i = 0; i < H; ++i)
    if (en[i] >= 0) emit(er[i], en[i], v[i], es[i]);
}

// A dgrad link: every element k < K (rounded up to 4) of dZ W; lane = (CT consecutive k, quarter of n).
template <int R, int CT, typename Side, typename Emit>
__device__ __forceinline__ void link_dgrad(const float* dZ, int pz, const float* W, int pw, int N, int K, const Side& side, const Emit& emit) {
  constexpr int RP = R >= 4 ? 2 : 1, RT = R / RP, V = RT * CT, VP = (V + 3) / 4 * 4, H = VP / 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sl = lane >> 3;
  const int rp = warp % RP, k0 = warp / RP * 8 * CT + (lane & 7) * CT;
  if (warp / RP * 8 * CT >= K) return;
  float v[VP];
#pragma unroll
  for (int i = 0; i < VP; ++i) v[i] = 0.f;
  const float* wk = W + min(k0, pw - CT);                   // lanes beyond the row read its end and are not emitted
  const float* A = dZ + rp * RT * pz;
  const int K4 = up(K, 4);
  int er[H], ek[H];
  float2 es[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    int j;
    element_of<CT, H, 4>(i, sl, er[i], j);
    ek[i] = k0 + j;
    if (er[i] >= RT || ek[i] >= K4) ek[i] = -1;
    er[i] += rp * RT;
    if (ek[i] >= 0) es[i] = side(er[i], ek[i]);
  }
  // chunks of four n in rounds of four lane groups, as in dot_rows: in the last round, which also holds a chunk that N cuts,
  // what lies beyond N is zeros on both sides
  auto round = [&](int c, auto last) {
    const bool own = !decltype(last)::value || 4 * c < N;
    if (decltype(last)::value) c = min(c, (N - 1) >> 2);
    float w[4][CT];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool ok = !decltype(last)::value || (own && 4 * c + u < N);
      const float* row = wk + (decltype(last)::value ? min(4 * c + u, N - 1) : 4 * c + u) * pw;
      if constexpr (CT == 4) { const float4 t = lds4(row); w[u][0] = t.x; w[u][1] = t.y; w[u][2] = t.z; w[u][3] = t.w; }
      else if constexpr (CT == 2) { const float2 t = *reinterpret_cast<const float2*>(row); w[u][0] = t.x; w[u][1] = t.y; }
      else w[u][0] = row[0];
      if (!ok) {
#pragma unroll
        for (int j = 0; j < CT; ++j) w[u][j] = 0.f;
      }
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      float4 a = lds4(A + r * pz + 4 * c);                  // zero between N and the end of the chunk
      if (!own) a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.x, w[0][j], v[r * CT + j]);
#pragma unroll
      for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.y, w[1][j], v[r * CT + j]);
#pragma unroll
      for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.z, w[2][j], v[r * CT + j]);
#pragma unroll
      for (int j = 0; j < CT; ++j) v[r * CT + j] = fmaf(a.w, w[3][j], v[r * CT + j]);
    }
  };
  const int full = N >> 4;
#pragma unroll 2
  for (int i = 0; i < full; ++i) round(4 * i + sl, std::false_type{});
  if ((N & 15) != 0) round(4 * full + sl, std::true_type{});
  reduce_scatter<V, 4>(v, lane);
#pragma unroll
  for (int i = 0; i < H; ++i)
    if (ek[i] >= 0) emit(er[i], ek[i], v[i], es[i]);
}

// Columns per lane of a link with N columns: the smallest for which the warps cover them in one pass.
template <int R, typename F1, typename F2, typename F4>
__device__ __forceinline__ void by_width(int N, const F1& f1, const F2& f2, const F4& f4) {
  constexpr int blocks = SS_WARPS / (R >= 4 ? 2 : 1);
  if (N <= 8 * blocks) f1();
  else if (N <= 16 * blocks) f2();
  else f4();
}

// CT0: columns per lane in the split first layer (16 lanes along the columns); 0: the first layer is an ordinary link (C = 1).
template <int R, int CT0>
__global__ void __launch_bounds__(SS_THREADS, 1)
small_fwd_bwd_kernel(const __grid_constant__ SmallStep p, const float* __restrict__ x, const int32_t* __restrict__ cls,
                     const float* __restrict__ gather, float* loss_to, const __grid_constant__ SmallPlan q, float* y,
                     const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w0,
                     const __grid_constant__ CUtensorMap map_stage) {
  constexpr bool SPLIT = CT0 > 0;
  extern __shared__ __align__(128) float sm[];
  __shared__ uint64_t bars[3 + kSmallMaxLayers];            // x (and W_0) tiles; biases; received sums; weights of layer l
  __shared__ int cls_s[128];                                // classes of the cluster's rows (C * R <= 128)
  __shared__ float red[SS_WARPS];
  uint64_t *bar_x = bars, *bar_bias = bars + 1, *bar_recv = bars + 2, *bar_w = bars + 3;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, L = p.n_layers;
  const int C = SPLIT ? q.C : 1, rank = SPLIT ? (int)cluster_rank() : 0;
  const int RB = C * R;                                     // rows of the cluster's block
  const int rb0 = (int)blockIdx.x / C * RB;
  const int row0 = rb0 + rank * R, nv = max(0, min(R, p.batch - row0));
  const int nvb = min(RB, p.batch - rb0);                   // valid rows of the block
  constexpr int first = SPLIT ? 1 : 0;                      // first layer whose weights sit in a slot
  const int n0 = p.widths[0], NL = p.widths[L], N1 = p.widths[1];
  const bool train = !q.forward_only;
  const int k0 = SPLIT ? rank * q.ks : 0;                   // first feature of this CTA's slice
  float* xs = sm + q.off_x;
  float* bias_s = sm + q.off_bias;
  auto act_s = [&](int l) { return sm + q.off_act[l]; };
  auto slot = [&](int l) { return sm + q.off_slot[l]; };
  const float* xsrc = gather != nullptr ? gather : x;
  const bool x_tensor = small_input_by_tensor(x, gather, n0);       // the host built map_x under the same condition
  const bool stage = train && k0 < n0;
  const uint32_t recv_bytes = SPLIT ? (uint32_t)(SS_WARPS / C * R * up(N1, 4) * 4) : 0u;   // from each CTA of the cluster

  if (tid == 0) {
    for (int i = 0; i < 3 + kSmallMaxLayers; ++i) bar_init(bars + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async();
    if (SPLIT) bar_expect(bar_recv, (uint32_t)(C - 1) * recv_bytes);
  }
  __syncthreads();
  if (SPLIT) cluster_arrive_release();                      // "my barriers exist"; waited for before the first send
  pdl_wait();
  pdl_trigger();

  auto load_weight = [&](int l) {                           // by the issuing thread: the whole matrix, rows at their global pitch
    const uint32_t bytes = (uint32_t)p.widths[l + 1] * (uint32_t)p.ldw[l] * 4u;
    bar_expect(bar_w + l, bytes);
    bulk_load(slot(l), p.params + p.w_off[l], bytes, bar_w + l);
  };
  auto load_chain = [&]() {
    const int last = q.streamed ? min(L, first + 2) : L;
    for (int l = first; l < last; ++l) load_weight(l);
  };
  if (warp == 0) {
    if (elect_one()) {
      const uint32_t xb = x_tensor ? (uint32_t)(RB * q.ks * 4) : 0u, wb = SPLIT ? (uint32_t)(N1 * q.ks * 4) : 0u;
      bar_expect(bar_x, xb + wb);
      if (SPLIT) tensor_load(sm + q.off_w0, &map_w0, k0, 0, bar_x);
      if (x_tensor) tensor_load(xs, &map_x, k0, rb0, bar_x);
      uint32_t bb = 0;
      for (int l = 0; l < L; ++l) bb += (uint32_t)up(p.widths[l + 1], 4) * 4u;
      bar_expect(bar_bias, bb);
      for (int l = 0; l < L; ++l)
        bulk_load(bias_s + l * kSmallMaxWidth, p.params + p.b_off[l], (uint32_t)up(p.widths[l + 1], 4) * 4u, bar_bias);
      if (!q.late) load_chain();
    }
  }
  // classes of the block's rows, clamped (by the upper half of the threads: the first warp is issuing copies)
  const int crow = tid - SS_THREADS / 2;
  if (train && crow >= 0 && crow < RB) {
    int c = 0;
    if (crow < nvb) {
      c = cls[rb0 + crow];
      if (c < 0 || c >= p.n_classes) {
        if (rank == 0) atomicOr(p.dev_status, (int)DEV_BAD_CLASS);
        c = min(max(c, 0), p.n_classes - 1);
      }
      if (rank == 0) p.cls_stage[rb0 + crow] = c;
    }
    cls_s[crow] = c;
  }
  // step counter, Adam's bias corrections, where the loss goes
  if (train && blockIdx.x == 0 && tid == 32) {
    const unsigned long long step = *p.t + 1ull;
    *p.t = step;
    if (p.optimizer == SEG_ADAM) {                          // beta^t by repeated squaring, in double precision
      double r1 = 1.0, r2 = 1.0, b1 = (double)p.beta1, b2 = (double)p.beta2;
      for (unsigned long long e = step; e != 0; e >>= 1) {
        if (e & 1ull) { r1 *= b1; r2 *= b2; }
        b1 *= b1; b2 *= b2;
      }
      p.bc[0] = (float)(1.0 - r1);
      p.bc[1] = (float)(1.0 - r2);
    }
    *p.loss_dst = loss_to;
  }
  __syncthreads();                                          // cls_s
  if (!x_tensor) {
    // label rows gathered by class, or a batch whose rows are not whole 16-byte groups: plain loads, a row per warp.  The
    // column of ones is put down as well where it shares a 16-byte group with the last features: the staging store clips
    // whole groups only (the weights of that column are zero)
    for (int r = warp; r < RB; r += SS_WARPS) {
      const float* src = gather != nullptr ? gather + (int64_t)cls_s[r] * n0 : xsrc + (int64_t)(rb0 + min(r, nvb - 1)) * n0;
      for (int k = lane; k < q.ks; k += 32) xs[r * q.ks + k] = (r < nvb && k0 + k < n0) ? src[k0 + k] : (k0 + k == n0 && (n0 & 3) != 0 ? 1.f : 0.f);
    }
    fence_async();                                          // the staging store below reads them through the async proxy
    __syncthreads();
  }
  // the loss targets of the CTA's rows, in flight during the forward pass
  const int NL4 = up(NL, 4);
  float tgt_v[(R * kSmallMaxWidth + SS_THREADS - 1) / SS_THREADS];
  const bool want_targets = train && !p.is_final;
  if (want_targets) {
#pragma unroll
    for (int i = 0; i < (R * kSmallMaxWidth + SS_THREADS - 1) / SS_THREADS; ++i) {
      const int e = tid + i * SS_THREADS, r = e >> 7, n = e & 127;
      tgt_v[i] = (r < nv && n < NL) ? __ldg(p.sil + (int64_t)cls_s[rank * R + r] * NL + n) : 0.f;
    }
  }

  // output of layer l, element (r, n): bias, ReLU, shared and global memory; on the last layer of a non-final segment
  // also the loss  mean (a - t)^2  and  dZ = 2 (a - t) / (B N_P) * [a > 0]
  float lsum = 0.f;
  const float gscale = 2.0f / (float)((int64_t)p.batch * NL);
  float* dz_cur = sm + q.off_dz[0];
  const float* tgt_s = sm + q.off_tgt;
  struct Out { int N, pa; bool last, relu; float *a_s, *a_g, *y_g, *dz_g; int64_t ld, ld_y; };
  auto out_of = [&](int l) {                                // where layer l's output goes
    Out o;
    o.N = p.widths[l + 1]; o.pa = up(o.N, 4);
    o.last = l == L - 1; o.relu = !o.last || p.last_relu;
    o.a_s = act_s(l + 1);
    o.ld = p.ld_act[l + 1]; o.a_g = q.forward_only == 2 ? nullptr : p.act[l + 1] + (int64_t)row0 * o.ld;
    o.ld_y = o.N; o.y_g = (o.last && y != nullptr) ? y + (int64_t)row0 * o.N : nullptr;
    o.dz_g = p.dz[l] + (int64_t)row0 * o.ld;
    return o;
  };
  auto side_forward = [&](const Out& o, int l, int r, int n) {      // bias and, on the last layer, the loss target
    return make_float2(bias_s[l * kSmallMaxWidth + n], (o.last && want_targets) ? tgt_s[r * NL4 + n] : 0.f);
  };
  auto emit_forward = [&](const Out& o, int r, int n, float v, const float2& sd) {
    v += sd.x;
    if (o.relu) v = fmaxf(v, 0.f);
    if (n >= o.N) v = 0.f;
    const bool store = r < nv && n < o.N;
    if (store && o.a_g != nullptr) o.a_g[r * o.ld + n] = v;
    if (store && o.y_g != nullptr) o.y_g[r * o.ld_y + n] = v;
    if (o.last && want_targets) {
      float g = 0.f;
      if (store) {
        const float d = v - sd.y;
        lsum = fmaf(d, d, lsum);
        g = (p.last_relu && !(v > 0.f)) ? 0.f : d * gscale;
        o.dz_g[r * o.ld + n] = g;
      }
      dz_cur[r * kSmallMaxWidth + n] = g;
    } else {
      o.a_s[r * o.pa + n] = v;
    }
  };
  auto put_targets = [&]() {
    if (!want_targets) return;
#pragma unroll
    for (int i = 0; i < (R * kSmallMaxWidth + SS_THREADS - 1) / SS_THREADS; ++i) {
      const int e = tid + i * SS_THREADS, r = e >> 7, n = e & 127;
      if (r < R && n < NL4) sm[q.off_tgt + r * NL4 + n] = tgt_v[i];
    }
  };

  // ---- first layer, split over the cluster --------------------------------------------------------
  if constexpr (SPLIT) {
    const int N4 = up(N1, 4);
    constexpr int V = R * CT0, VP = (V + 1) / 2 * 2, H = VP / 2;
    const int KW = SS_WARPS / C, owner = warp % C, kw = warp / C;    // a warp contracts for one owner's rows; KW warps share its k
    float v[VP];
#pragma unroll
    for (int i = 0; i < VP; ++i) v[i] = 0.f;
    const float* wp[CT0];
#pragma unroll
    for (int j = 0; j < CT0; ++j) wp[j] = sm + q.off_w0 + min((lane & 15) + 16 * j, N1 - 1) * q.ks;
    bar_wait(bar_x, 0, p.dev_status);
    if (warp == 0 && stage) {                               // the staged input of the second kernel
      if (elect_one()) tensor_store(&map_stage, xs, k0, rb0);
    }
    const int kc = max(0, min(q.ks, n0 - k0) + 3) >> 2;     // 16-byte groups that hold features
    dot_rows<R, CT0, VP>(v, xs + owner * R * q.ks, q.ks, wp, 2 * kw + (lane >> 4), kc, 2 * KW);
    reduce_scatter<V, 2>(v, lane);
    // [owner][kw][row][column] in the send buffer, the own rows' share straight into the receive buffer
    float* out = owner == rank ? sm + q.off_recv + (size_t)(rank * KW + kw) * R * N4 : sm + q.off_send + (size_t)(owner * KW + kw) * R * N4;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      int r, j;
      element_of<CT0, H, 2>(i, lane >> 4, r, j);
      const int n = (lane & 15) + 16 * j;
      if (r < R && n < N4) out[r * N4 + n] = v[i];
    }
    fence_async();
    cluster_wait_acquire();                                 // every peer's receive barrier exists
    __syncthreads();
    if (warp == 0) {
      if (elect_one()) {
        for (int d = 1; d < C; ++d) {
          const int dest = (rank + d) & (C - 1);
          bulk_send(in_cta(smem_addr(sm + q.off_recv), (uint32_t)dest) + (uint32_t)rank * recv_bytes,
                    reinterpret_cast<const char*>(sm + q.off_send) + (size_t)dest * recv_bytes, recv_bytes,
                    in_cta(smem_addr(bar_recv), (uint32_t)dest));
        }
      }
      if (q.late) {                                         // the x and W_0 tiles are free once the staging store has read them
        if (stage) store_wait_source();
        __syncwarp();
        if (elect_one()) load_chain();
      }
    }
    put_targets();
    bar_wait(bar_bias, 0, p.dev_status);
    bar_wait(bar_recv, 0, p.dev_status);
    cluster_arrive_release();                               // "I have received everything"; waited for at the very end
    if (L == 1) __syncthreads();                            // the targets
    const int G = N4 / 4;
    const Out o = out_of(0);
    for (int e = tid; e < R * G; e += SS_THREADS) {
      const int r = e / G, g = e - r * G;
      const float* src = sm + q.off_recv + r * N4 + 4 * g;
      float4 s[SS_WARPS];
#pragma unroll
      for (int u = 0; u < SS_WARPS; ++u) s[u] = lds4(src + u * R * N4);
      float2 sd[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) sd[j] = side_forward(o, 0, r, 4 * g + j);
      float4 t = s[0];
#pragma unroll
      for (int u = 1; u < SS_WARPS; ++u) add4(t, s[u]);
      emit_forward(o, r, 4 * g, t.x, sd[0]); emit_forward(o, r, 4 * g + 1, t.y, sd[1]);
      emit_forward(o, r, 4 * g + 2, t.z, sd[2]); emit_forward(o, r, 4 * g + 3, t.w, sd[3]);
    }
  } else {
    put_targets();
    bar_wait(bar_bias, 0, p.dev_status);
    if (x_tensor) bar_wait(bar_x, 0, p.dev_status);
    if (warp == 0 && stage) {
      if (elect_one()) tensor_store(&map_stage, xs, 0, rb0);
    }
  }

  // ---- the forward chain ------------------------------------------------------------------------------
  for (int l = first; l < L; ++l) {
    const int K = p.widths[l], N = p.widths[l + 1];
    const float *A = l == 0 ? xs : act_s(l), *W = slot(l);
    const int pa = l == 0 ? q.ks : up(K, 4), pw = (int)p.ldw[l];
    const Out o = out_of(l);
    __syncthreads();                                        // the layer's input is complete
    bar_wait(bar_w + l, 0, p.dev_status);
    auto side = [&](int r, int n) { return side_forward(o, l, r, n); };
    auto emit = [&](int r, int n, float v, const float2& sd) { emit_forward(o, r, n, v, sd); };
    by_width<R>(N, [&]() { link_forward<R, 1>(A, pa, W, pw, K, N, side, emit); },
                [&]() { link_forward<R, 2>(A, pa, W, pw, K, N, side, emit); },
                [&]() { link_forward<R, 4>(A, pa, W, pw, K, N, side, emit); });
    if (q.streamed && l + 2 < L) {                          // two slots: refill this one for the layer after the next
      __syncthreads();
      if (warp == 0) { if (elect_one()) { fence_async(); load_weight(l + 2); } }
    }
  }
  if (!train) {
    if (SPLIT) cluster_wait_acquire();
    return;
  }
  __syncthreads();

  // ---- softmax cross-entropy of a final segment, 16 lanes per row:  dZ = (softmax(z) - onehot) / B -------
  if (p.is_final) {
    constexpr int M = kSmallMaxWidth / 16;
    const int r = tid >> 4, i0 = tid & 15;
    const float inv_b = 1.0f / (float)p.batch;
    const float* z = act_s(L) + min(r, R - 1) * NL4;
    float v[M], mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      v[j] = i0 + 16 * j < NL ? z[i0 + 16 * j] : -INFINITY;
      mx = fmaxf(mx, v[j]);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    float ex[M], se = 0.f, zc = 0.f;
    const int c = cls_s[rank * R + min(r, R - 1)];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      ex[j] = 0.f;
      if (16 * j < NL) ex[j] = i0 + 16 * j < NL ? expf(v[j] - mx) : 0.f;
      se += ex[j];
      if (i0 + 16 * j == c) zc = v[j];
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) { se += __shfl_xor_sync(0xFFFFFFFFu, se, o); zc += __shfl_xor_sync(0xFFFFFFFFu, zc, o); }
    const float inv_se = 1.0f / se;
    if (r < R) {
#pragma unroll
      for (int j = 0; j < M; ++j) {
        const int i = i0 + 16 * j;
        if (i < NL4) {
          float g = 0.f;
          if (r < nv && i < NL) {
            g = (ex[j] * inv_se - (i == c ? 1.f : 0.f)) * inv_b;
            if (p.last_relu && !(v[j] > 0.f)) g = 0.f;
            p.dz[L - 1][(int64_t)(row0 + r) * p.ld_act[L] + i] = g;
          }
          dz_cur[r * kSmallMaxWidth + i] = g;
        }
      }
      if (i0 == 0 && r < nv) lsum = logf(se) - (zc - mx);
    }
  }
  lsum = warp_sum(lsum);
  if (lane == 0) red[warp] = lsum;
  __syncthreads();
  if (tid == 0) {                                           // the CTA's share of the batch loss; the second kernel adds them up
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < SS_WARPS; ++w) t += red[w];
    p.loss_partials[blockIdx.x] = t;
  }

  // ---- dgrad chain:  dZ_{l-1} = (dZ_l W_l) * [A_{l-1} > 0] -----------------------------------------------
  for (int l = L - 1; l >= 1; --l) {
    const int K = p.widths[l], K4 = up(K, 4), N = p.widths[l + 1], pw = (int)p.ldw[l];
    if (q.streamed && l + 2 < L) bar_wait(bar_w + l, 1, p.dev_status);   // loaded a second time
    float* dz_next = dz_cur == sm + q.off_dz[0] ? sm + q.off_dz[1] : sm + q.off_dz[0];
    const float *al = act_s(l), *W = slot(l);
    const int64_t ld = p.ld_act[l];
    float* dz_g = p.dz[l - 1] + (int64_t)row0 * ld;
    auto side = [&](int r, int k) { return make_float2(al[r * K4 + k], 0.f); };
    auto emit = [&](int r, int k, float v, const float2& sd) {
      if (!(sd.x > 0.f)) v = 0.f;                           // columns beyond the width hold 0: masked as well
      dz_next[r * kSmallMaxWidth + k] = v;
      if (r < nv && k < K) dz_g[r * ld + k] = v;
    };
    by_width<R>(K, [&]() { link_dgrad<R, 1>(dz_cur, kSmallMaxWidth, W, pw, N, K, side, emit); },
                [&]() { link_dgrad<R, 2>(dz_cur, kSmallMaxWidth, W, pw, N, K, side, emit); },
                [&]() { link_dgrad<R, 4>(dz_cur, kSmallMaxWidth, W, pw, N, K, side, emit); });
    if (l > 1) __syncthreads();
    if (q.streamed && l - 2 >= 1) {
      if (warp == 0) { if (elect_one()) { fence_async(); load_weight(l - 2); } }
    }
    dz_cur = dz_next;
  }
  if (warp == 0 && stage) store_wait_all();                 // (a no-op for the threads that issued no store)
  if (SPLIT) cluster_wait_acquire();                        // the peers have read what this CTA sent
}

// ---- weight gradients of all layers, bias gradients and the update ---------------------------------
constexpr int WBOX = 32, WK = 64, W_STAGES = 3;             // batch rows per tensor copy and per stage, stages at most

__host__ __device__ inline int wgrad_tiles(int in, int nt) { return (in + 1 + nt - 1) / nt; }

// Floats of dynamic shared memory: the operand ring, which also holds the thread groups' partial tiles, and the received slices.
__host__ __device__ inline int wgrad_ring_floats(int mt, int nt, int stages) {
  const int ring = stages * WK * (mt + nt), parts = (SS_THREADS / mt) * mt * nt;
  return ring > parts ? ring : parts;
}

template <int OPT, int NT>
__global__ void __launch_bounds__(SS_THREADS, 2)
small_wgrad_update_kernel(const __grid_constant__ SmallStep p, const __grid_constant__ SmallMaps maps, int S, int rows_per_cta,
                          int n_partials, int stages) {
  constexpr int CN = NT / 8;                                // columns per thread
  constexpr int CPR = NT / 4;                               // 16-byte groups per row of B
  extern __shared__ __align__(128) float sm[];
  __shared__ uint64_t full[W_STAGES], empty[W_STAGES];
  __shared__ float red[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = S > 1 ? (int)cluster_rank() : 0;
  int l = 0, t = (int)blockIdx.x / S;
  for (; l < p.n_layers - 1; ++l) {
    const int nt = wgrad_tiles(p.widths[l], NT);
    if (t < nt) break;
    t -= nt;
  }
  const int in = p.widths[l], out = p.widths[l + 1], MT = up(out, 8), n0 = t * NT;
  const int items = MT;                                     // (MT / 8) x 8 threads hold the tile
  const int G = SS_THREADS / items, grp = tid / items, it = tid - grp * items;
  const int tx = it & 7, ty = it >> 3;
  const int k_begin = rank * rows_per_cta, k_end = min(p.batch, k_begin + rows_per_cta);
  const int rows = max(0, k_end - k_begin), steps = (rows + WK - 1) / WK;
  float* ringA = sm;                                        // [stage][WK][MT]
  float* ringB = sm + stages * WK * MT;                     // [stage][WK][NT]
  float* recv = sm + wgrad_ring_floats(MT, NT, stages);     // [source CTA][MT / S rows][NT]
  const CUtensorMap* map_a = maps.m + 3 * l;                // (m = o, k = b) at dz[b * ld + o]
  const CUtensorMap* map_b = map_a + (NT == 32 ? 1 : 2);    // (k = b, n = i) at act[b * ld + i]; column `in` holds ones
  const uint32_t box_bytes = (uint32_t)(WBOX * (MT + NT) * 4);
  auto load = [&](int step) {                               // by the issuing thread
    const int s = step % stages, boxes = min(WK / WBOX, (rows - step * WK + WBOX - 1) / WBOX);
    bar_expect(full + s, (uint32_t)boxes * box_bytes);
    for (int b = 0; b < boxes; ++b) {
      const int r = b * WBOX;
      tensor_load(ringA + (s * WK + r) * MT, map_a, 0, k_begin + step * WK + r, full + s);
      tensor_load(ringB + (s * WK + r) * NT, map_b, n0, k_begin + step * WK + r, full + s);
    }
  };
  if (tid == 0) {
    for (int i = 0; i < stages; ++i) { bar_init(full + i, 1); bar_init(empty + i, SS_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async();
  }
  __syncthreads();
  if (S > 1) cluster_arrive_release();
  pdl_wait();
  pdl_trigger();
  if (warp == 0) {
    if (elect_one())
      for (int s = 0; s < min(stages, steps); ++s) load(s);
  }
  float lpart = 0.f;                                        // the batch loss: the first block adds the first kernel's shares
  if (blockIdx.x == 0)
    for (int i = tid; i < n_partials; i += SS_THREADS) lpart += p.loss_partials[i];

  uint64_t acc2[4][CN];                                     // rows 2i and 2i + 1
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < CN; ++j) acc2[i][j] = 0;
  for (int step = 0; step < steps; ++step) {
    const int s = step % stages;
    bar_wait(full + s, (uint32_t)(step / stages) & 1u, p.dev_status);
    if (grp < G) {
      const int kmax = min(WK, rows - step * WK);           // rows beyond this CTA's share are never multiplied
      const float* a_s = ringA + (s * WK + grp) * MT + ty * 8;
      const float* b_s = ringB + (s * WK + grp) * NT + (CN == 2 ? 2 : 4) * tx;
#pragma unroll 4
      for (int k = grp; k < kmax; k += G, a_s += G * MT, b_s += G * NT) {
        const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(a_s), a1 = *reinterpret_cast<const ulonglong2*>(a_s + 4);
        const uint64_t a[4] = {a0.x, a0.y, a1.x, a1.y};
        float b[CN];
        if constexpr (CN == 4) {
          const float4 b0 = lds4(b_s);
          b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w;
        } else {
          const float2 b0 = *reinterpret_cast<const float2*>(b_s);
          b[0] = b0.x; b[1] = b0.y;
        }
#pragma unroll
        for (int j = 0; j < CN; ++j) {
          uint64_t bb;
          asm("mov.b64 %0, {%1, %1};" : "=l"(bb) : "f"(b[j]));
#pragma unroll
          for (int i = 0; i < 4; ++i) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[i][j]) : "l"(a[i]), "l"(bb));
        }
      }
    }
    if (step + stages < steps) {                            // the stage is needed again
      __syncwarp();
      if (lane == 0) bar_arrive(empty + s);
      if (warp == 0) {
        if (elect_one()) {
          bar_wait(empty + s, (uint32_t)(step / stages) & 1u, p.dev_status);
          load(step + stages);
        }
      }
    }
  }
  float acc[8][CN];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < CN; ++j)
      asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * i][j]), "=f"(acc[2 * i + 1][j]) : "l"(acc2[i][j]));
  __syncthreads();                                          // the ring is free: partial tiles [group][MT][NT] take its place
  if (grp < G) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float* d = sm + (grp * MT + ty * 8 + i) * NT;
      if constexpr (CN == 4) {
        *reinterpret_cast<float4*>(d + 4 * tx) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      } else {
        *reinterpret_cast<float2*>(d + 2 * tx) = make_float2(acc[i][0], acc[i][1]);
      }
    }
  }
  const int slice = MT / S;                                 // rows each CTA of the cluster ends up with
  // four consecutive columns of one row per thread and pass.  A group that lies wholly inside the weight matrix moves with
  // 16-byte accesses; the ragged group at the matrix edge, which also carries the bias element, goes element by element.
  struct Item { int64_t e[4]; bool wide, any; float w[4], m[4], v[4]; };
  auto fetch = [&](int e, Item& q) {
    const int o = rank * slice + e / CPR, c0 = n0 + 4 * (e % CPR);
    q.any = e < slice * CPR && o < out && c0 <= in;
    q.wide = q.any && c0 + 3 < in;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + j;
      q.e[j] = !q.any || c > in ? -1 : (c < in ? p.w_off[l] + (int64_t)o * p.ldw[l] + c : p.b_off[l] + o);
      q.w[j] = q.m[j] = q.v[j] = 0.f;
    }
    if (q.wide) {
      const float4 a = *reinterpret_cast<const float4*>(p.params + q.e[0]);
      q.w[0] = a.x; q.w[1] = a.y; q.w[2] = a.z; q.w[3] = a.w;
      if constexpr (OPT != SEG_SGD) {
        const float4 b = *reinterpret_cast<const float4*>(p.s1 + q.e[0]);
        q.m[0] = b.x; q.m[1] = b.y; q.m[2] = b.z; q.m[3] = b.w;
      }
      if constexpr (OPT == SEG_ADAM) {
        const float4 b = *reinterpret_cast<const float4*>(p.s2 + q.e[0]);
        q.v[0] = b.x; q.v[1] = b.y; q.v[2] = b.z; q.v[3] = b.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (q.e[j] < 0) continue;
        q.w[j] = p.params[q.e[j]];
        if constexpr (OPT != SEG_SGD) q.m[j] = p.s1[q.e[j]];
        if constexpr (OPT == SEG_ADAM) q.v[j] = p.s2[q.e[j]];
      }
    }
  };
  Item q;
  fetch(tid, q);                                            // in flight during the exchange
  float inv_bc1 = 1.0f, inv_bc2 = 1.0f;
  if constexpr (OPT == SEG_ADAM) { inv_bc1 = 1.0f / __ldg(p.bc); inv_bc2 = 1.0f / __ldg(p.bc + 1); }
  if (S > 1) cluster_wait_acquire();                        // every peer has started: its shared memory may be written
  __syncthreads();
  const uint32_t inv_slice = (65536u + (uint32_t)slice - 1u) / (uint32_t)slice;     // row / slice for row < 128, exactly
  for (int e0 = tid; e0 < MT * CPR; e0 += 4 * SS_THREADS) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * SS_THREADS;
      if (e < MT * CPR) {
        v[u] = lds4(sm + 4 * e);
        for (int g = 1; g < G; ++g) add4(v[u], lds4(sm + g * MT * NT + 4 * e));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * SS_THREADS;
      if (e < MT * CPR) {
        const int row = e / CPR, c = e % CPR, owner = (int)(((uint32_t)row * inv_slice) >> 16);
        const uint32_t off = 4u * (uint32_t)((rank * slice + row - owner * slice) * NT + 4 * c);
        if (S > 1) store_cluster4(in_cta(smem_addr(recv), (uint32_t)owner) + off, v[u]);
        else *reinterpret_cast<float4*>(recv + off / 4) = v[u];
      }
    }
  }
  if (S > 1) { cluster_arrive_release(); cluster_wait_acquire(); } else __syncthreads();
  for (int e = tid; e < slice * CPR; e += SS_THREADS) {
    if (e != tid) fetch(e, q);
    if (!q.any) continue;
    float4 g4 = lds4(recv + 4 * e);
    for (int s = 1; s < S; ++s) add4(g4, lds4(recv + s * slice * NT + 4 * e));
    const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (q.e[j] >= 0) opt_step<OPT>(q.w[j], gv[j], q.m[j], q.v[j], p, inv_bc1, inv_bc2);
    if (q.wide) {
      *reinterpret_cast<float4*>(p.grads + q.e[0]) = g4;
      if constexpr (OPT != SEG_SGD) *reinterpret_cast<float4*>(p.s1 + q.e[0]) = make_float4(q.m[0], q.m[1], q.m[2], q.m[3]);
      if constexpr (OPT == SEG_ADAM) *reinterpret_cast<float4*>(p.s2 + q.e[0]) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
      *reinterpret_cast<float4*>(p.params + q.e[0]) = make_float4(q.w[0], q.w[1], q.w[2], q.w[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (q.e[j] < 0) continue;
        p.grads[q.e[j]] = gv[j];
        if constexpr (OPT != SEG_SGD) p.s1[q.e[j]] = q.m[j];
        if constexpr (OPT == SEG_ADAM) p.s2[q.e[j]] = q.v[j];
        p.params[q.e[j]] = q.w[j];
      }
    }
  }
  if (blockIdx.x == 0) {
    const float total = block_sum(lpart, red);
    if (tid == 0) {
      const int NL = p.widths[p.n_layers];
      const float scale = p.is_final ? 1.0f / (float)p.batch : 1.0f / (float)((int64_t)p.batch * NL);
      float* dst = *p.loss_dst;
      if (dst) *dst = total * scale;
    }
  }
}

__global__ void small_ones_kernel(float* a, int64_t ld, int col, int rows) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += gridDim.x * blockDim.x) a[(int64_t)i * ld + col] = 1.0f;
}

// ---- host side -------------------------------------------------------------------------------------
// Clusters of C CTAs the GPU runs at once with one CTA per SM (cudaOccupancyMaxActiveClusters on a B200: 148, 74, 33, 15 - a
// cluster lives inside one GPC, and what a GPC has beyond a multiple of C stays idle).
int resident_clusters(int C) { return C == 1 ? 148 : C == 2 ? 74 : C == 4 ? 33 : 15; }
// The same with two CTAs per SM.
int resident_clusters_2(int C) { return C == 1 ? 296 : C == 2 ? 148 : C == 4 ? 71 : 33; }

int cluster_of(int n0) { return n0 <= 128 ? 1 : n0 <= 256 ? 2 : n0 <= 512 ? 4 : 8; }   // CTAs per cluster: at most 128 features each

constexpr int kRowChoices[] = {1, 2, 4, 6, 8, 10, 12, 16};
int split_columns(int N1) { return N1 <= 32 ? 2 : N1 <= 64 ? 4 : N1 <= 80 ? 5 : 8; }   // columns per lane in the split first layer

// Lays out one launch with R rows per CTA; false when it does not fit into shared memory.
bool layout_small(const SmallStep& p, int R, SmallPlan* q) {
  const int L = p.n_layers, n0 = p.widths[0], N1 = p.widths[1];
  q->R = R;
  q->C = cluster_of(n0);
  const int first = q->C > 1 ? 1 : 0, n_slots = L - first;
  q->ks = q->C > 1 ? pitch_of((n0 + q->C - 1) / q->C) : up(n0, 4);
  int slot_max = 0, slot_sum = 0;
  for (int l = first; l < L; ++l) {
    const int f = up(p.widths[l + 1] * (int)p.ldw[l], 32);
    slot_max = std::max(slot_max, f); slot_sum += f;
  }
  const int t_x = up(q->C * R * q->ks, 32), t_w = q->C > 1 ? up(N1 * q->ks, 32) : 0;
  const int exch = q->C > 1 ? SS_WARPS * R * up(N1, 4) : 0;         // sums sent / received: one share per warp and row
  for (int mode = 0; mode < 4; ++mode) {                            // own slots, two slots; the same in the first layer's tiles
    q->late = mode >= 2; q->streamed = mode & 1;
    if (q->streamed && n_slots <= 2) continue;
    if (q->late && q->C == 1) continue;
    const int slots = q->streamed ? 2 * slot_max : slot_sum;
    q->off_x = 0; q->off_w0 = t_x;
    int so = q->late ? 0 : t_x + t_w;
    int off = q->late ? std::max(t_x + t_w, slots) : t_x + t_w + slots;
    for (int l = first; l < L; ++l) {
      if (q->streamed) q->off_slot[l] = so + ((l - first) & 1) * slot_max;
      else { q->off_slot[l] = so; so += up(p.widths[l + 1] * (int)p.ldw[l], 32); }
    }
    q->off_send = off; off += exch;
    q->off_recv = off; off += exch;
    for (int l = 1; l <= L; ++l) { q->off_act[l] = off; off += R * up(p.widths[l], 4); }
    for (int i = 0; i < 2; ++i) { q->off_dz[i] = off; off += R * kSmallMaxWidth; }
    q->off_bias = off; off += L * kSmallMaxWidth;
    q->off_tgt = off; off += p.is_final ? 0 : R * up(p.widths[L], 4);
    q->floats = off;
    if ((size_t)off * sizeof(float) <= SS_SMEM_LIMIT) return true;
  }
  return false;
}

// Rows per CTA: the split with the smallest estimate of waves x time of a CTA.  A link costs its fixed latency, the pass
// over the weights in shared memory, and arithmetic in proportion to the rows; the first layer's share grows with the
// cluster's rows (cycles, fitted to clock stamps inside the kernel).
bool plan_small(const SmallStep& p, SmallPlan* best) {
  double best_t = 1e30;
  for (int R : kRowChoices) {
    SmallPlan q{};
    if (!layout_small(p, R, &q)) continue;
    const int clusters = (p.batch + q.C * R - 1) / (q.C * R);
    const int waves = (clusters + resident_clusters(q.C) - 1) / resident_clusters(q.C);
    double links = 0;
    for (int l = q.C > 1 ? 1 : 0; l < p.n_layers; ++l)
      links += (l > 0 ? 2 : 1) * (600.0 + p.widths[l] * p.widths[l + 1] * (0.04 + 0.012 * R));
    const double t0 = q.C > 1 ? 2500.0 + (double)up(q.C * R, 8) * p.widths[1] * q.ks / 90.0 : 0.0;
    const double t = waves * (3000.0 + t0 + links);
    if (t < best_t) { best_t = t; *best = q; }
  }
  return best_t < 1e30;
}

int chain_grid(const SmallStep& p, const SmallPlan& q) { return (p.batch + q.C * q.R - 1) / (q.C * q.R) * q.C; }

template <typename Kern>
cudaError_t launch_clustered(Kern kern, int grid, int cluster, size_t smem, cudaStream_t s, void** args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(SS_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (g_use_pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster; attr[n].val.clusterDim.y = 1; attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr; cfg.numAttrs = n;
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kern), args);
}

// Allows a kernel its largest dynamic shared memory, once per device.
cudaError_t allow_smem(const void* kern, size_t bytes, std::atomic<bool>* flags) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (flags[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) flags[dev].store(true, std::memory_order_release);
  return e;
}

struct ChainArgs {
  SmallStep p; SmallPlan q;
  const float* x; const int32_t* cls; const float* gather; float* loss_to; float* y;
  CUtensorMap map_x, map_w0, map_stage;
};

}  // namespace

// Everything about a launch that depends on the batch size only: split, shared-memory layout, tensor maps of the handle's
// own buffers, tiles of the second kernel.
struct SmallPrepared {
  ChainArgs a;
  SmallMaps maps;
  int nt, S, tiles, rows, stages;
  size_t wgrad_smem;
};

namespace {

template <int R, int CT0>
cudaError_t launch_chain(ChainArgs& a, cudaStream_t s) {
  static std::atomic<bool> allowed[64];
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(small_fwd_bwd_kernel<R, CT0>), SS_SMEM_LIMIT, allowed);
  if (e != cudaSuccess) return e;
  void* args[] = {&a.p, &a.x, &a.cls, &a.gather, &a.loss_to, &a.q, &a.y, &a.map_x, &a.map_w0, &a.map_stage};
  return launch_clustered(small_fwd_bwd_kernel<R, CT0>, chain_grid(a.p, a.q), a.q.C, (size_t)a.q.floats * sizeof(float), s, args);
}

template <int R>
cudaError_t launch_chain(ChainArgs& a, cudaStream_t s) {
  if (a.q.C == 1) return launch_chain<R, 0>(a, s);
  switch (split_columns(a.p.widths[1])) {
    case 2: return launch_chain<R, 2>(a, s);
    case 4: return launch_chain<R, 4>(a, s);
    case 5: return launch_chain<R, 5>(a, s);
    default: return launch_chain<R, 8>(a, s);
  }
}

cudaError_t launch_chain(ChainArgs& a, cudaStream_t s) {
  const SmallStep& p = a.p;
  const SmallPlan& q = a.q;
  if (small_input_by_tensor(a.x, a.gather, p.widths[0]) &&
      !make_map_f32(&a.map_x, a.x, (uint64_t)p.widths[0], (uint64_t)p.batch, (uint64_t)p.widths[0] * 4, (uint32_t)q.ks, (uint32_t)(q.C * q.R)))
    return cudaErrorInvalidValue;
  switch (q.R) {
    case 1: return launch_chain<1>(a, s);
    case 2: return launch_chain<2>(a, s);
    case 4: return launch_chain<4>(a, s);
    case 6: return launch_chain<6>(a, s);
    case 8: return launch_chain<8>(a, s);
    case 10: return launch_chain<10>(a, s);
    case 12: return launch_chain<12>(a, s);
    case 16: return launch_chain<16>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

size_t wgrad_smem_bytes(const SmallStep& p, int nt, int stages) {
  size_t b = 0;
  for (int l = 1; l <= p.n_layers; ++l) {
    const int mt = up(p.widths[l], 8);
    b = std::max(b, (size_t)(wgrad_ring_floats(mt, nt, stages) + mt * nt) * sizeof(float));
  }
  return b;
}

// Tile width and batch split of the second kernel with the smallest estimate: a wave of CTAs costs its fixed latencies, its
// arithmetic at the rate the register tile reaches (8 x 2 bound by shared-memory loads, 8 x 4 by FFMA issue) and the exchange.
// The constants follow from timing all splits of six networks at 64 to 1410 rows: at most 6 % off the best of them, most
// exactly it.  Eight warps per SM are bound by latency, so a grid of two CTAs per SM wins although each redoes the fixed part:
// 784-80-60 at 1410 rows 28.2 us per step with 32 columns x 8 CTAs (224 CTAs), 29.8 with 64 x 8 (120), which also lost
// everywhere else and is not built.
void plan_wgrad(SmallPrepared* w) {
  const SmallStep& p = w->a.p;
  double best_t = 1e30;
  for (int nt : {32, 16}) {
    int tiles = 0, mt = 8;
    for (int l = 0; l < p.n_layers; ++l) { tiles += wgrad_tiles(p.widths[l], nt); mt = std::max(mt, up(p.widths[l + 1], 8)); }
    for (int S : {1, 2, 4, 8}) {
      if (S > 1 && p.batch < 8 * S) continue;
      const int rows = (p.batch + S - 1) / S;
      const bool pairs = tiles > resident_clusters(S);               // two CTAs share an SM
      const int waves = pairs ? (tiles + resident_clusters_2(S) - 1) / resident_clusters_2(S) : 1;
      const double rate = pairs ? (nt == 32 ? 61.5 : 50.5) : (nt == 32 ? 87.0 : 65.0);   // multiply-adds per cycle and CTA
      const double exchange = S == 1 ? 500.0 : S == 2 ? 450.0 : S == 4 ? 950.0 : 1500.0;
      const double t = exchange + waves * (700.0 + rows * (double)mt * nt / rate + mt * nt / 12.0 * (1.0 + 1.0 / S));
      if (t < best_t) { best_t = t; w->nt = nt; w->S = S; w->tiles = tiles; w->rows = rows; }
    }
  }
  // all of a CTA's rows in flight at once where the stages allow it; two CTAs on an SM where the grid needs them
  w->stages = std::max(1, std::min((w->rows + WK - 1) / WK, W_STAGES));
  if (w->tiles > resident_clusters(w->S))
    while (w->stages > 2 && wgrad_smem_bytes(p, w->nt, w->stages) > 112 * 1024) --w->stages;
  w->wgrad_smem = wgrad_smem_bytes(p, w->nt, w->stages);
}

template <int OPT, int NT>
cudaError_t launch_wgrad(SmallPrepared& w, cudaStream_t s) {
  static std::atomic<bool> allowed[64];
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(small_wgrad_update_kernel<OPT, NT>), SS_SMEM_LIMIT, allowed);
  if (e != cudaSuccess) return e;
  int n_partials = chain_grid(w.a.p, w.a.q);
  void* args[] = {&w.a.p, &w.maps, &w.S, &w.rows, &n_partials, &w.stages};
  return launch_clustered(small_wgrad_update_kernel<OPT, NT>, w.tiles * w.S, w.S, w.wgrad_smem, s, args);
}

template <int OPT>
cudaError_t launch_wgrad(SmallPrepared& w, cudaStream_t s) {
  if (w.nt == 32) return launch_wgrad<OPT, 32>(w, s);
  return launch_wgrad<OPT, 16>(w, s);
}

}  // namespace

bool small_step_supported(int n_layers, const int* widths) {
  if (n_layers < 1 || n_layers > kSmallMaxLayers || widths[0] > kSmallMaxInput) return false;
  for (int l = 1; l <= n_layers; ++l)
    if (widths[l] > kSmallMaxWidth) return false;
  return true;
}

SmallPrepared* small_prepare(const SmallStep& p, const SmallMaps& maps) {
  SmallPrepared* w = new (std::nothrow) SmallPrepared();
  if (!w) return nullptr;
  w->maps = maps;
  ChainArgs& a = w->a;
  a.p = p;
  bool ok = plan_small(p, &a.q);
  if (ok) {
    const SmallPlan& q = a.q;
    // x_stage: clipped to the input width and the batch, so that the column of ones behind the width stays
    ok = make_map_f32(&a.map_stage, p.act[0], (uint64_t)p.widths[0], (uint64_t)p.batch, (uint64_t)p.ld_act[0] * 4, (uint32_t)q.ks,
                      (uint32_t)(q.C * q.R));
    a.map_x = a.map_w0 = a.map_stage;
    if (ok && q.C > 1)
      ok = make_map_f32(&a.map_w0, p.params + p.w_off[0], (uint64_t)p.widths[0], (uint64_t)p.widths[1], (uint64_t)p.ldw[0] * 4,
                        (uint32_t)q.ks, (uint32_t)p.widths[1]);
  }
  if (!ok) { delete w; return nullptr; }
  return w;
}

void small_release(SmallPrepared* w) { delete w; }

bool small_can_train(const SmallPrepared& w) { return chain_grid(w.a.p, w.a.q) <= loss_max_partials(); }

// A batch runs in waves of 16 rows per CTA (1920 rows with clusters of 8, 2368 with one CTA per block of rows); past a few of
// them the layer-by-layer products, whose tiles share a layer's weights among 64 rows, catch up.  Rows that cannot be loaded by a
// tensor copy (by_tensor false: plain loads of a warp per row) make a wave longer.  us, this path / layer by layer:
//   forward   784-80-60 at 1536 / 3072 / 8192 rows 17/24 32/36 79/63, 784-128-128-64 31/28 55/42 127/78, 60-60-60-47 7/17 12/18 30/20;
//             without tensor copies 31/40 60/56 148/85, 45/38 80/62 187/101, 8/19 14/20 34/24
//   training  784-80-60 at 2048 / 8192 / 16384 rows 46/56 143/148 272/298, 784-128-128-64 at 2048 / 4096 / 8192 75/75 136/113 241/204,
//             300-81-33 34/43 66/60 125/98, 60-60-60-47 22/47 38/59 72/81; without tensor copies 784-80-60 62/60 103/92 213/160,
//             784-128-128-64 91/78 169/119 323/218, 300-81-33 39/44 77/62 147/102, 60-60-60-47 23/47 40/60 75/82
int small_max_rows(const SmallStep& p, bool train, bool by_tensor) {
  const int C = cluster_of(p.widths[0]), wave = 16 * C * resident_clusters(C);
  if (!train) return by_tensor ? (C == 1 ? 2 * wave : wave) : (C == 8 ? wave / 2 : wave);
  if (C == 1 || (by_tensor && (C == 2 || (C == 8 && p.widths[1] <= 96)))) return INT_MAX;   // (one loss partial per CTA: 16384 rows)
  return by_tensor ? 2 * wave : C == 2 ? 3 * wave : wave;
}
// A whole data set in one launch takes many waves at a constant time per row, which the layer-by-layer pass undercuts in batches
// of this many rows (784-80-60: 8.7 ns per row against 8.8 in batches of 4096; 60-60-60-47: 3.4 against 4.4 and, at 8192, 2.4;
// without tensor copies 784-80-60 17.7 against 14 in batches of 2048).
int small_dataset_batch(const SmallStep& p, bool by_tensor) {
  const int C = cluster_of(p.widths[0]);
  return C == 1 ? 8192 : by_tensor || C < 8 ? 4096 : 2048;
}

bool small_step_maps(const SmallStep& p, int max_batch, SmallMaps* maps) {
  for (int l = 0; l < p.n_layers; ++l) {
    CUtensorMap* m = maps->m + 3 * l;
    const uint32_t mt = (uint32_t)up(p.widths[l + 1], 8);
    if (!make_map_f32(m, p.dz[l], mt, (uint64_t)max_batch, (uint64_t)p.ld_act[l + 1] * 4, mt, WBOX)) return false;
    const uint32_t nts[2] = {32, 16};
    for (int i = 0; i < 2; ++i)
      if (!make_map_f32(m + 1 + i, p.act[l], (uint64_t)p.widths[l] + 1, (uint64_t)max_batch, (uint64_t)p.ld_act[l] * 4, nts[i], WBOX)) return false;
  }
  return true;
}

cudaError_t launch_small_ones(float* act, int64_t ld, int col, int rows, cudaStream_t s) {
  small_ones_kernel<<<std::min((rows + 255) / 256, 148), 256, 0, s>>>(act, ld, col, rows);
  return cudaGetLastError();
}

cudaError_t launch_small_fwd_bwd(SmallPrepared& w, const float* x, const int32_t* cls, const float* gather, float* loss_to,
                                 cudaStream_t s) {
  ChainArgs& a = w.a;
  a.x = x; a.cls = cls; a.gather = gather; a.loss_to = loss_to; a.y = nullptr;
  a.q.forward_only = 0;
  return launch_chain(a, s);
}

cudaError_t launch_small_forward(SmallPrepared& w, const float* x, float* y, bool keep, cudaStream_t s) {
  ChainArgs& a = w.a;
  a.x = x; a.cls = nullptr; a.gather = nullptr; a.loss_to = nullptr; a.y = y;
  a.q.forward_only = keep ? 1 : 2;
  return launch_chain(a, s);
}

cudaError_t launch_small_wgrad_update(SmallPrepared& w, cudaStream_t s) {
  if (w.tiles == 0) plan_wgrad(&w);              // the first training step of this batch size
  switch (w.a.p.optimizer) {
    case SEG_SGD: return launch_wgrad<SEG_SGD>(w, s);
    case SEG_SGD_MOMENTUM: return launch_wgrad<SEG_SGD_MOMENTUM>(w, s);
    case SEG_ADAM: return launch_wgrad<SEG_ADAM>(w, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace segk
