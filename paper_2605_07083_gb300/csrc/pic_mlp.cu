// pic_mlp.cu -- the surrogate MLP 5 -> 128 -> 128 -> 128 -> 4 (GELU hidden
// layers, linear output): fused forward+backward and fused reduce+Adam.
//
// Mixed precision: the forward and backward read bfloat16 weights (a copy of
// the FP32 master weights), FP32 biases, and keep FP32 activations and
// accumulators; the optimiser updates the FP32 master and re-rounds the
// bfloat16 copy.  Deterministic: per-CTA gradient partials are summed in a
// fixed order.
//
// Parameter layout (flat FP32 master, bfloat16 copy with the same indices):
// for each layer, W (n_out x n_in row-major) then b (n_out).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pic.h"

namespace pic {
namespace mlp {

constexpr int IN = 5, H = 128, OUT = 4;
constexpr int oW1 = 0, ob1 = oW1 + H * IN, oW2 = ob1 + H, ob2 = oW2 + H * H, oW3 = ob2 + H,
              ob3 = oW3 + H * H, oW4 = ob3 + H, ob4 = oW4 + OUT * H, NP = ob4 + OUT;
static_assert(NP == PIC_MLP_PARAMS, "parameter count");

// The block works on a tile of TS samples (8, 16 or 32) with 16 warps.  Every
// activation array is [unit][sample] with rows of TS + 4 floats: the samples
// of a unit are consecutive (128-bit loads of four), and rows start 4 banks
// apart (mod 8 groups of 4), so lanes on neighbouring units never collide.
// The two square weight matrices lie in shared memory as bfloat16, transposed
// ([k][j], rows of 136): the forward reads four j of a k, the backward eight
// j of a k, both without conflicts.
//
// What bounds it: FP32 FMAs on the SM (6 x 128 x 128 x TS per training tile,
// two per fma.rn.f32x2 over two samples), then the erf of the activations and
// the partials' stores.  A 4 x 4 register tile needs two shared loads per 16
// FMAs; with one thread per unit each FMA row had a 2-byte global load and a
// scalar shared load per FMA, 150 us even for one tile.  Measured before and
// after: training step of 4096 samples 161 -> 41 us, gradient of 100 samples
// 154 -> 18.6 us, prediction of 41216 samples 287 -> 82 us.
constexpr int kThr = 512, kWarps = kThr / 32;
constexpr int kWRow = H + 8;                 // bfloat16 per row of a transposed matrix
constexpr int kSms = 152;                    // tiles are kept to one wave while they fit

template <int TS>
struct Tile {
  static constexpr int kRow = TS + 4;        // floats per row of an activation array
  static constexpr int kSg = TS / 4;         // groups of the four samples that a warp takes
  static constexpr int kSplit = kWarps / kSg;    // warps that share a group's contraction
  static_assert(kSplit > 1, "the partial sums of a group go through shared memory");
};

template <int TS>
struct Smem {
  __nv_bfloat16 w2t[H][kWRow], w3t[H][kWRow];
  float w1t[IN][H], w4[OUT][H];
  float b1[H], b2[H], b3[H], b4[OUT];
  float a0[IN][Tile<TS>::kRow];
  float dy[OUT][Tile<TS>::kRow];
  float part[Tile<TS>::kSplit][H][Tile<TS>::kRow];   // partial sums
  float ypart[kThr / TS][TS];                // output-layer partial sums
  float a1[H][Tile<TS>::kRow], a2[H][Tile<TS>::kRow];
};
// training only: the last activations (prediction reuses a1), and gelu'(z) of
// each layer, then (in place) its delta
template <int TS>
struct SmemGrad {
  float a3[H][Tile<TS>::kRow];
  float red[kThr];
  float g1[H][Tile<TS>::kRow], g2[H][Tile<TS>::kRow], g3[H][Tile<TS>::kRow];
};

using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float a, float b) {
  return ((f2)__float_as_uint(b) << 32) | (f2)__float_as_uint(a);
}
__device__ __forceinline__ float lo2(f2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(f2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// both halves of a pair = bfloat16 element 0 / 1 of a 32-bit word
__device__ __forceinline__ f2 dup_lo(unsigned w) {
  const float x = __uint_as_float(w << 16);
  return pack2(x, x);
}
__device__ __forceinline__ f2 dup_hi(unsigned w) {
  const float x = __uint_as_float(w & 0xffff0000u);
  return pack2(x, x);
}

// gelu(x) and, for training, gelu'(x) from the same erf
template <bool kGrad>
__device__ __forceinline__ float gelu(float x, float& slope) {
  const float e1 = 1.0f + erff(x * 0.70710678118654752f);
  if (kGrad) slope = 0.5f * e1 + x * (0.39894228040143268f * __expf(-0.5f * x * x));
  return 0.5f * x * e1;
}

// 128 x 128 bfloat16 W (row-major [j][k]) into shared memory as [k][j]: a
// thread takes two rows' next eight columns and writes eight (j, j + 1) words.
// Fetch and store are apart so that the loads of both matrices and of the
// small arrays are in flight together.
constexpr int kTasks = (H / 2) * (H / 8);      // (row pair, eight columns)

__device__ __forceinline__ void fetch_rows(const __nv_bfloat16* __restrict__ W, int t, uint4& u,
                                           uint4& v) {
  const unsigned short* p0 =
      reinterpret_cast<const unsigned short*>(W) + (2 * (t & (H / 2 - 1))) * H + (t >> 6) * 8;
  if ((reinterpret_cast<unsigned long long>(W) & 15ull) == 0ull) {
    u = *reinterpret_cast<const uint4*>(p0);
    v = *reinterpret_cast<const uint4*>(p0 + H);
  } else {
    unsigned x[4], y[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      x[q] = (unsigned)p0[2 * q] | ((unsigned)p0[2 * q + 1] << 16);
      y[q] = (unsigned)p0[H + 2 * q] | ((unsigned)p0[H + 2 * q + 1] << 16);
    }
    u = make_uint4(x[0], x[1], x[2], x[3]);
    v = make_uint4(y[0], y[1], y[2], y[3]);
  }
}

__device__ __forceinline__ void store_rows(__nv_bfloat16 (*wt)[kWRow], int t, const uint4& u,
                                           const uint4& v) {
  unsigned* dst = reinterpret_cast<unsigned*>(wt);
  const int jp = t & (H / 2 - 1), k0 = (t >> 6) * 8;
  const unsigned x[4] = {u.x, u.y, u.z, u.w}, y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    dst[(k0 + 2 * q) * (kWRow / 2) + jp] = __byte_perm(x[q], y[q], 0x5410);
    dst[(k0 + 2 * q + 1) * (kWRow / 2) + jp] = __byte_perm(x[q], y[q], 0x7632);
  }
}

__device__ __forceinline__ void load_transposed(const __nv_bfloat16* __restrict__ W,
                                                __nv_bfloat16 (*wt)[kWRow], int threads) {
#pragma unroll 2
  for (int t = threadIdx.x; t < kTasks; t += threads) {
    uint4 u, v;
    fetch_rows(W, t, u, v);
    store_rows(wt, t, u, v);
  }
}

// the weights, biases and the tile's inputs; the caller's first barrier follows
template <int TS>
__device__ __forceinline__ void load_tile(Smem<TS>& S, const float* __restrict__ master,
                                          const __nv_bfloat16* __restrict__ w,
                                          const float* __restrict__ x, long long s0, int ns) {
  static_assert(kTasks == 2 * kThr && H * IN <= 2 * kThr && OUT * H == kThr && 3 * H <= kThr &&
                    TS * IN <= kThr, "loads per thread");
  const int tid = threadIdx.x;
  uint4 u2[2], v2[2], u3[2], v3[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    fetch_rows(w + oW2, tid + r * kThr, u2[r], v2[r]);
    fetch_rows(w + oW3, tid + r * kThr, u3[r], v3[r]);
  }
  const int xs = tid / IN, xk = tid - xs * IN;
  const float xv = tid < TS * IN && xs < ns ? x[s0 * IN + tid] : 0.0f;
  const __nv_bfloat16 wa = w[oW1 + tid];
  const bool more = tid + kThr < H * IN;
  const __nv_bfloat16 wb = more ? w[oW1 + tid + kThr] : wa;
  const __nv_bfloat16 wo = w[oW4 + tid];
  const int bl = tid / H, bj = tid % H;        // bias of hidden layer bl
  const float bv = bl < 3 ? master[(bl == 0 ? ob1 : bl == 1 ? ob2 : ob3) + bj]
                          : (bj < OUT ? master[ob4 + bj] : 0.0f);
  if (tid < TS * IN) S.a0[xk][xs] = xv;
  S.w1t[tid % IN][tid / IN] = __bfloat162float(wa);
  if (more) S.w1t[(tid + kThr) % IN][(tid + kThr) / IN] = __bfloat162float(wb);
  S.w4[tid / H][tid % H] = __bfloat162float(wo);
  if (bl == 0) S.b1[bj] = bv;
  else if (bl == 1) S.b2[bj] = bv;
  else if (bl == 2) S.b3[bj] = bv;
  else if (bj < OUT) S.b4[bj] = bv;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    store_rows(S.w2t, tid + r * kThr, u2[r], v2[r]);
    store_rows(S.w3t, tid + r * kThr, u3[r], v3[r]);
  }
}

// acc[r][p] += over this warp's part of the contraction index c of
// wt[c][4 lane + r] * in[c][first sample of the group + 2 p (+1)]: the forward
// product of unit 4 lane + r, two samples per FMA
template <int TS>
__device__ __forceinline__ void product_forward(const __nv_bfloat16 (*wt)[kWRow],
                                                const float (*in)[Tile<TS>::kRow], int sg, int part,
                                                f2 (&acc)[4][2]) {
  constexpr int kLen = H / Tile<TS>::kSplit;
  const int lane = threadIdx.x & 31, c0 = part * kLen;
#pragma unroll 8
  for (int c = c0; c < c0 + kLen; ++c) {
    const uint2 wv = *reinterpret_cast<const uint2*>(&wt[c][4 * lane]);
    const f2 d[4] = {dup_lo(wv.x), dup_hi(wv.x), dup_lo(wv.y), dup_hi(wv.y)};
    const ulonglong2 av = *reinterpret_cast<const ulonglong2*>(&in[c][4 * sg]);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      acc[r][0] = fma2(d[r], av.x, acc[r][0]);
      acc[r][1] = fma2(d[r], av.y, acc[r][1]);
    }
  }
}

// acc[r][p] += over this warp's part of j of W[j][lane + 32 r] * in[j][...]:
// the backward product (wt[k][j] read along j, eight at a time)
template <int TS>
__device__ __forceinline__ void product_backward(const __nv_bfloat16 (*wt)[kWRow],
                                                 const float (*in)[Tile<TS>::kRow], int sg,
                                                 int part, f2 (&acc)[4][2]) {
  constexpr int kLen = H / Tile<TS>::kSplit;
  const int lane = threadIdx.x & 31, j0 = part * kLen;
#pragma unroll 2
  for (int j = j0; j < j0 + kLen; j += 8) {
    uint4 wv[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) wv[r] = *reinterpret_cast<const uint4*>(&wt[lane + 32 * r][j]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(&in[j + 2 * q][4 * sg]);
      const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(&in[j + 2 * q + 1][4 * sg]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const unsigned u = q == 0 ? wv[r].x : q == 1 ? wv[r].y : q == 2 ? wv[r].z : wv[r].w;
        const f2 e = dup_lo(u), o = dup_hi(u);
        acc[r][0] = fma2(e, a0.x, acc[r][0]);
        acc[r][1] = fma2(e, a0.y, acc[r][1]);
        acc[r][0] = fma2(o, a1.x, acc[r][0]);
        acc[r][1] = fma2(o, a1.y, acc[r][1]);
      }
    }
  }
}

// z (4 units x 4 samples per thread) -> activation and slope
template <bool kGrad>
__device__ __forceinline__ void activate4(const float (&z)[4], float* act, float* slope) {
  float4 av, gv;
  float* a = reinterpret_cast<float*>(&av);
  float* g = reinterpret_cast<float*>(&gv);
#pragma unroll
  for (int k = 0; k < 4; ++k) a[k] = gelu<kGrad>(z[k], g[k]);
  *reinterpret_cast<float4*>(act) = av;
  if (kGrad) *reinterpret_cast<float4*>(slope) = gv;
}

// a hidden layer: out = gelu(W in + b), slopes for training, for the first
// `live` samples of the tile (rounded up to a group).  The contraction is split
// over kSplit warps and summed part by part after a barrier.
template <int TS, bool kGrad>
__device__ __forceinline__ void hidden_layer(Smem<TS>& S, const __nv_bfloat16 (*wt)[kWRow],
                                             const float* b, const float (*in)[Tile<TS>::kRow],
                                             float (*out)[Tile<TS>::kRow],
                                             float (*slope)[Tile<TS>::kRow], int live) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sg = warp % Tile<TS>::kSg, part = warp / Tile<TS>::kSg;
  if (4 * sg < live) {
    f2 acc[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float b0 = part == 0 ? b[4 * lane + r] : 0.0f;
      acc[r][0] = acc[r][1] = pack2(b0, b0);
    }
    product_forward<TS>(wt, in, sg, part, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r)
      *reinterpret_cast<ulonglong2*>(&S.part[part][4 * lane + r][4 * sg]) =
          make_ulonglong2(acc[r][0], acc[r][1]);
  }
  __syncthreads();
  for (int e = tid; e < H * (TS / 4); e += kThr) {
    const int j = e / (TS / 4), s = 4 * (e % (TS / 4));
    float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q < Tile<TS>::kSplit; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(&S.part[q][j][s]);
      z[0] += v.x; z[1] += v.y; z[2] += v.z; z[3] += v.w;
    }
    if (s < live) activate4<kGrad>(z, &out[j][s], kGrad ? &slope[j][s] : nullptr);
  }
  __syncthreads();
}

// delta of the layer below: slope <- (W^T delta) * slope
template <int TS>
__device__ __forceinline__ void back_delta(Smem<TS>& S, const __nv_bfloat16 (*wt)[kWRow],
                                           const float (*delta)[Tile<TS>::kRow],
                                           float (*slope)[Tile<TS>::kRow]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sg = warp % Tile<TS>::kSg, part = warp / Tile<TS>::kSg;
  f2 acc[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = 0ull;
  product_backward<TS>(wt, delta, sg, part, acc);
#pragma unroll
  for (int r = 0; r < 4; ++r)
    *reinterpret_cast<ulonglong2*>(&S.part[part][lane + 32 * r][4 * sg]) =
        make_ulonglong2(acc[r][0], acc[r][1]);
  __syncthreads();
  for (int e = tid; e < H * (TS / 4); e += kThr) {
    const int k = e / (TS / 4), s = 4 * (e % (TS / 4));
    float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int q = 0; q < Tile<TS>::kSplit; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(&S.part[q][k][s]);
      z.x += v.x; z.y += v.y; z.z += v.z; z.w += v.w;
    }
    float4* p = reinterpret_cast<float4*>(&slope[k][s]);
    const float4 g = *p;
    *p = make_float4(z.x * g.x, z.y * g.y, z.z * g.z, z.w * g.w);
  }
  __syncthreads();
}

// gW[j][k] = sum_s d[j][s] a[k][s], gb[j] = sum_s d[j][s]: thread (jg, kg) has
// the 4 x 8 outputs (jg + 32 r, kg + 16 t); even and odd samples are summed
// apart, two per FMA.  Samples past the batch have d = 0.
template <int TS>
__device__ __forceinline__ void weight_grad(const float (*d)[Tile<TS>::kRow],
                                            const float (*a)[Tile<TS>::kRow], float* gW, float* gb) {
  constexpr int kR = H * 16 / kThr;          // rows per thread
  const int tid = threadIdx.x, jg = tid >> 4, kg = tid & 15;
  f2 acc[kR][8];
#pragma unroll
  for (int r = 0; r < kR; ++r)
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[r][t] = 0ull;
#pragma unroll 2
  for (int s = 0; s < TS; s += 4) {
    ulonglong2 dv[kR];
#pragma unroll
    for (int r = 0; r < kR; ++r)
      dv[r] = *reinterpret_cast<const ulonglong2*>(&d[jg + (kThr / 16) * r][s]);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const ulonglong2 av = *reinterpret_cast<const ulonglong2*>(&a[kg + 16 * t][s]);
#pragma unroll
      for (int r = 0; r < kR; ++r) acc[r][t] = fma2(dv[r].x, av.x, acc[r][t]);
#pragma unroll
      for (int r = 0; r < kR; ++r) acc[r][t] = fma2(dv[r].y, av.y, acc[r][t]);
    }
  }
#pragma unroll
  for (int r = 0; r < kR; ++r)
#pragma unroll
    for (int t = 0; t < 8; ++t)
      gW[(jg + (kThr / 16) * r) * H + kg + 16 * t] = lo2(acc[r][t]) + hi2(acc[r][t]);
  if (tid < H) {
    float g = 0.0f;
#pragma unroll
    for (int s = 0; s < TS; s += 4) {
      const float4 v = *reinterpret_cast<const float4*>(&d[tid][s]);
      g += v.x; g += v.y; g += v.z; g += v.w;
    }
    gb[tid] = g;
  }
}

// layers 1 to 3 and the output partial sums of a loaded tile; y of
// output o and sample s is then y_of(S, o, s)
template <int TS, bool kGrad>
__device__ __forceinline__ void forward_tile(Smem<TS>& S, SmemGrad<TS>* G, int ns) {
  // training computes whole tiles (samples past the batch read zeros and get
  // delta 0), prediction only the groups of four that hold samples
  const int live = kGrad ? TS : (ns + 3) & ~3;
  const int tid = threadIdx.x;
  __syncthreads();                     // load_tile
  for (int e = tid; e < H * (live / 4); e += kThr) {
    const int j = e % H, s = 4 * (e / H);
    float z[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) z[q] = S.b1[j];
#pragma unroll
    for (int k = 0; k < IN; ++k) {
      const float wv = S.w1t[k][j];
#pragma unroll
      for (int q = 0; q < 4; ++q) z[q] = fmaf(wv, S.a0[k][s + q], z[q]);
    }
    activate4<kGrad>(z, &S.a1[j][s], kGrad ? &G->g1[j][s] : nullptr);
  }
  __syncthreads();
  hidden_layer<TS, kGrad>(S, S.w2t, S.b2, S.a1, S.a2, kGrad ? G->g2 : nullptr, live);
  float (*a3)[Tile<TS>::kRow] = kGrad ? G->a3 : S.a1;
  hidden_layer<TS, kGrad>(S, S.w3t, S.b3, S.a2, a3, kGrad ? G->g3 : nullptr, live);
  // output layer: (output, part of the contraction) per group of TS lanes
  {
    constexpr int kParts = kThr / TS / OUT, kLen = H / kParts;
    const int grp = tid / TS, s = tid % TS, o = grp & 3, part = grp >> 2;
    float acc = part == 0 ? S.b4[o] : 0.0f;
#pragma unroll 8
    for (int k = part * kLen; k < (part + 1) * kLen; ++k) acc = fmaf(S.w4[o][k], a3[k][s], acc);
    S.ypart[part * OUT + o][s] = acc;
  }
  __syncthreads();
}

template <int TS>
__device__ __forceinline__ float y_of(const Smem<TS>& S, int o, int s) {
  constexpr int kParts = kThr / TS / OUT;
  float y = S.ypart[o][s];
#pragma unroll
  for (int q = 1; q < kParts; ++q) y += S.ypart[q * OUT + o][s];
  return y;
}

// Prediction of up to a wave of tiles: one block per tile
template <int TS>
__global__ void __launch_bounds__(kThr) k_mlp_forward(const float* __restrict__ master,
                                                      const __nv_bfloat16* __restrict__ w,
                                                      const float* __restrict__ x, long long batch,
                                                      float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TS>& S = *reinterpret_cast<Smem<TS>*>(raw);
  const long long s0 = (long long)blockIdx.x * TS;
  const int ns = (int)min((long long)TS, batch - s0);
  load_tile<TS>(S, master, w, x, s0, ns);
  forward_tile<TS, false>(S, nullptr, ns);
  for (int i = threadIdx.x; i < TS * OUT; i += kThr) {
    const int s = i / OUT, o = i - s * OUT;
    if (s < ns) y[(s0 + s) * OUT + o] = y_of<TS>(S, o, s);
  }
}

// Prediction of large batches: the weights stay in shared memory, and a warp
// takes eight samples at a time through all layers on its own, so no block
// barrier ties the warps' FMA phases and erf phases together.  What bounds it:
// the FMA pipe in the products (16 fma.rn.f32x2 to 8 conversions and 3 shared
// loads) and issue in the erf, 51 % and 58 % busy over the kernel.  41216
// samples take 82 us (84 with block tiles of 128 samples, 287 with one thread
// per unit).  A lane has units 4 l ... 4 l + 3 of all eight samples; the
// warp's activations are [unit][sample], eight floats a row and four floats
// of padding every four rows, so that a lane's rows start on banks of their
// own.
constexpr int kWideSamples = 8, kWideMaxWarps = 20;
struct WideSmem {
  __nv_bfloat16 w2t[H][kWRow], w3t[H][kWRow];
  float w1t[IN][H], w4[OUT][H];
  float b1[H], b2[H], b3[H], b4[OUT];
};
constexpr int kWideBuf = H * kWideSamples + (H / 4) * 4 + IN * kWideSamples;   // floats per warp
__device__ __forceinline__ int wide_at(int unit) { return unit * kWideSamples + (unit >> 2) * 4; }

// acc (samples 2 p, 2 p + 1 of unit 4 lane + r) -> activations
__device__ __forceinline__ void wide_activate(const f2 (&acc)[4][4], float* buf, int lane) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float a[8], unused;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      a[2 * p] = gelu<false>(lo2(acc[r][p]), unused);
      a[2 * p + 1] = gelu<false>(hi2(acc[r][p]), unused);
    }
    float4* row = reinterpret_cast<float4*>(buf + wide_at(4 * lane + r));
    row[0] = make_float4(a[0], a[1], a[2], a[3]);
    row[1] = make_float4(a[4], a[5], a[6], a[7]);
  }
}

__device__ __forceinline__ void wide_layer(const __nv_bfloat16 (*wt)[kWRow], const float* b,
                                           float* buf, int lane) {
  f2 acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[r][p] = pack2(b[4 * lane + r], b[4 * lane + r]);
#pragma unroll 4
  for (int c = 0; c < H; ++c) {
    const uint2 wv = *reinterpret_cast<const uint2*>(&wt[c][4 * lane]);
    const ulonglong2* row = reinterpret_cast<const ulonglong2*>(buf + wide_at(c));
    const ulonglong2 a0 = row[0], a1 = row[1];
    const f2 d[4] = {dup_lo(wv.x), dup_hi(wv.x), dup_lo(wv.y), dup_hi(wv.y)};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      acc[r][0] = fma2(d[r], a0.x, acc[r][0]);
      acc[r][1] = fma2(d[r], a0.y, acc[r][1]);
      acc[r][2] = fma2(d[r], a1.x, acc[r][2]);
      acc[r][3] = fma2(d[r], a1.y, acc[r][3]);
    }
  }
  __syncwarp();                        // every lane has read the layer below
  wide_activate(acc, buf, lane);
  __syncwarp();
}

__global__ void __launch_bounds__(32 * kWideMaxWarps, 1)
    k_mlp_forward_wide(const float* __restrict__ master, const __nv_bfloat16* __restrict__ w,
                       const float* __restrict__ x, long long batch, float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char raw[];
  WideSmem& S = *reinterpret_cast<WideSmem*>(raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = (int)(blockDim.x >> 5);
  float* buf = reinterpret_cast<float*>(raw + sizeof(WideSmem)) + (size_t)warp * kWideBuf;
  float* xs = buf + H * kWideSamples + (H / 4) * 4;        // [IN][samples]
  load_transposed(w + oW2, S.w2t, (int)blockDim.x);
  load_transposed(w + oW3, S.w3t, (int)blockDim.x);
  for (int i = tid; i < H * IN; i += blockDim.x) S.w1t[i % IN][i / IN] = __bfloat162float(w[oW1 + i]);
  for (int i = tid; i < OUT * H; i += blockDim.x) S.w4[i / H][i % H] = __bfloat162float(w[oW4 + i]);
  for (int i = tid; i < H; i += blockDim.x) {
    S.b1[i] = master[ob1 + i];
    S.b2[i] = master[ob2 + i];
    S.b3[i] = master[ob3 + i];
  }
  if (tid < OUT) S.b4[tid] = master[ob4 + tid];
  __syncthreads();
  const long long groups = (batch + kWideSamples - 1) / kWideSamples;
  // consecutive groups to the same warp number of all blocks: every SM gets
  // its share of the last round
  for (long long g = (long long)warp * gridDim.x + blockIdx.x; g < groups;
       g += (long long)warps * gridDim.x) {
    const long long s0 = g * kWideSamples;
    const int ns = (int)min((long long)kWideSamples, batch - s0);
    for (int i = lane; i < IN * kWideSamples; i += 32) {
      const int s = i / IN, k = i - s * IN;
      xs[k * kWideSamples + s] = s < ns ? x[(s0 + s) * IN + k] : 0.0f;
    }
    __syncwarp();
    {
      f2 acc[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[r][p] = pack2(S.b1[4 * lane + r], S.b1[4 * lane + r]);
#pragma unroll
      for (int k = 0; k < IN; ++k) {
        const ulonglong2* row = reinterpret_cast<const ulonglong2*>(xs + k * kWideSamples);
        const ulonglong2 a0 = row[0], a1 = row[1];
        const float4 wv = *reinterpret_cast<const float4*>(&S.w1t[k][4 * lane]);
        const float ws[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const f2 d = pack2(ws[r], ws[r]);
          acc[r][0] = fma2(d, a0.x, acc[r][0]);
          acc[r][1] = fma2(d, a0.y, acc[r][1]);
          acc[r][2] = fma2(d, a1.x, acc[r][2]);
          acc[r][3] = fma2(d, a1.y, acc[r][3]);
        }
      }
      wide_activate(acc, buf, lane);
    }
    __syncwarp();
    wide_layer(S.w2t, S.b2, buf, lane);
    wide_layer(S.w3t, S.b3, buf, lane);
    // output o of sample s by lane 8 o + s
    {
      const int s = lane & 7, o = lane >> 3;
      float acc = S.b4[o];
#pragma unroll 8
      for (int k = 0; k < H; ++k) acc = fmaf(S.w4[o][k], buf[wide_at(k) + s], acc);
      if (s < ns) y[(s0 + s) * OUT + o] = acc;
    }
    __syncwarp();                      // the buffer is reused
  }
}

// Training: one block per tile; per-block gradient partials [gridDim.x][NP]
// and sum of squared errors.
template <int TS>
__global__ void __launch_bounds__(kThr, 1) k_mlp_fwd_bwd(const float* __restrict__ master,
                                                         const __nv_bfloat16* __restrict__ w,
                                                         const float* __restrict__ x,
                                                         const float* __restrict__ t,
                                                         long long batch, float* __restrict__ part,
                                                         float* __restrict__ lpart) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TS>& S = *reinterpret_cast<Smem<TS>*>(raw);
  SmemGrad<TS>& G = *reinterpret_cast<SmemGrad<TS>*>(raw + sizeof(Smem<TS>));
  const int tid = threadIdx.x;
  const long long s0 = (long long)blockIdx.x * TS;
  const int ns = (int)min((long long)TS, batch - s0);
  load_tile<TS>(S, master, w, x, s0, ns);
  forward_tile<TS, true>(S, &G, ns);
  // d(loss)/dy and the squared errors
  {
    float e2 = 0.0f;
    if (tid < OUT * TS) {
      const int o = tid / TS, s = tid % TS;
      float d = 0.0f;
      if (s < ns) {
        const float diff = y_of<TS>(S, o, s) - t[(s0 + s) * OUT + o];
        d = 2.0f * diff / (float)(batch * OUT);
        e2 = diff * diff;
      }
      S.dy[o][s] = d;
    }
    G.red[tid] = e2;
  }
  __syncthreads();
  float* g = part + (size_t)blockIdx.x * NP;
  if (tid < 32) {                              // loss partial, fixed order
    float v = 0.0f;
#pragma unroll
    for (int q = 0; q < kThr / 32; ++q) v += G.red[tid + 32 * q];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (tid == 0) lpart[blockIdx.x] = v;
  }
  // output layer gradients, and the delta of layer 3 in place of its slope
  {
    const int k = tid & (H - 1), o = tid >> 7;  // kThr / H == OUT
    static_assert(kThr == H * OUT, "one output-layer weight per thread");
    float gw = 0.0f;
#pragma unroll
    for (int s = 0; s < TS; s += 4) {
      const float4 av = *reinterpret_cast<const float4*>(&G.a3[k][s]);
      const float4 d = *reinterpret_cast<const float4*>(&S.dy[o][s]);
      gw = fmaf(d.x, av.x, gw); gw = fmaf(d.y, av.y, gw);
      gw = fmaf(d.z, av.z, gw); gw = fmaf(d.w, av.w, gw);
    }
    g[oW4 + o * H + k] = gw;
    if (tid < OUT) {
      float gb = 0.0f;
      for (int s = 0; s < TS; ++s) gb += S.dy[tid][s];
      g[ob4 + tid] = gb;
    }
    const float w0 = S.w4[0][k], w1 = S.w4[1][k], w2 = S.w4[2][k], w3 = S.w4[3][k];
    for (int s = 4 * o; s < TS; s += 4 * OUT) {
      float4* p = reinterpret_cast<float4*>(&G.g3[k][s]);
      float4 v = *p;
      float* f = reinterpret_cast<float*>(&v);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a = fmaf(w0, S.dy[0][s + q], 0.0f);
        a = fmaf(w1, S.dy[1][s + q], a);
        a = fmaf(w2, S.dy[2][s + q], a);
        a = fmaf(w3, S.dy[3][s + q], a);
        f[q] *= a;
      }
      *p = v;
    }
  }
  __syncthreads();
  back_delta<TS>(S, S.w3t, G.g3, G.g2);        // g2 <- delta of layer 2
  weight_grad<TS>(G.g3, S.a2, g + oW3, g + ob3);
  back_delta<TS>(S, S.w2t, G.g2, G.g1);        // g1 <- delta of layer 1
  weight_grad<TS>(G.g2, S.a1, g + oW2, g + ob2);
  for (int i = tid; i < H * (IN + 1); i += kThr) {
    const int j = i % H, k = i / H;
    float gw = 0.0f;
#pragma unroll
    for (int s = 0; s < TS; s += 4) {
      const float4 d = *reinterpret_cast<const float4*>(&G.g1[j][s]);
      if (k < IN) {
        const float4 a = *reinterpret_cast<const float4*>(&S.a0[k][s]);
        gw = fmaf(d.x, a.x, gw); gw = fmaf(d.y, a.y, gw);
        gw = fmaf(d.z, a.z, gw); gw = fmaf(d.w, a.w, gw);
      } else {
        gw += d.x; gw += d.y; gw += d.z; gw += d.w;
      }
    }
    if (k < IN) g[oW1 + j * IN + k] = gw;
    else g[ob1 + j] = gw;
  }
}

constexpr int kRedThreads = 128, kRedUnroll = 16;   // 16 partials in flight per thread
constexpr int kRedBlocks = (NP + kRedThreads - 1) / kRedThreads;
static_assert(kRedBlocks * kRedThreads - 32 >= NP, "a warp for the loss");

__device__ __forceinline__ float tree_sum(float (&x)[kRedUnroll]) {
#pragma unroll
  for (int w = kRedUnroll / 2; w > 0; w >>= 1)
#pragma unroll
    for (int u = 0; u < w; ++u) x[u] += x[u + w];
  return x[0];
}

// s += x, the rounding error of that into low (Knuth's two-sum).  One number's
// error does not average out as a gradient's does, and a 64-bit sum, whose
// dependent additions take ~150 clocks each, made the kernel end 2 us later.
__device__ __forceinline__ void add_exactly(float& s, float& low, float x) {
  const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
  low += __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
  s = t;
}

// grad[p] = sum over CTAs of the partials; optional Adam update of the FP32
// master with the bfloat16 copy re-rounded (Kingma & Ba 2015).  The order is
// fixed: a tree over sixteen partials, the trees one after another.  (The tiles
// of 8 or 16 samples that a batch of less than a wave is cut into are up to
// four times as many partials as tiles of 32; one after another, 152 of them
// have an error of up to 151 roundings of the sum, so 13.  Sixteen running sums
// with one tree at the end are as exact, but left the compiler fewer loads in
// flight: the training step of 4096 samples 45.2 us instead of 41.0.)
__global__ void k_mlp_reduce_adam(const float* part, const float* lpart,
                                  int n_part, long long batch, float* __restrict__ grad,
                                  float* __restrict__ loss, float* __restrict__ master,
                                  __nv_bfloat16* __restrict__ w, float* __restrict__ m,
                                  float* __restrict__ v, float lr, float beta1, float beta2,
                                  float eps, float bc1, float bc2, int do_adam) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  // launched while the tiles still run (launch_reduce): everything below reads
  // what they, or launches before them, wrote (the partials through plain
  // loads: they change during this kernel's life, so no __restrict__ const)
  cudaGridDependencySynchronize();
  if (p >= kRedBlocks * kRedThreads - 32 && loss) {     // a warp without parameters
    float L = 0.0f, low = 0.0f;                // the sum and what its roundings dropped
    for (int b = threadIdx.x & 31; b < n_part; b += 32) add_exactly(L, low, lpart[b]);
    for (int off = 16; off > 0; off >>= 1) {
      const float other = __shfl_down_sync(0xffffffffu, L, off);
      low += __shfl_down_sync(0xffffffffu, low, off);
      add_exactly(L, low, other);
    }
    if ((threadIdx.x & 31) == 0) *loss = (L + low) / (float)(batch * OUT);
  }
  if (p >= NP) return;
  float gsum = 0.0f;
  int b = 0;
  for (; b + kRedUnroll <= n_part; b += kRedUnroll) {
    float x[kRedUnroll];
#pragma unroll
    for (int u = 0; u < kRedUnroll; ++u) x[u] = part[(size_t)(b + u) * NP + p];
    gsum += tree_sum(x);
  }
  if (b < n_part) {
    float x[kRedUnroll];
#pragma unroll
    for (int u = 0; u < kRedUnroll; ++u)
      x[u] = b + u < n_part ? part[(size_t)(b + u) * NP + p] : 0.0f;
    gsum += tree_sum(x);
  }
  if (grad) grad[p] = gsum;
  if (!do_adam) return;
  const float mm = beta1 * m[p] + (1.0f - beta1) * gsum;
  const float vv = beta2 * v[p] + (1.0f - beta2) * gsum * gsum;
  m[p] = mm;
  v[p] = vv;
  const float th = master[p] - lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
  master[p] = th;
  w[p] = __float2bfloat16_rn(th);
}

__global__ void k_mlp_cast(const float* __restrict__ master, __nv_bfloat16* __restrict__ w) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < NP) w[p] = __float2bfloat16_rn(master[p]);
}

// Samples per tile: the smallest of 8, 16, 32 whose tiles are one wave of
// blocks (a small batch is bound by one tile's chain of layers, which is
// shorter the fewer samples it has), else 32.  For gradients the partials of
// the tiles also have to fit in the caller's scratch.
int tile_size(long long batch, long long max_tiles) {
  for (int ts : {8, 16}) {
    const long long tiles = (batch + ts - 1) / ts;
    if (tiles <= kSms && tiles <= max_tiles) return ts;
  }
  return 32;
}

// Enough for the tile size of this batch and of every smaller one (a scratch
// taken for the largest batch serves the others).
size_t scratch_floats(long long batch) {
  const long long by32 = (batch + 31) / 32, by8 = (batch + 7) / 8;
  const long long nblk = by32 > kSms ? by32 : (by8 < kSms ? by8 : (long long)kSms);
  return (size_t)(nblk > by32 ? nblk : by32) * (NP + 1);
}

template <int TS>
cudaError_t forward_limit() {
  return cudaFuncSetAttribute(k_mlp_forward<TS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(Smem<TS>));
}
template <int TS>
cudaError_t grad_limit() {
  return cudaFuncSetAttribute(k_mlp_fwd_bwd<TS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(sizeof(Smem<TS>) + sizeof(SmemGrad<TS>)));
}

constexpr size_t wide_smem(int warps) {
  return sizeof(WideSmem) + (size_t)warps * kWideBuf * sizeof(float);
}

// the kernels' shared-memory limits, once for every device (the attribute is
// the current device's)
bool prepare_kernels() {
  static bool done[64] = {false};
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return false;
  const bool known = device >= 0 && device < 64;
  if (known && done[device]) return true;
  const bool ok = forward_limit<8>() == cudaSuccess && forward_limit<16>() == cudaSuccess &&
                  forward_limit<32>() == cudaSuccess &&
                  cudaFuncSetAttribute(k_mlp_forward_wide,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)wide_smem(kWideMaxWarps)) == cudaSuccess &&
                  grad_limit<8>() == cudaSuccess && grad_limit<16>() == cudaSuccess &&
                  grad_limit<32>() == cudaSuccess;
  if (ok && known) done[device] = true;
  return ok;
}

// The reduction's launch overlaps the end of the tiles (programmatic stream
// serialisation): its blocks wait for them to finish.
cudaError_t launch_reduce(const float* part, const float* lpart, int n_part, long long batch,
                          float* grad, float* loss, float* master, uint16_t* w, float* m, float* v,
                          float lr, float beta1, float beta2, float eps, float bc1, float bc2,
                          int do_adam, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kRedBlocks);
  cfg.blockDim = dim3(kRedThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mlp_reduce_adam, part, lpart, n_part, batch, grad, loss, master,
                            reinterpret_cast<__nv_bfloat16*>(w), m, v, lr, beta1, beta2, eps, bc1,
                            bc2, do_adam);
}

template <int TS>
void launch_grad(const float* master, const uint16_t* w, const float* x, const float* t,
                 long long batch, float* part, float* lpart, int nblk, cudaStream_t s) {
  k_mlp_fwd_bwd<TS><<<(unsigned)nblk, kThr, sizeof(Smem<TS>) + sizeof(SmemGrad<TS>), s>>>(
      master, reinterpret_cast<const __nv_bfloat16*>(w), x, t, batch, part, lpart);
}

// forward and backward of every tile; *nblk partials, then as many losses
int launch_fwd_bwd(const float* master, const uint16_t* w, const float* x, const float* t,
                   long long batch, float* scratch, size_t scratch_bytes, cudaStream_t s,
                   int* nblk_out) {
  const long long max_tiles = (long long)(scratch_bytes / (sizeof(float) * (NP + 1)));
  const int ts = tile_size(batch, max_tiles);
  const long long nblk = (batch + ts - 1) / ts;
  if (nblk > max_tiles) return PIC_EINVAL;
  if (!prepare_kernels()) return PIC_ECUDA;
  float* lpart = scratch + (size_t)nblk * NP;
  if (ts == 8) launch_grad<8>(master, w, x, t, batch, scratch, lpart, (int)nblk, s);
  else if (ts == 16) launch_grad<16>(master, w, x, t, batch, scratch, lpart, (int)nblk, s);
  else launch_grad<32>(master, w, x, t, batch, scratch, lpart, (int)nblk, s);
  *nblk_out = (int)nblk;
  return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

template <int TS>
void launch_predict(const float* master, const uint16_t* w, const float* x, long long batch,
                    float* y, cudaStream_t s) {
  k_mlp_forward<TS><<<(unsigned)((batch + TS - 1) / TS), kThr, sizeof(Smem<TS>), s>>>(
      master, reinterpret_cast<const __nv_bfloat16*>(w), x, batch, y);
}

// One block per SM, of the 12, 16 or 20 warps that leave the fewest idle in
// the last round (41216 samples: 34 groups per SM are three rounds of 12; two
// rounds of 17 took 88 us instead of 82: the FMA pipe is no fuller, and the
// warps' registers spill).
void launch_predict_wide(const float* master, const uint16_t* w, const float* x, long long batch,
                         float* y, cudaStream_t s) {
  const long long groups = (batch + kWideSamples - 1) / kWideSamples;
  const long long per_sm = (groups + kSms - 1) / kSms;
  int warps = 16;
  long long best = -1;
  for (int n : {16, 20, 12}) {
    const long long slots = (per_sm + n - 1) / n * n;
    if (best < 0 || slots < best) {
      best = slots;
      warps = n;
    }
  }
  k_mlp_forward_wide<<<kSms, 32 * warps, wide_smem(warps), s>>>(
      master, reinterpret_cast<const __nv_bfloat16*>(w), x, batch, y);
}

int launch_forward(const float* master, const uint16_t* w, const float* x, long long batch,
                   float* y, cudaStream_t s) {
  if (!prepare_kernels()) return PIC_ECUDA;
  const int ts = tile_size(batch, batch);
  if (ts == 8) launch_predict<8>(master, w, x, batch, y, s);
  else if (ts == 16) launch_predict<16>(master, w, x, batch, y, s);
  else if (batch <= 32ll * kSms) launch_predict<32>(master, w, x, batch, y, s);
  else launch_predict_wide(master, w, x, batch, y, s);
  return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

}  // namespace mlp
}  // namespace pic

using namespace pic::mlp;

extern "C" {

size_t pic_mlp_scratch_bytes(int64_t batch) {
  return batch > 0 ? pic::mlp::scratch_floats(batch) * sizeof(float) : 0;
}

int pic_mlp_cast_bf16(const float* master, uint16_t* w_bf16, void* stream) {
  if (!master || !w_bf16) return PIC_EINVAL;
  k_mlp_cast<<<(NP + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      master, reinterpret_cast<__nv_bfloat16*>(w_bf16));
  return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

int pic_mlp_forward(const float* master, const uint16_t* w_bf16, const float* x, int64_t batch,
                    float* y, void* stream) {
  if (!master || !w_bf16 || !x || !y || batch < 0) return PIC_EINVAL;
  if (batch == 0) return PIC_OK;
  return launch_forward(master, w_bf16, x, batch, y, (cudaStream_t)stream);
}

int pic_mlp_grad(const float* master, const uint16_t* w_bf16, const float* x, const float* t,
                 int64_t batch, float* grad, float* loss, float* scratch, size_t scratch_bytes,
                 void* stream) {
  if (!master || !w_bf16 || !x || !t || !grad || batch <= 0 || !scratch) return PIC_EINVAL;
  int nblk = 0;
  int rc = launch_fwd_bwd(master, w_bf16, x, t, batch, scratch, scratch_bytes,
                          (cudaStream_t)stream, &nblk);
  if (rc != PIC_OK) return rc;
  const cudaError_t e = launch_reduce(scratch, scratch + (size_t)nblk * NP, nblk, batch, grad, loss,
                                      nullptr, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f, 0.f, 1.f,
                                      1.f, 0, (cudaStream_t)stream);
  return e == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

int pic_mlp_train_step(float* master, uint16_t* w_bf16, float* adam_m, float* adam_v,
                       int64_t step, float lr, float beta1, float beta2, float eps, const float* x,
                       const float* t, int64_t batch, float* loss, float* scratch,
                       size_t scratch_bytes, void* stream) {
  if (!master || !w_bf16 || !adam_m || !adam_v || !x || !t || batch <= 0 || step < 1 || !scratch)
    return PIC_EINVAL;
  int nblk = 0;
  int rc = launch_fwd_bwd(master, w_bf16, x, t, batch, scratch, scratch_bytes,
                          (cudaStream_t)stream, &nblk);
  if (rc != PIC_OK) return rc;
  const float bc1 = 1.0f - powf(beta1, (float)step), bc2 = 1.0f - powf(beta2, (float)step);
  const cudaError_t e = launch_reduce(scratch, scratch + (size_t)nblk * NP, nblk, batch, nullptr,
                                      loss, master, w_bf16, adam_m, adam_v, lr, beta1, beta2, eps,
                                      bc1, bc2, 1, (cudaStream_t)stream);
  return e == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

}  // extern "C"
