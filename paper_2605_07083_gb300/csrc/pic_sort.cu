// pic_sort.cu -- stable counting sort of every (instance, species) particle
// segment by cell, run every few steps so that the blocks of the push kernel
// see narrow cell ranges (short charge flushes, local shared-memory atomics).
//
// The four kernels of pic_sort_core.cuh, each a 2D grid (chunk or histogram
// tile, segment), then a copy of the sorted scratch arrays back.  The cell of
// a particle is the fixed-point deposit's cell rule.  The grids are sized by
// the segments' capacities, since the host does not know the live counts;
// blocks past a segment's live particles return at once.
#include "pic_sort_core.cuh"

namespace pic {

using sortcore::kThreads;
using sortcore::kTile;
using sortcore::View;

constexpr int kCopyChunk = 8192;             // particles per k_sort_copy block
// 16 warps: two blocks per SM overlap their phases, and a state sorted a few
// steps ago has long runs in chunks of 8192 already
constexpr int kScatWarps = 16;

// segment g of the handle; its histogram starts on a multiple of kTile
__device__ __forceinline__ View seg_view(const DevState& st, int g) {
  const InstConst& ic = st.ic[g / 3];
  const long long off = st.seg_off[g], hoff = st.sort_hoff[g];
  View v;
  v.z = st.z + off; v.vx = st.vx + off; v.vy = st.vy + off; v.vz = st.vz + off; v.id = st.id + off;
  v.zo = st.z2 + off; v.vxo = st.vx2 + off; v.vyo = st.vy2 + off; v.vzo = st.vz2 + off;
  v.ido = st.id2 + off;
  v.hist = st.sort_hist + hoff;
  v.tsum = st.sort_tsum + hoff / kTile;
  v.n = st.seg_count[g];
  v.chunk = sortcore::chunk_of(v.n, kScatWarps, st.sort_slots);
  v.nch = (v.n + v.chunk - 1) / v.chunk;
  v.Nz = ic.Nz;
  v.inv_dz = ic.inv_dz_f;
  return v;
}

__global__ void __launch_bounds__(kThreads) k_sort_hist(DevState st) {
  extern __shared__ __align__(16) unsigned char smem[];
  const View v = seg_view(st, blockIdx.y);
  if ((int)blockIdx.x >= v.nch) return;
  sortcore::sort_hist(v, blockIdx.x, reinterpret_cast<int*>(smem));
}

__global__ void __launch_bounds__(kThreads) k_sort_tilesum(DevState st) {
  __shared__ int ws[32];
  const View v = seg_view(st, blockIdx.y);
  if ((int)blockIdx.x >= sortcore::tile_count(v)) return;
  sortcore::sort_tilesum(v, blockIdx.x, ws);
}

__global__ void __launch_bounds__(kThreads) k_sort_scan(DevState st) {
  __shared__ int ws[32];
  const View v = seg_view(st, blockIdx.y);
  if ((int)blockIdx.x >= sortcore::tile_count(v)) return;
  sortcore::sort_scan(v, blockIdx.x, ws);
}

__global__ void __launch_bounds__(32 * kScatWarps, 2) k_sort_scatter(DevState st) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int ws[32];
  const View v = seg_view(st, blockIdx.y);
  if ((int)blockIdx.x >= v.nch) return;
  sortcore::sort_scatter<kScatWarps>(v, blockIdx.x, smem, ws);
}

// The sorted particles back into the handle's arrays, four slots per access:
// segments start on a multiple of 32 slots and hold a multiple of 32, so the
// last access of a segment stays inside it (its slots past the live ones
// hold nothing).
__global__ void __launch_bounds__(kThreads) k_sort_copy(DevState st) {
  const int g = blockIdx.y;
  const int N = st.seg_count[g];
  const int q0 = blockIdx.x * (kCopyChunk / 4), q1 = min((N + 3) >> 2, q0 + kCopyChunk / 4);
  const long long off = st.seg_off[g];
  const float* from[4] = {st.z2 + off, st.vx2 + off, st.vy2 + off, st.vz2 + off};
  float* to[4] = {st.z + off, st.vx + off, st.vy + off, st.vz + off};
  const uint4* ifrom = reinterpret_cast<const uint4*>(st.id2 + off);
  uint4* ito = reinterpret_cast<uint4*>(st.id + off);
  for (int q = q0 + threadIdx.x; q < q1; q += kThreads) {
    float4 x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = reinterpret_cast<const float4*>(from[k])[q];
    const uint4 i = ifrom[q];
#pragma unroll
    for (int k = 0; k < 4; ++k) reinterpret_cast<float4*>(to[k])[q] = x[k];
    ito[q] = i;
  }
}

// Blocks per wave that a segment's chunks are cut for: the segments share the
// chip, with two blocks per SM where the counters of two fit
int sort_slots(int sms, int n_seg, int max_nz) {
  const int per_sm = sortcore::scatter_smem(max_nz, kScatWarps) <= 110 * 1024 ? 2 : 1;
  return max(1, per_sm * sms / n_seg);
}

static long long seg_hist_ints(int cap, int nz, int slots) {
  return (long long)nz * sortcore::max_columns(cap, kScatWarps, slots);
}

// histogram entries of all segments (each segment's a multiple of kTile)
size_t sort_hist_ints(const int32_t* seg_cap, const int* seg_nz, int n_seg, int slots,
                      int64_t* hoff) {
  size_t tot = 0;
  for (int g = 0; g < n_seg; ++g) {
    hoff[g] = (int64_t)tot;
    tot += (size_t)(seg_hist_ints(seg_cap[g], seg_nz[g], slots) + kTile - 1) / kTile * kTile;
  }
  return tot;
}

size_t sort_tiles(size_t hist_ints) { return hist_ints / kTile; }

// grid sizes: chunks, histogram tiles and copy blocks of the largest segment
SortGrid sort_grid(const int32_t* seg_cap, const int* seg_nz, int n_seg, int slots) {
  SortGrid r{1, 1, 1};
  for (int g = 0; g < n_seg; ++g) {
    const long long e = seg_hist_ints(seg_cap[g], seg_nz[g], slots);
    r.chunks = max(r.chunks, sortcore::max_columns(seg_cap[g], kScatWarps, slots));
    r.tiles = max(r.tiles, (int)((e + kTile - 1) / kTile));
    r.copies = max(r.copies, (seg_cap[g] + kCopyChunk - 1) / kCopyChunk);
  }
  return r;
}

// raise the kernels' dynamic shared-memory limit to the opt-in maximum less
// their static shared memory
cudaError_t sort_prepare(int optin) {
  const void* fns[] = {(const void*)k_sort_scatter, (const void*)k_sort_hist};
  for (const void* f : fns) {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, f);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               optin - (int)a.sharedSizeBytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void sort_launch(const DevState& st, const SortGrid& r, int max_nz, cudaStream_t s) {
  const dim3 chunks(r.chunks, st.n_seg), tiles(r.tiles, st.n_seg), copies(r.copies, st.n_seg);
  k_sort_hist<<<chunks, kThreads, max_nz * sizeof(int), s>>>(st);
  k_sort_tilesum<<<tiles, kThreads, 0, s>>>(st);
  k_sort_scan<<<tiles, kThreads, 0, s>>>(st);
  k_sort_scatter<<<chunks, 32 * kScatWarps, sortcore::scatter_smem(max_nz, kScatWarps), s>>>(st);
  k_sort_copy<<<copies, kThreads, 0, s>>>(st);
}

}  // namespace pic
