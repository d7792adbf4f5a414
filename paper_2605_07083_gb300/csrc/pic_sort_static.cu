// pic_sort_static.cu -- stable sort of one particle set by cell that
// allocates nothing: its (cell, chunk) histogram lives in a fixed device array
// of this library (see pic_sort_by_cell_static in include/pic.h).
//
// The kernels of the handle's periodic sort (pic_sort_core.cuh) with plain
// pointers, and the scratch taken from static arrays instead of a handle.
#include <cuda_runtime.h>

#include <climits>
#include <mutex>

#include "../../include/pic.h"
#include "pic_sort_core.cuh"

constexpr int kStaticHistInts = 1 << 20;     // 4 MiB of scratch on every device
constexpr int kLimitChunk = 8192;            // the chunk of the documented limit on n and n_cells

// The scratch: the histogram and the sums of its tiles.  Every GPU that loads
// the library holds it until exit.  Host code must not pass these symbols to a
// kernel: on the host they are only stand-ins; their device addresses come
// from cudaGetSymbolAddress below.
static __device__ __align__(256) int g_static_hist[kStaticHistInts];
static __device__ __align__(256) int g_static_tsum[kStaticHistInts / pic::sortcore::kTile];

namespace pic {
namespace {

using sortcore::View;
using sortcore::kThreads;

__global__ void __launch_bounds__(kThreads) k_static_hist(View v) {
  extern __shared__ __align__(16) unsigned char smem[];
  sortcore::sort_hist(v, blockIdx.x, reinterpret_cast<int*>(smem));
}

__global__ void __launch_bounds__(kThreads) k_static_tilesum(View v) {
  __shared__ int ws[32];
  sortcore::sort_tilesum(v, blockIdx.x, ws);
}

__global__ void __launch_bounds__(kThreads) k_static_scan(View v) {
  __shared__ int ws[32];
  sortcore::sort_scan(v, blockIdx.x, ws);
}

template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps) k_static_scatter(View v) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int ws[32];
  sortcore::sort_scatter<kWarps>(v, blockIdx.x, smem, ws);
}

// Per-device set-up, once, with that device current: the device address of
// the scratch arrays, the SM count and the scatter kernels' shared-memory limits.
std::mutex g_setup_mu;
int* g_hist_addr[64] = {nullptr};
int* g_tsum_addr[64] = {nullptr};
int g_sms[64] = {0};

int static_setup(int device, int** hist, int** tsum, int* sms) {
  if (device < 0 || device >= 64) return PIC_EINVAL;
  std::lock_guard<std::mutex> lock(g_setup_mu);
  if (!g_hist_addr[device]) {
    void* ptr = nullptr;
    void* tptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_hist) != cudaSuccess || !ptr) return PIC_ECUDA;
    if (cudaGetSymbolAddress(&tptr, g_static_tsum) != cudaSuccess || !tptr) return PIC_ECUDA;
    // 32 warps take up to 2048 cells, 16 warps the rest
    const size_t s32 = sortcore::scatter_smem(2048, 32), s16 = sortcore::scatter_smem(kMaxNz, 16);
    if (cudaFuncSetAttribute(k_static_scatter<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)s32) != cudaSuccess ||
        cudaFuncSetAttribute(k_static_scatter<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)s16) != cudaSuccess ||
        cudaDeviceGetAttribute(&g_sms[device], cudaDevAttrMultiProcessorCount, device) !=
            cudaSuccess)
      return PIC_ECUDA;
    g_tsum_addr[device] = static_cast<int*>(tptr);
    g_hist_addr[device] = static_cast<int*>(ptr);
  }
  *hist = g_hist_addr[device];
  *tsum = g_tsum_addr[device];
  *sms = g_sms[device];
  return PIC_OK;
}

}  // namespace
}  // namespace pic

extern "C" int pic_sort_by_cell_static(const float* z, const float* vx, const float* vy,
                                       const float* vz, const uint32_t* id, int64_t n,
                                       int32_t n_cells, double gap_m, float* z_out,
                                       float* vx_out, float* vy_out, float* vz_out,
                                       uint32_t* id_out, void* cuda_stream) {
  using namespace pic;
  if (n < 0 || n_cells < 1 || n_cells > kMaxNz || !(gap_m > 0)) return PIC_EINVAL;
  if (n == 0) return PIC_OK;
  if (!z || !vx || !vy || !vz || !id || !z_out || !vx_out || !vy_out || !vz_out || !id_out)
    return PIC_EINVAL;
  // histogram entries and output positions are 32-bit
  if (n > (int64_t)INT32_MAX) return PIC_ECAPACITY;
  if ((long long)n_cells * ((n + kLimitChunk - 1) / kLimitChunk) > kStaticHistInts)
    return PIC_ECAPACITY;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return PIC_ECUDA;
  View v;
  int sms = 0;
  int rc = static_setup(dev, &v.hist, &v.tsum, &sms);
  if (rc != PIC_OK) return rc;
  // the chunk that fills the SMs evenly, unless its columns would not fit in
  // the scratch: the longest chunk, at least the limit's own, always does
  const int warps = n_cells <= 2048 ? 32 : 16;
  static_assert(sortcore::max_chunk(16) >= kLimitChunk, "every accepted size fits");
  v.chunk = sortcore::chunk_of((int)n, warps, sms);
  if ((long long)n_cells * ((n + v.chunk - 1) / v.chunk) > kStaticHistInts)
    v.chunk = sortcore::max_chunk(warps);
  const long long nch = (n + v.chunk - 1) / v.chunk;
  v.z = z; v.vx = vx; v.vy = vy; v.vz = vz; v.id = id;
  v.zo = z_out; v.vxo = vx_out; v.vyo = vy_out; v.vzo = vz_out; v.ido = id_out;
  v.n = (int)n;
  v.nch = (int)nch;
  v.Nz = n_cells;
  v.inv_dz = (float)((double)n_cells / gap_m);
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const unsigned tiles =
      (unsigned)(((long long)n_cells * nch + sortcore::kTile - 1) / sortcore::kTile);
  // up to a column's particles the scatter alone is the sort: 100 particles over
  // 128 cells take 13 us, with the histogram and its prefix 29
  if (nch > 1) {
    k_static_hist<<<(unsigned)nch, kThreads, n_cells * sizeof(int), s>>>(v);
    k_static_tilesum<<<tiles, kThreads, 0, s>>>(v);
    k_static_scan<<<tiles, kThreads, 0, s>>>(v);
  }
  const size_t smem = sortcore::scatter_smem(n_cells, warps);
  if (warps == 32) k_static_scatter<32><<<(unsigned)nch, 1024, smem, s>>>(v);
  else k_static_scatter<16><<<(unsigned)nch, 512, smem, s>>>(v);
  return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}
