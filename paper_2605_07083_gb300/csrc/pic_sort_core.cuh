// pic_sort_core.cuh -- stable counting sort of one particle set by cell: the
// bodies of the four kernels that the handle's periodic sort (pic_sort.cu)
// and the allocation-free entry point (pic_sort_static.cu) share.
//
//   1. sort_hist     per-chunk cell histogram        -> hist[cell][chunk]
//   2. sort_tilesum  sums of kTile consecutive entries -> tsum[tile]
//   3. sort_scan     exclusive prefix of hist in (cell, chunk) order, which is
//                    the first output position of each (cell, chunk)
//   4. sort_scatter  ranks a chunk's particles, reorders them in shared
//                    memory and writes runs of equal cells
//
// What bounds it: 44 B per particle (z twice, the other fields and the output
// once), so HBM for a set larger than L2; below ~1e5 particles the four
// dependent launches.  4M particles over 2048 cells in random order: 91 us
// (1.9 TB/s), 930 us before, of which the prefix took 865 us in one block and
// the scatter 261 us; the handle's sort of 2.1M particles 75 us with its copy
// back, 320 us before.  A set of one chunk needs the scatter alone.
//   * The prefix runs over all entries of the histogram: a block per tile of
//     4096 entries, ~4 us for the sums and ~5 us for the prefix (each block
//     adds up the sums of the tiles before its own).
//   * Writing each particle straight to its place touches 32 sectors per warp
//     store.  Through shared memory a chunk is first put in cell order, one
//     field at a time, so a warp writes a few runs; the longer the chunk the
//     longer the runs (at 2048 cells 4 particles per run in chunks of 8192:
//     135 us; 6.5 in chunks of 13.3k: 80 us, both with spilled registers).  What is left of the scatter is
//     those partial lines: with contiguous writes the same kernel took 30 %
//     less.
//   * A warp ranks its 32 particles without __match_any_sync (about 50 clocks
//     of an SM's time each) while their cells are all different: the ranking
//     of 8192 particles went from 27k to 8k clocks.
#pragma once

#include "pic_internal.cuh"

namespace pic {
namespace sortcore {

constexpr int kThreads = 256;                // blocks of sort_hist and the scans
constexpr int kItems = 16;                   // particles per thread of sort_scatter
constexpr int kMinChunk = 2048;
constexpr int kTile = 4096;                  // histogram entries per scan block
constexpr int kTilePer = kTile / kThreads;   // 16

// sort_scatter runs with 16 or 32 warps per block.  A 16-bit counter per
// (warp, cell) has to fit in shared memory beside the rest, so 32 warps take
// up to 2048 cells.
__host__ __device__ constexpr int max_chunk(int warps) { return warps * 32 * kItems; }

// Particles per histogram column (one block of sort_scatter): the most that a
// block takes, cut to whole waves of `slots` blocks -- on 152 SMs 4M particles
// are two waves of 13.2k instead of one and a half of 16.4k -- and rounded up
// to a multiple of 32 per warp.
__host__ __device__ __forceinline__ int chunk_of(int n, int warps, int slots) {
  const int most = max_chunk(warps), unit = 32 * warps;
  const long long waves = ((long long)n + (long long)slots * most - 1) / ((long long)slots * most);
  const long long blocks = waves > 0 ? waves * slots : 1;
  long long c = ((long long)n + blocks - 1) / blocks;
  c = (c + unit - 1) / unit * unit;
  if (c < kMinChunk) c = kMinChunk;
  return (int)(c < most ? c : most);
}

// most columns that chunk_of gives any n <= cap (it is not monotone in n)
__host__ __device__ __forceinline__ int max_columns(int cap, int warps, int slots) {
  const long long wave = (long long)slots * max_chunk(warps);
  const long long by_wave = ((long long)cap + wave - 1) / wave * slots;
  const long long by_min = ((long long)cap + kMinChunk - 1) / kMinChunk;
  return (int)(by_wave < by_min ? by_wave : by_min);
}

struct View {
  const float* z; const float* vx; const float* vy; const float* vz; const uint32_t* id;
  float* zo; float* vxo; float* vyo; float* vzo; uint32_t* ido;
  int* hist;                 // [Nz * nch] counts, then output positions
  int* tsum;                 // [ceil(Nz * nch / kTile)]
  int n;
  int chunk;                 // particles per column (chunk_of)
  int nch;                   // columns: ceil(n / chunk)
  int Nz;
  float inv_dz;
};

__device__ __forceinline__ int cell_index(float z, float inv_dz, int Nz) {
  int j;
  float f;
  cell_of(z, inv_dz, Nz, j, f);
  return j;
}

// hs: [Nz] ints of shared memory
__device__ __forceinline__ void sort_hist(const View& v, int c, int* hs) {
  for (int j = threadIdx.x; j < v.Nz; j += kThreads) hs[j] = 0;
  __syncthreads();
  const int i0 = c * v.chunk, m = min(v.n - i0, v.chunk);
  const float* zc = v.z + i0;
  constexpr int kU = 16;                     // loads in flight per thread
  for (int b = 0; b < m; b += kU * kThreads) {
    float z[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = b + u * kThreads + (int)threadIdx.x;
      z[u] = i < m ? zc[i] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = b + u * kThreads + (int)threadIdx.x;
      if (i < m) atomicAdd(&hs[cell_index(z[u], v.inv_dz, v.Nz)], 1);
    }
  }
  __syncthreads();
  // every (cell, column) entry is written, so nothing an earlier sort left
  // is read
  for (int j = threadIdx.x; j < v.Nz; j += kThreads) v.hist[(long long)j * v.nch + c] = hs[j];
}

__device__ __forceinline__ int tile_count(const View& v) {
  return (int)(((long long)v.Nz * v.nch + kTile - 1) / kTile);
}

// a thread's kTilePer consecutive entries of tile t (zero past the end)
__device__ __forceinline__ void load_tile(const View& v, int t, int (&x)[kTilePer]) {
  const long long n = (long long)v.Nz * v.nch;
  const long long at = (long long)t * kTile + (long long)threadIdx.x * kTilePer;
  if (at + kTilePer <= n) {
    const int4* p = reinterpret_cast<const int4*>(v.hist + at);
#pragma unroll
    for (int q = 0; q < kTilePer / 4; ++q) {
      const int4 w = p[q];
      x[4 * q] = w.x; x[4 * q + 1] = w.y; x[4 * q + 2] = w.z; x[4 * q + 3] = w.w;
    }
  } else {
#pragma unroll
    for (int u = 0; u < kTilePer; ++u) x[u] = at + u < n ? v.hist[at + u] : 0;
  }
}

__device__ __forceinline__ void sort_tilesum(const View& v, int t, int* ws) {
  int x[kTilePer], s = 0;
  load_tile(v, t, x);
#pragma unroll
  for (int u = 0; u < kTilePer; ++u) s += x[u];
  const int tot = block_sum<int>(s, ws);
  if (threadIdx.x == 0) v.tsum[t] = tot;
}

__device__ __forceinline__ void sort_scan(const View& v, int t, int* ws) {
  int x[kTilePer], s = 0, before = 0;
  load_tile(v, t, x);
  for (int k = threadIdx.x; k < t; k += kThreads) before += v.tsum[k];
#pragma unroll
  for (int u = 0; u < kTilePer; ++u) s += x[u];
  const int base = block_sum<int>(before, ws);
  int tot;
  int run = base + block_exclusive_scan<int>(s, &tot, ws);
#pragma unroll
  for (int u = 0; u < kTilePer; ++u) {
    const int c = x[u];
    x[u] = run;
    run += c;
  }
  const long long n = (long long)v.Nz * v.nch;
  const long long at = (long long)t * kTile + (long long)threadIdx.x * kTilePer;
  if (at + kTilePer <= n) {
    int4* p = reinterpret_cast<int4*>(v.hist + at);
#pragma unroll
    for (int q = 0; q < kTilePer / 4; ++q)
      p[q] = make_int4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
  } else {
#pragma unroll
    for (int u = 0; u < kTilePer; ++u)
      if (at + u < n) v.hist[at + u] = x[u];
  }
}

// Shared memory of sort_scatter: per-warp 16-bit cell counters, which two
// staged fields (a chunk of words each) take the place of once the ranks are
// known; the cells' output offsets; the cell of each reordered particle.
__host__ __device__ constexpr int cells_even(int Nz) { return (Nz + 1) & ~1; }
__host__ __device__ constexpr size_t scatter_stage_bytes(int Nz, int warps) {
  return (size_t)warps * cells_even(Nz) * 2 > (size_t)max_chunk(warps) * 8
             ? (((size_t)warps * cells_even(Nz) * 2 + 15) & ~(size_t)15)
             : (size_t)max_chunk(warps) * 8;
}
__host__ __device__ constexpr size_t scatter_smem(int Nz, int warps) {
  return scatter_stage_bytes(Nz, warps) + (size_t)cells_even(Nz) * 4 +
         (size_t)max_chunk(warps) * 2;
}

// One chunk: thread (warp w, lane l) holds particles w * chunk / kWarps + 32 k
// + l, so that (warp, k, lane) is the input order.  Equal cells are ranked
// within a warp's 32 particles and the warp's own counter carries the rank
// from one 32 to the next: stable without an atomic.
template <int kWarps>
__device__ __forceinline__ void sort_scatter(const View& v, int c, unsigned char* smem, int* ws) {
  constexpr int kThr = 32 * kWarps, kMax = max_chunk(kWarps);
  static_assert(kMax <= 0xffff && kItems % 2 == 0, "16-bit counters and positions");
  const int Nz = v.Nz, Nze = cells_even(Nz);
  uint16_t* cnt = reinterpret_cast<uint16_t*>(smem);                  // [kWarps][Nze]
  uint32_t* stage = reinterpret_cast<uint32_t*>(smem);                // [2][kMax], later
  int* delta = reinterpret_cast<int*>(smem + scatter_stage_bytes(Nz, kWarps));
  uint16_t* cell_s = reinterpret_cast<uint16_t*>(delta + Nze);        // [kMax]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = c * v.chunk, total = min(v.n - c0, v.chunk);
  const int per_warp = v.chunk / kWarps;
  const int w0 = warp * per_warp;
  const int left = min(total - w0, per_warp);                         // this warp's particles
  const int nk = left > lane ? (left - lane + 31) >> 5 : 0;           // this lane's
  uint32_t x[kItems];                        // the field in flight, z first
#pragma unroll
  for (int k = 0; k < kItems; ++k)
    x[k] = k < nk ? __float_as_uint(v.z[c0 + w0 + lane + 32 * k]) : 0u;
  // with one column in all, the place within the chunk is the place
  const bool whole = v.nch == 1;
  for (int j = tid; j < Nz; j += kThr) delta[j] = whole ? 0 : v.hist[(long long)j * v.nch + c];
  for (int k = tid; k < kWarps * Nze / 2; k += kThr) reinterpret_cast<uint32_t*>(cnt)[k] = 0u;
  __syncthreads();
  // ---- cells and ranks: key[k] = (cell << 16) | rank among the warp's equals
  int key[kItems];
  {
    volatile uint16_t* my = cnt + warp * Nze;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      key[k] = 0;
      if (32 * k < left) {                                            // uniform over the warp
        const bool act = k < nk;
        const int j = act ? cell_index(__uint_as_float(x[k]), v.inv_dz, Nz) : Nze;
        // all 32 cells different (each lane finds its own mark): every rank
        // is the counter itself
        const int base = act ? my[j] : 0;
        __syncwarp();
        if (act) my[j] = (uint16_t)lane;
        __syncwarp();
        const bool twin = act && my[j] != (uint16_t)lane;
        unsigned before = 0u, all = 1u;
        if (__any_sync(0xffffffffu, twin)) {
          const unsigned peers = __match_any_sync(0xffffffffu, j);
          before = __popc(peers & lt);
          all = __popc(peers);
        }
        __syncwarp();
        if (act && before == 0u) my[j] = (uint16_t)(base + all);
        __syncwarp();
        key[k] = (j << 16) | (int)(base + before);
      }
    }
  }
  __syncthreads();
  // ---- counts -> positions within the chunk: per cell the prefix over the
  // warps, over the cells a block scan (two cells per word, consecutive words
  // per thread; a chunk holds fewer than 2^16 particles, so the halves of a
  // word never carry into each other)
  {
    uint32_t* cw = reinterpret_cast<uint32_t*>(cnt);
    constexpr int kPer = (kWarps == 32 ? 2048 : kMaxNz) / 2 / kThr;
    const int nw = Nze / 2, per = (nw + kThr - 1) / kThr;             // <= kPer words
    const int k0 = tid * per;
    unsigned tw[kPer];
    unsigned sum = 0u;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      tw[q] = 0u;
      if (q < per && k0 + q < nw) {
#pragma unroll 8
        for (int w = 0; w < kWarps; ++w) tw[q] += cw[w * nw + k0 + q];
      }
      sum += tw[q];
    }
    int tot;
    int run = block_exclusive_scan<int>((int)((sum & 0xffffu) + (sum >> 16)), &tot, ws);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int k = k0 + q;
      if (q < per && k < nw) {
        const unsigned lo = (unsigned)run, hi = lo + (tw[q] & 0xffffu);
        delta[2 * k] -= (int)lo;
        if (2 * k + 1 < Nz) delta[2 * k + 1] -= (int)hi;
        unsigned at = lo | (hi << 16);
#pragma unroll 8
        for (int w = 0; w < kWarps; ++w) {
          const unsigned n = cw[w * nw + k];
          cw[w * nw + k] = at;
          at += n;
        }
        run = (int)(hi + (tw[q] >> 16));
      }
    }
  }
  __syncthreads();
  unsigned lp[kItems / 2];                   // positions within the chunk, two per word
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    unsigned at = 0u;
    if (k < nk) {
      const int j = key[k] >> 16;
      at = cnt[warp * Nze + j] + (unsigned)(key[k] & 0xffff);
      cell_s[at] = (uint16_t)j;
    }
    lp[k >> 1] = (k & 1) ? lp[k >> 1] | (at << 16) : at;
  }
  __syncthreads();                           // the counters make room for the staged fields
  int to[kItems];
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    const int s = k * kThr + tid;
    to[k] = s < total ? (whole ? s : delta[cell_s[s]] + s) : 0;
  }
  // ---- the fields, through two stages in turn: the next field's loads are
  // in flight while this one is written (a rolled loop: unrolled, the
  // compiler keeps every position's address and spills)
#pragma unroll 1
  for (int f = 0; f < 5; ++f) {
    uint32_t* sg = stage + (f & 1) * kMax;
#pragma unroll
    for (int k = 0; k < kItems; ++k)
      if (k < nk) sg[(lp[k >> 1] >> (16 * (k & 1))) & 0xffffu] = x[k];
    if (f < 4) {
      const float* nf = f == 0 ? v.vx : f == 1 ? v.vy : v.vz;
      const uint32_t* src = (f < 3 ? reinterpret_cast<const uint32_t*>(nf) : v.id) + c0 + w0 + lane;
#pragma unroll
      for (int k = 0; k < kItems; ++k) x[k] = k < nk ? src[32 * k] : 0u;
    }
    __syncthreads();
    float* of = f == 0 ? v.zo : f == 1 ? v.vxo : f == 2 ? v.vyo : v.vzo;
    uint32_t* dst = f < 4 ? reinterpret_cast<uint32_t*>(of) : v.ido;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const int s = k * kThr + tid;
      if (s < total) dst[to[k]] = sg[s];
    }
  }
}

}  // namespace sortcore
}  // namespace pic
