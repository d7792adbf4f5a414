// pic_fused.cuh -- whole time steps of small diodes in one kernel.
//
// A step of a diode with a few tens of thousands of particles is bound by the
// three dependent kernels and the round trips inside them (17.1 us a step for
// 22k particles), not by its work.  Here a thread-block cluster (1 to 16
// blocks, by how many diodes share the chip) owns a diode and runs n_steps of
// it: field, constants, counts and tallies stay in shared memory, the
// particles in L2, and the phases of a step meet at hardware cluster
// barriers (9.4 us a step; 128 diodes of 5.3k particles 32 -> 11.8 us).  What
// is left is the phases' own round trips: about 40 % push, the rest lists, charge,
// field and compaction, of which only latency counts; a block keeps its
// registers below the limit, since a spilled one is fetched from L2 after
// every barrier (768 threads, which spill, took 28 us).  It computes exactly
// what k_push, k_mid and k_post compute, in the same arithmetic and array
// order (included by pic_kernels.cu for the functions they share), so a run
// may switch between the two at any step.
//
// Phases of a step (each ends at a cluster barrier):
//   A  push of the cluster's particles (contiguous quads per block and warp),
//      charge into shared histograms (electrons, ions), absorbed slots listed
//      per warp, candidates per block
//   B  the warps' absorbed lists into the diode's ordered list; the charge
//      summed over the blocks; collisions of the blocks' candidates
//   C  kinetic energies of the absorbed particles read (last block); the
//      particles that will fill their slots looked up and read; the field, by
//      every block for itself, the prefix in its last warp (in all
//      of them from kFusedWarpCells cells on)
//   D  the tallies summed (last block), hole filling and appends (a species
//      per block, or per part of the block's warps)
//
// k_route, on the device since only the device knows the live counts, picks
// this kernel or the three for every captured step graph.
#pragma once

#include <cooperative_groups.h>

namespace pic {

namespace cg = cooperative_groups;

constexpr int kFusedWarps = kFusedThreads / 32;
constexpr int kFusedMaxC = 16;         // blocks per cluster (non-portable above 8)
constexpr int kFusedList = 1024;       // absorbed slots of a species held in shared memory
constexpr int kFusedWarpList = 32;     // of a warp and species
constexpr int kFusedTeamWarps = kFusedWarps - 1;   // warps of phase D's teams

// shared memory: (E_j, dE_j) pairs, E, two histograms, the blocks' and the
// diode's node charge (up to kFusedWarpCells cells every block writes its own
// into all of them, else they are read from it), the candidate list, the absorbed
// lists (three species; a warp's share of them), the event keys of two species
__host__ __device__ constexpr size_t fused_smem(int nodes) {
  return (size_t)((nodes + 3) & ~3) *
             (8 + 4 + 12 + 12 + 16 + 8 * (nodes <= kFusedWarpCells + 1 ? kFusedMaxC : 1)) +
         (size_t)kFusedCand * 16 +
         (size_t)3 * kFusedList * 4 + (size_t)3 * kFusedWarps * kFusedWarpList * 4 +
         (size_t)2 * kEvCap * 8;
}

size_t fused_smem_bytes(int nodes) { return fused_smem(nodes); }

struct FusedShared {                   // static shared memory of k_fused
  InstConst ic;
  long long ws64[32];
  int ws32[32];
  int cnt[3];
  alignas(16) int wcnt[3][kFusedWarps];  // absorbed slots per warp (read by the cluster)
  int total[kFusedMaxC][4];            // absorbed slots of each block (written by them)
  int ncand, nemit;
  // window tallies of the collisions: at most 2^20 candidates a step and
  // kRouteSteps steps (64-bit shared adds are compare-and-swap loops, which a
  // warp of collisions enters 32 deep: 128 diodes of 20k particles 24.4 -> 22.9 us)
  unsigned coll[kTallies];
  long long wcount[6];                 // window tallies of the electrodes, as in InstDyn
  double wke[6];
  long long tcnt[3][kMaxParts][2];     // the step's, per part
  double tke[3][kMaxParts][2];
  double fA, fB;                       // the field's constants
  int cap[3];
  long long off[3];
  // what thread 0 keeps between the steps (in shared memory: a register held
  // over a cluster barrier may spill, and the barrier drops L1)
  long long step, pushed, win_steps, emitted, replenished;
  uint32_t base_id;
  int ids_out;
};

// Candidates and absorbed slots of up to four particles per lane, at slots
// slot + k (all 32 lanes call).
__device__ __forceinline__ void fused_events(FusedShared& S, uint4* cand, int sp, int slot,
                                             unsigned cm, unsigned dm, const float (&z)[4],
                                             const float (&v)[4], const uint32_t (&id)[4],
                                             uint32_t* wlist, uint32_t* dbuf, int& run, int lane) {
  if (cm) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (cm & (1u << k)) {
        const int at = atomicAdd(&S.ncand, 1);
        if (at < kFusedCand)
          cand[at] = make_uint4((unsigned)(slot + k) | ((unsigned)sp << 30), id[k],
                                __float_as_uint(z[k]), __float_as_uint(v[k]));
      }
  }
  const int dc = __popc(dm);
  int di = dc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, di, o);
    if (lane >= o) di += y;
  }
  int w = run + di - dc;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (dm & (1u << k)) {
      if (w < kFusedWarpList) wlist[w] = (uint32_t)(slot + k);
      else dbuf[w] = (uint32_t)(slot + k);
      ++w;
    }
  run += __shfl_sync(0xffffffffu, di, 31);
}

// Push of quads [wq0, wq1) of one segment by one warp; returns its absorbed
// slots' count (in slot order: the first kFusedWarpList in wlist, the rest at
// their places in dbuf).
__device__ __forceinline__ int fused_push(const DevState& st, FusedShared& S, const SegCtx& c,
                                          const float2* Es2, const Hist& hist, uint4* cand, int sp,
                                          long long off, int N, int wq0, int wq1, uint32_t* wlist,
                                          uint32_t* dbuf, int lane) {
  // (no __restrict__: these arrays change between steps, by other blocks too,
  // so their loads must not take the read-only path)
  float4* zp = reinterpret_cast<float4*>(st.z + off);
  float4* vp = reinterpret_cast<float4*>(st.vz + off);
  uint4* ip = reinterpret_cast<uint4*>(st.id + off);
  int run = 0;
  const int full = min(wq1, N >> 2);   // the segment's last quad may be partial
  float4 zn = make_float4(0.f, 0.f, 0.f, 0.f), vn = zn;
  uint4 in = make_uint4(0u, 0u, 0u, 0u);
  if (wq0 + lane < full) {
    zn = zp[wq0 + lane];
    vn = vp[wq0 + lane];
    in = ip[wq0 + lane];
  }
  for (int b = wq0; b < full; b += 32) {
    const int q = b + lane;
    float4 z4 = zn, v4 = vn;
    const uint4 i4 = in;
    if (q + 32 < full) {               // the next quad is in flight meanwhile
      zn = zp[q + 32];
      vn = vp[q + 32];
      in = ip[q + 32];
    }
    unsigned dm = 0u, cm = 0u;
    if (q < full) {
      push_quad(c, Es2, z4, v4, i4, dm, cm);
      zp[q] = z4;
      vp[q] = v4;
      if (dm == 0u) {
        deposit_quad(hist, z4, c.inv_dz, c.Nz, false);
      } else {
        const float z[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (!(dm & (1u << k))) {
            int j;
            float f;
            cell_of(z[k], c.inv_dz, c.Nz, j, f);
            hist_add(hist, j, frac_units(f));
          }
      }
    }
    if (__any_sync(0xffffffffu, (cm | dm) != 0u)) {
      const float z[4] = {z4.x, z4.y, z4.z, z4.w}, v[4] = {v4.x, v4.y, v4.z, v4.w};
      const uint32_t id[4] = {i4.x, i4.y, i4.z, i4.w};
      fused_events(S, cand, sp, 4 * q, cm, dm, z, v, id, wlist, dbuf, run, lane);
    }
  }
  if (full < wq1) {                    // at most one quad, the segment's last: a lane per particle
    const int i = 4 * full + lane;
    unsigned r = 0u;
    float z = 0.0f, v = 0.0f;
    uint32_t id = 0u;
    if (lane < 4 && i < N) {
      z = st.z[off + i];
      v = st.vz[off + i];
      id = st.id[off + i];
      r = push_one(c, Es2, z, v, id);
      st.z[off + i] = z;
      st.vz[off + i] = v;
      if (!(r & 1u)) {
        int j;
        float f;
        cell_of(z, c.inv_dz, c.Nz, j, f);
        hist_add(hist, j, frac_units(f));
      }
    }
    if (__any_sync(0xffffffffu, r != 0u)) {
      const float z1[4] = {z, 0.f, 0.f, 0.f}, v1[4] = {v, 0.f, 0.f, 0.f};
      const uint32_t id1[4] = {id, 0u, 0u, 0u};
      fused_events(S, cand, sp, i, (r >> 1) & 1u, r & 1u, z1, v1, id1, wlist, dbuf, run, lane);
    }
  }
  return run;
}

__device__ __forceinline__ void fused_collide(const DevState& st, FusedShared& S, int inst,
                                              long long slot, int sp, uint32_t id, float z,
                                              float vx, float vy, float vz, long long step) {
  const int code = collide(S.ic, st.dyn + inst, st.ev_buf + (long long)inst * kEvCap, sp, id, step,
                           z, vx, vy, vz);
  if (code != 0) {
    st.vx[slot] = vx;
    st.vy[slot] = vy;
    st.vz[slot] = vz;
  }
  if (step >= S.ic.window_start) {
    atomicAdd(&S.coll[code], 1u);
    atomicAdd(&S.coll[6 + sp], 1u);
  }
}

// An absorbed particle: its wall and kinetic energy.
struct FusedDead {
  long long c0, c1;
  double e0, e1;
};
__device__ __forceinline__ void fused_dead(const DevState& st, const InstConst& ic, int sp,
                                           long long off, uint32_t idx, FusedDead& d) {
  const double mw = 0.5 * ic.m_d[sp] * ic.weight;
  const float z = st.z[off + idx];
  const double vx = st.vx[off + idx], vy = st.vy[off + idx], vz = st.vz[off + idx];
  const double ke = mw * (vx * vx + vy * vy + vz * vz);
  if (z < 0.0f) { d.c0 += 1; d.e0 += ke; } else { d.c1 += 1; d.e1 += ke; }
}

// Sum over a warp as block_reduce4 takes it: shuffles down, the FP64 adds only
// if some lane holds an energy.  Valid in lane 0.
__device__ __forceinline__ void fused_warp_sum(FusedDead& d) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    d.c0 += __shfl_down_sync(0xffffffffu, d.c0, o);
    d.c1 += __shfl_down_sync(0xffffffffu, d.c1, o);
  }
  if (__any_sync(0xffffffffu, d.e0 != 0.0 || d.e1 != 0.0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      d.e0 += __shfl_down_sync(0xffffffffu, d.e0, o);
      d.e1 += __shfl_down_sync(0xffffffffu, d.e1, o);
    }
  }
}

// A part of the block's warps working as one block does: its threads' numbers
// and a named barrier.
struct FusedTeam {
  int tid, n, bar;
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory");
  }
};

// sort_events by a team: evb[0, E) by parent id, keys in evk
__device__ __forceinline__ void fused_sort_events(const FusedTeam& t, const Event* evb, int E,
                                                  unsigned long long* evk) {
  int P2 = 1;
  while (P2 < E) P2 <<= 1;
  for (int k = t.tid; k < P2; k += t.n)
    evk[k] = (k < E) ? (((unsigned long long)evb[k].parent << 32) | (unsigned)k) : ~0ull;
  t.sync();
  for (int kk = 2; kk <= P2; kk <<= 1)
    for (int jj = kk >> 1; jj > 0; jj >>= 1) {
      for (int i = t.tid; i < P2; i += t.n) {
        const int ixj = i ^ jj;
        if (ixj > i) {
          const unsigned long long a = evk[i], b = evk[ixj];
          const bool up = (i & kk) == 0;
          if ((a > b) == up) { evk[i] = b; evk[ixj] = a; }
        }
      }
      t.sync();
    }
}

// Hole filling and appends of one species by a team: what a block of k_post
// does.  dd: the species' D absorbed slots in order.  A thread's first move is
// looked up and loaded a phase ahead (fused_move), its first emitted electron
// (z, v) drawn there.
struct FusedMove {
  int to;                              // destination slot, -1: none
  float z, vx, vy, vz;
  uint32_t id;
};

__device__ __forceinline__ void fused_move(const DevState& st, int k, int N, int D, long long off,
                                           const uint32_t* dd, FusedMove& m) {
  m.to = -1;
  if (k >= D) return;
  const int Nn = N - D, t0 = Nn + k;
  const int a2 = lower_bound(dd, D, t0);
  if (a2 < D && (int)dd[a2] == t0) return;         // absorbed itself
  m.to = (int)dd[k - (a2 - lower_bound(dd, D, Nn))];
  const long long src = off + t0;
  m.z = st.z[src];
  m.vx = st.vx[src];
  m.vy = st.vy[src];
  m.vz = st.vz[src];
  m.id = st.id[src];
}

__device__ __forceinline__ void fused_post(const DevState& st, const InstConst& ic,
                                           const FusedTeam& t, int inst, int sp, int N, int D,
                                           int Di, int Nemit, long long step, uint32_t base_id,
                                           long long off, int cap, const uint32_t* dd,
                                           unsigned long long* evk, FusedMove& m,
                                           const float4& drawn) {
  const int Nn = N - D;
  int E = *(volatile int*)&st.dyn[inst].ev_count;   // all collisions are done
  for (int k = t.tid;;) {
    if (m.to >= 0) put_particle(st, off, m.to, m.z, m.vx, m.vy, m.vz, m.id);
    k += t.n;
    if (k >= D) break;
    fused_move(st, k, N, D, off, dd, m);
  }
  if (E > kEvCap) {
    if (t.tid == 0) atomicOr(&st.dyn[inst].err, ERR_CAPACITY);
    E = kEvCap;
  }
  t.sync();                            // tail slots are read
  bool overflow = false;
  const uint32_t id_emit = base_id + 2u * (uint32_t)E;
  if (sp == 0) {
    for (int k = t.tid; k < Nemit; k += t.n) {
      float z = drawn.x, vx = drawn.y, vy = drawn.z, vz = drawn.w;
      if (k != t.tid) emitted_electron(ic, k, step, z, vx, vy, vz);
      const long long sl = (long long)Nn + k;
      if (sl < cap) put_particle(st, off, sl, z, vx, vy, vz, id_emit + (uint32_t)k);
      else overflow = true;
    }
  } else {
    const bool ion = sp == 2;
    const uint32_t idb = ion ? 1u : 0u, id_repl = id_emit + (uint32_t)Nemit;
    const Event* evb = st.ev_buf + (long long)inst * kEvCap;
    if (E > 1) fused_sort_events(t, evb, E, evk);
    for (int k = t.tid; k < E; k += t.n) {
      const Event e = evb[E > 1 ? (int)(evk[k] & 0xffffffffu) : 0];
      const long long sl = (long long)Nn + k;
      if (sl < cap)
        put_particle(st, off, sl, e.z, ion ? e.vi[0] : e.ve[0], ion ? e.vi[1] : e.ve[1],
                     ion ? e.vi[2] : e.ve[2], base_id + 2u * k + idb);
      else
        overflow = true;
    }
    const int P = ic.replenish ? Di : 0;
    for (int k = t.tid; k < P; k += t.n) {
      float z, vx, vy, vz;
      replenished(ic, k, step, ion, z, vx, vy, vz);
      const long long sl = (long long)Nn + E + k;
      if (sl < cap) put_particle(st, off, sl, z, vx, vy, vz, id_repl + 2u * k + idb);
      else overflow = true;
    }
  }
  if (overflow) atomicOr(&st.dyn[inst].err, ERR_CAPACITY);
}

// The prefix of field_solve by one warp, for Nz <= kFusedWarpCells: rho (at
// fused_at) becomes G_j, and the constants of E_j = A + B (G_j + G_{j-1}) are
// left in S.  Lane l takes the nodes l c + u, u < c = ceil(Nz / 32); the
// padding of fused_at keeps those accesses off one another's banks.
__device__ __forceinline__ int fused_at(int j) { return j + (j >> 4); }

__device__ __forceinline__ void fused_field_prefix(FusedShared& S, long long* rho, int lane) {
  const InstConst& ic = S.ic;
  const int Nz = ic.Nz, c = (Nz + 31) >> 5, j0 = lane * c;
  long long loc = 0, wl = 0;
  for (int u = 0; u < c; ++u) {
    const int j = j0 + u;
    const long long v = (j >= 1 && j < Nz) ? rho[fused_at(j)] : 0LL;
    loc += v;
    wl += v * (long long)(Nz - j);
  }
  long long x = loc, y = wl;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long px = __shfl_up_sync(0xffffffffu, x, o);
    const long long py = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) {
      x += px;
      y += py;
    }
  }
  const long long Htot = __shfl_sync(0xffffffffu, y, 31);
  const double kap = ic.kappa;
  const double d0 = (ic.V + kap * (double)Htot) * ic.inv_nz;
  if (lane == 0) {
    S.fA = -d0 * ic.inv_dz;
    S.fB = 0.5 * kap * ic.inv_dz;
  }
  long long G = x - loc;
  for (int u = 0; u < c; ++u) {
    const int j = j0 + u;
    if (j < Nz) {
      if (j >= 1) G += rho[fused_at(j)];
      rho[fused_at(j)] = G;
    }
  }
}

// The charge of a block that holds more particles than its 32-bit histograms
// can (kHistMaxParticles): quads [lo, hi) of the diode's segments, pushed
// already, are binned again, kRebin at a time into sum (plain, not padded), and
// the block's node charge is written once more.  Replenishment adds a particle
// per absorbed ion, so nothing the route kernel could check bounds a diode's
// growth over its steps.
constexpr int kRebin = kHistMaxParticles / 2;

__device__ __noinline__ void fused_rebin(const DevState& st, const FusedShared& S, unsigned* hE,
                                         unsigned* hI, long long* sum, long long* node,
                                         int mn, int lo, int hi) {
  const InstConst& ic = S.ic;
  const Hist histE{hE}, histI{hI};
  const int Nz = ic.Nz, tid = threadIdx.x, nt = kFusedThreads;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  __syncthreads();                     // the histograms have been read
  for (int j = tid; j <= Nz; j += nt) sum[j] = 0;
  hist_zero(histE, Nz);
  hist_zero(histI, Nz);
  __syncthreads();
  int s0 = 0;
#pragma unroll 1
  for (int sp = 0; sp < 3; ++sp) {
    const int n = S.cnt[sp], s1 = s0 + ((n + 3) >> 2);
    const int end = min(4 * (min(hi, s1) - s0), n);
#pragma unroll 1
    for (int a = 4 * (max(lo, s0) - s0); a < end; a += kRebin) {
      const int b = min(end, a + kRebin);
      for (int i = a + tid; i < b; i += nt) {
        const float z = st.z[S.off[sp] + i];
        if (z >= 0.0f && z < ic.L_f) {
          int j;
          float f;
          cell_of(z, ic.inv_dz_f, Nz, j, f);
          hist_add(sp == 2 ? histI : histE, j, frac_units(f));
        }
      }
      __syncthreads();
      for (int j = tid; j <= Nz; j += nt)
        sum[j] += hist_node(histI, j, Nz) - hist_node(histE, j, Nz);
      __syncthreads();
      hist_zero(histE, Nz);
      hist_zero(histI, Nz);
      __syncthreads();
    }
    s0 = s1;
  }
  if (rank == C - 1)                   // the electrons of this step, as emit_charge binned them
    for (int k = tid; k < S.nemit; k += nt) {
      float z, vx, vy, vz, f;
      int j;
      emitted_electron(ic, k, S.step, z, vx, vy, vz);
      cell_of(z, ic.inv_dz_f, Nz, j, f);
      hist_add(histE, j, frac_units(f));
    }
  __syncthreads();
  for (int j = tid; j <= Nz; j += nt) {
    const long long v = sum[j] + hist_node(histI, j, Nz) - hist_node(histE, j, Nz);
    if (mn > 0) {
      for (int b = 0; b < C; ++b) cl.map_shared_rank(node, b)[rank * mn + j] = v;
    } else {
      node[j] = v;
    }
  }
}

// kRebins: a diode's room and its replenishment let a block outgrow its
// histograms within a launch (set_fused_shape).  A template, since the test
// alone cost every step of the others 0.1 of 10 us.
template <bool kRebins>
__device__ __forceinline__ void fused_body(const DevState& st, int n_steps) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ FusedShared S;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), last = C - 1;
  const int inst = (int)blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = kFusedThreads;
  const int mn = (st.max_nodes + 3) & ~3;
  float2* Es2 = reinterpret_cast<float2*>(smem);
  const bool warp_field = st.max_nodes <= kFusedWarpCells + 1;
  long long* node = reinterpret_cast<long long*>(smem + (size_t)mn * 8);    // [blocks or 1][mn]
  long long* rho_s = node + (warp_field ? kFusedMaxC : 1) * mn;    // [2 mn]: padded
  unsigned* hE = reinterpret_cast<unsigned*>(rho_s + 2 * mn);
  unsigned* hI = hE + 3 * mn;
  float* E = reinterpret_cast<float*>(hI + 3 * mn);
  uint4* cand = reinterpret_cast<uint4*>(E + mn);
  unsigned long long* evk = reinterpret_cast<unsigned long long*>(cand + kFusedCand);  // [2][kEvCap]
  uint32_t* dlist = reinterpret_cast<uint32_t*>(evk + 2 * kEvCap);          // [3][kFusedList]
  uint32_t* wlist = dlist + 3 * kFusedList;                                 // [3][warps][...]
  const Hist histE{hE}, histI{hI};
  InstDyn* dyn = st.dyn + inst;

  {
    const int* src = reinterpret_cast<const int*>(st.ic + inst);
    int* dst = reinterpret_cast<int*>(&S.ic);
    for (int w = tid; w < (int)(sizeof(InstConst) / 4); w += nt) dst[w] = src[w];
    if (tid < 3) {
      S.cnt[tid] = st.seg_count[3 * inst + tid];
      S.cap[tid] = st.seg_cap[3 * inst + tid];
      S.off[tid] = st.seg_off[3 * inst + tid];
    }
    if (tid < kTallies) S.coll[tid] = 0u;
    if (tid == 0) {
      S.ncand = 0;
      S.step = dyn->step;
      S.base_id = dyn->next_id;
      S.pushed = S.win_steps = S.emitted = S.replenished = 0;
      S.ids_out = 0;
    }
    if (tid < 6) {
      S.wcount[tid] = dyn->count[tid >> 1][tid & 1];
      S.wke[tid] = dyn->ke[tid >> 1][tid & 1];
    }
  }
  const auto off_of = [&](int sp) { return S.off[sp]; };
  __syncthreads();
  const InstConst& ic = S.ic;
  const int Nz = ic.Nz;
  // species s is finished by block s % C; its warps but the last are shared
  // out among the block's species
  const int post_n = C == 1 ? 3 : C == 2 ? 2 - rank : rank < 3 ? 1 : 0;
  const int team_warps = post_n > 0 ? kFusedTeamWarps / post_n : kFusedTeamWarps;
  const int team = warp / team_warps;
  const FusedTeam tm{tid - 32 * team_warps * team, 32 * team_warps, 1 + team};
  const int post_sp = rank + C * team;           // this team's species
  stage_field(Es2, st.E + ic.node_off, Nz);
  hist_zero(histE, Nz);
  hist_zero(histI, Nz);
  // The charge of the electrons a step emits goes into the last block's
  // histogram while the step before it ends: threads t, t + n, ...
  const auto emit_charge = [&](long long at, int t, int n) {
    const int Ne = emitted_count(ic, at);
    for (int k = t; k < Ne; k += n) {
      float z, vx, vy, vz, f;
      int j;
      emitted_electron(ic, k, at, z, vx, vy, vz);
      cell_of(z, ic.inv_dz_f, Nz, j, f);
      hist_add(histE, j, frac_units(f));
    }
  };
  __syncthreads();
  if (rank == last) emit_charge(S.step, tid, nt);
  cl.sync();                           // every block has read the state before any changes it

  for (int it = 0; it < n_steps; ++it) {
    // ---- A: push
    const long long step = S.step;
    const int n0 = S.cnt[0], n1 = S.cnt[1], n2 = S.cnt[2];
    const auto n_of = [&](int sp) { return sp == 0 ? n0 : sp == 1 ? n1 : n2; };
    if (tid == nt - 1) S.nemit = emitted_count(ic, step);
    if (tid == 0 && rank == 0) dyn->ev_count = 0;
    const int qs1 = (n0 + 3) >> 2, qs2 = qs1 + ((n1 + 3) >> 2), qs3 = qs2 + ((n2 + 3) >> 2);
    const auto qs_of = [&](int sp) { return sp == 0 ? 0 : sp == 1 ? qs1 : sp == 2 ? qs2 : qs3; };
    const int lo = (int)((long long)qs3 * rank / C), hi = (int)((long long)qs3 * (rank + 1) / C);
    int wq_first[3];                   // this warp's first quad of each segment
    int runs[3];                       // and its absorbed slots there
#pragma unroll
    for (int sp = 0; sp < 3; ++sp) wq_first[sp] = runs[sp] = 0;
#pragma unroll 1
    for (int sp = 0; sp < 3; ++sp) {
      const int s0 = qs_of(sp), s1 = qs_of(sp + 1);
      const int q0 = max(lo, s0) - s0, q1 = min(hi, s1) - s0;
      int run = 0, wq0 = 0;
      if (q0 < q1) {
        wq0 = (int)warp_start(q0, q1, warp, kFusedWarps);
        const int wq1 = (int)warp_start(q0, q1, warp + 1, kFusedWarps);
        SegCtx c;
        c.inv_dz = ic.inv_dz_f;
        c.Lf = ic.L_f;
        c.dt = ic.dt_f;
        c.qmdt = ic.qmdt[sp];
        c.Nz = Nz;
        c.tc = ic.t_cand[sp];
        c.ck = ic.ckey[sp];
        c.stepw = (uint32_t)step;
#pragma unroll
        for (int r = 0; r < 10; ++r) c.rk[r] = c.ck + (uint32_t)r * 0x9E3779B9u;
        run = fused_push(st, S, c, Es2, sp == 2 ? histI : histE, cand, sp, off_of(sp), n_of(sp), wq0,
                         wq1, wlist + (sp * kFusedWarps + warp) * kFusedWarpList,
                         st.dead_dense + off_of(sp) + 4 * wq0, lane);
      }
      if (sp == 0) { wq_first[0] = wq0; runs[0] = run; }
      else if (sp == 1) { wq_first[1] = wq0; runs[1] = run; }
      else { wq_first[2] = wq0; runs[2] = run; }
      if (lane == 0) S.wcnt[sp][warp] = run;
    }
    __syncthreads();
    for (int j = tid; j <= Nz; j += nt) {
      const long long v = hist_node(histI, j, Nz) - hist_node(histE, j, Nz);
      if (warp_field) {
#pragma unroll 2
        for (int b = 0; b < C; ++b) cl.map_shared_rank(node, b)[rank * mn + j] = v;
      } else {
        node[j] = v;
      }
    }
    if (kRebins && 4 * (hi - lo) + S.nemit > kHistMaxParticles)
      fused_rebin(st, S, hE, hI, rho_s, node, warp_field ? mn : 0, lo, hi);
    if (warp < 3) {
      const int x = lane < kFusedWarps ? S.wcnt[warp][lane] : 0;
      const int sum = __reduce_add_sync(0xffffffffu, x);
      if (lane < C) cl.map_shared_rank(&S.total[0][0], lane)[4 * rank + warp] = sum;
    }
    cl.sync();

    // ---- B: absorbed lists, charge, collisions
    const int nc = S.ncand, Nem = S.nemit;
    int D[3], start[3];
    {
      // this warp's first entry and the total: blocks and warps are in slot order
#pragma unroll
      for (int sp = 0; sp < 3; ++sp) {
        const int tb = lane < C ? S.total[lane][sp] : 0;
        const int tw = lane < warp ? S.wcnt[sp][lane] : 0;       // warp <= 15 < 32
        D[sp] = __reduce_add_sync(0xffffffffu, tb);
        start[sp] = __reduce_add_sync(0xffffffffu, (lane < rank ? tb : 0) + tw);
      }
    }
    const auto D_of = [&](int sp) { return sp == 0 ? D[0] : sp == 1 ? D[1] : D[2]; };
#pragma unroll
    for (int sp = 0; sp < 3; ++sp) {
      const int n = runs[sp];
      if (n == 0) continue;
      const uint32_t* near = wlist + (sp * kFusedWarps + warp) * kFusedWarpList;
      const uint32_t* far = st.dead_dense + S.off[sp] + 4 * wq_first[sp];
      uint32_t* to = D[sp] <= kFusedList ? cl.map_shared_rank(dlist + sp * kFusedList, sp % C)
                                         : st.dead_buf + S.off[sp];
      for (int k = lane; k < n; k += 32) to[start[sp] + k] = k < kFusedWarpList ? near[k] : far[k];
    }
    if (warp_field) {
      for (int j = tid; j <= Nz; j += nt) {
        long long v = 0;
#pragma unroll 4
        for (int b = 0; b < C; ++b) v += node[b * mn + j];
        rho_s[fused_at(j)] = v;
        if (rank == 0 && it == n_steps - 1) st.rho[ic.node_off + j] = v;
      }
    } else {
      // a slice of the nodes per block, summed from and written to all of them
      const int j0 = (int)((long long)(Nz + 1) * rank / C), j1 = (int)((long long)(Nz + 1) * (rank + 1) / C);
      for (int j = j0 + tid; j < j1; j += nt) {
        long long v = 0;
#pragma unroll 4
        for (int b = 0; b < C; ++b) v += cl.map_shared_rank(node, b)[j];
#pragma unroll 2
        for (int b = 0; b < C; ++b) cl.map_shared_rank(rho_s, b)[j] = v;
        if (it == n_steps - 1) st.rho[ic.node_off + j] = v;
      }
    }
    if (nc <= kFusedCand) {
      for (int k = nt - 1 - tid; k < nc; k += nt) {
        const uint4 cr = cand[k];
        const int sp = (int)(cr.x >> 30);
        const long long slot = off_of(sp) + (long long)(cr.x & 0x3fffffffu);
        fused_collide(st, S, inst, slot, sp, cr.y, __uint_as_float(cr.z), st.vx[slot], st.vy[slot],
                      __uint_as_float(cr.w), step);
      }
    } else {
      // more candidates than the list holds: the block looks through its
      // particles again (the test depends on id, step and the final z alone)
      if (nc > st.cand_cap && tid == 0) atomicOr(&dyn->err, ERR_CAPACITY);
#pragma unroll 1
      for (int sp = 0; sp < 3; ++sp) {
        const int s0 = qs_of(sp), s1 = qs_of(sp + 1);
        const int a = 4 * (max(lo, s0) - s0);
        const int b = min(4 * (min(hi, s1) - s0), n_of(sp));
        uint32_t rk[10];
#pragma unroll
        for (int r = 0; r < 10; ++r) rk[r] = ic.ckey[sp] + (uint32_t)r * 0x9E3779B9u;
        for (int i = a + tid; i < b; i += nt) {
          const long long slot = off_of(sp) + i;
          const float z = st.z[slot];
          const uint32_t id = st.id[slot];
          if (z >= 0.0f && z < ic.L_f && philox2x32_w0_rk(id, (uint32_t)step, rk) < ic.t_cand[sp])
            fused_collide(st, S, inst, slot, sp, id, z, st.vx[slot], st.vy[slot], st.vz[slot], step);
        }
      }
    }
    hist_zero(histE, Nz);              // the nodes hold what they counted
    hist_zero(histI, Nz);
    cl.sync();

    // ---- C: the field's prefix in the last warp; the absorbed particles'
    // energies, before their slots are reused; the moves that fill the slots
    // looked up and loaded.  Warp (species, part) of the last block takes
    // entries part + kp (t + 512 i) as thread t of k_mid's list block would,
    // so that the sums agree bit for bit; up to 32 entries stay in the lanes
    // over the barrier.
    if (warp_field && warp == kFusedWarps - 1) fused_field_prefix(S, rho_s, lane);
    const int kp = st.kp, item_sp = warp / kp, item_part = warp - kp * item_sp;
    const bool item = rank == last && warp < 3 * kp;
    FusedDead d{0, 0, 0.0, 0.0};
    if (item) {
      const int Di = D_of(item_sp);
      const int n_item = Di > item_part ? (Di - item_part + kp - 1) / kp : 0;
      const uint32_t* dd = Di <= kFusedList
                               ? cl.map_shared_rank(dlist + item_sp * kFusedList, item_sp % C)
                               : st.dead_buf + off_of(item_sp);
      if (n_item <= 32) {
        if (lane < n_item) fused_dead(st, ic, item_sp, off_of(item_sp), dd[item_part + kp * lane], d);
      } else {
        FusedDead sum{0, 0, 0.0, 0.0};           // lane v < 16: virtual warp v
        const int nv = min(kPostThreads / 32, (n_item + 31) >> 5);   // the others hold zeros
        for (int v = 0; v < nv; ++v) {
          FusedDead e{0, 0, 0.0, 0.0};
          for (int t = 32 * v + lane; t < n_item; t += kPostThreads)
            fused_dead(st, ic, item_sp, off_of(item_sp), dd[item_part + kp * t], e);
          fused_warp_sum(e);
          const long long c0 = __shfl_sync(0xffffffffu, e.c0, 0), c1 = __shfl_sync(0xffffffffu, e.c1, 0);
          const double e0 = __shfl_sync(0xffffffffu, e.e0, 0), e1 = __shfl_sync(0xffffffffu, e.e1, 0);
          if (lane == v) sum = FusedDead{c0, c1, e0, e1};
        }
        d = sum;
      }
    }
    const int Dp = team < post_n && warp < kFusedWarps - 1 ? D_of(post_sp) : 0;
    const uint32_t* dd_post = Dp <= kFusedList ? dlist + (team < post_n ? post_sp : 0) * kFusedList
                                               : st.dead_buf + off_of(post_sp);
    FusedMove mv;
    mv.to = -1;
    float4 drawn = make_float4(0.f, 0.f, 0.f, 0.f);
    if (team < post_n && warp < kFusedWarps - 1 && post_sp == 0 && tm.tid < Nem)
      emitted_electron(ic, tm.tid, step, drawn.x, drawn.y, drawn.z, drawn.w);
    if (Dp > 0) fused_move(st, tm.tid, n_of(post_sp), Dp, off_of(post_sp), dd_post, mv);
    if (!warp_field) {
      field_solve(ic, rho_s, E, nullptr, S.ws64);
    } else {
      __syncthreads();                 // the prefix
      const double A = S.fA, B = S.fB;
      for (int j = tid; j <= Nz; j += nt) {
        const long long gl = j > 0 ? rho_s[fused_at(j - 1)] : 0LL;
        const long long g = j < Nz ? rho_s[fused_at(j)] : gl;
        E[j] = (float)fma(B, (double)(j == 0 ? 0LL : g + gl), A);
      }
    }
    if (tid == 0) S.ncand = 0;         // every thread holds nc; the next push counts again
    cl.sync();

    // ---- D: hole filling, appends, tallies
    for (int j = tid; j < Nz; j += nt) Es2[j] = make_float2(E[j], E[j + 1] - E[j]);
    if (warp == kFusedWarps - 1) {
      if (rank == last) emit_charge(step + 1, lane, 32);
    } else if (team < post_n) {
      fused_post(st, ic, tm, inst, post_sp, n_of(post_sp), Dp, D[2], Nem, step, S.base_id,
                 off_of(post_sp), S.cap[post_sp], dd_post, evk + (post_sp == 2 ? kEvCap : 0), mv,
                 drawn);
    }
    if (item) {
      // (one virtual warp and zeros: the second level of the sum adds nothing)
      fused_warp_sum(d);
      if (lane == 0) {
        S.tcnt[item_sp][item_part][0] = d.c0;
        S.tcnt[item_sp][item_part][1] = d.c1;
        S.tke[item_sp][item_part][0] = d.e0;
        S.tke[item_sp][item_part][1] = d.e1;
      }
    }
    const int Ev = min(*(volatile int*)&dyn->ev_count, kEvCap);
    cl.sync();                         // the particles, the tallies
    // ---- the step closes: every block for itself
    const bool in_win = step >= ic.window_start;
    const int Pt = ic.replenish ? D[2] : 0;
    if (rank == last && in_win && tid >= 32 && tid < 38) {
      const int i = tid - 32;
      long long c = 0;
      double e = 0.0;
      for (int r = 0; r < kp; ++r) {
        c += S.tcnt[i >> 1][r][i & 1];
        e += S.tke[i >> 1][r][i & 1];
      }
      S.wcount[i] += c;
      S.wke[i] += e;
    }
    if (tid < 3) {
      const int add = tid == 0 ? Nem : Ev + Pt;
      S.cnt[tid] = min(n_of(tid) - D_of(tid) + add, S.cap[tid]);
    }
    if (tid == 64) {
      const uint32_t id0 = S.base_id;
      if ((unsigned long long)id0 + 2ull * (unsigned)Ev + (unsigned)Nem + 2ull * (unsigned)Pt >
          0xFFFFFFFFull)
        S.ids_out = 1;
      S.base_id = id0 + 2u * (uint32_t)Ev + (uint32_t)Nem + 2u * (uint32_t)Pt;
      S.pushed += (long long)n0 + n1 + n2;
      if (in_win) {
        S.win_steps += 1;
        S.emitted += Nem;
        S.replenished += Pt;
      }
      S.step = step + 1;
    }
    __syncthreads();
  }

  // ---- the state for whoever comes next
  if (rank == 0) {
    for (int j = tid; j <= Nz; j += nt) {
      st.E[ic.node_off + j] = E[j];
    }
    if (tid < 3) st.seg_count[3 * inst + tid] = S.cnt[tid];
    if (tid == 0) {
      dyn->step = S.step;
      dyn->next_id = S.base_id;
      dyn->pushed += S.pushed;
      dyn->win_steps += S.win_steps;
      dyn->emitted += S.emitted;
      dyn->replenished += S.replenished;
      if (S.ids_out) atomicOr(&dyn->err, ERR_CAPACITY);
    }
  }
  if (rank == last && tid < 6) {
    dyn->count[tid >> 1][tid & 1] = S.wcount[tid];
    dyn->ke[tid >> 1][tid & 1] = S.wke[tid];
  }
  if (tid < kTallies && S.coll[tid] != 0u)
    atomicAdd(tid < 6 ? &dyn->coll[tid] : &dyn->cand[tid - 6],
              (unsigned long long)S.coll[tid]);
  cl.sync();                           // no block leaves while its shared memory is read
}

__global__ void __launch_bounds__(kFusedThreads, 1) k_fused(DevState st, int n_steps) {
  fused_body<false>(st, n_steps);
}
__global__ void __launch_bounds__(kFusedThreads, 1) k_fused_rebins(DevState st, int n_steps) {
  fused_body<true>(st, n_steps);
}

// Which way the next steps run: 1 (the fused kernel) if its estimated time per
// step is the smaller.
// The fused kernel's histograms hold kHistMaxParticles per block, and a block
// with more bins its particles a second time (fused_rebin), so it is not taken
// where a diode with `growth` more (most that emission and ionisation can add
// over the steps; replenishment comes on top) would pass that, nor where the
// expected candidates come near the size of the three kernels' buffer, whose
// overflow is an error.
__global__ void k_route(DevState st, int C, int sms, long long growth, int n_steps,
                        cudaGraphConditionalHandle handle) {
  __shared__ float ws[6][32];
  float longest = 0.0f, most = 0.0f, emit = 0.0f, sum = 0.0f, cands = 0.0f, total = 0.0f;
  for (int i = threadIdx.x; i < st.n_inst; i += blockDim.x) {
    const InstConst& ic = st.ic[i];
    PostScratch& ps = st.post[i];
    int n = 0;
    float cand = 0.0f, dead = 0.0f;
    for (int sp = 0; sp < 3; ++sp) {
      const int ns = st.seg_count[3 * i + sp];
      n += ns;
      cand += (float)ns * ((float)ic.t_cand[sp] * 2.3283064e-10f);
    }
    // absorbed per step since the last decision: every particle that came has an
    // id (what an injection or a load makes of it only sways one choice)
    const long long step = st.dyn[i].step, past = step - ps.route_step;
    const uint32_t id = st.dyn[i].next_id;
    const long long gone = (long long)ps.route_n + (long long)(uint32_t)(id - ps.route_id) - n;
    if (past > 0 && past <= 4096 && gone > 0) dead = (float)gone / (float)past;
    ps.route_step = step;
    ps.route_n = n;
    ps.route_id = id;
    const DiodeLoad d{(float)n, (float)ic.emit_floor + (float)ic.t_frac * 2.3283064e-10f,
                      dead, cand};
    const float t = fused_estimate(d, C, st.kp, st.max_nodes);
    longest = fmaxf(longest, t);
    sum += t;
    most = fmaxf(most, (float)n);
    emit = fmaxf(emit, d.emit);
    cands += cand;
    total += d.n;
  }
  for (int o = 16; o > 0; o >>= 1) {
    longest = fmaxf(longest, __shfl_down_sync(0xffffffffu, longest, o));
    most = fmaxf(most, __shfl_down_sync(0xffffffffu, most, o));
    emit = fmaxf(emit, __shfl_down_sync(0xffffffffu, emit, o));
    sum += __shfl_down_sync(0xffffffffu, sum, o);
    cands += __shfl_down_sync(0xffffffffu, cands, o);
    total += __shfl_down_sync(0xffffffffu, total, o);
  }
  if ((threadIdx.x & 31) == 0) {
    const int w = threadIdx.x >> 5;
    ws[0][w] = longest;
    ws[1][w] = most;
    ws[2][w] = emit;
    ws[3][w] = sum;
    ws[4][w] = cands;
    ws[5][w] = total;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      longest = fmaxf(longest, ws[0][w]);
      most = fmaxf(most, ws[1][w]);
      emit = fmaxf(emit, ws[2][w]);
      sum += ws[3][w];
      cands += ws[4][w];
      total += ws[5][w];
    }
    const StepEstimate e = estimate_step(st.n_inst, longest, sum, total, cands, emit, C, sms);
    const bool one = e.fused < e.three && 2.0f * cands + 4096.0f < (float)st.cand_cap &&
                     (long long)most + growth < (long long)kHistMaxParticles;
    if (one) st.post[0].fused_steps += (uint32_t)n_steps;
    cudaGraphSetConditional(handle, one ? 1u : 0u);
  }
}

}  // namespace pic
