#pragma once
// What the two lattice solvers share (mf_lattice2.cu: images, a CTA per tile;
// mf_lattice3.cu: volumes, a warp per tile): geometry, grid barrier, set-up,
// relabel and cut preparation, outputs.
//
// The problem and the outputs are those of mf_solver.cuh, for single graphs that
// are lattices: the vertices other than s and t, numbered in order without those
// two, are the cells of a row-major box X x Y (x Z), and every arc joins
// neighbouring cells or a cell and s or t, at most one slot per direction and
// terminal (found on the device when the graph is created, mf_lattice.cu). A
// cell's neighbours are then known from its place, and the cells are kept in
// tiles of 512 (32 x 16 or 8 x 8 x 8).
//
// Why tiles: the list solver runs one round of Algorithm 1 per grid barrier. On
// a 256x256x128 volume that is 50,000 rounds and 13,000 BFS phases of 7-50 us,
// each a chain of dependent L2 and DRAM round trips, whatever the number of
// vertices in it. A tile's state fits a CTA's (or a warp's) shared memory and
// registers; a visit loads it, runs several rounds on it without leaving the SM,
// and writes it back. Excess crosses a whole tile per visit, and a BFS label too.
//
//  * Inside a tile a cell pushes along residual arcs to lower labels and relabels
//    (one above the least residual neighbour): in 2D after the push, with excess
//    left, and pushes once more; in 3D before it, when no such arc is there. Cells
//    of a tile do so at the same time on labels that may be one round old, as in
//    the paper's synchronous rounds, and without its win rule: a label may then
//    rise past the distance, which costs detours, not correctness.
//  * A push over a tile face uses the neighbour's label as it was when the tile
//    was loaded, takes the residual from the pusher's side at once and adds the
//    amount to the receiver's inbox; it joins the receiver's excess and its side
//    of the arc when its tile is next loaded. Until then the receiver
//    underestimates its residual, which only delays it. (Amounts fit int32: they
//    come out of one residual.)
//  * Global relabel: exact distances by label-correcting relaxation, a tile to
//    its fixpoint per visit, tiles whose neighbour's face improved visited again.
//    The labels are those of Algorithm 2's BFS.
//  * A phase ends, as in the list solver, when a global relabel (which takes in
//    every inbox) finds no vertex with excess and a finite label. Whatever the
//    order of pushes before that, the result is a maximum preflow (phase 1) or a
//    flow (phase 2, the excess that is left back to s), so the value and S_min
//    are exact.
//  * That a solve ends is not proven: between two relabels labels only rise, but one
//    that rose past its distance falls at the next relabel, and the list solver's
//    argument (rounds whose labels stay below the distances) does not hold. So a
//    solve is given up after LAT_EFFORT sweeps (2D) or visits of one warp (3D), far
//    beyond any measured (256x256x128: 20,000 visits a warp), and the host runs the
//    list solver on the graph.
#include <cuda_runtime.h>
#include <limits.h>

#include "mf.h"
#include "mf_check.cuh"
#include "mf_device.cuh"

#undef MF_FILE
#define MF_FILE 1

namespace mf {

namespace {

constexpr unsigned LFULL = 0xffffffffu;
constexpr int LT = 256;      // threads per CTA
constexpr int LW = LT / 32;
constexpr int TV = 512;      // cells per tile: 32 x 16 or 8 x 8 x 8
constexpr int LINF = UNV;    // label of a cell that does not reach the sink
#ifndef MF_LATTICE_EFFORT      // (a test builds it with less)
#define MF_LATTICE_EFFORT 2000000
#endif
constexpr int LAT_EFFORT = MF_LATTICE_EFFORT;

template <int DIM>
struct Geo {
  static constexpr int ND = 2 * DIM;               // directions: -x, +x, -y, +y (, -z, +z)
  static constexpr int FS = DIM == 3 ? 64 : 32;    // entries per face (a 2D x face uses 16)
  static constexpr int EX = DIM == 3 ? 8 : 32;     // tile extents
  static constexpr int EY = DIM == 3 ? 8 : 16;
  static constexpr int NH = ND * FS;

  static __device__ __forceinline__ int stride(int j) { return j < 2 ? 1 : j < 4 ? EX : EX * EY; }
  // cell u's neighbour in direction j lies in the same tile
  static __device__ __forceinline__ bool inside(int j, int u) {
    if (j == 0) return (u & (EX - 1)) > 0;
    if (j == 1) return (u & (EX - 1)) < EX - 1;
    const int y = DIM == 3 ? (u >> 3) & 7 : u >> 5;
    if (j == 2) return y > 0;
    if (j == 3) return y < EY - 1;
    return j == 4 ? u >= 64 : u < TV - 64;
  }
  static __device__ __forceinline__ int step(int j) { return (j & 1) ? stride(j) : -stride(j); }
  // labels of a tile with its halo, one cell wide on every side
  static constexpr int PX = EX + 2, PY = EY + 2;
  static constexpr int PAD = PX * PY * (DIM == 3 ? 10 : 1);
  static __device__ __forceinline__ int pad(int u) {
    return DIM == 3 ? ((u >> 6) + 1) * (PX * PY) + (((u >> 3) & 7) + 1) * PX + (u & 7) + 1 : ((u >> 5) + 1) * PX + (u & 31) + 1;
  }
  static __device__ __forceinline__ int pstep(int j) {
    const int w = j < 2 ? 1 : j < 4 ? PX : PX * PY;
    return (j & 1) ? w : -w;
  }
  // entry of cell u on face j
  static __device__ __forceinline__ int face(int j, int u) {
    if (DIM == 2) return j < 2 ? u >> 5 : u & 31;
    return j < 2 ? u >> 3 : j < 4 ? (u >> 6) * 8 + (u & 7) : u & 63;
  }
  static __device__ __forceinline__ bool face_entry(int j, int f) { return DIM == 3 || j >= 2 || f < EY; }
  // cell of entry f on face j
  static __device__ __forceinline__ int cell(int j, int f) {
    if (DIM == 2) return j == 0 ? f * 32 : j == 1 ? f * 32 + 31 : j == 2 ? f : TV - 32 + f;
    switch (j) {
      case 0: return f * 8;
      case 1: return f * 8 + 7;
      case 2: return (f >> 3) * 64 + (f & 7);
      case 3: return (f >> 3) * 64 + 56 + (f & 7);
      case 4: return f;
      default: return TV - 64 + f;
    }
  }
};

// State of a CTA between tiles.
struct LShared {
  unsigned long long bars;
  int err;                     // control words as they stood at the last grid barrier
  int cnt, req;                // (2D) tiles of the next sweep, relabel request
  int done;                    // (3D) the phase's queue has run dry
  unsigned long long deadline; // (3D) end of a push phase (%globaltimer)
  int tick;
  long long sum[LW];
};

__device__ __forceinline__ unsigned long long lat_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long lat_acquire(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void lat_err(const Dev &D, int code, int where) {
  if (atomicCAS(&D.ctl->err, 0, code) == 0) atomicExch(&D.ctl->err_where, where);
}

// Grid barrier (as the list solver's grid_sync): every wait is bounded by
// D.timeout_ns. Shares the error word, the size of tile list `gen` and the
// relabel request of sweep `sweep` with the CTA. False after an error.
static __device__ bool lat_sync(const Dev &D, LShared &sh, int where, int gen = 0, int sweep = 0) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long *c = reinterpret_cast<unsigned long long *>(&D.ctl->bar);
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(c), "l"(1ULL) : "memory");
    const unsigned long long target = (sh.bars + 1) * (unsigned long long)gridDim.x;
    if (lat_acquire(c) < target) {
      const unsigned long long t0 = lat_timer();
      unsigned spins = 0;
      while (lat_acquire(c) < target) {
        if ((++spins & 31u) == 0 && lat_timer() - t0 > D.timeout_ns) {
          lat_err(D, MF_ERR_TIMEOUT, where);
          break;
        }
        __nanosleep(20);
      }
    }
    sh.bars++;
    const int e = __ldcg(&D.ctl->err), n = __ldcg(&D.ctl->cnt[gen & 3]), q = __ldcg(&D.ctl->gr_req[sweep & 1]);
    sh.err = e;
    sh.cnt = n;
    sh.req = q;
    sh.done = 0;
  }
  __syncthreads();
  return sh.err == 0;
}

// Tile adjacent to t over face j, -1 if none.
template <int DIM>
__device__ __forceinline__ int next_tile(const Lat &L, int t, int j) {
  const int tx = t % L.TX, q = t / L.TX, ty = q % L.TY, tz = q / L.TY;
  const int at = j < 2 ? tx : j < 4 ? ty : tz, end = j < 2 ? L.TX : j < 4 ? L.TY : L.TZ;
  const int st = j < 2 ? 1 : j < 4 ? L.TX : L.TX * L.TY;
  return (j & 1) ? (at + 1 < end ? t + st : -1) : (at > 0 ? t - st : -1);
}

// Scans count what a lattice solve looks at. Volumes: slots of the graph (Lat::slots),
// of a discharged cell those to its neighbours and the one to the phase's sink, in
// a BFS those to the neighbours of a cell that offers its label. Images: directions,
// with a slot or without, the drain among them once per visit of a cell; in a BFS
// those of all cells of a visited tile once per visit (counting slots cost 2-4% of a
// solve there: 64 registers, and a round's work is little more than the count).
struct LStat {
  unsigned tiles_dis = 0, tiles_bfs = 0;  // visits of tiles
  unsigned scans_dis = 0, scans_res = 0, scans_bfs = 0, pushes = 0, relabels = 0, visits_dis = 0, visits_bfs = 0;
  long long to_sink = 0;
};

// Start of a global relabel toward `drain`: inboxes taken in, residual masks set
// up, label 1 where the drain is open. faces(t): the faces whose inbox holds
// something; seed(t, b) (lane 0): whether tile t has such cells.
template <int DIM, typename F, typename S>
__device__ __forceinline__ void start_relabel(const Dev &D, const int *drain, F faces, S seed_tile) {
  using G = Geo<DIM>;
  const Lat &L = D.lat;
  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x, nwarps = (int)gridDim.x * LW;
  for (int t = warp; t < L.tiles; t += nwarps) {
    const int bits = faces(t);
    bool seed = false;
    if (bits) {
#pragma unroll 1
      for (int k = lane; k < G::NH; k += 32) {
        const int j = k / G::FS, f = k % G::FS;
        if (!((bits >> j) & 1) || !G::face_entry(j, f)) continue;
        const int a = __ldcg(&L.inbox[MF_INBOX(D, (size_t)t * G::NH + k)]);
        if (a) {
          const int u = G::cell(j, f);
          L.inbox[MF_INBOX(D, (size_t)t * G::NH + k)] = 0;
          int *const r = &L.r[MF_RES(D, ((size_t)t * G::ND + j) * TV + u)];
          *r = __ldcg(r) + a;
          atomicAdd(reinterpret_cast<unsigned long long *>(&L.ex[MF_CELL(D, (size_t)t * TV + u)]), (unsigned long long)a);
        }
      }
      __syncwarp();
    }
#pragma unroll 2
    for (int i = 0; i < TV / 128; i++) {
      const int u = 4 * (i * 32 + lane);
      const int4 dr = __ldcg(reinterpret_cast<const int4 *>(&drain[MF_CELL(D, (size_t)t * TV + u)]));
      unsigned m = 0;
#pragma unroll
      for (int j = 0; j < G::ND; j++) {
        const int4 r = __ldcg(reinterpret_cast<const int4 *>(&L.r[MF_RES(D, ((size_t)t * G::ND + j) * TV + u)]));
        m |= ((unsigned)(r.x > 0) | (unsigned)(r.y > 0) << 8 | (unsigned)(r.z > 0) << 16 | (unsigned)(r.w > 0) << 24) << j;
      }
      *reinterpret_cast<unsigned *>(&L.mask[MF_CELL(D, (size_t)t * TV + u)]) = m;
      *reinterpret_cast<int4 *>(&L.d[MF_CELL(D, (size_t)t * TV + u)]) =
          make_int4(dr.x > 0 ? 1 : LINF, dr.y > 0 ? 1 : LINF, dr.z > 0 ? 1 : LINF, dr.w > 0 ? 1 : LINF);
      seed |= dr.x > 0 || dr.y > 0 || dr.z > 0 || dr.w > 0;
    }
    seed = __any_sync(LFULL, seed);
    if (lane == 0) seed_tile(t, seed);
  }
}

// Calls queue(t) (lane 0) for the tiles with an active cell.
template <typename F>
__device__ __forceinline__ void queue_active(const Dev &D, F queue) {
  const Lat &L = D.lat;
  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x, nwarps = (int)gridDim.x * LW;
  for (int t = warp; t < L.tiles; t += nwarps) {
    bool a = false;
#pragma unroll 4
    for (int i = 0; i < TV / 64; i++) {
      const size_t at = (size_t)t * TV + 2 * (i * 32 + lane);
      const longlong2 e = __ldcg(reinterpret_cast<const longlong2 *>(&L.ex[MF_CELL(D, at)]));
      const int2 d = __ldcg(reinterpret_cast<const int2 *>(&L.d[MF_CELL(D, at)]));
      a |= (e.x > 0 && d.x < LINF) || (e.y > 0 && d.y < LINF);
    }
    if (__any_sync(LFULL, a) && lane == 0) queue(t);
  }
}

// Start of the cut's BFS. Seeds are the cells s reaches directly (those that
// returned excess to it), with cut_only those that kept excess; arcs lead from
// the neighbour to the cell, so bit j of the mask is the neighbour's residual
// (taken from the residual masks of the last global relabel, after which nothing
// was pushed). Calls queue(t) (thread 0) for the tiles with a seed; returns this
// thread's count of cells that kept excess though
// phase 2 is over.
template <int DIM, typename F>
__device__ __forceinline__ long long start_cut(const Dev &D, F queue) {
  using G = Geo<DIM>;
  const Lat &L = D.lat;
  long long left = 0;
  for (int t = blockIdx.x; t < L.tiles; t += gridDim.x) {
    bool seed = false;
#pragma unroll 1
    for (int u = threadIdx.x; u < TV; u += LT) {
      const size_t at = (size_t)t * TV + u;
      unsigned m = 0;
#pragma unroll
      for (int j = 0; j < G::ND; j++) {
        size_t q;
        if (G::inside(j, u)) {
          q = at + G::step(j);
        } else {
          const int nt = next_tile<DIM>(L, t, j);
          if (nt < 0) continue;
          q = (size_t)nt * TV + G::cell(j ^ 1, G::face(j, u));
        }
        m |= ((__ldcg(&L.mask[MF_CELL(D, q)]) >> (j ^ 1)) & 1u) << j;
      }
      const long long e = __ldcg(&L.ex[MF_CELL(D, at)]);
      const bool sd = D.cut_only ? e > 0 : __ldcg(&L.ret[MF_CELL(D, at)]) != 0;
      if (!D.cut_only && e != 0) left++;
      L.ret[MF_CELL(D, at)] = (unsigned char)m;  // from here on the mask of the cut
      L.d[MF_CELL(D, at)] = sd ? 0 : LINF;
      seed |= sd;
    }
    if (__syncthreads_or(seed) && threadIdx.x == 0) queue(t);
  }
  return left;
}

// Cell index of vertex v, and vertex of cell p.
__device__ __forceinline__ int cell_of(const Lat &L, int v) { return v - (v > L.s) - (v > L.t); }
__device__ __forceinline__ int vertex_of(const Lat &L, int p) {
  const int lo = min(L.s, L.t), hi = max(L.s, L.t);
  int v = p + (p >= lo);
  return v + (v >= hi);
}

// Place of cell p in the tiled arrays.
template <int DIM>
__device__ __forceinline__ size_t place_of(const Lat &L, int p) {
  if (DIM == 2) {
    const int x = p % L.X, y = p / L.X;
    return (size_t)((y >> 4) * L.TX + (x >> 5)) * TV + (y & 15) * 32 + (x & 31);
  }
  const int x = p % L.X, q = p / L.X, y = q % L.Y, z = q / L.Y;
  return (size_t)(((z >> 3) * L.TY + (y >> 3)) * L.TX + (x >> 3)) * TV + (z & 7) * 64 + (y & 7) * 8 + (x & 7);
}

// Cell at place u of tile t, -1 outside the box or past the last cell.
template <int DIM>
__device__ __forceinline__ int cell_at(const Lat &L, int t, int u) {
  const int tx = t % L.TX, ty = (t / L.TX) % L.TY, tz = t / (L.TX * L.TY);
  const int x = tx * Geo<DIM>::EX + (u & (Geo<DIM>::EX - 1));
  const int y = ty * Geo<DIM>::EY + (DIM == 3 ? (u >> 3) & 7 : u >> 5);
  const int z = DIM == 3 ? tz * 8 + (u >> 6) : 0;
  if (x >= L.X || y >= L.Y || z >= L.Z) return -1;
  const long long p = ((long long)z * L.Y + y) * L.X + x;
  return p < L.cells ? (int)p : -1;
}

// Direction of the arc from cell p to cell q (they are neighbours).
template <int DIM>
__device__ __forceinline__ int dir_of(const Lat &L, int p, int q) {
  const int x = q - p;
  if (x == 1 || x == -1) return x > 0;
  if (DIM == 2) return 2 + (x > 0);
  return x == L.X ? 3 : x == -L.X ? 2 : 4 + (x > 0);
}

// Sum over the CTA (in every thread).
__device__ __forceinline__ long long lat_sum(long long x, long long *buf) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(LFULL, x, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = x;
  __syncthreads();
  long long s = 0;
  for (int i = 0; i < LW; i++) s += buf[i];
  __syncthreads();
  return s;
}

// Initialisation with the source's arcs saturated: every cell's residuals from
// its row, excess from s, an empty inbox.
template <int DIM>
__device__ __forceinline__ void init_cells(const Dev &D) {
  using G = Geo<DIM>;
  const Lat &L = D.lat;
  for (int t = blockIdx.x; t < L.tiles; t += gridDim.x) {
    for (int c = 0; c < 2; c++) {
      const int u = threadIdx.x + c * LT, p = cell_at<DIM>(L, t, u);
      long long ex = 0;
      int dr = 0, rs = 0, slots = 0, r[G::ND];
#pragma unroll
      for (int j = 0; j < G::ND; j++) r[j] = 0;
      if (p >= 0) {
        const int v = vertex_of(L, p);
        const int b = __ldg(&D.row[MF_ROW(D, v)]), e = __ldg(&D.row[MF_ROW(D, v + 1)]);
        for (int a = b; a < e; a++) {
          const int w = __ldg(&D.head[MF_SLOT(D, a)]), cp = __ldg(&D.cap[MF_SLOT(D, a)]);
          if (w == L.t) {
            dr = cp;
            slots += 8;
          } else if (w == L.s) {
            slots += 16;
            const int cs = __ldg(&D.cap[MF_SLOT(D, __ldg(&D.rev[MF_SLOT(D, a)]))]);
            rs = cp + cs;
            ex = cs;
          } else {
            const int jj = dir_of<DIM>(L, p, cell_of(L, w));
            slots++;
#pragma unroll
            for (int j = 0; j < G::ND; j++)
              if (j == jj) r[j] = cp;
          }
        }
      }
      const size_t at = (size_t)t * TV + u;
      L.ex[MF_CELL(D, at)] = ex;
      L.drain[MF_CELL(D, at)] = dr;
      L.back[MF_CELL(D, at)] = rs;
      L.ret[MF_CELL(D, at)] = 0;
      if (DIM == 3) L.slots[MF_CELL(D, at)] = (unsigned char)slots;
#pragma unroll
      for (int j = 0; j < G::ND; j++) L.r[MF_RES(D, ((size_t)t * G::ND + j) * TV + u)] = r[j];
    }
    for (int k = threadIdx.x; k < G::NH; k += LT) L.inbox[MF_INBOX(D, (size_t)t * G::NH + k)] = 0;
    if (threadIdx.x == 0) L.state[MF_TILE(D, t)] = L.bits[MF_BITS(D, t)] = L.bits[MF_BITS(D, (size_t)L.tiles + t)] = 0;
  }
}

// Value, cut bitmap and per-slot flows of a finished solve.
template <int DIM>
__device__ __forceinline__ void write_outputs(const Dev &D) {
  using G = Geo<DIM>;
  const Lat &L = D.lat;
  const int tid = blockIdx.x * LT + threadIdx.x, nthr = gridDim.x * LT;
  if (tid == 0 && D.out_value) D.out_value[0] = __ldcg(&D.ctl->value);
  if (D.out_cut) {
    const int words = (D.n + 31) >> 5, lane = threadIdx.x & 31;
    for (int wd = tid >> 5; wd < words; wd += nthr >> 5) {
      const int v = wd * 32 + lane;
      const bool in =
          v < D.n && v != L.t && (v == L.s || __ldcg(&L.d[MF_CELL(D, place_of<DIM>(L, cell_of(L, v)))]) < LINF);
      const unsigned b = __ballot_sync(LFULL, in);
      if (lane == 0) D.out_cut[wd] = b;
    }
  }
  if (D.out_flow)
    for (int p = tid; p < L.cells; p += nthr) {
      const int v = vertex_of(L, p);
      const size_t at = place_of<DIM>(L, p);
      const size_t rt = at / TV * G::ND * TV + at % TV;
      const int b = __ldg(&D.row[MF_ROW(D, v)]), e = __ldg(&D.row[MF_ROW(D, v + 1)]);
      for (int a = b; a < e; a++) {
        const int w = __ldg(&D.head[MF_SLOT(D, a)]), cp = __ldg(&D.cap[MF_SLOT(D, a)]);
        if (w == L.t) {
          D.out_flow[MF_SLOT(D, a)] = cp - __ldcg(&L.drain[MF_CELL(D, at)]);
          D.out_flow[MF_SLOT(D, __ldg(&D.rev[MF_SLOT(D, a)]))] = 0;
        } else if (w == L.s) {
          const int net = __ldcg(&L.back[MF_CELL(D, at)]) - cp;  // flow s -> p
          D.out_flow[MF_SLOT(D, a)] = max(-net, 0);
          D.out_flow[MF_SLOT(D, __ldg(&D.rev[MF_SLOT(D, a)]))] = max(net, 0);
        } else {
          const int res = __ldcg(&L.r[MF_RES(D, rt + (size_t)dir_of<DIM>(L, p, cell_of(L, w)) * TV)]);
          D.out_flow[MF_SLOT(D, a)] = max(cp - res, 0);
        }
      }
    }
}

// Adds a thread's counters to the control block (all threads call).
static __device__ __forceinline__ void add_stats(const Dev &D, LShared &sh, const LStat &st) {
  const unsigned cnts[9] = {st.tiles_dis, st.tiles_bfs, st.scans_dis, st.scans_res, st.scans_bfs, st.pushes, st.relabels, st.visits_dis, st.visits_bfs};
  long long *dst[9] = {&D.ctl->rounds, &D.ctl->levels, &D.ctl->scans_dis, &D.ctl->scans_res, &D.ctl->scans_bfs, &D.ctl->pushes,
                       &D.ctl->relabels, &D.ctl->visits_dis, &D.ctl->visits_bfs};
#pragma unroll
  for (int i = 0; i < 9; i++) {
    const long long x = lat_sum((long long)cnts[i], sh.sum);
    if (threadIdx.x == 0 && x) atomicAdd(reinterpret_cast<unsigned long long *>(dst[i]), (unsigned long long)x);
  }
}

}  // namespace

}  // namespace mf
