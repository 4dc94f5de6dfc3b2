// Lattice solver for images: a CTA per tile, sweeps over the active tiles with a
// grid barrier between them (see mf_lattice.cuh).
//
// What bounds it: a solve is some 20 sweeps and 20 BFS sweeps of 5-20 us, most of
// that the rounds of the busiest tile. On an image most cells are active at first
// (every pixel has a terminal arc), so a tile keeps 256 threads busy; a warp per
// tile, as for volumes, takes two to three times as long (64x64: 0.35 ms against
// 0.14 ms; 1024x1024: 1.05 ms against 0.72 ms).
#include "mf_lattice.cuh"
#include "mf_internal.h"

#undef MF_FILE
#define MF_FILE 2

namespace mf {

namespace {

constexpr int DIM = 2;
using G = Geo<DIM>;
constexpr int LAT_ROUNDS = 8;  // push-relabel rounds per visit of a tile (16: 5-15% slower, 32: 20-70%)

// A CTA's tile.
struct CTile {
  int lab[G::PAD];  // labels with the halo
  int delta[2 * DIM][TV];  // amount cell u pushed in direction j this round
  int flag[TV];            // directions from which cell u received this round
  int nt[2 * DIM];         // tiles across the faces (-1: none)
  int out, need;
};

// Queues tile t for sweep `sweep` (list generation gen), once.
__device__ __forceinline__ void queue_tile(const Dev &D, int t, int sweep, int gen) {
  if (atomicExch(&D.lat.state[MF_TILE(D, t)], sweep) != sweep) {
    const int i = atomicAdd(&D.ctl->cnt[gen & 3], 1);
    if (i < D.lat.tiles)
      D.lat.list[gen & 1][MF_TILE(D, i)] = t;
    else
      lat_err(D, MF_ERR_INTERNAL, 11);
  }
}

// CTA 0 clears the counters of the list generation after next.
__device__ __forceinline__ void clear_next(const Dev &D, int gen) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    D.ctl->cnt[(gen + 2) & 3] = 0;
    D.ctl->lcnt[(gen + 2) & 3] = 0;
  }
}

// The tiles of list generation gen (n of them), one after another: the first
// by block index, the rest by ticket (a visit takes between one and LAT_ROUNDS
// rounds).
template <typename F>
__device__ __forceinline__ void for_tiles(const Dev &D, LShared &sh, int gen, int n, F f) {
  clear_next(D, gen);
  for (int i = blockIdx.x; i < n;) {
    int nx = 0;
    if (threadIdx.x == 0) nx = (int)gridDim.x + atomicAdd(&D.ctl->lcnt[gen & 3], 1);
    f(__ldcg(&D.lat.list[gen & 1][MF_TILE(D, i)]));
    __syncthreads();  // the visit's shared state may be overwritten
    if (threadIdx.x == 0) sh.tick = nx;
    __syncthreads();
    i = sh.tick;
  }
}

// Labels of the cells across the tile's faces.
__device__ __forceinline__ void load_halo(const Dev &D, CTile &w, int t) {
  const Lat &L = D.lat;
  const int tx = t % L.TX, ty = t / L.TX;
  for (int k = threadIdx.x; k < G::NH; k += LT) {
    const int j = k / G::FS, f = k % G::FS;
    if (!G::face_entry(j, f)) continue;
    const bool up = j & 1;
    const int at = j < 2 ? tx : ty, end = j < 2 ? L.TX : L.TY, st = j < 2 ? 1 : L.TX;
    const bool there = up ? at + 1 < end : at > 0;
    const int n = up ? t + st : t - st;
    w.lab[MF_LAB(D, G::pad(G::cell(j, f)) + G::pstep(j))] =
        there ? __ldcg(&L.d[MF_CELL(D, (size_t)n * TV + G::cell(j ^ 1, f))]) : LINF;
  }
}

// One visit of an active tile in sweep `sweep` (list generation gen): load,
// inboxes, rounds, store; tiles that received excess, and the tile itself if it
// is still active, are queued for the next sweep. `drain` holds the residuals
// toward the phase's sink (t, then s); `ret` (phase 2) marks cells that returned
// excess to s.
//
// A thread holds two cells' residuals and excess in registers for the whole
// visit and shares only labels: a push leaves its amount in `delta` and a bit at
// the receiver, who adds it to its own registers after the CTA barrier. (With
// residuals and 64-bit excess in shared memory, updated by the pusher, a round
// was a chain of dependent shared-memory accesses and took 2 us instead of 1.)
__device__ void push_visit(const Dev &D, CTile &w, int t, int sweep, int gen, int *drain, unsigned char *ret,
                           LStat &st) {
  const Lat &L = D.lat;
  const int bits = __ldcg(&L.bits[MF_BITS(D, (size_t)(sweep & 1) * L.tiles + t)]);
  int r[2][G::ND], d[2], dr[2];
  long long ex[2];
  unsigned in[2], ch = 0;  // directions that stay in the tile; bits c, 2 + c, 4 + c: residuals/excess, label, drain changed
#pragma unroll
  for (int c = 0; c < 2; c++) {
    const int u = threadIdx.x + c * LT;
    const size_t at = (size_t)t * TV + u;
#pragma unroll
    for (int j = 0; j < G::ND; j++) r[c][j] = __ldcg(&L.r[MF_RES(D, ((size_t)t * G::ND + j) * TV + u)]);
    ex[c] = __ldcg(&L.ex[MF_CELL(D, at)]);
    d[c] = __ldcg(&L.d[MF_CELL(D, at)]);
    dr[c] = __ldcg(&drain[MF_CELL(D, at)]);
    in[c] = 0;
#pragma unroll
    for (int j = 0; j < G::ND; j++) in[c] |= (unsigned)G::inside(j, u) << j;
    w.flag[u] = 0;
  }
  if (threadIdx.x < G::ND) w.nt[threadIdx.x] = next_tile<DIM>(L, t, threadIdx.x);
  load_halo(D, w, t);
  if (threadIdx.x == 0) w.out = 0;
  if (bits) {  // uniform in the CTA
#pragma unroll
    for (int c = 0; c < 2; c++)
#pragma unroll
      for (int j = 0; j < G::ND; j++)
        if ((bits >> j) & 1 & ~(in[c] >> j)) {
          const int a =
              atomicExch(&L.inbox[MF_INBOX(D, (size_t)t * G::NH + j * G::FS + G::face(j, threadIdx.x + c * LT))], 0);
          r[c][j] += a;
          ex[c] += a;
          ch |= 1u << c;
        }
  }
#pragma unroll
  for (int c = 0; c < 2; c++) w.lab[MF_LAB(D, G::pad(threadIdx.x + c * LT))] = d[c];
  __syncthreads();  // every thread has read the tile's bits
  if (bits && threadIdx.x == 0) L.bits[MF_BITS(D, (size_t)(sweep & 1) * L.tiles + t)] = 0;
  const int cap = D.n_cap;
  unsigned outb = 0;
  for (int k = 0; k < LAT_ROUNDS; k++) {
    bool any = false;
#pragma unroll
    for (int c = 0; c < 2; c++) {
      if (ex[c] <= 0 || d[c] >= cap) continue;
      const int u = threadIdx.x + c * LT, q = G::pad(u);
      any = true;
      st.visits_dis++;
      st.scans_dis += G::ND + 1;
      int dl[G::ND];
#pragma unroll
      for (int j = 0; j < G::ND; j++) dl[j] = w.lab[MF_LAB(D, q + G::pstep(j))];
      int left = (int)min(ex[c], (long long)INT_MAX);
      ex[c] -= left;
      ch |= 1u << c;
      if (dr[c] > 0) {
        const int a = min(dr[c], left);
        dr[c] -= a;
        left -= a;
        st.to_sink += a;
        st.pushes++;
        ch |= 16u << c;
        if (ret) ret[MF_CELL(D, (size_t)t * TV + u)] = 0x80;
      }
#pragma unroll 1
      for (int pass = 0; left > 0; pass++) {
        int m = LINF;
#pragma unroll
        for (int j = 0; j < G::ND; j++) {
          const int a = dl[j] < d[c] ? min(r[c][j], left) : 0;
          if (a > 0) {
            left -= a;
            r[c][j] -= a;
            st.pushes++;
            if ((in[c] >> j) & 1) {
              w.delta[j][u] = a;
              atomicOr(&w.flag[u + G::step(j)], 1 << (j ^ 1));
            } else {
              atomicAdd(&L.inbox[MF_INBOX(D, (size_t)w.nt[j] * G::NH + (j ^ 1) * G::FS + G::face(j, u))], a);
              outb |= 1u << j;
            }
          }
          if (r[c][j] > 0) m = min(m, dl[j]);
        }
        if (left == 0 || m + 1 <= d[c]) break;
        d[c] = min(m + 1, LINF);
        w.lab[MF_LAB(D, q)] = d[c];
        ch |= 4u << c;
        st.relabels++;
        if (pass || d[c] >= cap) break;
      }
      ex[c] += left;
    }
    if (!__syncthreads_or(any)) break;
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const int u = threadIdx.x + c * LT;
      const int f = w.flag[u];
      if (f) {
        w.flag[u] = 0;
        ch |= 1u << c;
#pragma unroll
        for (int j = 0; j < G::ND; j++)
          if ((f >> j) & 1) {
            const int a = w.delta[j ^ 1][u + G::step(j)];
            r[c][j] += a;
            ex[c] += a;
          }
      }
    }
    __syncthreads();
  }
  if (outb) atomicOr(&w.out, (int)outb);
  const bool act = __syncthreads_or((ex[0] > 0 && d[0] < cap) || (ex[1] > 0 && d[1] < cap));
#pragma unroll
  for (int c = 0; c < 2; c++) {
    const int u = threadIdx.x + c * LT;
    const size_t at = (size_t)t * TV + u;
    if ((ch >> c) & 1) {
#pragma unroll
      for (int j = 0; j < G::ND; j++) L.r[MF_RES(D, ((size_t)t * G::ND + j) * TV + u)] = r[c][j];
      L.ex[MF_CELL(D, at)] = ex[c];
    }
    if ((ch >> (2 + c)) & 1) L.d[MF_CELL(D, at)] = d[c];
    if ((ch >> (4 + c)) & 1) drain[MF_CELL(D, at)] = dr[c];
  }
  if (threadIdx.x < G::ND && ((w.out >> threadIdx.x) & 1)) {
    const int q = w.nt[threadIdx.x];
    atomicOr(&L.bits[MF_BITS(D, (size_t)((sweep + 1) & 1) * L.tiles + q)], 1 << (threadIdx.x ^ 1));
    queue_tile(D, q, sweep + 1, gen + 1);
  }
  if (threadIdx.x == 32 && act) queue_tile(D, t, sweep + 1, gen + 1);
}

// One visit of a tile in a BFS sweep: labels relaxed to the tile's fixpoint;
// neighbours that a lowered face label can improve are queued. Bit j of `mask`:
// the arc between the cell and its neighbour in direction j leads toward the
// seeds (global relabel: the cell's residual; cut: the neighbour's).
__device__ void bfs_visit(const Dev &D, CTile &w, int t, int sweep, int gen, const unsigned char *mask, LStat &st) {
  const Lat &L = D.lat;
  int d0[2], d[2];
  unsigned mk[2];
#pragma unroll
  for (int c = 0; c < 2; c++) {
    const size_t at = (size_t)t * TV + threadIdx.x + c * LT;
    d0[c] = d[c] = __ldcg(&L.d[MF_CELL(D, at)]);
    mk[c] = __ldcg(&mask[MF_CELL(D, at)]);
  }
  if (threadIdx.x < G::ND) w.nt[threadIdx.x] = next_tile<DIM>(L, t, threadIdx.x);
  load_halo(D, w, t);
  if (threadIdx.x == 0) w.need = 0;
#pragma unroll
  for (int c = 0; c < 2; c++) w.lab[MF_LAB(D, G::pad(threadIdx.x + c * LT))] = d[c];
  __syncthreads();
  bool ch;
  do {
    ch = false;
#pragma unroll
    for (int rep = 0; rep < 2; rep++)  // labels only fall: reading a neighbour's old or new one is both right
#pragma unroll
      for (int c = 0; c < 2; c++) {
        const int q = G::pad(threadIdx.x + c * LT);
        int m = LINF;
#pragma unroll
        for (int j = 0; j < G::ND; j++) {
          const int x = *(volatile int *)&w.lab[MF_LAB(D, q + G::pstep(j))];
          if ((mk[c] >> j) & 1) m = min(m, x);
        }
        if (m + 1 < d[c]) {
          d[c] = m + 1;
          *(volatile int *)&w.lab[MF_LAB(D, q)] = d[c];
          ch = true;
        }
      }
  } while (__syncthreads_or(ch));
#pragma unroll
  for (int c = 0; c < 2; c++)
    if (d[c] != d0[c]) L.d[MF_CELL(D, (size_t)t * TV + threadIdx.x + c * LT)] = d[c];
  st.scans_bfs += 2 * G::ND;
  st.visits_bfs += 2;
  unsigned need = 0;
  for (int k = threadIdx.x; k < G::NH; k += LT) {
    const int j = k / G::FS, f = k % G::FS;
    const int q = w.nt[j];
    if (q < 0 || !G::face_entry(j, f)) continue;
    const int at = G::pad(G::cell(j, f));
    if (w.lab[MF_LAB(D, at)] + 1 < w.lab[MF_LAB(D, at + G::pstep(j))] &&
        ((__ldcg(&mask[MF_CELL(D, (size_t)q * TV + G::cell(j ^ 1, f))]) >> (j ^ 1)) & 1))
      need |= 1u << j;
  }
  if (need) atomicOr(&w.need, (int)need);
  __syncthreads();
  if (threadIdx.x < G::ND && ((w.need >> threadIdx.x) & 1)) queue_tile(D, w.nt[threadIdx.x], sweep + 1, gen + 1);
}

// Relaxes labels from the tiles of list generation gen on; false after an error.
__device__ __forceinline__ bool bfs_sweeps(const Dev &D, LShared &sh, CTile &w, int &sweep, int &gen,
                                           const unsigned char *mask, LStat &st) {
  while (sh.cnt > 0) {
    for_tiles(D, sh, gen, sh.cnt, [&](int t) { bfs_visit(D, w, t, sweep, gen, mask, st); });
    if (blockIdx.x == 0 && threadIdx.x == 0) st.tiles_bfs++;
    if (!lat_sync(D, sh, 2, gen + 1)) return false;
    gen++;
    sweep++;
  }
  return true;
}

// Four CTAs per SM (64 registers): visits wait for memory first and for CTA
// barriers after, so other tiles' visits have to fill both.
__global__ void __launch_bounds__(LT, 4) lattice2_kernel(Dev D) {
  __shared__ CTile w;
  __shared__ LShared sh;
  const Lat &L = D.lat;
  LStat st;
  const bool timer = blockIdx.x == 0 && threadIdx.x == 0;
  if (threadIdx.x == 0) sh.bars = 0;
  if (timer) D.ctl->t_start = lat_timer();
  init_cells<DIM>(D);
  bool ok = lat_sync(D, sh, 0);
  // Stages: phase 1 (excess toward t), phase 2 (what is left back to s), the cut.
  // A phase is a global relabel, sweeps until no tile is active or (gr_time_ratio)
  // they took longer than that many relabels, and so on until a relabel finds no
  // active cell.
  int sweep = 1, gen = 0;
  long long rounds = 0;
  for (int stage = 1; ok;) {
    const bool cutting = stage == 3;
    int *const drain = stage == 1 ? L.drain : L.back;
    const unsigned long long t0 = lat_timer();
    auto queue = [&](int t) { queue_tile(D, t, sweep + 1, gen + 1); };
    auto next = [&](int where) {  // the tiles queued become the list
      ok = lat_sync(D, sh, where, gen + 1, sweep);
      gen++;
      sweep++;
      return ok;
    };
    clear_next(D, gen);
    if (cutting) {
      const long long left = lat_sum(start_cut<DIM>(D, queue), sh.sum);
      if (threadIdx.x == 0 && left) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&D.ctl->leftover), (unsigned long long)left);
        lat_err(D, MF_ERR_INTERNAL, 8);
      }
      if (!next(9)) break;
      ok = bfs_sweeps(D, sh, w, sweep, gen, L.ret, st);
      break;
    }
    if (timer) D.ctl->grs++;
    start_relabel<DIM>(
        D, drain,
        [&](int t) { return __ldcg(&L.bits[MF_BITS(D, t)]) | __ldcg(&L.bits[MF_BITS(D, (size_t)L.tiles + t)]); },
        [&](int t, bool seeds) {
          L.bits[MF_BITS(D, t)] = L.bits[MF_BITS(D, (size_t)L.tiles + t)] = 0;
          if (seeds) queue(t);
        });
    if (!next(2)) break;
    if (!(ok = bfs_sweeps(D, sh, w, sweep, gen, L.mask, st))) break;
    clear_next(D, gen);
    queue_active(D, queue);
    if (!next(3)) break;
    const unsigned long long t1 = lat_timer();
    if (timer) D.ctl->t_gr += t1 - t0;
    if (sh.cnt == 0) {
      if (stage == 1) {  // the flow value: what the cells delivered to t
        const long long x = lat_sum(st.to_sink, sh.sum);
        if (threadIdx.x == 0 && x) atomicAdd(reinterpret_cast<unsigned long long *>(&D.ctl->value), (unsigned long long)x);
        if (timer) {
          D.ctl->t_preflow = lat_timer();
          D.ctl->rounds_phase1 = rounds;
        }
      }
      stage = stage == 1 && !D.cut_only ? 2 : 3;
      continue;
    }
    do {
      rounds++;
      if (sweep > LAT_EFFORT) {  // (here only: a relabel ends by itself, as labels only fall in it)
        lat_err(D, MF_ERR_ITER_LIMIT, 10);
        ok = false;
        break;
      }
      if (timer) {
        D.ctl->gr_req[sweep & 1] = (double)(lat_timer() - t1) > D.gr_time_ratio * (double)(t1 - t0);
        st.tiles_dis++;
      }
      unsigned char *const ret = stage == 2 ? L.ret : nullptr;
      for_tiles(D, sh, gen, sh.cnt, [&](int t) { push_visit(D, w, t, sweep, gen, drain, ret, st); });
    } while (next(4) && sh.cnt > 0 && !sh.req);
    if (timer) D.ctl->t_dis += lat_timer() - t1;
  }
  if (ok) write_outputs<DIM>(D);
  add_stats(D, sh, st);
  if (timer) D.ctl->t_end = lat_timer();
}

}  // namespace

const void *lattice2_fn() { return (const void *)lattice2_kernel; }

}  // namespace mf
