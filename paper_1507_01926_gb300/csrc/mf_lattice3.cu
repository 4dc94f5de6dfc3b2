// Lattice solver for volumes: a warp per tile (see mf_lattice.cuh).
//
// What bounds it: latency. On a volume about 1% of the cells of an active tile are
// active in a round, three or four of them, so a round is a short dependent chain
// on a few lanes. With a CTA per tile, nearly every warp has one active lane and
// all of them wait at the CTA barriers (a round took 1.3 us, four tiles per SM); a
// warp per tile runs the same round in 0.6 us, eight tiles per SM. A visit is
// about 16 us: 4 us to load 22 KB and take in the inboxes, ten rounds, 2.5 us to
// write the touched cells back and hand on to the neighbours. A scheduler issues
// an instruction every 8 cycles; of a warp's time a quarter is waiting for a tile
// (97x80x61 has fewer active tiles than the GPU has warps), a quarter loads, a
// third the dependent instructions and branches of the rounds.
// Measured, solve of 97x80x61 / 256x256x128: list solver 96 / 870 ms, a CTA per
// tile in sweeps 30 / 750 ms, this 33-41 / 375-480 ms by input.
#include "mf_lattice.cuh"
#include "mf_tile_queue.cuh"
#include "mf_internal.h"

#undef MF_FILE
#define MF_FILE 3

namespace mf {

namespace {

constexpr int DIM = 3;
using G = Geo<DIM>;
constexpr int LAT_ROUNDS = 16;  // push-relabel rounds per visit of a tile (8 and 32 measured 3-8% slower)

// A warp's tile.
struct __align__(16) LTile {
  int r[2 * DIM][TV];
  long long ex[TV];
  int drain[TV];
  int lab[G::PAD];  // labels with the halo
  unsigned lo[TV], hi[TV]; // excess received and not taken in yet: sums of the low 16 bits and of the rest
  union {
    unsigned short q[TV];    // the cells of this round
    int got[G::NH];   // while loading: amounts from the inbox, by face entry
  };
  __align__(16) unsigned char slots[TV];  // Lat::slots
  unsigned inq[TV / 32];   // bitmap of the cells of the next round
  int nt[8];               // tiles across the faces (-1: none)
};

// The tiles to visit are in a queue that all warps of the grid share
// (mf_tile_queue.cuh): no barrier between visits, and nobody waits for the longest
// visit of a sweep (with a grid barrier per sweep over the active tiles, warps
// spent three quarters of their time at it: one tile in a sweep of 500 used all
// its rounds, most a few). Queues of successive phases alternate between two
// buffers, and their counters between four sets; those of the phase before are
// cleared while the next one runs.
//
// The queue's memory operations.
struct QMem {
  const Dev *D;
  unsigned long long deadline;  // end of a push phase (%globaltimer)
  unsigned long long t0;

  __device__ __forceinline__ int add(int *p, int x) { return atomicAdd(p, x); }
  __device__ __forceinline__ int or_relaxed(int *p, int x) { return atomicOr(p, x); }
  __device__ __forceinline__ int or_acquire(int *p, int x) {
    int old;
    asm volatile("atom.acquire.gpu.global.or.b32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(x) : "memory");
    return old;
  }
  __device__ __forceinline__ int and_acquire(int *p, int x) {
    int old;
    asm volatile("atom.acquire.gpu.global.and.b32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(x) : "memory");
    return old;
  }
  __device__ __forceinline__ int exch_acquire(int *p, int x) {
    int old;
    asm volatile("atom.acquire.gpu.global.exch.b32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(x) : "memory");
    return old;
  }
  __device__ __forceinline__ unsigned cas(unsigned *p, unsigned expect, unsigned x) { return atomicCAS(p, expect, x); }
  __device__ __forceinline__ unsigned load(unsigned *p) { return *(volatile unsigned *)p; }
  __device__ __forceinline__ void store(unsigned *p, unsigned x) { *(volatile unsigned *)p = x; }
  __device__ __forceinline__ void release() { __threadfence(); }
  __device__ __forceinline__ void acquire() { __threadfence(); }
  // Wait for a place to become empty: given up when the phase ends (the warp whose
  // entry lies there may have left at the deadline, and the relabel that follows
  // queues afresh), after an error, and after D.timeout_ns.
  __device__ __forceinline__ bool wait(unsigned spins) {
    const unsigned long long now = lat_timer();
    if (spins == 1) t0 = now;
    if (now > deadline || *(volatile int *)&D->ctl->err) return false;
    if (now - t0 > D->timeout_ns) {
      lat_err(*D, MF_ERR_TIMEOUT, 4);
      return false;
    }
    __nanosleep(100);
    return true;
  }
};

// The queue of phase ph, which ends by itself or at the deadline.
__device__ __forceinline__ TileQueue<QMem> queue_of(const Dev &D, int ph, unsigned long long deadline = ~0ull) {
  return TileQueue<QMem>{reinterpret_cast<unsigned *>(D.lat.list[ph & 1]), &D.ctl->qhead[ph & 3], &D.ctl->qtail[ph & 3],
                         D.lat.state, D.lat.tiles, QMem{&D, deadline, 0}};
}

// Between phases: empties the queue the phase before `ph` left (a push phase may
// stop before its queue is empty) and its counters.
__device__ __forceinline__ void q_clear(const Dev &D, int ph) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
  if (tid == 0) D.ctl->qhead[(ph + 3) & 3] = D.ctl->qtail[(ph + 3) & 3] = D.ctl->qidle[(ph + 3) & 3] = 0;
  const TileQueue<QMem> q = queue_of(D, ph + 1);
  for (unsigned i = tid; i < q_slots(D.lat.tiles); i += nthr) *q.place(i) = 0;
}

// Takes the next tile (lane 0's work, the result in every lane); -1: the phase
// is over. It is when every warp of the grid waits and no place that one of them
// waits for is filled: head == tail + warps (idle warps queue nothing, so this
// does not change any more; the first warp of each CTA looks), or at the
// deadline, which a warp's first tile of a phase does not heed (every phase gets
// something done). A wait during which no tile is queued is bounded by
// D.timeout_ns, and a solve by LAT_EFFORT visits of this warp (a phase counts as
// eight: its barriers and set-up), which also keeps the grid's tickets below 2^32.
static __device__ int q_pop(const Dev &D, LShared &sh, int ph, bool timed, bool first, const LStat &st) {
  int t = -1;
  const bool over = st.tiles_dis + st.tiles_bfs + 8u * (unsigned)ph > (unsigned)LAT_EFFORT;
  if (over && (threadIdx.x & 31) == 0) lat_err(D, MF_ERR_ITER_LIMIT, 10);
  if ((threadIdx.x & 31) == 0 && !over && !(timed && !first && lat_timer() > sh.deadline)) {
    TileQueue<QMem> q = queue_of(D, ph);
    const unsigned ticket = q.ticket();
    const bool looks = threadIdx.x == 0;
    const int nwarps = (int)gridDim.x * LW;
    t = q.look(ticket);
    if (t < 0) {
      atomicAdd(&D.ctl->qidle[ph & 3], 1);
      unsigned long long t0 = lat_timer();
      int tail0 = 0;
      // plain loads some way apart, few of them of the shared counters
      for (unsigned spins = 1;; spins++) {
        __nanosleep(spins < 8 ? 100 : 400);
        t = q.look(ticket);
        if (t >= 0 || *(volatile int *)&sh.done) break;
        if (looks && (spins & 1)) {
          if (*(volatile int *)&D.ctl->qidle[ph & 3] == nwarps) {
            __threadfence();
            const int head = *(volatile int *)&D.ctl->qhead[ph & 3];
            __threadfence();
            if (head == *(volatile int *)&D.ctl->qtail[ph & 3] + nwarps) {
              *(volatile int *)&sh.done = 1;
              break;
            }
          }
        }
        if ((spins & 15) == 0) {
          const unsigned long long now = lat_timer();
          if (timed && now > sh.deadline) break;
          const int tail = *(volatile int *)&D.ctl->qtail[ph & 3];
          if (tail != tail0) {
            tail0 = tail;
            t0 = now;
          } else if (now - t0 > D.timeout_ns) {
            lat_err(D, MF_ERR_TIMEOUT, 4);
            break;
          }
          if (*(volatile int *)&D.ctl->err) break;
        }
      }
      if (t >= 0) atomicAdd(&D.ctl->qidle[ph & 3], -1);
    }
    if (t >= 0) q.take(ticket);
  }
  t = __shfl_sync(LFULL, t, 0);
  __syncwarp();  // (a shuffle does not order memory) lane 0's fence holds for all lanes
  return t;
}

// Starts the visit of tile t. Lane 0 gets the faces whose inbox holds something
// (shifted by FACES), which the warp reads later with q_faces: the exchange is in
// flight with the tile's loads.
__device__ __forceinline__ int q_begin(const Dev &D, int ph, int t) {
  return (threadIdx.x & 31) == 0 ? queue_of(D, ph).begin(MF_TILE(D, t)) : 0;
}
__device__ __forceinline__ int q_faces(int old) {
  old = __shfl_sync(LFULL, old, 0);
  __syncwarp();  // what lane 0 acquired, every lane sees
  return old >> FACES;
}

// Ends the visit of tile t: the tiles across the faces in `out` have work now, and
// t itself if `again`. All lanes; the warp's writes are released first.
__device__ __forceinline__ void q_done(const Dev &D, LTile &w, int ph, unsigned long long deadline, int t, unsigned out,
                                       bool again) {
  const int lane = threadIdx.x & 31;
  TileQueue<QMem> q = queue_of(D, ph, deadline);
  __syncwarp();  // also: the warp's tile may be overwritten
  __threadfence();
  int put = -1;
  if (lane < G::ND) {
    if (((out >> lane) & 1) && q.mark(MF_TILE(D, w.nt[lane]), 1 << (lane ^ 1))) put = w.nt[lane];
  } else if (lane == 31) {
    if (q.end(MF_TILE(D, t), again)) put = t;
  }
  __syncwarp();  // the pushes of all lanes together
  if (put >= 0) q.push(put, lane < 31);
  __syncwarp();  // the entries made are counted before lane 0 takes the next ticket
}

__device__ __forceinline__ void copy16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Labels of tile t and of the cells across its faces, into w.lab, and the tiles
// across its faces, into w.nt (the caller synchronises the warp).
__device__ __forceinline__ void load_labels(const Dev &D, LTile &w, int t) {
  const Lat &L = D.lat;
  const int lane = threadIdx.x & 31;
  const int nt = next_tile<DIM>(L, t, lane);
  if (lane < G::ND) w.nt[lane] = nt;
  int4 own[4];
#pragma unroll
  for (int i = 0; i < 4; i++)
    own[i] = __ldcg(reinterpret_cast<const int4 *>(&L.d[MF_CELL(D, (size_t)t * TV)]) + i * 32 + lane);
  int h[G::NH / 32];
#pragma unroll
  for (int i = 0; i < G::NH / 32; i++) {
    const int j = i * 32 / G::FS, f = i * 32 % G::FS + lane, q = __shfl_sync(LFULL, nt, j);
    h[i] = LINF;
    if (q >= 0) h[i] = __ldcg(&L.d[MF_CELL(D, (size_t)q * TV + G::cell(j ^ 1, f))]);
  }
#pragma unroll
  for (int i = 0; i < 4; i++) {  // four cells of one row
    const int p = G::pad(4 * (i * 32 + lane));
    w.lab[MF_LAB(D, p)] = own[i].x;
    w.lab[MF_LAB(D, p + 1)] = own[i].y;
    w.lab[MF_LAB(D, p + 2)] = own[i].z;
    w.lab[MF_LAB(D, p + 3)] = own[i].w;
  }
#pragma unroll
  for (int i = 0; i < G::NH / 32; i++) {
    const int j = i * 32 / G::FS, f = i * 32 % G::FS + lane;
    w.lab[MF_LAB(D, G::pad(G::cell(j, f)) + G::pstep(j))] = h[i];
  }
}

// Marks cell u for the next list.
__device__ __forceinline__ void mark(LTile &w, int u) {
  atomicOr(&w.inq[u >> 5], 1u << (u & 31));
}

// Appends one cell of every lane with `on` to the list of n cells.
__device__ __forceinline__ void put(LTile &w, int u, bool on, int &n) {
  const unsigned b = __ballot_sync(LFULL, on);
  if (on) w.q[n + __popc(b & ((1u << (threadIdx.x & 31)) - 1))] = (unsigned short)u;
  n += __popc(b);
}

// Adds a to the excess cell u receives: two 32-bit sums that 6 arcs cannot
// overflow (a 64-bit add to shared memory is a compare-and-swap loop).
__device__ __forceinline__ void give(LTile &w, int u, int a) {
  atomicAdd(&w.lo[u], (unsigned)a & 0xffffu);
  atomicAdd(&w.hi[u], (unsigned)a >> 16);
}

// Takes what cell u received.
__device__ __forceinline__ long long take(LTile &w, int u) {
  const unsigned l = w.lo[u], h = w.hi[u];
  w.lo[u] = 0;
  w.hi[u] = 0;
  return (long long)l + ((long long)h << 16);
}

// The marked cells become the warp's list (their number is returned, in every
// lane), join `touched` (lane i < 16: cells 32 i to 32 i + 31), and the marks are
// cleared.
__device__ __forceinline__ int next_list(LTile &w, unsigned &touched) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  unsigned x = lane < TV / 32 ? w.inq[lane] : 0;
  touched |= x;
  if (lane < TV / 32) w.inq[lane] = 0;
  const int c = __popc(x);
  int at = c;
#pragma unroll
  for (int o = 1; o < TV / 32; o <<= 1) {
    const int y = __shfl_up_sync(LFULL, at, o);
    if (lane >= o) at += y;
  }
  const int n = __shfl_sync(LFULL, at, TV / 32 - 1);
  at -= c;
  for (; x; x &= x - 1) w.q[at++] = (unsigned short)(lane * 32 + __ffs(x) - 1);
  __syncwarp();
  return n;
}

// A push over face j: the amount joins the inbox of the tile across it.
__device__ __forceinline__ void push_out(const Dev &D, const LTile &w, int j, int u, int a) {
  atomicAdd(&D.lat.inbox[MF_INBOX(D, (size_t)w.nt[j] * G::NH + (j ^ 1) * G::FS + G::face(j, u))], a);
}

// A round over the warp's list (n cells), 32 at a time, a lane per cell: every lane
// reads its cell and its neighbours' labels, relabels first if no residual arc
// leads to a lower label, and pushes along those that do. Excess left after that
// waits for the next round. (Pushing, relabeling and pushing again in one round
// took 5-10% longer on 97x80x61 and 256x256x128: fewer rounds, but the second pass
// ran in nearly all of them.) Returns the number of cells on the next list.
// Residuals change by atomics, as a relabeled cell and its neighbour may push over
// the same pair at once (then its labels are not valid in the sense of Section 2.1,
// which costs detours, not correctness). Nothing waits for an atomic's result: what
// a cell received and whether it is active next are sums and bits read in the next
// round.
__device__ __forceinline__ int push_round(const Dev &D, LTile &w, int t, int n, unsigned char *ret, unsigned &out,
                                          unsigned &touched, LStat &st) {
  const int lane = threadIdx.x & 31, cap = D.n_cap;
  for (int b = 0; b < n; b += 32) {
    const bool on = b + lane < n;
    const int u = w.q[on ? b + lane : 0], q = G::pad(u);
    const int du = w.lab[MF_LAB(D, q)];
    long long e = 0;
    int left = 0, dr = 0;
    int r[G::ND], dl[G::ND];
#pragma unroll
    for (int j = 0; j < G::ND; j++) {
      dl[j] = w.lab[MF_LAB(D, q + G::pstep(j))];
      r[j] = on ? w.r[j][u] : 0;
      st.scans_res += r[j] > 0;
    }
    if (on) {
      e = w.ex[u] + take(w, u);
      // at most INT_MAX leaves a cell per round, so the chain of pushes is 32-bit
      left = du < cap ? (int)min(e, (long long)INT_MAX) : 0;
      e -= left;
      dr = w.drain[u];
      st.visits_dis++;
      st.scans_dis += (w.slots[u] & 7) + ((w.slots[u] >> (ret ? 4 : 3)) & 1);
      st.scans_res += dr > 0;
      if (dr > 0 && left > 0) {  // the drain is an arc to label 0
        const int a = min(dr, left);
        w.drain[u] = dr -= a;
        left -= a;
        st.to_sink += a;
        st.pushes++;
        if (ret) ret[MF_CELL(D, (size_t)t * TV + u)] = 0x80;
      }
    }
    __syncwarp();  // every lane has read its cell
    int m = LINF;
#pragma unroll
    for (int j = 0; j < G::ND; j++) m = min(m, r[j] > 0 ? dl[j] : LINF);
    int lab = du;
    if (left > 0 && m >= lab) {
      lab = min(m + 1, LINF);
      st.relabels++;
    }
    const int can = lab < cap ? left : 0;
    e += left - can;
    left = can;
#pragma unroll
    for (int j = 0; j < G::ND; j++) {
      const int a = dl[j] < lab ? min(r[j], left) : 0;
      left -= a;
      if (a > 0) {
        st.pushes++;
        atomicAdd(&w.r[j][u], -a);
        if (G::inside(j, u)) {
          const int x = u + G::step(j);
          atomicAdd(&w.r[j ^ 1][x], a);
          give(w, x, a);
          mark(w, x);
        } else {
          push_out(D, w, j, u, a);
          out |= 1u << j;
        }
      }
    }
    if (on) {
      e += left;
      w.ex[u] = e;
      if (lab != du) w.lab[MF_LAB(D, q)] = lab;
      if (e > 0 && lab < cap) mark(w, u);
    }
    __syncwarp();
  }
  return next_list(w, touched);
}

// One visit of an active tile in phase `ph` by a warp: load, inboxes, rounds,
// store of the cells that took part; tiles that received excess, and the tile
// itself if it is still active, are queued. `drain` holds the residuals toward the phase's sink (t, then s); `ret`
// (phase 2) marks cells that returned excess to s.
//
// On a volume about 1% of the cells of an active tile are active in a round: with
// a CTA per tile and two cells per thread, nearly every warp had one active lane
// and a round took 1.3 us.
__device__ void push_visit(const Dev &D, LTile &w, int t, int ph, unsigned long long deadline, int *drain,
                           unsigned char *ret, LStat &st) {
  const Lat &L = D.lat;
  const int lane = threadIdx.x & 31, cap = D.n_cap;
  const int state = q_begin(D, ph, t);
#pragma unroll 4
  for (int i = 0; i < G::ND * TV / 128; i++)
    copy16(&w.r[0][0] + 4 * (i * 32 + lane), &L.r[MF_RES(D, (size_t)t * G::ND * TV + 4 * (i * 32 + lane))]);
#pragma unroll 4
  for (int i = 0; i < TV / 64; i++)
    copy16(&w.ex[2 * (i * 32 + lane)], &L.ex[MF_CELL(D, (size_t)t * TV + 2 * (i * 32 + lane))]);
#pragma unroll
  for (int i = 0; i < TV / 128; i++)
    copy16(&w.drain[4 * (i * 32 + lane)], &drain[MF_CELL(D, (size_t)t * TV + 4 * (i * 32 + lane))]);
  copy16(w.slots + 16 * lane, &L.slots[MF_CELL(D, (size_t)t * TV + 16 * lane)]);
  load_labels(D, w, t);  // (a halo older than the inbox is as good)
  const int bits = q_faces(state);
  if (bits) {
    int a[G::NH / 32];
#pragma unroll
    for (int i = 0; i < G::NH / 32; i++) {
      const int j = i * 32 / G::FS;
      a[i] = 0;
      if ((bits >> j) & 1) a[i] = atomicExch(&L.inbox[MF_INBOX(D, (size_t)t * G::NH + i * 32 + lane)], 0);
    }
#pragma unroll
    for (int i = 0; i < G::NH / 32; i++) w.got[i * 32 + lane] = a[i];
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  if (bits) {
#pragma unroll 1
    for (int k = lane; k < G::NH; k += 32) {
      const int a = w.got[k];
      if (a) {
        const int j = k / G::FS, u = G::cell(j, k % G::FS);
        w.r[j][u] += a;  // one entry per (face, cell)
        give(w, u, a);
        mark(w, u);
      }
    }
    __syncwarp();
  }
  unsigned active = 0;
#pragma unroll 4
  for (int i = 0; i < TV / 32; i++) {
    const unsigned b = __ballot_sync(LFULL, w.ex[i * 32 + lane] > 0 && w.lab[MF_LAB(D, G::pad(i * 32 + lane))] < cap);
    if (lane == i) active = b;
  }
  if (lane < TV / 32) w.inq[lane] |= active;
  unsigned out = 0, touched = 0;  // lane i of touched: cells 32 i ... 32 i + 31 to be written back
  int n = next_list(w, touched);
  for (int k = 0; k < LAT_ROUNDS && n > 0; k++) {
    n = push_round(D, w, t, n, ret, out, touched, st);
  }
  __syncwarp();
#pragma unroll 1
  for (int i = 0; i < TV / 32; i++) {
    const unsigned b = __shfl_sync(LFULL, touched, i);
    if ((b >> lane) & 1) {
      const int u = i * 32 + lane;
      const size_t at = (size_t)t * TV + u;
#pragma unroll
      for (int j = 0; j < G::ND; j++) L.r[MF_RES(D, ((size_t)t * G::ND + j) * TV + u)] = w.r[j][u];
      L.ex[MF_CELL(D, at)] = w.ex[u] + take(w, u);
      L.d[MF_CELL(D, at)] = w.lab[MF_LAB(D, G::pad(u))];
      drain[MF_CELL(D, at)] = w.drain[u];
    }
  }
  out = __reduce_or_sync(LFULL, out);
  q_done(D, w, ph, deadline, t, out, n > 0);
  st.tiles_dis += lane == 0;
}

// One visit of a tile in a BFS phase by a warp: cells take better labels over the
// faces that woke the tile, and cells whose label fell offer it on inside the
// tile until none does; neighbouring tiles that a lowered face label can improve are
// queued. Bit j of `mask`: the arc between the cell and its neighbour in
// direction j leads toward the seeds (global relabel: the cell's residual; cut:
// the neighbour's).
__device__ void bfs_visit(const Dev &D, LTile &w, int t, int ph, const unsigned char *mask, LStat &st) {
  const Lat &L = D.lat;
  const int lane = threadIdx.x & 31;
  unsigned char *mk = reinterpret_cast<unsigned char *>(w.ex);
  copy16(mk + 16 * lane, mask + (size_t)t * TV + 16 * lane);
  copy16(w.slots + 16 * lane, &L.slots[MF_CELL(D, (size_t)t * TV + 16 * lane)]);
  const int from = q_faces(q_begin(D, ph, t)), faces = from & 63;
  const bool seeds = from & (SEEDS >> FACES);
  load_labels(D, w, t);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  int n = 0;
  unsigned touched = 0;
#pragma unroll 1
  for (int f6 = faces; f6; f6 &= f6 - 1) {  // the tile is at its fixpoint but for what lies across these faces
    const int j = __ffs(f6) - 1;
#pragma unroll
    for (int f = lane; f < G::FS; f += 32) {
      const int u = G::cell(j, f), q = G::pad(u), x = w.lab[MF_LAB(D, q + G::pstep(j))] + 1;
      if (((mk[u] >> j) & 1) && x < w.lab[MF_LAB(D, q)]) {  // one entry per cell and face
        w.lab[MF_LAB(D, q)] = x;
        mark(w, u);
      }
    }
    __syncwarp();
  }
  n = next_list(w, touched);
  if (seeds) {  // first visit: every cell with a label offers it
    n = 0;
#pragma unroll 1
    for (int i = 0; i < TV / 32; i++) {
      const int u = i * 32 + lane;
      put(w, u, w.lab[MF_LAB(D, G::pad(u))] < LINF, n);
    }
    __syncwarp();
  }
  while (n > 0) {
    for (int b = 0; b < n; b += 32)
      if (b + lane < n) {
        const int u = w.q[b + lane], q = G::pad(u);
        const int l = w.lab[MF_LAB(D, q)] + 1;
        int x[G::ND];
        unsigned k[G::ND];
#pragma unroll
        for (int j = 0; j < G::ND; j++) {
          x[j] = w.lab[MF_LAB(D, q + G::pstep(j))];
          k[j] = G::inside(j, u) ? mk[u + G::step(j)] : 0;
        }
#pragma unroll
        for (int j = 0; j < G::ND; j++)
          if (((k[j] >> (j ^ 1)) & 1) && x[j] > l) {
            atomicMin(&w.lab[MF_LAB(D, q + G::pstep(j))], l);
            mark(w, u + G::step(j));
          }
        st.scans_bfs += w.slots[u] & 7;
        st.visits_bfs++;
      }
    n = next_list(w, touched);
  }
  __syncwarp();
#pragma unroll 1
  for (int i = 0; i < TV / 32; i++) {
    const unsigned b = __shfl_sync(LFULL, touched, i);
    if ((b >> lane) & 1) L.d[MF_CELL(D, (size_t)t * TV + i * 32 + lane)] = w.lab[MF_LAB(D, G::pad(i * 32 + lane))];
  }
  unsigned need = 0;
#pragma unroll
  for (int i = 0; i < G::NH / 32; i++) {
    const int j = i * 32 / G::FS, f = i * 32 % G::FS + lane;
    const int at = G::pad(G::cell(j, f));
    // (a halo cell without a tile has label LINF and no arc)
    if (w.nt[j] >= 0 && w.lab[MF_LAB(D, at)] + 1 < w.lab[MF_LAB(D, at + G::pstep(j))])
      need |= (unsigned)((__ldcg(&mask[MF_CELL(D, (size_t)w.nt[j] * TV + G::cell(j ^ 1, f))]) >> (j ^ 1)) & 1) << j;
  }
  need = __reduce_or_sync(LFULL, need);
  q_done(D, w, ph, ~0ull, t, need, false);
  st.tiles_bfs += lane == 0;
}

// One CTA of 8 warps per SM, a tile (28 KB) per warp.
__global__ void __launch_bounds__(LT, 1) lattice3_kernel(Dev D) {
  extern __shared__ __align__(16) unsigned char lat_smem[];
  __shared__ LShared sh;
  LTile &w = reinterpret_cast<LTile *>(lat_smem)[threadIdx.x >> 5];
  const Lat &L = D.lat;
  const int tid = blockIdx.x * LT + threadIdx.x, nthr = gridDim.x * LT;
  LStat st;
  if (threadIdx.x == 0) sh.bars = 0;
  for (int i = threadIdx.x & 31; i < TV; i += 32) w.lo[i] = w.hi[i] = 0;
  if ((threadIdx.x & 31) < TV / 32) w.inq[threadIdx.x & 31] = 0;
  __syncthreads();
  if (tid == 0) D.ctl->t_start = lat_timer();
  init_cells<DIM>(D);
  for (unsigned i = tid; i < q_slots(L.tiles); i += nthr) *queue_of(D, 0).place(i) = *queue_of(D, 1).place(i) = 0;
  bool ok = lat_sync(D, sh, 0);
  // Stages: phase 1 (excess toward t), phase 2 (what is left back to s), the cut.
  // A phase is a global relabel, visits until no tile is active or (gr_time_ratio)
  // they took longer than that many relabels, and so on until a relabel finds no
  // active cell. (One loop for all of it, so that the code of a visit exists
  // once.)
  const bool timer = tid == 0;
  int ph = 0;
  for (int stage = 1; ok; ph++) {
    const bool cutting = stage == 3;
    int *const drain = stage == 1 ? L.drain : L.back;
    const unsigned long long t0 = lat_timer();
    q_clear(D, ph);
    if (cutting) {
      const long long left = lat_sum(start_cut<DIM>(D, [&](int t) {
        L.state[MF_TILE(D, t)] = QUEUED | SEEDS;
        queue_of(D, ph).push(t, false);
      }), sh.sum);
      if (threadIdx.x == 0 && left) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&D.ctl->leftover), (unsigned long long)left);
        lat_err(D, MF_ERR_INTERNAL, 8);
      }
    } else {
      if (timer) D.ctl->grs++;
      start_relabel<DIM>(
          D, drain, [&](int t) { return __ldcg(&L.state[MF_TILE(D, t)]) >> FACES; },
          [&](int t, bool seeds) {
            L.state[MF_TILE(D, t)] = seeds ? QUEUED | SEEDS : 0;
            if (seeds) queue_of(D, ph).push(t, false);
          });
    }
    ok = lat_sync(D, sh, 2);
    if (!ok) break;
    const unsigned char *const mask = cutting ? L.ret : L.mask;
    for (int t; (t = q_pop(D, sh, ph, false, false, st)) >= 0;) bfs_visit(D, w, t, ph, mask, st);
    ok = lat_sync(D, sh, cutting ? 9 : 2);
    if (!ok || cutting) break;
    ph++;
    q_clear(D, ph);
    queue_active(D, [&](int t) {
      L.state[MF_TILE(D, t)] = QUEUED;
      queue_of(D, ph).push(t, false);
    });
    ok = lat_sync(D, sh, 3);
    if (!ok) break;
    const unsigned long long t1 = lat_timer();
    if (timer) D.ctl->t_gr += t1 - t0;
    if (__ldcg(&D.ctl->qtail[ph & 3]) == 0) {  // (nobody adds to it before the next barrier if it is 0)
      if (stage == 1) {  // the flow value: what the cells delivered to t
        const long long x = lat_sum(st.to_sink, sh.sum), vis = lat_sum((long long)st.tiles_dis, sh.sum);
        if (threadIdx.x == 0) {
          if (x) atomicAdd(reinterpret_cast<unsigned long long *>(&D.ctl->value), (unsigned long long)x);
          if (vis) atomicAdd(reinterpret_cast<unsigned long long *>(&D.ctl->rounds_phase1), (unsigned long long)vis);
        }
        if (timer) D.ctl->t_preflow = lat_timer();
      }
      stage = stage == 1 && !D.cut_only ? 2 : 3;
      continue;
    }
    // every CTA times its own relabel: they end at the same barrier, and which warp stops when changes no result
    if (threadIdx.x == 0) sh.deadline = t1 + (unsigned long long)fmin(D.gr_time_ratio * (double)(t1 - t0), 1e18);
    __syncthreads();
    unsigned char *const ret = stage == 2 ? L.ret : nullptr;
    bool first = true;
    for (int t; (t = q_pop(D, sh, ph, true, first, st)) >= 0; first = false) push_visit(D, w, t, ph, sh.deadline, drain, ret, st);
    ok = lat_sync(D, sh, 4);
    if (timer) D.ctl->t_dis += lat_timer() - t1;
  }
  if (ok) write_outputs<DIM>(D);
  add_stats(D, sh, st);
  if (tid == 0) D.ctl->t_end = lat_timer();
}

}  // namespace

const void *lattice3_fn() { return (const void *)lattice3_kernel; }
// Bytes of one tile queue.
size_t lattice_queue_bytes(int tiles) {
  return (size_t)q_slots(tiles) * Q_STRIDE * 4;
}
size_t lattice3_smem() { return LW * sizeof(LTile); }

}  // namespace mf
