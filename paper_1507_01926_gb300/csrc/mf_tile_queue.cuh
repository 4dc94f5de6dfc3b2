#pragma once
// The queue of tiles that the warps of a volume solve share (mf_lattice3.cu).
//
// A tile is queued at most once. Its state word: QUEUED (it is in the queue, or,
// while RUNNING, to be queued again after its visit), RUNNING (a warp has it),
// and above them the faces whose inbox holds something (in a BFS: beyond which a
// label fell) and, in a BFS, whether cells of the tile are seeds. A ticket (head)
// names the place a warp waits for; an entry (tail) fills the next place.
//
// Places are reused in turn, and an entry may still lie in its place when the
// ring comes round to it, if the warp with its ticket has not looked since. So
// an entry carries its lap, which only the ticket of that lap takes, and is
// written only into an empty place. Fewer entries than places are out at a time
// (a tile has one at most), so the ticket of an entry in the way has been drawn
// and its warp is looking: the wait ends when it does.
//
// What a visit wrote is handed on twice: over the tile's state word, to whoever
// queues it next, and over the entry, to the warp that takes it. Each hand-over
// is a fence before the atomic that others read and a fence (or an acquire)
// after the one that reads it. The caller fences what a visit wrote before it
// calls mark or end.
//
// M names the memory operations: relaxed ones, RMWs that acquire, and fences
// (device: mf_lattice3.cu; a model that checks the order: the CPU tests).
#ifdef __CUDACC__
#define MF_QUEUE_FN __host__ __device__ __forceinline__
#else
#define MF_QUEUE_FN inline
#endif

namespace mf {

enum : int { QUEUED = 1, RUNNING = 2, FACES = 2, SEEDS = 64 << FACES };  // FACES: shift of the face bits

// Places of a queue: at most `tiles` are filled, and at most one per warp of the
// grid (2 tiles + 8, see lattice_grid) is waited for ahead of them.
MF_QUEUE_FN unsigned q_slots(int tiles) { return 3u * (unsigned)tiles + 8u; }

constexpr int Q_STRIDE = 8;      // ints per place: a sector of its own (idle warps look at neighbouring ones)
constexpr int Q_TILE_BITS = 23;  // of an entry: tile + 1 (there are at most 2^22 tiles); above them the lap

template <class M>
struct TileQueue {
  unsigned *ring;
  int *head, *tail;
  int *state;  // per tile
  int tiles;
  M m;

  MF_QUEUE_FN unsigned *place(unsigned i) const { return ring + (size_t)(i % q_slots(tiles)) * Q_STRIDE; }
  MF_QUEUE_FN unsigned entry(unsigned i, int t) const { return (i / q_slots(tiles)) << Q_TILE_BITS | (unsigned)(t + 1); }

  // Tile t joins the queue: `handed` after `mark` (what the last visitor of t wrote
  // was handed to this warp over the state word and is passed on), else after `end`
  // (the visitor is this warp, whose writes the caller fenced). False if the wait
  // for the place was given up (M::wait).
  MF_QUEUE_FN bool push(int t, bool handed) {
    const unsigned i = (unsigned)m.add(tail, 1);
    if (handed) m.release();
    for (unsigned spins = 1; m.cas(place(i), 0u, entry(i, t)) != 0; spins++)
      if (!m.wait(spins)) return false;
    return true;
  }
  // Tile t has work (an inbox of a face in `faces`, or lower labels around it):
  // true if it is to be pushed.
  MF_QUEUE_FN bool mark(int t, int faces) {
    return !(m.or_acquire(&state[t], QUEUED | (faces << FACES)) & (QUEUED | RUNNING));
  }
  // Starts the visit of tile t: its state word as it stood. What the warps that
  // marked t wrote before is visible after it.
  MF_QUEUE_FN int begin(int t) { return m.exch_acquire(&state[t], RUNNING); }
  // Ends the visit of tile t; `again`: it still has work. True if it is to be pushed.
  MF_QUEUE_FN bool end(int t, bool again) {
    if (again) m.or_relaxed(&state[t], QUEUED);
    return m.and_acquire(&state[t], ~RUNNING) & QUEUED;
  }

  MF_QUEUE_FN unsigned ticket() { return (unsigned)m.add(head, 1); }
  // The tile in the place of ticket i, -1 if it is not there yet.
  MF_QUEUE_FN int look(unsigned i) {
    const unsigned v = m.load(place(i));
    return v && v >> Q_TILE_BITS == entry(i, 0) >> Q_TILE_BITS ? (int)(v & ((1u << Q_TILE_BITS) - 1)) - 1 : -1;
  }
  // The warp with ticket i has seen its tile and takes it.
  MF_QUEUE_FN void take(unsigned i) {
    m.acquire();  // what was written before the entry was made is visible from here on
    m.store(place(i), 0u);
  }
};

}  // namespace mf
